"""The rounds of kernels (plans on the FP64 tensor cores, and degrees whose digit sums are not
exact): launch tuning, CUDA graphs, compaction, the FP32 kernels' shapes and contractions, the
grid cache and EIH, which plans with the default contraction run no more; and the degrees that
take the rounds whatever the plan asks."""
import numpy as np
import pytest

from paper_2301_03989_gb300 import workloads as W
from test_gpu_eih import run_gpu_eih, run_oracle_eih
from test_gpu_parity import TOL, rel_err, run_gpu, run_oracle
from test_gpu_resident import _work
from test_gpu_tuning import DEFAULT_TUNING, _run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    import torch
    from paper_2301_03989_gb300 import build, pcprop
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return pcprop


def _rounds_plan(pc, w, precision, **opts):
    import torch
    plan = pc.plan_from_workload(w, precision=precision, contraction=pc.PC_CONTRACT_DMMA, **opts)
    return plan, torch.as_tensor(W.to_planar(w.x0), device="cuda")


def _same(a, b, note):
    import torch
    for x, y in zip(a[2:], b[2:]):
        assert torch.equal(x, y), note


SETTINGS = {
    0: [dict(graphs=0), dict(rounds_per_batch=2), dict(contract_ctas_per_sm=1, setup_ctas_per_sm=1),
        dict(contract_ctas_per_sm=16, setup_ctas_per_sm=16), dict(repack_div=2, rounds_per_batch=16),
        dict(repack_div=64, rounds_per_batch=5), dict(grid_cache=0)],
    1: [dict(graphs=0), dict(rounds_per_batch=2, contract_ctas_per_sm=1), dict(side_priority=0, grid_cache=0),
        dict(repack_div=2, rounds_per_batch=16, fp32_ctas_per_sm=16), dict(fp32_rows=0, fp32_ctas_per_sm=4),
        dict(fp32_rows=4, fp32_slots=8, fp32_ctas_per_sm=2), dict(fp32_rows=8, fp32_slots=32),
        dict(fp32_rows=4, fp32_slots=64, fp32_ctas_per_sm=3), dict(fp32_rows=8, fp32_slots=16, graphs=0)],
}


@pytest.mark.parametrize("precision,workload,fp32_mma", [(0, "flyby", 0), (0, "study", 0), (1, "flyby", 0),
                                                         (1, "study", 0), (1, "study", 1)])
def test_tuning_is_bitwise_neutral(pc, precision, workload, fp32_mma):
    """Ten bodies with segments by osculating period (every grid its own) and the three-body
    study on a common arc (shared grids); a stream of the caller's besides."""
    import torch
    w = W.config2(M=384) if workload == "flyby" else W.config3(M=600)
    tf = (0.15 if workload == "flyby" else 0.3) * W.YEAR
    plan, x0 = _rounds_plan(pc, w, precision, fp32_mma=fp32_mma, switch_tol=1e-6 if workload == "study" else 0.0)
    base = _run(pc, plan, w, x0, tf)
    assert base[0] in (pc.PC_OK, pc.PC_ENOTCONV)
    for kw in SETTINGS[precision]:
        pc.set_tuning(plan, **kw)
        _same(base, _run(pc, plan, w, x0, tf), kw)
        pc.set_tuning(plan, **DEFAULT_TUNING)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        _same(base, _run(pc, plan, w, x0, tf, stream=s), "stream")
    plan.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_grid_cache_two_epochs_and_over_capacity(pc, precision):
    """Arcs from two epochs (two families of grids in a round); in FP64 also 40,000 segments of
    their own lengths in the first round, more grids than the cache's 32,768."""
    import torch
    w = W.config3(M=500)
    plan, x0 = _rounds_plan(pc, w, precision, switch_tol=1e-6 if precision else 0.0)
    t0 = torch.full((500,), w.t0, dtype=torch.float64, device="cuda")
    t0[1::2] += 3.0 * W.DAY
    tf, outs = t0 + 0.2 * W.YEAR, []
    for gc in (1, 0):
        pc.set_tuning(plan, grid_cache=gc)
        xf = torch.zeros_like(x0)
        assert pc.propagate_groups([plan], [500], x0, t0, tf, xf)[0] == pc.PC_OK
        torch.cuda.synchronize()
        outs.append(xf)
    assert torch.equal(*outs)
    plan.close()
    if precision == 0:
        w = W.config2(M=40000)
        plan, x0 = _rounds_plan(pc, w, 0)
        base = _run(pc, plan, w, x0, w.t0 + 2.0 * W.DAY)
        pc.set_tuning(plan, grid_cache=0)
        _same(base, _run(pc, plan, w, x0, w.t0 + 2.0 * W.DAY), "over capacity")
        plan.close()


def test_fp32_mma_sweeps_and_error(pc, ora):
    """TF32 tensor-core sweeps against FP32 multiply-adds: the oracle's result, and the FP64 and
    FP32 sweeps within 2 and 10 per cent."""
    w = W.config3(M=128)
    o = run_oracle(ora, w, w.x0)
    counts = {}
    for mma in (0, 1):
        plan, x0 = _rounds_plan(pc, w, 1, fp32_mma=mma, switch_tol=1e-6)
        pc.kernel_times(plan)
        r = _run(pc, plan, w, x0, w.tf)
        kt = pc.kernel_times(plan)
        counts[mma] = (kt["sweeps64"], kt["sweeps32"])
        er, ev = rel_err(W.from_planar(r[2].cpu().numpy()), o["xf"])
        assert r[0] == pc.PC_OK and er.max() < TOL and ev.max() < TOL
        plan.close()
    assert abs(counts[1][0] - counts[0][0]) <= 0.02 * counts[0][0]
    assert abs(counts[1][1] - counts[0][1]) <= 0.1 * counts[0][1]


@pytest.mark.parametrize("precision", [0, 1])
def test_eih_on_the_rounds(pc, ora, precision):
    w = W.config2(M=16)
    tf = 20 * W.DAY
    g = run_gpu_eih(pc, w, w.x0, tf=tf, precision=precision, contraction=pc.PC_CONTRACT_DMMA)
    o = run_oracle_eih(ora, w, w.x0, tf=tf)
    er, ev = rel_err(g["xf"], o["xf"])
    assert er.max() < TOL and ev.max() < TOL, (er.max(), ev.max())


@pytest.mark.parametrize("N,truncated,precision", [(270, 1, 0), (275, 1, 1), (276, 1, 0), (276, 1, 1), (287, 1, 0),
                                                   (288, 0, 0), (300, 0, 0), (511, 0, 0)])
def test_degrees_around_the_digit_limit(pc, ora, N, truncated, precision):
    """Truncated operators whose digit sums are exact (270, 275) and are not (276, 287), and the
    degrees beyond 287: forward against the oracle, the gradient against that of degree 64."""
    import torch
    w = _work(5, N, 4, years=0.15)
    g = run_gpu(pc, w, w.x0, truncated=truncated, precision=precision)
    o = run_oracle(ora, w, w.x0)
    assert g["code"] == pc.PC_OK
    er, ev = rel_err(g["xf"], o["xf"])
    assert er.max() < TOL and ev.max() < TOL, (er.max(), ev.max())
    if precision or N > 400:
        return
    bar = torch.as_tensor(np.random.default_rng(6).standard_normal((6, 5)), device="cuda")
    x0 = torch.as_tensor(W.to_planar(w.x0), device="cuda")
    grads = []
    for degree, opts in ((N, dict(truncated=truncated)), (64, {})):
        w.N = degree
        plan = pc.plan_from_workload(w, **opts)
        out = torch.zeros_like(x0)
        assert pc.propagate_adjoint(plan, x0, w.t0, w.tf, bar, out) == pc.PC_OK
        torch.cuda.synchronize()
        grads.append(out.cpu().numpy())
        plan.close()
    for h in (slice(0, 3), slice(3, 6)):
        assert (np.linalg.norm((grads[0] - grads[1])[h], axis=0) <= TOL * np.linalg.norm(grads[1][h], axis=0)).all()
