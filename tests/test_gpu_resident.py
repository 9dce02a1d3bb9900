"""The resident FP64 kernel (one launch per propagation).  Its digit products are
exact sums, so a trajectory's result is bitwise the same whatever batch, tile size
(1 to 16 slots per CTA) or scratch placement it ran with; it agrees with the
oracle within the parity tolerance and, being the same fixed point stopped at
1e-13, with the launch-per-step rounds (FP64 tensor cores) within 1e-11."""
import numpy as np
import pytest

from paper_2301_03989_gb300 import workloads as W
from test_gpu_parity import TOL, rel_err, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    import torch
    from paper_2301_03989_gb300 import build, pcprop
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return pcprop


def _work(M, N, segments, years=0.3, bodies=2):
    w = W.config3(M=M, seed=11)
    w.N, w.segments, w.tf = N, segments, years * W.YEAR
    w.x0 = w.x0 * (1.0 + 1e-3 * np.random.default_rng(3).standard_normal(w.x0.shape))
    w.mu, w.coef = w.mu[:bodies], w.coef[:bodies]
    return w


def _run(pc, w, n, **opts):
    import torch
    plan = pc.plan_from_workload(w, **opts)
    x0 = torch.as_tensor(W.to_planar(w.x0[:n]), device="cuda")
    xf = torch.zeros_like(x0)
    st = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    it, ns = torch.zeros_like(st), torch.zeros_like(st)
    code, _ = pc.propagate(plan, x0, w.t0, w.tf, xf, status=st, iters=it, nseg=ns)
    torch.cuda.synchronize()
    plan.close()
    return code, W.from_planar(xf.cpu().numpy()), st.cpu().numpy(), it.cpu().numpy(), ns.cpu().numpy()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("N", [32, 65, 128])
def test_batch_sizes_are_bitwise_neutral(pc, order, N, precision):
    """Sizes on both sides of every change of shape: 1, 2, 4 and 8 slots per CTA and, at
    degree 128 for the largest, the tcgen05 product (65 rows of 128 filled at degree 65)."""
    w = _work(5000, N, {32: 12, 65: 8, 128: 6}[N], years=0.3 if N == 32 else 0.15)
    prec = pc.PC_PREC_MIXED if precision == "mixed" else pc.PC_PREC_FP64
    full = _run(pc, w, w.n_ic, order=order, precision=prec)
    assert full[0] == pc.PC_OK
    for n in (1, 3, 152, 305, 609, 1217, 1300, 2433):
        part = _run(pc, w, n, order=order, precision=prec)
        assert part[0] == pc.PC_OK
        for a, b in zip(part[1:], full[1:]):
            np.testing.assert_array_equal(a, b[:n], err_msg=str(n))


@pytest.mark.parametrize("order,N,segments,bodies",
                         [(o, *c) for o in (1, 2) for c in ((8, 60, 2), (20, 20, 2), (33, 12, 0), (100, 6, 1), (255, 4, 2))]
                         + [(1, 256, 4, 2), (1, 287, 4, 2)])
def test_against_oracle_and_rounds(pc, ora, order, N, segments, bodies):
    """Degrees that leave ragged k-steps and node tiles, no and one body, degrees beyond
    255 (first order)."""
    w = _work(5, N, segments, years=0.15, bodies=bodies)
    g = _run(pc, w, 5, order=order)
    o = run_oracle(ora, w, w.x0, order=order)
    np.testing.assert_array_equal(g[2], o["status"])
    np.testing.assert_array_equal(g[4], o["nseg"])
    er, ev = rel_err(g[1], o["xf"])
    assert er.max() < TOL and ev.max() < TOL
    for prec in (pc.PC_PREC_FP64, pc.PC_PREC_MIXED):
        m = g if prec == pc.PC_PREC_FP64 else _run(pc, w, 5, order=order, precision=prec)
        # the rounds, on the FP64 tensor cores (first order only)
        r = _run(pc, w, 5, precision=prec, contraction=pc.PC_CONTRACT_DMMA)
        er, ev = rel_err(m[1], r[1])
        assert m[0] == r[0] and er.max() < 1e-11 and ev.max() < 1e-11


def test_adjoint_batch_sizes_are_bitwise_neutral(pc):
    """The reverse sweep's shapes (one slot in 256 or 128 threads, two slots) and the
    scratch placement change no bit of a trajectory's gradient."""
    import torch
    w = _work(1300, 32, 12)
    plan = pc.plan_from_workload(w)
    rec, cap = pc.tape_record(plan), 12
    dev = dict(dtype=torch.float64, device="cuda")
    x0 = torch.as_tensor(W.to_planar(w.x0), device="cuda")
    xb = torch.as_tensor(np.random.default_rng(5).standard_normal((6, w.n_ic)), device="cuda")
    full = None
    for n in (1300, 1, 3, 305, 700, 1217):
        t0, tf = torch.full((n,), w.t0, **dev), torch.full((n,), w.tf, **dev)
        a, b = x0[:, :n].contiguous(), xb[:, :n].contiguous()
        xf, out = torch.empty_like(a), torch.empty_like(a)
        ns = torch.zeros(n, dtype=torch.int32, device="cuda")
        tape = torch.empty(n * cap * rec, **dev)
        it, st = torch.zeros_like(ns), torch.zeros_like(ns)
        assert pc.propagate_tape(plan, a, t0, tf, xf, ns, tape, cap) == pc.PC_OK
        assert pc.adjoint_tape(plan, ns, cap, tape, b, out, status=st, iters=it) == pc.PC_OK
        torch.cuda.synchronize()
        got = (out.clone(), it.clone(), st.clone())
        full = full or got
        for x, y in zip(got, full):
            assert torch.equal(x, y[..., :n]), n
    plan.close()
