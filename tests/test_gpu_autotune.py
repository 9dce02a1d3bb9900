"""The autotuner on plans whose propagations run resident (which read no launch tuning) and on
plans that run rounds (FP64 tensor cores)."""
import pytest

from paper_2301_03989_gb300 import workloads as W
from test_gpu_tuning import DEFAULT_TUNING, _run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    import torch
    from paper_2301_03989_gb300 import build, pcprop
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return pcprop


def _plan(pc, w, **opts):
    import torch
    return pc.plan_from_workload(w, **opts), torch.as_tensor(W.to_planar(w.x0), device="cuda")


@pytest.mark.parametrize("precision", [0, 1])
def test_resident_plan_is_not_timed(pc, precision):
    w = W.config1(M=16)
    plan, x0 = _plan(pc, w, precision=precision)
    pc.kernel_times(plan)
    assert pc.autotune(plan, x0, w.t0, w.tf, max_rounds=16) == DEFAULT_TUNING == pc.get_tuning(plan)
    assert pc.kernel_times(plan)["kernel_launches"] == 0
    # what a trial would have refused is still refused
    for t0, tf in ((w.t0, 1e30), (float("nan"), w.tf)):
        with pytest.raises(pc.PCError) as e:
            pc.autotune(plan, x0, t0, tf, max_rounds=16)
        assert e.value.code == pc.PC_EINVAL
    plan.close()


def test_rounds_are_timed_and_the_choice_is_neutral(pc):
    import torch
    w = W.config2(M=256)
    plan, x0 = _plan(pc, w, precision=pc.PC_PREC_MIXED, contraction=pc.PC_CONTRACT_DMMA)
    tf = 0.1 * W.YEAR
    base = _run(pc, plan, w, x0, tf)
    pc.kernel_times(plan)
    best = pc.autotune(plan, x0, w.t0, tf, max_rounds=32)
    assert pc.kernel_times(plan)["kernel_launches"] > 0
    assert pc.get_tuning(plan) == best
    r = _run(pc, plan, w, x0, tf)
    for a, b in zip(base[2:], r[2:]):
        assert torch.equal(a, b)
    plan.close()
