"""The reverse sweep applies the operator as the plan asks: PC_CONTRACT_DMMA on the FP64 tensor
cores (one launch per segment step back), PC_CONTRACT_SPLIT by digit products (one launch)."""
import numpy as np
import pytest

from paper_2301_03989_gb300 import workloads as W
from test_gpu_resident import _work

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    import torch
    from paper_2301_03989_gb300 import build, pcprop
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return pcprop


@pytest.mark.parametrize("N,segments", [(32, 12), (128, 4), (200, 3)])
def test_contraction_of_the_reverse_sweep(pc, N, segments):
    import torch
    w = _work(9, N, segments)
    x0 = torch.as_tensor(W.to_planar(w.x0), device="cuda")
    bar = torch.as_tensor(np.random.default_rng(8).standard_normal((6, 9)), device="cuda")
    got = {}
    for mode in (pc.PC_CONTRACT_DMMA, pc.PC_CONTRACT_SPLIT):
        plan = pc.plan_from_workload(w, contraction=mode)
        t0 = torch.full((9,), w.t0, dtype=torch.float64, device="cuda")
        tf = torch.full((9,), w.tf, dtype=torch.float64, device="cuda")
        ns = torch.zeros(9, dtype=torch.int32, device="cuda")
        xf, out = torch.zeros_like(x0), torch.zeros_like(x0)
        tape = torch.empty(9 * 2 * segments * pc.tape_record(plan), dtype=torch.float64, device="cuda")
        assert pc.propagate_tape(plan, x0, t0, tf, xf, ns, tape, 2 * segments) == pc.PC_OK
        pc.kernel_times(plan)
        assert pc.adjoint_tape(plan, ns, 2 * segments, tape, bar, out) == pc.PC_OK
        torch.cuda.synchronize()
        launches = pc.kernel_times(plan)["kernel_launches"]
        assert launches == (int(ns.max()) if mode == pc.PC_CONTRACT_DMMA else 1)
        got[mode] = out.cpu().numpy()
        plan.close()
    a, b = got.values()
    # both sweeps stop at a change of 1e-13, on forward nodes that differ by no more
    for h in (slice(0, 3), slice(3, 6)):
        size = np.linalg.norm(b[h], axis=0)
        assert (np.linalg.norm(a[h] - b[h], axis=0) <= 1e-11 * size).all()
