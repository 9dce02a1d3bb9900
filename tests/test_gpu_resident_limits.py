"""The resident kernel where its launch is near a limit: shared memory of one block,
and several host threads launching the same kernel at different sizes."""
import numpy as np
import pytest

from paper_2301_03989_gb300 import workloads as W
from test_gpu_resident import _run, _work

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    import torch
    from paper_2301_03989_gb300 import build, pcprop
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return pcprop


@pytest.mark.parametrize("N,bodies,M", [(71, 0, 500), (71, 1, 400), (72, 1, 400)])
def test_scratch_at_the_shared_memory_limit(pc, N, bodies, M):
    """16-slot tiles whose scratch ends within 2 KB of what a block may have: the call is
    served, and as single slots (whose scratch is far below the limit) give it."""
    w = _work(M, N, 8, bodies=bodies)
    code, xf, st, it, ns = _run(pc, w, M, order=2)
    assert code == pc.PC_OK
    one = _run(pc, w, 100, order=2)
    for a, b in zip((xf[:100], st[:100], it[:100], ns[:100]), one[1:]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("reverse", [False, True])
def test_threads_with_plans_of_different_sizes(pc, reverse):
    """One plan and stream a thread, the same kernel instance in all (a single slot, one
    thread at degree 128 and three at degree 16): no launch is refused for the shared
    memory that another thread's needs."""
    import threading
    import torch
    errors, barrier, over = [], threading.Barrier(4), threading.Event()

    def worker(N):
        try:
            w = _work(1, N, 1, years=0.002)
            plan = pc.plan_from_workload(w)
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                x0 = torch.as_tensor(W.to_planar(w.x0), device="cuda")
                xf, out, bar = torch.zeros_like(x0), torch.zeros_like(x0), torch.ones_like(x0)
                arc = torch.tensor([w.t0, w.tf], dtype=torch.float64, device="cuda")
                ns = torch.zeros(1, dtype=torch.int32, device="cuda")
                tape = torch.empty(pc.tape_record(plan), dtype=torch.float64, device="cuda")
                pc.propagate_tape(plan, x0, arc[:1], arc[1:], xf, ns, tape, 1, stream=stream)
                stream.synchronize()
                barrier.wait()
                for _ in range(2000):
                    if reverse:
                        pc.adjoint_tape(plan, ns, 1, tape, bar, out, stream=stream)
                    else:
                        pc.propagate(plan, x0, w.t0, w.tf, xf, stream=stream)
                    if N < 128 and over.is_set():
                        break
            plan.close()
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(e)
            barrier.abort()
        if N == 128:
            over.set()

    threads = [threading.Thread(target=worker, args=(N,)) for N in (128, 16, 16, 16)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
