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
