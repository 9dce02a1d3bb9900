"""The force of the resident kernel (tile_accel): the kernel-level entry point evaluates the
same function as a propagation, bit for bit, so that what is shown of one holds for the other."""
import numpy as np
import pytest

from paper_2301_03989_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    import torch
    from paper_2301_03989_gb300 import build, pcprop
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return pcprop


def _dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("eih", [False, True])
@pytest.mark.parametrize("N", [40, 128])
def test_entry_point_is_the_force_of_a_propagation(pc, ora, N, eih):
    """One sweep from a cold start (every node at x0) over a segment with omega2 = 2^20 s
    exactly: its end state is x0 + omega2 K f, and scaling by a power of two changes no
    digit, so it equals the operator applied to omega2 times the forces of the entry point.
    States near Venus and far from every body; the ten-body system, indirect term on."""
    import torch
    w = W.config2(M=8)
    rng = np.random.default_rng(12)
    m = ora.Model.from_workload(w)
    t0, half = 2.0 ** 21, 2.0 ** 20
    tf = t0 + 2.0 * half
    venus = ora.ephem_eval(m, t0)[1]
    x0 = np.zeros((6, 6))
    for i in range(6):
        d = rng.standard_normal(3)
        x0[:3, i] = venus + d / np.linalg.norm(d) * 10.0 ** (4 + i) if i < 4 else rng.standard_normal(3) * 2e8
        x0[3:, i] = rng.standard_normal(3) * 30.0
    opts = pc.options_default(warm_start=0, trunc_tol=0.0, div_limit=1e30, max_depth=0)
    plan = pc.plan_create(N, 1, w.mu_central, w.mu, w.t_begin, w.granule, w.coef, w.indirect, opts,
                          c_light=299792.458 if eih else 0.0)
    xf = torch.zeros((6, 6), dtype=torch.float64, device="cuda")
    it = torch.zeros(6, dtype=torch.int32, device="cuda")
    code, _ = pc.propagate(plan, _dev(x0), t0, tf, xf, tol=1e25, iters=it)
    assert code == pc.PC_OK and (it.cpu().numpy() == 1).all()
    K, tau = pc.plan_operator(plan)
    t = (0.5 * (tf + t0) + half * tau)[:, None] + np.zeros(6)
    y = np.broadcast_to(x0[:, None, :], (6, N + 1, 6))                      # [component][node][trajectory]
    f = torch.zeros((6, (N + 1) * 6), dtype=torch.float64, device="cuda")
    pc.eval_dynamics(plan, _dev(t.reshape(-1)), _dev(y.reshape(6, -1)), f)
    g = (half * f).reshape(6, N + 1, 6).permute(1, 0, 2).contiguous()
    out = torch.zeros_like(g)
    pc.apply_operator(plan, _dev(x0), g, out)
    torch.cuda.synchronize()
    got, ref = xf.cpu().numpy(), out[N].cpu().numpy()
    if not eih:
        np.testing.assert_array_equal(got, ref)
    else:
        # the sweeps form both parts in one pass: two rounding orders of the same sum, each within
        # 2e-15 of its terms (the bound of the kernel-level dynamics test), over sum_j |K_Nj| = 2
        F = f.cpu().numpy().reshape(6, N + 1, 6)
        sep = np.abs(x0[:3] - venus[:, None])
        near = w.mu[1] / (sep ** 2).sum(0)
        mag = np.abs(F[3:]).max((0, 1)) + near + W.MU_SUN / (x0[:3] ** 2).sum(0)
        assert (np.abs(got[3:] - ref[3:]) <= 2 * 2 * half * 2e-15 * mag + 2e-16 * np.abs(ref[3:])).all()
        np.testing.assert_array_equal(got[:3], ref[:3])
    plan.close()
