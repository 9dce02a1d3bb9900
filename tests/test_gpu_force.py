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


def _sky(center, granules, seed):
    """Bodies that stand still within a granule, in random directions: (mu_central, mu,
    positions [granule][body][3])."""
    rng = np.random.default_rng(seed)
    if center == "earth":  # Sun and Moon
        mu_c, mu, dist = 398600.4418, [W.MU_SUN, 4902.8], [1.496e8, 384400.0]
    else:                  # eight planets
        mu_c = W.MU_SUN
        mu = [2.2032e4, 3.24859e5, 3.986e5, 4.2828e4, 1.26686e8, 3.7931e7, 5.794e6, 6.8365e6]
        dist = [a * W.AU for a in (0.387, 0.723, 1.0, 1.524, 5.203, 9.54, 19.2, 30.1)]
    d = rng.standard_normal((granules, len(mu), 3))
    d *= (np.array(dist) * rng.uniform(0.95, 1.05, (granules, len(mu))) / np.linalg.norm(d, axis=2))[:, :, None]
    return mu_c, np.array(mu), d


def _force_error(pc, center, seed, **opts):
    """Largest error of the entry point's acceleration against extended precision, over the sum
    of the terms' sizes, for nodes from near the centre to beyond every body and close to bodies."""
    import torch
    G, per = 64, 40
    mu_c, mu, pos = _sky(center, G, seed)
    rng = np.random.default_rng(seed + 1)
    lo, hi = (7.0e3, 1.5e6) if center == "earth" else (0.3 * W.AU, 40.0 * W.AU)
    g = np.repeat(np.arange(G), per)
    u = rng.standard_normal((G * per, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    r = u * np.exp(rng.uniform(np.log(lo), np.log(hi), G * per))[:, None]
    near = rng.random(G * per) < 0.5       # by a body, between a 4th and a 200th of its distance from the centre
    b = rng.integers(0, len(mu), G * per)
    p = pos[g, b]
    r[near] = (p + u * (np.linalg.norm(p, axis=1) / rng.uniform(4.0, 200.0, G * per))[:, None])[near]
    t = g + 0.5
    coef = np.ascontiguousarray(pos.transpose(1, 0, 2)[..., None])  # [body][granule][axis][1]
    plan = pc.plan_create(32, 1, mu_c, mu, 0.0, 1.0, coef, True, pc.options_default(**opts))
    f = torch.zeros((6, G * per), dtype=torch.float64, device="cuda")
    pc.eval_dynamics(plan, _dev(t), _dev(np.concatenate([r.T, r.T])), f)
    torch.cuda.synchronize()
    plan.close()
    ld = np.longdouble
    R, P = r.astype(ld), pos[g].astype(ld)
    d = R[:, None] - P
    dn, pn, rn = (np.sqrt((x * x).sum(-1)) for x in (d, P, R))
    m = mu.astype(ld)
    ref = -ld(mu_c) * R / rn[:, None] ** 3 - (m[None, :, None] * (d / dn[..., None] ** 3 + P / pn[..., None] ** 3)).sum(1)
    mag = ld(mu_c) / rn ** 2 + (m * (1 / dn ** 2 + 1 / pn ** 2)).sum(1)
    return float((np.abs(f[3:].T.cpu().numpy() - ref).max(1) / mag).max())


@pytest.mark.parametrize("center", ["earth", "sun"])
def test_force_against_extended_precision(pc, center):
    """About the Earth the Sun's indirect term is up to a dozen times the central attraction;
    about the Sun bodies lie on both sides of the switch to float pairs.  Bound: eight
    roundings (the difference, the reciprocal cube, the product, the sum) of each term's size,
    as in the kernel-level dynamics test."""
    err = max(_force_error(pc, center, seed) for seed in range(4))
    assert err <= 2e-15, err


def test_indirect_term_does_not_depend_on_the_company(pc):
    """About the Earth, on per-trajectory arcs: slots that share their node times share the
    body data of one of them, which decides whether the FP64 term is formed with them or by
    the nodes that want it.  A trajectory's result is the same, bit for bit, alone, in company
    and with the body data of the call's table."""
    import torch
    mu_c, mu, pos = _sky("earth", 1, 3)
    coef = np.ascontiguousarray(pos.transpose(1, 0, 2)[..., None])
    M, tf = 2600, 4.0e5   # two and more slots a CTA
    rng = np.random.default_rng(4)
    a = np.exp(rng.uniform(np.log(5.0e3), np.log(8.0e5), M))   # Sun's term from 2^-11.4 to several times the Earth's
    u, v = rng.standard_normal((2, 3, M))
    u /= np.linalg.norm(u, axis=0)
    v -= (u * v).sum(0) * u
    v /= np.linalg.norm(v, axis=0)
    x0 = _dev(np.concatenate([a * u, np.sqrt(mu_c / a) * v]))
    plan = pc.plan_create(32, 40, mu_c, mu, 0.0, 1.0e6, coef, True, pc.options_default())

    def run(cols, common):
        x = x0[:, cols].contiguous()
        out = torch.zeros_like(x)
        if common:
            pc.propagate(plan, x, 0.0, tf, out)
        else:
            arc = torch.zeros((2, len(cols)), dtype=torch.float64, device="cuda")
            arc[1] = tf
            pc.propagate_groups([plan], [len(cols)], x, arc[0].contiguous(), arc[1].contiguous(), out)
        torch.cuda.synchronize()
        return out

    everyone = list(range(M))
    full = run(everyone, False)
    assert torch.equal(full, run(everyone, True))
    for cols in ([0], everyone[:700], everyone[1300::-1]):
        assert torch.equal(run(cols, False), full[:, cols])
    plan.close()
