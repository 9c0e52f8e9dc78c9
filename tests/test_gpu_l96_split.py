"""FP64 Lorenz-96 integrations of a few columns with the state split over CTAs, at the sizes where
the split can go wrong: rings of one CTA (n <= 256) and the first split state, more steps than one
launch takes, no steps, observations of the initial state only, steps after the last observation,
repeated observations.  Tolerances as for the other FP64 products: 1e-10 of the column norm."""
import numpy as np
import pytest

from oracle import bcov, l96, riot as orc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def _problem(n, T, steps, dup):
    rng = np.random.default_rng(1000 * n + T)
    ix = np.sort(rng.choice(n, max(1, n // 3), replace=False))
    if dup:
        ix = np.sort(np.concatenate([ix, ix[:3]]))
    st, ix = np.repeat(steps, ix.size), np.tile(ix, len(steps))
    x0 = l96.nl(8.0 + rng.standard_normal(n), 60, 0.05, 8.0)[-1]
    sig = 0.5 + rng.random(st.size)
    y = l96.nl(x0, T, 0.02, 8.0)[st, ix] + sig * rng.standard_normal(st.size)
    L = bcov.bsqrt(n, 2.0, 1.0)
    return orc.L96Problem(n=n, T=T, dt=0.02, F=8.0, obs_step=st, obs_idx=ix, y=y, sigma_o=sig, L=L,
                          x_b=x0 + L @ rng.standard_normal(n))


@pytest.mark.parametrize("n,T,steps,dup", [(16, 1, [1], False), (33, 0, [0], True), (64, 5, [0], True),
                                           (256, 50, [0, 7, 49], False), (257, 50, [3, 48], True),
                                           (300, 13, [0, 13], True), (4111, 11, [2, 9], False)])
def test_split_integrations_match_the_oracle(gpu_lib, n, T, steps, dup):
    R = gpu_lib
    prob = _problem(n, T, steps, dup)
    traj = orc.trajectory(prob, prob.x_b)
    d = orc.innovation(prob, traj)
    W = np.random.default_rng(3).standard_normal((n, 3))
    ref = orc.hvp(prob, traj, W)
    gref = orc.gradient_b(prob, traj, d)
    for prec in (R.RIOT_PREC_FP64, R.RIOT_PREC_MIXED):
        ctx = R.Context(n=n, T=T, dt=prob.dt, F=prob.F, obs_step=prob.obs_step, obs_idx=prob.obs_idx, obs_y=prob.y,
                        obs_sigma=prob.sigma_o, length=2.0, sigma_b=1.0, precision=prec, kmax=3)
        J = R.riot_outer_begin(ctx.h, _t(prob.x_b))
        assert abs(J - 0.5 * np.sum((d / prob.sigma_o) ** 2)) <= 1e-12 * J
        g, dd = torch.empty(n, dtype=torch.float64, device=DEV), torch.empty(d.size, dtype=torch.float64, device=DEV)
        R.riot_get_state(ctx.h, g=g)
        R.riot_get_innovation(ctx.h, dd)
        np.testing.assert_allclose(g.cpu().numpy(), gref, rtol=0, atol=1e-10 * np.linalg.norm(gref))
        np.testing.assert_allclose(dd.cpu().numpy(), d, rtol=0, atol=1e-10 * np.abs(d).max())
        # the quadratic cost at 0 and at a step: the tangent-linear half alone
        dv = _t(0.1 * W[:, 0])
        Hdv = R.riot_quadratic_cost(ctx.h, dv)
        want = J + gref @ (0.1 * W[:, 0]) + 0.005 * W[:, 0] @ (W[:, 0] + ref[:, 0])
        assert abs(Hdv - want) <= 1e-10 * abs(want)
        if prec == R.RIOT_PREC_FP64:
            for nc in (1, 3):   # columns given at once take the same steps
                Wt = _t(W[:, :nc].T)
                Y = torch.empty_like(Wt)
                R.riot_hessian_apply(ctx.h, Wt, Y, add_identity=(nc == 3))
                got = Y.cpu().numpy().T - (W if nc == 3 else 0)
                err = np.linalg.norm(got - ref[:, :nc], axis=0) / np.linalg.norm(ref[:, :nc], axis=0)
                assert err.max() < 1e-10
        ctx.close()


@pytest.mark.parametrize("n,T", [(100, 97), (700, 30)])
def test_forecast_in_place(gpu_lib, n, T):
    """Only the final state is kept, in the start's own memory."""
    R = gpu_lib
    x0 = 8.0 + np.random.default_rng(n).standard_normal(n)
    x = _t(x0)
    R.riot_l96_forecast(n, T, 0.01, 8.0, x, x, store_all=False)
    ref = l96.nl(x0, T, 0.01, 8.0)[-1]
    np.testing.assert_allclose(x.cpu().numpy(), ref, rtol=0, atol=1e-11 * np.abs(ref).max())
