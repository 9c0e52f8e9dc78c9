"""J of riot_outer_begin on a Lorenz-96 window is formed in a fixed order: the same bits every time (at
v = 0), and the oracle's cost to 1e-12.  One CTA of observations, a part of one, and more observations
than the CTAs take at once."""
import numpy as np
import pytest

from oracle import l96

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("n,per_step,T", [(40, 1, 1), (300, 256, 1), (1000, 777, 6), (8000, 8000, 20)])
def test_cost_is_the_same_every_time(gpu_lib, n, per_step, T):
    R = gpu_lib
    rng = np.random.default_rng(n)
    st = np.repeat(np.arange(1, T + 1), per_step)
    ix = np.concatenate([np.sort(rng.choice(n, per_step, replace=False)) for _ in range(T)])
    x = l96.nl(8.0 + rng.standard_normal(n), 20, 0.05, 8.0)[-1]
    sig, y = 0.3 + rng.random(st.size), 8.0 + 3.0 * rng.standard_normal(st.size)
    ctx = R.Context(n=n, T=T, dt=0.01, F=8.0, obs_step=st, obs_idx=ix, obs_y=y, obs_sigma=sig, length=2.0, kmax=4)
    xd = torch.tensor(x, device=DEV)
    J = [R.riot_outer_begin(ctx.h, xd) for _ in range(40)]
    ctx.close()
    want = 0.5 * np.sum(((l96.nl(x, T, 0.01, 8.0)[st, ix] - y) / sig) ** 2)
    assert abs(J[0] - want) <= 1e-12 * want
    assert set(J) == {J[0]}
