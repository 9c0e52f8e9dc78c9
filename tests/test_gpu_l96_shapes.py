"""The FP32 Lorenz-96 product picks one or two columns per thread and the columns of a CTA by their
number; a column's arithmetic is the same in every shape, so its product is the same bit for bit
whether it is applied alone, with a few others or with many."""
import numpy as np
import pytest

from oracle import l96

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("n,T,many", [(40, 9, 700), (111, 6, 333), (1003, 5, 401), (4096, 4, 320)])
def test_products_do_not_depend_on_the_column_count(gpu_lib, n, T, many):
    R = gpu_lib
    rng = np.random.default_rng(n)
    st, ix = np.repeat(np.arange(T + 1), n // 3), np.concatenate([np.sort(rng.choice(n, n // 3, False)) for _ in range(T + 1)])
    ctx = R.Context(n=n, T=T, dt=0.02, F=8.0, obs_step=st, obs_idx=ix, obs_y=np.zeros(st.size), obs_sigma=np.ones(st.size),
                    length=2.5, kmax=many)
    R.riot_outer_begin(ctx.h, torch.tensor(l96.nl(8.0 + rng.standard_normal(n), 50, 0.05, 8.0)[-1], device=DEV))
    W = torch.randn(many, n, device=DEV, generator=torch.Generator(device=DEV).manual_seed(n))
    Y = torch.empty_like(W)
    R.riot_hessian_apply(ctx.h, W, Y)
    for nc in (1, 2, 5, 77):
        y = torch.empty(nc, n, device=DEV)
        R.riot_hessian_apply(ctx.h, W[many - nc:].contiguous(), y)
        assert torch.equal(y, Y[many - nc:])
    ctx.close()
