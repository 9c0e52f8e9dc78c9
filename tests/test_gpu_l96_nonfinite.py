"""An infinity or NaN in a column of an FP64 product reaches what the observations and the model carry it
to and nothing else: with only the initial state observed, and not at the places that are not finite,
the product is that of the column with zeros there (to the FP64 bound of the other tests)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("n,T,nc", [(100, 0, 1), (100, 2, 1), (700, 0, 1), (700, 1, 2), (4100, 1, 1), (300, 1, 60)])
def test_columns_that_are_not_finite(gpu_lib, n, T, nc, value):
    R = gpu_lib
    at = [0, n // 2]                                  # unobserved, and so are the neighbours L reaches
    ix = np.array([i for i in range(n) if min(min(abs(i - a), n - abs(i - a)) for a in at) > 12])
    ctx = R.Context(n=n, T=T, dt=0.01, F=8.0, obs_step=np.zeros(ix.size), obs_idx=ix, obs_y=np.zeros(ix.size),
                    obs_sigma=np.full(ix.size, 0.5), length=0.5, precision=R.RIOT_PREC_FP64, kmax=max(nc, 2))
    R.riot_outer_begin(ctx.h, torch.linspace(1, 9, n, dtype=torch.float64, device=DEV))
    W = torch.randn(nc, n, dtype=torch.float64, device=DEV, generator=torch.Generator(device=DEV).manual_seed(n))
    W[:, at] = 0.0
    want, got = torch.empty_like(W), torch.empty_like(W)
    R.riot_hessian_apply(ctx.h, W, want)
    W[0, at] = value
    R.riot_hessian_apply(ctx.h, W, got)
    ctx.close()
    assert bool(torch.isfinite(got).all())
    assert torch.linalg.norm(got - want).item() <= 1e-10 * torch.linalg.norm(want).item()
