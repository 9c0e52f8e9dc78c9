"""The FP32 Lorenz-96 product reads no shared memory that it has not written: applied after kernels
that left NaN in it, it gives the same bits as before, and the oracle's product to the FP32 bound
of the other tests (2e-5 of the column norm)."""
import numpy as np
import pytest

from oracle import bcov, l96, riot as orc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("n,nc,kernel", [(40, 3, "RIOT_HVP_CTA_BARRIER"), (1003, 152, "RIOT_HVP_CTA_BARRIER"),
                                         (1003, 400, "RIOT_HVP_CTA_BARRIER"), (1003, 400, "RIOT_HVP_CTA_TWO_PER_SM"),
                                         (8191, 40, "RIOT_HVP_CTA_BARRIER")])
def test_products_after_nan(gpu_lib, n, nc, kernel):
    R = gpu_lib
    T, rng = 4, np.random.default_rng(n)
    ix = np.sort(rng.choice(n, n // 3, replace=False))
    st, ix = np.repeat([0, 2, T], ix.size), np.tile(ix, 3)
    x0 = l96.nl(8.0 + rng.standard_normal(n), 50, 0.05, 8.0)[-1]
    ctx = R.Context(n=n, T=T, dt=0.02, F=8.0, obs_step=st, obs_idx=ix, obs_y=np.zeros(st.size),
                    obs_sigma=np.ones(st.size), length=2.0, kmax=nc)
    R.riot_set_hvp_kernel(ctx.h, getattr(R, kernel))
    R.riot_outer_begin(ctx.h, torch.tensor(x0, device=DEV))
    W = torch.randn(nc, n, device=DEV, generator=torch.Generator(device=DEV).manual_seed(n))
    first, Y = torch.empty_like(W), torch.empty_like(W)
    R.riot_hessian_apply(ctx.h, W, first)
    if n <= 1003:
        prob = orc.L96Problem(n=n, T=T, dt=0.02, F=8.0, obs_step=st, obs_idx=ix, y=np.zeros(st.size),
                              sigma_o=np.ones(st.size), L=bcov.bsqrt(n, 2.0, 1.0), x_b=x0)
        ref = orc.hvp(prob, orc.trajectory(prob, x0), W[:3].double().cpu().numpy().T).T
        err = np.linalg.norm(first[:3].double().cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)
        assert err.max() < 2e-5
    bad = torch.full((512, 512), float("nan"), dtype=torch.float64, device=DEV)
    for _ in range(25):
        with pytest.raises(RuntimeError):
            R.riot_symm_eig(bad, bad.new_empty(512), torch.empty_like(bad))
        R.riot_hessian_apply(ctx.h, W, Y)
        assert torch.equal(Y, first)
    ctx.close()
