"""FP32 tracer products on grids and column counts that take the level-marching stepper, at the
edges of its tiles: one and several tiles in x and y, even and odd nx, the fewest and the most
levels.  Reference: the FP64 products of the same window (compared with the oracle in
test_gpu_advdiff.py).  Tolerance: rounding errors along the 8 T stages of a product add like a
random walk, four roundings on the longest path per stage, times 4: 16 sqrt(8 T) 2^-24 of the
column norm."""
import numpy as np
import pytest

from synth import advdiff as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("nx,ny,nz,P", [(45, 23, 2, 128), (26, 28, 32, 128), (100, 56, 30, 64), (101, 57, 31, 64)])
def test_level_marching_products(gpu_lib, nx, ny, nz, P):
    R = gpu_lib
    T = 6
    cfg = S.AdvDiffConfig(name="lv", nx=nx, ny=ny, nz=nz, T=T, nblocks=2, n_hotspots=4, n_tracks=4, pts_per_track=50,
                          alt_lo=100.0, alt_hi=6000.0)
    u, v = cfg.winds()
    step, pos = cfg.tracks()
    pos[:, 2] = np.minimum(pos[:, 2], nz - 1.0)
    box = dict(nx=nx, ny=ny, nz=nz, nblocks=2, T=T, dt=cfg.dt, dx=cfg.dx, dy=cfg.dy, dz=cfg.dz, u=u, v=v,
               amp=cfg.amplitude(), kz=cfg.kz(), emis_b=cfg.background_emissions(), obs_step=step, obs_pos=pos,
               obs_y=np.zeros(step.size), obs_sigma=np.ones(step.size), length=cfg.ell, sigma_b=cfg.sigma_b, kmax=P)
    x = torch.tensor(0.2 * cfg.background_perturbation(), device=DEV)
    W = torch.randn(P, cfg.n, device=DEV, generator=torch.Generator(device=DEV).manual_seed(nx))
    out = {}
    for prec, dt in ((R.RIOT_PREC_FP64, torch.float64), (R.RIOT_PREC_MIXED, torch.float32)):
        ctx = R.Context(precision=prec, **box)
        R.riot_outer_begin(ctx.h, x)
        Y = torch.empty(P, cfg.n, dtype=dt, device=DEV)
        R.riot_hessian_apply(ctx.h, W.to(dt), Y)
        out[prec] = Y.double()
        ctx.close()
    err = (out[R.RIOT_PREC_MIXED] - out[R.RIOT_PREC_FP64]).norm(dim=1) / out[R.RIOT_PREC_FP64].norm(dim=1)
    assert float(err.max()) <= 16.0 * (8 * T) ** 0.5 * 2.0 ** -24
