"""A CTA of the batched Hessian kernel that takes several items lays the next window's coefficient ring
over bytes that the last one used as halo and state.  Windows of every chunk width, with one column
group per item so that each CTA takes several, end as they do alone, run after run: eigenvalues to
1e-12, as in test_gpu_batch.py."""
import numpy as np
import pytest

from synth import configs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("S", [2, 4])
def test_items_of_several_shapes_per_cta(gpu_lib, S):
    R = gpu_lib
    from paper_1906_01413_gb300 import workloads
    spec = [(8192, 3, 64), (16, 12, 16), (4096, 4, 96), (333, 6, 128), (5001, 3, 64), (100, 9, 100), (2047, 4, 128), (40, 9, 40)]
    cfgs = [configs.L96Config(name="bi%d" % i, n=n, F=8.0, T=T, obs_every=2, obs_frac=0.3, obs_layout="random", ell=3.0,
                              k=k, q=0, spinup=100, seed=configs.BASE_SEED + 700 + i) for i, (n, T, k) in enumerate(spec)]
    ctxs, alone = [], []
    for c in cfgs:
        ctx, xb, _ = workloads.l96_twin(R, torch, c, DEV, R.RIOT_PREC_MIXED, c.k)
        R.riot_outer_begin(ctx.h, xb)
        alone.append(np.array(R.riot_rsvd(ctx.h, c.k, 0, sketch_stream=configs.STREAM_SKETCH0)))
        ctxs.append(ctx)
    b = R.riot_batch_create([ctx.h for ctx in ctxs], [c.k for c in cfgs], 0)
    R.riot_batch_set_config(b, 1, S)
    for _ in range(12):
        assert R.riot_batch_run(b, len(cfgs), sketch_stream=configs.STREAM_SKETCH0, use_graph=False) == [0] * len(cfgs)
        for c, ctx, want in zip(cfgs, ctxs, alone):
            lam = torch.empty(c.k, dtype=torch.float64, device=DEV)
            R.riot_get_state(ctx.h, lam=lam)
            np.testing.assert_allclose(lam.cpu().numpy(), want, rtol=1e-12, err_msg=c.name)
    R.riot_batch_destroy(b)
    for ctx in ctxs:
        ctx.close()
