"""Sketch network kernels at the edges of their tiles: odd positions and channels, every tap count,
one window and several, more targets than directions.  Reference: the FP64 oracle; tolerances as
in test_gpu_sketchnet.py (outputs 1e-5 of their scale, gradients 1e-4 in the 2-norm)."""
import numpy as np
import pytest

from oracle import sketchnet as N

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("c_in,width,m,ksize,n,B,r", [(1, 1, 1, 1, 16, 1, 2), (3, 9, 5, 3, 131, 2, 7),
                                                      (5, 67, 70, 5, 257, 1, 66), (8, 64, 128, 7, 300, 9, 64)])
def test_loss_and_gradient(gpu_lib, c_in, width, m, ksize, n, B, r):
    R = gpu_lib
    rng = np.random.default_rng(n)
    chan = [c_in, width, width, m]
    params = [(rng.standard_normal((o, c, ksize)) / np.sqrt(c * ksize), 0.1 * rng.standard_normal(o))
              for c, o in zip(chan, chan[1:])]
    flat = N.flatten(params).astype(np.float32)
    params = N.unflatten(flat.astype(np.float64), [W.shape for W, _ in params])
    xs = rng.standard_normal((B, c_in, n)).astype(np.float32)
    Us = np.stack([np.linalg.qr(rng.standard_normal((n, r)))[0].T for _ in range(B)]).astype(np.float32)
    net = R.riot_sketchnet_create(c_in, width, m, depth=3, ksize=ksize, n_max=n + 5, batch_max=B, r_max=r + 3)
    R.riot_sketchnet_set_params(net, torch.tensor(flat, device=DEV))
    x, U = torch.tensor(xs, device=DEV), torch.tensor(Us, device=DEV).contiguous()
    Z = torch.empty(B, m, n, dtype=torch.float32, device=DEV)
    R.riot_sketchnet_forward(net, x, Z)
    ref, _ = N.forward(params, xs[-1].astype(np.float64))
    np.testing.assert_allclose(Z[-1].cpu().numpy(), ref, atol=1e-5 * np.abs(ref).max())
    g = torch.empty(flat.size, dtype=torch.float32, device=DEV)
    L = R.riot_sketchnet_loss_grad(net, x, U, 0.2, g)
    Lo, go = N.batch_loss_grad(params, [v.astype(np.float64) for v in xs], [V.T.astype(np.float64) for V in Us], 0.2)
    go = N.flatten(go)
    assert L == pytest.approx(Lo, rel=1e-5)
    assert np.linalg.norm(g.cpu().numpy() - go) <= 1e-4 * max(np.linalg.norm(go), 1e-3)
    # a network whose products leave the FP32 range ends as sums in 64 bits do
    R.riot_sketchnet_forward(net, x * 1e30, Z)
    assert bool(torch.isfinite(Z).all())
    R.riot_sketchnet_destroy(net)
