"""Narrow layers take a form of the convolution that skips the channels a tile does not have.  A network
and the same one with zero channels added to its hidden layers (which takes the other form) give the
same outputs bit for bit: the added terms are zeros, the order of the others is the same."""
import numpy as np
import pytest

from oracle import sketchnet as N

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("c_in,width,m,ksize,n", [(8, 1, 64, 5, 131), (9, 3, 40, 3, 64), (8, 8, 33, 1, 257), (12, 9, 70, 7, 130),
                                                  (8, 31, 64, 5, 512), (16, 32, 65, 3, 129)])
def test_zero_channels_change_nothing(gpu_lib, c_in, width, m, ksize, n, bf16):
    R = gpu_lib
    rng = np.random.default_rng(width)
    wide = 48
    chan, pad = [c_in, width, width, m], [c_in, wide, wide, m]
    params, padded = [], []
    for o, c, po, pc in zip(chan[1:], chan, pad[1:], pad):
        W, b = rng.standard_normal((o, c, ksize)) / np.sqrt(c * ksize), 0.1 * rng.standard_normal(o)
        params.append((W, b))
        Wp, bp = np.zeros((po, pc, ksize)), np.zeros(po)
        Wp[:o, :c], bp[:o] = W, b
        padded.append((Wp, bp))
    x = torch.randn(2, c_in, n, device=DEV, generator=torch.Generator(device=DEV).manual_seed(n))
    out = []
    for p, w in ((params, width), (padded, wide)):
        net = R.riot_sketchnet_create(c_in, w, m, depth=3, ksize=ksize, n_max=n, batch_max=2, r_max=2)
        R.riot_sketchnet_set_params(net, torch.tensor(N.flatten(p).astype(np.float32), device=DEV))
        Z = torch.empty(2, m, n, dtype=torch.float32, device=DEV)
        R.riot_sketchnet_forward(net, x, Z, bf16=bf16)
        out.append(Z)
        R.riot_sketchnet_destroy(net)
    assert torch.equal(out[0], out[1])
    if not bf16:
        ref, _ = N.forward([(W.astype(np.float32).astype(float), b.astype(np.float32).astype(float)) for W, b in params],
                           x[1].double().cpu().numpy())
        np.testing.assert_allclose(out[0][1].cpu().numpy(), ref, atol=1e-5 * np.abs(ref).max())
