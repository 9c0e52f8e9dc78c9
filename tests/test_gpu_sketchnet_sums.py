"""Weight gradients of the sketch network are sums of FP32 factors to the accuracy of sums in 64 bits:
where the terms of a lane cancel (to 2^-21 of their size), where products leave the FP32 range and
where they fall below it.  The second input channel has zero weights, so that its values x1 act on
its own weights' gradient alone, sum_i g[o][i] x1[i + d - h]; inputs and targets repeat every 32
positions, so that g does, to the bit, and x1 decides how the terms cancel.  Bound: 1e-3 of the gradient's
2-norm against the FP64 oracle.  g itself, FP32 as everywhere, is good to about 1e-6 of its largest
value and sums in 64 bits add nothing to that; rounding a lane's cancelling terms to FP32 once per
pair costs 2^-25 / 2^-21 = 6 % of what remains, products of 30 units of the smallest FP32 number
rounded one by one about 1 %."""
import numpy as np
import pytest

from oracle import sketchnet as N

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


def _problem(ksize, n, seed):
    rng = np.random.default_rng(seed)
    chan = [2, 7, 3]
    params = [(rng.standard_normal((o, c, ksize)) / np.sqrt(c * ksize), 0.1 * rng.standard_normal(o))
              for c, o in zip(chan, chan[1:])]
    params[0][0][:, 1, :] = 0.0
    flat = N.flatten(params).astype(np.float32)
    x0 = np.tile(rng.standard_normal(32), n // 32).astype(np.float32)
    U = np.tile(np.linalg.qr(rng.standard_normal((32, 2)))[0], (n // 32, 1)) / np.sqrt(n / 32)
    return flat, N.unflatten(flat.astype(np.float64), [W.shape for W, _ in params]), x0, U.T.astype(np.float32)


def _g1(params, x0, x1, U, mu):
    """The oracle's gradient of the second channel's weights."""
    x = np.stack([x0, x1]).astype(np.float64)
    return N.batch_loss_grad(params, [x], [U.T.astype(np.float64)], mu)[1][0][0][:, 1, :]


@pytest.mark.parametrize("ksize", [1, 3, 5, 7])
@pytest.mark.parametrize("kind", ["cancel", "overflow", "underflow"])
def test_gradient_sums(gpu_lib, kind, ksize):
    R = gpu_lib
    n = 4096
    flat, params, x0, U = _problem(ksize, n, 10 * ksize)
    a, block = np.tile(np.random.default_rng(3).uniform(0.5, 1.0, 32), n // 32), np.arange(n) // 32
    e = np.zeros((32, n))
    mu = 0.2
    e[0, n // 2] = 1.0
    g = np.abs(_g1(params, x0, e[0], U, mu)).max()   # size of g: the gradient for x1 = 1 at one position
    if kind == "cancel":      # neighbouring terms of a lane, 32 positions apart
        x1 = np.where(block % 2 == 0, a.astype(np.float32), -a.astype(np.float32) * np.float32(1.0 - 2.0 ** -21))
    elif kind == "overflow":  # two halves that cancel to 2^-20
        mu *= 100.0 / g
        x1 = 1e38 * np.where(block < n // 64, a, -a * (1.0 - 2.0 ** -20))
    else:
        x1 = a * (30.0 * 2.0 ** -149 / g)
    x1 = x1.astype(np.float32)
    want = _g1(params, x0, x1, U, mu)
    assert np.all(np.isfinite(want.astype(np.float32)))
    net = R.riot_sketchnet_create(2, 7, 3, depth=2, ksize=ksize, n_max=n, batch_max=1, r_max=2)
    R.riot_sketchnet_set_params(net, torch.tensor(flat, device=DEV))
    grad = torch.empty(flat.size, dtype=torch.float32, device=DEV)
    R.riot_sketchnet_loss_grad(net, torch.tensor(np.stack([x0, x1])[None], device=DEV),
                               torch.tensor(U[None], device=DEV).contiguous(), mu, grad)
    R.riot_sketchnet_destroy(net)
    got = grad[:7 * 2 * ksize].view(7, 2, ksize)[:, 1].double().cpu().numpy()
    print(kind, ksize, g, np.linalg.norm(want), np.linalg.norm(got - want) / np.linalg.norm(want))
    assert np.linalg.norm(got / np.abs(want).max() - want / np.abs(want).max()) <= 1e-3 * np.linalg.norm(want / np.abs(want).max())
