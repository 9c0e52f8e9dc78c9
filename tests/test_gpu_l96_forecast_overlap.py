"""A stored forecast may start from any place of its own trajectory buffer (a run continued from its
last state): the rows are those of a start elsewhere, to the FP64 bound of the other forecasts."""
import numpy as np
import pytest

from oracle import l96

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("n,T,at", [(100, 5, 5.0), (700, 3, 3.0), (700, 9, 1.0), (700, 9, 9.0), (700, 9, 0.0),
                                    (700, 9, 0.37), (4096, 5, 2.0), (4096, 60, 60.0), (8192, 4, 3.5), (700, 0, 0.0),
                                    (700, 0, 0.5)])
def test_start_inside_the_trajectory(gpu_lib, n, T, at):
    R = gpu_lib
    x0 = 8.0 + np.random.default_rng(n).standard_normal(n)
    ref = l96.nl(x0, T, 0.01, 8.0)
    for _ in range(10):
        buf = torch.zeros((T + 2) * n, dtype=torch.float64, device=DEV)   # one row more than the trajectory
        start = buf[int(at * n):int(at * n) + n]
        start.copy_(torch.tensor(x0))
        R.riot_l96_forecast(n, T, 0.01, 8.0, start, buf)
        got = buf.view(T + 2, n)[:T + 1].cpu().numpy()
        np.testing.assert_allclose(got, ref, rtol=0, atol=1e-11 * np.abs(ref).max())
