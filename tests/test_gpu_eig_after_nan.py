"""The inverse iteration reads nothing that it has not written: an eigenproblem solved after one
whose kernels left NaN in shared memory gives the eigenvalues of a plain solve.  The bound is the
FP64 eigensolvers' usual one, 1e-13 of the norm times the order's square root."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("k,k_nan", [(37, 64), (128, 300), (128, 128), (201, 512)])
def test_eigenproblem_after_nan(gpu_lib, k, k_nan):
    R = gpu_lib
    K = np.random.default_rng(k).standard_normal((k, 2 * k))
    K = K @ K.T
    want = np.linalg.eigvalsh(K)[::-1]
    good = torch.tensor(K, device=DEV)
    bad = torch.full((k_nan, k_nan), float("nan"), dtype=torch.float64, device=DEV)
    for _ in range(20):
        with pytest.raises(RuntimeError):
            R.riot_symm_eig(bad, bad.new_empty(k_nan), torch.empty_like(bad))
        lam, Z = good.new_empty(k), torch.empty_like(good)
        R.riot_symm_eig(good, lam, Z)
        np.testing.assert_allclose(lam.cpu().numpy(), want, rtol=0, atol=1e-13 * np.sqrt(k) * want[0])
