"""Eigenproblems of order 1 to 4, whose workspace pieces lie closest together, against LAPACK, and a
batch of windows with one sketch vector against the window alone (1e-12, as for batches).  The bound is the FP64 eigensolvers' usual one, 1e-13 of the norm times the order's square root."""
import numpy as np
import pytest

from oracle import l96

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("k", [1, 2, 3, 4])
def test_tiny_eigenproblems(gpu_lib, k):
    R = gpu_lib
    for seed in range(20):
        K = np.random.default_rng(seed).standard_normal((k, 2 * k))
        K = K @ K.T
        want = np.linalg.eigvalsh(K)[::-1]
        good = torch.tensor(K, device=DEV)
        lam, Z = good.new_empty(k), torch.empty_like(good)
        R.riot_symm_eig(good, lam, Z)
        np.testing.assert_allclose(lam.cpu().numpy(), want, rtol=0, atol=1e-13 * np.sqrt(k) * want[0])
        U = Z.cpu().numpy()   # rows are the eigenvectors
        np.testing.assert_allclose((U * want[:, None]).T @ U, K, rtol=0, atol=1e-12 * np.sqrt(k) * want[0])


def test_batch_with_one_sketch_vector(gpu_lib):
    R = gpu_lib

    def context(seed):
        x = l96.nl(8.0 + np.random.default_rng(seed).standard_normal(40), 40, 0.05, 8.0)[-1]
        st, ix = np.repeat([2, 4], 20), np.tile(np.arange(0, 40, 2), 2)
        c = R.Context(n=40, T=4, dt=0.02, F=8.0, obs_step=st, obs_idx=ix, obs_y=np.zeros(40),
                      obs_sigma=np.ones(40), length=2.0, kmax=4, seed=seed)
        R.riot_outer_begin(c.h, torch.tensor(x, device=DEV))
        return c

    def state(c):
        x = torch.empty(40, dtype=torch.float64, device=DEV)
        R.riot_get_state(c.h, x=x)
        return x.cpu().numpy()

    alone, both = [context(i) for i in range(2)], [context(i) for i in range(2)]
    for c in alone:
        R.riot_rsvd(c.h, 1, 1, sketch_stream=16)
        R.riot_increment(c.h)
    b = R.riot_batch_create([c.h for c in both], [1, 1], 1)
    R.riot_batch_run(b, 2, sketch_stream=16)
    for c, a in zip(both, alone):
        np.testing.assert_allclose(state(c), state(a), rtol=0, atol=1e-12 * np.abs(state(a)).max())
    R.riot_batch_destroy(b)
