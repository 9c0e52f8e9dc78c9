"""Eigensolvers of a batch run side by side in one cooperative launch; each must give what the
window gives alone, also when the batch mixes the smallest problems (no reflector, one column),
sizes around a multiple of four columns, more problems than one launch takes, and windows of the
Jacobi option.  Tolerance 1e-12, as for batches: the arithmetic of a problem does not depend on its
CTAs, the Cholesky forms of a batch differ in rounding only."""
import numpy as np
import pytest

from oracle import l96

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("ks", [[1, 2, 3, 4, 5], [64, 7, 129, 128, 33], list(range(4, 60))])
def test_batched_eigensolvers_equal_those_alone(gpu_lib, ks):
    R = gpu_lib

    def contexts():
        out = []
        for i, k in enumerate(ks):
            n = max(40, 2 * k)
            rng = np.random.default_rng(k)
            x = l96.nl(8.0 + rng.standard_normal(n), 40, 0.05, 8.0)[-1]
            st, ix = np.repeat([2, 4], n // 2), np.tile(np.arange(0, 2 * (n // 2), 2), 2)
            c = R.Context(n=n, T=4, dt=0.02, F=8.0, obs_step=st, obs_idx=ix, obs_y=np.zeros(st.size),
                          obs_sigma=np.ones(st.size), length=2.0, kmax=k, seed=i,
                          eig_method=R.RIOT_EIG_JACOBI if k == 33 else R.RIOT_EIG_TRIDIAG)
            R.riot_outer_begin(c.h, torch.tensor(x, device=DEV))
            out.append(c)
        return out

    def state(c, k):
        lam = torch.empty(k, dtype=torch.float64, device=DEV)
        U = torch.empty(k, c.n, dtype=torch.float64, device=DEV)
        x = torch.empty(c.n, dtype=torch.float64, device=DEV)
        R.riot_get_state(c.h, x=x, U=U, lam=lam)
        return lam, U, x

    alone = contexts()
    for c, k in zip(alone, ks):
        R.riot_rsvd(c.h, k, 1, sketch_stream=16)
        R.riot_increment(c.h)
    both = contexts()
    b = R.riot_batch_create([c.h for c in both], ks, 1)
    R.riot_batch_run(b, len(ks), sketch_stream=16)
    for c, a, k in zip(both, alone, ks):
        for got, want in zip(state(c, k), state(a, k)):
            np.testing.assert_allclose(got.cpu().numpy(), want.cpu().numpy(), rtol=0, atol=1e-12 * float(want.abs().max()))
    R.riot_batch_destroy(b)
