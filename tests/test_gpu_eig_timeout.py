"""A wait at the eigensolver's barrier that runs out is reported by the call that met it, before it
changes the state, and the context goes on: RIOT-PSAS, block Lanczos and the FP64 inner loop."""
import numpy as np
import pytest

from oracle import l96

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("precision", ["RIOT_PREC_FP64", "RIOT_PREC_MIXED"])
@pytest.mark.parametrize("call", ["psas", "varbl", "varcg", "rsvd"])
def test_eigensolver_wait_that_runs_out(gpu_lib, precision, call):
    R = gpu_lib
    n, T, m = 200, 5, 64
    rng = np.random.default_rng(9)
    x0 = l96.nl(8.0 + rng.standard_normal(n), 100, 0.05, 8.0)[-1]
    ix = np.arange(0, n, 2)
    st, ix = np.repeat([2, T], ix.size), np.tile(ix, 2)
    ctx = R.Context(n=n, T=T, dt=0.02, F=8.0, obs_step=st, obs_idx=ix, obs_y=8.0 + rng.standard_normal(st.size),
                    obs_sigma=np.ones(st.size), length=2.0, precision=getattr(R, precision), kmax=2 * m)
    B0 = torch.tensor(rng.standard_normal((2, n)), device=DEV)
    run = {"psas": lambda: R.riot_psas(ctx.h, m, 0, sketch_stream=5), "varbl": lambda: R.riot_varbl(ctx.h, 2, m // 2, B0),
           "varcg": lambda: R.riot_varcg(ctx.h, m), "rsvd": lambda: R.riot_rsvd(ctx.h, m, 0, sketch_stream=5)}[call]
    x, v, x1, v1 = (torch.empty(n, dtype=torch.float64, device=DEV) for _ in range(4))
    R.riot_outer_begin(ctx.h, torch.tensor(x0, device=DEV))
    R.riot_get_state(ctx.h, x=x, v=v)
    R.riot_set_wait_limit(ctx.h, 0)
    with pytest.raises(R.RiotError) as e:
        run()
    assert e.value.status == -5 and "bounded device wait" in str(e.value)
    R.riot_get_state(ctx.h, x=x1, v=v1)
    assert torch.equal(x, x1) and torch.equal(v, v1)
    R.riot_set_wait_limit(ctx.h, -1)
    got = run()[0] if call != "rsvd" else run()
    ctx.close()
    # the same call on a context whose waits never ran out
    ctx = R.Context(n=n, T=T, dt=0.02, F=8.0, obs_step=st, obs_idx=ix, obs_y=np.zeros(st.size), obs_sigma=np.ones(st.size),
                    length=2.0, precision=getattr(R, precision), kmax=2 * m)
    R.riot_outer_begin(ctx.h, torch.tensor(x0, device=DEV))
    if call != "varcg":   # whose Krylov space starts at the gradient, another one here
        want = run()[0] if call != "rsvd" else run()
        np.testing.assert_allclose(got, want, rtol=0, atol=1e-9 * np.abs(want).max())
    assert np.all(np.isfinite(got))
    ctx.close()
