"""The workspace that spreads FP64 integrations over the GPU never takes memory that something else of
the context needs: a budget that the rest fits is enough for riot_setup and for RIOT-PSAS's blocks, and
results are those of a context with the workspace (one CTA a column then, another order of the FP64
sums: 1e-10 of the norm, as against the oracle)."""
import numpy as np
import pytest

from oracle import l96

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


class Budget:
    """An allocator of the library's that refuses what goes beyond a number of bytes."""

    def __init__(self, R, limit):
        self.left, self.sizes, self.live = limit, [], {}
        self.alloc, self.free = R.DEV_ALLOC_FN(self._alloc), R.DEV_FREE_FN(self._free)

    def _alloc(self, nbytes, stream, user):
        self.sizes.append(nbytes)
        if nbytes > self.left:
            return None
        t = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
        self.left -= nbytes
        self.live[t.data_ptr()] = t
        return t.data_ptr()

    def _free(self, ptr, nbytes, stream, user):
        self.left += self.live.pop(ptr).numel()


def _run(R, monkeypatch, precision, limit):
    n, T, m = 520, 12, 40
    rng = np.random.default_rng(5)
    st, ix = np.repeat(np.arange(1, T + 1), 60), np.tile(np.sort(rng.choice(n, 60, replace=False)), T)
    x0 = l96.nl(8.0 + rng.standard_normal(n), 60, 0.05, 8.0)[-1]
    y = 8.0 + 3.0 * rng.standard_normal(st.size)
    b = Budget(R, limit)
    monkeypatch.setattr(R, "TORCH_ALLOC", b.alloc)
    monkeypatch.setattr(R, "TORCH_FREE", b.free)
    ctx = R.Context(n=n, T=T, dt=0.02, F=8.0, obs_step=st, obs_idx=ix, obs_y=y, obs_sigma=np.ones(st.size), length=2.0,
                    precision=precision, kmax=m)
    setup = list(b.sizes)
    f64 = dict(dtype=torch.float64, device=DEV)
    g, x = torch.empty(n, **f64), torch.empty(n, **f64)
    out = [np.array([R.riot_outer_begin(ctx.h, torch.tensor(x0, device=DEV))])]
    R.riot_get_state(ctx.h, g=g)
    out += [g.cpu().numpy(), np.array([R.riot_quadratic_cost(ctx.h, torch.tensor(0.1 * x0, device=DEV))])]
    R.riot_psas(ctx.h, m, 0, sketch_stream=3)
    R.riot_get_state(ctx.h, x=x)
    out.append(x.cpu().numpy())
    out.append(np.array([R.riot_outer_begin(ctx.h)]))   # after the workspace may have gone
    peak = list(b.sizes)
    ctx.close()
    assert not b.live
    return out, setup, peak


@pytest.mark.parametrize("precision", ["RIOT_PREC_FP64", "RIOT_PREC_MIXED"])
def test_a_budget_without_the_optional_workspace(gpu_lib, monkeypatch, precision):
    R = gpu_lib
    prec = getattr(R, precision)
    want, setup, peak = _run(R, monkeypatch, prec, 1 << 40)
    optional = setup[-1]   # the last request of the setup
    assert optional > max(setup[-5:-1])
    for limit in (sum(peak) - optional,        # refused at the setup, or given back to RIOT-PSAS's blocks
                  sum(peak) - optional // 2):
        got, again, _ = _run(R, monkeypatch, prec, limit)
        assert again == setup
        for a, w in zip(got, want):
            assert np.linalg.norm(a - w) <= 1e-10 * np.linalg.norm(w)
    # exactly what the setup needs without it
    with pytest.raises(R.RiotError) as e:
        _run(R, monkeypatch, prec, sum(setup) - optional)
    assert e.value.status == -2 and "riot_psas" in str(e.value)
