"""Contexts of different sizes side by side, in two host threads or in two batches: a kernel's limit of shared
memory belongs to the process, and the small one's calls leave the large one's launches alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("precision", ["RIOT_PREC_FP64", "RIOT_PREC_MIXED"])
def test_contexts_of_two_sizes_side_by_side(gpu_lib, precision):
    R = gpu_lib
    real = torch.float64 if precision == "RIOT_PREC_FP64" else torch.float32
    bad, start = [], threading.Barrier(2, timeout=60)

    def work(n, length):
        try:
            stream = torch.cuda.Stream(DEV)
            ctx = R.Context(n=n, T=0, dt=0.01, F=8.0, obs_step=np.zeros(n // 2, int), obs_idx=np.arange(n // 2),
                            obs_y=np.zeros(n // 2), obs_sigma=np.ones(n // 2), length=length, precision=getattr(R, precision),
                            kmax=2, stream=stream)
            with torch.cuda.stream(stream):
                R.riot_outer_begin(ctx.h, torch.ones(n, dtype=torch.float64, device=DEV))
                W = torch.randn(1, n, dtype=real, device=DEV)
                Y, first = torch.empty_like(W), torch.empty_like(W)
                R.riot_hessian_apply(ctx.h, W, first)
                start.wait()
                for _ in range(30000):
                    R.riot_hessian_apply(ctx.h, W, Y)
                assert torch.equal(Y, first)
            ctx.close()
        except Exception as e:
            start.abort()
            bad.append(repr(e))

    threads = [threading.Thread(target=work, args=a) for a in ((700, 300.0), (16, 0.5))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_batches_of_two_sizes(gpu_lib):
    """The second batch's plan asks for less shared memory than the first's, which runs afterwards."""
    R = gpu_lib
    ctxs, batches = [], []
    for n, k in ((8192, 16), (40, 8)):
        ctx = R.Context(n=n, T=2, dt=0.01, F=8.0, obs_step=np.full(n // 2, 1), obs_idx=np.arange(n // 2),
                        obs_y=np.zeros(n // 2), obs_sigma=np.ones(n // 2), length=1.0, kmax=k)
        R.riot_outer_begin(ctx.h, 8.0 + torch.sin(torch.arange(n, dtype=torch.float64, device=DEV)))
        ctxs.append(ctx)
        batches.append(R.riot_batch_create([ctx.h], [k], 0))
    for b in batches:
        assert R.riot_batch_run(b, 1, sketch_stream=3) == [0]
        R.riot_batch_destroy(b)
    for ctx in ctxs:
        ctx.close()
