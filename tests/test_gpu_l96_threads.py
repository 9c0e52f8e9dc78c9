"""Two host threads with contexts of different sizes: the square root of B of one asks for nine times the
shared memory that the other's does, and neither call disturbs the other's launch."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


def test_contexts_of_two_sizes_side_by_side(gpu_lib):
    R = gpu_lib
    bad, start = [], threading.Barrier(2, timeout=60)

    def work(n, length):
        try:
            stream = torch.cuda.Stream(DEV)
            ctx = R.Context(n=n, T=0, dt=0.01, F=8.0, obs_step=np.zeros(n // 2, int), obs_idx=np.arange(n // 2),
                            obs_y=np.zeros(n // 2), obs_sigma=np.ones(n // 2), length=length, precision=R.RIOT_PREC_FP64,
                            kmax=2, stream=stream)
            with torch.cuda.stream(stream):
                R.riot_outer_begin(ctx.h, torch.ones(n, dtype=torch.float64, device=DEV))
                W = torch.randn(1, n, dtype=torch.float64, device=DEV)
                Y, first = torch.empty_like(W), torch.empty_like(W)
                R.riot_hessian_apply(ctx.h, W, first)
                start.wait()
                for _ in range(30000):
                    R.riot_hessian_apply(ctx.h, W, Y)
                assert torch.equal(Y, first)
            ctx.close()
        except Exception as e:
            bad.append(repr(e))

    threads = [threading.Thread(target=work, args=a) for a in ((700, 300.0), (16, 0.5))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
