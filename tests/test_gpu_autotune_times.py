"""epfft_autotune times the tilings of a small lattice alike, as whole solves by
the schedule each takes: a time per iteration that of a long solve plus the warm
start, the last evaluation and the final pass of its 30 iterations (at most three
more: 10 %) and the launch."""
import time

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [16, 64, 128, 256])
def test_times_are_those_of_whole_solves(L):
    import torch
    from paper_0802_2488_gb300 import binding as B
    E = [[0.0, 0.0, 0.0, 1.5 / (2 * 3 ** 0.5)]]  # the autotuner's lattice and load
    with B.Context(0) as ctx:
        chosen, ms = B.epfft_autotune(ctx, L, "fp32", 1)
        true = {}
        for v in range(4):
            if not B.epfft_supported_tiling(L, "fp32", v):
                continue
            B.epfft_set_tiling(ctx, L, "fp32", v)
            best = []
            for n in (200, 1000):
                p = B.Problem(L=L, precision="fp32", void_fraction=0.2, seed=7, max_iter=n, tol_eq=0.0, tol_macro=0.0)
                B.epfft_solve(ctx, p, E)
                t = []
                for _ in range(5):
                    torch.cuda.synchronize()
                    t0 = time.perf_counter()
                    B.epfft_solve(ctx, p, E)
                    t.append(time.perf_counter() - t0)
                best.append(min(t))
            true[v] = (best[1] - best[0]) / 800 * 1e3
        for v, t in true.items():
            assert 0.9 < ms[v] / t < 1.3, (v, ms[v], t)
        assert true[chosen] < 1.1 * min(true.values())
