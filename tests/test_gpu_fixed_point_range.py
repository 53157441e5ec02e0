"""The double-precision projection scales exactly by powers of two over the whole
normal range, as FP64 arithmetic does: the transforms' block exponents
(fft64.cuh) reach down to 2^-1022 as well as up."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiling", [0, 1])
@pytest.mark.parametrize("L", [4, 16, 64, 256, 512, 1024, 2048, 4096])
def test_projection_scales_exactly(L, tiling):
    import torch
    from paper_0802_2488_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(L)
    p = torch.randn((3, L, L), generator=g, device="cuda", dtype=torch.float64)
    E = np.array([0.3, -0.2, 0.0, 0.1])
    with B.Context(0) as ctx:
        B.epfft_set_tiling(ctx, L, "fp64", tiling)
        ref = B.epfft_project(ctx, L, "fp64", 1.5, 1.0, E, p)
        for k in (-985, -960, -300, 900):
            s = 2.0 ** k
            got = B.epfft_project(ctx, L, "fp64", 1.5, 1.0, E * s, p * s)
            # numbers whose scaled value leaves the normal range may round
            err = ((got / s - ref).abs() * (ref.abs() * s > 2.0 ** -1000)).max()
            assert float(err) == 0.0, k
