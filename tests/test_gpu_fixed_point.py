"""The double-precision transforms run in 64-bit fixed point on a block
exponent (fft64.cuh): the projection of Eqs. 2-3 at the edges of their range,
against the same projection with torch's FP64 transforms on the GPU.

Tolerance: each side's rounding error grows like u sqrt(log2 N) per transform
(u = 2^-53); 4 u log2(L^2) of the result's 2-norm leaves a factor of a few
over both.  Inputs whose transform is far from white (a single pixel, a large
mean) and extreme scales are what a fixed-point transform can lose."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LAM, MU = 1.5, 1.0


def _reference(p, L):
    import torch
    q = 2.0 * np.pi * torch.arange(L, device=p.device, dtype=torch.float64) / L
    k = torch.complex(torch.sin(q), 2.0 * torch.sin(0.5 * q) ** 2)
    k1, k2 = k[None, :L // 2 + 1], k[:, None]
    a1, a2 = k1.abs() ** 2, k2.abs() ** 2
    n11, n22 = LAM * a1 + MU * (a1 + a2) + MU * a1, LAM * a2 + MU * (a1 + a2) + MU * a2
    n12 = LAM * k1.conj() * k2 + MU * k1 * k2.conj()
    det = n11 * n22 - n12.abs() ** 2
    det[0, 0] = 1.0
    c11, c22, c12 = torch.fft.rfft2(p)
    w1, w2 = k1.conj() * c11 + k2.conj() * c12, k1.conj() * c12 + k2.conj() * c22
    v1, v2 = (n22 * w1 - n12 * w2) / det, (n11 * w2 - n12.conj() * w1) / det
    e = torch.stack([-(k1 * v1), -(k2 * v2), -0.5 * (k1 * v2 + k2 * v1)])
    e[:, 0, 0] = 0.0
    return torch.fft.irfft2(e, s=(L, L))


@pytest.mark.parametrize("tiling", [0, 1])
@pytest.mark.parametrize("L", [4, 8, 16, 32, 128, 256, 512, 1024, 2048, 4096])
def test_projection_fp64(L, tiling):
    import torch
    from paper_0802_2488_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(L + tiling)
    white = torch.randn((3, L, L), generator=g, device="cuda", dtype=torch.float64)
    pixel = torch.zeros_like(white)
    pixel[:, L // 3, L // 2 + 1] = torch.tensor([1.0, -2.0, 0.5], device="cuda", dtype=torch.float64)
    with B.Context(0) as ctx:
        B.epfft_set_tiling(ctx, L, "fp64", tiling)
        for p in (white, 1e140 * white, 1e-140 * white, pixel):
            got = B.epfft_project(ctx, L, "fp64", LAM, MU, [0.0, 0.0, 0.0, 0.0], p)
            ref = _reference(p, L)
            # norms of scaled copies: squares of 1e140 stay below the range's end
            s = ref.abs().max()
            err = float(torch.linalg.norm((got - ref) / s) / torch.linalg.norm(ref / s))
            assert err < 4 * 2.0 ** -53 * 2 * np.log2(L), err
        # a large mean: projected out, its rounding stays relative to it
        got = B.epfft_project(ctx, L, "fp64", LAM, MU, [0.0, 0.0, 0.0, 0.0], white + 1e3)
        err = float(torch.linalg.norm(got - _reference(white, L)) / torch.linalg.norm(white + 1e3))
        assert err < 4 * 2.0 ** -53 * 2 * np.log2(L), err
        # zero stays zero; a NaN or an infinity reaches every output
        assert float(B.epfft_project(ctx, L, "fp64", LAM, MU, [0.0] * 4, torch.zeros_like(white)).abs().max()) == 0.0
        for bad in (float("nan"), float("inf")):
            p = white.clone()
            p[0, 1, 2] = bad
            assert not bool(torch.isfinite(B.epfft_project(ctx, L, "fp64", LAM, MU, [0.0] * 4, p)).any())
