"""The double-precision transforms hold each sequence on a block exponent of its
own (fft64.cuh): a component far below the others keeps the accuracy of its own
norm where the operator does not couple it to them.  Fields that vary along x1
only decouple (k2 = 0): Eqs. 2-3 give

    e11 = -(p11 - <p11>) / (lambda0 + 2 mu0),  e12 = -(p12 - <p12>) / (2 mu0),  e22 = 0,

and u2 of the displacement is the sum of 2 (eps12 - <eps12>) along x1.  (Fields
along x2 do not: the m1 = 0 and m1 = L/2 columns share a sequence, and the
rounding of one couples the components through the other.)

Tolerance: that of test_gpu_fixed_point.py, 4 u log2(L^2) of the component's own
2-norm (u = 2^-53)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LAM, MU = 1.5, 1.0


def _tol(L):
    return 4 * 2.0 ** -53 * 2 * np.log2(L)


def _rel(got, ref):
    s = np.abs(ref).max()
    return float(np.linalg.norm((got - ref) / s) / np.linalg.norm(ref / s))


def _line(rng, L, scale):
    """(L, L) array that varies along x1 ([x2][x1]), and its deviation from the mean."""
    v = scale * rng.standard_normal(L)
    v64 = v.astype(np.longdouble)
    d = (v64 - v64.mean()).astype(np.float64)
    return np.tile(v, (L, 1)), np.tile(d, (L, 1))


@pytest.mark.parametrize("tiling", [0, 1])
@pytest.mark.parametrize("L", [4, 8, 16, 32, 64, 128, 256, 512, 1024, 2048, 4096])
def test_small_component_of_a_projection(L, tiling):
    import torch
    from paper_0802_2488_gb300 import binding as B
    rng = np.random.default_rng(L)
    with B.Context(0) as ctx:
        B.epfft_set_tiling(ctx, L, "fp64", tiling)
        for small in (1e-10, 1e-60):
            p11, d11 = _line(rng, L, 1.0)
            p22, _ = _line(rng, L, 1e3)
            p12, d12 = _line(rng, L, small)
            p = torch.tensor(np.stack([p11, p22, p12]), device="cuda")
            e = B.epfft_project(ctx, L, "fp64", LAM, MU, [0.0] * 4, p).cpu().numpy()
            assert _rel(e[2], -d12 / (2 * MU)) < _tol(L), small
            assert _rel(e[0], -d11 / (LAM + 2 * MU)) < _tol(L), small


@pytest.mark.parametrize("L", [16, 256, 1024])
def test_displacement_of_a_small_shear(L):
    import torch
    from paper_0802_2488_gb300 import binding as B
    rng = np.random.default_rng(L)
    eps = np.zeros((L, L, 4))
    eps[..., 0], eps[..., 3] = _line(rng, L, 1.0)[0], _line(rng, L, 1e-12)[0]
    v = eps[0, :, 3].astype(np.longdouble)
    u = np.concatenate([[0.0], np.cumsum(2 * (v - v.mean()))[:-1]])
    ref = np.tile((u - u.mean()).astype(np.float64), (L, 1))
    with B.Context(0) as ctx:
        got = B.epfft_displacement(ctx, L, "fp64", torch.tensor(eps, device="cuda")).cpu().numpy()
    assert _rel(got[..., 1], ref) < _tol(L)


@pytest.mark.parametrize("L", [16, 64, 256])
def test_small_mean_shear_of_a_homogeneous_lattice(L):
    """Without voids the strain is the mean strain, component by component."""
    from paper_0802_2488_gb300 import binding as B
    E = np.array([[0.1, 0.05, 0.0, 1e-12]])
    with B.Context(0) as ctx:
        _, rec, f = B.epfft_solve(ctx, B.Problem(L=L, precision="fp64", max_iter=30), E, fields=True)
    for c in (0, 1, 3):
        assert np.abs(f.eps[..., c] / E[0, c] - 1).max() < _tol(L), c
    assert abs(rec["sig_mean"][0][3] / (2 * E[0, 3]) - 1) < _tol(L)
