"""The problem is homogeneous of degree one in strain and flow stress: with both
times 2^k every number of a double-precision solve is 2^k times the other's,
exactly, also where squared strains and stresses leave the FP32 range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [-400, -70, -63, 64, 70, 400])
@pytest.mark.parametrize("L", [16, 64, 256])
def test_solve_scales_exactly_with_the_units(L, k):
    from paper_0802_2488_gb300 import binding as B
    from paper_0802_2488_gb300 import inputs
    s = 2.0 ** k
    path = inputs.load_path("shear", 3, 3.0)
    with B.Context(0) as ctx:
        def solve(u):
            prob = B.Problem(L=L, precision="fp64", void_fraction=0.15, seed=2, yield_stress=u, max_iter=25,
                             tol_eq=1e-6, tol_macro=1e-6)
            return B.epfft_solve(ctx, prob, path * u, fields=True)
        rc0, r0, f0 = solve(1.0)
        rc1, r1, f1 = solve(s)
    assert rc0 == rc1 and f0.plastic[-1].any()
    for key in ("iterations", "n_plastic", "n_clusters", "status", "eta1", "eta2", "eta3"):
        assert np.array_equal(r0[key], r1[key]), key
    assert np.array_equal(r0["sig_mean"] * s, r1["sig_mean"])
    assert np.array_equal(r0["eps_mean"] * s, r1["eps_mean"])
    assert np.array_equal(f0.eps * s, f1.eps) and np.array_equal(f0.plastic, f1.plastic)
