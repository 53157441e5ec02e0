"""Loop graphs kept from call to call (over the context's own records, at most eight)
give the bytes of a fresh context: other shapes on the same records in between,
other operators, tilings, materials, tolerances, load paths and refresh
intervals of the same shape, shapes put out by newer ones, and a batch too large
for the records."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (L, precision, tiling, solves, operator): shapes the resident schedule declines
SHAPES = [(256, "fp64", 0, 1, "eq3"), (256, "fp64", 1, 1, "eq3"), (256, "fp64", 0, 2, "dg1"), (256, "fp64", 0, 1, "dg1"),
          (128, "fp32", 0, 1, "eq3"), (128, "fp32", 0, 3, "eq3"), (64, "fp32_defect", 0, 1, "eq3"),
          (64, "fp32_defect", 0, 2, "eq3"), (64, "fp32_defect", 1, 1, "eq3"), (8, "fp32", 0, 100, "eq3"),
          (8, "fp32", 0, 130, "eq3")]


def _solve(ctx, shape, k):
    """Call k of a shape: its materials, tolerances, path and refresh interval differ."""
    from paper_0802_2488_gb300 import binding as B
    from paper_0802_2488_gb300 import inputs
    L, prec, tiling, n, green = shape
    B.epfft_set_tiling(ctx, L, prec, tiling)
    B.epfft_set_defect_refresh(ctx, 3 + 4 * k)
    probs = [B.Problem(L=L, precision=prec, void_fraction=0.1 + 0.05 * k, seed=10 * k + i, mu=1.0 + 0.2 * k,
                       yield_stress=1.0 - 0.1 * k, tol_eq=10.0 ** -(2 + k), tol_macro=1e-2, max_iter=12 + i % 3,
                       green=green) for i in range(n)]
    paths = [inputs.load_path("shear" if k else "equibiaxial", 1 + k, 3.0)] * n
    rc, recs, fs = B.epfft_solve_batch(ctx, probs, paths, fields=True)
    return [rc] + [r.tobytes() for r in recs] + [f.eps.tobytes() + f.plastic.tobytes() + f.labels.tobytes() for f in fs]


def test_kept_graphs_equal_fresh_contexts():
    from paper_0802_2488_gb300 import binding as B
    ref = {}
    for s in SHAPES:
        for k in range(3):
            with B.Context(0) as ctx:
                ref[s, k] = _solve(ctx, s, k)
    rng = np.random.default_rng(0)
    with B.Context(0) as ctx:
        # every shape in turn (eleven: the first ones are put out), then in any order
        order = [(s, 0) for s in SHAPES] + [(s, 1) for s in SHAPES[:4]] + [(s, 2) for s in SHAPES[:4]]
        order += [(SHAPES[i], int(k)) for i, k in zip(rng.integers(0, len(SHAPES), 60), rng.integers(0, 3, 60))]
        for s, k in order:
            assert _solve(ctx, s, k) == ref[s, k], (s, k)
