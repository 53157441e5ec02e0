"""n_plastic of a record is the number of plastic flags of that increment: both
come from the test of the accepted strain.  A lattice without voids loaded
exactly to first yield holds every pixel at the threshold to rounding, where
two different tests would part."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _yield_path(rng, mu, Y):
    """Half the yield strain, then yield twice: E scaled to 2 mu |dev E| = sqrt(2/3) Y."""
    E = rng.uniform(-1.0, 1.0, 4)
    d = E[:3] - E[:3].mean()
    E *= np.sqrt(2.0 / 3.0) * Y / (2.0 * mu * np.sqrt((d ** 2).sum() + 2.0 * E[3] ** 2))
    return np.stack([0.5 * E, E, E])


@pytest.mark.parametrize("schedule", ["device", "host"])
@pytest.mark.parametrize("L,n", [(16, 60), (64, 20), (256, 10)])
def test_count_equals_the_flags_at_first_yield(L, n, schedule, monkeypatch):
    from paper_0802_2488_gb300 import binding as B
    if schedule == "host":
        monkeypatch.setenv("EPFFT_SYNC_CHECK", "1")
    rng = np.random.default_rng(L)
    with B.Context(0) as ctx:
        for i in range(n):
            mu, lam, Y = rng.uniform(0.5, 2.0, 3)
            prob = B.Problem(L=L, precision="fp64", mu=mu, lambda_=lam, yield_stress=Y, max_iter=20,
                             tol_eq=1e-8, tol_macro=1e-8)
            _, rec, f = B.epfft_solve(ctx, prob, _yield_path(rng, mu, Y), fields=True)
            assert [int(x) for x in rec["n_plastic"]] == [int(p.sum()) for p in f.plastic], i


@pytest.mark.parametrize("L", [32, 128, 512])
def test_count_equals_the_flags_of_a_porous_lattice(L):
    from paper_0802_2488_gb300 import binding as B
    from paper_0802_2488_gb300 import inputs
    with B.Context(0) as ctx:
        probs = [B.Problem(L=L, precision="fp64", void_fraction=0.15, seed=s, max_iter=40) for s in range(2)]
        _, recs, fs = B.epfft_solve_batch(ctx, probs, [inputs.load_path("shear", 4, 3.0)] * 2, fields=True)
        for rec, f in zip(recs, fs):
            assert [int(x) for x in rec["n_plastic"]] == [int(p.sum()) for p in f.plastic]
            assert rec["n_plastic"][-1] > 0


@pytest.mark.parametrize("big", [1e3, 1e6, 1e12, 1e16])
def test_count_equals_the_flags_under_a_large_mean_strain(big):
    """A mean strain far above the yield deviator leaves the stored deviator few
    exact bits: the branch taken and the flags' test part at any distance."""
    from paper_0802_2488_gb300 import binding as B
    rng = np.random.default_rng(3)
    with B.Context(0) as ctx:
        for i in range(30):
            mu, lam, Y = rng.uniform(0.5, 2.0, 3)
            E = _yield_path(rng, mu, Y) * rng.uniform(0.5, 1.5)
            E[:, :3] += big * Y
            prob = B.Problem(L=16, precision="fp64", mu=mu, lambda_=lam, yield_stress=Y, max_iter=20)
            _, rec, f = B.epfft_solve(ctx, prob, E, fields=True)
            assert [int(x) for x in rec["n_plastic"]] == [int(p.sum()) for p in f.plastic], i
