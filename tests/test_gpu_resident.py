"""The resident schedule (one cooperative launch runs whole solves of small
and medium lattices): the same bits as the two passes launched one by one, for
every side and tiling it is built for, alone, in a batch, with the general
Green operator, and in a call mixed with another size (which runs the two-pass
loop)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = ([("fp64", L, v) for v in (0, 1) for L in (8, 16, 32, 64, 128)] +
         [("fp32", L, 0) for L in (32, 64)] + [("fp32", L, 1) for L in (8, 16, 32, 64, 128, 256, 512)])


def _same(a, b):
    assert a[0] == b[0]
    for ra, rb, fa, fb in zip(a[1], b[1], a[2], b[2]):
        assert ra.tobytes() == rb.tobytes()
        assert np.array_equal(fa.eps, fb.eps) and np.array_equal(fa.plastic, fb.plastic)
        assert np.array_equal(fa.labels, fb.labels)


@pytest.mark.parametrize("prec,L,tiling", SIZES)
def test_same_bits_as_the_passes(prec, L, tiling, monkeypatch):
    from paper_0802_2488_gb300 import binding as B
    from paper_0802_2488_gb300 import inputs
    with B.Context(0) as ctx:
        B.epfft_set_tiling(ctx, L, prec, tiling)
        for n, green in ((1, "eq3"), (2, "eq3"), (2, "dg1")):
            probs = [B.Problem(L=L, precision=prec, void_fraction=0.2, seed=s, max_iter=6 + 3 * s, green=green,
                               tol_eq=1e-2, tol_macro=1e-1) for s in range(n)]
            paths = [inputs.load_path("shear", 2 + s, 3.0) for s in range(n)]
            got = B.epfft_solve_batch(ctx, probs, paths, fields=True)
            # the starting state, one loop launch, the check records and the
            # labels (batches of the larger sides may exceed the GPU's CTAs and
            # run the passes)
            assert B.epfft_last_stats(ctx)["kernel_launches"] == 3 + 3 * n or (n > 1 and L >= 256)
            monkeypatch.setenv("EPFFT_SYNC_CHECK", "1")
            ref = B.epfft_solve_batch(ctx, probs, paths, fields=True)
            monkeypatch.delenv("EPFFT_SYNC_CHECK")
            _same(got, ref)


def test_mixed_call_equals_resident_alone():
    from paper_0802_2488_gb300 import binding as B
    from paper_0802_2488_gb300 import inputs
    with B.Context(0) as ctx:
        B.epfft_set_tiling(ctx, 128, "fp32", 1)
        probs = [B.Problem(L=64, precision="fp64", void_fraction=0.1, seed=1, max_iter=40),
                 B.Problem(L=128, precision="fp32", void_fraction=0.2, seed=2, max_iter=30)]
        paths = [inputs.load_path("shear", 2, 2.0), inputs.load_path("equibiaxial", 3, 2.0)]
        rc, recs, fs = B.epfft_solve_batch(ctx, probs, paths, fields=True)
        for i in range(2):
            _same(B.epfft_solve_batch(ctx, probs[i:i + 1], paths[i:i + 1], fields=True),
                  (rc, recs[i:i + 1], fs[i:i + 1]))


def test_iterate_accepts_a_strain_off_the_16_byte_boundary():
    """The accepted strain is written back by a kernel of 16-byte words, or by a
    copy where the caller's buffer does not start on such a boundary."""
    import torch
    from paper_0802_2488_gb300 import binding as B
    L = 32
    base = torch.rand(4 * L * L + 1, device="cuda", generator=torch.Generator("cuda").manual_seed(3)) * 0.5
    a = base[:-1].clone().view(L, L, 4)
    b = torch.empty(4 * L * L + 1, device="cuda")[1:].view(L, L, 4)
    b.copy_(a)
    assert b.data_ptr() % 16 == 4
    with B.Context(0) as ctx:
        prob = B.Problem(L=L, precision="fp32", void_fraction=0.2, seed=1)
        for t in (a, b):
            B.epfft_iterate(ctx, prob, [0.3, 0.2, 0.0, 0.1], t, 3)
    assert torch.equal(a, b)
