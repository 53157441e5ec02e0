"""Cluster labels and void-plastic clusters at the edges of the labelling's
tiles (64 x 32 pixels in shared memory, whole images below): against the
oracle, whole numbers, for every way a cluster can cross a tile or image
border."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def _images(L):
    rng = np.random.default_rng(L)
    im = [rng.random((L, L)) < p for p in (0.1, 0.5, 0.59, 0.8)]
    x, y = np.meshgrid(np.arange(L), np.arange(L))
    im += [np.ones((L, L), bool), np.zeros((L, L), bool), (x + y) % 2 == 0, x % 2 == 0, y % 2 == 0,
           (y % 2 == 0) | (x == np.where(y % 4 == 1, L - 1, 0)),  # one winding cluster
           (x == y) | (x == (y + 1) % L)]                          # a diagonal staircase
    return np.stack(im).astype(np.uint8)


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("L", [2, 4, 8, 16, 32, 64, 128, 256])
def test_labels(L, periodic):
    import torch
    from paper_0802_2488_gb300 import binding as B
    im = _images(L)
    with B.Context(0) as ctx:
        lab, counts = B.epfft_label(ctx, torch.tensor(im, device="cuda"), periodic)
    lab = lab.cpu().numpy()
    for i in range(len(im)):
        ref, n = O.label(im[i], periodic)
        np.testing.assert_array_equal(lab[i], ref)
        assert counts[i] == n


@pytest.mark.parametrize("L", [4, 16, 32, 64, 128])
def test_void_plastic_images(L):
    from paper_0802_2488_gb300 import binding as B
    im = _images(L)
    rng = np.random.default_rng(L + 1)
    with B.Context(0) as ctx:
        for mask in ((rng.random((L, L)) < 0.05).astype(np.uint8), np.zeros((L, L), np.uint8),
                     np.ones((L, L), np.uint8)):
            pl = im & (1 - mask)  # plastic pixels are matrix pixels
            st, lab = B.epfft_void_plastic(ctx, mask, pl, labels=True)
            only = B.epfft_void_plastic(ctx, mask, pl)
            np.testing.assert_array_equal(st, only)
            lab = lab.cpu().numpy()
            for i in range(len(pl)):
                ref = O.void_plastic(mask, pl[i])
                np.testing.assert_array_equal(lab[i], ref[0])
                np.testing.assert_array_equal(st[i], ref[1])
