"""Calls whose scratch cannot be had in one piece, or at all, take the form that
needs less, with the same results.  The context's allocator hook (torch's caching
allocator) is wrapped to refuse allocations."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture
def hook(monkeypatch):
    """Records the sizes asked for; refuses those `refuse(index, size)` names,
    index counting from the last reset."""
    import torch

    class Hook:
        sizes, granted = [], []
        refuse = staticmethod(lambda i, n: False)

        def reset(self, refuse=None):
            self.sizes, self.granted = [], []
            self.refuse = refuse or (lambda i, n: False)
    h = Hook()
    h.reset()
    real = torch.cuda.caching_allocator_alloc

    def alloc(size, device=None, stream=None):
        i = len(h.sizes)
        h.sizes.append(int(size))
        if h.refuse(i, int(size)):
            raise torch.cuda.OutOfMemoryError("refused by the test")
        h.granted.append(int(size))
        return real(size, device, stream)
    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    return h


@pytest.mark.parametrize("prec,L,tiling", [("fp64", 64, 1), ("fp32", 256, 1)])
def test_small_solve_without_the_resident_schedules_scratch(hook, prec, L, tiling):
    from paper_0802_2488_gb300 import binding as B
    from paper_0802_2488_gb300 import inputs
    with B.Context(0) as ctx:
        B.epfft_set_tiling(ctx, L, prec, tiling)
        prob = B.Problem(L=L, precision=prec, void_fraction=0.2, seed=1, max_iter=20)
        path = inputs.load_path("shear", 2, 3.0)
        solve = lambda: B.epfft_solve(ctx, prob, path, fields=True)
        solve()  # tables and the context's own blocks
        hook.reset()
        rc, rec, f = solve()
        resident = B.epfft_last_stats(ctx)["kernel_launches"]
        # the batch's block first, then the schedule's two buffers
        for k in (1, 2):
            hook.reset(lambda i, n: i == k)
            rc2, rec2, f2 = solve()
            assert B.epfft_last_stats(ctx)["kernel_launches"] > resident + 10
            assert rc2 == rc and rec2.tobytes() == rec.tobytes()
            assert np.array_equal(f2.eps, f.eps) and np.array_equal(f2.labels, f.labels)


def test_cluster_counts_and_void_plastic_take_what_scratch_there_is(hook):
    """A refused size is halved until it can be had: with 3 images' worth there,
    8 images are labelled 2 at a time and not one by one."""
    import torch
    from paper_0802_2488_gb300 import binding as B
    from paper_0802_2488_gb300 import inputs
    L, n = 64, 8
    g = torch.Generator(device="cuda").manual_seed(4)
    mask = (torch.rand((L, L), generator=g, device="cuda") < 0.2).to(torch.uint8)
    plastic = ((torch.rand((n, L, L), generator=g, device="cuda") < 0.4) & (mask == 0)).to(torch.uint8)
    with B.Context(0) as ctx:
        ref, lab = B.epfft_void_plastic(ctx, mask, plastic, labels=True)
        per = 26 * L * L
        hook.reset(lambda i, s: s > 3 * per)
        got, lab2 = B.epfft_void_plastic(ctx, mask, plastic, labels=True)
        assert hook.granted[0] == 2 * per
        assert np.array_equal(got, ref) and torch.equal(lab, lab2)
        # a solve without fields counts the clusters of its increments' flags
        prob = B.Problem(L=L, precision="fp64", void_fraction=0.2, seed=1, max_iter=20)
        path = inputs.load_path("shear", n, 3.0)
        _, rec = B.epfft_solve(ctx, prob, path)
        per = 4 * L * L
        hook.reset(lambda i, s: s == n * per)
        _, rec2 = B.epfft_solve(ctx, prob, path)
        assert n * per in hook.sizes and n // 2 * per in hook.granted
        assert rec.tobytes() == rec2.tobytes()
