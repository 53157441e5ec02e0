"""Performance cases: the work a user of the library has it do, each through
the package's public entry points.

Six kinds of call:

* ``solve``     epfft_solve_batch: one lattice or a batch through a loading
                path, capped iterations per increment, as the studies of the
                paper run it (the library's main call);
* ``iterate``   epfft_iterate: a fixed number of augmented-Lagrangian
                iterations of one lattice from a given strain field, with any
                of the Green operators;
* ``project``   epfft_project: the compatible-strain projection of Eqs. 2-3;
* ``displace``  epfft_displacement: the displacement field of a strain field;
* ``serve``     a burst of requests of mixed sides through the serving engine;
* ``clusters``  epfft_void_plastic: the void-plastic clusters of Sec. 3 for the
                plastic zones of successive increments.

The context of a state is tuned once (epfft_autotune), as the benchmark and
the README do, and kept.

Outputs are returned by the precision their form computes in: the records
of the single-precision and defect-correction forms hold numbers of single
accuracy in double fields and are returned as float32.  Plastic flags, labels
and counts are returned where the form is double precision throughout; in the
other forms a pixel at the yield threshold may fall on either side of it.
"""
import math

import numpy as np
import torch

from paper_0802_2488_gb300 import binding as B
from paper_0802_2488_gb300 import inputs

DEV = "cuda:0"
MU, LAM, Y = inputs.MU, inputs.LAMBDA, inputs.YIELD
L2_BYTES = 126 << 20


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # The smallest study (the L = 64, f = 0.1 lattice under equibiaxial
        # loading to twice the yield strain), plain double precision, all
        # fields wanted: every iteration is launch and latency.
        dict(name="solve_fp64_L64", kind="solve", precision="fp64", L=64, n=1, f=0.10, mode="equibiaxial",
             n_inc=4, max_iter=100, fields=True),
        # The single-lattice study in shear, plain double precision with
        # all fields (the reference against which the other forms are judged).
        dict(name="solve_fp64_L256", kind="solve", precision="fp64", L=256, n=1, f=0.20, mode="shear",
             n_inc=2, max_iter=100, fields=True),
        # The same lattice in single precision: one ordinary lattice alone.
        dict(name="solve_fp32_L256", kind="solve", precision="fp32", L=256, n=1, f=0.20, mode="shear",
             n_inc=4, max_iter=100, fields=False),
        # Many realizations of a small cell: statistics over disorder.
        dict(name="solve_fp32_96xL32", kind="solve", precision="fp32", L=32, n=96, f=0.20, mode="shear",
             n_inc=4, max_iter=100, fields=False),
        # The batched study: 64 realizations of L = 512 (the headline of the
        # benchmark), macroscopic curves only.
        dict(name="solve_fp32_64xL512", kind="solve", precision="fp32", L=512, n=64, f=0.20, mode="equibiaxial",
             n_inc=2, max_iter=30, fields=False),
        # A batch solved in plain double precision, all fields to page-locked
        # buffers.
        dict(name="solve_fp64_8xL512", kind="solve", precision="fp64", L=512, n=8, f=0.10, mode="equibiaxial",
             n_inc=1, max_iter=25, fields=True),
        # The same batch in the defect-correction form, which certifies
        # double-precision tolerances at single-precision cost.
        dict(name="solve_defect_8xL512", kind="solve", precision="fp32_defect", L=512, n=8, f=0.10,
             mode="equibiaxial", n_inc=1, max_iter=100, fields=False),
        # The largest lattice, single precision: iterations of its field.
        dict(name="iterate_fp32_L4096", kind="iterate", precision="fp32", L=4096, f=0.35, green="eq3", n_iter=20),
        # The symmetrized operator of the operator comparison at L = 1024.
        dict(name="iterate_dg1_L1024", kind="iterate", precision="fp32", L=1024, f=0.10, green="dg1", n_iter=25),
        # The projection alone on a large field (one application of Gamma).
        dict(name="project_fp32_L2048", kind="project", precision="fp32", L=2048),
        # A burst of requests of the serving mix (L = 128 .. 1024).
        dict(name="serve_fp32_mix", kind="serve", precision="fp32", n=12, n_inc=4, max_iter=20),
        # Sec. 3 analysis of a solve: void-plastic clusters of the plastic
        # zone of each increment.
        dict(name="clusters_10xL1024", kind="clusters", L=1024, n=10, f=0.20),
    ]


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "iterate", "iterate", "project", "displace", "serve", "clusters"])
    f = round(rng.uniform(0.05, 0.35), 3)
    if kind == "solve":
        prec = rng.choice(["fp64", "fp32", "fp32_defect"])
        L = 2 ** rng.randint(4, 10)
        most = (4 if prec == "fp64" else 16) * 512 * 512  # pixels of the batch
        n = int(math.exp(rng.uniform(0.0, math.log(max(1, min(96, most // (L * L))) + 0.999))))
        budget = (40e6 if prec == "fp64" else 300e6) / (n * L * L)  # iterations
        n_inc = rng.randint(1, 4)
        cap = max(3, min(rng.randint(20, 100), int(budget / n_inc)))
        return dict(kind="solve", precision=prec, L=L, n=n, f=f, mode=rng.choice(["equibiaxial", "shear"]),
                    n_inc=n_inc, max_iter=cap, fields=prec == "fp64" and n <= 16)
    if kind == "iterate":
        prec = rng.choice(["fp64", "fp32", "fp32"])
        L = 2 ** rng.randint(5, 11 if prec == "fp64" else 12)
        k = int(math.exp(rng.uniform(math.log(2), math.log(25.9))))
        if prec == "fp64":
            k = max(1, min(k, int(40e6 / (L * L))))
        return dict(kind="iterate", precision=prec, L=L, f=f, green=rng.choice(["eq3", "eq3", "cg1", "dg1"]), n_iter=k)
    if kind in ("project", "displace"):
        return dict(kind=kind, precision=rng.choice(["fp64", "fp32"]), L=2 ** rng.randint(5, 12),
                    f=f)
    if kind == "serve":
        return dict(kind="serve", precision="fp32", n=rng.randint(3, 12), n_inc=rng.randint(2, 4),
                    max_iter=rng.randint(8, 20))
    L = 2 ** rng.randint(7, 11)
    return dict(kind="clusters", L=L, n=rng.randint(1, max(1, min(16, 10 * 1024 * 1024 // (L * L)))), f=f)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _path(case):
    return inputs.load_path(case["mode"], case["n_inc"], 2.0 if case["mode"] == "equibiaxial" else 3.0)


def _void_seeds(case, seed):
    return [int(seed) * 1009 + i for i in range(case["n"])]


def _requests(case, seed):
    """The burst's problems: the recipe of the serving stream."""
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["n"]):
        L = (128, 256, 512, 1024)[i % 4]
        mode = "equibiaxial" if rng.random() < 0.5 else "shear"
        out.append(dict(L=L, n=1, f=float(rng.uniform(0.05, 0.35)), mode=mode, n_inc=case["n_inc"],
                        max_iter=case["max_iter"], seed=int(seed) * 1009 + i))
    return out


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _mean_strain(seed):
    r = np.random.default_rng(seed)
    return np.array([0.35, 0.30, 0.0, 0.15]) + 0.1 * r.uniform(-1, 1, 4) * np.array([1.0, 1.0, 0.0, 1.0])


def _iterate_inputs(case, seed):
    """Void mask, mean strain and a generic strain field around it."""
    L, g = case["L"], _gen(seed)
    mask = (torch.rand((L, L), generator=g, device=DEV) < case["f"]).to(torch.uint8)
    E = _mean_strain(seed)
    dt = torch.float32 if case["precision"] == "fp32" else torch.float64
    eps = torch.rand((L, L, 4), generator=g, device=DEV, dtype=dt).sub_(0.5).mul_(0.6)
    eps += torch.tensor(E, device=DEV, dtype=dt)
    return mask, E, eps


def _field(case, seed, shape):
    dt = torch.float32 if case["precision"] == "fp32" else torch.float64
    return torch.randn(shape, generator=_gen(seed), device=DEV, dtype=dt)


def _cluster_inputs(case, seed):
    """Voids, and plastic zones that grow around them from image to image: a
    smoothed void density plus noise above a falling threshold."""
    L, n, g = case["L"], case["n"], _gen(seed)
    mask = (torch.rand((L, L), generator=g, device=DEV) < case["f"]).to(torch.uint8)
    q = torch.fft.fftfreq(L, device=DEV) * L
    k = torch.exp(-0.5 * ((q[:, None] ** 2 + q[None, :L // 2 + 1] ** 2) / (L / 12.0) ** 2))
    s = torch.fft.irfft2(torch.fft.rfft2(mask.float() + 0.5 * torch.randn((L, L), generator=g, device=DEV)) * k,
                         s=(L, L))
    s = (s - s.mean()) / s.std() + 0.3 * torch.randn((L, L), generator=g, device=DEV)
    lev = torch.linspace(2.2, 0.2, n + 1, device=DEV)[1:]
    plastic = ((s[None] > lev[:, None, None]) & (mask[None] == 0)).to(torch.uint8)
    return mask, plastic.contiguous()


def prepare(case, seed):
    ctx = B.Context(0)
    st = dict(case=case, ctx=ctx)
    k = case["kind"]
    if k == "solve":
        if case["precision"] == "fp32_defect":
            B.epfft_autotune(ctx, case["L"], "fp64", case["n"])  # the reference refresh's passes
        B.epfft_autotune(ctx, case["L"], case["precision"], case["n"])
        st["problems"] = [B.Problem(L=case["L"], precision=case["precision"], void_fraction=case["f"], seed=s,
                                    max_iter=case["max_iter"]) for s in _void_seeds(case, seed)]
        st["paths"] = [_path(case)] * case["n"]
        if case["fields"]:
            st["out"] = [B.pinned_fields(p, case["n_inc"]) for p in st["problems"]]
    elif k == "iterate":
        B.epfft_autotune(ctx, case["L"], case["precision"], 1)
        mask, st["E"], st["eps"] = _iterate_inputs(case, seed)
        st["problem"] = B.Problem(L=case["L"], precision=case["precision"], mask=mask, green=case["green"])
    elif k == "project":
        B.epfft_autotune(ctx, case["L"], case["precision"], 1)
        st["E"], st["p"] = _mean_strain(seed), _field(case, seed, (3, case["L"], case["L"]))
    elif k == "displace":
        B.epfft_autotune(ctx, case["L"], case["precision"], 1)
        st["eps"] = _field(case, seed, (case["L"], case["L"], 4))
    elif k == "serve":
        for L in (128, 256, 512, 1024):
            B.epfft_autotune(ctx, L, case["precision"], 16)
        st["requests"] = [(B.Problem(L=r["L"], precision=case["precision"], void_fraction=r["f"], seed=r["seed"],
                                     max_iter=r["max_iter"]), _path(r)) for r in _requests(case, seed)]
    else:
        st["mask"], st["plastic"] = _cluster_inputs(case, seed)
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def _record_values(recs, double):
    """Macroscopic curves and indicators of the increments of each solve."""
    dt = np.float64 if double else np.float32
    out = {"sigma": np.stack([r["sig_mean"] for r in recs]).astype(dt),
           "strain": np.stack([r["eps_mean"] for r in recs]).astype(dt),
           "eta": np.stack([np.stack([r["eta1"], r["eta2"], r["eta3"]], -1) for r in recs]).astype(dt),
           "iterations": np.stack([r["iterations"] for r in recs]),
           "status": np.stack([r["status"] for r in recs])}
    if double:
        out["n_plastic"] = np.stack([r["n_plastic"] for r in recs])
        out["n_clusters"] = np.stack([r["n_clusters"] for r in recs])
    return out


def run(state):
    case, ctx = state["case"], state["ctx"]
    k = case["kind"]
    if k == "solve":
        if case["fields"]:
            _, recs, f = B.epfft_solve_batch(ctx, state["problems"], state["paths"], fields=True, out=state["out"])
            out = _record_values(recs, case["precision"] == "fp64")
            out["eps"] = [x.eps for x in f]
            out["plastic"] = [x.plastic for x in f]
            out["labels"] = [x.labels for x in f]
            return out
        _, recs = B.epfft_solve_batch(ctx, state["problems"], state["paths"])
        return _record_values(recs, case["precision"] == "fp64")
    if k == "iterate":
        rec = B.epfft_iterate(ctx, state["problem"], state["E"], state["eps"], case["n_iter"])
        dt = np.float32 if case["precision"] == "fp32" else np.float64
        return {"eps": state["eps"], "sigma": rec["sig_mean"].astype(dt), "strain": rec["eps_mean"].astype(dt)}
    if k == "project":
        return {"e": B.epfft_project(ctx, case["L"], case["precision"], LAM, MU, state["E"], state["p"])}
    if k == "displace":
        return {"u": B.epfft_displacement(ctx, case["L"], case["precision"], state["eps"])}
    if k == "serve":
        B.epfft_serve_open(ctx, 64 << 30, 16, 32)
        try:
            tickets = [B.epfft_submit(ctx, p, path) for p, path in state["requests"]]
            res = [None] * len(tickets)
            while any(r is None for r in res):
                B.epfft_serve_step(ctx)
                for i, t in enumerate(tickets):
                    if res[i] is None:
                        res[i] = B.epfft_poll(ctx, t, state["requests"][i][0], case["n_inc"])
        finally:
            B.epfft_serve_close(ctx)
        return _record_values([r[1] for r in res], False)
    stats, labels = B.epfft_void_plastic(ctx, state["mask"], state["plastic"], labels=True)
    return {"stats": stats, "labels": labels}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _iteration_work(L, n, iters, rs):
    """Flops of the transforms (30 log2 L per pixel for three components both
    ways), the Green operator and the local step; bytes of strain, stress and
    spectrum per iteration (20 reals per pixel) where the batch exceeds the
    last-level cache, else one read and write of the state."""
    px = n * L * L
    flops = px * iters * (30.0 * math.log2(L) + 85.0)
    state = px * (8 * rs + 1)
    return (px * iters * (20.0 * rs + 1) if px * 11 * rs > L2_BYTES else 2.0 * state), flops


def work(case):
    k = case["kind"]
    L = case.get("L", 0)
    rs = 8 if case.get("precision") == "fp64" else 4
    if k == "solve":
        b, f = _iteration_work(L, case["n"], case["n_inc"] * (case["max_iter"] + 1), rs)
        if case["fields"]:
            b += case["n"] * L * L * (4 * rs + 5 * case["n_inc"])
        return {"bytes": b, "flops": f}
    if k == "iterate":
        b, f = _iteration_work(L, 1, case["n_iter"], rs)
        return {"bytes": b, "flops": f}
    if k == "project":
        return {"bytes": 6.0 * L * L * rs, "flops": L * L * (30.0 * math.log2(L) + 25.0)}
    if k == "displace":
        return {"bytes": 6.0 * L * L * rs, "flops": L * L * (25.0 * math.log2(L) + 25.0)}
    if k == "serve":
        b = f = 0.0
        for r in _requests(case, 0):
            x, y = _iteration_work(r["L"], 1, r["n_inc"] * (r["max_iter"] + 1), rs)
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    return {"bytes": L * L * (1.0 + case["n"] * (1.0 + 4.0)), "flops": 0.0}


# ---------------------------------------------------------------------------
# The same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _void_mask(L, f, seed):
    """i.i.d. voids of the SplitMix64 stream of `seed`: pixel x is a void iff
    the top 53 bits of output x are below floor(f 2^53)."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, L * L + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z ^= z >> np.uint64(31)
    v = (z >> np.uint64(11)) < np.uint64(math.floor(f * 2.0 ** 53))
    return torch.from_numpy(v.reshape(L, L)).to(DEV)


def _apply(k1, k2, c):
    """Eq. 3 at symbols k1, k2 on a spectrum c (n, 3, L, L/2 + 1): the strain
    -(k_a v_b + k_b v_a) / 2 with N v = w, w_a = k*_b p_ab, N the acoustic
    tensor of the reference medium (the matrix); zero where k = 0."""
    p11, p22, p12 = c[:, 0], c[:, 1], c[:, 2]
    j1, j2 = k1.conj(), k2.conj()
    a1, a2 = (k1 * j1).real, (k2 * j2).real
    n11, n22 = LAM * a1 + MU * (a1 + a2) + MU * a1, LAM * a2 + MU * (a1 + a2) + MU * a2
    n12 = LAM * j1 * k2 + MU * k1 * j2
    det = n11 * n22 - (n12 * n12.conj()).real
    det = torch.where(det == 0, torch.ones_like(det), det)
    w1, w2 = j1 * p11 + j2 * p12, j1 * p12 + j2 * p22
    v1, v2 = (n22 * w1 - n12 * w2) / det, (n11 * w2 - n12.conj() * w1) / det
    return torch.stack([-(k1 * v1), -(k2 * v2), -0.5 * (k1 * v2 + k2 * v1)], 1)


class _Gamma:
    """e = E + Gamma p for (n, 3, L, L) fields indexed [x2][x1]."""

    def __init__(self, L, green="eq3"):
        self.L, self.green = L, green
        m = torch.arange(L, device=DEV, dtype=torch.float64)
        q = 2.0 * math.pi * m / L
        if green == "cg1":
            k = torch.where(m > L // 2, q - 2.0 * math.pi, q).to(torch.complex128)
        else:
            k = torch.complex(torch.sin(q), 2.0 * torch.sin(0.5 * q) ** 2)
        h = L // 2 + 1
        neg = (-torch.arange(L, device=DEV)) % L
        self.k1, self.k2 = k[None, :h], k[:, None]
        if green == "cg1":  # both signs of the ambiguous Nyquist momenta
            s = torch.ones(L, device=DEV, dtype=torch.float64)
            s[L // 2] = -1.0
            self.n1, self.n2 = (k * s)[None, :h], (k * s)[:, None]
        else:
            self.n1, self.n2 = k[neg][None, :h], k[neg][:, None]

    def hat(self, c):
        if self.green == "eq3":
            return _apply(self.k1, self.k2, c)
        if self.green == "cg1":
            return 0.25 * (_apply(self.k1, self.k2, c) + _apply(self.n1, self.k2, c) + _apply(self.k1, self.n2, c) +
                           _apply(self.n1, self.n2, c))
        d = torch.tensor([1.0, 1.0, -1.0], device=DEV, dtype=torch.float64)[None, :, None, None]
        return 0.25 * (_apply(self.k1, self.k2, c) + _apply(self.n1, self.n2, c) +
                       d * (_apply(self.n1, self.k2, d * c) + _apply(self.k1, self.n2, d * c)))

    def __call__(self, p, E):
        c = self.hat(torch.fft.rfft2(p))
        c[:, :, 0, 0] = 0.0
        e = torch.fft.irfft2(c, s=(self.L, self.L))
        return e + torch.as_tensor(E, device=DEV, dtype=torch.float64)[:, [0, 1, 3]][:, :, None, None]


def _c0(a):
    t = LAM * (a[:, 0] + a[:, 1] + a[:, 2])
    return torch.stack([t + 2 * MU * a[:, 0], t + 2 * MU * a[:, 1], t + 2 * MU * a[:, 2], 2 * MU * a[:, 3]], 1)


def _split(a):
    m = (a[:, 0] + a[:, 1] + a[:, 2]) / 3.0
    d = torch.stack([a[:, 0] - m, a[:, 1] - m, a[:, 2] - m, a[:, 3]], 1)
    return m, d, torch.sqrt(d[:, 0] ** 2 + d[:, 1] ** 2 + d[:, 2] ** 2 + 2.0 * d[:, 3] ** 2)


def _join(m, d):
    return torch.stack([d[:, 0] + m, d[:, 1] + m, d[:, 2] + m, d[:, 3]], 1)


_CAP = math.sqrt(2.0 / 3.0) * Y
_K = LAM + 2.0 * MU / 3.0


def _stress(e, void):
    m, d, r = _split(e)
    g = torch.where(2 * MU * r > _CAP, _CAP / r.clamp_min(1e-300), torch.full_like(r, 2 * MU))
    return torch.where(void[:, None], torch.zeros_like(e), _join(3 * _K * m, g[:, None] * d))


def _local(t, void):
    """Strain with sigma(eps) + C0:eps = t (C0 the matrix)."""
    m, d, r = _split(t)
    el = torch.full_like(r, 1.0 / (4.0 * MU))
    sc = torch.where(0.5 * r > _CAP, (1.0 - _CAP / r.clamp_min(1e-300)) / (2.0 * MU), el)
    sc = torch.where(void, torch.full_like(r, 1.0 / (2.0 * MU)), sc)
    return _join(torch.where(void, m / (3.0 * _K), m / (6.0 * _K)), sc[:, None] * d)


def _iterate64(gam, void, eps, E, iters):
    """`iters` iterations at mean strains E (n, 4) from eps (n, 4, L, L):
    the last strain and its record values."""
    E = np.asarray(E, dtype=np.float64).reshape(-1, 4)
    E33 = torch.tensor(E[:, 2], device=DEV)[:, None, None]
    lam = _stress(eps, void)
    sm = lam.mean((2, 3))
    for _ in range(iters):
        p = lam - _c0(eps)
        ei = gam(p[:, [0, 1, 3]], E)
        e = torch.stack([ei[:, 0], ei[:, 1], E33.expand_as(ei[:, 0]), ei[:, 2]], 1)
        tau = lam + _c0(e)
        eps = _local(tau, void)
        lam = tau - _c0(eps)
        prev, sm = sm, lam.mean((2, 3))
    lam = _stress(eps, void)
    d1 = lam[:, 0] - lam[:, 0].roll(1, 2) + lam[:, 3] - lam[:, 3].roll(1, 1)
    d2 = lam[:, 3] - lam[:, 3].roll(1, 2) + lam[:, 1] - lam[:, 1].roll(1, 1)
    sm = lam.mean((2, 3))
    dot = lambda a: a[:, 0] ** 2 + a[:, 1] ** 2 + 2.0 * a[:, 3] ** 2  # noqa: E731
    r = eps - e
    comp = (r[:, 0] ** 2 + r[:, 1] ** 2 + r[:, 2] ** 2 + 2.0 * r[:, 3] ** 2).mean((1, 2))
    Et = torch.tensor(E, device=DEV)
    EE = Et[:, 0] ** 2 + Et[:, 1] ** 2 + Et[:, 2] ** 2 + 2.0 * Et[:, 3] ** 2
    eta = torch.stack([torch.sqrt((d1 ** 2 + d2 ** 2).mean((1, 2)) / dot(sm)), torch.sqrt(dot(sm - prev) / dot(sm)),
                       torch.sqrt(comp / EE)], -1)
    return eps, sm, eps.mean((2, 3)), eta


def _solve64(L, void, paths, max_iter):
    """The solves of void masks (n, L, L) along paths (n, n_inc, 4)."""
    gam = _Gamma(L)
    n, n_inc = paths.shape[:2]
    eps = torch.zeros((n, 4, L, L), device=DEV, dtype=torch.float64)
    last = np.zeros((n, 4))
    rec = []
    for k in range(n_inc):
        eps = eps + torch.tensor(paths[:, k] - last, device=DEV)[:, :, None, None]
        last = paths[:, k]
        eps, s, e, eta = _iterate64(gam, void, eps, paths[:, k], max_iter)
        rec.append((s, e, eta))
    cols = [torch.stack([r[j] for r in rec], 1) for j in range(3)]
    return eps, cols


def exact(case, seed):
    k = case["kind"]
    if k == "clusters":
        return None  # whole numbers only
    if k == "solve":
        L, n = case["L"], case["n"]
        sig, strain, eta, fields = [], [], [], []
        path = _path(case)
        seeds = _void_seeds(case, seed)
        step = max(1, (1 << 22) // (L * L))  # lattices at a time
        for i in range(0, n, step):
            void = torch.stack([_void_mask(L, case["f"], s) for s in seeds[i:i + step]])
            eps, c = _solve64(L, void, np.stack([path] * len(void)), case["max_iter"])
            sig, strain, eta = sig + [c[0]], strain + [c[1]], eta + [c[2]]
            if case["fields"]:
                fields += [x.permute(1, 2, 0).contiguous() for x in eps]
        out = {"sigma": torch.cat(sig), "strain": torch.cat(strain), "eta": torch.cat(eta)}
        if case["fields"]:
            out["eps"] = fields
        return out
    if k == "iterate":
        mask, E, eps = _iterate_inputs(case, seed)
        gam = _Gamma(case["L"], case["green"])
        e, s, m, _ = _iterate64(gam, (mask != 0)[None], eps.double().permute(2, 0, 1)[None].contiguous(), E[None],
                                case["n_iter"])
        return {"eps": e[0].permute(1, 2, 0).contiguous(), "sigma": s[0], "strain": m[0]}
    if k == "project":
        p = _field(case, seed, (3, case["L"], case["L"])).double()
        return {"e": _Gamma(case["L"])(p[None], _mean_strain(seed)[None])[0]}
    if k == "displace":
        return {"u": _displacement64(_field(case, seed, (case["L"], case["L"], 4)).double(), case["L"])}
    out = []
    for r in _requests(case, seed):
        void = _void_mask(r["L"], r["f"], r["seed"])[None]
        out.append(_solve64(r["L"], void, _path(r)[None], r["max_iter"])[1])
    return {"sigma": torch.cat([c[0] for c in out]), "strain": torch.cat([c[1] for c in out]),
            "eta": torch.cat([c[2] for c in out])}


def _displacement64(eps, L):
    """Displacement of Sec. 2: (u1, u2) from e11, e22, e12 with the complex
    k^2 = k1^2 + k2^2, and with |k|^2 at the two modes where k^2 vanishes."""
    g = _Gamma(L)
    k1, k2 = g.k1.expand(L, -1), g.k2.expand(-1, L // 2 + 1)
    e = torch.fft.rfft2(eps.permute(2, 0, 1))
    e11, e22, e12 = e[0], e[1], e[3]
    kk = k1 * k1 + k2 * k2
    zero = torch.zeros_like(kk, dtype=torch.bool)
    if L % 4 == 0:
        zero[3 * L // 4, L // 4] = True  # (m1, m2) = (L/4, 3L/4); the other one is its mirror
    den = torch.where(zero, torch.ones_like(kk), kk)
    den[0, 0] = 1.0
    u1 = -1j / den * (k1 * (e11 - e22) + 2 * k2 * e12)
    u2 = 1j / den * (k2 * (e11 - e22) - 2 * k1 * e12)
    nk = (k1 * k1.conj() + k2 * k2.conj()).real
    nk[0, 0] = 1.0
    w1, w2 = k1.conj() * e11 + k2.conj() * e12, k1.conj() * e12 + k2.conj() * e22
    s = -1j * (k1.conj() * w1 + k2.conj() * w2) / nk
    u1 = torch.where(zero, (-2j * w1 - k1 * s) / nk, u1)
    u2 = torch.where(zero, (-2j * w2 - k2 * s) / nk, u2)
    u1[0, 0] = 0.0
    u2[0, 0] = 0.0
    return torch.stack([torch.fft.irfft2(u1, s=(L, L)), torch.fft.irfft2(u2, s=(L, L))], -1)
