"""The workloads this library's speed is judged on: what a user of the plane-wave Kohn-Sham
library has it do, through its public entry points (``paper_2507_08578_gb300.kss``), from the
smallest call to the largest.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (the
system handle with its tables, band blocks, start values), ``run`` is one call (or the few calls
that belong together), ``exact`` the same result from plain torch in 64 bits, ``work`` the bytes
and operations the result cannot do without.

The systems are the seeded synthetic ones of ``workloads``: cubic cells, Gaussian local potential,
one s and three p projectors per atom; only their atoms, projector energies and band blocks come
from the seed, their sizes from the case.
"""
import math
import random

import numpy as np
import torch

import paper_2507_08578_gb300.kss as K

DEV = "cuda"
_ctx = None

# coefficients of a Chebyshev step in the middle of a filter (alpha H psi + beta psi + gamma psi_prev)
CHEB = (0.043, -1.07, -0.82)


def listed():
    return [
        # the smallest ordinary call: H on the block of a 4-atom cell at Gamma (latency, launches)
        {"name": "h_a10_fp64", "kind": "apply", "prec": "fp64", "a": 10.0, "ecut": 10.0, "natom": 4, "box": 24,
         "k": 0, "nb": 20},
        # one filter step of the 64-atom cell, 512 bands and their buffer, in double precision
        {"name": "cheb_a20_fp64", "kind": "cheb", "prec": "fp64", "a": 20.0, "ecut": 20.0, "natom": 64, "box": 96,
         "k": 1, "nb": 564},
        # the same step in the mixed form (complex64 transforms, split-BF16 projector products)
        {"name": "cheb_a20_mixed", "kind": "cheb", "prec": "mixed", "a": 20.0, "ecut": 20.0, "natom": 64, "box": 96,
         "k": 1, "nb": 564},
        # H on the many bands of a small cell at Gamma (real-space-real bands, two per transform)
        {"name": "h_gamma_a10_mixed", "kind": "gamma", "prec": "mixed", "a": 10.0, "ecut": 10.0, "natom": 4,
         "box": 24, "k": 0, "nb": 1127},
        # one system of a high-throughput campaign, mixed form: uneven box, ragged band count
        {"name": "cheb_a12_mixed", "kind": "cheb", "prec": "mixed", "a": 12.3, "ecut": 15.7, "natom": 37, "box": 0,
         "k": 1, "nb": 82},
        # another one in double precision: uneven box, odd band count
        {"name": "h_a14_fp64", "kind": "apply", "prec": "fp64", "a": 13.9, "ecut": 17.3, "natom": 21, "box": 0,
         "k": 2, "nb": 47},
        # the subspace products of Rayleigh-Ritz at 512 + 52 bands: Gram matrix and rotation
        {"name": "products_564_fp64", "kind": "products", "nb": 564, "npw": 34181},
        # the subspace eigenproblem of the 64-atom cell
        {"name": "eigen_564", "kind": "eigen", "n": 564, "real": False},
        # the subspace eigenproblem of 1024 + 103 bands at Gamma (real pencil)
        {"name": "eigen_1127_real", "kind": "eigen", "n": 1127, "real": True},
        # electron density of the 64-atom cell's bands at one k-point
        {"name": "density_a20_fp64", "kind": "density", "prec": "fp64", "a": 20.0, "ecut": 20.0, "natom": 64,
         "box": 96, "k": 1, "nb": 512},
        # a whole eigensolve of the 4-atom cell to residual 1e-8, and the density of its bands
        {"name": "solve_a10_fp64", "kind": "solve", "a": 10.0, "ecut": 10.0, "natom": 4, "box": 24, "k": 0,
         "nband": 16},
        # a batch of uneven systems solved together, mixed form
        {"name": "batch_12_mixed", "kind": "batch", "units": 12, "mix": 45},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["apply", "cheb", "cheb", "apply", "gamma", "products", "eigen", "density", "solve", "batch"])
    if kind in ("apply", "cheb", "gamma", "density"):
        prec = rng.choice(["fp64", "mixed"])
        a, ecut = round(_log(rng, 8.0, 20.0), 2), round(rng.uniform(10.0, 20.0), 2)
        natom = max(4, min(64, int(a ** 3 / 125 * rng.uniform(0.6, 1.6))))
        nb = int(_log(rng, 2, 512))
        while kind == "density" and a * math.sqrt(2 * ecut) / (2 * math.pi) > 14.7:  # boxes it accepts
            a, ecut = round(_log(rng, 8.0, 20.0), 2), round(rng.uniform(10.0, 20.0), 2)
        return {"kind": kind, "prec": prec, "a": a, "ecut": ecut, "natom": natom, "box": 0,
                "k": 0 if kind == "gamma" else rng.randint(0, 3), "nb": nb}
    if kind == "products":
        return {"kind": kind, "nb": int(_log(rng, 20, 564)), "npw": int(_log(rng, 1500, 34181))}
    if kind == "eigen":
        real = rng.random() < 0.5
        return {"kind": kind, "n": int(_log(rng, 20, 1127 if real else 700)), "real": real}
    if kind == "solve":
        return {"kind": kind, "a": round(rng.uniform(7.0, 11.0), 2), "ecut": round(rng.uniform(8.0, 11.0), 2),
                "natom": rng.randint(2, 6), "box": 0, "k": rng.randint(0, 3), "nband": rng.randint(6, 24)}
    return {"kind": "batch", "units": rng.randint(3, 12), "mix": rng.randint(0, 1 << 20)}


# ------------------------------------------------------------------------------------------------
# inputs

KPTS = [(0.0, 0.0, 0.0), (0.25, 0.25, 0.25), (0.25, 0.25, -0.25), (0.25, -0.25, 0.25), (-0.25, 0.25, 0.25)]


def _context():
    """One context for the process, on the stream torch uses."""
    global _ctx
    if _ctx is None:
        _ctx = K.kss_create(0)
    return _ctx


class Sys:
    """A system handle that is given back when the last state that holds it goes."""

    def __init__(self, a, ecut, natom, box, kpts, seed):
        self.d = _atoms(a, natom, seed)
        self.a, self.ecut, self.kpts = a, ecut, kpts
        self.h = K.kss_setup(_context(), np.eye(3) * a, ecut, kpts, self.d[0], self.d[1], fft_box=(box, box, box))

    def __del__(self):
        if getattr(self, "h", None) is not None:
            K.kss_sys_destroy(self.h)


def _atoms(a, natom, seed):
    r = np.random.default_rng(seed)
    return r.random((natom, 3)) * a, r.uniform(-1.0, 1.0, 4 * natom)


def _prec(case):
    return K.KSS_PREC_FP64 if case.get("prec", "fp64") == "fp64" else K.KSS_PREC_MIXED


def _type(case):
    return torch.complex128 if case.get("prec", "fp64") == "fp64" else torch.complex64


def _block(q2, nb, seed, dtype, gamma=False):
    """Bands like those of an iterate: random, falling off with the kinetic energy, unit norm."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    x = torch.randn(nb, q2.numel(), dtype=dtype, device=DEV, generator=g)
    if gamma:  # psi(-G) = conj psi(G): the canonical order of the sphere at Gamma is symmetric
        x = x + x.flip(1).conj()
    x *= 1.0 / (1.0 + 0.5 * q2.to(x.real.dtype))
    x /= torch.linalg.vector_norm(x, dim=1, keepdim=True)
    return x


def _q(miller, k, a):
    return (torch.as_tensor(np.asarray(miller, np.float64), device=DEV) + torch.tensor(k, dtype=torch.float64, device=DEV)) * (2 * math.pi / a)


def _batch_units(case):
    """Sizes of the batch: cells of 8 to 16 bohr, cutoffs of 12 to 20 Ha, 8 to 64 atoms, up to four
    k-points."""
    r, units = random.Random(case["mix"]), []
    while len(units) < case["units"]:
        a, ecut, natom = r.uniform(8.0, 16.0), r.uniform(12.0, 20.0), r.randint(8, 64)
        nk = min(r.randint(1, 4), case["units"] - len(units))
        units += [(a, ecut, natom, KPTS[1:1 + nk], ik) for ik in range(nk)]
    return units


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("apply", "cheb", "gamma", "density"):
        s = Sys(case["a"], case["ecut"], case["natom"], case["box"], [KPTS[case["k"]]], seed)
        q2 = (_q(K.kss_sphere(s.h, 0), KPTS[case["k"]], case["a"]) ** 2).sum(1)
        st = {"kind": kind, "sys": s, "prec": _prec(case)}
        st["psi"] = _block(q2, case["nb"], seed, _type(case), kind == "gamma")
        if kind == "cheb":
            st["prev"] = _block(q2, case["nb"], seed + 1, _type(case))
        if kind == "density":
            st["occ"] = np.where(np.arange(case["nb"]) < (case["nb"] * 9) // 10, 2.0, 0.7)
            st["shape"] = K.kss_sys_info_get(s.h)["fft_box"][::-1]
        else:
            st["out"] = torch.empty_like(st["psi"])
        return st
    if kind == "products":
        _context()
        g = torch.Generator(device=DEV).manual_seed(seed)
        nb, npw = case["nb"], case["npw"]
        t = torch.rand(npw, dtype=torch.float64, device=DEV, generator=g) * 40.0
        y = _block(t, nb, seed, torch.complex128)
        q = torch.randn(nb, nb, dtype=torch.complex128, device=DEV, generator=g) / math.sqrt(nb)
        return {"kind": kind, "y": y, "q": q, "s": torch.empty(nb, nb, dtype=torch.complex128, device=DEV),
                "x": torch.empty_like(y)}
    if kind == "eigen":
        _context()
        a, b = _pencil(case, seed)
        n = case["n"]
        return {"kind": kind, "real": case["real"], "a0": a, "b0": b, "a": torch.empty_like(a),
                "b": torch.empty_like(b), "w": torch.empty(n, dtype=torch.float64, device=DEV)}
    if kind == "solve":
        s = Sys(case["a"], case["ecut"], case["natom"], case["box"], [KPTS[case["k"]]], seed)
        npw = K.kss_sphere(s.h, 0).shape[0]
        return {"kind": kind, "sys": s, "nband": case["nband"], "opts": K.make_opts(tol=1e-8, seed=seed),
                "occ": np.full(case["nband"], 2.0), "shape": K.kss_sys_info_get(s.h)["fft_box"][::-1],
                "evecs": torch.empty(case["nband"], npw, dtype=torch.complex128, device=DEV)}
    systems, made = [], {}
    for a, ecut, natom, kpts, ik in _batch_units(case):
        if (a, ecut) not in made:
            made[a, ecut] = Sys(a, ecut, natom, 0, kpts, seed + len(made))
        systems.append(made[a, ecut])
    units = _batch_units(case)
    return {"kind": kind, "systems": systems, "iks": [u[4] for u in units], "nbands": [2 * u[2] for u in units],
            "opts": K.make_opts(degree=20, prec=K.KSS_PREC_MIXED, seed=seed)}


def _pencil(case, seed):
    """The pencil of a filtered block: eigenvectors nearly along the axes, columns of uneven norm."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    n, dt = case["n"], torch.float64 if case["real"] else torch.complex128
    u = torch.rand(n, dtype=torch.float64, device=DEV, generator=g)  # levels that keep apart
    lam = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.7 * u) * (6.0 / n) - 2.0
    m = torch.eye(n, dtype=dt, device=DEV) + 0.3 / math.sqrt(n) * torch.randn(n, n, dtype=dt, device=DEV, generator=g)
    m = m * (0.3 + torch.rand(n, dtype=torch.float64, device=DEV, generator=g))
    b = m.mH @ m
    a = m.mH @ (lam[:, None] * m)
    # one column per row: the transpose of a Hermitian matrix is its conjugate
    col = [((x + x.mH) * 0.5).to(torch.complex128).t().contiguous() for x in (a, b)]
    return col


def _fix_gauge(x):
    """Eigenvectors (rows of x) with the phase that makes their leading component positive."""
    c = x.diagonal()
    return x * (c.conj() / c.abs())[:, None]


# ------------------------------------------------------------------------------------------------
# one pass

def run(st):
    kind = st["kind"]
    if kind == "apply":
        K.kss_apply_H(st["sys"].h, 0, st["psi"], st["out"], st["prec"])
        return st["out"]
    if kind == "cheb":
        K.kss_cheb_step(st["sys"].h, 0, st["psi"], st["prev"], st["out"], *CHEB, prec=st["prec"])
        return st["out"]
    if kind == "gamma":
        K.kss_apply_H_gamma(st["sys"].h, 0, st["psi"], st["out"], st["prec"])
        return st["out"]
    if kind == "density":
        rho = torch.zeros(st["shape"], dtype=torch.float64, device=DEV)
        K.kss_density_accumulate(st["sys"].h, 0, st["psi"], st["occ"], rho, st["prec"])
        return rho
    if kind == "products":
        K.kss_gemm(_ctx, 0, st["y"], st["y"], st["s"])
        K.kss_gemm(_ctx, 1, st["y"], st["q"], st["x"])
        return {"gram": st["s"], "rotated": st["x"]}
    if kind == "eigen":  # the call overwrites its matrices
        st["a"].copy_(st["a0"])
        st["b"].copy_(st["b0"])
        K.kss_dense_hegv(_ctx, [st["a"]], [st["b"]], [st["w"]], real=st["real"])
        return {"values": st["w"], "vectors": _fix_gauge(st["a"])}
    if kind == "solve":
        ev, _, _, _ = K.kss_chebfi_solve(st["sys"].h, 0, st["nband"], st["opts"], evecs=st["evecs"])
        rho = torch.zeros(st["shape"], dtype=torch.float64, device=DEV)
        K.kss_density_accumulate(st["sys"].h, 0, st["evecs"], st["occ"], rho)
        return {"values": ev, "rho": rho}
    ev, _, _, _ = K.kss_solve_batch(_ctx, [s.h for s in st["systems"]], st["iks"], st["nbands"], st["opts"],
                                    allow_noconv=True)
    # eigenvalues of the mixed form are good to 1e-6 Ha: single-precision results
    return [e.astype(np.float32) for e in ev]


# ------------------------------------------------------------------------------------------------
# the same in 64 bits, without the library

def _sphere(a, ecut, k):
    r = int(a * math.sqrt(2 * ecut) / (2 * math.pi)) + 2
    m = np.arange(-r, r + 1)
    m3, m2, m1 = np.meshgrid(m, m, m, indexing="ij")
    m = np.stack([m1.ravel(), m2.ravel(), m3.ravel()], 1)
    q = (m + np.array(k)) * (2 * math.pi / a)
    return m[0.5 * ((q[:, 0] ** 2 + q[:, 1] ** 2) + q[:, 2] ** 2) <= ecut]


def _smooth(n):
    while True:
        r = n
        for p in (2, 3, 5):
            while r % p == 0:
                r //= p
        if r == 1:
            return n
        n += 1


class Dense:
    """H of one cubic system at one k-point as plain torch operations in 64 bits."""

    def __init__(self, a, ecut, natom, box, k, seed, kpts=None):
        pos, self.D = (torch.as_tensor(x, device=DEV) for x in _atoms(a, natom, seed))
        self.m = _sphere(a, ecut, k)
        self.N = N = box or _smooth(4 * max(int(np.abs(_sphere(a, ecut, x)).max()) for x in (kpts or [k])) + 1)
        q = _q(self.m, k, a)
        self.q2 = (q ** 2).sum(1)
        self.T = 0.5 * self.q2
        mm = torch.as_tensor(self.m % N, device=DEV)
        self.off = (mm[:, 2] * N + mm[:, 1]) * N + mm[:, 0]
        # V: a periodic sum of Gaussians, a product over the axes of a cubic cell
        x = torch.arange(N, dtype=torch.float64, device=DEV) * (a / N)
        im = torch.arange(-3, 4, dtype=torch.float64, device=DEV) * a
        e = torch.exp(-0.5 * (x[None, None, :, None] - pos.t()[:, :, None, None] - im) ** 2).sum(3)  # axis, atom, point
        self.V = -2.0 * torch.einsum("az,ay,ax->zyx", e[2], e[1], e[0])
        al, vol = 0.25, a ** 3
        cs = math.sqrt((2 * math.pi) ** 3 * (2 * al / math.pi) ** 1.5 / vol)
        f = torch.exp(-al * self.q2) * torch.exp(-1j * (pos @ q.t()))
        cp = cs * math.sqrt(4 * al)
        self.beta = torch.stack([cs * f] + [cp * q[:, i] * f for i in range(3)], 1).reshape(4 * natom, -1)
        self.vol = vol

    def grid(self, x):
        N = self.N
        g = torch.zeros(x.shape[0], N ** 3, dtype=torch.complex128, device=DEV)
        g[:, self.off] = x
        return torch.fft.ifftn(g.view(-1, N, N, N), dim=(1, 2, 3)) * N ** 3

    def apply(self, psi):
        out = torch.empty(psi.shape, dtype=torch.complex128, device=DEV)
        for i in range(0, psi.shape[0], 32):
            x = psi[i:i + 32].to(torch.complex128)
            v = torch.fft.fftn(self.grid(x) * self.V, dim=(1, 2, 3)).reshape(x.shape[0], -1)[:, self.off] / self.N ** 3
            c = x @ self.beta.mH
            out[i:i + 32] = self.T * x + v + (c * self.D) @ self.beta
        return out

    def density(self, psi, occ):
        rho = torch.zeros(self.N, self.N, self.N, dtype=torch.float64, device=DEV)
        for i in range(0, psi.shape[0], 32):
            g = self.grid(psi[i:i + 32].to(torch.complex128))
            w = torch.as_tensor(occ[i:i + 32], device=DEV) / self.vol
            rho += torch.einsum("n,nzyx->zyx", w, g.real ** 2 + g.imag ** 2)
        return rho

    def matrix(self):
        return self.apply(torch.eye(len(self.m), dtype=torch.complex128, device=DEV)).t()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("apply", "cheb", "gamma", "density"):
        d = Dense(case["a"], case["ecut"], case["natom"], case["box"], KPTS[case["k"]], seed)
        psi = _block(d.q2, case["nb"], seed, _type(case), kind == "gamma")
        if kind == "density":
            return d.density(psi, np.where(np.arange(case["nb"]) < (case["nb"] * 9) // 10, 2.0, 0.7))
        h = d.apply(psi)
        if kind == "cheb":
            h = CHEB[0] * h + CHEB[1] * psi.to(torch.complex128)
            h += CHEB[2] * _block(d.q2, case["nb"], seed + 1, _type(case)).to(torch.complex128)
        return h
    if kind == "products":
        st = prepare(case, seed)
        return {"gram": (st["y"].conj() @ st["y"].t()).t(), "rotated": st["q"] @ st["y"]}
    if kind == "eigen":
        a, b = (x.t() for x in _pencil(case, seed))
        c = torch.linalg.cholesky(b)
        t = torch.linalg.solve_triangular(c, a, upper=False)
        t = torch.linalg.solve_triangular(c, t.mH, upper=False)
        if case["real"]:
            w, z = torch.linalg.eigh(((t + t.mH) * 0.5).real)
            z = z.to(torch.complex128)
        else:
            w, z = torch.linalg.eigh((t + t.mH) * 0.5)
        x = torch.linalg.solve_triangular(c.mH, z, upper=True)
        return {"values": w, "vectors": _fix_gauge(x.t().contiguous())}
    if kind == "solve":
        d = Dense(case["a"], case["ecut"], case["natom"], case["box"], KPTS[case["k"]], seed)
        w, z = torch.linalg.eigh(d.matrix())
        n = case["nband"]
        return {"values": w[:n], "rho": d.density(z[:, :n].t(), np.full(n, 2.0))}
    out, made = [], {}
    for a, ecut, natom, kpts, ik in _batch_units(case):
        made.setdefault((a, ecut), seed + len(made))
        d = Dense(a, ecut, natom, 0, kpts[ik], made[a, ecut], kpts)
        out.append(torch.linalg.eigvalsh(d.matrix())[:2 * natom] if len(d.m) <= 4000 else None)
    return out if any(v is not None for v in out) else None


# ------------------------------------------------------------------------------------------------

def _apply_work(a, ecut, natom, box, k, nb, size, blocks):
    """Bytes: the band blocks and V and the projector table once.  Operations: the transforms of
    the pencils that can hold data, there and back, and the two projector products."""
    npw = a ** 3 * (2 * ecut) ** 1.5 / (6 * math.pi ** 2)
    N = box or K.kss_default_box(np.eye(3) * a, ecut, [KPTS[k]])[0]
    w = 2 * a * math.sqrt(2 * ecut) / (2 * math.pi) + 1
    pencils = math.pi / 4 * w * w + w * N + N * N
    fft = 2 * pencils * 5 * N * math.log2(N)
    return (blocks * nb * npw * size + N ** 3 * size / 2 + 4 * natom * npw * size,
            nb * (fft + 2 * 8 * 4 * natom * npw))


def work(case):
    kind = case["kind"]
    size = 16 if case.get("prec", "fp64") == "fp64" else 8
    if kind in ("apply", "cheb", "gamma"):
        b, f = _apply_work(case["a"], case["ecut"], case["natom"], case["box"], case["k"], case["nb"], size,
                           3 if kind == "cheb" else 2)
        return {"bytes": b, "flops": f / (2 if kind == "gamma" else 1)}
    if kind == "density":
        b, f = _apply_work(case["a"], case["ecut"], 0, case["box"], case["k"], case["nb"], size, 1)
        return {"bytes": b, "flops": f / 2}
    if kind == "products":
        nb, npw = case["nb"], case["npw"]
        return {"bytes": 16 * (2 * nb * npw + 2 * nb * nb), "flops": 2 * 8 * nb * nb * npw}
    if kind == "eigen":
        n = case["n"]
        return {"bytes": 3 * 16 * n * n, "flops": (1 if case["real"] else 4) * 8 * n ** 3}
    if kind == "solve":  # at least two filters of degree ten
        b, f = _apply_work(case["a"], case["ecut"], case["natom"], case["box"], case["k"], case["nband"], 16, 2)
        return {"bytes": 22 * b, "flops": 22 * f}
    b = f = 0.0
    for a, ecut, natom, kpts, ik in _batch_units(case):
        x, y = _apply_work(a, ecut, natom, 0, 1, 2 * natom, 8, 2)
        b, f = b + 42 * x, f + 42 * y
    return {"bytes": b, "flops": f}
