"""The fixed-point double-precision local part through the C ABI, where block exponents can go wrong.

* Bands of one call at scales from 1e-150 to 1e150, a zero band, a single plane wave and a band
  concentrated at one point: each band has exponents of its own, so each is as accurate as alone
  (1e-14 of its own |H psi|: a few roundings of 2^-53 each in the oracle's FP64 sums of at most
  1e4 terms and in the library).
* A band with a NaN or an infinity gives NaN and leaves the others bit for bit as they are.
* Gamma pairs of very different norms: the smaller band's error is relative to the pair (as in the
  transform of the sum), 1e-14 of the pair's |H psi|.
* Boxes whose y/z split runs pruned and full, odd edges among them.
"""
import numpy as np
import pytest

import oracle as O
import workloads as W
import paper_2507_08578_gb300.kss as K
from tests.kss_helpers import ensure_built, make_ctx, setup

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    ensure_built()
    c = make_ctx()
    yield c
    torch.cuda.synchronize()
    K.kss_destroy(c)


def _apply(sysh, c, gamma=False):
    import torch
    psi = torch.from_numpy(c).cuda()
    out = torch.empty_like(psi)
    (K.kss_apply_H_gamma if gamma else K.kss_apply_H)(sysh, 0, psi, out, K.KSS_PREC_FP64)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("box,a,ecut,kpt", [
    ((24, 24, 24), 10.0, 10.0, 0), ((25, 25, 25), 8.0, 10.0, 1), ((27, 30, 30), 8.0, 8.0, 1),
    ((54, 54, 54), 13.9, 17.3, 1), ((96, 96, 96), 9.0, 9.0, 1), ((45, 48, 48), 10.0, 16.0, 0)])
def test_scales_and_special_bands(ctx, box, a, ecut, kpt):
    s = W.make_system("fx", a, ecut, 3, 4, seed=17, kpts=[[0.25 * kpt] * 3], fft_box=box, nproj_per_atom=0)
    sysh = setup(ctx, s)
    try:
        p = O.build_problem(s, 0, box=box)
        npw = p.basis.npw
        c = W.random_block(npw, 9, seed=5)
        c[1] *= 1e-150
        c[2] *= 1e150
        c[3] = 0
        c[4] = 0
        c[4, npw // 3] = 1
        c[5] = 1.0 / np.sqrt(npw)
        c[6] *= 10.0 ** np.random.default_rng(1).uniform(-14, 0, npw)
        out = _apply(sysh, c)
        scale = np.array([1, 1e150, 1e-150, 1, 1, 1, 1, 1, 1])[:, None]
        ref = p.apply(c * scale)
        err = np.linalg.norm(out * scale - ref, axis=1)
        assert err[3] == 0
        nz = [i for i in range(9) if i != 3]
        assert np.all(err[nz] < 1e-14 * np.linalg.norm(ref[nz], axis=1)), err[nz] / np.linalg.norm(ref[nz], axis=1)
        bad = c.copy()
        bad[0, 3] = np.nan
        bad[7, npw - 1] = np.inf
        o2 = _apply(sysh, bad)
        assert np.all(np.isnan(o2[0])) and np.all(np.isnan(o2[7]))
        keep = [i for i in range(9) if i not in (0, 7)]
        assert np.array_equal(o2[keep], out[keep])
    finally:
        K.kss_sys_destroy(sysh)


def test_gamma_pairs_of_uneven_norm(ctx):
    s = W.make_system("fxg", 10.0, 10.0, 4, 4, seed=18, fft_box=(30, 30, 30), nproj_per_atom=0)
    sysh = setup(ctx, s)
    try:
        p = O.build_problem(s, 0, box=(30, 30, 30))
        c = W.random_block(p.basis.npw, 5, seed=6)
        c = c + c[:, ::-1].conj()  # the canonical order at Gamma is symmetric
        c[1] *= 1e-9
        c[2] *= 1e-6
        c[4] *= 1e120
        out = _apply(sysh, c, gamma=True)
        ref = np.concatenate([p.apply(c[:4]), 1e120 * p.apply(c[4:] * 1e-120)])
        err = np.linalg.norm((out - ref) / np.array([1, 1, 1, 1, 1e120])[:, None], axis=1)
        big = np.linalg.norm(ref / np.array([1, 1, 1, 1, 1e120])[:, None], axis=1)
        assert np.all(err[:2] < 1e-14 * big[:2].max())
        assert np.all(err[2:4] < 1e-14 * big[2:4].max())
        assert err[4] < 1e-14 * big[4]
    finally:
        K.kss_sys_destroy(sysh)


@pytest.mark.parametrize("box,a,ecut,kpt", [((24, 24, 24), 10.0, 10.0, 0), ((25, 25, 25), 8.0, 10.0, 1),
                                            ((45, 48, 48), 10.0, 16.0, 0), ((96, 96, 96), 9.0, 9.0, 1)])
def test_density_scales_and_special_bands(ctx, box, a, ecut, kpt):
    """Bands at scales whose squares leave single weights and densities in range: w |psi|^2 of each
    is of order one, so the sum is as accurate as in the oracle (1e-13 of its maximum: roundings of
    2^-53 of |psi| in sums of at most 1e4 terms, twice that in the square)."""
    import torch
    s = W.make_system("fx", a, ecut, 3, 4, seed=17, kpts=[[0.25 * kpt] * 3], fft_box=box, nproj_per_atom=0)
    sysh = setup(ctx, s)
    try:
        b = O.make_basis(s.lattice, s.ecut, s.kpts[0], box)
        _, vol = O.reciprocal_lattice(s.lattice)
        c = W.random_block(b.npw, 7, seed=5) / np.sqrt(b.npw)
        c[3] = 0
        c[4] = 0
        c[4, b.npw // 3] = 1  # one plane wave: a constant density
        c[5] = 1.0 / b.npw    # a peak at the origin
        w = np.array([1.0, 0.7, 1.3, 2.0, 1.0, 0.5, -0.25])
        scale = np.array([1, 1e-150, 1e150, 1, 1, 1, 1])

        def rho_of(c, w):
            rho = torch.zeros(tuple(reversed(box)), dtype=torch.float64, device="cuda")
            K.kss_density_accumulate(sysh, 0, torch.from_numpy(c).cuda(), w, rho)
            torch.cuda.synchronize()
            return rho.cpu().numpy()

        got = rho_of(c * scale[:, None], w / scale ** 2)
        ref = O.density(c, b, w, vol)
        assert np.max(np.abs(got - ref)) < 1e-13 * np.max(ref), np.max(np.abs(got - ref)) / np.max(ref)
        assert np.all(rho_of(c[3:4], w[3:4]) == 0)
        one = rho_of(c[4:5], w[4:5])
        assert np.max(np.abs(one - 1.0 / vol)) < 1e-14 / vol
        bad = c.copy()
        bad[6, 0] = np.inf
        assert np.all(np.isnan(rho_of(bad, w)))
    finally:
        K.kss_sys_destroy(sysh)


@pytest.mark.parametrize("box,a,ecut", [((24, 24, 24), 10.0, 10.0), ((30, 30, 30), 8.0, 10.0)])
def test_density_no_further_from_the_true_one_than_fp64_transforms(ctx, box, a, ecut):
    """Against the density in extended precision (at least 11 bits beyond double, from the sums
    themselves): closer than the one from FP64 FFTs, whose rounded factors act on every band alike, and
    within 2^-52 of it in the mean square: the blocks' values are off by a few 2^-56 of their rms, and the
    last operations round at most twice a band (four bands)."""
    import torch
    ld, cl = np.longdouble, np.clongdouble
    assert np.finfo(ld).nmant >= 63
    s = W.make_system("fd", a, ecut, 3, 4, seed=17, kpts=[[0.25] * 3], fft_box=box, nproj_per_atom=0)
    sysh = setup(ctx, s)
    try:
        b = O.make_basis(s.lattice, s.ecut, s.kpts[0], box)
        _, vol = O.reciprocal_lattice(s.lattice)
        m = np.asarray(b.miller) % np.array(box)
        w = np.array([2.0, 2.0, 0.7, 1.3])
        c = W.random_block(b.npw, 4, seed=5) / (1.0 + np.asarray(b.kinetic))
        c /= np.linalg.norm(c, axis=1)[:, None]
        rho = torch.zeros(tuple(reversed(box)), dtype=torch.float64, device="cuda")
        K.kss_density_accumulate(sysh, 0, torch.from_numpy(c).cuda(), w, rho)
        torch.cuda.synchronize()
        pi = ld("3.14159265358979323846264338327950288419716939937510")
        k = np.arange(box[0])
        t = (np.outer(k, k) % box[0]).astype(ld) * (2 * pi / box[0])
        F = np.cos(t) + 1j * np.sin(t)
        ref = np.zeros(rho.shape, ld)
        grid = np.zeros((4,) + rho.shape, complex)
        grid[:, m[:, 2], m[:, 1], m[:, 0]] = c
        for n in range(4):
            g = grid[n].astype(cl)
            g = np.einsum("zyx,xa->zya", g, F)
            g = np.einsum("zya,yb->zba", g, F)
            g = np.einsum("zba,zc->cba", g, F)
            ref += ld(w[n]) * (g.real ** 2 + g.imag ** 2) / ld(vol)
        r = np.fft.ifftn(grid, axes=(1, 2, 3)) * np.prod(box)
        fft = np.einsum("n,nzyx->zyx", w / vol, r.real ** 2 + r.imag ** 2)

        def err(x):
            return float(np.sqrt(np.sum((x.astype(ld) - ref) ** 2) / np.sum(ref ** 2)))

        got = err(rho.cpu().numpy())
        assert got < 2.0 ** -52
        assert got < err(fft)
    finally:
        K.kss_sys_destroy(sysh)
