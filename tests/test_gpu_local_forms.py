"""Which form of the double-precision local passes runs, through the C ABI.

A box without fixed-point instances (an x edge outside their list, or uneven y and z edges) keeps the
CTA-wide passes in FP64.  The forms differ in the order of their roundings, so the schedule that runs
shows in the last bits: the tuned CTA-wide schedule and the per-warp form pinned in its place give the
same H psi to rounding (1e-13 of a row) and not bit for bit.
"""
import numpy as np
import pytest

import oracle as O
import workloads as W
import paper_2507_08578_gb300.kss as K
from tests.kss_helpers import ensure_built, make_ctx, rel_err_rows, setup

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    ensure_built()
    c = make_ctx()
    yield c
    torch.cuda.synchronize()
    K.kss_autotune_clear()
    K.kss_autotune_set(c, 1)
    K.kss_destroy(c)


def apply(sysh, c):
    import torch
    psi = torch.from_numpy(c).cuda()
    out = torch.empty_like(psi)
    K.kss_apply_H(sysh, 0, psi, out, K.KSS_PREC_FP64)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("box", [(64, 48, 48), (72, 60, 60), (32, 30, 30)])
def test_listed_schedule_runs_without_fixed_point(ctx, box):
    s = W.make_system("fl", 8.0, 10.0, 3, 4, seed=23, fft_box=box, nproj_per_atom=0)
    sysh = setup(ctx, s)
    try:
        p = O.build_problem(s, 0, box=box)
        c = W.random_block(p.basis.npw, 64, seed=8)
        K.kss_autotune_clear()
        K.kss_autotune_set(ctx, 1)
        tuned = apply(sysh, c)
        (e,) = K.kss_autotune_table()
        assert (e["N1"], e["N"]) == box[:2] and e["threads"] > 0
        assert rel_err_rows(tuned, p.apply(c)) < 1e-13
        for nt in (256, 384, 0):
            K.kss_autotune_put(e["device"], e["precision"], e["N1"], e["N"], e["W3"], e["A"], e["B"], nt)
            (listed,) = K.kss_autotune_table()
            assert listed["threads"] == nt
            out = apply(sysh, c)
            assert rel_err_rows(out, tuned) < 1e-13
            assert np.array_equal(out, tuned) == (nt != 0)  # the thread count changes no rounding
    finally:
        K.kss_sys_destroy(sysh)
        K.kss_autotune_clear()


@pytest.mark.parametrize("box", [(96, 48, 54), (96, 30, 36), (64, 48, 54)])
def test_uneven_boxes_match_oracle(ctx, box):
    """A CTA-wide x edge beside a y/z pair that has no CTA-wide form, and neither."""
    s = W.make_system("fl", 8.0, 10.0, 3, 4, seed=24, kpts=[[0.25, 0.25, -0.25]], fft_box=box)
    sysh = setup(ctx, s)
    try:
        p = O.build_problem(s, 0, box=box)
        c = W.random_block(p.basis.npw, 5, seed=9)
        assert rel_err_rows(apply(sysh, c), p.apply(c)) < 1e-13
    finally:
        K.kss_sys_destroy(sysh)
        K.kss_autotune_clear()


@pytest.mark.parametrize("box,a,ecut,natom,nb,nproj", [
    ((24, 24, 24), 10.0, 10.0, 4, 12, 0),      # every band in one chunk
    ((24, 24, 24), 10.0, 10.0, 4, 1700, 0),    # more bands than the scratch holds: several chunks
    ((36, 36, 36), 9.0, 8.0, 60, 8729, 4),     # room for one slab and not for its exponents
    ((64, 48, 48), 10.0, 10.0, 4, 12, 0)])     # CTA-wide passes in FP64
def test_noalloc_runs_the_same_passes(ctx, box, a, ecut, natom, nb, nproj):
    """The entry point that allocates nothing takes the passes of kss_apply_H however much of its
    scratch the band block leaves, so the local part agrees bit for bit (projector energies of zero
    where there are projectors: their products are summed in another order)."""
    import torch
    s = W.make_system("fn", a, ecut, natom, 4, seed=25, fft_box=box, nproj_per_atom=nproj)
    s.D = np.zeros_like(s.D)
    sysh = setup(ctx, s)
    try:
        K.kss_autotune_clear()
        K.kss_autotune_set(ctx, 1)
        npw = K.kss_sphere(sysh, 0).shape[0]
        g = torch.Generator(device="cuda").manual_seed(4)
        psi = torch.randn(nb, npw, dtype=torch.complex128, device="cuda", generator=g)
        ref, out = torch.empty_like(psi), torch.empty_like(psi)
        K.kss_apply_H(sysh, 0, psi, ref, K.KSS_PREC_FP64)
        K.kss_apply_H_noalloc(sysh, 0, psi, out, K.KSS_PREC_FP64)
        torch.cuda.synchronize()
        assert torch.equal(ref, out)
    finally:
        K.kss_sys_destroy(sysh)
        K.kss_autotune_clear()


@pytest.mark.parametrize("box", [(64, 48, 48), (96, 48, 54), (72, 30, 36)])
def test_gamma_pairs_without_fixed_point(ctx, box):
    """Real-space-real bands, two per transform, an odd one left over, in the FP64 forms: 1e-13 of the
    pair's |H psi|, as the transform is of the pair's sum."""
    import torch
    s = W.make_system("fg", 8.0, 10.0, 3, 4, seed=26, fft_box=box)
    sysh = setup(ctx, s)
    try:
        p = O.build_problem(s, 0, box=box)
        c = W.random_block(p.basis.npw, 7, seed=10)
        c = c + c[:, ::-1].conj()  # the canonical order at Gamma is symmetric
        psi = torch.from_numpy(c).cuda()
        out = torch.empty_like(psi)
        K.kss_apply_H_gamma(sysh, 0, psi, out, K.KSS_PREC_FP64)
        torch.cuda.synchronize()
        ref = p.apply(c)
        err = np.linalg.norm(out.cpu().numpy() - ref, axis=1)
        norm = np.linalg.norm(ref, axis=1)
        pair = np.maximum(norm, np.append(norm.reshape(-1)[:6].reshape(3, 2)[:, ::-1].reshape(-1), 0.0))
        assert np.all(err < 1e-13 * pair)
    finally:
        K.kss_sys_destroy(sysh)
        K.kss_autotune_clear()
