"""Parity of the CUDA 3D-Fourier forms (through the C-ABI) with the FP64 oracle: Eq. 12
(CT step, then the 3D CTF inversion, rerun for a second sigma) and the Fourier-gridding
UTR (with and without the NSR noise filter).  Float32 tolerance 1e-5 relative L2, except
where the noise filter decides per coefficient whether to keep it: those decisions are
taken in float32 on the GPU and in float64 by the oracle, so coefficients at the
threshold may go either way (1e-3 there)."""
import math

import numpy as np
import pytest
import torch

import oracle as O
from oracle import fourier as F
from paper_2206_09151_gb300 import phantoms as ph

pytestmark = pytest.mark.gpu

TOL_F32 = 1e-5


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.fail("the gpu tests need a CUDA device")
    from paper_2206_09151_gb300.build import build
    build()


def rel_l2(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _scan(grid, nu, nv, D, span, lam, R, photons=None, cone=False, seed=8):
    phan = ph.blob_phantom(grid, 12, seed=seed, s_vox=1.5, amp_unit=2e-6)
    rot = ph.cone_rotations(D, 60.0, seed=seed) if cone else ph.single_axis_rotations(D, span=span)
    Rs = np.full(D, R) if np.isscalar(R) else np.asarray(R)
    img = ph.multislice_images(phan, rot, nu, nv, 1e-9, lam, Rs, 0.3, n_slabs=16, photons=photons, seed=3).numpy()
    return img, rot, Rs


@pytest.mark.parametrize("grid,nu,nv", [((32, 32, 32), 32, 32), ((24, 20, 12), 30, 22)])
def test_swapped_order_matches_oracle_and_reruns_for_another_sigma(grid, nu, nv):
    from paper_2206_09151_gb300.recon import Reconstructor
    D, lam, R = 60, 4e-10, 20e-9
    img, rot, Rs = _scan(grid, nu, nv, D, 2 * math.pi, lam, R)
    r = Reconstructor(rot, nu, nv, grid, lam=lam, delta=1e-9, defocus=Rs, nz_layers=8, sigma=0.3, eps=1e-2,
                      filter="pair")
    ws = r.swap_ct(torch.from_numpy(img).cuda())
    vc, vs = F.swap_ct(img, rot, lam=lam, delta=1e-9, defocus=Rs, nz_layers=8, grid=grid)
    for sig, eps in ((0.3, 1e-2), (0.05, 0.1)):
        got = r.swap_phase(ws, sig, eps).cpu().numpy()
        ref = F.swap_phase(vc, vs, lam=lam, delta=1e-9, defocus=R, sigma=sig, eps=eps)
        assert rel_l2(got, ref) <= TOL_F32, (sig, rel_l2(got, ref))
    r.close()


@pytest.mark.parametrize("grid,nu,nv,cone", [((32, 32, 32), 32, 32, False), ((24, 20, 12), 30, 22, True)])
def test_gridding_matches_oracle(grid, nu, nv, cone):
    from paper_2206_09151_gb300.recon import Reconstructor
    D, lam = 60, 4e-10
    Rs = np.random.default_rng(4).uniform(15e-9, 25e-9, D)
    img, rot, Rs = _scan(grid, nu, nv, D, 2 * math.pi, lam, Rs, cone=cone)
    r = Reconstructor(rot, nu, nv, grid, lam=lam, delta=1e-9, defocus=Rs, nz_layers=4, sigma=0.3, eps=1e-2,
                      ramp="density" if cone else "single_axis")
    got = r.grid_run(torch.from_numpy(img).cuda()).cpu().numpy()
    r.close()
    ref = F.recon_gridding(img, rot, lam=lam, delta=1e-9, defocus=Rs, grid=grid, sigma=0.3, eps=1e-2)
    assert rel_l2(got, ref) <= TOL_F32, rel_l2(got, ref)


def test_gridding_noise_filter_matches_oracle():
    from paper_2206_09151_gb300.recon import Reconstructor
    grid, D, lam = (32, 32, 32), 60, 1e-10
    img, rot, Rs = _scan(grid, 32, 32, D, 2 * math.pi, lam, 30e-9, photons=1e4)
    r = Reconstructor(rot, 32, 32, grid, lam=lam, delta=1e-9, defocus=Rs, nz_layers=4, sigma=0.3, eps=1e-2)
    got = r.grid_run(torch.from_numpy(img).cuda(), nsr=1e-2).cpu().numpy()
    r.close()
    ref = F.recon_gridding(img, rot, lam=lam, delta=1e-9, defocus=Rs, grid=grid, sigma=0.3, eps=1e-2, nsr=1e-2)
    assert rel_l2(got, ref) <= 1e-3, rel_l2(got, ref)


@pytest.mark.parametrize("grid", [(1, 5, 9), (17, 3, 33), (300, 2, 3), (2, 3, 520)])
def test_line_transforms_of_every_length_match_oracle(grid):
    """Grid sides whose padded lengths run from 2 to 2048 (a thread per line, the 8-value and
    the 16-value transform), odd sides (a last unpaired line of the complex-to-real pass) and
    sides that leave part of a thread block without lines.  Both forms, the gridding on the
    grids whose cells are near the images' bins."""
    from paper_2206_09151_gb300.recon import Reconstructor
    nu, nv, D, lam = 21, 18, 7, 4e-10
    rng = np.random.default_rng(5)
    img = (1.0 + 0.05 * rng.standard_normal((D, nv, nu))).astype(np.float32)
    Rs = np.full(D, 20e-9)
    kw = dict(lam=lam, delta=1e-9, defocus=Rs, nz_layers=3)
    rot = ph.single_axis_rotations(D, span=2 * math.pi, start=0.1)
    r = Reconstructor(rot, nu, nv, grid, sigma=0.3, eps=1e-2, filter="pair", **kw)
    got = r.swap_phase(r.swap_ct(torch.from_numpy(img).cuda()), 0.3, 1e-2).cpu().numpy()
    r.close()
    vc, vs = F.swap_ct(img, rot, grid=grid, **kw)
    ref = F.swap_phase(vc, vs, lam=lam, delta=1e-9, defocus=20e-9, sigma=0.3, eps=1e-2)
    assert rel_l2(got, ref) <= TOL_F32, rel_l2(got, ref)
    if max(grid) > 64:
        # a 64-bin image spectrum stretched over 1024 or 2048 cells: the float32 coordinates of the
        # splat (up to 1000 cells, 6e-5 cell of rounding) are further off than the transforms
        return
    rot = ph.cone_rotations(D, 60.0, seed=3)
    r = Reconstructor(rot, nu, nv, grid, sigma=0.3, eps=1e-2, ramp="density", **kw)
    got = r.grid_run(torch.from_numpy(img).cuda()).cpu().numpy()
    r.close()
    ref = F.recon_gridding(img, rot, lam=lam, delta=1e-9, defocus=Rs, grid=grid, sigma=0.3, eps=1e-2)
    assert rel_l2(got, ref) <= TOL_F32, rel_l2(got, ref)


@pytest.mark.parametrize("side,n,D", [(24, 24, 150), (12, 48, 60)])
def test_noise_filter_decides_alike_in_whatever_order_its_sums_are_added(side, n, D):
    """The noise filter keeps or drops whole cells, so a cell next to the threshold must not hang on the
    order of the float atomics that sum it.  Steps of the volume over nsr, one cell pair each, are bisected down to
    neighbouring float32 thresholds; there and a few steps around, every call gives one and the same volume.  Also a volume much smaller than the images,
    whose cells take thousands of samples each."""
    from paper_2206_09151_gb300.recon import Reconstructor
    rng = np.random.default_rng(7)
    img = torch.from_numpy((1.0 + 0.1 * rng.standard_normal((D, n, n))).astype(np.float32)).cuda()
    r = Reconstructor(ph.cone_rotations(D, 60.0, seed=3), n, n, (side, side, side), lam=4e-10, delta=1e-9,
                      defocus=rng.uniform(10e-9, 20e-9, D), nz_layers=2, sigma=0.3, eps=1e-2, ramp="density")

    def vol(bits):  # at the float32 threshold nsr sqrt(nu nv) with these bits
        return r.grid_run(img, float(np.int32(bits).view(np.float32)) / n)

    def same(a, b):
        return float((a - b).norm()) <= 1e-5 * float(b.norm())

    for t in (0.3, 0.8, 1.5, 2.5, 4.0) if side == n else (1.0, 2.0, 4.0):
        lo, hi = (int(np.float32(x).view(np.int32)) for x in (t, t * (1.05 if side == n else 1.5)))
        vlo = vol(lo)
        assert not same(vlo, vol(hi))
        while hi - lo > 1:
            mid = (lo + hi) // 2
            if same(vol(mid), vlo):
                lo = mid
            else:
                hi = mid
        for bits in range(lo - 2, hi + 3):
            first = vol(bits)
            assert all(same(vol(bits), first) for _ in range(15)), (t, bits - lo)
    r.close()


def test_gridding_with_a_noise_ratio_below_float32_is_the_one_without_the_filter():
    from paper_2206_09151_gb300.recon import Reconstructor
    grid, D = (20, 24, 16), 12
    img, rot, Rs = _scan(grid, 24, 24, D, 2 * math.pi, 4e-10, 20e-9)
    r = Reconstructor(rot, 24, 24, grid, lam=4e-10, delta=1e-9, defocus=Rs, nz_layers=4, sigma=0.3, eps=1e-2)
    im = torch.from_numpy(img).cuda()
    ref, got = (r.grid_run(im, nsr).cpu().numpy() for nsr in (0.0, 1e-50))
    r.close()
    assert rel_l2(got, ref) <= TOL_F32, rel_l2(got, ref)


@pytest.mark.parametrize("grid,n", [((300, 2, 3), 300), ((3, 270, 2), 270), ((2, 3, 511), 511), ((520, 2, 1), 520),
                                    ((1, 600, 2), 600), ((2, 1, 700), 700)])
def test_gridding_on_long_axes_matches_oracle(grid, n):
    """Padded sides of 1024 and 2048 along each axis in turn, with images of that length.  The splat forms its coordinates
    (up to P3 / 2 cells) in three float32 roundings, d = 1.5 2^-24 P3 / 2 cells off at most; a weight changes by d per
    axis and a cell by its difference from its neighbours, so the volume is within 2 sqrt(3) d."""
    from paper_2206_09151_gb300.recon import Reconstructor
    rng = np.random.default_rng(n)
    D, lam = 2, 1e-10
    nu, nv = (n, 24) if grid[1] < n else (24, n)
    img = (1.0 + 0.05 * rng.standard_normal((D, nv, nu))).astype(np.float32)
    rot, Rs = ph.single_axis_rotations(D, start=0.2), rng.uniform(15e-9, 25e-9, D)
    r = Reconstructor(rot, nu, nv, grid, lam=lam, delta=1e-9, defocus=Rs, nz_layers=2, sigma=0.3, eps=1e-2)
    got = r.grid_run(torch.from_numpy(img).cuda()).cpu().numpy()
    r.close()
    ref = F.recon_gridding(img, rot, lam=lam, delta=1e-9, defocus=Rs, grid=grid, sigma=0.3, eps=1e-2)
    P3 = 2 << (max(grid) - 1).bit_length()
    assert rel_l2(got, ref) <= 2 * math.sqrt(3) * 1.5 * 2.0 ** -24 * P3 / 2, rel_l2(got, ref)
