"""GPU: grids at the edges of the kernels' size rules (tiles, chunks, remainders), against the oracle."""
import os

import numpy as np
import pytest

from paper_2211_16718_gb300 import inputs as I
from tests._util import flux_scale, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ns3d():
    from paper_2211_16718_gb300 import build as B
    B.build()
    from paper_2211_16718_gb300 import ns3d as N
    N.lib()
    return N


@pytest.fixture(scope="module")
def orc(oracle):
    oracle.set_threads(os.cpu_count() or 1)
    return oracle


def _gpu(u):
    import torch
    return torch.from_numpy(np.ascontiguousarray(u)).cuda()


# more x-y tiles than resident blocks; a last z-chunk shorter than the others; one block
@pytest.mark.parametrize("nx,ny,nz", [(640, 256, 3), (70, 33, 129), (32, 8, 1)])
@pytest.mark.parametrize("prec", [0, 2])
def test_stats_chunks(ns3d, orc, nx, ny, nz, prec):
    u = I.random_smooth(nx, ny, nz, seed=3, amp=0.1, mach=0.4)
    so = orc.stats(orc.Params(nx, ny, nz), u)
    s = ns3d.Solver(nx, ny, nz, precision=prec)
    sg = s.stats(_gpu(u))
    s.close()
    for k, v in so.items():  # sums of n terms: the tolerance of the statistics tests
        assert abs(sg[k] - v) <= 1e-12 * (so["mass"] if k.startswith("mom") else abs(v)), k


def test_stats_minima_of_bad_states(ns3d):
    """Minima over a state with a negative pressure and a NaN: the NaN is ignored, the status set."""
    u = I.random_smooth(20, 9, 6, seed=4)
    u[4, 1, 2, 3] = -1.0
    u[0, 3, 4, 5] = np.nan
    rho = u[0]
    p = 0.4 * (u[4] - 0.5 * (u[1] ** 2 + u[2] ** 2 + u[3] ** 2) / rho)
    s = ns3d.Solver(20, 9, 6)
    sg = s.stats(_gpu(u))
    s.close()
    assert sg["status"] == ns3d.NS3D_ENONPHYSICAL
    assert sg["rho_min"] == np.nanmin(rho)
    assert sg["p_min"] == pytest.approx(np.nanmin(p), rel=1e-14)


# one-plane chunks, a shorter last chunk, more x-y tiles than resident blocks, one plane of points
@pytest.mark.parametrize("nx,ny,nz", [(33, 9, 70), (21, 40, 131), (640, 256, 3), (40, 24, 1)])
def test_viscous_chunks(ns3d, orc, nx, ny, nz):
    u = I.random_smooth(nx, ny, nz, seed=6, amp=0.1, mach=0.4)
    ref = orc.rhs(orc.Params(nx, ny, nz, mu_eff=1e-4), u)
    out = []
    for storage in (1, 2):
        s = ns3d.Solver(nx, ny, nz, mu_eff=1e-4, storage=storage)
        out.append(s.rhs(_gpu(u)).cpu().numpy())
        s.close()
    # mu is small because the composite second difference amplifies the double-float rounding of the
    # temperature (a few 2^-48) by (18/12)^2 / dx^2, times kappa = mu / (0.4 * 0.72): at 640 points and
    # mu = 1e-4 that is 3.5e-4 * 4 * 3.6e-15 * 2.25 * 1.04e4 = 1.2e-13, below the 1e-12 of a right-hand
    # side (max |R| is 2)
    assert rel_err(out[0], ref) <= 1e-12
    assert np.array_equal(out[0], out[1])
    s = ns3d.Solver(nx, ny, nz, mu_eff=1e-4, precision=1)
    r32 = s.rhs(_gpu(u)).cpu().numpy()
    s.close()
    # FP32 fluxes: 1e-5 of the flux scale over the smallest spacing (as the FP32-bulk tests)
    assert np.abs(r32 - ref).max() <= 1e-5 * flux_scale(u, (2 * np.pi,) * 3)


# lines shorter than a tile, one point over one and two tiles, one-point lines, lengths that are no
# multiple of 4 (x tiles start on 32-byte sectors), wide remainders; every tile shape, both FP64 modes
@pytest.mark.parametrize("nx,ny,nz", [(25, 49, 33), (32, 23, 7), (1, 26, 5), (47, 3, 64), (73, 17, 25), (2, 41, 97)])
def test_balanced_tiles(ns3d, orc, nx, ny, nz):
    u = I.random_smooth(nx, ny, nz, seed=7, amp=0.1, mach=0.5)
    ref = orc.rhs(orc.Params(nx, ny, nz, mu_eff=0.003), u)
    for prec, variants in ((0, (0, 1, 2)), (2, (0,))):
        out = []
        for v in variants:
            s = ns3d.Solver(nx, ny, nz, mu_eff=0.003, precision=prec)
            ns3d.set_solver_variant(s, v)
            out.append(s.rhs(_gpu(u)).cpu().numpy())
            s.close()
            assert rel_err(out[-1], ref) <= 1e-12, (prec, v)
            assert np.array_equal(out[0], out[-1]), (prec, v)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nx", [24, 26, 27])
def test_step_of_a_state_on_8_byte_boundaries(ns3d, nx, prec):
    """The z pass takes 16-byte copies only where U_n allows it: the same bits either way."""
    import torch
    u = _gpu(I.random_smooth(nx, 10, 30, seed=8, amp=0.1, mach=0.4))
    buf = torch.empty(u.numel() + 1, dtype=torch.float64, device="cuda")
    v = buf[1:].view(u.shape)
    v.copy_(u)
    assert v.data_ptr() % 16 == 8
    s = ns3d.Solver(nx, 10, 30, mu_eff=0.003, precision=prec)
    s.rk_step(u, 0.01, 2)
    s.rk_step(v, 0.01, 2)
    s.check()
    s.close()
    assert torch.equal(u, v)


# one tile, one point over one and two tiles, x lengths that are no multiple of 4, one-point lines;
# against the all-FP64 adjoint kernels, which have their own tiles and algebra (both pinned to the
# oracle's dense adjoint elsewhere): the tolerance of that comparison
@pytest.mark.parametrize("nx,ny,nz", [(32, 33, 5), (65, 3, 31), (2, 66, 35), (39, 7, 64), (1, 9, 34)])
def test_adjoint_tiles(ns3d, nx, ny, nz):
    u = _gpu(I.random_smooth(nx, ny, nz, seed=9, amp=0.1, mach=0.5))
    lam = _gpu(np.random.default_rng(5).normal(size=(5, nz, ny, nx)))
    out = []
    for prec in (0, 2):
        s = ns3d.Solver(nx, ny, nz, mu_eff=0.003, precision=prec)
        out.append(s.rhs_vjp(u, lam).cpu().numpy())
        s.check()
        s.close()
    assert rel_err(out[0], out[1]) <= 1e-11


@pytest.mark.parametrize("prec,rk", [(0, 0), (0, 1), (2, 0)])
@pytest.mark.parametrize("nx,ny,nz", [(25, 30, 9), (64, 5, 1), (33, 26, 50)])
def test_merged_xy_passes_give_the_same_bits(ns3d, prec, rk, nx, ny, nz):
    """The x and y passes in one launch (small grids) against separate launches: contexts whose
    kernels are timed, and lean storage, launch them apart."""
    import torch
    u = _gpu(I.random_smooth(nx, ny, nz, seed=10, amp=0.1, mach=0.5))
    out = []
    for timed, storage in ((False, 1), (True, 1), (False, 2)):
        s = ns3d.Solver(nx, ny, nz, mu_eff=0.003, precision=prec, rk=rk, storage=storage)
        s.timing_enable(timed)
        v = u.clone()
        s.rk_step(v, 0.01, 2)
        out.append((s.rhs(u), v))
        s.close()
    for r, v in out[1:]:
        assert torch.equal(r, out[0][0]) and torch.equal(v, out[0][1])


# FP32-bulk tiles: lines of one and two tiles, lengths whose last segment of four interfaces is partial
@pytest.mark.parametrize("nx,ny,nz", [(27, 26, 28), (53, 29, 3), (1, 55, 27), (30, 2, 79)])
def test_balanced_tiles_fp32_bulk(ns3d, orc, nx, ny, nz):
    u = I.random_smooth(nx, ny, nz, seed=11, amp=0.1, mach=0.5)
    ref = orc.rhs(orc.Params(nx, ny, nz, mu_eff=0.003), u)
    s = ns3d.Solver(nx, ny, nz, mu_eff=0.003, precision=1)
    r = s.rhs(_gpu(u)).cpu().numpy()
    s.check()
    s.close()
    # FP32 fluxes: 1e-5 of the flux scale over the smallest spacing (as the FP32-bulk tests)
    assert np.abs(r - ref).max() <= 1e-5 * flux_scale(u, (2 * np.pi,) * 3)


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_adjoint_of_jumps_between_tiles(ns3d, axis):
    """A shock tube whose jumps lie between the adjoint's tiles (along x 24, 24 and 17 points of 65,
    else 22, 22 and 21), and one with them inside; as test_adjoint_tiles."""
    shp = [5, 4, 6]
    shp[axis] = 65
    lam = _gpu(np.random.default_rng(6).normal(size=[5] + shp))
    for lo, hi in ((24, 48) if axis == 2 else (22, 44), (10, 33)):
        left = np.ones(65, dtype=bool)
        left[lo:hi] = False
        left = left[tuple(slice(None) if k == axis else None for k in range(3))]
        wave = 1.0 + 0.02 * np.random.default_rng(7).uniform(-1.0, 1.0, shp)
        vel = [0.1 * (m + 1) * (wave - 1.0) for m in range(3)]
        u = _gpu(I.to_conserved(np.where(left, 1.0, 0.125) * wave, *vel, np.where(left, 1.0, 0.1) * wave / 1.4))
        out = []
        for prec in (0, 2):
            s = ns3d.Solver(*shp[::-1], mu_eff=0.003, precision=prec)
            out.append(s.rhs_vjp(u, lam).cpu().numpy())
            s.check()
            s.close()
        assert rel_err(out[0], out[1]) <= 1e-11
