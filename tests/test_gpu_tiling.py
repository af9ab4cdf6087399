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
    ref = orc.rhs(orc.Params(nx, ny, nz, mu_eff=0.02), u)
    out = []
    for storage in (1, 2):
        s = ns3d.Solver(nx, ny, nz, mu_eff=0.02, storage=storage)
        out.append(s.rhs(_gpu(u)).cpu().numpy())
        s.close()
    assert rel_err(out[0], ref) <= 1e-12  # the tolerance of one right-hand side
    assert np.array_equal(out[0], out[1])
    s = ns3d.Solver(nx, ny, nz, mu_eff=0.02, precision=1)
    r32 = s.rhs(_gpu(u)).cpu().numpy()
    s.close()
    # FP32 fluxes: 1e-5 of the flux scale over the smallest spacing (as the FP32-bulk tests)
    assert np.abs(r32 - ref).max() <= 1e-5 * flux_scale(u, (2 * np.pi,) * 3)
