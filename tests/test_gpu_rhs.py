"""The right-hand side in two passes (stored normals) where its indexing can go wrong: odd
numbers of planes (the last one has no partner in its Philox call), the smallest sides,
sides shorter than a block, and the FP32 grids on either side of the size above which the
marching kernel takes over."""
import numpy as np
import pytest

from oracle import icm as oracle

from _gpu_helpers import TOL, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def icm():
    import paper_1212_6427_gb300 as m
    from paper_1212_6427_gb300 import build
    build.build_library()
    return m


CASES = [((6, 6, 9), 64), ((6, 6, 9), 32), ((27, 8, 27), 64), ((27, 8, 27), 32), ((8, 162, 6), 64), ((8, 162, 6), 32),
         ((128, 128, 64), 32), ((128, 128, 72), 32),
         ((108, 144, 81), 32)]


@pytest.mark.parametrize("grid,precision", CASES)
@pytest.mark.parametrize("hist", [True, False])
def test_right_hand_side_at_the_edges(icm, grid, precision, hist):
    prm = oracle.Params(grid, h=0.9, rho=1.2, eta=0.7, kT=2e-3, dt=0.04, kernel=3, seed=(5 << 33) + 17)
    nx, ny, nz = grid
    rng = np.random.default_rng(nx + ny + nz)
    v = 0.1 * rng.standard_normal((3, nz, ny, nx))
    prev = 0.1 * rng.standard_normal((3, nz, ny, nx)) if hist else None
    sim = icm.Simulation(grid, prm.h, prm.rho, prm.eta, prm.kT, prm.dt, 3, prm.seed, precision)
    r, a = icm.icm_op_explicit_rhs(sim.handle, v.ravel(), None if prev is None else prev.ravel(), 5)
    want_r, want_a = oracle.explicit_rhs(v, prev, 5, prm)
    assert rel(r, want_r) < TOL[precision] and rel(a, want_a) < TOL[precision]
    sim.close()
