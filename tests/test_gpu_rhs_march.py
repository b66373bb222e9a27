"""The marching right-hand side (FP32 above 2^20 cells, and below where there are normals that do not fit in the
scratch): persistent blocks and fixed marches with remainders and odd first planes, tiles wider than
the short sides (several periodic wraps), ragged tiles, an odd number of planes, with and without noise,
history and advection, against the oracle, and bit for bit between the launch shapes."""
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


# more than 2^20 cells march with and without noise; the smaller grids with noise only
CASES = [((8, 384, 384), kT) for kT in (1e-3, 0.0)] + [((24, 216, 243), kT) for kT in (1e-3, 0.0)] + \
        [((486, 54, 48), kT) for kT in (1e-3, 0.0)] + [((27, 9, 27), 1e-3), ((48, 16, 9), 1e-3), ((96, 6, 81), 1e-3)]


@pytest.mark.parametrize("grid,kT", CASES)
@pytest.mark.parametrize("hist,advection", [(True, True), (False, False)])
def test_every_march_gives_the_same_right_hand_side(icm, grid, kT, hist, advection):
    prm = oracle.Params(grid, h=0.9, rho=1.2, eta=0.7, kT=kT, dt=0.04, kernel=3, seed=(5 << 33) + 17, advection=advection)
    nx, ny, nz = grid
    rng = np.random.default_rng(nx + ny + nz)
    v = 0.1 * rng.standard_normal((3, nz, ny, nx))
    prev = 0.1 * rng.standard_normal((3, nz, ny, nx)) if hist else None
    want_r, want_a = oracle.explicit_rhs(v, prev, 5, prm)
    sim = icm.Simulation(grid, prm.h, prm.rho, prm.eta, kT, prm.dt, 3, prm.seed, 32, 0 if advection else 0x1)
    first = None
    for kz in (None, 0, 4, 7, 16):                 # the default march, then these
        if kz is not None:
            icm.icm_set_plan(sim.handle, rhs_kz=kz)
        r, a = icm.icm_op_explicit_rhs(sim.handle, v.ravel(), None if prev is None else prev.ravel(), 5)
        assert rel(r, want_r) < TOL[32] and rel(a, want_a) < TOL[32], kz
        if first is None:
            first = (r, a)
        assert np.array_equal(r, first[0]) and np.array_equal(a, first[1]), kz
    sim.close()
