"""Solves and coupling matrices in units in which the spacing is far from one: |d|^2 and a + b|d|^2 are
numbers of any size, and so is their product, but the solution is the unit one, scaled."""
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


# spacing, and the factor of a and b h^2
UNITS = [(1e-100, 1e120), (1e100, 1e-120), (1e-10, 1e18), (3.0, 0.2)]


@pytest.mark.parametrize("grid", [(16, 12, 9), (32, 32, 32), (48, 16, 128)])
@pytest.mark.parametrize("h,factor", UNITS)
@pytest.mark.parametrize("ab", [(1.7, 0.4), (0.0, 0.6)])
def test_solve_in_any_units(icm, grid, h, factor, ab):
    nx, ny, nz = grid
    sim = icm.Simulation(grid, h, 1.0, 1.0, 0.0, 1.0, 3, 1, 64)
    r = np.random.default_rng(nx + nz).standard_normal((3, nz, ny, nx))
    got = icm.icm_op_spectral_solve(sim.handle, ab[0] * factor, ab[1] * factor * h * h, r.ravel()) * factor
    assert rel(got, oracle.spectral_solve(r, ab[0], ab[1], 1.0)) < TOL[64]
    sim.close()


@pytest.mark.parametrize("h,factor", [(1e-60, 1e200), (1e60, 1e-200), (3.0, 0.2)])
@pytest.mark.parametrize("ab", [(1.7, 0.4), (0.0, 0.6)])
def test_coupling_in_any_units(icm, h, factor, ab):
    grid = (16, 12, 9)
    sim = icm.Simulation(grid, h, 1.0, 1.0, 0.0, 1.0, 3, 1, 64)
    q = np.random.default_rng(5).uniform(0, 1, size=(2, 1, 3)) * grid
    got = icm.icm_op_coupling(sim.handle, q[0] * h, q[1] * h, ab[0] * factor, ab[1] * factor * h * h)
    want = oracle.coupling_matrix(q[0, 0], q[1, 0], grid, 3, 1.0, *ab)
    assert rel(got[0] * factor * h ** 3, want) < 10 * TOL[64]   # q h / h is rounded: stencils move by an ulp of 16
    sim.close()
