"""Spectra whose rows are one wave number longer than whole tiles: the last wave number of
several rows (z pass) or planes (y pass) shares a tile.  Row and plane counts that do and do
not fill the last such tile, fewer rows than one tile takes, every z kernel (tensor copies, plain, any
side) and sides whose rows do not fold, against the oracle."""
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


GRIDS = [(16, 6, 32), (32, 6, 64), (64, 27, 48), (128, 36, 32), (48, 9, 96), (18, 12, 32), (384, 32, 18), (48, 384, 9),
         (96, 512, 6), (512, 48, 32), (256, 192, 27), (384, 96, 12), (64, 64, 64), (36, 64, 128)]


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("tma", [1, 0])
def test_solve_with_folded_last_column(icm, precision, grid, tma):
    nx, ny, nz = grid
    sim = icm.Simulation(grid, 0.8, 1.3, 0.7, 0.0, 0.05, 3, 1, precision)
    icm.icm_set_plan(sim.handle, tma_z=tma)
    r = np.random.default_rng(nx + 2 * ny + nz).standard_normal((3, nz, ny, nx))
    got = icm.icm_op_spectral_solve(sim.handle, 1.7, 0.4, r.ravel())
    assert rel(got, oracle.spectral_solve(r, 1.7, 0.4, 0.8)) < TOL[precision] / 2
    sim.close()
