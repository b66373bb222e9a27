"""The coupling sums' split into segments of kx and columns of (ky, kz), against the oracle's transforms:
one and several segments, ragged last ones, more columns than threads, and every pair of a call
alike."""
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


@pytest.mark.parametrize("grid,pairs", [((32, 27, 16), 3), ((162, 8, 9), 3), ((36, 6, 6), 70), ((128, 81, 6), 2),
                                        ((192, 128, 128), 1), ((243, 128, 128), 1), ((6, 512, 486), 2)])
@pytest.mark.parametrize("ab", [(1.0, 0.5), (0.0, 0.6)])
def test_every_split_of_the_sum(icm, grid, pairs, ab):
    sim = icm.Simulation(grid, 0.9, 1.0, 0.6, 0.0, 0.05, 3, 1, 64, 0)
    L = np.array(grid) * 0.9
    q = np.random.default_rng(sum(grid)).uniform(0, 1, size=(2, pairs, 3)) * L
    got = icm.icm_op_coupling(sim.handle, q[0], q[1], *ab)
    for p in {0, pairs - 1}:
        want = oracle.coupling_matrix(q[0, p], q[1, p], grid, 3, 0.9, *ab)
        assert rel(got[p], want) < TOL[64]
        assert np.array_equal(icm.icm_op_coupling(sim.handle, q[0, p], q[1, p], *ab)[0], got[p])
    sim.close()
