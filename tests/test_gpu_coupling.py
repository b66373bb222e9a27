"""The coupling matrices as sums over wave vectors (icm_op_coupling) against the oracle's
transforms, where the sum's indexing can go wrong: odd and smallest sides, a Nyquist
plane on some axes and not on others, positions on the seams and outside the box, more
pairs than one chunk of the library's, and a spacing other than one."""
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


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("grid,kernel,h", [((6, 6, 6), 3, 1.0), ((9, 18, 8), 4, 0.8), ((27, 12, 9), 3, 1.3),
                                           ((54, 16, 32), 4, 1.0), ((8, 81, 27), 3, 0.7)])
@pytest.mark.parametrize("ab", [(1.0, 0.0), (0.0, 0.6)])
def test_coupling_on_ragged_grids(icm, precision, grid, kernel, h, ab):
    sim = icm.Simulation(grid, h, 1.0, 0.6, 0.0, 0.05, kernel, 1, precision, 0)
    rng = np.random.default_rng(sum(grid) + kernel)
    L = np.array(grid) * h
    qj = rng.uniform(0, 1, size=(5, 3)) * L
    qi = qj + rng.uniform(-2, 2, size=(5, 3)) * h
    qj[0] = [0.0, L[1], 0.5 * h]
    qi[0] = [L[0] - 0.5 * h, -0.25 * h, L[2] + 1.0]
    qi[1] = qj[1]
    got = icm.icm_op_coupling(sim.handle, qi, qj, *ab)
    want = np.array([oracle.coupling_matrix(np.mod(qi[p], L), np.mod(qj[p], L), grid, kernel, h, *ab)
                     for p in range(5)])
    assert rel(got, want) < TOL[precision]
    sim.close()


def test_coupling_of_many_pairs_equals_each_alone(icm):
    grid = (8, 6, 9)
    sim = icm.Simulation(grid, 1.0, 1.0, 1.0, 0.0, 0.05, 3, 1, 64, 0)
    rng = np.random.default_rng(8)
    q = rng.uniform(0, 1, size=(2, 600, 3)) * grid
    got = icm.icm_op_coupling(sim.handle, q[0], q[1], 0.5, 0.25)
    for p in (0, 1, 511, 512, 513, 599):
        one = icm.icm_op_coupling(sim.handle, q[0, p], q[1, p], 0.5, 0.25)
        assert np.array_equal(one[0], got[p])
    sim.close()
