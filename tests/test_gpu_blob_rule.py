"""Who does the blob work of a step on a grid with plane passes: the planes up to a number of blobs, row
blocks or separate kernels past it.  On either side of every line, the path taken (by its stages)
and the step against the oracle; and the plane passes with lists that fill, and with more blobs
than one window of them, which only FP64 grids without row blocks still give them."""
import numpy as np
import pytest

import icm_workloads as wl
from oracle import icm as oracle

from _gpu_helpers import TOL, compare_states, make_sim, read_oracle_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def icm():
    import paper_1212_6427_gb300 as m
    from paper_1212_6427_gb300 import build
    build.build_library()
    return m


def _path(sim, state):
    sim.write(state.q, state.u, state.v.ravel(), None, state.slip_g, state.step)   # the step just compared, again
    stages = [name for name, _, _ in sim.profile(1)]
    if "spread" in stages:
        return "apart"
    return "planes" if "rt1.yx_inv" in stages else "rows"


def _state(grid, nb, kernel, inertial, prm, seed):
    rng = np.random.default_rng(seed)
    return oracle.State(wl.random_fluid(grid, 0.05, 3), rng.uniform(0.0, 1.0, size=(nb, 3)) * prm.box,
                        0.05 * rng.standard_normal((nb, 3)), rng.uniform(-0.5, 2.0, size=nb) * inertial,
                        0.01 * rng.standard_normal((nb, 3)))


def _step_and_compare(sim, prm, state, precision):
    sim.step(1)
    want = oracle.icm_step(state, prm)
    got, _ = read_oracle_state(sim, prm, state.me, state.force)
    for key, e in compare_states(got, want, prm, state.q).items():
        assert e < TOL[precision], (key, e)


LINES = [((16, 16, 16), 32, True, 640, "apart"), ((32, 32, 32), 32, True, 1280, "apart"),
         ((24, 24, 27), 32, True, 1080, "apart"), ((128, 128, 54), 32, True, 1728, "rows"),
         ((32, 32, 192), 32, True, 2048, "rows"), ((32, 32, 32), 32, False, 2048, "apart"),
         ((32, 32, 32), 64, True, 5120, "rows"), ((32, 64, 192), 64, False, 16384, "rows")]


@pytest.mark.parametrize("grid,precision,inertial,most,beyond", LINES)
def test_the_blob_work_moves_at_the_line(icm, grid, precision, inertial, most, beyond):
    prm = oracle.Params(grid, h=0.9, rho=1.1, eta=0.8, kT=1e-3, dt=0.05, kernel=3, seed=5)
    for nb, path in ((most, "planes"), (most + 1, beyond)):
        state = _state(grid, nb, 3, inertial, prm, nb)
        sim = make_sim(prm, state, precision)
        _step_and_compare(sim, prm, state, precision)
        assert _path(sim, state) == path, nb
        sim.close()


def test_few_large_planes_leave_the_blobs_to_row_blocks(icm):
    prm = oracle.Params((128, 96, 12), kT=1e-3, dt=0.05, kernel=4, seed=5)
    state = _state((128, 96, 12), 3, 4, True, prm, 1)
    sim = make_sim(prm, state, 32)
    _step_and_compare(sim, prm, state, 32)
    assert _path(sim, state) == "rows"
    sim.close()


def test_full_lists_and_more_blobs_than_a_window(icm):
    """66000 blobs on a few planes (many lists for those, an empty window for the others), 4000 after them."""
    grid, nb = (24, 24, 48), 70000
    prm = oracle.Params(grid, kT=1e-3, dt=0.05, kernel=3, seed=5)
    state = _state(grid, nb, 3, True, prm, 2)
    state.q[:66000, 2] = 10.0 + 2.0 * np.random.default_rng(3).uniform(size=66000)
    state.q[66000:, 2] = 30.0 + 4.0 * np.random.default_rng(4).uniform(size=4000)
    sim = make_sim(prm, state, 64)
    _step_and_compare(sim, prm, state, 64)
    assert _path(sim, state) == "planes"
    sim.close()
