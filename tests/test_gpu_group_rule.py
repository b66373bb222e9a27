"""Group solves by plane passes or by separate x and y passes: the members of one launch decide (full rounds
of blocks in FP32, one member in FP64).  On either side of every line, the launches of a step and
every member's result against its run alone."""
import numpy as np
import pytest

from _gpu_helpers import TOL, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def icm():
    import paper_1212_6427_gb300 as m
    from paper_1212_6427_gb300 import build
    build.build_library()
    m.use_torch_allocator()
    return m


def _make(icm, grid, k, precision):
    rng = np.random.default_rng(k)
    sim = icm.Simulation(grid, 1.0, 1.0, 1.0, 1e-3, 0.05, 3, 50 + k, precision)
    sim.add_blobs(rng.uniform(0.0, 1.0, size=(9, 3)) * grid, 0.05 * rng.standard_normal((9, 3)),
                  rng.uniform(-0.5, 2.0, size=9))
    sim.set_forces(0.01 * rng.standard_normal((9, 3)))
    return sim


@pytest.mark.parametrize("grid,precision,members,planes",
                         [((32, 32, 32), 32, 4, True), ((32, 32, 32), 32, 5, False), ((32, 32, 32), 32, 9, True),
                          ((32, 32, 32), 32, 10, False), ((96, 96, 32), 32, 5, True), ((32, 32, 32), 64, 1, True),
                          ((32, 32, 32), 64, 2, False), ((48, 48, 48), 64, 2, False)])
def test_members_decide_the_passes_of_a_group_solve(icm, grid, precision, members, planes):
    sims = [_make(icm, grid, k, precision) for k in range(members)]
    b = icm.icm_batch_create()
    icm.icm_batch_set(b, [s.handle for s in sims])
    icm.icm_batch_set_grouped(b, 2)
    icm.icm_batch_step(b, 3)
    icm.icm_batch_sync(b)
    # twelve launches of stages, and three solves of three launches (planes) or five
    assert icm.icm_batch_kernels_per_step(b) == 12 + 3 * (3 if planes else 5)
    for k, s in enumerate(sims):
        alone = _make(icm, grid, k, precision)
        alone.step(3)
        want, got = alone.read(fluid=True), s.read(fluid=True)
        for name in ("vel", "fluid"):
            assert rel(got[name], want[name]) < 2 * TOL[precision], name
        alone.close()
    icm.icm_batch_destroy(b)
    for s in sims:
        s.close()
