"""The plane passes' blob work takes no memory beyond the row blocks' on grids that have both, and on grids that
only have planes it is left apart where there is none for it, with the same steps."""
import numpy as np
import pytest

import icm_workloads as wl
from oracle import icm as oracle

from _gpu_helpers import TOL, flags_of, rel
from test_gpu_coupling_limits import _KEEP, Limited

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def icm():
    import paper_1212_6427_gb300 as m
    from paper_1212_6427_gb300 import build
    build.build_library()
    m.use_torch_allocator()
    yield m
    m.use_torch_allocator()


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("blobs,slots", [(5, 64), (100, 128)])
def test_blob_slots_take_what_the_row_blocks_need(icm, precision, blobs, slots):
    sim = icm.Simulation((32, 32, 32), 1.0, 1.0, 1.0, 1e-3, 0.05, 3, 1, precision)
    before = icm.icm_device_bytes(sim.handle)
    sim.add_blobs(np.random.default_rng(1).uniform(0, 32, size=(blobs, 3)), None, np.ones(blobs))
    # blob arrays, stencil records, accumulators, and the bin list of 49 blocks per blob
    assert icm.icm_device_bytes(sim.handle) - before == slots * (41 * 8 + 336 + 12 * 8) + -(-slots * 49 * 4 // 256) * 256
    sim.close()


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("kernel,slip", [(3, "visc"), (4, "full")])
def test_steps_without_room_for_the_records(icm, precision, kernel, slip):
    grid = (24, 27, 18)
    prm = oracle.Params(grid, h=0.9, rho=1.1, eta=0.8, kT=1e-3, dt=0.05, kernel=kernel, seed=5, slip=slip)
    rng = np.random.default_rng(3)
    state = oracle.State(wl.random_fluid(grid, 0.05, 3), rng.uniform(0.0, 1.0, size=(9, 3)) * prm.box,
                         0.05 * rng.standard_normal((9, 3)), rng.uniform(-0.5, 2.0, size=9),
                         0.01 * rng.standard_normal((9, 3)))
    for limited in (False, True):
        mem = Limited(icm)
        _KEEP.append(mem)
        sim = icm.icm_create(grid, prm.h, prm.rho, prm.eta, prm.kT, prm.dt, kernel, prm.seed, precision, flags_of(prm), None)
        if limited:
            mem.limit = sum(mem.held.values()) + 64 * 41 * 8     # the blob arrays, and no records
        icm.icm_add_blobs(sim, state.q, state.u, state.me)
        mem.limit = None
        icm.icm_set_blob_forces(sim, state.force)
        icm.icm_write_state(sim, state.q, state.u, state.v.ravel(), None, state.slip_g, 0)
        assert ("spread" in [name for name, _, _ in icm.icm_profile_steps(sim, 1)]) == limited
        vel, fluid = icm.icm_read_state(sim, int(np.prod(grid)), fluid=True)[1:3]
        want = oracle.icm_step(state, prm)
        assert rel(vel, want.u) < TOL[precision] and rel(fluid, want.v) < TOL[precision]
        icm.icm_destroy(sim)
