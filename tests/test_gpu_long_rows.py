"""x sides above 256 with more blobs per block of rows than the inverse x pass stages (32 in FP32): the
records past those are read in place.  Sides 384 and 512, store, gather-only and adding passes,
against the oracle step by step."""
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


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("grid,nb,kernel", [((384, 32, 6), 400, 3), ((512, 16, 8), 500, 4), ((512, 48, 8), 20, 4)])
def test_steps_with_crowded_row_blocks(icm, precision, grid, nb, kernel):
    prm = oracle.Params(grid, h=0.9, rho=1.1, eta=0.8, kT=1e-3, dt=0.05, kernel=kernel, seed=5)
    rng = np.random.default_rng(nb + kernel)
    state = oracle.State(wl.random_fluid(grid, 0.05, 3), rng.uniform(0.0, 1.0, size=(nb, 3)) * prm.box,
                         0.05 * rng.standard_normal((nb, 3)), rng.uniform(-0.5, 2.0, size=nb),
                         0.01 * rng.standard_normal((nb, 3)))
    sim = make_sim(prm, state, precision)
    for _ in range(2):
        sim.step(1)
        want = oracle.icm_step(state, prm)
        got, _ = read_oracle_state(sim, prm, state.me, state.force)
        for key, e in compare_states(got, want, prm, state.q).items():
            assert e < TOL[precision], (key, e)
        state = got
    sim.close()
