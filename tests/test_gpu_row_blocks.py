"""The blob work inside the x passes of sides up to 256 with crowded row blocks (more records than a block stages)
and row blocks that straddle z planes, alone and in batched stages, against the oracle step by step."""
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


def _crowd(grid, nb, kernel, seed, side=14.0):
    """Half of the blobs in a corner of `side` cells across the periodic seams, the others anywhere."""
    prm = oracle.Params(grid, h=0.9, rho=1.1, eta=0.8, kT=1e-3, dt=0.02, kernel=kernel, seed=seed)
    rng = np.random.default_rng(seed)
    q = rng.uniform(0.0, 1.0, size=(nb, 3)) * prm.box
    q[: nb // 2] = np.mod(rng.uniform(-0.5, 0.5, size=(nb // 2, 3)) * np.minimum(side * prm.h, prm.box), prm.box)
    state = oracle.State(wl.random_fluid(grid, 0.05, 3), q, 0.02 * rng.standard_normal((nb, 3)),
                         rng.uniform(-0.5, 2.0, size=nb), 0.01 * rng.standard_normal((nb, 3)))
    return prm, state


def _compare(sim, prm, state, precision):
    want = oracle.icm_step(state, prm)
    got, _ = read_oracle_state(sim, prm, state.me, state.force)
    for key, e in compare_states(got, want, prm, state.q).items():
        assert e < TOL[precision], (key, e)
    return got


CASES = [((128, 128, 8), 64, 700, 4), ((256, 192, 8), 32, 900, 4), ((256, 192, 8), 64, 700, 3),
         ((192, 144, 8), 64, 700, 3), ((256, 216, 8), 32, 900, 3), ((256, 243, 9), 32, 1100, 4),
         ((32, 32, 192), 32, 2200, 3)]


@pytest.mark.parametrize("grid,precision,nb,kernel", CASES)
def test_crowded_row_blocks(icm, grid, precision, nb, kernel):
    prm, state = _crowd(grid, nb, kernel, 7)
    sim = make_sim(prm, state, precision)
    for _ in range(2):
        sim.step(1)
        state = _compare(sim, prm, state, precision)
    stages = [name for name, _, _ in sim.profile(1)]
    assert "bins" in stages and "rt1.x_inv" in stages and "spread" not in stages
    sim.close()


@pytest.mark.parametrize("precision", [64, 32])
def test_crowded_row_blocks_in_batched_stages(icm, precision):
    members = [_crowd((32, 32, 32), 500, 3, 11), _crowd((32, 32, 32), 300, 4, 12), _crowd((48, 48, 48), 600, 4, 13),
               _crowd((64, 64, 64), 800, 3, 14)]
    sims = [make_sim(prm, state, precision) for prm, state in members]
    b = icm.icm_batch_create()
    icm.icm_batch_set(b, [s.handle for s in sims])
    icm.icm_batch_set_grouped(b, 3)
    states = [state for _, state in members]
    for _ in range(2):
        icm.icm_batch_step(b, 1)
        icm.icm_batch_sync(b)
        states = [_compare(s, prm, state, precision) for s, (prm, _), state in zip(sims, members, states)]
    # ten launches of stages (one precision, every member with noise), three solves of five for each of three grids
    assert icm.icm_batch_kernels_per_step(b) == 10 + 3 * 3 * 5
    icm.icm_batch_destroy(b)
    for s in sims:
        s.close()
