"""Solves and steps on grids whose planes do not fit in shared memory (or whose other side is 384 or 512): the
general x and y passes with every factorisation of a side, odd sides and sides of three factors
among them, alone and beside register passes, against the oracle."""
import numpy as np
import pytest

import icm_workloads as wl
from oracle import icm as oracle

from _gpu_helpers import TOL, compare_states, make_sim, read_oracle_state, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def icm():
    import paper_1212_6427_gb300 as m
    from paper_1212_6427_gb300 import build
    build.build_library()
    return m


def _passes(sim):
    return {name.split(".")[1] for name, _, _ in sim.profile(1) if name.startswith("rt1.")}


X_SIDES = [6, 9, 12, 16, 18, 24, 27, 36, 54, 72, 81, 108, 144, 162, 216, 243, 288, 324, 432, 486]
SOLVES = [(n, 384 if n % 4 else 512, 6) for n in X_SIDES] + [(512 if n % 4 else 384, n, 6) for n in X_SIDES] + \
         [(486, 486, 6), (324, 216, 8), (243, 432, 6)]


@pytest.mark.parametrize("precision,grid", [(p, g) for p in (64, 32) for g in SOLVES] + [(64, (144, 216, 8))])
def test_solve_by_the_general_passes(icm, precision, grid):
    nx, ny, nz = grid
    sim = icm.Simulation(grid, 0.8, 1.3, 0.7, 0.0, 0.05, 3, 1, precision)
    r = np.random.default_rng(nx + ny + nz).standard_normal((3, nz, ny, nx))
    got = icm.icm_op_spectral_solve(sim.handle, 1.7, 0.4, r.ravel())
    assert rel(got, oracle.spectral_solve(r, 1.7, 0.4, 0.8)) < TOL[precision] / 2
    assert _passes(sim) == {"x_fwd", "y_fwd", "z_sym", "y_inv", "x_inv"}
    sim.close()


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("grid,nb,kernel", [((243, 384, 6), 40, 3), ((384, 243, 6), 40, 3), ((54, 512, 8), 30, 4),
                                            ((162, 486, 9), 30, 3)])
def test_steps_with_blobs_on_the_general_passes(icm, precision, grid, nb, kernel):
    prm = oracle.Params(grid, h=0.9, rho=1.1, eta=0.8, kT=1e-3, dt=0.05, kernel=kernel, seed=5)
    rng = np.random.default_rng(nb + kernel)
    q = rng.uniform(0.0, 1.0, size=(nb, 3)) * prm.box
    q[0], q[1] = 0.0, prm.box - 0.25 * prm.h                    # on the seams
    state = oracle.State(wl.random_fluid(grid, 0.05, 3), q, 0.05 * rng.standard_normal((nb, 3)),
                         rng.uniform(-0.5, 2.0, size=nb), 0.01 * rng.standard_normal((nb, 3)))
    sim = make_sim(prm, state, precision)
    for _ in range(2):
        sim.step(1)
        want = oracle.icm_step(state, prm)
        got, _ = read_oracle_state(sim, prm, state.me, state.force)
        for key, e in compare_states(got, want, prm, state.q).items():
            assert e < TOL[precision], (key, e)
        state = got
    assert "x_fwd" in _passes(sim)
    sim.close()
