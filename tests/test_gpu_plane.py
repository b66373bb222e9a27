"""The plane passes (x and y transforms of a whole z plane in one pass) where they can go
wrong: odd numbers of rows, odd rows, rows that are not 16-byte aligned, one to three
factors per side, the smallest sides, planes of one block and of several rounds of blobs,
blobs whose stencils start on every plane (so the Laplacian's reach wraps), both blob
paths, against the oracle step by step; and the size above which separate passes take over."""
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


SOLVES = [(6, 6, 6), (9, 27, 8), (27, 9, 6), (54, 18, 9), (162, 24, 8), (24, 243, 6), (216, 108, 16), (128, 36, 9),
          (32, 81, 12), (192, 64, 8), (144, 162, 27), (81, 288, 6), (432, 6, 9), (384, 16, 8), (16, 512, 8)]


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("grid", SOLVES)
def test_solve_on_any_sides(icm, precision, grid):
    nx, ny, nz = grid
    sim = icm.Simulation(grid, 0.8, 1.3, 0.7, 0.0, 0.05, 3, 1, precision)
    r = np.random.default_rng(nx + ny + nz).standard_normal((3, nz, ny, nx))
    got = icm.icm_op_spectral_solve(sim.handle, 1.7, 0.4, r.ravel())
    assert rel(got, oracle.spectral_solve(r, 1.7, 0.4, 0.8)) < TOL[precision] / 2
    sim.close()


STEPS = [((12, 9, 16), 16, 4, "visc"), ((27, 12, 9), 9, 3, "full"), ((24, 54, 12), 12, 3, "visc"),
         ((32, 48, 18), 18, 4, "zero"), ((64, 64, 32), 700, 4, "full"), ((16, 16, 16), 600, 3, "visc")]


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("grid,nb,kernel,slip", STEPS)
@pytest.mark.parametrize("in_plane", [1, 0])
def test_steps_with_blobs_on_every_plane(icm, precision, grid, nb, kernel, slip, in_plane):
    prm = oracle.Params(grid, h=0.9, rho=1.1, eta=0.8, kT=1e-3, dt=0.05, kernel=kernel, seed=5, slip=slip)
    rng = np.random.default_rng(nb + kernel)
    q = rng.uniform(0.0, 1.0, size=(nb, 3)) * prm.box
    n = min(nb, grid[2])
    q[:n, 2] = (np.arange(n) + 0.4) * prm.h       # a stencil that starts on every plane
    state = oracle.State(wl.random_fluid(grid, 0.05, 3), q, 0.05 * rng.standard_normal((nb, 3)),
                         rng.uniform(-0.5, 2.0, size=nb), 0.01 * rng.standard_normal((nb, 3)))
    sim = make_sim(prm, state, precision)
    icm.icm_set_plan(sim.handle, fused_blobs=in_plane)
    for _ in range(3):
        sim.step(1)
        want = oracle.icm_step(state, prm)
        got, mom = read_oracle_state(sim, prm, state.me, state.force)
        for key, e in compare_states(got, want, prm, state.q).items():
            assert e < TOL[precision], (key, e)
        assert rel(got.slip_g, want.slip_g) < 30 * TOL[precision]   # a difference of nearby velocities over h^2
        scale = np.abs(want.v).sum() * prm.rho * prm.h ** 3
        assert np.abs(mom - oracle.total_momentum(want, prm)).max() < TOL[precision] * scale
        state = got
    sim.close()
