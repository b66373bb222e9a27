"""Both builders of the WCA cell list (one block for short lists, three launches otherwise)
and the warp-per-blob forces against the oracle's all-pairs forces, through the impulse
and the blob displacement of a step: many cells, few cells per axis (two, and one), and
more blobs than one block's list."""
import numpy as np
import pytest

import icm_workloads as wl
from oracle import icm as oracle

from _gpu_helpers import TOL, compare_states, make_sim, read_oracle_state

pytestmark = pytest.mark.gpu

# grid, blobs, sigma: 28^3 cells (three launches); 14^3 cells; 3 x 2 x 1 cells of a crowded box;
# 8200 blobs (three launches)
CASES = [((32, 32, 32), 300, 1.0), ((32, 32, 32), 900, 2.0), ((24, 16, 9), 60, 3.9), ((64, 32, 36), 8200, 1.0)]


@pytest.mark.parametrize("grid,nb,sigma", CASES)
def test_wca_step_through_either_list(grid, nb, sigma):
    rng = np.random.default_rng(nb)
    q = rng.uniform(0.0, 1.0, size=(nb, 3)) * grid
    if nb < 1000:   # no pair so close that its force dwarfs the rest
        q = wl.random_sequential_addition(nb, grid, 1.0, 0.75 * sigma, nb)
    eps = 1e-4 if nb < 1000 else 1e-12
    prm = oracle.Params(grid, kT=1e-3, dt=0.02, kernel=3, seed=3, wca_epsilon=eps, wca_sigma=sigma)
    st = oracle.State(wl.random_fluid(grid, 0.02, 1), q, np.zeros((nb, 3)), np.zeros(nb), np.zeros((nb, 3)))
    sim = make_sim(prm, st, 64)
    sim.step(1)
    got, mom = read_oracle_state(sim, prm, st.me, st.force)
    sim.close()
    if nb > 1000:   # all pairs in blocks of rows: the force's sum is zero, its norm compared through u
        force = np.zeros((nb, 3))
        tr = {}
        prm0 = oracle.Params(grid, kT=1e-3, dt=0.02, kernel=3, seed=3)
        oracle.icm_step(st, prm0, tr)
        qh = tr["q_half"]
        for a in range(0, nb, 500):
            d = qh[a:a + 500, None, :] - qh[None, :, :]
            d -= prm.box * np.round(d / prm.box)
            r2 = (d * d).sum(axis=2)
            r2[np.arange(r2.shape[0]), a + np.arange(r2.shape[0])] = np.inf
            ok = r2 < (2.0 ** (1.0 / 6.0) * sigma) ** 2
            s6 = np.where(ok, sigma ** 6 / r2 ** 3, 0.0)
            force[a:a + 500] = (np.where(ok, 24.0 * eps * (2.0 * s6 * s6 - s6) / r2, 0.0)[:, :, None] * d).sum(axis=1)
        want = oracle.icm_step(oracle.State(st.v, st.q, st.u, st.me, force), prm0)
    else:
        want = oracle.icm_step(st, prm)
    for key, e in compare_states(got, want, prm, st.q).items():
        assert e < TOL[64], (key, e)
