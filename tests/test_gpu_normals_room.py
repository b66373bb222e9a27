"""The stress normals take no device memory of their own: they live in the spectrum scratch, in slabs of
planes where it does not hold all of them (FP64; FP32 grids march and store none).  What a simulation holds, what jobs are admitted by, and the
right-hand side against the oracle in one slab and in several: an odd number of planes, ragged
last slabs, one plane at a time."""
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
    m.use_torch_allocator()
    return m


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("grid", [(32, 32, 32), (48, 48, 48), (96, 24, 27)])
def test_noise_takes_no_memory(icm, grid, precision):
    held = []
    for kT in (0.0, 1e-3):
        sim = icm.icm_create(grid, 1.0, 1.0, 1.0, kT, 0.05, 3, 1, precision, 0, None)
        icm.icm_step(sim, 2)
        icm.icm_sync(sim)
        held.append(icm.icm_device_bytes(sim))
        icm.icm_destroy(sim)
    assert held[0] == held[1]
    # three face fields and the padded spectrum, and little else
    nx, ny, nz = grid
    reals = 9 * nx * ny * nz + 6 * nz * ny * ((nx // 2 + 1 + 15) // 16 * 16)
    estimate = icm.icm_estimate_device_bytes(grid, precision, 0)
    assert held[1] <= estimate <= reals * precision // 8 + 200_000
    server = icm.icm_server_create(estimate, 1)
    job = icm.icm_server_submit(server, grid, 1.0, 1.0, 1.0, 1e-3, 0.05, 3, 5, precision, 0, np.zeros((0, 3)), None,
                                np.zeros(0), None, 2)
    for _ in range(100000):
        icm.icm_server_pump(server, 2)
        if icm.icm_server_result(server, job, 0)["state"] >= 2:
            break
    assert icm.icm_server_result(server, job, 0)["state"] == 2
    icm.icm_server_destroy(server)


SLABS = [((16, 16, 9), 1), ((24, 12, 27), 2), ((48, 16, 48), 2), ((162, 8, 9), 3), ((512, 8, 6), 6), ((486, 6, 16), 3)]


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("grid,slabs", SLABS)
@pytest.mark.parametrize("hist", [True, False])
def test_right_hand_side_slab_by_slab(icm, grid, slabs, precision, hist):
    nx, ny, nz = grid
    fit = nz * ((nx // 2 + 1 + 15) // 16 * 16) // nx            # planes of normals in the spectrum scratch
    assert slabs == (1 if fit >= nz else -(-nz // (fit - 2)))
    prm = oracle.Params(grid, h=0.9, rho=1.2, eta=0.7, kT=2e-3, dt=0.04, kernel=3, seed=(5 << 33) + 17)
    rng = np.random.default_rng(nx + ny + nz)
    v = 0.1 * rng.standard_normal((3, nz, ny, nx))
    prev = 0.1 * rng.standard_normal((3, nz, ny, nx)) if hist else None
    sim = icm.Simulation(grid, prm.h, prm.rho, prm.eta, prm.kT, prm.dt, 3, prm.seed, precision)
    r, a = icm.icm_op_explicit_rhs(sim.handle, v.ravel(), None if prev is None else prev.ravel(), 5)
    want_r, want_a = oracle.explicit_rhs(v, prev, 5, prm)
    assert rel(r, want_r) < TOL[precision] and rel(a, want_a) < TOL[precision]
    sim.close()
