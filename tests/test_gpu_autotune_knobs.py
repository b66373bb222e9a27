"""The autotuners leave rhs_kz alone where no right-hand side marches (FP64; small FP32 grids whose normals fit
in the scratch): its trials could only pick a value by timing noise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def icm():
    import paper_1212_6427_gb300 as m
    from paper_1212_6427_gb300 import build
    build.build_library()
    m.use_torch_allocator()
    return m


def _sim(icm, grid, precision, kT, seed):
    sim = icm.Simulation(grid, 1.0, 1.0, 1.0, kT, 0.05, 3, seed, precision)
    sim.add_blobs(np.random.default_rng(seed).uniform(0, 16, size=(5, 3)), None, np.ones(5))
    return sim


@pytest.mark.parametrize("grid,precision,kT", [((32, 32, 32), 32, 1e-3), ((16, 16, 48), 32, 1e-3),
                                               ((48, 48, 24), 32, 0.0), ((48, 48, 24), 64, 1e-3)])
def test_a_simulation_keeps_its_march(icm, grid, precision, kT):
    sim = _sim(icm, grid, precision, kT, 1)
    for kz in (7, 11, 23):                    # none of them a candidate
        icm.icm_set_plan(sim.handle, rhs_kz=kz)
        plan, _ = icm.icm_autotune(sim.handle, 3)
        assert plan["rhs_kz"] == kz
    sim.close()


def test_a_batch_keeps_its_march(icm):
    for precision, grid in ((64, (48, 32, 32)), (32, (32, 32, 32))):
        for trial in range(2):
            sims = [_sim(icm, grid, precision, 1e-3, k) for k in range(3)]
            b = icm.icm_batch_create()
            icm.icm_batch_set(b, [s.handle for s in sims])
            icm.icm_batch_autotune(b, 2)
            assert all(icm.icm_get_plan(s.handle)["rhs_kz"] == 16 for s in sims)   # the plan the tuner starts from
            icm.icm_batch_destroy(b)
            for s in sims:
                s.close()
