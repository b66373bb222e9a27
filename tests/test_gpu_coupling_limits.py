"""icm_op_coupling where there is no device memory but for the positions and results of the pairs: the
sums take their tables from the simulation's own scratch, with the same matrices."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def icm():
    import paper_1212_6427_gb300 as m
    from paper_1212_6427_gb300 import build
    build.build_library()
    yield m
    m.use_torch_allocator()


class Limited:
    """torch's allocator, with an upper bound on what is held."""

    def __init__(self, icm):
        import torch
        self.held, self.limit = {}, None
        make = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)
        drop = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)

        def give(_, size, stream):
            if self.limit is not None and sum(self.held.values()) + size > self.limit:
                return None
            p = torch.cuda.caching_allocator_alloc(int(size), stream=int(stream or 0))
            self.held[p] = int(size)
            return p

        def take(_, p, stream):
            self.held.pop(p, None)
            torch.cuda.caching_allocator_delete(p)

        self.calls = make(give), drop(take)
        icm.lib().icm_set_default_allocator(self.calls[0], self.calls[1], None)


_KEEP = []   # the simulations keep the function pointers


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("grid,pairs", [((6, 6, 6), 40), ((16, 16, 16), 1100), ((6, 6, 486), 3), ((64, 6, 9), 200)])
def test_coupling_needs_room_for_positions_and_results_only(icm, precision, grid, pairs):
    mem = Limited(icm)
    _KEEP.append(mem)
    sim = icm.icm_create(grid, 1.0, 1.0, 1.0, 0.0, 0.05, 3, 1, precision, 0, None)
    q = np.random.default_rng(pairs).uniform(0.0, 1.0, size=(2, pairs, 3)) * grid
    want = icm.icm_op_coupling(sim, q[0], q[1], 0.5, 0.25)
    mem.limit = sum(mem.held.values()) + (6 + 9) * 8 * pairs
    got = icm.icm_op_coupling(sim, q[0], q[1], 0.5, 0.25)
    assert np.array_equal(got, want)
    mem.limit = sum(mem.held.values())
    with pytest.raises(icm.IcmError) as ei:
        icm.icm_op_coupling(sim, q[0], q[1], 0.5, 0.25)
    assert ei.value.status == icm.ICM_ENOMEM
    icm.icm_destroy(sim)
