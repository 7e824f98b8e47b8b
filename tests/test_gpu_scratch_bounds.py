"""The allocation-free call stays inside its static array, or refuses."""
import ctypes

import numpy as np
import pytest

SCRATCH = 64 << 20


def _network(n, seed=0):
    """n tensors of 2^16 entries (half a megabyte each) over one shared 16-valued index and three of their own: a
    slice is a few thousand operations a tensor, and the entries are what takes memory."""
    rng = np.random.default_rng(seed)
    dims, tensors = [16], []
    for _ in range(n):
        own = list(range(len(dims), len(dims) + 3))
        dims += [16] * 3
        tensors.append(([0] + own, rng.standard_normal((16,) * 4) / 64 + 0j))
    return dims, tensors


def _plan(tnq_lib, n):
    dims, tensors = _network(n)
    return dims, tensors, tnq_lib.Plan.from_network(dims, tensors, min_p=4, max_p=4)


def _items(tnq_lib, plan, items, cap):
    f = tnq_lib.lib().tnq_internal_noalloc_small
    f.restype = ctypes.c_size_t
    f.argtypes = [ctypes.c_void_p, ctypes.c_uint32, ctypes.c_uint64, ctypes.POINTER(ctypes.c_int32)]
    batch = ctypes.c_int32()
    return f(plan.handle, items, cap, ctypes.byref(batch)), batch.value


def test_what_runs_at_once_fits(tnq_lib):
    for n in (100, 127):
        plan = _plan(tnq_lib, n)[2]
        for cap in (1, 2, 16):
            batch = _items(tnq_lib, plan, 1, cap)[1]
            assert 0 <= batch <= cap and (n > 100 or batch)
            assert batch == 0 or _items(tnq_lib, plan, batch, cap)[0] <= SCRATCH
            assert batch == cap or _items(tnq_lib, plan, max(1, 2 * batch), cap)[0] > SCRATCH


def test_tables_beyond_the_array_do_not_fit(tnq_lib):
    plan = _plan(tnq_lib, 140)[2]
    used, batch = _items(tnq_lib, plan, 1, 16)
    assert used > SCRATCH and batch == 0


@pytest.mark.gpu
def test_refused_with_the_byte_counts(cuda, tnq_lib):
    dims, tensors, plan = _plan(tnq_lib, 140)
    with pytest.raises(tnq_lib.TnqError) as e:
        tnq_lib.contract_sliced_noalloc(plan)
    assert e.value.status == tnq_lib.ENOMEM and "static scratch" in str(e.value)
    # the last size that fits gives the workspace call's values
    dims, tensors, plan = _plan(tnq_lib, 100)
    ref = tnq_lib.contract_sliced(plan, per_slice=True)[1]
    assert np.any(ref != 0) and np.array_equal(tnq_lib.contract_sliced_noalloc(plan, per_slice=True)[1], ref)
