"""Batches that are not full: the kernels work on the valid items only, so a
slice's value must be the same bits whatever range it was asked for in."""
import ctypes

import numpy as np
import pytest

from paper_2004_10892_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("rows,cols,depth,seed,bag", [(5, 5, 24, 2, 11), (6, 6, 20, 3, 13), (6, 6, 28, 1, 20)])
def test_every_range_gives_the_same_slices(cuda, tnq_lib, precision, rows, cols, depth, seed, bag):
    torch = cuda
    circ = I.random_grid_circuit(rows, cols, depth, seed)
    plan = tnq_lib.Plan(circ, max_bag_log2=bag, min_p=4, max_p=6, precision=precision, gemm_min_k_log2=3, reorder_every=1)
    f = tnq_lib.lib().tnq_internal_small  # (step by step: the launches are what is tested here)
    f.argtypes = [ctypes.c_void_p, ctypes.c_int]
    f(plan.handle, 0)
    n = plan.info()["n_slices"]
    bits = I.random_bitstring(circ.n_qubits, seed)
    ws = torch.empty(plan.workspace_bytes(16), dtype=torch.uint8, device="cuda")
    _, ref = tnq_lib.contract_sliced(plan, bits, 0, 16, workspace=ws, max_batch=16, per_slice=True)
    assert np.all(np.isfinite(ref)) and np.any(ref != 0)
    for begin, end in [(0, 1), (0, 3), (5, 10), (1, 16), (7, 16)]:
        ws.fill_(0xFF)  # what is left out must not be read: NaN in every tensor
        amp, got = tnq_lib.contract_sliced(plan, bits, begin, end, workspace=ws, max_batch=16, per_slice=True)
        assert np.array_equal(got, ref[begin:end])
        assert abs(amp - ref[begin:end].sum()) <= 1e-14 * np.abs(ref[begin:end]).sum()
    # bitstrings as items: three of them, 3 n of the batch's 4 n items
    more = [bits] + [I.random_bitstring(circ.n_qubits, seed + k) for k in (1, 2)]
    out = tnq_lib.amplitudes_batch([plan], [more])
    one = tnq_lib.contract_sliced(plan, bits, 0, n)
    assert abs(out[0] - one) <= 1e-9 * abs(one)
