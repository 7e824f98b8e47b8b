"""Early buckets (k_bucket_level): blocks of 1, 2, 4 and 8 pieces of 256
entries, items inside and across blocks, against the FP64 oracle and against
other batch sizes (a slice's value must not depend on the batch)."""
import ctypes
import re

import numpy as np
import pytest

from paper_2004_10892_gb300 import inputs as I

ROWS, COLS, DEPTH, SEED, BITSTRINGS = 5, 6, 32, 1, 32


@pytest.fixture(scope="module")
def work(tnq_lib):
    circ = I.random_grid_circuit(ROWS, COLS, DEPTH, SEED)
    plan = tnq_lib.Plan(circ, max_bag_log2=20, min_p=4, max_p=20, reorder_every=1)
    f = tnq_lib.lib().tnq_internal_small  # launches by level are what is tested here
    f.argtypes = [ctypes.c_void_p, ctypes.c_int]
    f(plan.handle, 0)
    return circ, plan, [I.random_bitstring(circ.n_qubits, SEED + i) for i in range(BITSTRINGS)]


def _pieces(tnq_lib, plan, mode, batch):
    """log2 of a block's pieces -> early buckets that have it."""
    f = tnq_lib.lib().tnq_internal_group_text
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_uint32, ctypes.c_char_p, ctypes.c_size_t]
    buf = ctypes.create_string_buffer(1 << 20)
    assert f(plan.handle, mode, batch, buf, 1 << 20) == 0
    return {int(r) for _, _, r in re.findall(r"early: (\d+) (\d+) (\d+)", buf.value.decode())}


def test_batch_sizes_reach_every_block_size(tnq_lib, work):
    _, plan, _ = work
    assert _pieces(tnq_lib, plan, 1, 32) == {0, 1}
    assert _pieces(tnq_lib, plan, 1, 128) == {0, 1, 2, 3}
    assert _pieces(tnq_lib, plan, 1, 512) == {0, 3}


@pytest.mark.gpu
def test_batches_match_oracle_and_each_other(cuda, tnq_lib, oracle_lib, work):
    import torch

    circ, plan, bits = work
    n = plan.info()["n_slices"]
    ref = np.array([oracle_lib.contract(circ, bits[0], order=plan.order(), mu=plan.sliced(), slices=(s, s + 1))
                    for s in range(2)])
    # complex64: ~100 buckets in sequence, each adding a few 2^-24 roundings
    scale = 2.0 ** (-(circ.n_qubits + plan.info()["p"]) / 2)
    one = np.array([tnq_lib.contract_sliced(plan, bits[0], s, s + 1, per_slice=True)[1][0] for s in range(2)])
    assert np.max(np.abs(one - ref) / np.maximum(np.abs(ref), scale)) <= 1e-5
    for batch in (3, 16):
        total, got = tnq_lib.contract_sliced(plan, bits[0], 0, n, per_slice=True, max_batch=batch)
        assert np.max(np.abs(got[:2] - one)) <= 1e-9 * scale
        assert abs(total - np.sum(got)) <= 1e-12 * np.sum(np.abs(got))  # FP64 sums of the slices' FP64 values
    sums = [tnq_lib.contract_sliced(plan, b, 0, n) for b in bits]
    for batch in (32, 128, 512):
        ws = torch.empty(plan.workspace_bytes(batch), dtype=torch.uint8, device="cuda")
        out = np.array(tnq_lib.amplitudes_batch([plan], [bits], workspace=ws))
        assert np.max(np.abs(out - np.array(sums))) <= 1e-9 * scale * n
