"""3xBF16 plans give 3xBF16 values on every route that a plan can take."""
import ctypes

import numpy as np
import pytest

from paper_2004_10892_gb300 import inputs as I

# small enough for one kernel, with GEMM chains (rows, cols, depth, seed, plan options)
SMALL = [
    (5, 5, 22, 8835, dict(max_bag_log2=20, min_p=2, max_p=40)),
    (6, 6, 20, 3416, dict(max_bag_log2=25, max_p=40)),
    (5, 4, 31, 4704, dict(max_bag_log2=26, min_p=2, max_p=40)),
]


def _plan(tnq_lib, case, precision):
    rows, cols, depth, seed, kw = case
    circ = I.random_grid_circuit(rows, cols, depth, seed)
    return circ, tnq_lib.Plan(circ, precision=precision, reorder_every=1, **kw)


def _small(tnq_lib, plan, use):
    f = tnq_lib.lib().tnq_internal_small
    f.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return f(plan.handle, use)


def _few(plan):
    """What the rule takes in complex64."""
    return plan.info()["flops_per_slice"] <= 6e6


@pytest.mark.parametrize("case", SMALL, ids=str)
def test_gemm_chains_in_bf16_keep_their_launches(tnq_lib, case):
    _, plan = _plan(tnq_lib, case, tnq_lib.PREC_SPLIT_BF16)
    assert plan.info()["n_gemm_buckets"] > 0
    assert _small(tnq_lib, plan, 1) == 1  # it has a one-kernel form,
    assert _small(tnq_lib, plan, 2) == 0  # which the rule does not take
    plan.keep_chains([])  # without GEMM chains every product is FP32
    assert plan.info()["n_gemm_buckets"] == 0 and _small(tnq_lib, plan, 2) == _few(plan)
    _, plan = _plan(tnq_lib, case, tnq_lib.PREC_C64)
    assert _small(tnq_lib, plan, 2) == _few(plan)


@pytest.mark.gpu
@pytest.mark.parametrize("case", SMALL, ids=str)
def test_small_bf16_plans_run_their_gemm_chains(cuda, tnq_lib, case):
    circ, plan = _plan(tnq_lib, case, tnq_lib.PREC_SPLIT_BF16)
    bits = I.random_bitstring(circ.n_qubits, 1)
    _, got = tnq_lib.contract_sliced(plan, bits, per_slice=True)
    _, loc = tnq_lib.contract_sliced_noalloc(plan, bits, per_slice=True)
    _small(tnq_lib, plan, 0)
    _, steps = tnq_lib.contract_sliced(plan, bits, per_slice=True)
    assert np.array_equal(got, steps) and np.array_equal(loc, steps)


# GEMM chains of mostly padding: every tile that they get, small tensors folded into either operand
PADDED = [
    (7, 5, 28, 2045, dict(max_bag_log2=22, max_p=40)),
    (5, 6, 31, 2775, dict(max_bag_log2=20, max_p=40)),
    (7, 6, 29, 6996, dict(max_bag_log2=23, max_p=40)),
    (6, 6, 20, 3416, dict(max_bag_log2=25, max_p=40)),
]


@pytest.mark.gpu
@pytest.mark.parametrize("case", PADDED, ids=str)
def test_padded_bf16_chains_give_the_gemm_values(cuda, tnq_lib, case):
    """FP32 sums in another order (2^-24 per addition, ~50 steps), and operands
    of later splits that they move across a rounding boundary (2^-17 each, with
    a probability of 2^-6): 5e-6 in all. FP32 products differ by up to 2e-5."""
    circ, plan = _plan(tnq_lib, case, tnq_lib.PREC_SPLIT_BF16)
    bits = I.random_bitstring(circ.n_qubits, 88)
    n = min(8, plan.info()["n_slices"])
    f = tnq_lib.lib().tnq_internal_pair
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    f.restype = None
    launches = tnq_lib.lib().tnq_internal_launches_per_batch
    launches.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_uint32]
    got = tnq_lib.contract_sliced(plan, bits, 0, n, per_slice=True)[1]
    fewer = launches(plan.handle, 0, 1)
    f(plan.handle, 1, 0)
    assert launches(plan.handle, 0, 1) > fewer  # (a GEMM packs its operands first)
    gemm = tnq_lib.contract_sliced(plan, bits, 0, n, per_slice=True)[1]
    assert np.linalg.norm(got - gemm) <= 5e-6 * np.linalg.norm(gemm)
