"""Small plans as one kernel (k_small): against the FP64 oracle, the state of
every level on the host, and the same plan run step by step."""
import ctypes

import numpy as np
import pytest

from oracle import network as onet
from paper_2004_10892_gb300 import inputs as I

TOL = 1e-5  # ~50 buckets of <= 8 complex64 factors in sequence

# circuits (rows, cols, depth, seed, plan options): one bucket level and many, only narrow levels and
# levels that a cluster shares, wires without a gate, every slicing depth
CASES = [
    (1, 2, 2, 0, {}),
    (2, 2, 5, 1, {}),
    (3, 3, 8, 2, dict(min_p=2, max_p=2)),
    (4, 4, 16, 0, {}),
    (4, 4, 16, 3, dict(min_p=4, max_p=4, leaf_absorb=0)),
    (5, 5, 20, 2, dict(precision=1, gemm_min_k_log2=3)),
    (5, 5, 24, 5, dict(min_p=1, max_p=1, precision=2)),
    (6, 6, 20, 1, {}),
    (6, 6, 24, 0, dict(max_bag_log2=24, min_p=4, max_p=8)),
    (5, 6, 26, 3, dict(max_bag_log2=15, max_p=9)),
]


def _plan(tnq_lib, case):
    rows, cols, depth, seed, kw = case
    circ = I.random_grid_circuit(rows, cols, depth, seed)
    return circ, tnq_lib.Plan(circ, **kw)


def _small(tnq_lib, plan, use):
    f = tnq_lib.lib().tnq_internal_small
    f.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return f(plan.handle, use)


@pytest.mark.parametrize("case", CASES, ids=str)
def test_levels_and_memory(tnq_lib, case):
    _, plan = _plan(tnq_lib, case)
    assert _small(tnq_lib, plan, 1) == 1
    msg = ctypes.create_string_buffer(256)
    assert tnq_lib.lib().tnq_internal_validate(plan.handle, 0, 2, msg, 256) == 0, msg.value


def test_large_plans_run_step_by_step(tnq_lib):
    plan = tnq_lib.Plan(I.random_grid_circuit(6, 6, 32, 0), max_bag_log2=26, max_p=30)
    assert plan.info()["flops_per_slice"] > 1 << 25
    assert _small(tnq_lib, plan, 1) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES, ids=str)
def test_matches_oracle_and_steps(cuda, tnq_lib, oracle_lib, case):
    circ, plan = _plan(tnq_lib, case)
    n, p = circ.n_qubits, plan.info()["p"]
    bits = [I.random_bitstring(n, s) for s in (1, 2, 3)]
    assert _small(tnq_lib, plan, 1) == 1
    amp, got = tnq_lib.contract_sliced(plan, bits[0], per_slice=True)
    ref = [oracle_lib.contract(circ, b, order=plan.order(), mu=plan.sliced(), per_slice=True) for b in bits]
    scale = 2.0 ** (-(n + p) / 2)
    assert np.max(np.abs(got - ref[0][1]) / np.maximum(np.abs(ref[0][1]), scale)) <= TOL
    assert abs(amp - ref[0][0]) <= TOL * max(abs(ref[0][0]), 2.0 ** (-n / 2))
    # batches of any size, the batched call and the allocation-free one give the same bits
    for batch in (1, 2):
        assert np.array_equal(tnq_lib.contract_sliced(plan, bits[0], max_batch=batch, per_slice=True)[1], got)
    assert np.array_equal(tnq_lib.contract_sliced_noalloc(plan, bits[0], per_slice=True)[1], got)
    out = tnq_lib.amplitudes_batch([plan], [bits])
    for a, r in zip(out, ref):
        assert abs(a - r[0]) <= TOL * max(abs(r[0]), 2.0 ** (-n / 2))
    assert abs(out[0] - amp) <= 1e-14 * np.abs(got).sum()
    _small(tnq_lib, plan, 0)
    _, steps = tnq_lib.contract_sliced(plan, bits[0], per_slice=True)
    tol = 1e-4 if case[4].get("precision", 0) else TOL  # (the steps may take split-precision GEMMs)
    assert np.max(np.abs(got - steps) / np.maximum(np.abs(steps), scale)) <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols,dim,p", [(3, 3, 2, 0), (4, 4, 3, 1), (4, 5, 5, 2), (5, 5, 3, 3)])
def test_networks(cuda, tnq_lib, rows, cols, dim, p):
    """Tensors with more than two variables (leaf value table), digits sliced."""
    net = I.random_lattice_network(rows, cols, dim, 7)
    plan = tnq_lib.Plan.from_network(net.dims, net.tensors, min_p=p, max_p=p)
    assert _small(tnq_lib, plan, 1) == 1
    _, got = tnq_lib.contract_sliced(plan, None, per_slice=True)
    ref = onet.contract_network(net.dims, net.tensors)
    assert abs(got.sum() - ref) <= TOL * max(abs(ref), np.abs(got).max())
    _small(tnq_lib, plan, 0)
    _, steps = tnq_lib.contract_sliced(plan, None, per_slice=True)
    assert np.max(np.abs(got - steps)) <= TOL * np.max(np.abs(steps))
