"""The one-kernel form of a small plan against its launches, bit by bit."""
import ctypes

import numpy as np
import pytest

from paper_2004_10892_gb300 import inputs as I

# (rows, cols, depth, seed, plan options): no fused chains, so that every bucket is summed on its own
CIRCUITS = [
    (4, 4, 12, 4, {}),
    (4, 4, 16, 0, dict(min_p=2, max_p=2)),
    (5, 5, 20, 3, dict(leaf_absorb=0)),
    (5, 6, 26, 3, dict(max_bag_log2=15, max_p=9)),
    (6, 6, 20, 4116, dict(max_bag_log2=20, max_p=30, reorder_every=1)),
]


def _form(tnq_lib, plan, use):
    """1: one kernel, 0: its launches."""
    f = tnq_lib.lib().tnq_internal_small
    f.argtypes = [ctypes.c_void_p, ctypes.c_int]
    assert f(plan.handle, use) == use


def _equal(a, b):
    """Every slice is a product of FP32 tensors in FP64, whose factors are multiplied in another order."""
    assert np.max(np.abs(a - b)) <= 1e-14 * np.max(np.abs(b))


@pytest.mark.gpu
@pytest.mark.parametrize("case", CIRCUITS, ids=str)
def test_circuits_have_the_launches_bits(cuda, tnq_lib, case):
    rows, cols, depth, seed, kw = case
    circ = I.random_grid_circuit(rows, cols, depth, seed)
    plan = tnq_lib.Plan(circ, fuse_min_rank=0, **kw)
    bits = I.random_bitstring(circ.n_qubits, 5)
    n = min(8, plan.info()["n_slices"])
    _form(tnq_lib, plan, 1)
    one = tnq_lib.contract_sliced(plan, bits, 0, n, per_slice=True)[1]
    _form(tnq_lib, plan, 0)
    _equal(one, tnq_lib.contract_sliced(plan, bits, 0, n, per_slice=True)[1])


# plans whose chains are fused: in k_group's general form, with a register tail, with two lean stages
CHAINS = [
    (4, 4, 16, 21, dict(min_p=2, max_p=2, fuse_min_rank=1)),
    (5, 5, 20, 21, dict(min_p=3, max_p=3, fuse_min_rank=4)),
    (4, 5, 24, 22, dict(min_p=4, max_p=4, fuse_min_rank=8)),
    (6, 6, 24, 0, dict(max_bag_log2=24, min_p=4, max_p=8)),
    (6, 6, 24, 5, dict(max_bag_log2=18, max_p=20, reorder_every=1, fuse_min_rank=8)),
    (5, 5, 28, 2, dict(min_p=2, max_p=2, reorder_every=1)),
    (4, 7, 26, 3, dict(max_bag_log2=20, max_p=20, reorder_every=1, fuse_min_rank=6)),
]


@pytest.mark.gpu
@pytest.mark.parametrize("case", CHAINS, ids=str)
def test_chains_have_their_kernels_bits(cuda, tnq_lib, case):
    """k_group's arithmetic, stage by stage (k_pair, off here, sums in another order)."""
    rows, cols, depth, seed, kw = case
    circ = I.random_grid_circuit(rows, cols, depth, seed)
    plan = tnq_lib.Plan(circ, **kw)
    assert plan.info()["n_fused_groups"] > 0
    bits = I.random_bitstring(circ.n_qubits, 5)
    n = min(8, plan.info()["n_slices"])
    _form(tnq_lib, plan, 1)
    one = tnq_lib.contract_sliced(plan, bits, 0, n, per_slice=True)[1]
    _form(tnq_lib, plan, 0)
    f = tnq_lib.lib().tnq_internal_pair
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    f.restype = None
    f(plan.handle, 0, 0)
    _equal(one, tnq_lib.contract_sliced(plan, bits, 0, n, per_slice=True)[1])


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols,dim,p", [(3, 3, 2, 0), (4, 4, 3, 1), (4, 5, 5, 2), (5, 5, 3, 3)])
def test_networks_have_the_launches_bits(cuda, tnq_lib, rows, cols, dim, p):
    net = I.random_lattice_network(rows, cols, dim, 7)
    plan = tnq_lib.Plan.from_network(net.dims, net.tensors, min_p=p, max_p=p, fuse_min_rank=0)
    _form(tnq_lib, plan, 1)
    one = tnq_lib.contract_sliced(plan, None, per_slice=True)[1]
    _form(tnq_lib, plan, 0)
    _equal(one, tnq_lib.contract_sliced(plan, None, per_slice=True)[1])
