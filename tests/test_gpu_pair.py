"""Fused chains as register-tiled products (k_pair): every shape that the rule
accepts, against the FP64 oracle and against the same plan run bucket by
bucket. The shape of a chain is (C: a third large tensor, loops over summed
variables outside the register tile n1 / n2, summed variables among the
register bits nkx / nky, tile bits or one tile, small tensors folded into A)."""
import ctypes
import re

import numpy as np
import pytest

from paper_2004_10892_gb300 import inputs as I

# complex64 chains: products of <= 3 tensors, sums of <= 2^5 terms per chain
# and ~50 buckets in sequence, each adding a few 2^-24 roundings
TOL = 1e-5

# (rows, cols, depth, seed, shapes that the plan's chains have)
CASES = [
    (4, 5, 26, 3, {("-", 1, 0, 0, 0)}),
    (4, 5, 29, 2, {("-", 4, 0, 0, 0)}),
    (4, 5, 32, 3, {("-", 3, 0, 0, 0)}),
    (4, 7, 29, 5, {("-", 2, 0, 0, 0)}),
    (4, 5, 26, 1, {("c", 0, 0, 0, 1)}),
    (4, 7, 23, 2, {("c", 0, 0, 0, 2)}),
    (4, 7, 23, 8, {("c", 0, 0, 1, 1)}),
    (4, 5, 23, 5, {("c", 0, 0, 1, 2)}),
    (5, 6, 23, 2, {("c", 0, 0, 2, 1)}),
    (5, 5, 26, 5, {("c", 0, 0, 2, 2)}),
    (5, 5, 20, 9, {("c", 0, 1, 1, 1)}),
    (4, 7, 26, 1, {("c", 0, 1, 1, 2)}),
    (5, 6, 20, 0, {("c", 0, 1, 2, 1)}),
    (4, 5, 29, 1, {("c", 0, 2, 0, 2)}),
    (4, 5, 26, 8, {("c", 1, 0, 1, 1)}),
    (4, 7, 26, 3, {("c", 1, 0, 1, 2)}),
    (4, 7, 29, 4, {("c", 1, 0, 2, 1)}),
    (5, 5, 23, 0, {("c", 1, 1, 1, 1)}),
    (4, 5, 26, 4, {("c", 2, 0, 1, 1)}),
    (4, 5, 32, 9, {("c", 2, 1, 0, 1)}),
    (4, 7, 29, 9, {("c", 3, 0, 0, 1)}),
]


# (precision, rows, cols, depth, seed, forms): what runs as a product (0 a bucket, 1 a chain, 2 a GEMM chain of mostly
# padding), C ("B": B alone, "X": and small tensors with other variables), whether it holds the first eliminated variable, register bits along A / B, those of them that are summed
FORMS = [
    (0, 4, 7, 23, 7, {(0, "-", 0, 1, 3, 0, 0)}),
    (1, 4, 5, 26, 1, {(0, "-", 0, 2, 2, 0, 0)}),
    (1, 4, 7, 29, 0, {(0, "-", 0, 2, 3, 0, 0)}),
    (0, 4, 5, 29, 5, {(0, "c", 1, 2, 2, 0, 0)}),
    (1, 4, 7, 29, 9, {(1, "-", 0, 0, 1, 0, 0)}),
    (1, 5, 6, 17, 3, {(2, "-", 0, 0, 1, 0, 0)}),
    (0, 4, 5, 29, 7, {(1, "-", 0, 1, 3, 0, 0)}),
    (1, 5, 5, 26, 8, {(1, "-", 0, 2, 3, 0, 0)}),
    (0, 5, 5, 28, 10, {(1, "c", 0, 2, 3, 0, 1)}),
    (0, 6, 6, 26, 2, {(1, "c", 0, 2, 3, 0, 2)}),
    (0, 4, 5, 30, 0, {(1, "c", 0, 2, 3, 1, 1)}),
    (0, 4, 5, 30, 11, {(1, "c", 0, 2, 3, 1, 2)}),
    (0, 5, 5, 26, 12, {(1, "c", 0, 2, 3, 2, 1)}),
    (0, 5, 5, 26, 5, {(1, "c", 0, 2, 3, 2, 2)}),
    (0, 5, 5, 29, 2, {(1, "c", 1, 2, 2, 0, 0)}),
    (0, 4, 5, 26, 7, {(1, "c", 1, 2, 2, 0, 1)}),
    (0, 6, 6, 29, 0, {(1, "c", 1, 2, 2, 0, 2)}),
    (0, 5, 5, 23, 1, {(1, "c", 1, 2, 2, 1, 1)}),
    (1, 4, 5, 32, 2, {(2, "-", 0, 2, 2, 0, 0)}),
    (0, 4, 5, 29, 1, {(0, "B", 0, 0, 3, 0, 0)}),
    (0, 4, 5, 26, 0, {(1, "B", 0, 0, 3, 0, 0)}),
    (0, 4, 5, 32, 4, {(1, "B", 0, 0, 1, 0, 0)}),  # one chunk, 2^6 products of small tensors
    (0, 4, 5, 32, 0, {(1, "B", 0, 0, 1, 0, 0)}),  # two chunks
    (1, 5, 6, 29, 6, {(1, "B", 0, 0, 1, 0, 0)}),  # four
    (0, 5, 6, 32, 9, {(0, "X", 0, 0, 3, 0, 0)}),
    (0, 5, 6, 32, 0, {(0, "X", 0, 0, 3, 0, 0)}),  # 2^7 products of small tensors
    (0, 4, 5, 26, 5, {(1, "X", 0, 0, 3, 0, 0)}),
]


def _plan(tnq_lib, rows, cols, depth, seed, bag=20, **kw):
    circ = I.random_grid_circuit(rows, cols, depth, seed)
    plan = tnq_lib.Plan(circ, max_bag_log2=bag, max_p=20, reorder_every=1, **kw)
    f = tnq_lib.lib().tnq_internal_small  # these plans are small: their chains are what is tested here
    f.argtypes = [ctypes.c_void_p, ctypes.c_int]
    f(plan.handle, 0)
    return circ, plan


def _bag(forms):
    """C with 4 x 8 tiles needs the outputs of a larger plan."""
    return 22 if any(f[1] == "c" and f[4] == 3 for f in forms) else 20


def _words(tnq_lib, plan):
    f = tnq_lib.lib().tnq_internal_group_text
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_uint32, ctypes.c_char_p, ctypes.c_size_t]
    buf = ctypes.create_string_buffer(1 << 20)
    assert f(plan.handle, 0, 2, buf, 1 << 20) == 0
    for line in re.findall(r"pair: (.*)", buf.value.decode()):
        w = line.split()
        d = dict(zip(w[::2], map(int, w[1::2])))
        outside = d["b"] < 8 + d["ry"] + d["n1"] - d["chunks"] // 2  # local outputs that the large tensor lacks
        yield dict(d, c="BX"[outside] if d["a"] == 0 else "-" if d["c"] < 0 else "c")


def _shapes(tnq_lib, plan):
    return {tuple(d[k] for k in ("c", "n1", "n2", "nkx", "nky")) for d in _words(tnq_lib, plan) if not d["c_u0"]}


def _forms(tnq_lib, plan):
    return {tuple(d[k] for k in ("kind", "c", "c_u0", "rx", "ry", "nkx", "nky")) for d in _words(tnq_lib, plan)}


@pytest.mark.parametrize("rows,cols,depth,seed,shapes", CASES)
def test_every_launch_stays_in_bounds(tnq_lib, rows, cols, depth, seed, shapes):
    """Host only: the rule gives these shapes, and every staged, folded and
    written index of both modes and several batch sizes is inside its tensor."""
    _, plan = _plan(tnq_lib, rows, cols, depth, seed)
    assert shapes <= _shapes(tnq_lib, plan)
    msg = ctypes.create_string_buffer(512)
    for mode in (0, 1):
        for batch in (1, 2, 16):
            assert tnq_lib.lib().tnq_internal_validate(plan.handle, mode, batch, msg, 512) == 0, msg.value


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols,depth,seed,shapes", CASES)
def test_chain_matches_oracle_and_separate_buckets(cuda, tnq_lib, oracle_lib, rows, cols, depth, seed, shapes):
    circ, plan = _plan(tnq_lib, rows, cols, depth, seed)
    assert shapes <= _shapes(tnq_lib, plan)
    _check(tnq_lib, oracle_lib, circ, plan, _plan(tnq_lib, rows, cols, depth, seed, fuse_min_rank=0)[1], seed, TOL)


@pytest.mark.parametrize("precision,rows,cols,depth,seed,forms", FORMS)
def test_every_form_stays_in_bounds(tnq_lib, precision, rows, cols, depth, seed, forms):
    _, plan = _plan(tnq_lib, rows, cols, depth, seed, _bag(forms), precision=precision)
    assert forms <= _forms(tnq_lib, plan)
    msg = ctypes.create_string_buffer(512)
    for mode in (0, 1):
        for batch in (1, 2, 16):
            assert tnq_lib.lib().tnq_internal_validate(plan.handle, mode, batch, msg, 512) == 0, msg.value


@pytest.mark.gpu
@pytest.mark.parametrize("precision,rows,cols,depth,seed,forms", FORMS)
def test_form_matches_oracle_and_separate_buckets(cuda, tnq_lib, oracle_lib, precision, rows, cols, depth, seed, forms):
    bag = _bag(forms)
    circ, plan = _plan(tnq_lib, rows, cols, depth, seed, bag, precision=precision)
    assert forms <= _forms(tnq_lib, plan)
    # (split precision: the plan's other GEMM chains keep 16 to 22 bits of their operands)
    _check(tnq_lib, oracle_lib, circ, plan, _plan(tnq_lib, rows, cols, depth, seed, bag, fuse_min_rank=0)[1], seed,
           1e-4 if precision else TOL)


def _check(tnq_lib, oracle_lib, circ, plan, plain, seed, tol):
    n = min(plan.info()["n_slices"], 4)
    bits = I.random_bitstring(circ.n_qubits, seed)
    _, got = tnq_lib.contract_sliced(plan, bits, 0, n, per_slice=True)
    _, sep = tnq_lib.contract_sliced(plain, bits, 0, n, per_slice=True)
    ref = np.array([oracle_lib.contract(circ, bits, order=plan.order(), mu=plan.sliced(), slices=(s, s + 1))
                    for s in range(n)])
    scale = np.maximum(np.abs(ref), 2.0 ** (-(circ.n_qubits + plan.info()["p"]) / 2))
    assert np.max(np.abs(got - ref) / scale) <= tol
    assert np.max(np.abs(got - sep) / scale) <= tol
    # three bitstrings at once: the item dimension carries (bitstring, slice)
    more = [bits, I.random_bitstring(circ.n_qubits, seed + 1), I.random_bitstring(circ.n_qubits, seed + 2)]
    # (the GEMM packs multiply the small tensors in another order when one of them depends on the item)
    if plan.info()["p"] == 0 and plan.info()["n_gemm_buckets"] == 0:
        out = tnq_lib.amplitudes_batch([plan], [more])
        assert abs(out[0] - got[0]) <= 1e-9 * abs(got[0])
