"""k_pair with inputs far below one: every input has its own power of two, and
the product of two or three of them is beyond FP32's range."""
import ctypes
import re

import numpy as np
import pytest

from oracle import network as onet

TINY = 1e-21  # two such scales are 2^139, three 2^209


def network(seed):
    """Sites of rank 7 and more over indices that two or three of them share. Each site is the sum over an index of its
    own of a tensor and a weight that are large at opposite values, so its entries are about TINY. Returns the network,
    and the sites alone as tensors of ordinary size."""
    rng = np.random.default_rng(seed)
    n = int(rng.integers(3, 8))
    dims, ends = [], [[] for _ in range(n)]
    while min(map(len, ends)) < 7:
        room = [s for s in range(n) if len(ends[s]) < 10]
        k = min(len(room), int(rng.choice([2, 2, 2, 3])))
        few = sorted(room, key=lambda s: (len(ends[s]), rng.random()))[: k + 1]
        for s in rng.choice(few, size=k, replace=False):
            ends[s].append(len(dims))
        dims.append(2)
    for _ in range(int(rng.integers(0, 6))):  # small ones
        ends.append([int(i) for i in rng.choice(len(dims), size=2, replace=False)])
    tensors, sites, plain = [], [], list(dims)
    for e in ends:
        shape = [dims[i] for i in e]
        a, b = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape) for _ in range(2))
        v = len(dims)
        dims.append(2)
        tensors.append(([v] + e, np.stack([a, TINY * b])))
        tensors.append(([v], np.array([TINY, 1.0], complex)))
        sites.append((e, a + b))
    return dims, tensors, plain, sites


def pairs(text):
    for line in re.findall(r"pair: (.*)", text):
        w = line.split()
        yield dict(zip(w[::2], map(int, w[1::2])))


def form(d):
    """Bucket or chain, and k_pair's kind: two tensors, a third without or with the first variable, one alone."""
    return d["kind"], "one" if d["a"] == 0 else "two" if d["c"] < 0 else "three, u" if d["c_u0"] else "three"


# seed of a network, sliced variables, k_pair's launches in its plan
CASES = [
    (7, 0, {(1, "three")}),
    (13, 0, {(1, "three"), (1, "two")}),
    (20, 0, {(1, "three")}),
    (91, 0, {(0, "one"), (1, "two")}),
    (96, 0, {(0, "one"), (1, "three"), (1, "two")}),
    (109, 0, {(0, "one"), (0, "two"), (1, "two")}),
    (122, 0, {(1, "three, u")}),
    (166, 0, {(0, "one"), (0, "two"), (1, "two")}),
    (197, 0, {(0, "one"), (0, "three, u"), (1, "two")}),
    (733, 0, {(1, "three, u"), (1, "two")}),
    # (several slices: every item has its own powers of two)
    (96, 2, {(1, "three"), (1, "two")}),
    (166, 1, {(0, "one"), (0, "two"), (1, "two")}),
    (733, 1, {(1, "three, u")}),
]


def _forms(tnq_lib, plan):
    f = tnq_lib.lib().tnq_internal_group_text
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_uint32, ctypes.c_char_p, ctypes.c_size_t]
    buf = ctypes.create_string_buffer(1 << 20)
    assert f(plan.handle, 0, 1, buf, 1 << 20) == 0
    return [form(d) for d in pairs(buf.value.decode())]


def _plan(tnq_lib, seed, p=0):
    dims, tensors, plain, sites = network(seed)
    plan = tnq_lib.Plan.from_network(dims, tensors, fuse_min_rank=8, min_p=p, max_p=p)
    f = tnq_lib.lib().tnq_internal_small  # (its launches are what is tested here)
    f.argtypes = [ctypes.c_void_p, ctypes.c_int]
    f(plan.handle, 0)
    # the chains that k_pair runs (k_group multiplies a stage's scales into one factor); the others bucket by bucket
    chains, kept = plan.fused_chains(), []
    for last in chains:
        plan.keep_chains([last])
        if [kind for kind, _ in _forms(tnq_lib, plan)].count(1) == 1:
            kept.append(last)
    plan.keep_chains(kept)
    assert [kind for kind, _ in _forms(tnq_lib, plan)].count(1) == len(kept) == plan.info()["n_fused_groups"]
    return plan, plain, sites


@pytest.mark.parametrize("seed,p,forms", CASES)
def test_plans_have_these_forms(tnq_lib, seed, p, forms):
    assert forms <= set(_forms(tnq_lib, _plan(tnq_lib, seed, p)[0]))


@pytest.mark.gpu
@pytest.mark.parametrize("seed,p,forms", CASES)
def test_tiny_inputs_keep_their_value(cuda, tnq_lib, seed, p, forms):
    """complex64: about 30 buckets in sequence, each adding a few 2^-24 roundings."""
    plan, dims, sites = _plan(tnq_lib, seed, p)
    got = tnq_lib.contract_sliced(plan)
    scale = TINY ** len(sites)
    ref = onet.contract_network(dims, sites) * scale
    assert abs(got - ref) <= 1e-5 * max(abs(ref), onet.typical_magnitude(dims, sites) * scale)
