"""Workspace of small plans: what sufficed for their launches is accepted, and the sizes asked for grow by at most the
room of sixteen items."""
import ctypes

import numpy as np
import pytest

from paper_2004_10892_gb300 import inputs as I

MB = 1 << 20
# (rows, cols, depth, seed, plan options)
CASES = [
    (5, 5, 20, 3, dict(min_p=3, max_p=3)),
    (6, 6, 24, 0, dict(max_bag_log2=24, min_p=4, max_p=8)),
    (6, 6, 32, 0, dict(max_bag_log2=18, max_p=40)),
]


def _plan(tnq_lib, case):
    rows, cols, depth, seed, kw = case
    circ = I.random_grid_circuit(rows, cols, depth, seed)
    plan = tnq_lib.Plan(circ, **kw)
    assert _small(tnq_lib, plan, 1) == 1
    return circ, plan


def _small(tnq_lib, plan, use):
    f = tnq_lib.lib().tnq_internal_small
    f.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return f(plan.handle, use)


def _steps_bytes(tnq_lib, case, batch):
    plan = _plan(tnq_lib, case)[1]
    _small(tnq_lib, plan, 0)
    return plan.workspace_bytes(batch)


@pytest.mark.parametrize("case", CASES, ids=str)
def test_sizes(tnq_lib, case):
    plan = _plan(tnq_lib, case)[1]
    for batch in (1, 2, 8, 16, 64, 512, 1 << 14):
        steps, got = _steps_bytes(tnq_lib, case, batch), plan.workspace_bytes(batch)
        assert steps <= got <= max(steps, min(batch, 16) * (8 * MB + 1024))
    assert got == steps  # (many items: the launches' batch is the larger)


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES, ids=str)
def test_every_size_that_the_launches_accept(cuda, tnq_lib, case):
    import torch

    circ, plan = _plan(tnq_lib, case)
    bits = I.random_bitstring(circ.n_qubits, 3)
    n = min(40, plan.info()["n_slices"])
    ref = tnq_lib.contract_sliced(plan, bits, 0, n, per_slice=True)[1]
    room = plan.workspace_bytes(1)
    least = _steps_bytes(tnq_lib, case, 1)
    for size in sorted({least, _steps_bytes(tnq_lib, case, 8), room, 3 * room, 5 * room + 64}):
        ws = torch.full((size + 256,), 0xFF, dtype=torch.uint8, device="cuda")
        _, got = tnq_lib.contract_sliced(plan, bits, 0, n, workspace=ws[:size], per_slice=True)
        assert np.all(ws[size:].cpu().numpy() == 0xFF)
        if size >= room:  # one kernel: the same bits however many items are at once
            assert np.array_equal(got, ref)
        else:  # ~50 buckets of complex64 in another grouping
            assert np.max(np.abs(got - ref)) <= 1e-5 * np.max(np.abs(ref))
    with pytest.raises(tnq_lib.TnqError) as e:
        tnq_lib.contract_sliced(plan, bits, 0, n, workspace=torch.empty(least - 256, dtype=torch.uint8, device="cuda"))
    assert e.value.status == tnq_lib.ENOMEM


@pytest.mark.gpu
def test_batched_call_in_every_size(cuda, tnq_lib):
    import torch

    plans, bits = [], []
    for k, case in enumerate(CASES[:2]):
        circ, plan = _plan(tnq_lib, case)
        plans.append(plan)
        bits.append([I.random_bitstring(circ.n_qubits, 10 * k + j) for j in range(5)])
    ref = tnq_lib.amplitudes_batch(plans, bits)
    least = max(_steps_bytes(tnq_lib, case, 1) for case in CASES[:2])
    for size in (least + (1 << 14), 2 * least + (1 << 14), plans[1].workspace_bytes(1) + (1 << 14), 16 * MB):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        got = tnq_lib.amplitudes_batch(plans, bits, workspace=ws)
        assert np.max(np.abs(got - ref) / np.abs(ref)) <= 1e-5
