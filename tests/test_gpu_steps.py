"""The tests of chains, GEMMs, levels, autotuning, lanes and the allocation-free
steps, on plans that run step by step: small plans run as one kernel by default,
where these launches do not happen."""
import ctypes

import numpy as np
import pytest
import test_gpu_gemm
import test_gpu_network
import test_gpu_parity
import test_zz_no_alloc

from paper_2004_10892_gb300 import inputs as I

# (module, test, its arguments)
CASES = [
    (test_gpu_parity, "test_4x4_zero_amplitude", dict(seed=0)),
    (test_gpu_parity, "test_6x6_sliced_per_slice", dict(p=4)),
    (test_gpu_parity, "test_batch_size_does_not_change_slices", {}),
    (test_gpu_parity, "test_slice_sum_matches_unsliced", {}),
    (test_gpu_parity, "test_closed_forms_on_gpu", {}),
    (test_gpu_parity, "test_wire_without_nondiagonal_gate", {}),
    (test_gpu_parity, "test_tiny_amplitudes_are_rescaled", {}),
    (test_gpu_parity, "test_random_small_circuits_all_gates", {}),
    (test_gpu_parity, "test_uneven_batch_of_plans", {}),
    *[(test_gpu_parity, "test_fused_chains_match_oracle", dict(fuse=f)) for f in (1, 4, 8)],
    (test_gpu_parity, "test_fused_equals_unfused", {}),
    *[(test_gpu_parity, "test_leaf_absorption_matches_oracle", dict(fuse=f)) for f in (0, 12)],
    (test_gpu_parity, "test_autotune_keeps_results", {}),
    *[(test_gpu_parity, "test_split_precision_gemm_buckets_match_oracle", dict(precision=p)) for p in (1, 2)],
    *[(test_gpu_parity, "test_reordered_plans_match_oracle", dict(precision=p)) for p in (0, 1, 2)],
    (test_gpu_parity, "test_split_precision_agrees_with_c64", {}),
    *[(test_gpu_parity, "test_every_slicer_gives_the_same_amplitude", dict(slicer=s)) for s in (0, 4)],
    (test_gpu_parity, "test_autotuned_tuning_reproduces_and_matches_oracle", {}),
    (test_gpu_parity, "test_batched_call_lanes_duplicates_and_small_workspace", {}),
    (test_gpu_gemm, "test_fused_a_gemm_matches_packed_form_and_oracle", dict(case="6x6-24")),
    *[(test_gpu_network, "test_lattice_sliced_per_slice", dict(L=L, p=p)) for L, p in ((3, 4), (4, 5))],
    (test_gpu_network, "test_mixed_dimensions_and_torus", {}),
    *[(test_gpu_network, "test_degenerate_small_networks", dict(seed=s)) for s in (0, 3)],
    (test_gpu_network, "test_fused_chains_and_tiles_on_a_larger_lattice", {}),
    *[(test_gpu_network, "test_split_precision_network", dict(precision=p)) for p in (1, 2)],
    (test_zz_no_alloc, "test_noalloc_matches_workspace_entry_point_and_oracle", {}),
    (test_zz_no_alloc, "test_noalloc_second_plan_after_first", {}),
    (test_zz_no_alloc, "test_noalloc_split_precision_gemm_and_register_tail_steps", {}),
    (test_zz_no_alloc, "test_noalloc_allocates_no_device_memory", {}),
]


@pytest.fixture
def steps(tnq_lib, monkeypatch):
    """Every plan that a test makes runs step by step."""
    small = tnq_lib.lib().tnq_internal_small
    small.argtypes = [ctypes.c_void_p, ctypes.c_int]
    init, network = tnq_lib.Plan.__init__, tnq_lib.Plan.from_network

    def from_circuit(self, *args, **opts):
        init(self, *args, **opts)
        assert small(self.handle, 0) == 0

    def from_network(*args, **opts):
        plan = network(*args, **opts)
        assert small(plan.handle, 0) == 0
        return plan

    monkeypatch.setattr(tnq_lib.Plan, "__init__", from_circuit)
    monkeypatch.setattr(tnq_lib.Plan, "from_network", from_network)


@pytest.mark.gpu
@pytest.mark.parametrize("module,name,args", CASES, ids=[f"{n[5:]}-{'-'.join(map(str, a.values()))}" for _, n, a in CASES])
def test_step_by_step(request, steps, module, name, args):
    test = getattr(module, name)
    code = test.__code__
    given = {a: request.getfixturevalue(a) for a in code.co_varnames[: code.co_argcount] if a not in args}
    test(**given, **args)


@pytest.mark.gpu
def test_noalloc_batches_that_are_not_full(cuda, tnq_lib, steps):
    """GEMM and register-tail steps in the static array, 3, 5 and 6 of a batch of 4 or 8 items: the slices' bits."""
    circ = I.random_grid_circuit(5, 6, 24, 0)
    bits = I.random_bitstring(30, 0)
    plan = tnq_lib.Plan(circ, max_bag_log2=18, min_p=3, max_p=30, precision=1, gemm_min_k_log2=3, fuse_min_rank=8,
                        reorder_every=1)
    kinds, tails = test_zz_no_alloc._step_kinds(tnq_lib, plan)
    assert (kinds == 2).sum() >= 1 and (tails > 0).sum() >= 1
    ref = tnq_lib.contract_sliced_noalloc(plan, bits, per_slice=True)[1]
    want = tnq_lib.contract_sliced(plan, bits, per_slice=True)[1]
    assert np.array_equal(ref, want)
    for begin, end in ((0, 3), (2, 8), (1, 6)):
        assert np.array_equal(tnq_lib.contract_sliced_noalloc(plan, bits, begin, end, per_slice=True)[1], ref[begin:end])
