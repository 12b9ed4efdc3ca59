"""GPU parity for the kernel variants that only large launches select, each at the smallest shape that
still selects it, against the fp64 oracle on sampled (batch, head) units (units are independent end to
end, so the oracle run on a unit alone is that unit's exact reference):

  * the fold-decision kernels of states with more units than SMs;
  * the decode kernel's direct-output branch (one row split per head) at head_dim 128, with and without
    grouped queries;
  * config 5's structure at a batch wide enough to select the kernels that the full batch selects;
  * the minimum of two memory-key slots (one block of look-ahead), which very large batches run with;
  * what states that fill the GPU do: folds on the caller's stream with one readout copy, new-row products
    inside the decision kernel for folds that append few rows, memory keys recomputed from their fp16 copy.
"""
import numpy as np
import pytest
import torch

from paper_2605_09877_b200 import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


def _sampled(wl, units, params=None, gate=False, decode_from=None, flags=0):
    params = params or synth.make_layer_params(wl)
    tensors = synth.make_inputs(wl)
    if gate:
        tensors["gate"] = synth.make_gate(wl)
    y_gpu, st = pu.run_gpu(wl, tensors, params, decode_from=decode_from, flags=flags)
    y_ref, o = pu.run_oracle(wl, tensors, params, units=units)
    stats = pu.compare(wl, y_gpu, st, y_ref, o, units=units)
    stats["counters"] = st.debug_counters()
    st.free()
    return stats


def test_fold_decide_two_ctas_per_sm_variant_head_dim_128():
    """160 units x block 256 at head_dim 128, more units than SMs: folds that append rows take the bounds-first decision
    kernel (its 128-register build, two CTAs per SM); gates and affine LayerNorm included."""
    wl = synth.Workload("t", 1, 160, 160, 128, 4 * 256 + 70, 256, "sqrt", sqrt_coeff=14, r=32, seed=31, kind="mixture")
    params = synth.make_layer_params(wl, trivial=False)
    print(_sampled(wl, [(0, 0), (0, 37), (0, 101), (0, 148), (0, 159)], params=params, gate=True))


def test_decode_direct_output_branch_head_dim_128():
    """416 query heads need no row split: the decode kernel writes its output directly.  40 steps from position 1004
    cross the block boundary at 1024, so one of them folds."""
    from paper_2605_09877_b200 import kvm
    wl = synth.Workload("t", 13, 32, 32, 128, 1004 + 40, 256, "sqrt", r=0, seed=32)
    assert {kvm.decode_plan(13, 32, 32, 128, _decode_rows(wl, t)) for t in range(1004, wl.T)} == {(1, 1, 1)}
    print(_sampled(wl, [(0, 0), (7, 13), (12, 31)], decode_from=1004))


def test_decode_grouped_queries_direct_and_split():
    """Four query heads per kv head: 640 query heads (direct output) and 8 query heads (row splits)."""
    from paper_2605_09877_b200 import kvm
    wl = synth.Workload("t", 5, 128, 32, 128, 500 + 30, 128, "sqrt", r=32, seed=33)
    assert {kvm.decode_plan(5, 128, 32, 128, _decode_rows(wl, t)) for t in range(500, wl.T)} == {(4, 1, 1)}
    params = synth.make_layer_params(wl, trivial=False)
    print(_sampled(wl, [(0, 0), (2, 17), (4, 31)], params=params, decode_from=500))
    wl = synth.Workload("t", 1, 8, 2, 128, 700 + 30, 128, "sqrt", r=32, seed=34)
    assert all(kvm.decode_plan(1, 8, 2, 128, _decode_rows(wl, t))[1] > 1 for t in range(700, wl.T))
    print(_sampled(wl, [(0, 0), (0, 1)], decode_from=700))


def test_config5_structure_at_a_batch_that_selects_the_full_batch_kernels():
    """B8 x H32 = 256 units, block 256, sqrt growth, N(0,1) tokens, two prefill segments and a few decode
    steps: every kernel selection that depends on the number of units (decision kernel build, rows-per-warp
    apply, attention tail split, routing filter splits, decode without row splits) is the full batch's."""
    wl = synth.CONFIGS["cfg5"].scaled(B=8, T=3072 + 20)
    units = [(0, 0), (3, 9), (7, 31)]
    params = synth.make_layer_params(wl)
    tensors = synth.make_inputs(wl)
    y_gpu, st = pu.run_gpu(wl, tensors, params, cuts=[0, 2048, 3072], decode_from=3072)
    y_ref, o = pu.run_oracle(wl, tensors, params, units=units)
    print(pu.compare(wl, y_gpu, st, y_ref, o, units=units))
    st.free()


def test_two_memory_key_slots_one_block_of_look_ahead():
    """With only two memory-key slots every fold's keys are computed while the fold before it runs, and a
    slot is rewritten as soon as its fold is done: routing must still see its own block's keys."""
    from paper_2605_09877_b200 import kvm
    wl = synth.CONFIGS["cfg3"].scaled(Hq=3, Hkv=3, T=256 * 12 + 31)
    print(_sampled(wl, None, flags=kvm.FLAG_MIN_KEY_SLOTS))
    wl = synth.CONFIGS["cfg2"].scaled(B=2, Hq=2, Hkv=2, T=128 * 14)
    print(_sampled(wl, None, flags=kvm.FLAG_MIN_KEY_SLOTS, gate=True))


def test_serial_folds_one_readout_copy():
    """What states of 256 or more units do by themselves, forced on small shapes: folds on the caller's stream
    between the attention launches, one readout copy written in place; segmented prefill, gates, decode with a
    fold."""
    from paper_2605_09877_b200 import kvm
    wl = synth.CONFIGS["cfg3"].scaled(Hq=3, Hkv=3, T=256 * 9 + 31)
    print(_sampled(wl, None, flags=kvm.FLAG_SERIAL_FOLDS))
    wl = synth.Workload("t", 2, 4, 2, 128, 128 * 11 + 40, 128, "fixed", fixed_slots=400, r=32, seed=35)
    params = synth.make_layer_params(wl, trivial=False)
    tensors = synth.make_inputs(wl)
    tensors["gate"] = synth.make_gate(wl)
    y_gpu, st = pu.run_gpu(wl, tensors, params, cuts=[0, 300, 1000, 128 * 11], decode_from=128 * 11, flags=kvm.FLAG_SERIAL_FOLDS)
    y_ref, o = pu.run_oracle(wl, tensors, params)
    print(pu.compare(wl, y_gpu, st, y_ref, o))
    st.free()


def test_small_appends_compute_their_products_in_the_decision_kernel_and_keys_are_recomputed():
    """Serial states: a fold that appends at most 32 rows computes the products of its new rows with the block's
    keys itself (here every fold after the first: 4 sqrt(N) slots), larger ones use the batched launch (the
    second case, 16 sqrt(N): both kinds in one run).  64 units x block 128 is also the size from which no fp64
    memory keys are kept: every fp64 key the fold kernels use is recomputed from the fp16 key and the token's
    LayerNorm statistics.  Exact slots against the oracle say that the recomputed keys equal the stored ones."""
    from paper_2605_09877_b200 import kvm
    wl = synth.Workload("t", 2, 32, 32, 128, 128 * 12 + 31, 128, "sqrt", sqrt_coeff=4, r=32, seed=36)
    params = synth.make_layer_params(wl, trivial=False)
    stats = _sampled(wl, [(0, 0), (0, 19), (1, 7), (1, 31)], params=params, gate=True, flags=kvm.FLAG_SERIAL_FOLDS)
    print(stats)
    wl = synth.Workload("t", 2, 32, 32, 128, 128 * 40 + 77, 128, "sqrt", sqrt_coeff=16, r=32, seed=37, kind="mixture")
    print(_sampled(wl, [(0, 3), (1, 30)], flags=kvm.FLAG_SERIAL_FOLDS, decode_from=128 * 40 + 40))
    # the same small-append shape below the size threshold keeps its fp64 keys: products inside the kernel only
    wl = synth.Workload("t", 1, 3, 3, 64, 64 * 14 + 9, 64, "sqrt", sqrt_coeff=3, r=16, seed=38)
    print(_sampled(wl, None, flags=kvm.FLAG_SERIAL_FOLDS))


def test_bounds_first_decisions_head_dim_64_three_sink_rows_duplicated_keys():
    """More units than SMs: the decision kernel that ranks the tokens by the filter's bounds first and scores
    only the ones in doubt.  Head dimension 64, three sink rows (a sink row in reach takes a token's bounds
    away), mixture keys (near-duplicates inside a block: new rows in reach of many tokens), with the batched
    new-row products and with the products computed inside the kernel."""
    from paper_2605_09877_b200 import kvm
    wl = synth.Workload("t", 1, 160, 160, 64, 64 * 11 + 20, 64, "sqrt", sqrt_coeff=5, r=16, seed=39, kind="mixture", S=3)
    params = synth.make_layer_params(wl, trivial=False)
    units = [(0, 0), (0, 77), (0, 159)]
    print(_sampled(wl, units, params=params, gate=True))
    print(_sampled(wl, units, params=params, gate=True, flags=kvm.FLAG_SERIAL_FOLDS))
    wl = synth.Workload("t", 5, 32, 32, 128, 128 * 9 + 3, 128, "fixed", fixed_slots=300, r=32, seed=40, S=2)
    print(_sampled(wl, [(0, 0), (3, 11), (4, 31)], flags=kvm.FLAG_SERIAL_FOLDS))


def test_bounds_first_decisions_with_exactly_tied_scores():
    """More units than SMs, every key of a sequence equal (all similarities tie exactly) or every key repeated in
    the next block half (ties in pairs): the bounds decide nothing, every token is scored, and appended tokens,
    rows and merge targets must follow the tie rules (smaller token, lowest row) as in the oracle."""
    wl = synth.Workload("t", 1, 160, 160, 64, 32 * 9 + 5, 32, "sqrt", sqrt_coeff=3, r=0, seed=41)
    params = synth.make_layer_params(wl)
    units = [(0, 0), (0, 80), (0, 159)]
    tensors = synth.make_inputs(wl)
    tensors["k"] = torch.full_like(tensors["k"], 0.5)
    y_gpu, st = pu.run_gpu(wl, tensors, params)
    y_ref, o = pu.run_oracle(wl, tensors, params, units=units)
    print(pu.compare(wl, y_gpu, st, y_ref, o, units=units))
    st.free()
    tensors = synth.make_inputs(wl)
    k = tensors["k"]
    for b0 in range(0, wl.T - 31, 32):   # second half of every block repeats the first half
        k[:, :, b0 + 16:b0 + 32] = k[:, :, b0:b0 + 16]
    y_gpu, st = pu.run_gpu(wl, tensors, params)
    y_ref, o = pu.run_oracle(wl, tensors, params, units=units)
    print(pu.compare(wl, y_gpu, st, y_ref, o, units=units))
    st.free()


def test_many_units_run_to_run_and_across_variants_identical_bits():
    """256 units (bounds-first decisions, one readout copy, recomputed memory keys, one apply CTA per unit): three
    runs give identical bits, and the same problem run as 160 + 96 units in two states leaves the same state bit
    for bit (units are independent: the fold kernels chosen by the number of units must not change any unit's
    sums or counts)."""
    wl = synth.Workload("t", 8, 32, 32, 128, 256 * 6 + 77, 256, "sqrt", sqrt_coeff=12, r=32, seed=42, kind="mixture")
    tensors = synth.make_inputs(wl)
    params = synth.make_layer_params(wl)
    outs = []
    for _ in range(3):
        y, st = pu.run_gpu(wl, tensors, params)
        e = st.export()
        outs.append((y, e["sum_k"].copy(), e["sum_v"].copy(), e["count"].copy()))
        st.free()
    for y, sk, sv, c in outs[1:]:
        assert torch.equal(y, outs[0][0]) and np.array_equal(sk, outs[0][1]) and np.array_equal(sv, outs[0][2])
    # batch rows 0-4 (160 units: bounds-first kernel, two readout copies) and 5-7 (96 units: sliced decision kernel)
    for lo, hi in ((0, 5), (5, 8)):
        sub = wl.scaled(B=hi - lo)
        t = {k: v[lo:hi].contiguous() for k, v in tensors.items()}
        y, st = pu.run_gpu(sub, t, params)
        e = st.export()
        U0, U1 = lo * wl.Hkv, hi * wl.Hkv
        # (the attention launch may cut the last wave's tiles along the keys at one size and not at the other:
        #  outputs agree to the rounding of a different summation order, the state bit for bit)
        assert (y.float() - outs[0][0][lo:hi].float()).abs().max() <= 2e-2
        assert np.array_equal(e["sum_k"], outs[0][1][U0:U1]) and np.array_equal(e["sum_v"], outs[0][2][U0:U1])
        assert np.array_equal(e["count"], outs[0][3][U0:U1])
        st.free()


_SWEEP = [
    # (B, Hq, Hkv, d, C, blocks, extra, growth kwargs, r, S, w, kind, flags_serial, gate, decode)
    (5, 32, 32, 64, 16, 14, 3, dict(growth="sqrt", sqrt_coeff=2), 0, 0, 2, "normal", False, False, 0),
    (3, 64, 64, 64, 32, 10, 9, dict(growth="fixed", fixed_slots=96), 16, 2, 3, "mixture", True, True, 12),
    (10, 32, 16, 128, 64, 8, 1, dict(growth="power", sqrt_coeff=6, pow_num=2, pow_den=3), 32, 1, 2, "scaled_keys", False, True, 0),
    (6, 32, 32, 128, 128, 7, 50, dict(growth="saturating", fixed_slots=400, sat_half=600), 0, 4, 2, "needles", True, False, 20),
    (20, 8, 8, 64, 64, 9, 0, dict(growth="sqrt", sqrt_coeff=9), 16, 1, 4, "mixture", True, False, 0),
    (1, 150, 150, 128, 256, 4, 17, dict(growth="sqrt", sqrt_coeff=16), 32, 1, 2, "normal", True, True, 0),
]


@pytest.mark.parametrize("case", range(len(_SWEEP)))
def test_shape_sweep_with_more_units_than_sms(case):
    """Seeded sweep over the shapes the many-unit kernels meet: head dimension, block length from 16 to 256, every
    budget rule, sink rows from 0 to 4, window lengths, grouped queries, gates, rotary dimensions, with and without
    the serial-fold flag, prefill followed by decode steps; sampled units against the oracle."""
    from paper_2605_09877_b200 import kvm
    B, Hq, Hkv, d, C, nb, extra, gk, r, S, w, kind, serial, gate, dec = _SWEEP[case]
    T = C * nb + extra + dec
    wl = synth.Workload("sweep", B, Hq, Hkv, d, T, C, r=r, S=S, w=w, seed=100 + case, kind=kind, **gk)
    assert B * Hkv > 148
    params = synth.make_layer_params(wl, trivial=(case % 2 == 0))
    units = [(0, 0), (B // 2, Hkv // 2), (B - 1, Hkv - 1)]
    stats = _sampled(wl, units, params=params, gate=gate, decode_from=(T - dec) if dec else None,
                     flags=kvm.FLAG_SERIAL_FOLDS if serial else 0)
    print(case, stats)


_DECIDE = [
    # (B, Hq, Hkv, d, C, blocks, extra, growth kwargs, r, S, w, kind, flags_serial, gate)
    (1, 1, 1, 64, 16, 12, 5, dict(growth="sqrt", sqrt_coeff=3), 0, 0, 2, "normal", False, False),          # one CTA
    (1, 1, 1, 128, 256, 9, 1, dict(growth="sqrt", sqrt_coeff=16), 32, 1, 2, "mixture", False, True),       # eight CTAs
    (1, 3, 3, 64, 136, 10, 40, dict(growth="fixed", fixed_slots=200), 16, 4, 3, "needles", False, True),   # slices of 17
    (3, 6, 3, 128, 200, 7, 0, dict(growth="power", sqrt_coeff=6, pow_num=2, pow_den=3), 0, 0, 1, "scaled_keys", False, False),
    (2, 20, 10, 64, 72, 11, 3, dict(growth="saturating", fixed_slots=300, sat_half=400), 0, 1, 2, "mixture", True, True),
    (4, 10, 10, 128, 256, 5, 9, dict(growth="sqrt", sqrt_coeff=20), 32, 2, 2, "normal", True, False),      # keys recomputed
    (5, 15, 15, 64, 104, 6, 0, dict(growth="fixed", fixed_slots=104), 0, 1, 2, "normal", False, False),    # one CTA per unit
    (4, 37, 37, 64, 48, 6, 7, dict(growth="sqrt", sqrt_coeff=5), 16, 1, 2, "mixture", False, True),        # 148 units
    (10, 15, 15, 64, 48, 8, 0, dict(growth="fixed", fixed_slots=64), 0, 2, 2, "normal", False, True),      # decisions alone
]


@pytest.mark.parametrize("case", range(len(_DECIDE)))
def test_decisions_over_cluster_sizes_and_slices(case):
    """One to eight CTAs per unit, slices of the block that are no multiple of a warp, every budget rule, full states
    that append nothing, one and two readout copies, up to 150 units."""
    from paper_2605_09877_b200 import kvm
    B, Hq, Hkv, d, C, nb, extra, gk, r, S, w, kind, serial, gate = _DECIDE[case]
    wl = synth.Workload("step", B, Hq, Hkv, d, C * nb + extra, C, r=r, S=S, w=w, seed=300 + case, kind=kind, **gk)
    params = synth.make_layer_params(wl, trivial=(case % 2 == 0))
    units = [(0, 0), (B // 2, Hkv // 2), (B - 1, Hkv - 1)]
    print(case, _sampled(wl, units, params=params, gate=gate, flags=kvm.FLAG_SERIAL_FOLDS if serial else 0))


def test_decisions_scan_every_row_for_tokens_with_too_many_candidates():
    """Keys repeated over whole blocks: most rows of the state tie, the filter's lists overflow, and the tokens are
    scored against every row (and, where rows are appended, against every new row)."""
    wl = synth.Workload("t", 1, 4, 4, 64, 64 * 8 + 3, 64, "sqrt", sqrt_coeff=8, r=0, S=2, seed=320)
    tensors = synth.make_inputs(wl)
    tensors["k"][:, 0] = tensors["k"][:, 0, :1]                        # one key
    for j in range(wl.T):
        tensors["k"][:, 1, j] = tensors["k"][:, 1, j % 3]             # three keys in turn
    tensors["k"][:, 2, 64:] = tensors["k"][:, 2, 64:65]
    params = synth.make_layer_params(wl)
    y_gpu, st = pu.run_gpu(wl, tensors, params)
    y_ref, o = pu.run_oracle(wl, tensors, params)
    print(pu.compare(wl, y_gpu, st, y_ref, o))
    assert st.debug_counters()["exhaustive_tokens"] > 0
    st.free()


def _decode_rows(wl, t):
    """State rows and window tokens that the decode step at position t attends over."""
    from paper_2605_09877_b200 import kvm
    g = kvm.growth(wl.growth, wl.fixed_slots, wl.sqrt_coeff, wl.pow_num, wl.pow_den, wl.sat_half)
    return kvm.kvm_plan_capacity(wl.C, wl.w, g, t // wl.C * wl.C) + t + 1 - max(0, (t // wl.C + 1 - wl.w) * wl.C)


@pytest.mark.parametrize("B,Hq,Hkv,d,pos,steps,plans", [
    (1, 1, 1, 64, 40, 30, {(1, 1, 1)}), (1, 2, 1, 128, 900, 20, {(2, 6, 1)}), (3, 32, 4, 64, 1300, 10, {(4, 7, 1)}),
    (7, 21, 21, 128, 300, 9, {(1, 2, 1)}), (9, 64, 64, 64, 700, 6, {(1, 1, 1)}), (40, 32, 8, 128, 300, 4, {(4, 1, 1)}),
    (1, 1, 1, 128, 60, 20, {(1, 1, 1), (1, 2, 1)}), (1, 2, 2, 128, 110, 10, {(1, 2, 1)}), (1, 3, 3, 64, 400, 5, {(1, 4, 1)}),
    (1, 1, 1, 64, 1000, 5, {(1, 6, 1)}), (1, 2, 2, 128, 260, 5, {(1, 5, 1)}),
    (1, 2, 2, 128, 452, 5, {(1, 8, 1)}), (6, 32, 16, 128, 70, 8, {(2, 2, 1)}), (10, 32, 8, 64, 500, 5, {(4, 2, 1)}),
    (5, 32, 4, 64, 20, 5, {(8, 1, 1)}), (5, 32, 4, 128, 130, 8, {(8, 3, 1)}), (12, 32, 4, 128, 300, 5, {(8, 2, 1)}),
    (5, 32, 4, 128, 392, 5, {(8, 4, 1)}), (1, 2, 2, 128, 392, 5, {(1, 7, 1)})])
def test_decode_row_splits_from_one_to_eight(B, Hq, Hkv, d, pos, steps, plans):
    """One to eight CTAs in the cluster of a group of heads, one to eight query heads per CTA: how the looping kernel cuts these
    steps.  Those of few heads run the kernel that fetches its rows ahead (test_kernels_of_the_row_split_cases)."""
    from paper_2605_09877_b200 import kvm
    wl = synth.Workload("dec", B, Hq, Hkv, d, pos + steps, 64, "sqrt", sqrt_coeff=20, r=32, seed=330 + pos)
    assert {kvm.decode_plan(B, Hq, Hkv, d, _decode_rows(wl, t)) for t in range(pos, pos + steps)} == plans
    params = synth.make_layer_params(wl, trivial=False)
    print(_sampled(wl, [(0, 0), (B - 1, Hkv - 1)], params=params, decode_from=pos))


def _decode_kernels(B, Hq, Hkv, d, rows):
    """What the decode steps over these numbers of rows run: ("ahead", query heads per CTA, CTAs per cluster) or (query heads per CTA,
    CTAs per cluster, clusters) of the kernel that loops over its rows."""
    from paper_2605_09877_b200 import kvm
    ahead = {n: kvm.decode_ahead(B, Hq, Hkv, d, n) for n in rows}
    return {("ahead", a[1], a[0]) if a[0] else kvm.decode_plan(B, Hq, Hkv, d, n) for n, a in ahead.items()}


@pytest.mark.parametrize("B,Hq,Hkv,d,pos,steps,kernels", [
    (1, 1, 1, 64, 40, 30, {("ahead", 1, 1)}), (1, 2, 1, 128, 900, 20, {("ahead", 2, 6)}), (3, 32, 4, 64, 1300, 10, {("ahead", 2, 4)}),
    (7, 21, 21, 128, 300, 9, {(1, 2, 1)}), (9, 64, 64, 64, 700, 6, {(1, 1, 1)}), (40, 32, 8, 128, 300, 4, {(4, 1, 1)}),
    (1, 1, 1, 128, 60, 20, {("ahead", 1, 1)}), (1, 2, 2, 128, 110, 10, {("ahead", 1, 1)}), (1, 3, 3, 64, 400, 5, {("ahead", 1, 2)}),
    (1, 1, 1, 64, 1000, 5, {("ahead", 1, 3)}), (1, 2, 2, 128, 260, 5, {("ahead", 1, 3)}),
    (1, 2, 2, 128, 452, 5, {("ahead", 1, 4)}), (6, 32, 16, 128, 70, 8, {("ahead", 2, 1)}), (10, 32, 8, 64, 500, 5, {(4, 2, 1)}),
    (5, 32, 4, 64, 20, 5, {("ahead", 2, 1)}), (5, 32, 4, 128, 130, 8, {("ahead", 2, 2)}), (12, 32, 4, 128, 300, 5, {(8, 2, 1)}),
    (5, 32, 4, 128, 392, 5, {(8, 4, 1)}), (1, 2, 2, 128, 392, 5, {("ahead", 1, 4)})])
def test_kernels_of_the_row_split_cases(B, Hq, Hkv, d, pos, steps, kernels):
    """What the steps of test_decode_row_splits_from_one_to_eight run."""
    wl = synth.Workload("dec", B, Hq, Hkv, d, pos + steps, 64, "sqrt", sqrt_coeff=20, r=32, seed=330 + pos)
    assert _decode_kernels(B, Hq, Hkv, d, {_decode_rows(wl, t) for t in range(pos, pos + steps)}) == kernels


@pytest.mark.parametrize("B,Hq,Hkv,d,serial", [(1, 2, 1, 64, False), (1, 4, 4, 128, False), (2, 8, 2, 128, True)])
def test_decode_steps_launched_back_to_back_equal_steps_one_at_a_time(B, Hq, Hkv, d, serial):
    """A step is on the GPU while the one before it stores its token, and while a fold rewrites readout rows: every slot
    of the window ring is reused several times, and the outputs are those of steps that are waited for one by one."""
    from paper_2605_09877_b200 import kvm
    wl = synth.Workload("pdl", B, Hq, Hkv, d, 40 + 16 * 13, 16, "sqrt", sqrt_coeff=5, r=16, seed=360 + Hq)
    params = synth.make_layer_params(wl, trivial=False)
    t = {n: x.cuda() for n, x in synth.make_inputs(wl).items() if n in "qkv"}
    outs = []
    for wait in (False, True):
        st, g = pu.gpu_layer(wl, params, flags=kvm.FLAG_SERIAL_FOLDS if serial else 0)
        st.prefill(t["q"][:, :, :40], t["k"][:, :, :40], t["v"][:, :, :40], wl.C, g, wl.r)
        steps = [[t[n][:, :, i].contiguous() for n in "qkv"] for i in range(40, wl.T)]
        y = [torch.empty_like(s[0]) for s in steps]
        torch.cuda.synchronize()
        for s, o in zip(steps, y):
            st.decode_step(*s, out=o)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert st.check() == 0
        outs.append(torch.stack(y))
        st.free()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("B,Hq,Hkv,d,slots,clusters", [
    (1, 1, 1, 128, 3000, 7), (1, 8, 1, 128, 2500, 6), (1, 4, 2, 128, 4000, 9), (1, 2, 2, 64, 9000, 10), (1, 32, 8, 128, 4200, 3),
    (2, 8, 8, 64, 9000, 3), (1, 16, 1, 64, 6000, 7), (1, 64, 8, 128, 4200, 2)])
def test_decode_clusters_of_the_same_heads_merge_through_global_memory(B, Hq, Hkv, d, slots, clusters):
    """Few heads over many rows: one to four query heads per CTA, an odd number of clusters, the last ones with few rows or
    none; steps across a block boundary, with a fold between them, against the oracle and from run to run."""
    from paper_2605_09877_b200 import kvm
    C = 256
    start = (slots // C + 4) * C - 5
    wl = synth.Workload("far", B, Hq, Hkv, d, start + 9, C, "fixed", fixed_slots=slots, r=32, seed=370 + slots)
    got = {kvm.decode_plan(B, Hq, Hkv, d, slots + n)[1:] for n in (2 * C - 5, 2 * C, C + 1, C + 4)}
    assert all(s == 8 and c > 1 for s, c in got) and any(c == clusters for _, c in got), got
    params = synth.make_layer_params(wl, trivial=False)
    tensors = synth.make_inputs(wl)
    ys = []
    for _ in range(2):
        y, st = pu.run_gpu(wl, tensors, params, decode_from=start)
        ys.append(y)
        if len(ys) == 1:
            units = [(0, 0), (B - 1, Hkv - 1)]
            y_ref, o = pu.run_oracle(wl, tensors, params, units=units)
            print(pu.compare(wl, y, st, y_ref, o, units=units))
        st.free()
    assert torch.equal(ys[0], ys[1])


@pytest.mark.parametrize("B,Hq,Hkv,d,C,T,slots", [(1, 3, 3, 128, 64, 1500, 700), (8, 32, 32, 64, 64, 1111, 200), (4, 128, 64, 128, 128, 1400, 300)])
def test_kernels_that_start_under_the_ones_before_equal_kernels_one_at_a_time(B, Hq, Hkv, d, C, T, slots):
    """One readout copy: attention under the end of the fold, the routing filter under the attention.  With the timing hook on
    nothing starts early; outputs, sums, rows and the slots of all tokens are the same, in calls of whole and of odd pieces."""
    from paper_2605_09877_b200 import kvm
    wl = synth.Workload("early", B, Hq, Hkv, d, T, C, "fixed", fixed_slots=slots, r=32, seed=400 + B, kind="mixture")
    params = synth.make_layer_params(wl, trivial=False)
    t = {n: x.cuda() for n, x in synth.make_inputs(wl).items() if n in "qkv"}
    outs = []
    for hook in (True, False, False):
        st, g = pu.gpu_layer(wl, params, flags=kvm.FLAG_SERIAL_FOLDS)
        st.profile_enable(hook)
        y = torch.zeros_like(t["q"])
        for a, z in ((0, 5 * C), (5 * C, 7 * C + 13), (7 * C + 13, T)):
            st.prefill(t["q"][:, :, a:z], t["k"][:, :, a:z], t["v"][:, :, a:z], C, g, wl.r, out=y[:, :, a:z])
        torch.cuda.synchronize()
        assert st.check() == 0
        e = st.export()
        outs.append([y.cpu().view(torch.int16).numpy(), e["sum_k"], e["sum_v"], e["k_read"].view(torch.int16).numpy(), e["v_read"].view(torch.int16).numpy()] + list(st.assignments()))
        st.free()
    for o in outs[1:]:
        for a, b in zip(outs[0], o):
            assert np.array_equal(a, b)


def _equal_keys(wl, where):
    """Inputs in which the tokens `where(position in block)` of every block have one and the same key per head."""
    tensors = synth.make_inputs(wl)
    pos = [t for t in range(wl.T) if where(t % wl.C)]
    tensors["k"][:, :, pos] = tensors["k"][:, :, :1].clone()
    return tensors


@pytest.mark.parametrize("B,Hkv,d,C,T,kind", [
    (1, 1, 64, 256, 256 * 9 + 3, dict(growth="sqrt", sqrt_coeff=16)),      # eight CTAs per unit
    (1, 9, 128, 256, 256 * 7, dict(growth="sqrt", sqrt_coeff=20)),         # four
    (1, 1, 128, 128, 128 * 12, dict(growth="fixed", fixed_slots=300)),     # eight, nothing appended
    (1, 20, 64, 64, 64 * 9 + 1, dict(growth="fixed", fixed_slots=150)),    # two, nothing appended
    (2, 20, 64, 64, 64 * 9 + 1, dict(growth="fixed", fixed_slots=150)),    # one, nothing appended
    (2, 20, 64, 256, 256 * 6, dict(growth="sqrt", sqrt_coeff=16)),         # two
    (4, 25, 64, 256, 256 * 6, dict(growth="sqrt", sqrt_coeff=16)),         # one CTA per unit
    (10, 16, 64, 128, 128 * 8, dict(growth="fixed", fixed_slots=128)),     # more units than SMs, nothing appended
])
def test_runs_of_equal_keys_in_one_slice_of_the_block(B, Hkv, d, C, T, kind):
    """The tokens whose candidate lists overflow are neighbours, all in the slice of one CTA (and of one or two of its warps); the
    other CTAs of the unit have none.  Scores, targets and slots against the oracle."""
    wl = synth.Workload("runs", B, Hkv, Hkv, d, T, C, r=0, S=1, seed=410 + Hkv, **kind)
    params = synth.make_layer_params(wl)
    for lo, hi in ((0, 16), (C - 21, C)):
        tensors = _equal_keys(wl, lambda p: lo <= p < hi)
        y_gpu, st = pu.run_gpu(wl, tensors, params)
        units = [(0, 0), (B - 1, Hkv - 1)]
        y_ref, o = pu.run_oracle(wl, tensors, params, units=units)
        print(pu.compare(wl, y_gpu, st, y_ref, o, units=units))
        assert st.debug_counters()["exhaustive_tokens"] > 0
        st.free()


@pytest.mark.parametrize("units", [1, 40, 100])
def test_runs_of_equal_keys_cost_what_scattered_ones_cost(units):
    """Sixteen tokens of every block scan the state: neighbours (one or two warps' own tokens) or one every sixteen tokens
    (one per warp).  The same number of scans, dealt over all warps of the unit: about the same time (ten times more for
    the neighbours when every warp scanned for its own tokens)."""
    from paper_2605_09877_b200 import kvm
    wl = synth.Workload("deal", 1, units, units, 64, 256 * 14, 256, "fixed", fixed_slots=1500, r=0, seed=430)
    ms = []
    for where in (lambda p: p < 16, lambda p: p % 16 == 0):
        t = {n: x.cuda() for n, x in _equal_keys(wl, where).items() if n in "qkv"}
        st, g = pu.gpu_layer(wl, {})
        best = float("inf")
        for _ in range(3):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            st.reset()
            a.record()
            st.prefill(t["q"], t["k"], t["v"], wl.C, g, 0)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
        assert st.check() == 0 and st.debug_counters()["exhaustive_tokens"] > 100 * units
        st.free()
    print(units, ms)
    assert ms[0] < 2 * ms[1], ms


@pytest.mark.parametrize("Hkv,d,C", [(80, 64, 256), (148, 64, 256), (100, 128, 128), (160, 64, 256), (40, 64, 256), (9, 128, 256), (1, 64, 256)])
def test_crowded_runs_are_compared_pair_by_pair(Hkv, d, C):
    """Every key of a block occurs eight times, the same keys in every block: each token has eight candidate rows, the most that
    a list holds, and up to sixteen neighbouring tokens share a warp's list.  None is scanned against every row."""
    wl = synth.Workload("crowd", 1, Hkv, Hkv, d, C * 6 + 5, C, "fixed", fixed_slots=C, r=0, S=1, seed=440 + Hkv)
    tensors = synth.make_inputs(wl)
    tensors["k"] = tensors["k"][:, :, torch.arange(wl.T) % C // 8 * 8].clone()
    y_gpu, st = pu.run_gpu(wl, tensors, synth.make_layer_params(wl))
    units = [(0, 0), (0, Hkv - 1)]
    y_ref, o = pu.run_oracle(wl, tensors, synth.make_layer_params(wl), units=units)
    print(pu.compare(wl, y_gpu, st, y_ref, o, units=units), st.debug_counters())
    assert st.debug_counters()["exhaustive_tokens"] == 0
    st.free()


@pytest.mark.parametrize("B,Hkv,d,C,slots,rows4", [
    (1, 3, 128, 256, 64, False),    # one row per warp: four members a row on average, many rows with more than a batch of four
    (1, 2, 64, 200, 24, False),
    (2, 9, 128, 64, 1, False),      # every token of a block joins one of the 64 rows of the first fold
    (3, 24, 128, 256, 300, True),   # four rows per warp with stored memory keys
    (2, 25, 64, 256, 256, True),
    (5, 32, 64, 192, 64, True),     # (four CTAs per unit)
    (2, 24, 64, 128, 90, True),
    (1, 47, 64, 128, 300, False),
])
def test_rows_with_many_members_in_both_apply_kernels(B, Hkv, d, C, slots, rows4):
    """The kernel that a state's folds run to write the touched rows, at rows with none, one and many members, appended rows
    among them; the state means and readout rows against the oracle."""
    rows = C * B * Hkv
    assert rows4 == ((rows > 12288 if C > 128 else rows >= 6144) if d == 64 else C > 128 and rows > 16384 and B * Hkv < 128)
    wl = synth.Workload("t", B, Hkv, Hkv, d, C * 5 + 11, C, "fixed", fixed_slots=slots, r=32, seed=61, kind="mixture")
    params = synth.make_layer_params(wl, trivial=False)
    units = sorted({(0, 0), (B - 1, Hkv - 1)})
    stats = _sampled(wl, units, params=params, gate=True)
    print(stats)


@pytest.mark.parametrize("B,Hkv,d,C,slots,rows_per_warp,run", [
    (1, 3, 128, 256, 64, 1, False), (1, 2, 64, 200, 24, 1, False), (2, 9, 128, 64, 1, 1, False), (3, 24, 128, 256, 300, 1, False),
    (2, 25, 64, 256, 256, 4, False), (5, 32, 64, 192, 64, 4, False), (2, 24, 64, 128, 90, 4, False), (1, 47, 64, 128, 300, 1, False),
    (1, 36, 64, 256, 256, 4, True),   # eight CTAs per unit
    (2, 34, 64, 136, 100, 4, True)])
def test_rows_per_warp_of_states_with_many_members(B, Hkv, d, C, slots, rows_per_warp, run):
    """Which of the two kernels the library takes, for the cases of the test above too, which holds a rule of its own; the others run."""
    from paper_2605_09877_b200 import kvm
    assert kvm.apply_plan(B * Hkv, d, C)[0] == rows_per_warp
    if run:
        wl = synth.Workload("t", B, Hkv, Hkv, d, C * 5 + 11, C, "fixed", fixed_slots=slots, r=32, seed=61, kind="mixture")
        print(_sampled(wl, [(0, 0), (B - 1, Hkv - 1)], params=synth.make_layer_params(wl, trivial=False), gate=True))


@pytest.mark.parametrize("Hq,Hkv,d,blocks", [(8, 8, 128, 21), (16, 4, 128, 22), (24, 8, 64, 23), (3, 3, 128, 25)])
def test_attention_of_few_heads_over_many_rows_splits_the_keys(Hq, Hkv, d, blocks):
    """Key splits of launches of 6 to 48 tiles over 10 to 40 key tiles: two to eight splits, ragged last ones."""
    wl = synth.Workload("t", 1, Hq, Hkv, d, 256 * blocks + 70, 256, "unbounded", r=32, seed=62)
    print(_sampled(wl, [(0, 0), (0, Hkv - 1)]))


@pytest.mark.parametrize("Hq,Hkv,d,blocks,splits", [
    (8, 8, 128, 21, {1, 2, 3, 4, 5}), (16, 4, 128, 22, {1, 2, 3}), (24, 8, 64, 23, {1, 2}), (3, 3, 128, 25, {1, 2, 3, 4, 5, 6})])
def test_key_splits_of_the_cases_with_few_heads_over_many_rows(Hq, Hkv, d, blocks, splits):
    """The splits that the test above meets: 6 to 48 tiles over 1 to 49 key tiles."""
    from paper_2605_09877_b200 import kvm
    assert {kvm.attention_plan(1, Hq, Hkv, d, 256, 256 * max(b - 1, 0), decides=False)[1] for b in range(blocks + 1)} == splits


def _short_splits(n_q, group, d, n):
    """CTAs per cluster of the decode kernel that fetches its rows ahead (0: the step is not one of its)."""
    groups, cta = (n_q // 2 if group % 2 == 0 else n_q), 64 * (256 // d)
    fit = (296, 148, 88, 71, 56, 45, 37, 33)
    if groups > fit[0] or n > 16 * cta:
        return 0
    ns = -(-n // cta)
    ns = 8 if ns > 8 or 8 <= groups <= 16 else ns
    return ns if groups <= fit[ns - 1] else 0


@pytest.mark.parametrize("Hq,Hkv,d,C,slots,r,splits", [
    (1, 1, 64, 16, 40, 0, {1}), (3, 1, 128, 16, 80, 32, {1}), (2, 2, 128, 32, 170, 32, {2}), (2, 1, 128, 64, 300, 64, {3, 4}),
    (5, 5, 64, 64, 960, 16, {4, 5}), (4, 2, 128, 64, 600, 0, {6}), (3, 3, 128, 64, 700, 32, {6, 7}), (12, 12, 64, 32, 300, 0, {8}),
    (24, 12, 128, 64, 900, 32, {8}), (33, 33, 128, 64, 930, 0, {8}),
    (2, 2, 128, 64, 1500, 32, {8}), (1, 1, 64, 256, 3500, 0, {8}), (66, 33, 64, 64, 2700, 32, {8}),   # two passes over a warp's rows
])
def test_decode_steps_that_fetch_their_rows_ahead(Hq, Hkv, d, C, slots, r, splits):
    """One to eight CTAs per group of heads, one and two passes, warps with few rows or none; steps back to back across a fold, of
    which each fetches what the ones before leave complete, against the oracle and against steps that are waited for."""
    start = (slots // C + 4) * C - 6
    wl = synth.Workload("short", 1, Hq, Hkv, d, start + 14, C, "fixed", fixed_slots=slots, r=r, seed=400 + slots)
    assert {_short_splits(Hq, Hq // Hkv, d, _decode_rows(wl, t)) for t in range(start, wl.T)} <= splits
    params = synth.make_layer_params(wl, trivial=False)
    tensors = synth.make_inputs(wl)
    y, st = pu.run_gpu(wl, tensors, params, decode_from=start)
    units = sorted({(0, 0), (0, Hkv - 1)})
    y_ref, o = pu.run_oracle(wl, tensors, params, units=units)
    print(pu.compare(wl, y, st, y_ref, o, units=units))
    st.free()
    t = {n: x.cuda() for n, x in tensors.items() if n in "qkv"}
    outs = []
    for wait in (False, True):
        st, g = pu.gpu_layer(wl, params, max_call_tokens=start)
        st.prefill(t["q"][:, :, :start], t["k"][:, :, :start], t["v"][:, :, :start], wl.C, g, wl.r)
        steps = [[t[n][:, :, i].contiguous() for n in "qkv"] for i in range(start, wl.T)]
        ys = [torch.empty_like(s[0]) for s in steps]
        torch.cuda.synchronize()
        for s, out in zip(steps, ys):
            st.decode_step(*s, out=out)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert st.check() == 0
        outs.append(torch.stack(ys, 2).cpu())
        st.free()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], y[:, :, start:])


@pytest.mark.parametrize("Hq,Hkv,d,C,slots,r,splits,run", [
    (1, 1, 64, 16, 40, 0, {1}, False), (3, 1, 128, 16, 80, 32, {1}, False), (2, 2, 128, 32, 170, 32, {2}, False),
    (2, 1, 128, 64, 300, 64, {3, 4}, False), (5, 5, 64, 64, 960, 16, {5}, False), (4, 2, 128, 64, 600, 0, {6}, False),
    (3, 3, 128, 64, 700, 32, {6, 7}, False), (12, 12, 64, 32, 300, 0, {8}, False), (24, 12, 128, 64, 900, 32, {8}, False),
    (32, 32, 128, 64, 930, 0, {8}, True), (16, 16, 128, 16, 60, 32, {1}, True), (24, 12, 64, 64, 300, 32, {2}, True),
    (2, 2, 128, 64, 1500, 32, {8}, False), (1, 1, 64, 256, 3500, 0, {8}, False), (40, 20, 64, 64, 2500, 32, {8}, True)])
def test_splits_of_the_steps_that_fetch_their_rows_ahead(Hq, Hkv, d, C, slots, r, splits, run):
    """The library's splits, for cases of the test above too, which holds a rule of its own; the others run."""
    from paper_2605_09877_b200 import kvm
    start = (slots // C + 4) * C - 6
    wl = synth.Workload("short", 1, Hq, Hkv, d, start + 14, C, "fixed", fixed_slots=slots, r=r, seed=400 + slots)
    assert {kvm.decode_ahead(1, Hq, Hkv, d, _decode_rows(wl, t))[0] for t in range(start, wl.T)} == splits
    if run:
        test_decode_steps_that_fetch_their_rows_ahead(Hq, Hkv, d, C, slots, r, set(range(9)))


@pytest.mark.parametrize("B,Hq,Hkv,d,pos,steps,plan", [
    (1, 1, 1, 64, 40, 30, (1, 1, 1)), (1, 2, 1, 128, 900, 20, (2, 6, 1)), (3, 32, 4, 64, 1300, 10, (4, 7, 1)), (7, 21, 21, 128, 300, 9, (1, 2, 1)),
    (1, 2, 2, 128, 260, 5, (1, 5, 1)), (1, 2, 2, 128, 452, 5, (1, 8, 1)), (5, 32, 4, 64, 20, 5, (8, 1, 1)), (5, 32, 4, 128, 130, 8, (8, 3, 1))])
def test_decode_kernel_that_loops_over_rows_at_few_rows(B, Hq, Hkv, d, pos, steps, plan):
    """With the timing hook on no step overlaps the one before it; steps that fetch their rows ahead otherwise and steps of the kernel
    that loops over them."""
    from paper_2605_09877_b200 import kvm
    wl = synth.Workload("dec", B, Hq, Hkv, d, pos + steps, 64, "sqrt", sqrt_coeff=20, r=32, seed=330 + pos)
    assert {kvm.decode_plan(B, Hq, Hkv, d, _decode_rows(wl, t)) for t in range(pos, pos + steps)} == {plan}
    params = synth.make_layer_params(wl, trivial=False)
    tensors = synth.make_inputs(wl)
    units = sorted({(0, 0), (B - 1, Hkv - 1)})
    y, st = pu.run_gpu(wl, tensors, params, decode_from=pos, timed=True)
    y_ref, o = pu.run_oracle(wl, tensors, params, units=units)
    print(pu.compare(wl, y, st, y_ref, o, units=units))
    st.free()


@pytest.mark.parametrize("B,Hq,Hkv,d,C,slots,plan", [
    (10, 24, 8, 128, 16, 110, (1, 1, 1)), (10, 15, 5, 128, 16, 110, (1, 2, 1)), (10, 9, 9, 128, 32, 220, (1, 3, 1)), (8, 9, 9, 128, 32, 370, (1, 4, 1)),
    (6, 9, 9, 64, 64, 960, (1, 5, 1)), (3, 11, 11, 128, 32, 1010, (1, 6, 1)), (8, 1, 1, 64, 64, 4120, (1, 7, 1)), (8, 1, 1, 128, 64, 2200, (1, 8, 1)),
    (10, 30, 5, 128, 16, 110, (2, 1, 1)), (12, 16, 8, 64, 64, 440, (2, 2, 1)), (12, 10, 5, 128, 32, 490, (2, 3, 1)), (2, 22, 11, 128, 32, 1010, (2, 6, 1)),
    (10, 64, 16, 128, 16, 16, (4, 1, 1)), (10, 16, 4, 128, 32, 370, (4, 4, 1)), (10, 8, 2, 128, 32, 770, (4, 7, 1)), (6, 12, 3, 128, 64, 820, (4, 8, 1)),
    (10, 64, 8, 64, 16, 16, (8, 1, 1)), (10, 24, 3, 128, 32, 220, (8, 3, 1)), (12, 16, 2, 128, 32, 230, (8, 5, 1)), (6, 24, 3, 128, 64, 620, (8, 6, 1))])
def test_decode_steps_that_loop_over_their_rows(B, Hq, Hkv, d, C, slots, plan):
    """One to eight splits and query heads per CTA of the kernel that loops over its rows, each where the library takes it; steps
    across a fold, behind which some run the other kernel, against the oracle."""
    start = (slots // C + 4) * C - 4
    wl = synth.Workload("loop", B, Hq, Hkv, d, start + 8, C, "fixed", fixed_slots=slots, r=32, seed=500 + slots)
    assert plan in _decode_kernels(B, Hq, Hkv, d, {_decode_rows(wl, t) for t in range(start, wl.T)})
    params = synth.make_layer_params(wl, trivial=False)
    print(_sampled(wl, sorted({(0, 0), (B - 1, Hkv - 1)}), params=params, decode_from=start))


@pytest.mark.parametrize("B,Hq,Hkv,d,C,slots", [(1, 4, 4, 128, 64, 500), (1, 16, 4, 64, 64, 1200), (2, 4, 2, 128, 64, 1500), (10, 64, 16, 128, 16, 16)])
def test_timed_decode_steps_run_the_kernels_that_serve(B, Hq, Hkv, d, C, slots):
    """With the timing hook on no step overlaps the one before it, but it is the same kernel: bit for bit the same outputs."""
    start = (slots // C + 4) * C - 6
    wl = synth.Workload("hook", B, Hq, Hkv, d, start + 12, C, "fixed", fixed_slots=slots, r=32, seed=520 + slots)
    params = synth.make_layer_params(wl, trivial=False)
    t = {n: x.cuda() for n, x in synth.make_inputs(wl).items() if n in "qkv"}
    outs = []
    for hook in (False, True):
        st, g = pu.gpu_layer(wl, params, max_call_tokens=start)
        st.prefill(t["q"][:, :, :start], t["k"][:, :, :start], t["v"][:, :, :start], wl.C, g, wl.r)
        st.profile_enable(hook)
        outs.append(torch.stack([st.decode_step(*(t[n][:, :, i].contiguous() for n in "qkv")) for i in range(start, wl.T)]).cpu())
        assert st.check() == 0 and (not hook or st.profile_read()["decode"][1] == wl.T - start)
        st.free()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("Hq,Hkv,d,slots", [(4, 4, 128, 600), (2, 1, 64, 1500), (1, 1, 128, 1300)])
def test_replayed_steps_fetch_no_rows_of_an_earlier_replay_ahead(Hq, Hkv, d, slots):
    """A captured run of steps carries the numbers it was captured with.  Replayed behind a prefill of another sequence, and once
    more behind itself, its steps give what the same steps give one by one."""
    C, n = 64, 12
    start = (slots // C + 4) * C + 5
    wl = synth.Workload("replay", 1, Hq, Hkv, d, start + n, C, "fixed", fixed_slots=slots, r=32, seed=530 + slots)
    assert {k[0] for k in _decode_kernels(1, Hq, Hkv, d, {_decode_rows(wl, t) for t in range(start, wl.T)})} == {"ahead"}
    params = synth.make_layer_params(wl, trivial=False)
    seqs = [{m: x.cuda() for m, x in synth.make_inputs(wl.scaled(seed=530 + slots + i)).items() if m in "qkv"} for i in range(3)]

    def prefill(st, g, t):
        st.prefill(t["q"][:, :, :start], t["k"][:, :, :start], t["v"][:, :, :start], C, g, wl.r)

    want = []
    for t in seqs:
        st, g = pu.gpu_layer(wl, params, max_call_tokens=start)
        prefill(st, g, t)
        ys = []
        for i in range(start, wl.T):
            ys.append(st.decode_step(*(t[m][:, :, i].contiguous() for m in "qkv")))
            torch.cuda.synchronize()
        want.append(torch.stack(ys))
        st.free()
    st, g = pu.gpu_layer(wl, params, max_call_tokens=start)
    prefill(st, g, seqs[0])
    steps = [[seqs[0][m][:, :, i].clone(memory_format=torch.contiguous_format) for m in "qkv"] for i in range(start, wl.T)]
    out = torch.empty_like(want[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for s, y in zip(steps, out):
            st.decode_step(*s, out=y)
    for t, y_ref in zip(seqs, want):
        if t is not seqs[0]:
            st.reset()
            prefill(st, g, t)
            for i, s in zip(range(start, wl.T), steps):
                for m, x in zip("qkv", s):
                    x.copy_(t[m][:, :, i])
        for _ in range(2):
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, y_ref)
    assert st.check() == 0
    del graph
    st.free()


def test_steps_of_two_states_in_turn_on_one_stream():
    """The layers of a model: a step is resident under the one of another state, across the folds of both."""
    wls = [synth.Workload("la", 1, 4, 4, 128, 700 + 40, 64, "fixed", fixed_slots=400, r=32, seed=541),
           synth.Workload("lb", 1, 8, 2, 64, 690 + 40, 64, "sqrt", sqrt_coeff=16, r=0, seed=542)]
    starts, outs = (700, 690), []
    for together in (False, True):
        made = []
        for wl, start in zip(wls, starts):
            t = {n: x.cuda() for n, x in synth.make_inputs(wl).items() if n in "qkv"}
            st, g = pu.gpu_layer(wl, synth.make_layer_params(wl), max_call_tokens=start)
            st.prefill(t["q"][:, :, :start], t["k"][:, :, :start], t["v"][:, :, :start], wl.C, g, wl.r)
            made.append((st, [[t[n][:, :, i].contiguous() for n in "qkv"] for i in range(start, wl.T)]))
        ys = [[torch.empty_like(s[0]) for s in steps] for _, steps in made]
        torch.cuda.synchronize()
        order = [(l, i) for i in range(40) for l in range(2)] if together else [(l, i) for l in range(2) for i in range(40)]
        for l, i in order:
            made[l][0].decode_step(*made[l][1][i], out=ys[l][i])
            if not together:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert all(st.check() == 0 for st, _ in made)
        outs.append([torch.stack(y) for y in ys])
        for st, _ in made:
            st.free()
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
