"""Forwards of a few token rows (weight-streaming products, attention of few rows) against the tensor-core path of larger
forwards on the same weights: one to 32 rows, widths that leave shares of K and slices ragged, key counts around the slice
of 32 and around the lengths at which a head's keys go to two and to four CTAs."""
import os

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _logits(few, heads, plens, gamma, steps):
    import paper_2408_05636_b200 as sdd
    n_ctx, V, d = 512, 700, 64 * heads
    t, q = synth.ModelShape(V, 2, d, heads, n_ctx, True), synth.ModelShape(V, 1, 128, 2, n_ctx, False)
    names = synth.tensor_names(t)
    wt = synth.model_weights(t, 3, "bf16", bias_std=0.05, perturb_ln=True)
    dt = sdd.DeviceModel(t, wt, names, "bf16")
    dq = sdd.DeviceModel(q, synth.model_weights(q, 4, "bf16"), synth.tensor_names(q), "bf16")
    prompts = synth.prompt_ids(V, len(plens), max(plens), 9)
    old = os.environ.get("SDD_FEW_ROWS")
    os.environ["SDD_FEW_ROWS"] = few
    try:
        s = sdd.Session(dt, dq, prompts, plens, gamma, 1, 60, 1.0, 1.0, 5)
    finally:
        if old is None:
            del os.environ["SDD_FEW_ROWS"]
        else:
            os.environ["SDD_FEW_ROWS"] = old
    rows = gamma + 1 if steps == "round" else 1
    (s.sdd_step if steps == "round" else s.sdd_ar_step)()
    p = s.tap_numpy(sdd.TAP_LOGITS_P)[: len(plens) * rows * V].reshape(len(plens), rows, V).copy()
    slots = s.tap_numpy(sdd.TAP_DRAFT_IDS).copy()
    s.close()
    return p, slots


@pytest.mark.parametrize("heads", [2, 5, 25])
@pytest.mark.parametrize("plens", [[1], [31, 33], [190, 191, 5], [33] * 7, [300] * 9, [383, 384, 2] * 6, [60] * 25])
def test_decoding_rows(heads, plens):
    few, _ = _logits("32", heads, plens, 8, "ar")
    ref, _ = _logits("0", heads, plens, 8, "ar")
    assert np.abs(few - ref).max() < 2e-2 and np.linalg.norm(few - ref) < 1e-2 * np.linalg.norm(ref)


@pytest.mark.parametrize("plens,gamma", [([40], 1), ([380], 7), ([420, 3], 7), ([100], 30), ([250, 31, 64], 4)])
def test_verification_rows(plens, gamma):
    few, slots = _logits("32", 5, plens, gamma, "round")
    ref, slots_ref = _logits("0", 5, plens, gamma, "round")
    assert np.array_equal(slots, slots_ref)          # the drafts do not depend on the target's path
    assert np.abs(few - ref).max() < 2e-2 and np.linalg.norm(few - ref) < 1e-2 * np.linalg.norm(ref)


# column groups of 5, 6 and 8, 48-feature CTAs (width 1600 from 17 rows on), the row limits of both widths, row groups of 8
@pytest.mark.parametrize("heads", [5, 25])
@pytest.mark.parametrize("plens,gamma", [([100], 16), ([300], 32), ([40, 190, 2], 12), ([400], 40), ([100, 333, 7], 15), ([200], 48),
                                         ([31], 63), ([250, 9, 63, 64], 15)])
def test_verification_rows_wide(heads, plens, gamma):
    few, slots = _logits("64", heads, plens, gamma, "round")
    ref, slots_ref = _logits("0", heads, plens, gamma, "round")
    assert np.array_equal(slots, slots_ref)
    assert np.abs(few - ref).max() < 2e-2 and np.linalg.norm(few - ref) < 1e-2 * np.linalg.norm(ref)
