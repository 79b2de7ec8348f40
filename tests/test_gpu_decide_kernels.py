"""The decision behind the LM head (ebd_step) in each of its launch forms
(tests/forms.py), against the oracle:

* degenerate windows (empty, one row, the longest all masked, the longest with
  nothing masked, |M| <= L_min) with no active block (the LBS runs) and inside
  one; the statistics of every row, masked and not, are the step's;
* non-finite hidden rows: reported, not committed, other sequences exact;
* the baselines' threshold and Top-m rules;
* sweep points of 16 and 64 sequences at the LLaDA-8B head shape;
* ebd_decide (statistics as inputs) on a step's own statistics takes that
  step's decision bit for bit."""
import numpy as np
import pytest

import synth
from oracle import ebd_oracle as o
from tests import parity
from tests import test_gpu_configs as C
from tests import test_gpu_edges as G
from tests.forms import FORMS, ragged_step

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _step(sh, inp, expect=0, **over):
    from paper_2609_16450_gb300 import _ebd as E
    from paper_2609_16450_gb300 import runtime as rt
    w = rt.upload_weights(inp)
    h = rt.Handle(rt.config_for(sh, **over), w.w_emb)
    try:
        ds = rt.DeviceStep(inp, w, attention=False)
        E.check(E.ebd_step(h.h, ds.args(), rt.stream_handle(None)), h.h)
        assert h.sync_status() == expect, E.ebd_last_error(h.h)
        return ds.fetch()
    finally:
        h.close()


@pytest.mark.parametrize("state", ["select", "inblock"])
@pytest.mark.parametrize("form", FORMS)
def test_degenerate_windows(form, state):
    sh, inp = ragged_step(form, state)
    gpu = _step(sh, inp)
    res = o.step(inp, G._weights(sh), G._prm(sh), attention=False)
    parity.compare_stats(res.stats, gpu)
    rep = parity.compare_decision(res, gpu, inp, G._prm(sh))
    assert rep["flagged_sequences"] <= rep["sequences"] // 2, rep
    cu = inp.cu_rows
    for b in range(3, sh.batch, 7):  # nothing masked: no commit, no block
        sl = slice(int(cu[b]), int(cu[b + 1]))
        assert not gpu["accepted"][sl].any() and np.array_equal(gpu["tokens"][sl], inp.tokens[sl])
        assert tuple(gpu["blk_meta"][b]) == (0, 0)
    if state == "select":
        for b in range(0, sh.batch, 7):  # the LBS ran over the whole window
            assert np.isfinite(gpu["lbs_logit"][int(cu[b]):int(cu[b + 1])]).all()
        for b in range(5, sh.batch, 7):  # |M| <= L_min
            assert np.isnan(gpu["lbs_logit"][int(cu[b]):int(cu[b + 1])]).all()


@pytest.mark.parametrize("form", FORMS)
def test_nonfinite_rows(form):
    from paper_2609_16450_gb300 import _ebd as E
    sh, inp = ragged_step(form, seed=100)
    cu = inp.cu_rows
    res = o.step(inp, G._weights(sh), G._prm(sh), attention=False)
    bad = [int(cu[0]) + 2, int(cu[1]) - 1]
    inp.hidden[bad[0]] = G.BF16_NAN
    inp.hidden[bad[1]] = G.BF16_INF
    gpu = _step(sh, inp, expect=E.EBD_ERR_NONFINITE)
    assert np.all(gpu["argmax"][bad] == -1) and np.all(gpu["mask"][bad] == 1)
    assert not gpu["accepted"][bad].any() and np.array_equal(gpu["tokens"][bad], inp.tokens[bad])
    rest = np.arange(int(cu[1]), inp.rows)
    sub = o.RowStats(*(np.asarray(getattr(res.stats, f))[rest] for f in
                       ("conf", "entropy", "ent_norm", "gap", "argmax", "logit_gap", "near_tie")))
    parity.compare_stats(sub, {k: gpu[k][rest] for k in ("conf", "entropy", "ent_norm", "gap", "argmax")})
    compared = 0
    for b in range(1, sh.batch):
        if res.flag_accept[b] or res.flag_lbs[b]:
            continue
        compared += 1
        sl = slice(int(cu[b]), int(cu[b + 1]))
        for k in ("accepted", "tokens", "mask", "in_block"):
            assert np.array_equal(np.asarray(gpu[k][sl], np.int64), np.asarray(getattr(res, k)[sl], np.int64)), (k, b)
        assert np.array_equal(gpu["blk_meta"][b], res.blk_meta[b]), b
    assert compared >= (sh.batch - 1) // 2


@pytest.mark.parametrize("mode,top_m", [("threshold", 1), ("topm", 5)])
@pytest.mark.parametrize("form", FORMS)
def test_baseline_modes(form, mode, top_m):
    sh, inp = ragged_step(form, seed=200)
    gpu = _step(sh, inp, decode_mode={"threshold": 1, "topm": 2}[mode], top_m=top_m)
    want = o.softmax_stats(o.lm_logits(inp.hidden.reshape(inp.rows, -1), inp.w_lm.reshape(sh.vocab, -1)))
    parity.compare_stats(want, gpu)
    compared = 0
    for b in range(sh.batch):
        sl = slice(int(inp.cu_rows[b]), int(inp.cu_rows[b + 1]))
        m, t = inp.mask[sl].copy(), inp.tokens[sl].copy()
        n = len(m)
        st = o.RowStats(*(gpu[k][sl].astype(np.float64) for k in ("conf", "entropy", "ent_norm", "gap")),
                        gpu["argmax"][sl].astype(np.int64), np.full(n, np.inf), np.zeros(n, bool))
        d = o.decide_fixed_block(m, t, st, mode, sh.tau, top_m)
        if d.flag_accept:
            continue
        compared += 1
        assert np.array_equal(gpu["accepted"][sl], d.accepted), b
        assert np.array_equal(gpu["mask"][sl], m) and np.array_equal(gpu["tokens"][sl], t), b
    assert compared >= sh.batch // 2
    assert np.array_equal(gpu["in_block"], inp.in_block) and np.array_equal(gpu["blk_meta"], inp.blk_meta)


@pytest.mark.parametrize("point", [(16, 256, 32), (64, 256, 8)])
def test_many_sequences(point):
    C.test_sweep_point(point)


@pytest.mark.parametrize("state", ["select", "inblock"])
def test_decide_entry_takes_the_steps_decision(state):
    """ebd_decide (statistics as inputs) on the statistics a step produced, from
    the same decode state, takes exactly that step's decision."""
    from paper_2609_16450_gb300 import _ebd as E
    from paper_2609_16450_gb300 import runtime as rt
    sh = synth.llada
    inp = synth.make_step_inputs(sh)
    if state == "inblock":
        synth.preset_in_block(inp, 20)
    w = rt.upload_weights(inp)
    h = rt.Handle(rt.config_for(sh), w.w_emb)
    try:
        ds = rt.DeviceStep(inp, w, attention=False)
        E.check(E.ebd_step(h.h, ds.args(), rt.stream_handle(None)), h.h)
        assert h.sync_status() == 0
        step = ds.fetch()
        ds.restore_state()
        E.check(E.ebd_decide(h.h, ds.args(), rt.stream_handle(None)), h.h)
        assert h.sync_status() == 0
        dec = ds.fetch()
        for k in ("tokens", "mask", "in_block", "blk_meta", "accepted"):
            np.testing.assert_array_equal(dec[k], step[k], err_msg=k)
        for k in ("lbs_logit", "lps_prob"):
            np.testing.assert_array_equal(dec[k], step[k], err_msg=k)  # NaN where not scored
        assert step["accepted"].sum() >= 1
    finally:
        h.close()
