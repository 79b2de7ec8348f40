"""The baselines' rules on statistics given to ebd_decide (one CTA per sequence,
windows of up to 64 and of up to 512 rows), against the oracle's rule: batches
and windows at the edges of a warp's and of a thread's rows, nothing masked,
equal confidences, statistics that are not usable, and the window lengths that
a handle takes and refuses."""
import numpy as np
import pytest

import synth
from oracle import ebd_oracle as o
from tests.test_gpu_decide_rows import _stats

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MODES = {"threshold": 1, "topm": 2}
STATE = ("tokens", "mask", "in_block", "blk_meta")


def _decide(ws, max_window, mode, top_m, stats, change=None, max_rows=None):
    """One ebd_decide; returns (status, inputs, outputs)."""
    from paper_2609_16450_gb300 import _ebd as E
    from paper_2609_16450_gb300 import runtime as rt
    sh = synth.tiny.with_(name="rule", batch=len(ws), windows=tuple(int(w) for w in ws), gen_len=512, prefix=0,
                          mask_frac=0.7, seed=int(sum(ws)) + len(ws))
    inp = synth.make_step_inputs(sh, weights=False)
    if change:
        change(inp, stats)
    conf, ent, gap, arg = stats
    cfg = rt.config_for(sh, max_window=max_window, max_rows=max_rows or min(4096, len(ws) * max_window),
                        decode_mode=MODES[mode], top_m=top_m)
    w_emb = torch.zeros((sh.vocab, sh.d_base), dtype=torch.int16, device="cuda")
    h = rt.Handle(cfg, w_emb)
    try:
        t = {k: rt._dev(np.asarray(v), "cuda") for k, v in dict(
            cu_rows=inp.cu_rows.astype(np.int32), row_pos=inp.row_pos.astype(np.int32),
            tokens=inp.tokens.astype(np.int32), mask=inp.mask.astype(np.uint8),
            in_block=inp.in_block.astype(np.uint8), blk_meta=inp.blk_meta.astype(np.int32), conf=conf, ent_norm=ent,
            gap=gap, argmax=arg).items()}
        n = inp.rows
        t.update(lbs_logit=torch.zeros(n, device="cuda"), lps_prob=torch.zeros(n, device="cuda"),
                 accepted=torch.full((n,), 9, dtype=torch.uint8, device="cuda"))
        a = E.ebd_step_args()
        a.batch, a.rows = len(ws), n
        for k, v in t.items():
            setattr(a, k, v.data_ptr())
        E.check(E.ebd_decide(h.h, a, rt.stream_handle(None)), h.h)
        status = h.sync_status()
        return status, sh, inp, {k: v.cpu().numpy() for k, v in t.items()}
    finally:
        h.close()


def _compare(sh, inp, got, stats, mode, top_m):
    conf, ent, gap, arg = stats
    usable = np.isfinite(conf) & np.isfinite(ent) & np.isfinite(gap) & (arg >= 0) & (arg < sh.vocab)
    compared = 0
    for b, (r0, r1) in enumerate(zip(inp.cu_rows[:-1], inp.cu_rows[1:])):
        sl = slice(int(r0), int(r1))
        m, t = inp.mask[sl].copy(), inp.tokens[sl].copy()
        held = (m != 0) & ~usable[sl]  # stays masked
        m[held] = 0
        st = o.RowStats(*(np.asarray(x)[sl] for x in (conf.astype(np.float64), ent, ent, gap, arg,
                                                      np.full(inp.rows, np.inf), np.zeros(inp.rows, bool))))
        d = o.decide_fixed_block(m, t, st, mode, sh.tau, top_m)
        if d.flag_accept:
            continue
        compared += 1
        m[held] = 1
        assert np.array_equal(got["accepted"][sl], d.accepted), b
        assert np.array_equal(got["mask"][sl], m) and np.array_equal(got["tokens"][sl], t), b
    assert compared >= (len(inp.cu_rows) - 1) // 2
    assert np.isnan(got["lbs_logit"]).all() and np.isnan(got["lps_prob"]).all()
    assert np.array_equal(got["in_block"], inp.in_block) and np.array_equal(got["blk_meta"], inp.blk_meta)


@pytest.mark.parametrize("mode,top_m", [("threshold", 1), ("topm", 1), ("topm", 7), ("topm", 600)])
@pytest.mark.parametrize("batch,window", [(1, 64), (1, 33), (5, 13), (16, 32), (40, 24), (63, 64), (300, 9), (1, 65),
                                          (2, 257), (1, 512), (9, 200)])
def test_rule_matches_oracle(batch, window, mode, top_m):
    rng = np.random.default_rng(batch * 997 + window)
    ws = rng.integers(0, window + 1, batch)
    ws[0] = window
    stats = _stats(rng, int(ws.sum()), synth.tiny.vocab, synth.tiny.eos_id)

    def change(inp, stats):
        r0, r1 = int(inp.cu_rows[-2]), int(inp.cu_rows[-1])
        if batch > 1:  # nothing left to unmask
            inp.mask[r0:r1] = 0
            inp.tokens[r0:r1] = 5
        conf, ent, gap, arg = stats
        n = len(conf)
        conf[rng.integers(0, n, 1 + n // 50)] = np.nan
        gap[rng.integers(0, n, 1 + n // 50)] = np.inf
        arg[rng.integers(0, n, 1 + n // 50)] = -1
        arg[rng.integers(0, n, 1 + n // 50)] = synth.tiny.vocab

    status, sh, inp, got = _decide(ws, window, mode, top_m, stats, change)
    assert status == 0
    _compare(sh, inp, got, stats, mode, top_m)


@pytest.mark.parametrize("window", [40, 400])
def test_equal_confidences_take_the_lower_positions(window):
    n = window
    stats = (np.full(n, 0.5, np.float32), np.full(n, 0.3, np.float32), np.full(n, 0.1, np.float32),
             np.arange(n, dtype=np.int32))
    status, _, inp, got = _decide([n], window, "topm", 3, stats)
    assert status == 0
    want = np.flatnonzero(inp.mask)[:3]
    assert np.array_equal(np.flatnonzero(got["accepted"]), want)
    assert np.array_equal(got["tokens"][want], want)


@pytest.mark.parametrize("batch,max_window,longest,ok", [(15, 32, 64, True), (16, 32, 32, True), (16, 32, 33, False),
                                                         (2, 64, 65, False), (2, 65, 128, True)])
def test_windows_a_handle_takes(batch, max_window, longest, ok):
    from paper_2609_16450_gb300 import _ebd as E
    ws = [longest] + [1] * (batch - 1)
    stats = _stats(np.random.default_rng(3), sum(ws), synth.tiny.vocab, synth.tiny.eos_id)
    status, sh, inp, got = _decide(ws, max_window, "threshold", 1, stats, max_rows=batch * max_window)
    if ok:
        assert status == 0
        _compare(sh, inp, got, stats, "threshold", 1)
    else:
        assert status == E.EBD_ERR_INVALID_ARG
        assert np.array_equal(got["mask"][:longest], inp.mask[:longest])
        assert np.array_equal(got["tokens"][:longest], inp.tokens[:longest])
