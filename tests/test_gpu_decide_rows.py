"""The decision's launch shapes at their boundaries, on statistics given to
ebd_decide: clusters of 8, 4 and 2 CTAs for windows of up to 64 rows (picked by
the batch), of 4, 2 and 1 for up to 32 rows in batches of 16 and more; above 64
rows a CTA per group of 8 rows, then clusters of 16, 8, 4 and 2 CTAs, also with
one window of 512 rows among many short ones; windows of a row, of whole groups
of 8 rows and one more or one less, with nothing masked, and blocks of every
masked row (the LPS over the whole window)."""
import dataclasses

import numpy as np
import pytest

import synth
from oracle import ebd_oracle as o
from tests import parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _stats(rng, n, vocab, eos):
    conf = rng.uniform(0.05, 0.99, n).astype(np.float32)
    # no kappa within the oracle's near-tie distance (1e-3) of tau, which with
    # hundreds of rows in one sequence would leave nothing to compare
    conf[np.abs(conf - 0.9) < 2e-3] = 0.8
    ent = ((1 - conf) * rng.uniform(0.2, 1.0, n)).astype(np.float32)
    gap = (conf * rng.uniform(0.3, 1.0, n)).astype(np.float32)
    arg = rng.integers(0, vocab, n).astype(np.int32)
    arg[rng.random(n) < 0.05] = eos
    return conf, ent, gap, arg


@pytest.mark.parametrize("bias", [0.0, 8.0])
@pytest.mark.parametrize("batch,window", [(1, 64), (1, 13), (2, 9), (9, 64), (20, 57), (37, 64), (44, 40),
                                          (16, 32), (40, 24), (90, 32), (140, 16), (1, 65), (2, 129), (1, 512),
                                          (3, 300), (400, 12), (9, 129), (20, 200), (60, 68)])
def test_decide_launch_shapes(batch, window, bias):
    rng = np.random.default_rng(batch * 1000 + window)
    ws = np.minimum(rng.integers(0, window + 1, batch), window)
    ws[0] = window
    ws[rng.integers(0, batch, batch // 4)] = 8 * (window // 8)
    while ws.sum() > 4096:
        ws[int(np.argmax(ws))] //= 2
    _check(rng, ws, window, bias)


@pytest.mark.parametrize("bias", [0.0, 8.0])
@pytest.mark.parametrize("batch", [7, 15, 36, 38])
def test_one_long_window_among_short_ones(batch, bias):
    rng = np.random.default_rng(batch)
    _check(rng, np.concatenate([[512], rng.integers(0, 70, batch - 1)]), 512, bias)


def _check(rng, ws, window, bias):
    from paper_2609_16450_gb300 import _ebd as E
    from paper_2609_16450_gb300 import runtime as rt
    batch = len(ws)
    sh = synth.tiny.with_(name=f"dec_{batch}_{window}", batch=batch, windows=tuple(int(w) for w in ws),
                          gen_len=max(512, window), prefix=0, mask_frac=0.8, seed=batch + window)
    inp = synth.make_step_inputs(sh)
    first = int(inp.cu_rows[1])
    inp.mask[:first] = 1  # the longest window entirely masked
    inp.tokens[:first] = -1
    n = inp.rows
    conf, ent, gap, arg = _stats(rng, n, sh.vocab, sh.eos_id)
    cfg = rt.config_for(sh, max_window=window, max_rows=min(4096, batch * window))
    W = synth.router_weights(sh.seed, sh.d_base, sh.gen_len)
    W = dict(W)
    W["lbs.head.b"] = synth.f32_to_bf16_bits(np.array([bias], np.float32)) if bias else W["lbs.head.b"]
    w_emb = rt._dev(inp.w_emb, "cuda")
    h = rt.Handle(cfg, w_emb)
    try:
        E.check(E.ebd_import_weights(h.h, synth.pack_blob(W, sh.d_base, sh.gen_len)), h.h)
        dev = {k: rt._dev(v, "cuda") for k, v in dict(
            cu_rows=inp.cu_rows, row_pos=inp.row_pos, tokens=inp.tokens, mask=inp.mask, in_block=inp.in_block,
            blk_meta=inp.blk_meta, conf=conf, ent_norm=ent, gap=gap, argmax=arg).items()}
        out = dict(lbs_logit=torch.full((n,), -7.0, device="cuda"), lps_prob=torch.full((n,), -7.0, device="cuda"),
                   accepted=torch.full((n,), 9, dtype=torch.uint8, device="cuda"))
        a = E.ebd_step_args()
        a.batch, a.rows = batch, n
        for k, v in {**dev, **out}.items():
            setattr(a, k, v.data_ptr())
        E.check(E.ebd_decide(h.h, a, rt.stream_handle(None)), h.h)
        assert h.sync_status() == 0, E.ebd_last_error(h.h)
        got = {k: v.cpu().numpy() for k, v in {**dev, **out}.items()}
    finally:
        h.close()
    f8 = lambda x: x.astype(np.float64)  # noqa: E731
    st = o.RowStats(conf=f8(conf), entropy=f8(ent), ent_norm=f8(ent), gap=f8(gap), argmax=arg,
                    logit_gap=np.ones(n), near_tie=np.zeros(n, bool))
    prm = o.DecisionParams(tau=sh.tau, tau_psi=sh.tau_psi, l_min=sh.l_min, l_b=sh.l_b, g_max=sh.g_max,
                           eos_id=sh.eos_id)
    ref = o.decide(inp.cu_rows, inp.row_pos, inp.tokens, inp.mask, inp.in_block, inp.blk_meta, st, inp.w_emb,
                   o.weights_f64(W), prm)
    flagged = ref.flag_accept | ref.flag_lbs
    keep = np.concatenate([np.full(w, not flagged[i]) for i, w in enumerate(np.diff(inp.cu_rows))])
    assert keep.mean() > 0.5
    for k in ("tokens", "mask", "in_block", "accepted"):
        assert np.array_equal(got[k][keep], getattr(ref, k)[keep]), k
    assert np.array_equal(got["blk_meta"][~flagged], ref.blk_meta[~flagged])
    # two bf16 planes hold 16 bits of an activation: logits of a few units
    # after some ten products of it stay within 1e-3 (one plane: 1e-1)
    for k in ("lbs_logit", "lps_prob"):
        x, y = got[k][keep], getattr(ref, k)[keep]
        assert np.array_equal(np.isnan(x), np.isnan(y)), k
        assert np.nanmax(np.abs(x - y), initial=0.0) <= 1e-3, k
