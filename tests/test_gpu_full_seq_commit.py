"""Windows of more than 64 rows whose decision runs no LPS (lps_enabled = 0, a
window with nothing masked): the commit overwrites the decode state that every
CTA of the sequence's cluster reads.  Called again and again from the same
state, the decision is the oracle's each time."""
import numpy as np
import pytest

import synth
from oracle import ebd_oracle as o
from tests.test_gpu_decide_rows import _stats

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("state", ["select", "inblock"])
def test_commit_in_place_without_lps(state):
    from paper_2609_16450_gb300 import _ebd as E
    from paper_2609_16450_gb300 import runtime as rt
    sh = synth.tiny.with_(name="nolps", batch=4, windows=(300, 65, 128, 80), gen_len=512, prefix=0, lps_enabled=0,
                          seed=41)
    inp = synth.make_step_inputs(sh)
    if state == "inblock":
        synth.preset_in_block(inp, 24)
    r0, r1 = (int(x) for x in inp.cu_rows[3:5])  # nothing left to unmask
    inp.mask[r0:r1], inp.in_block[r0:r1] = 0, 0
    inp.tokens[r0:r1], inp.blk_meta[3] = 3, 0
    conf, ent, gap, arg = _stats(np.random.default_rng(41), inp.rows, sh.vocab, sh.eos_id)
    h = rt.Handle(rt.config_for(sh), rt._dev(inp.w_emb, "cuda"))
    try:
        dev = {k: rt._dev(np.asarray(v), "cuda") for k, v in dict(
            cu_rows=inp.cu_rows.astype(np.int32), row_pos=inp.row_pos.astype(np.int32), conf=conf, ent_norm=ent,
            gap=gap, argmax=arg).items()}
        start = {k: rt._dev(v, "cuda") for k, v in dict(
            tokens=inp.tokens.astype(np.int32), mask=inp.mask.astype(np.uint8),
            in_block=inp.in_block.astype(np.uint8), blk_meta=inp.blk_meta.astype(np.int32)).items()}
        a = E.ebd_step_args()
        a.batch, a.rows = 4, inp.rows
        got = []
        for _ in range(40):
            st = {k: v.clone() for k, v in start.items()}
            acc = torch.full((inp.rows,), 9, dtype=torch.uint8, device="cuda")
            for k, v in {**dev, **st, "accepted": acc}.items():
                setattr(a, k, v.data_ptr())
            E.check(E.ebd_decide(h.h, a, rt.stream_handle(None)), h.h)
            got.append({**st, "accepted": acc})
        assert h.sync_status() == 0
        got = [{k: v.cpu().numpy() for k, v in g.items()} for g in got]
    finally:
        h.close()
    for g in got[1:]:
        for k in g:
            assert np.array_equal(g[k], got[0][k]), k
    f8 = lambda x: x.astype(np.float64)  # noqa: E731
    ref = o.decide(inp.cu_rows, inp.row_pos, inp.tokens, inp.mask, inp.in_block, inp.blk_meta,
                   o.RowStats(conf=f8(conf), entropy=f8(ent), ent_norm=f8(ent), gap=f8(gap), argmax=arg,
                              logit_gap=np.ones(inp.rows), near_tie=np.zeros(inp.rows, bool)),
                   inp.w_emb, o.weights_f64(synth.router_weights(sh.seed, sh.d_base, sh.gen_len)),
                   o.DecisionParams(tau=sh.tau, tau_psi=sh.tau_psi, l_min=sh.l_min, l_b=sh.l_b, g_max=sh.g_max,
                                    eos_id=sh.eos_id, lps_enabled=False))
    checked = 0
    for b in range(4):
        if ref.flag_accept[b] or ref.flag_lbs[b]:
            continue
        checked += 1
        sl = slice(int(inp.cu_rows[b]), int(inp.cu_rows[b + 1]))
        for k in ("accepted", "tokens", "mask", "in_block"):
            assert np.array_equal(np.asarray(got[0][k][sl], np.int64), np.asarray(getattr(ref, k)[sl], np.int64)), (k, b)
        assert np.array_equal(got[0]["blk_meta"][b], ref.blk_meta[b]), b
    assert checked >= 2
