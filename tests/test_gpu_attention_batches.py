"""The window attention of calls with fewer sequences, and shorter key ranges,
than the handle was made for: kernel and key splits follow the call's sequences
(the tcgen05 kernel for few, the mma.sync kernel for many), and a sequence with
few keys leaves splits out, beside sequences that take all of them."""
import numpy as np
import pytest

import synth
from oracle import ebd_oracle as o
from tests import parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("heads", [(8, 8, 128), (14, 2, 64)])
@pytest.mark.parametrize("prefix", [320, 1100])
def test_calls_below_the_largest_batch(heads, prefix):
    from paper_2609_16450_gb300 import _ebd as E
    from paper_2609_16450_gb300 import runtime as rt
    h = None
    try:
        for batch in (1, 2, 5, 19, 40):
            rng = np.random.default_rng(batch * 7 + prefix)
            lens = rng.integers(0, prefix + 1, batch)
            lens[0] = prefix
            if batch > 2:
                lens[1], lens[2] = 0, 250
            sh = synth.tiny.with_(name=f"mb{batch}", batch=batch, windows=tuple(int(w) for w in rng.integers(1, 17, batch)),
                                  n_heads_q=heads[0], n_heads_kv=heads[1], head_dim=heads[2], prefix=prefix,
                                  seed=batch)
            inp = synth.make_step_inputs(sh, weights=False, prefix_lens=lens)
            if h is None:
                h = rt.Handle(rt.config_for(sh, max_batch=40, max_window=16, max_rows=640))
            q, kw, vw, kc, vc = (rt._dev(x, "cuda") for x in (inp.q, inp.k_win, inp.v_win, inp.k_cache, inp.v_cache))
            cu, pl = (rt._dev(x.astype(np.int32), "cuda") for x in (inp.cu_rows, inp.prefix_len))
            out = torch.full((inp.rows, heads[0], heads[2]), -7.0, device="cuda")
            a = E.ebd_step_args()
            a.batch, a.rows = batch, inp.rows
            for k, t in dict(cu_rows=cu, prefix_len=pl, q=q, k_win=kw, v_win=vw, k_cache=kc, v_cache=vc,
                             attn_out=out).items():
                setattr(a, k, t.data_ptr())
            for _ in range(2):  # the second call finds the first one's tickets
                E.check(E.ebd_attention(h.h, a, rt.stream_handle(None)), h.h)
            assert h.sync_status() == 0, E.ebd_last_error(h.h)
            want = o.window_attention(inp.q, inp.k_win, inp.v_win, inp.k_cache, inp.v_cache, inp.cu_rows,
                                      inp.prefix_len, None)
            # fp32 sums of probabilities held in 16 bits: 2e-3 as for every attention output
            parity._close(f"batch {batch}", out.cpu().numpy().reshape(want.shape), want)
    finally:
        if h is not None:
            h.close()
