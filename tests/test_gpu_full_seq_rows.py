"""Windows of more than 64 rows: a step writes the statistics of every one of
its rows, also of those that no sequence's window holds (rows before the first
offset or past the last) and of rejected sequences (more rows than gen_len,
offsets that run backwards), and reports a non-finite row among them."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROWS = 130
STATS = ("conf", "entropy", "ent_norm", "gap", "argmax")


def _run(offsets, bad_row=None):
    from paper_2609_16450_gb300 import _ebd as E
    from paper_2609_16450_gb300 import runtime as rt
    sh = synth.tiny.with_(name="uncovered", batch=2, windows=(90, 40), gen_len=96, prefix=0, seed=31)
    inp = synth.make_step_inputs(sh)
    if bad_row is not None:
        inp.hidden[bad_row] = 0x7FC0  # NaN
    w = rt.upload_weights(inp)
    h = rt.Handle(rt.config_for(sh, max_batch=3, max_window=96, max_rows=ROWS), w.w_emb)
    try:
        ds = rt.DeviceStep(inp, w, attention=False)
        a = ds.args()
        E.check(E.ebd_lm_stats(h.h, a, rt.stream_handle(None)), h.h)
        h.sync_status()
        want = ds.fetch()
        for k in STATS:
            getattr(ds, k).fill_(-7)
        cu = torch.tensor(offsets, dtype=torch.int32, device="cuda")
        ds.blk_meta = torch.zeros((len(offsets) - 1, 2), dtype=torch.int32, device="cuda")
        a = ds.args()
        a.cu_rows, a.batch = cu.data_ptr(), len(offsets) - 1
        E.check(E.ebd_step(h.h, a, rt.stream_handle(None)), h.h)
        status = h.sync_status()
        return status, want, ds.fetch()
    finally:
        h.close()


@pytest.mark.parametrize("offsets,ok", [
    ((0, 90, ROWS), True),        # every row in a window
    ((0, 70, 100), True),         # rows past the last offset
    ((10, 75, ROWS), True),       # rows before the first
    ((0, 0, 60), True),           # an empty window, and rows past the end
    ((0, 100, ROWS), False),      # more rows than gen_len
    ((0, 20, ROWS), False),       # the last sequence rejected
    ((0, 40, 20, ROWS), False),   # offsets that run backwards
    ((0, 90, ROWS + 50), False),  # past the step's rows
])
def test_statistics_of_every_row(offsets, ok):
    from paper_2609_16450_gb300 import _ebd as E
    status, want, got = _run(offsets)
    assert status == (E.EBD_OK if ok else E.EBD_ERR_INVALID_ARG)
    # the same partial states through the same merge
    for k in STATS:
        np.testing.assert_allclose(got[k], want[k], rtol=1e-6, atol=1e-7, err_msg=k)


def test_nonfinite_row_outside_every_window():
    from paper_2609_16450_gb300 import _ebd as E
    status, _, got = _run((0, 70, 100), bad_row=120)
    assert status == E.EBD_ERR_NONFINITE and got["argmax"][120] == -1
