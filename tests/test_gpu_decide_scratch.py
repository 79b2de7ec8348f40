"""The decision's device scratch grows with the rows a handle may see, not with
the sequences it may see: a handle for 65535 sequences of 4096 rows in all takes
some 200 MB (of which up to 36864 scratch rows of 5.1 KB above 64 rows per
sequence), where 32 rows kept for each sequence took 5 to 11 GB."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("max_window", [32, 64, 128])
def test_scratch_is_bounded_by_rows(max_window):
    from paper_2609_16450_gb300 import runtime as rt
    rt.Handle(rt.config_for(synth.tiny)).close()  # the library's own context and code
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    h = rt.Handle(rt.config_for(synth.tiny, max_batch=65535, max_window=max_window, max_rows=4096))
    try:
        used = free - torch.cuda.mem_get_info()[0]
    finally:
        h.close()
    assert used < 400 << 20, used
