"""The mma.sync attention's split of a chunk's keys over its warps: tiles of up
to 16 rows (four key groups), up to 32 (two) and above (one), at their edges,
with chunks whose last keys leave whole groups without one, several splits of
the key range, rings of two and three stages, and both head widths."""
import numpy as np
import pytest

import synth
from tests.test_gpu_attention_kernels import _check

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("splits,stages", [("1", "3"), ("1", "2"), ("3", "2")])
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("heads", [(4, 4), (6, 2)])
def test_key_groups(monkeypatch, heads, head_dim, splits, stages):
    monkeypatch.setenv("EBD_ATTN_KERNEL", "mma")
    monkeypatch.setenv("EBD_ATTN_SPLITS", splits)
    monkeypatch.setenv("EBD_ATTN_STAGES", stages)
    windows = (1, 15, 16, 17, 32, 33, 5, 11)
    prefixes = np.array([0, 1, 16, 17, 33, 48, 64, 193])
    sh = synth.tiny.with_(name=f"groups_{heads[1]}_{head_dim}", batch=len(windows), windows=windows, n_heads_q=heads[0],
                          n_heads_kv=heads[1], head_dim=head_dim, prefix=200, seed=head_dim + heads[0])
    inp = synth.make_step_inputs(sh, weights=False, prefix_lens=prefixes)
    got = _check("groups", inp)
    assert np.isfinite(got).all()
