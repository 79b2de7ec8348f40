"""The launch forms of the decision (GPU tests), each with a batch that selects it
and a step whose windows reach its edges: CTAs per sequence by groups of 8 rows
per CTA for windows of up to 64 rows (the first three) and of up to 32 in batches
of 16 and more, CTAs per sequence above 64 rows (behind the statistics and LBS
grids).  The number of sequences at which one form gives way to the next is the
number of clusters that fit the GPU (GB300: 15 of 8 CTAs, 36 of 4; above 64 rows 7
of 16)."""
import numpy as np

import synth

FORMS = {"8x1": (3, 64), "4x2": (20, 64), "2x4": (40, 64), "4x1": (16, 32), "2x2": (40, 32), "1x4": (80, 32),
         "wide16": (3, 100), "wide8": (10, 100), "wide4": (20, 100), "wide2": (38, 100)}


def ragged_step(form, state="select", seed=0, weights=True):
    """(shape, inputs): the longest window with every row masked, an empty one, one
    row, the longest with nothing masked (more rows than a CTA's warps merge at
    once), half of it, one whose masked set is no larger than L_min, nine rows; over
    and over."""
    batch, longest = FORMS[form]
    kinds = (longest, 0, 1, longest, longest // 2 + 1, 20, 9)
    windows = tuple(kinds[i % len(kinds)] for i in range(batch))
    prefix = 128 if longest <= 64 else 0
    sh = synth.tiny.with_(name=f"form_{form}", batch=batch, windows=windows, prefix=prefix, seed=seed + batch)
    inp = synth.make_step_inputs(sh, weights=weights, prefix_lens=np.arange(batch) * 37 % (prefix + 1))
    if state == "inblock":
        synth.preset_in_block(inp, 16)
    for i in range(batch):
        r0, r1 = int(inp.cu_rows[i]), int(inp.cu_rows[i + 1])
        if i % 7 == 0:
            inp.mask[r0:r1], inp.tokens[r0:r1] = 1, -1
        elif i % 7 == 3:
            inp.mask[r0:r1], inp.tokens[r0:r1] = 0, 7
            inp.in_block[r0:r1], inp.blk_meta[i] = 0, 0
        elif i % 7 == 5:
            m = np.zeros(r1 - r0, np.uint8)
            m[[1, 4, 9, 10, 17]] = 1
            inp.mask[r0:r1], inp.tokens[r0:r1] = m, np.where(m == 1, -1, 11)
    return sh, inp
