"""Windows that start and end anywhere inside a group of codes: the part inside is staged and stored
in one piece, so the first and last elements of it may fall on either side of a 16-byte boundary
of the output.  Every length up to a few such pieces, at every alignment of the outputs and for groups of
1, 16, 81, 256 and 625 codes, inside guards and bit for bit against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2601_02311_b200 import synth
from test_gpu_canaries import FIELDS, ctx, guarded, guards_intact, ps, unsigned      # noqa: F401
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("mode_mask", [0b00001, 0b10010, 0b01011, 0b01111, 0b11111])
@pytest.mark.parametrize("ragged", [False, True])
def test_parts_of_groups(ctx, mode_mask, shift, ragged):      # noqa: F811
    space = dict(synth.config("C3", n_models=2), mode_mask=mode_mask)
    if ragged:
        space["n_values"] = np.asarray([6, 7, 96], dtype=np.uint32)
    gs, os_ = ctx.space(space), O.Space(space)
    codes = bin(mode_mask).count("1") ** 4
    want = os_.eval_range(0, 4 * codes + 32)
    windows = {(lo, n) for lo in (0, 1, 2, 3, codes - 1, codes, codes + 1, 2 * codes - 3)
               for n in (1, 2, 3, 4, 5, 7, 9, codes - 1, codes, codes + 3, 2 * codes + 1)}
    for first, count in sorted(w for w in windows if w[0] >= 0 and w[1] > 0):
        bufs, out = {}, {}
        for k in FIELDS:
            bufs[k], out[k] = guarded(count, torch.int32 if k == "flags" else torch.int64, shift, ctx.torch_device)
        gs.eval_batch_into(first, count, out)
        ctx.check_status()
        for k in FIELDS:
            assert guards_intact(bufs[k], shift, count), (k, first, count)
            assert np.array_equal(unsigned(out[k]), want[k][first:first + count]), (k, first, count)
