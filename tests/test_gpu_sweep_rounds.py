"""Top-k over tables around the sizes at which its kernel changes over (rounds of resident blocks): the
lists of a sample of the models and all counts, bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2601_02311_b200 import synth
from test_gpu_parity import VALID, assert_same_sweep, ctx, ps      # noqa: F401

pytestmark = pytest.mark.gpu
GB = synth.GB


@pytest.mark.parametrize("per_sm,over", [(4, 0), (4, 1), (5, 0), (5, 1), (8, 0), (8, 1)])
@pytest.mark.parametrize("mode_mask", [0b11111, 0b10110])
@pytest.mark.parametrize("name", ["C1", "C3"])            # (22 factorisations, 290)
def test_topk_where_blocks_fill_the_gpu(ctx, ps, name, mode_mask, per_sm, over):      # noqa: F811
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + over
    space = dict(synth.config(name, n_models=n), mode_mask=mode_mask)
    few = np.arange(0, n, 37)
    gs, os_ = ctx.space(space), O.Space(dict(space, models=space["models"][few]))
    ppm = gs.points_per_model
    for require, host, skip in ((VALID, O.NO_LIMIT, False), (VALID, 64 * GB, False), (VALID, 64 * GB, True),
                                (VALID, O.NO_LIMIT, True), (0, O.NO_LIMIT, False)):
        filt = dict(require_flags=require, host_cap=host)
        entries, counts = gs.sweep(dict(filt, skip_rejected=skip), [80 * GB], ps.REDUCE_TOPK, 9)
        got = entries[few].copy()
        there = np.arange(got.shape[2]) < counts[few][:, :, None]
        shift = np.broadcast_to(((few - np.arange(len(few))) * ppm).astype(np.uint64)[:, None, None], got.shape)
        got["idx"][there] -= shift[there]                      # as in the table of the sample
        assert_same_sweep((got, counts[few]), os_.sweep(filt, [80 * GB], O.KIND_TOPK, 9, n_threads=8))
