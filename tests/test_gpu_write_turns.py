"""Compactions that list more factorisations than the write pass has places for, so that its blocks take several
turns with one table of triples: a warp for each of one, two and four variants, counts that leave a part of a block
without a unit in the last turn, windows that start and end inside a group, units that are left out.  Bit for bit
against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2601_02311_b200 import synth
from test_gpu_parity import VALID, assert_same_arrays, both, ctx, ps      # noqa: F401

pytestmark = pytest.mark.gpu
GB = synth.GB


@pytest.mark.parametrize("variants", [(1, 1), (1, 2), (2, 1), (2, 2)])
@pytest.mark.parametrize("kind", ["powers of two", "copies", "ragged"])
def test_blocks_that_take_several_units(ctx, ps, kind, variants):      # noqa: F811
    nv, nt = variants
    space = dict(synth.config("C4", n_models=90), mode_mask=0b01001, n_act_variants=nv, n_tpa_variants=nt)
    if kind == "copies":
        space["replication_k"] = 2
    if kind == "ragged":
        space["n_values"] = np.asarray([1, 2, 3, 6, 7, 12, 24, 30, 36, 48, 96, 97, 360, 384, 768, 1000, 1536], dtype=np.uint32)
        space["t_enum_max"], space["k_enum_max"] = 12, 36
    gs, os_ = both(ctx, space)
    per_unit, teams = 16 * nv * nt, 4 // (nv * nt)                  # teams: units that a block takes in a turn
    places = 64 * teams * torch.cuda.get_device_properties(0).multi_processor_count       # of a turn, at most
    units = gs.size // per_unit // teams * teams - teams + 1        # one is left for a block's last turn
    count = units * per_unit - 5
    # nothing required; nothing of the composition; valid placements under a capacity
    for filt in (dict(require_flags=0), dict(require_flags=O.F_SC, cap_bytes=400 * GB),
                 dict(require_flags=VALID, cap_bytes=80 * GB)):
        want = os_.compact_range(3, count - 3, filt)
        if filt["require_flags"] == 0:
            listed = len(np.unique(want["idx"] // np.uint64(per_unit)))
            assert listed == units > places
        assert_same_arrays(gs.compact(3, count - 3, filt), want, str(filt))
