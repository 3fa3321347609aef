"""Sweeps and compaction where their kernels change over: more factorisations than a
segment of the sweep, so many survivors that its buffers fill and the passes resume,
byte counts beyond a double, windows that start or end inside a group, a factorisation or
a run of factorisations.  Bit for bit against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2601_02311_b200 import synth
from test_gpu_parity import VALID, assert_same_arrays, assert_same_sweep, both, ctx, ps      # noqa: F401

pytestmark = pytest.mark.gpu
GB = synth.GB


def space_of(kind):
    if kind == "segments":              # 1.4 thousand factorisations: two segments
        return synth._space(synth.zoo(2, 21), [2520 * k for k in (1, 2, 3, 4, 5, 6, 8, 9, 10, 12, 16, 18)], t_enum_max=16,
                            k_enum_max=16, n_act=1, n_tpa=1, mode_mask=0b11111)
    space = synth.config("C3", n_models=2)
    if kind == "copies":
        return dict(space, replication_k=3, grad_accum_steps=3, sstar_units=2, n_values=np.asarray([1, 6, 36, 96], dtype=np.uint32))
    if kind == "beyond a double":
        models = space["models"].copy()
        models["param_elems_override"] = [1 << 46, (1 << 46) - 12345]
        return dict(space, models=models)
    if kind == "few modes":
        return dict(space, mode_mask=0b11010)
    return space


@pytest.mark.parametrize("require", [0, VALID])
@pytest.mark.parametrize("kind", ["segments", "plain", "copies", "beyond a double", "few modes"])
def test_sweeps_where_buffers_fill_and_segments_change(ctx, ps, kind, require):      # noqa: F811
    space = space_of(kind)
    gs, os_ = both(ctx, space)
    caps = [80 * GB, 1 << 61] if kind == "beyond a double" else [80 * GB, 10 ** 6 * GB]
    for comm_kind in (ps.COMM_PAPER, ps.COMM_PAPER_PLUS_EXT):
        for host_cap in (O.NO_LIMIT, 64 * GB):
            filt = dict(require_flags=require, host_cap=host_cap, comm_kind=comm_kind)
            for got_kind, want_kind, k in ((ps.REDUCE_PARETO, O.KIND_PARETO, 96), (ps.REDUCE_TOPK, O.KIND_TOPK, 64),
                                           (ps.REDUCE_TOPK, O.KIND_TOPK, 1)):
                want = os_.sweep(filt, caps, want_kind, k, n_threads=8)
                assert_same_sweep(gs.sweep(filt, caps, got_kind, k), want)
                if require:
                    assert_same_sweep(gs.sweep(dict(filt, skip_rejected=1), caps, got_kind, k), want)


@pytest.mark.parametrize("kind", ["plain", "copies", "beyond a double", "few modes"])
def test_compaction_windows_at_the_edges_of_groups_and_runs(ctx, kind):      # noqa: F811
    gs, os_ = both(ctx, space_of(kind))
    nm = bin(space_of(kind)["mode_mask"]).count("1")
    group, unit = nm ** 4, 4 * nm ** 4
    run = 32 * unit
    for first, last in ((0, 1), (group - 1, group + 1), (unit - 1, unit), (3 * group + 7, unit + 2 * group - 1),
                        (run - 1, run + 1), (run, 2 * run), (run + group + 3, 3 * run - group - 5)):
        last = min(last, gs.size)
        if first >= last:
            continue
        for filt in (dict(cap_bytes=192 * GB, require_flags=0, host_cap=O.NO_LIMIT),
                     dict(cap_bytes=1 << 61, require_flags=O.F_GI | O.F_SC, host_cap=64 * GB)):
            assert_same_arrays(gs.compact(first, last - first, filt), os_.compact_range(first, last - first, filt),
                               f"{kind} [{first}, {last})")
