"""Sweeps and compaction where their kernels change over: more factorisations than a
segment of the sweep, so many survivors that its buffers fill and the passes resume,
byte counts beyond a double, windows that start or end inside a group, a factorisation or
a run of factorisations.  Bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2601_02311_b200 import synth
from test_gpu_parity import VALID, assert_same_arrays, assert_same_sweep, both, ctx, ps      # noqa: F401

pytestmark = pytest.mark.gpu
GB = synth.GB


def space_of(kind):
    if kind == "segments":              # 1.4 thousand factorisations: two segments
        return synth._space(synth.zoo(2, 21), [2520 * k for k in (1, 2, 3, 4, 5, 6, 8, 9, 10, 12, 16, 18)], t_enum_max=16,
                            k_enum_max=16, n_act=1, n_tpa=1, mode_mask=0b11111)
    if kind == "stress":                # points that cost nothing: one pair in each of 1360 (unit, variant)
        return synth.config("C4", n_models=2)
    if kind == "ragged":
        return dict(synth.config("C3", n_models=2), n_values=np.asarray([1, 7, 36, 96, 360, 1000, 1536], dtype=np.uint32),
                    t_enum_max=12, k_enum_max=36)
    if kind == "crowded cells":         # activations outweigh the rest: a quarter of the candidates pass the staircase
        return dict(space_of("ragged"), models=synth.zoo(2, 3, max_layers=160, max_hidden_mult=128, seqs=(1 << 17,),
                                                         max_micro_batch=64), n_act_variants=1, replication_k=3)
    if kind == "tied in a unit":        # 122 pairs of 460 (triple, variant) under a host budget of 6 GB
        models = synth.zoo(1, 5)
        models["unit_from_shape"], models["act_enabled"] = 0, 0
        return dict(synth._space(models, list(range(1, 65)), t_enum_max=1, k_enum_max=1, n_act=2, n_tpa=2,
                                 mode_mask=0b11111), grad_accum_steps=8)
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
@pytest.mark.parametrize("kind", ["segments", "plain", "copies", "beyond a double", "few modes", "stress", "ragged",
                                  "tied in a unit", "crowded cells"])
def test_sweeps_where_buffers_fill_and_segments_change(ctx, ps, kind, require):      # noqa: F811
    space = space_of(kind)
    gs, os_ = both(ctx, space)
    caps = [80 * GB, 1 << 61] if kind == "beyond a double" else [80 * GB, 10 ** 6 * GB]
    for comm_kind in (ps.COMM_PAPER, ps.COMM_PAPER_PLUS_EXT):
        for host_cap in (O.NO_LIMIT, (6 if kind == "tied in a unit" else 64) * GB):
            filt = dict(require_flags=require, host_cap=host_cap, comm_kind=comm_kind)
            for got_kind, want_kind, k in ((ps.REDUCE_PARETO, O.KIND_PARETO, 128), (ps.REDUCE_TOPK, O.KIND_TOPK, 64),
                                           (ps.REDUCE_TOPK, O.KIND_TOPK, 1)):
                want = os_.sweep(filt, caps, want_kind, k, n_threads=8)
                assert_same_sweep(gs.sweep(filt, caps, got_kind, k), want)
                if require:
                    assert_same_sweep(gs.sweep(dict(filt, skip_rejected=1), caps, got_kind, k), want)


def milliseconds(call):
    """The fastest of five, after one to warm up."""
    times = []
    for _ in range(6):
        begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        begin.record()
        call()
        end.record()
        end.synchronize()
        times.append(begin.elapsed_time(end))
    return min(times[1:])


@pytest.mark.parametrize("kind,reduce", [("plain", "pareto"), ("stress", "pareto"), ("ragged", "pareto"),
                                         ("tied in a unit", "pareto"), ("plain", "topk"), ("stress", "topk"),
                                         ("ragged", "topk")])
def test_tied_points_do_not_slow_a_sweep_down(ctx, ps, kind, reduce):      # noqa: F811
    """Many points of one (bytes, communication) pair are one entry of a frontier: the path for
    frontiers that outgrow the block's buffer, which evaluates every point again for each entry and
    takes fifty times as long or more, is not for them.  Nor does a top-k list look at each of tens
    of thousands of points that send nothing (sixteen times as long and more): their bytes decide.
    The same table without the ties takes about as long as with them, half at least."""
    few = space_of(kind)
    space = dict(few, models=np.tile(few["models"], 128))
    free = dict(require_flags=0, host_cap=O.NO_LIMIT)
    if kind == "tied in a unit":
        models = space["models"].copy()
        models["unit_from_shape"] = 1
        tied = dict(require_flags=VALID, host_cap=6 * GB, comm_kind=ps.COMM_PAPER_PLUS_EXT)
        other, without = dict(space, models=models), tied
    else:
        tied = dict(free, comm_kind=ps.COMM_PAPER)
        other, without = space, dict(free, comm_kind=ps.COMM_PAPER_PLUS_EXT)
    kind_of, entries = (ps.REDUCE_PARETO, 128) if reduce == "pareto" else (ps.REDUCE_TOPK, 64)
    took = []
    for description, filt in ((space, tied), (other, without)):
        gpu = ctx.space(description)
        out, counts = gpu.alloc_sweep(1, entries)
        took.append(milliseconds(lambda: gpu.sweep_into(filt, [10 ** 6 * GB], kind_of, entries, out, counts)))
        ctx.check_status()
        assert reduce == "topk" or int(counts.max()) <= 128
    assert took[0] < 8 * took[1], took


def test_tables_beyond_a_double_keep_their_pace(ctx, ps):      # noqa: F811
    """With 64 micro-batches a step the largest shapes' volumes pass 2^53 and the table is swept in
    64-bit integers, whose compares would take twice as long: device bytes stay in doubles."""
    took = []
    for accum in (64, 1):
        gpu = ctx.space(dict(synth.config("C4", n_models=512), grad_accum_steps=accum))
        out, counts = gpu.alloc_sweep(1, 64)
        filt = dict(require_flags=0, host_cap=O.NO_LIMIT)
        took.append(milliseconds(lambda: gpu.sweep_into(filt, [80 * GB], ps.REDUCE_TOPK, 64, out, counts)))
    assert took[0] < 1.6 * took[1], took


def test_capacities_beyond_a_double(ctx, ps):      # noqa: F811
    """Capacities at a point's bytes and one below, where a double no longer holds them."""
    models = synth.zoo(1, 0)
    for field, value in dict(param_elems_override=(1 << 46) - 5, layers=1, hidden=8191, heads=3275, vocab=1, seq=(1 << 17) - 1,
                             micro_batch=(1 << 10) - 1, w_param=15, w_opt=16, w_grad=13).items():
        models[field] = value
    space = synth._space(models, [1, 2, 3, 8], t_enum_max=2, k_enum_max=2, n_act=2, n_tpa=2, mode_mask=0b11111)
    gs, os_ = both(ctx, space)
    mem = np.unique(os_.eval_range(0, gs.size)["mem"])
    mem = mem[mem > 1 << 53]
    assert len(mem) > 100 and np.any(mem.astype(np.float64).astype(np.uint64) != mem)
    for exact in mem[::len(mem) // 12]:
        for cap in (int(exact), int(exact) - 1):
            filt = dict(cap_bytes=cap, require_flags=0, host_cap=O.NO_LIMIT)
            assert_same_arrays(gs.compact(0, gs.size, filt), os_.compact_range(0, gs.size, filt), f"capacity {cap}")
            for got_kind, want_kind, k in ((ps.REDUCE_PARETO, O.KIND_PARETO, 128), (ps.REDUCE_TOPK, O.KIND_TOPK, 64)):
                for require in (0, VALID):
                    filt = dict(require_flags=require, host_cap=O.NO_LIMIT)
                    assert_same_sweep(gs.sweep(filt, [cap], got_kind, k), os_.sweep(filt, [cap], want_kind, k))


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


@pytest.mark.parametrize("mode_mask", [0b11111, 0b11010])
@pytest.mark.parametrize("params", [1 << 41, 1 << 46])      # byte counts in doubles and in 64-bit integers
def test_host_bytes_at_the_end_of_their_range(ctx, ps, params, mode_mask):      # noqa: F811
    """Offloaded activations of 2^62 - 2^48.9 bytes with offloaded states on top: more than 2^62."""
    models = synth.zoo(1, 0)
    for field, value in dict(param_elems_override=params, layers=1, hidden=8192, heads=3276, vocab=1, seq=1 << 17,
                             micro_batch=1 << 10, w_param=16, w_opt=16, w_grad=16).items():
        models[field] = value
    space = dict(synth._space(models, [1, 2, 3, 8], t_enum_max=2, k_enum_max=2, n_act=2, n_tpa=2, mode_mask=mode_mask),
                 grad_accum_steps=8)
    gs, os_ = both(ctx, space)
    assert int(os_.eval_range(0, gs.size)["host"].max()) > 1 << 62
    for host_cap in (O.NO_LIMIT, 1 << 62, (1 << 62) + (1 << 45)):
        for cap in (1 << 50, O.NO_LIMIT):
            filt = dict(cap_bytes=cap, require_flags=0, host_cap=host_cap)
            assert_same_arrays(gs.compact(0, gs.size, filt), os_.compact_range(0, gs.size, filt), f"{cap}, {host_cap}")
            for got_kind, want_kind, k in ((ps.REDUCE_PARETO, O.KIND_PARETO, 128), (ps.REDUCE_TOPK, O.KIND_TOPK, 64)):
                assert_same_sweep(gs.sweep(filt, [cap], got_kind, k), os_.sweep(filt, [cap], want_kind, k))
