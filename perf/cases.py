"""The work that the library is used for, as cases that can be timed and compared.

A case is a dict of plain values.  Its "path" says which entry point it takes:

  check    one composition, answered on the host (ps_check_composition)
  sweep    a whole space reduced per model and capacity: the memory-vs-communication
           frontier or the top-k list (ps_sweep_pareto)
  window   every output of a window of points (ps_eval_batch without a filter)
  compact  the survivors of a filter in a window, in index order (ps_eval_batch with one)
  select   Algorithm 1 for a batch of queries (ps_select)
  verify   the brute-force verification of a batch of placements (ps_verify_batch)

Inputs follow the distributions of the repository's own configurations
(paper_2601_02311_b200/synth.py); only the seed differs.
"""
import math

import numpy as np
import torch

from paper_2601_02311_b200 import ps, synth

GB = synth.GB
CAPS = [80 * GB, 192 * GB, 141 * GB, 40 * GB]
DIMS = dict(accum=1, sstar=1, copies=1)

# The spaces, by what they stand for: the configuration whose device counts, limits and
# variants they take, and the distribution of their shapes.
#   job       one job of a given parameter count on a data axis of up to 64 devices (C0)
#   data      a zoo of shapes on a data axis of up to 1024 devices (C1)
#   grid      tensor x pipeline x data up to 4096 devices without offloading (C2)
#   pareto    the same with all five modes and larger shapes (C3)
#   stress    up to 16384 devices, every tensor degree, long sequences (C4)
#   ragged    device counts that are not powers of two (nodes of 6, 8, 12 and odd remainders)
SMALL = dict(max_layers=128, max_hidden_mult=128)
LARGE = dict(max_layers=160, max_hidden_mult=256)
LONG = dict(LARGE, seqs=(2048, 4096, 8192, 16384, 32768), max_micro_batch=64)
FAMILIES = {"job": ("C0", None), "data": ("C1", SMALL), "grid": ("C2", SMALL), "pareto": ("C3", LARGE),
            "stress": ("C4", LONG), "ragged": ("C3", LARGE)}
RAGGED_COUNTS = [1, 2, 3, 6, 7, 12, 24, 30, 36, 48, 96, 97, 360, 384, 768, 1000, 1536]
# factorisations x variants of a model, and placement codes of a factorisation and variant
GROUPS = {"job": 7, "data": 22, "grid": 1160, "pareto": 1160, "stress": 2720, "ragged": 2104}
CODES = {"job": 625, "data": 625, "grid": 256, "pareto": 625, "stress": 625, "ragged": 625}


def points_per_model(case):
    return GROUPS[case["family"]] * CODES[case["family"]]


def sweep(name, family, models, reduce, **more):
    case = dict(DIMS, path="sweep", family=family, models=models, reduce=reduce, entries=64, caps=1, host_gb=0,
                priced=False, skip=False, fresh=False)
    case.update(more)
    return dict(case, name=name)


def listed():
    return [
        # a planner or a command line asks about one composition and waits for the answer
        dict(path="check", devices=512, tensor=8, pipeline=4, code=49, variant=1, cap_gb=80, name="check_one"),
        # one job's frontier under two device sizes, read back on the host
        sweep("frontier_job", "job", 1, "pareto", caps=2, host_gb=64, fresh=True),
        # a handful of candidate shapes, changed between calls, frontier read back (interactive what-if)
        sweep("frontier_few", "pareto", 8, "pareto", caps=2, host_gb=64, fresh=True),
        # a zoo of shapes: the frontiers, leaving out what the filter rejects at sight
        sweep("frontier_zoo", "pareto", 1024, "pareto", caps=2, host_gb=64, skip=True),
        # the stress configuration: both reductions, every factorisation evaluated
        sweep("topk_stress", "stress", 4096, "topk"),
        sweep("frontier_stress", "stress", 4096, "pareto", caps=2, host_gb=64),
        # clusters of awkward sizes, gradient accumulation, two copies of every shard
        sweep("topk_ragged", "ragged", 250, "topk", entries=10, accum=4, copies=2),
        # every figure of a large window that starts anywhere (feeding another program)
        dict(DIMS, path="window", family="pareto", models=64, first=311, count=1 << 25, name="window_all"),
        # the valid points under 80 GB of a window: few survive
        dict(DIMS, path="compact", family="stress", models=64, first=12_345_678, count=1 << 25, cap_gb=80, valid=True,
             name="window_valid"),
        # every placement that fits, valid or not: many survive
        dict(DIMS, path="compact", family="grid", models=64, first=1001, count=(1 << 23) + 77, cap_gb=192, valid=False,
             name="window_fits"),
        # Algorithm 1 over a large table of jobs
        dict(path="select", queries=1 << 24, tensor=8, name="select_many"),
        # all 625 placements on one to four devices against single-device training
        dict(path="verify", units=4, width=16, batch=2, accum=2, steps=3, cases=2500, name="verify_grid"),
    ]


def between(rng, lo, hi):
    """A whole number, even over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    path = rng.choice(["sweep"] * 6 + ["window", "compact", "compact", "select", "verify", "check"])
    dims = dict(accum=rng.choice([1, 1, 1, 2, 4, 8]), sstar=rng.choice([1, 1, 2]), copies=rng.choice([1, 1, 1, 2, 3, 4]))
    if path == "check":
        tensor, pipeline = 1 << rng.randrange(5), rng.choice([1, 2, 3, 4, 6, 8])
        return dict(path=path, devices=tensor * pipeline * between(rng, 1, 512), tensor=tensor, pipeline=pipeline,
                    code=rng.randrange(625), variant=rng.randrange(2), cap_gb=rng.choice([40, 80, 141, 192]))
    if path == "select":
        return dict(path=path, queries=between(rng, 300, 1 << 24), tensor=rng.choice([2, 4, 8, 16, 72]))
    if path == "verify":
        case = dict(path=path, units=rng.randint(1, 6), width=rng.randint(1, 24), batch=rng.randint(1, 3),
                    accum=rng.randint(1, 3), steps=rng.randint(1, 4), cases=between(rng, 40, 5000))
        # no case's training is longer than the listed one's
        while case["units"] * case["width"] * case["steps"] * (case["batch"] * case["accum"] + 2) > 1000:
            case["width"] -= 1
        return case
    if path == "sweep":
        family = rng.choice(["job", "data", "grid", "pareto", "pareto", "stress", "ragged"])
        caps = rng.randint(1, 4)
        reduce = rng.choice(["pareto", "pareto", "topk"])
        # what the longest listed sweep evaluates, less where degrees are not powers of two or shards have copies
        most = 6_000_000_000 if family != "ragged" and dims["copies"] == 1 else 700_000_000
        most //= (caps if reduce == "topk" else 1) * points_per_model(dict(family=family))
        models = between(rng, 1, min(4096, most))
        entries = rng.choice([1, 5, 10, 33, 64]) if reduce == "topk" else rng.choice([32, 64, 100])
        return dict(dims, path=path, family=family, models=models, reduce=reduce, entries=entries, caps=caps,
                    host_gb=rng.choice([64, 64, 8, 500]) if reduce == "pareto" else rng.choice([0, 0, 64]),
                    priced=rng.random() < 0.2, skip=rng.random() < 0.5, fresh=rng.random() < 0.3)
    family = rng.choice(["data", "grid", "pareto", "stress", "ragged"])
    models = 64
    of_two = 2 * points_per_model(dict(family=family))
    room = models // 2 * of_two
    valid = rng.random() < 0.7
    if path == "window":
        count = between(rng, 700, min(room, 1 << 25))
    else:                                       # (valid points lie far apart: two models' worth has some)
        count = between(rng, of_two if valid else 5000, min(room, 1 << 24))
    case = dict(dims, path=path, family=family, models=models, first=rng.randint(0, room - count), count=count)
    if path == "compact":
        case.update(cap_gb=rng.choice([40, 80, 192]), valid=valid)
    return case


# ---------------------------------------------------------------- inputs
_contexts = {}


def context():
    """The one handle that a program keeps for its device and stream."""
    if 0 not in _contexts:
        _contexts[0] = ps.Context(0)
    return _contexts[0]


def shapes(family, n, seed):
    limits = FAMILIES[family][1]
    if limits is not None:
        return synth.zoo(n, seed, **limits)
    out = synth.zoo(n, seed, **SMALL)            # a job: its parameter count given, no activations
    rng = np.random.default_rng(seed)
    out["param_elems_override"] = rng.integers(10**9, 10**12, n)
    out["act_enabled"] = 0
    return out


def description(case, seed):
    space = synth.config(FAMILIES[case["family"]][0], n_models=1)
    space["models"] = shapes(case["family"], case["models"], seed)
    if case["family"] == "ragged":
        space["n_values"] = np.asarray(RAGGED_COUNTS, dtype=np.uint32)
        space["t_enum_max"], space["k_enum_max"] = 12, 36
    return dict(space, sstar_units=case["sstar"], grad_accum_steps=case["accum"], replication_k=case["copies"])


def queries(n, seed):
    """synth.select_queries' distribution as packed 32-byte records, drawn on the device."""
    g = torch.Generator("cuda").manual_seed(seed)

    def whole(lo, hi):
        return torch.randint(lo, hi + 1, (n,), generator=g, device="cuda", dtype=torch.int64)

    params = whole(1000, 9999) * torch.tensor([10**e for e in range(5, 10)], device="cuda")[whole(0, 4)]
    layer = torch.where(whole(0, 7) > 0, params // whole(12, 160), 0)
    memory = torch.tensor([16, 24, 40, 80, 141, 192], device="cuda")[whole(0, 5)] * GB
    devices = torch.where(whole(0, 5) > 0, torch.ones_like(params) << whole(0, 14), whole(1, 3000))
    last = devices | (2 << 32) | (2 << 40) | (12 << 48) | (whole(0, 1) << 56)
    return torch.stack([params, layer, memory, last], dim=1).contiguous().view(torch.uint8).view(-1)


def problems(case, seed):
    """Training problems for one to four devices and the (code, devices) pairs to run on them."""
    rng = np.random.default_rng(seed)
    size, per = case["units"] * case["width"], case["batch"] * case["width"]
    chunks, offsets, at = [], {}, 0
    for devices in (1, 2, 3, 4):
        samples = case["accum"] * devices * per
        chunks += [rng.uniform(0.5, 1.5, size), rng.normal(size=samples), rng.uniform(-0.8, 0.8, samples)]
        offsets[devices] = at
        at += size + 2 * samples
    grid = np.zeros(case["cases"], dtype=ps.VERIFY_CASE_DTYPE)
    k = np.arange(case["cases"]) if case["cases"] >= 2500 else np.sort(rng.choice(2500, case["cases"], replace=False))
    grid["code"], grid["D"] = k % 625, 1 + k // 625 % 4
    grid["data_offset"] = np.array([offsets[1 + i] for i in range(4)], dtype=np.uint64)[grid["D"] - 1]
    return grid, np.concatenate(chunks)


def prepare(case, seed):
    ctx, path = context(), case["path"]
    s = {"case": case, "ctx": ctx}
    if path == "check":
        s["shape"] = synth.zoo(1, seed, **LARGE)
    elif path == "select":
        s["queries"] = queries(case["queries"], seed)
        s["out"] = torch.empty(case["queries"] * 32, dtype=torch.uint8, device="cuda")
    elif path == "verify":
        s["grid"], s["data"] = problems(case, seed)
    else:
        description_ = description(case, seed)
        s["space"] = space = ctx.space(description_)
        if path == "sweep":
            s["caps"] = CAPS[:case["caps"]]
            s["kind"] = ps.REDUCE_PARETO if case["reduce"] == "pareto" else ps.REDUCE_TOPK
            s["filter"] = dict(require_flags=ps.F_VALID, host_cap=case["host_gb"] * GB if case["host_gb"] else ps.NO_LIMIT,
                               comm_kind=ps.COMM_PAPER if case["priced"] else ps.COMM_PAPER_PLUS_EXT,
                               skip_rejected=case["skip"])
            if case["fresh"]:
                s["table"] = torch.from_numpy(description_["models"].view(np.uint8).copy()).pin_memory()
            else:
                s["out"], s["counts"] = space.alloc_sweep(case["caps"], case["entries"])
        else:
            s["out"] = {k: v.zero_() for k, v in space.alloc_outputs(case["count"]).items()}
            if path == "compact":
                s["filter"] = dict(require_flags=ps.F_VALID if case["valid"] else 0, cap_bytes=case["cap_gb"] * GB)
                s["idx"] = torch.zeros(case["count"], dtype=torch.int64, device="cuda")
                s["n"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    case, ctx, path = s["case"], s["ctx"], s["case"]["path"]
    if path == "check":
        n, t, k = case["devices"], case["tensor"], case["pipeline"]
        return ctx.check_composition(s["shape"], n, t, k, n // (t * k), 156, 31, case["code"],
                                     act_variant=case["variant"], cap_bytes=case["cap_gb"] * GB)
    if path == "sweep":
        if case["fresh"]:                      # another table of shapes, the answer on the host
            s["space"].set_models(s["table"])
            entries, counts = s["space"].sweep(s["filter"], s["caps"], s["kind"], case["entries"])
            return entries.view(np.int64), counts.astype(np.int64)
        s["space"].sweep_into(s["filter"], s["caps"], s["kind"], case["entries"], s["out"], s["counts"])
        return s["out"].view(torch.int64), s["counts"]
    if path == "window":
        s["space"].eval_batch_into(case["first"], case["count"], s["out"])
        return s["out"]
    if path == "compact":
        s["space"].eval_batch_into(case["first"], case["count"], s["out"], s["filter"], s["idx"], s["n"])
        return dict(s["out"], idx=s["idx"], n=s["n"])
    if path == "select":
        ctx.select_into(s["queries"], case["queries"], s["out"], tp_degree=case["tensor"])
        return s["out"].view(torch.int64)
    shape = dict(units=case["units"], h=case["width"], b=case["batch"], accum=case["accum"], steps=case["steps"])
    result, theta = ctx.verify_batch(shape, s["grid"], s["data"], want_theta=True)
    return dict({k: result[k].astype(np.int64) for k in ("mem", "comm", "host", "match")},
                max_rel_err=np.ascontiguousarray(result["max_rel_err"]), theta=theta)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    path = case["path"]
    if path == "check":
        return {"bytes": 48 + 40, "flops": 100}
    if path == "select":
        return {"bytes": 64 * case["queries"], "flops": 20 * case["queries"]}
    if path == "verify":
        size = case["units"] * case["width"]
        samples = 2.5 * case["accum"] * case["batch"]           # over one to four devices
        data = 4 * size + 8 * samples * case["width"]
        # forward, backward and update of the placed and of the single-device run
        flops = 2 * case["steps"] * size * (50 * samples + 20 * 2.5)
        return {"bytes": 8 * data + case["cases"] * (16 + 40 + 8 * size), "flops": case["cases"] * flops}
    if path == "window":
        return {"bytes": 36 * case["count"], "flops": 4 * case["count"]}
    if path == "compact":
        # survivors: nearly all points that fit without a required flag, a few in ten thousand valid ones
        share = 0.0005 if case["valid"] else {40: 0.3, 80: 0.4}.get(case["cap_gb"], 0.5)
        return {"bytes": 44 * share * case["count"], "flops": case["count"]}
    rows = case["models"] * case["caps"]
    groups = case["models"] * GROUPS[case["family"]]
    # a compare per point; where rejected factorisations may be left out, a test per factorisation
    passes = case["caps"] if case["reduce"] == "topk" else 1
    flops = groups / 4 if case["skip"] else groups * CODES[case["family"]]
    return {"bytes": 48 * case["models"] + rows * (40 * case["entries"] + 4), "flops": passes * flops}


def tolerance(case):
    """Whole numbers are exact.  The verifier trains in fp64: with every input moved by one unit in the last
    place (what another order of the sums does to a result) its parameters move by 2e-16 of their norm and its
    largest relative error, a quotient with a small divisor where a placement has left the trajectory, by 1.5e-13."""
    return {"rel": 1e-12, "max": 1e-11, "differ": 0.0} if case["path"] == "verify" else "exact"
