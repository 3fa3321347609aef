"""The sweeps' screening holds rounded figures against the capacity: no factorisation may be lost
whose only survivor has exactly as many bytes as the capacity or the host budget allows.  Bit for
bit against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from test_gpu_parity import VALID, assert_same_sweep, both, ctx, ps      # noqa: F401
from test_gpu_reduction_edges import GB, space_of

pytestmark = pytest.mark.gpu


def some(values, n):
    values = np.unique(values)
    return [int(v) for v in values[::max(1, len(values) // n)]]


@pytest.mark.parametrize("require", [VALID, O.F_USES_HOST, O.F_PAPER_PRICED | O.F_CV, O.F_ACT_AVAIL])
@pytest.mark.parametrize("kind", ["plain", "ragged", "copies", "few modes", "beyond a double"])
def test_capacities_at_a_factorisations_least_bytes(ctx, ps, kind, require):      # noqa: F811
    space = space_of(kind)
    gs, os_ = both(ctx, space)
    nm = bin(space["mode_mask"]).count("1")
    all_ = os_.eval_range(0, gs.size)
    passes = (all_["flags"] & require) == require
    by_unit = np.where(passes, all_["mem"], np.uint64(1 << 63)).reshape(-1, 4 * nm ** 4)
    least = by_unit.min(axis=1)
    tries = [(cap, O.NO_LIMIT) for exact in some(least[least < 1 << 62], 5) for cap in (exact, max(exact, 1) - 1)]
    tries += [(O.NO_LIMIT, O.NO_LIMIT), (17, O.NO_LIMIT), (80 * GB, 0)]
    # with next to no capacity the offloaded points decide, and with them the host budget
    tries += [(cap, host) for exact in some(all_["host"][passes & (all_["mem"] == 0)], 4)
              for cap, host in ((0, exact), (1, max(exact, 1) - 1))]
    for cap, host in tries:
        filt = dict(require_flags=require, host_cap=host)
        for got_kind, want_kind, k in ((ps.REDUCE_PARETO, O.KIND_PARETO, 64), (ps.REDUCE_TOPK, O.KIND_TOPK, 3)):
            assert_same_sweep(gs.sweep(filt, [cap], got_kind, k), os_.sweep(filt, [cap], want_kind, k, n_threads=8))
