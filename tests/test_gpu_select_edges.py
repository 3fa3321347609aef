"""Algorithm 1 per query where its kernel changes over: records on 16-byte instead of 32-byte
boundaries, counts around a block's, quotients at and beyond what its divisions by a reciprocal
take, device counts that are not powers of two.  Whole numbers: equal to the oracle's."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2601_02311_b200 import synth
from test_gpu_parity import ctx, ps, to_query_records      # noqa: F401

pytestmark = pytest.mark.gpu
NAMES = ("mem", "comm", "branch", "T", "code_dp", "flags")


def edge_queries(n, seed):
    q = synth.select_queries(n, seed=seed)
    rng = np.random.default_rng(seed)
    q[::2, 3] = rng.integers(1, 1 << 24, len(q[::2]))
    q[::3, 0] = (1 << rng.integers(1, 46, len(q[::3]))) + rng.integers(-1, 2, len(q[::3]))
    ends = [(1 << 50) - 1, 1 << 50, (1 << 50) + 1, (1 << 52) - 1, 1 << 52, (1 << 55) - 3]
    q[5::7, 0] = np.resize(ends, len(q[5::7]))             # (beyond the documented range)
    q[5::7, 1] = np.resize(ends[::-1], len(q[5::7]))
    # multiples of the device count and their neighbours
    d = q[6::7, 3].astype(np.uint64)
    q[6::7, 0] = d * (((1 << 46) - 1) // d) - rng.integers(0, 2, len(d)).astype(np.uint64)
    q[::5, 2] = 1 << 30                                    # small devices: the tensor-parallel branch
    return q


@pytest.mark.parametrize("shift", [(0, 0), (16, 0), (0, 16), (16, 16)])
@pytest.mark.parametrize("n", [1, 127, 128, 257, 5003])
def test_select_on_every_alignment(ctx, ps, n, shift):      # noqa: F811
    q = edge_queries(max(n, 7), n)[:n]
    records = to_query_records(ps, q)
    d_q = torch.zeros(n * 32 + 32, dtype=torch.uint8, device="cuda")
    d_o = torch.full((n * 32 + 64,), 0xAB, dtype=torch.uint8, device="cuda")
    d_q[shift[0]:shift[0] + n * 32] = torch.from_numpy(records.view(np.uint8).reshape(-1).copy()).cuda()
    out = d_o[shift[1]:shift[1] + n * 32]
    for tp_degree in (1, 8, 64, 72):
        ctx.select_into(d_q[shift[0]:], n, out, tp_degree=tp_degree)
        ctx.check_status()
        got = out.cpu().numpy().view(ps.SELECT_RESULT_DTYPE)
        want = O.select(q, tp_degree=tp_degree)
        for j, name in enumerate(NAMES):
            assert np.array_equal(got[name].astype(np.uint64), want[:, j]), (name, tp_degree)
    rest = torch.cat([d_o[:shift[1]], d_o[shift[1] + n * 32:]])
    assert bool((rest == 0xAB).all())
