"""verify_batch around the size up to which its inputs and results travel through pinned memory, and without
cases: the same records and parameters as in small portions."""
import numpy as np
import pytest

from test_gpu_verify import ctx, problems, ps      # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("want_theta", [False, True])
def test_no_cases(ctx, ps, want_theta):      # noqa: F811
    none = np.zeros(0, dtype=ps.VERIFY_CASE_DTYPE)
    for data in (np.zeros(0), np.ones(7)):
        got = ctx.verify_batch(dict(units=3, h=5, b=2), none, data, want_theta=want_theta)
        records, theta = got if want_theta else (got, np.zeros((0, 15)))
        assert records.shape == (0,) and records.dtype == ps.VERIFY_RESULT_DTYPE
        assert theta.shape == (0, 15) and theta.dtype == np.float64


@pytest.mark.parametrize("many_inputs", [False, True])
@pytest.mark.parametrize("over", [-1, 0, 1])
def test_sizes_around_the_limit(ctx, ps, over, many_inputs):      # noqa: F811
    units, h, b = (4, 8, 2) if many_inputs else (6, 24, 2)
    data, offsets, _ = problems(units, h, b, 1, seed=5)
    shape, each = dict(units=units, h=h, b=b, steps=1), 40 + 8 * units * h
    n = (ps.PINNED_RESULT_BYTES // each if not many_inputs else 3000) + over
    cases = np.zeros(n, dtype=ps.VERIFY_CASE_DTYPE)
    k = np.arange(n)
    cases["code"], cases["D"] = k % 625, 1 + k // 625 % 4
    cases["data_offset"] = np.array([offsets[1 + d] for d in range(4)], dtype=np.uint64)[cases["D"] - 1]
    if many_inputs:                                    # as many problems as make the inputs that large
        copies = (ps.PINNED_RESULT_BYTES - cases.nbytes) // data.nbytes + (over > 0)
        cases["data_offset"] += (k % copies).astype(np.uint64) * np.uint64(len(data))
        data = np.tile(data, copies)
    data.flags.writeable = False
    records, theta = ctx.verify_batch(shape, cases, data, want_theta=True)
    assert np.array_equal(ctx.verify_batch(shape, cases, data), records)
    for first in range(0, n, 2500):
        some, some_theta = ctx.verify_batch(shape, cases[first:first + 2500], data, want_theta=True)
        assert np.array_equal(some, records[first:first + 2500])
        assert np.array_equal(some_theta, theta[first:first + 2500])
