"""Rows whose columns span few columns, which the warp-per-row numeric kernels
accumulate by column and the symbolic ones count by a bitmap: at the widest
span of each table, one column past it,
and with sums of zero, infinities and NaN (which stay entries of C), against
the CPU oracle."""

import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2206_07244_gb300 as ops  # noqa: E402

ops.build()


def product(size, span, first, seed):
    """37 rows of C with `size` entries whose columns span exactly `span`
    columns from `first` on, as sums of five overlapping B rows each."""
    rng = np.random.default_rng(seed)
    a, b = [], []
    for i in range(37):
        pool = np.sort(rng.choice(np.arange(1, span - 1), size - 2, replace=False))
        pool = np.concatenate([[0], pool, [span - 1]]) + first
        a.append(np.arange(len(b), len(b) + 5))
        parts = [np.sort(rng.choice(pool, size // 3, replace=False)) for _ in range(3)]
        b += [pool[: size // 2], pool[size // 2:]] + parts

    def csr(lists, cols):
        rpt = np.zeros(len(lists) + 1, dtype=np.int32)
        np.cumsum([len(x) for x in lists], out=rpt[1:])
        col = np.concatenate(lists).astype(np.int32)
        return W.Csr(len(lists), cols, rpt, col, rng.integers(-3, 4, col.size).astype(np.float64))

    return csr(a, len(b)), csr(b, first + span + 5)


@pytest.mark.parametrize("first", [0, (1 << 22) + 3])
@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("slots, size", [(256, 66), (256, 128), (512, 129), (512, 256), (1024, 257), (1024, 512)])
def test_widest_span(slots, size, extra, first):
    A, B = product(size, slots * 12 // 8 // 32 * 32 + extra, first, 3)
    dA, dB = (ops.CSR.from_arrays(m.rows, m.cols, m.rpt, m.col, m.val) for m in (A, B))
    with ops.Handle() as h:
        C = h.multiply(dA, dB)
        h.status()
        assert sum(h.stats()["num_bins"]) == A.rows
    for g, w in zip(C.numpy(), oracle.spgemm(A, B)[:3]):
        assert np.array_equal(g, w)


@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("slots, size", [(512, 150), (1024, 300)])   # about 2.5 size products a row
def test_widest_span_of_the_symbolic_bitmap(slots, size, extra):
    A, B = product(size, slots * 32 + extra, 11, 4)
    table = ops.kernel_table(0)
    kernel = next(k for k, t in enumerate(table) if t[0] == 32 and t[2] == slots)
    cfg = ops.default_config()
    cfg["sym_kernel"], cfg["sym_range"] = [kernel, len(table) - 1], [table[kernel][3], -1]
    dA, dB = (ops.CSR.from_arrays(m.rows, m.cols, m.rpt, m.col, m.val) for m in (A, B))
    with ops.Handle(cfg) as h:
        C = h.multiply(dA, dB)
        h.status()
    for g, w in zip(C.numpy(), oracle.spgemm(A, B)[:3]):
        assert np.array_equal(g, w)


def test_special_values():
    A, B = product(200, 400, 7, 5)
    A.val[:] = 1.0
    B.val[::7] = np.inf
    B.val[3::11] = np.nan
    B.val[5::13] = -np.inf
    B.val[1::2] = 0.0
    dA, dB = (ops.CSR.from_arrays(m.rows, m.cols, m.rpt, m.col, m.val) for m in (A, B))
    with ops.Handle() as h:
        C = h.multiply(dA, dB)
        h.status()
    rpt, col, val = oracle.spgemm(A, B)[:3]
    got = C.numpy()
    assert np.array_equal(got[0], rpt) and np.array_equal(got[1], col)
    assert np.array_equal(got[2], val, equal_nan=True)


def even(rows, per_row, cols, seed, reverse=False):
    """Every row `per_row` distinct columns, ascending (or descending)."""
    rng = np.random.default_rng(seed)
    col = np.sort(rng.random((rows, cols)).argpartition(per_row - 1, axis=1)[:, :per_row], axis=1)
    if reverse:
        col = col[:, ::-1]
    return W.Csr(rows, cols, np.arange(0, rows * per_row + 1, per_row, dtype=np.int32), col.astype(np.int32).ravel(),
                 rng.integers(-3, 4, rows * per_row).astype(np.float64))


def numeric_ms(h, dA, dB):
    C = h.multiply(dA, dB)
    best = np.inf
    for _ in range(9):
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        h.numeric_values(dA, dB, C)
        e1.record()
        h.status()
        best = min(best, e0.elapsed_time(e1))
    return best, C


@pytest.mark.parametrize("entries, length", [(200, 2), (400, 2), (400, 4), (1600, 4), (1600, 8)])
def test_short_rows_of_B_are_not_added_one_at_a_time(entries, length):
    # descending columns take the table whatever the rows of B are; ascending
    # ones must not be slower by more than a tenth of it and the noise
    times = []
    A = even(4000, entries, 2000, 1)
    for reverse in (False, True):
        B = even(2000, length, 100, 2, reverse)
        dA, dB = (ops.CSR.from_arrays(m.rows, m.cols, m.rpt, m.col, m.val) for m in (A, B))
        with ops.Handle() as h:
            ms, C = numeric_ms(h, dA, dB)
        times.append(ms)
        for g, w in zip(C.numpy(), oracle.spgemm(A, B)[:3]):
            assert np.array_equal(g, w)
    assert times[0] < 1.25 * times[1], times
