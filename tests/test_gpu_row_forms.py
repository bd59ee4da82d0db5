"""Rows of the 512- and 1024-slot numeric kernels that a warp takes and rows of
many products that a block takes, in one bin, on both sides of the limits:
against the CPU oracle (integer values: bit for bit), in the plain, the
values-only and the learned path, and the times of rows that belong to a
block."""

import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2206_07244_gb300 as ops  # noqa: E402
from paper_2206_07244_gb300 import learned  # noqa: E402

ops.build()

K = 3000   # rows of B


def right(columns, length, apart, order, seed):
    """B: `length` of `columns` columns a row, `apart` from each other."""
    rng = np.random.default_rng(seed)
    col = np.sort(rng.random((K, columns)).argpartition(length - 1, axis=1)[:, :length], axis=1) * apart
    if order == "descending":
        col = col[:, ::-1]
    return W.Csr(K, columns * apart, np.arange(0, K * length + 1, length, dtype=np.int32),
                 col.astype(np.int32).ravel(), rng.integers(-3, 4, K * length).astype(np.float64))


def left(lengths, seed):
    """A: rows of the given lengths, random entries."""
    rng = np.random.default_rng(seed)
    rpt = np.zeros(len(lengths) + 1, dtype=np.int32)
    np.cumsum(lengths, out=rpt[1:])
    return W.Csr(len(lengths), K, rpt, rng.integers(0, K, rpt[-1]).astype(np.int32),
                 rng.integers(-3, 4, rpt[-1]).astype(np.float64))


def lengths_of(rows, short, long_rows, long):
    """Long rows in the middle and at both ends."""
    n = np.full(rows, short)
    n[np.linspace(0, rows - 1, long_rows).astype(int)] = long
    return n


def dev(m):
    return ops.CSR.from_arrays(m.rows, m.cols, m.rpt, m.col, m.val)


def same(C, want):
    for g, w in zip(C.numpy(), want):
        assert np.array_equal(g, w)


@pytest.mark.parametrize("rows, long_rows", [(40, 2), (300, 300), (2500, 41), (2500, 2500), (17000, 3)])
@pytest.mark.parametrize("length, order, apart", [(24, "ascending", 1), (10, "ascending", 1), (3, "ascending", 1),
                                                  (24, "descending", 1), (24, "ascending", 250), (7, "descending", 250)])
@pytest.mark.parametrize("columns, products", [(200, 520), (400, 800)])   # 512 and 1024 slots
def test_long_rows_in_a_bin(columns, products, length, order, apart, rows, long_rows):
    B = right(columns, length, apart, order, 1)
    short, long = products // length + 1, 9000 // length
    A = left(lengths_of(rows, short, long_rows, long), 2)
    dA, dB = dev(A), dev(B)
    want = oracle.spgemm(A, B)[:3]
    sizes = np.diff(want[0])
    assert columns // 2 < np.median(sizes) <= columns
    with ops.Handle() as h:
        C = h.multiply(dA, dB)
        h.status()
        same(C, want)
        C.col.fill_(-1)
        C.val.fill_(float("nan"))
        h.numeric_values(dA, dB, C)
        h.status()
        same(C, want)
        # every row predicted to have as many entries as the larger ones
        theta = np.zeros_like(np.load(learned.WEIGHTS))
        theta[-1] = np.log1p(sizes.max())
        h.set_predictor(theta, 0.0)
        h.set_mode("learned")
        C = h.multiply(dA, dB)
        h.status()
        same(C, want)


def numeric_ms(A, B):
    dA, dB = dev(A), dev(B)
    with ops.Handle() as h:
        C = h.multiply(dA, dB)
        best = np.inf
        for _ in range(9):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            h.numeric_values(dA, dB, C)
            e1.record()
            h.status()
            best = min(best, e0.elapsed_time(e1))
    return best


@pytest.mark.parametrize("rows, short, long_rows, long", [(3000, 4, 1, 30000),    # one hub among short rows
                                                          (400, 400, 400, 400)])  # few rows, all long
@pytest.mark.parametrize("columns, length, order", [(200, 24, "descending"), (400, 10, "ascending"), (400, 24, "descending"),
                                                    (400, 48, "ascending")])
def test_long_rows_are_not_left_to_one_warp(columns, length, order, rows, short, long_rows, long):
    # B declared wider than the warps' sort takes leaves every row to a block:
    # the time with its own width must not be above that by more than an eighth
    # and 10 us for the second launch
    A = left(lengths_of(rows, short, long_rows, long), 2)
    B = right(columns, length, 1, order, 1)
    wide = W.Csr(B.rows, (1 << 23) + 1, B.rpt, B.col, B.val)
    t, t_block = numeric_ms(A, B), numeric_ms(A, wide)
    assert t < 1.125 * t_block + 0.010, (t, t_block)
