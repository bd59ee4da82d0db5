"""The setup scans at the edges of their tiles: row products, bin statistics
and the check of B's column order, against the oracle."""

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

TILE = 2048   # entries per tile of the scans


def rows_of(lengths, cols, seed):
    """CSR with the given row lengths, distinct ascending columns and small
    integer values."""
    rng = np.random.default_rng(seed)
    rpt = np.zeros(len(lengths) + 1, dtype=np.int64)
    np.cumsum(lengths, out=rpt[1:])
    col = np.concatenate([np.sort(rng.choice(cols, k, replace=False)) for k in lengths] or [np.zeros(0)])
    return W.Csr(len(lengths), cols, rpt.astype(np.int32), col.astype(np.int32),
                 rng.integers(-3, 4, col.size).astype(np.float64))


LENGTHS = {
    "one tile": [TILE],
    "one past": [TILE, 1],
    "edge inside a row": [TILE - 1, 3, 0, 5],
    "empty rows at the edge": [TILE] + [0] * 700 + [2] + [0] * 300,
    "long row over tiles": [1, 3 * TILE + 5, 2],
    "single entries": [1] * (TILE + 300),
    "empty ends": [0] * 400 + [7, 0, 9] + [0] * 400,
    "nothing": [0] * 5,
}


@pytest.mark.parametrize("i64", [False, True])
@pytest.mark.parametrize("name", LENGTHS)
def test_row_products_and_bin_statistics(name, i64):
    K = 7000
    A = rows_of(LENGTHS[name], K, 1)
    B = rows_of(np.random.default_rng(2).integers(0, 4, K), 900, 3)
    want = oracle.nprod(A, B)
    t = np.int64 if i64 else np.int32
    dA, dB = (ops.CSR.from_arrays(m.rows, m.cols, m.rpt.astype(t), m.col, m.val) for m in (A, B))
    with ops.Handle() as h:
        got = h.multiply(dA, dB)
        st = h.stats()
        h.status()
    rpt, col, val, _ = oracle.spgemm(A, B)
    assert st["total_nprod"] == want.sum() and st["max_nprod"] == want.max(initial=0)
    assert sum(st["sym_bins"]) == A.rows
    for g, w in zip(got.numpy(), (rpt, col, val)):
        assert np.array_equal(g, w)
    X = learned.features(dA, dB).cpu().numpy()
    length = np.diff(B.rpt)
    big = np.array([length[A.col[a:b]].max(initial=0) for a, b in zip(A.rpt[:-1], A.rpt[1:])])
    low = np.array([length[A.col[a:b]].min() if b > a else 0 for a, b in zip(A.rpt[:-1], A.rpt[1:])])
    # float32 log1p of whole numbers: half an ulp of the result and of the argument, and CUDA's 1 ulp
    for k, w in ((1, want), (2, big), (4, low)):
        np.testing.assert_allclose(X[:, k], np.log1p(w.astype(np.float64)), rtol=4e-7, atol=0)


@pytest.mark.parametrize("at", [0, TILE - 2, TILE - 1, TILE, 2 * TILE - 1, 2 * TILE + 3])
@pytest.mark.parametrize("kind", ["repeat", "decrease"])
def test_order_check_at_tile_edges(at, kind):
    # one row of B breaks the order between its entries `at` and `at` + 1:
    # kernels that rely on distinct columns must not be taken
    n = 2 * TILE + 10
    B = rows_of([0, n, 0], n + 50, 5)
    if kind == "repeat":
        B.col[at + 1] = B.col[at]
    else:
        B.col[[at, at + 1]] = B.col[[at + 1, at]]
    A = W.from_dense(np.array([[0.0, 2.0, 0.0], [1.0, 3.0, 1.0]]))
    with ops.Handle() as h:
        got = h.multiply(ops.CSR.from_workload(A), ops.CSR.from_workload(B))
        h.status()
    for g, w in zip(got.numpy(), oracle.spgemm(A, B)[:3]):
        assert np.array_equal(g, w)


# Entries in more rows than the scans walk (32 steps of at most 256 rows):
# their tiles search the rows instead.
SPARSE = {
    **{f"{k} empty rows": [5, 3] + [0] * k + [4, 2] for k in (8189, 8190, 8191, 8192, 8193)},
    "several gaps": [3] * 10 + [0] * 200000 + [2] * 3000 + [0] * 50000 + [1] + [0] * 30000,
    "a row in 37": [1 + i % 3 if i % 37 == 5 else 0 for i in range(150000)],
    "long rows apart": [1500] + [0] * 9000 + [1500] + [0] * 9000 + [2 * TILE + 700] + [0] * 9000 + [3],
    "gap at a tile's edge": [TILE - 1] + [0] * 20000 + [1] + [0] * 20000 + [1, 2],
}


@pytest.mark.parametrize("i64", [False, True])
@pytest.mark.parametrize("name", SPARSE)
def test_entries_in_far_apart_rows_of_A(name, i64):
    K = 7000
    A = rows_of(SPARSE[name], K, 1)
    B = rows_of(np.random.default_rng(2).integers(0, 4, K), 900, 3)
    want = oracle.nprod(A, B)
    t = np.int64 if i64 else np.int32
    dA, dB = (ops.CSR.from_arrays(m.rows, m.cols, m.rpt.astype(t), m.col, m.val) for m in (A, B))
    with ops.Handle() as h:
        got = h.multiply(dA, dB)
        st = h.stats()
        h.status()
        r0 = A.rows // 3
        h.symbolic(dA, dB, r0, A.rows)
        part = h.numeric(dA, dB)
        h.status()
    assert st["total_nprod"] == want.sum() and st["max_nprod"] == want.max(initial=0)
    for r, C in ((0, got), (r0, part)):
        for g, w in zip(C.numpy(), oracle.spgemm(A, B, r, A.rows)[:3]):
            assert np.array_equal(g, w)
    X = learned.features(dA, dB).cpu().numpy()
    length = np.diff(B.rpt)
    full = np.flatnonzero(np.diff(A.rpt))
    for k, f in ((2, np.maximum), (4, np.minimum)):
        w = f.reduceat(length[A.col], A.rpt[full])
        np.testing.assert_allclose(X[full, k], np.log1p(w.astype(np.float64)), rtol=4e-7, atol=0)


@pytest.mark.parametrize("fault", ["none", "repeat", "decrease"])
@pytest.mark.parametrize("name", SPARSE)
def test_order_check_with_far_apart_rows_of_B(name, fault):
    # one entry in B's last long row breaks the order; entries that only
    # follow the end of another row do not
    B = rows_of(SPARSE[name], 9000, 5)
    lens = np.diff(B.rpt)
    q = B.rpt[np.flatnonzero(lens >= 2)[-1]]
    if fault == "repeat":
        B.col[q + 1] = B.col[q]
    elif fault == "decrease":
        B.col[[q, q + 1]] = B.col[[q + 1, q]]
    full = np.flatnonzero(lens)[-40:]
    A = W.Csr(3, B.rows, np.array([0, full.size, full.size, 2 * full.size], dtype=np.int32),
              np.concatenate([full, full]).astype(np.int32), np.arange(2.0 * full.size) - 30)
    with ops.Handle() as h:
        got = h.multiply(ops.CSR.from_workload(A), ops.CSR.from_workload(B))
        h.status()
    for g, w in zip(got.numpy(), oracle.spgemm(A, B)[:3]):
        assert np.array_equal(g, w)


def test_repeating_rows_around_a_gap():
    # a band of 33 columns with 40,000 empty rows inside: repeating rows are
    # left out of the scan of a tile whose entries search their rows, too
    n, offs = 45000, np.arange(-16, 17)
    lists = [np.zeros(0, int) if 20000 <= i < 60000 else (j := i if i < 20000 else i - 40000) + offs[(j + offs >= 0) & (j + offs < n)]
             for i in range(n + 40000)]
    rpt = np.zeros(len(lists) + 1, dtype=np.int32)
    np.cumsum([x.size for x in lists], out=rpt[1:])
    col = np.concatenate(lists).astype(np.int32)
    rng = np.random.default_rng(4)
    A = W.Csr(len(lists), n, rpt, col, rng.integers(-3, 4, col.size).astype(np.float64))
    B = rows_of([9] * n, 300, 3)
    for k in range(n):   # rows that repeat the row before, moved by one
        B.col[9 * k:9 * k + 9] = k + np.arange(9)
    B.cols = n + 9
    with ops.Handle() as h:
        got = h.multiply(ops.CSR.from_workload(A), ops.CSR.from_workload(B))
        st = h.stats()
        h.status()
    assert st["total_nprod"] == oracle.nprod(A, B).sum()
    for g, w in zip(got.numpy(), oracle.spgemm(A, B)[:3]):
        assert np.array_equal(g, w)


@pytest.mark.parametrize("side", ["A", "B"])
def test_empty_rows_are_not_walked_by_one_block(side):
    # 8M empty rows between two ends of 20,000 rows: what a row costs with all
    # blocks at work (rows of A: row pointers, counters, bins and offsets,
    # about 100 bytes; rows of B: nothing) is below 3 ms at a fifth of the
    # memory rate; one block alone waits about 1.2 us for every 256 rows
    gap = 1 << 23
    lens = np.concatenate([np.full(20000, 4), np.zeros(gap, int), np.full(20000, 4)])
    rpt = np.zeros(lens.size + 1, dtype=np.int32)
    np.cumsum(lens, out=rpt[1:])
    other = rows_of([4] * 20000, 20000, 2)
    rng = np.random.default_rng(6)
    if side == "A":
        A = W.Csr(lens.size, 20000, rpt, rng.integers(0, 20000, rpt[-1]).astype(np.int32), np.ones(rpt[-1]))
        B = other
    else:
        A = W.Csr(20000, lens.size, other.rpt, (other.col % 20000 + (gap + 20000) * (other.col % 2)).astype(np.int32), other.val)
        B = W.Csr(lens.size, 20000, rpt, np.tile(np.arange(0, 20000, 5000, dtype=np.int32), 40000), np.ones(rpt[-1]))
    dA, dB = ops.CSR.from_workload(A), ops.CSR.from_workload(B)
    with ops.Handle() as h:
        best = np.inf
        for _ in range(6):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            C = h.multiply(dA, dB)
            e1.record()
            h.status()
            best = min(best, e0.elapsed_time(e1))
        for g, w in zip(C.numpy(), oracle.spgemm(A, B)[:3]):
            assert np.allclose(g, w, rtol=1e-12, atol=1e-12)
    assert best < (6.0 if side == "A" else 3.0), best


# Rows whose part of a tile is more than 32 steps of their threads (one thread
# a row up to 4 entries on average, then as many as a quarter of the average):
# at that limit, over tiles, in one warp and in rows next to each other.
HUBS = {
    "one thread a row": [1, 2, 32, 33, 34, 0, 31, 65] + [1] * 3000 + [900, 33, 1],
    "hub over tiles": [2] * 700 + [5 * TILE + 77] + [2] * 3000,
    "hubs side by side": [1] * 4000 + [TILE, TILE + 1, 40, 2 * TILE, 3] + [1] * 4000,
    "two threads a row": [7] * 400 + [64, 65, 66, 400] + [5] * 300 + [130, 63],
    "eight threads a row": [25] * 200 + [256, 257, 300, 1] + [30] * 100 + [2000],
    "sixteen threads a row": [60] * 100 + [512, 513, 1800] + [62] * 50,
    "a warp a row": [130] * 60 + [1024, 1025, 1500] + [140] * 30,
}


@pytest.mark.parametrize("i64", [False, True])
@pytest.mark.parametrize("name", HUBS)
def test_long_rows_among_short_ones(name, i64):
    K = 15000
    A = rows_of(HUBS[name], K, 1)
    B = rows_of(np.random.default_rng(2).integers(0, 4, K), 900, 3)
    want = oracle.nprod(A, B)
    t = np.int64 if i64 else np.int32
    dA, dB = (ops.CSR.from_arrays(m.rows, m.cols, m.rpt.astype(t), m.col, m.val) for m in (A, B))
    with ops.Handle() as h:
        got = h.multiply(dA, dB)
        st = h.stats()
        h.status()
    assert st["total_nprod"] == want.sum() and st["max_nprod"] == want.max()
    for g, w in zip(got.numpy(), oracle.spgemm(A, B)[:3]):
        assert np.array_equal(g, w)
    X = learned.features(dA, dB).cpu().numpy()
    length = np.diff(B.rpt)
    full = np.flatnonzero(np.diff(A.rpt))
    np.testing.assert_allclose(X[:, 1], np.log1p(want.astype(np.float64)), rtol=4e-7, atol=0)
    for k, f in ((2, np.maximum), (4, np.minimum)):
        w = f.reduceat(length[A.col], A.rpt[full])
        np.testing.assert_allclose(X[full, k], np.log1p(w.astype(np.float64)), rtol=4e-7, atol=0)


def test_full_last_row_of_a_tridiagonal_matrix():
    # the row repeats no other and is counted where most rows are left out;
    # 64 tiles are in flight at once, and the 64 loads that a lane takes there
    # wait for memory about 1 us each at most
    import ctypes
    from paper_2206_07244_gb300 import _abi
    n = 1 << 17
    lists = [np.arange(max(i - 1, 0), min(i + 2, n)) for i in range(n - 1)] + [np.arange(n)]
    rpt = np.zeros(n + 1, dtype=np.int32)
    np.cumsum([x.size for x in lists], out=rpt[1:])
    rng = np.random.default_rng(4)
    A = W.Csr(n, n, rpt, np.concatenate(lists).astype(np.int32), rng.integers(-3, 4, rpt[-1]).astype(np.float64))
    B = W.Csr(n, n, A.rpt.copy(), A.col, A.val)
    B.rpt[-1] = B.rpt[-2] + 2   # tridiagonal
    last = B.rpt[-2]
    B.col, B.val = np.concatenate([A.col[:last], [n - 2, n - 1]]).astype(np.int32), A.val[:last + 2].copy()
    dA, dB = ops.CSR.from_workload(A), ops.CSR.from_workload(B)
    ms, ln = (ctypes.c_double * 43)(), (ctypes.c_int64 * 43)()
    best = np.inf
    with ops.Handle() as h:
        _abi.check(_abi.lib().spgemm_set_timing(h._h, 1), "spgemm_set_timing")
        for _ in range(6):
            C = h.multiply(dA, dB)
            h.status()
            st = h.stats()
            _abi.check(_abi.lib().spgemm_kernel_times(h._h, ms, ln, 43, 1), "spgemm_kernel_times")
            best = min(best, 1e3 * ms[32])
        for g, w in zip(C.numpy(), oracle.spgemm(A, B)[:3]):
            assert np.array_equal(g, w)
    assert st["total_nprod"] == oracle.nprod(A, B).sum()
    assert best < 100.0, best
