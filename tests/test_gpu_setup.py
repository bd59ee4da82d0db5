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
