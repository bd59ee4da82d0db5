"""Rows of at most 8 products, which the 8-lane row groups keep in registers:
against the CPU oracle (integer values, exact sums) next to rows just past
the limit, empty rows, empty B rows, repeated and unsorted columns."""

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


def csr(lists, cols, rng, i64):
    rpt = np.zeros(len(lists) + 1, dtype=np.int64 if i64 else np.int32)
    np.cumsum([len(x) for x in lists], out=rpt[1:])
    col = (np.concatenate(lists) if rpt[-1] else np.zeros(0)).astype(np.int32)
    return W.Csr(len(lists), cols, rpt, col, rng.integers(-3, 4, col.size).astype(np.float64))


@pytest.mark.parametrize("i64", [False, True])
@pytest.mark.parametrize("most", [1, 7, 8, 9])     # products per row; 9 needs the table
@pytest.mark.parametrize("cols", [3, 40, 1 << 30])
def test_rows_of_few_products(most, cols, i64):
    rng = np.random.default_rng(most)
    b = [rng.integers(0, cols, n) for n in rng.integers(0, 10, 300)]   # unsorted, repeated
    size = np.array([len(x) for x in b])
    a = []
    for i in range(1003):
        row, left = [], int(rng.integers(0, most + 1)) if i % 97 else most
        while len(row) < 8 and rng.random() < 0.9:
            k = int(rng.choice(np.nonzero(size <= left)[0]))
            row.append(k)
            left -= int(size[k])
        a.append(np.array(row, dtype=np.int64))
    a[500] = np.zeros(0, dtype=np.int64)
    A, B = csr(a, 300, rng, i64), csr(b, cols, rng, i64)
    dA, dB = (ops.CSR.from_arrays(m.rows, m.cols, m.rpt, m.col, m.val) for m in (A, B))
    for r0, r1 in ((0, A.rows), (5, 38)):
        with ops.Handle() as h:
            h.symbolic(dA, dB, r0, r1)
            C = h.numeric(dA, dB)
            h.status()
        for g, w in zip(C.numpy(), oracle.spgemm(A, B, r0, r1)[:3]):
            assert np.array_equal(g, w)
