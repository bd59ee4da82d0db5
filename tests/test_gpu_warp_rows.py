"""The 512- and 1024-slot numeric kernels in their warp-per-row form (B of up
to 2^23 columns) and their block-per-row form (wider B), at the edges of the
register sort, against the CPU oracle with integer values (exact sums)."""

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


def product(size, cols, spread, sort, seed):
    """40 rows of C with `size` distinct entries each: A's rows reference
    overlapping pieces of B's rows, whose columns reach cols - 1."""
    rng = np.random.default_rng(seed)
    a_lists, b_lists = [], []
    for i in range(40):
        pool = np.sort(rng.choice(np.arange(cols - spread, cols), size, replace=False))
        pool[-1] = cols - 1
        # short or long B rows that cover the pool, every piece overlapping the next
        step = 11 if i % 2 else 150
        pieces = [pool[k:k + step + 3] for k in range(0, size, step)]
        a_lists.append(np.arange(len(b_lists), len(b_lists) + len(pieces)))
        b_lists += [p if sort else rng.permutation(p) for p in pieces]

    def csr(lists, n, seed):
        rpt = np.zeros(len(lists) + 1, dtype=np.int32)
        np.cumsum([len(x) for x in lists], out=rpt[1:])
        col = np.concatenate(lists).astype(np.int32)
        return W.Csr(len(lists), n, rpt, col, np.random.default_rng(seed).integers(-3, 4, col.size).astype(np.float64))

    return csr(a_lists, len(b_lists), seed + 1), csr(b_lists, cols, seed + 2)


@pytest.mark.parametrize("sort", [True, False])
@pytest.mark.parametrize("cols", [1 << 23, (1 << 23) + 1])
@pytest.mark.parametrize("spread", [1100, 1 << 20])
@pytest.mark.parametrize("slots, size", [(512, 129), (512, 256), (512, 257), (512, 512), (1024, 257), (1024, 512),
                                         (1024, 513), (1024, 1024)])
def test_rows_at_the_edges_of_the_sort(slots, size, cols, spread, sort):
    A, B = product(size, cols, spread, sort, 7)
    table = ops.kernel_table(1)
    kernel = next(k for k, t in enumerate(table) if t[2] == slots)
    cfg = ops.default_config()
    cfg["num_kernel"], cfg["num_range"] = [kernel, len(table) - 1], [table[kernel][3], -1]
    dA, dB = (ops.CSR.from_arrays(m.rows, m.cols, m.rpt, m.col, m.val) for m in (A, B))
    with ops.Handle(cfg) as h:
        C = h.multiply(dA, dB)
        h.status()
    for g, w in zip(C.numpy(), oracle.spgemm(A, B)[:3]):
        assert np.array_equal(g, w)
