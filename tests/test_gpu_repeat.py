"""Rows of C that repeat the column pattern of the row before (structured
grids, bands, several unknowns per point), which skip the symbolic phase and
are multiplied by a shared map: against the CPU oracle, at the limits of the
path (products and entries per row, run lengths, words of 32 rows) and where
the pattern breaks. Integer values: every partial sum is exact, so results
must match bit for bit."""

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

MIN_ROWS = 32768   # products of fewer and short rows do not look for repeating rows


def csr(rows, cols, lists, seed):
    """Rows from ascending column lists, small integer values."""
    lens = np.array([len(x) for x in lists])
    rpt = np.zeros(rows + 1, dtype=np.int32)
    np.cumsum(lens, out=rpt[1:])
    col = np.concatenate(lists).astype(np.int32)
    return W.Csr(rows, cols, rpt, col, np.random.default_rng(seed).integers(-3, 4, col.size).astype(np.float64))


def offsets(n, offs, seed, cols=None):
    """Row i holds the columns i + offs inside [0, cols)."""
    cols = cols or n
    offs = np.array(sorted(offs))
    return csr(n, cols, [(i + offs)[(i + offs >= 0) & (i + offs < cols)] for i in range(n)], seed)


def expand(m, dofs, seed):
    """Every point becomes `dofs` unknowns, all coupled."""
    lists = []
    for i in range(m.rows):
        c = (m.col[m.rpt[i]:m.rpt[i + 1], None] * dofs + np.arange(dofs)).ravel()
        lists += [c] * dofs
    return csr(m.rows * dofs, m.cols * dofs, lists, seed)


def box27(side):
    m = W.stencil27(side)
    return W.Csr(m.rows, m.cols, m.rpt, m.col, np.random.default_rng(1).integers(-3, 4, m.nnz).astype(np.float64))


def break_rows(m, every, seed):
    """Moves the last column of every `every`-th row."""
    lists = [m.col[m.rpt[i]:m.rpt[i + 1]].copy() for i in range(m.rows)]
    for i in range(3, m.rows, every):
        if lists[i].size > 1 and lists[i][-1] < m.cols - 1:
            lists[i][-1] += 1
    return csr(m.rows, m.cols, lists, seed)


N = MIN_ROWS + 77


def one_point(n=N):
    return offsets(n, [0], 5)


CASES = {
    "tridiagonal": lambda: (offsets(N, [-1, 0, 1], 1),) * 2,
    "one entry a row": lambda: (one_point(),) * 2,
    "grid 5": lambda: (offsets(N, [-128, -1, 0, 1, 128], 1),) * 2,
    "27 points": lambda: (box27(33),) * 2,
    "two unknowns a point": lambda: (expand(offsets(N // 2 + 1, [-90, -1, 0, 1, 90], 1), 2, 2),) * 2,
    "five unknowns a point": lambda: (expand(offsets(N // 5 + 1, [-60, -1, 0, 1, 60], 1), 5, 2),) * 2,
    "band 33 (products of the second class)": lambda: (offsets(N, range(-16, 16), 1),) * 2,
    "band 67 (third class)": lambda: (offsets(N, range(-33, 34), 1),) * 2,
    "band 135 (fourth class)": lambda: (offsets(N, range(-67, 68), 1),) * 2,
    "band 137 (past the last class)": lambda: (offsets(N, range(-68, 69), 1),) * 2,
    "apart: more entries than an accumulator": lambda: (
        offsets(N, [0, 3], 1, cols=N + 3),
        offsets(N + 3, [40 * j for j in range(513)], 2, cols=N + 40 * 513)),
    "A of 256 entries": lambda: (offsets(N, range(256), 1, cols=N + 256), one_point(N + 256)),
    "A of 257 entries": lambda: (offsets(N, range(257), 1, cols=N + 257), one_point(N + 257)),
    "other B": lambda: (offsets(N, [0, 2, 5, 64], 1, cols=N + 70), offsets(N + 70, [0, 1, 7, 30], 2, cols=N + 110)),
    "empty rows in B": lambda: (offsets(N, [0, 1], 1, cols=N + 1), csr(
        N + 1, N + 9, [np.zeros(0, dtype=int) if i % 50 == 7 else i + np.arange(4) for i in range(N + 1)], 3)),
    "B broken every 11 rows": lambda: (offsets(N, [-1, 0, 1], 1), break_rows(offsets(N, range(-4, 5), 1), 11, 2)),
    "A broken every 5 rows": lambda: (break_rows(offsets(N, [-2, 0, 2], 1), 5, 2), offsets(N, range(-4, 5), 1)),
    "A broken every 33 rows": lambda: (break_rows(offsets(N, [-2, 0, 2], 1), 33, 2), offsets(N, range(-4, 5), 1)),
}


def dev(m, i64=False):
    return ops.CSR.from_arrays(m.rows, m.cols, m.rpt.astype(np.int64 if i64 else np.int32), m.col, m.val)


def same(C, want):
    for g, w in zip(C.numpy(), want):
        assert np.array_equal(g, w)


@pytest.mark.parametrize("i64", [False, True])
@pytest.mark.parametrize("name", CASES)
def test_repeating_rows(name, i64):
    A, B = CASES[name]()
    dA = dev(A, i64)
    dB = dA if B is A else dev(B, i64)
    rpt, col, val, _ = oracle.spgemm(A, B)
    with ops.Handle() as h:
        C = h.multiply(dA, dB)
        st = h.stats()
        h.status()
        same(C, (rpt, col, val))
        assert st["total_nprod"] == oracle.nprod(A, B).sum()
        assert sum(st["sym_bins"]) == sum(st["num_bins"]) == A.rows
        # new values on the same structure
        A2 = W.Csr(A.rows, A.cols, A.rpt, A.col, np.random.default_rng(9).integers(-3, 4, A.nnz).astype(np.float64))
        C.val.fill_(float("nan"))
        h.numeric_values(dev(A2, i64), dB, C)
        h.status()
        same(C, oracle.spgemm(A2, B)[:3])


@pytest.mark.parametrize("r0, rows", [(0, MIN_ROWS), (1, MIN_ROWS), (37, MIN_ROWS + 1), (64, MIN_ROWS - 1)])
def test_row_window(r0, rows):
    A = offsets(N + 100, [-100, -1, 0, 1, 100], 1)
    with ops.Handle() as h:
        h.symbolic(dev(A), dev(A), r0, r0 + rows)
        C = h.numeric(dev(A), dev(A))
        h.status()
    same(C, oracle.spgemm(A, A, r0, r0 + rows)[:3])


@pytest.mark.parametrize("kind", ["repeated column", "unsorted"])
def test_columns_of_B_in_another_order(kind):
    # rows of A repeat, but B has a row whose columns are not ascending: no
    # row may be added without atomics
    A = offsets(N, [-1, 0, 1], 1)
    B = offsets(N, range(-4, 5), 2)
    q = B.rpt[N // 2]
    if kind == "unsorted":
        B.col[q:q + 2] = B.col[q:q + 2][::-1].copy()
    else:
        B.col[q + 1] = B.col[q]
    with ops.Handle() as h:
        C = h.multiply(dev(A), dev(B))
        h.status()
    same(C, oracle.spgemm(A, B)[:3])


def test_another_structure_is_reported():
    # the same sizes, but rows of B longer and shorter than the symbolic phase saw
    A = offsets(N, [-1, 0, 1], 1)
    lists = [A.col[A.rpt[i]:A.rpt[i + 1]] for i in range(N)]
    lists[5000], lists[5001] = np.array([4999, 5000]), np.array([5000, 5001, 5002, 5003])
    B = csr(N, N, lists, 2)
    assert B.nnz == A.nnz
    with ops.Handle() as h:
        C = h.multiply(dev(A), dev(A))
        h.status()
        h.numeric_values(dev(A), dev(B), C)
        with pytest.raises(ops.SpgemmError):
            h.status()
        same(h.multiply(dev(A), dev(B)), oracle.spgemm(A, B)[:3])
        h.status()


@pytest.mark.parametrize("trained", [True, False])   # False: every size predicted 1, rows overflow
@pytest.mark.parametrize("name", ["grid 5", "27 points", "band 33 (products of the second class)", "other B",
                                  "B broken every 11 rows", "empty rows in B"])
def test_learned_sizing(name, trained):
    from paper_2206_07244_gb300 import learned
    A, B = CASES[name]()
    dA = dev(A)
    dB = dA if B is A else dev(B)
    with ops.Handle() as h:
        theta = np.load(learned.WEIGHTS)
        h.set_predictor(theta if trained else np.zeros_like(theta), 0.25 if trained else 0.0)
        h.set_mode("learned")
        want = oracle.spgemm(A, B)[:3]
        for _ in range(2):
            C = h.multiply(dA, dB)
            h.status()
            same(C, want)
        st = h.learned_stats()
        assert st["one_phase_rows"] + st["mispredicted_rows"] + st["exact_rows"] == A.rows


def scatter(m, every, seed):
    """Every `every`-th row references columns far apart, as many as before."""
    rng = np.random.default_rng(seed)
    lists = [m.col[m.rpt[i]:m.rpt[i + 1]] for i in range(m.rows)]
    for i in range(every // 2, m.rows, every):
        lists[i] = np.sort(rng.choice(m.cols, lists[i].size, replace=False))
    return csr(m.rows, m.cols, lists, seed)


# Rows of 257 to 1024 products and at most 64 entries, the second class by
# their products and the first by their entries; a scattered row has as many
# products as its neighbours and several times their entries.
MIXED = {
    "band 17": lambda: offsets(40000, range(-8, 9), 1),
    "band 21": lambda: offsets(40000, range(-10, 11), 1),
    "band 31": lambda: offsets(40000, range(-15, 16), 1),
    "six unknowns a point": lambda: expand(offsets(40000 // 6, [-1, 0, 1], 1), 6, 2),
    "ten unknowns a point": lambda: expand(offsets(4000, [-1, 0, 1], 1), 10, 2),
    "blocks of 24": lambda: expand(offsets(40000 // 24, [0], 1), 24, 2),
}


@pytest.mark.parametrize("every", [10001, 39999])   # a handful of scattered rows, and one
@pytest.mark.parametrize("name", MIXED)
def test_learned_sizing_with_some_rows_mispredicted(name, every):
    from paper_2206_07244_gb300 import learned
    B = MIXED[name]()
    A = scatter(B, every, 4)
    dA, dB = dev(A), dev(B)
    want = oracle.spgemm(A, B)[:3]
    # predictions of the rows' own size, whatever the network says of them:
    # the output bias alone, log1p of the entries of an unscattered row
    theta = np.zeros_like(np.load(learned.WEIGHTS))
    theta[-1] = np.log1p(np.median(np.diff(want[0])))
    for weights in (np.load(learned.WEIGHTS), theta):
        with ops.Handle() as h:
            h.set_predictor(weights, 0.0)
            h.set_mode("learned")
            C = h.multiply(dA, dB)
            st = h.learned_stats()
            h.status()
            same(C, want)
            if weights is theta:
                assert 0 < st["mispredicted_rows"] < A.rows // 2


@pytest.mark.parametrize("kind", ["band", "unsorted rows of B", "window below the rule"])
def test_bin_statistics_tell_the_rows_that_the_kernels_take(kind):
    import ctypes
    from paper_2206_07244_gb300 import _abi
    A = offsets(N, range(-8, 9), 1)
    B = A
    rows = N
    if kind == "unsorted rows of B":
        B = W.Csr(A.rows, A.cols, A.rpt, A.col.copy(), A.val)
        B.col[5:7] = B.col[5:7][::-1].copy()
    elif kind == "window below the rule":
        rows = 4000
    with ops.Handle() as h:
        nnz = h.symbolic(dev(A), dev(B), 0, rows)
        st = []
        for phase in (0, 1):
            a = (ctypes.c_int64 * 64)()
            _abi.check(_abi.lib().spgemm_bin_stats(h._h, phase, a, 64), "spgemm_bin_stats")
            st.append(np.array(a).reshape(4, 16))
    for phase in (0, 1):
        assert st[phase][0].sum() == rows and st[phase][2].sum() == A.rpt[rows]
        taken = st[phase][3]
        if kind == "band":
            assert 0 < taken.sum() < rows // 8
        elif kind == "window below the rule" or phase == 1:   # numeric kernels need ascending rows of B
            assert np.array_equal(taken, st[phase][0])
        else:
            assert taken.sum() < rows // 8
    assert st[1][1].sum() == nnz
