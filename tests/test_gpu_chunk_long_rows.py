"""The one-launch chunk is chosen only where the rows are even enough for its
slices (a slice is as wide as its longest row): one long row, alone and in every
member of a batch or a family, goes to the per-iteration kernels, a moderate one
and rows that are all long stay; what is chosen, and the chunk where it is asked
for, has the row-block kernels' iterates bit for bit."""
import numpy as np
import pytest
import scipy.sparse as sp

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _as32(S):
    S = sp.csr_matrix(S)
    S.sort_indices()
    return sp.csr_matrix((S.data, S.indices.astype(np.int32), S.indptr.astype(np.int32)), shape=S.shape)


def _qp(n, m, long, every=None, seed=1):
    """Diagonal Q, ten entries a row of A, `long` in row 5 (in every `every`-th from there)."""
    rng = np.random.default_rng(seed)
    cnt = np.full(m, 10)
    cnt[5 if every is None else slice(5, None, every)] = long
    rows = np.repeat(np.arange(m), cnt)
    cols = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in cnt])
    A = sp.csr_matrix((rng.standard_normal(rows.size), (rows, cols)), shape=(m, n))
    b = A @ rng.uniform(-0.5, 0.5, n) - np.where(np.arange(m) < m // 2, 0.0, 0.1)
    return qpgen.QPInstance("long_rows", n, m, m // 2, _as32(sp.diags(rng.uniform(1, 2, n))), _as32(A),
                            rng.standard_normal(n), b, np.full(n, -1.0), np.full(n, 1.0))


CASES = {
    "alone_1500": (1, lambda s: _qp(1500, 750, 1500), False),
    "alone_200": (1, lambda s: _qp(1500, 750, 200), True),
    "alone_all_300": (1, lambda s: _qp(600, 64, 300, every=1), True),
    "batch_1000": (160, lambda s: _qp(1000, 500, 1000, seed=s % 4), False),
    "batch_every_slice": (160, lambda s: _qp(2000, 1000, 256, every=32, seed=s % 4), False),
    "batch_64": (24, lambda s: _qp(300, 150, 64, seed=s), True),
}


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("case", sorted(CASES))
def test_choice_and_bits(case, precision):
    pd = G.lib()
    count, make, chunk = CASES[case]
    insts = [make(s) for s in range(count)]
    N, M = sum(i.n for i in insts), sum(i.m for i in insts)
    asked = (2,) if count == 1 else ()              # at most 64 row blocks
    out = {}
    for nt in (256, 0, *asked):
        h = pd.batch_from_instances(insts)
        try:
            x, y = np.zeros(N), np.zeros(M)
            st, info = pd.pdqp_solve(h, pd.pdqp_default_options(precision=precision, spmv_threads=nt, max_iter=130,
                                                                eps=0.0), x_out=x, y_out=y)
            out[nt] = (st, x, y, info.spmv_threads)
        finally:
            pd.pdqp_destroy(h)
    assert (out[0][3] == 2) == chunk
    for nt in (0, *asked):
        assert out[nt][0] == out[256][0]
        np.testing.assert_array_equal(out[nt][1], out[256][1])
        np.testing.assert_array_equal(out[nt][2], out[256][2])


def test_family_with_a_long_row_runs_interleaved():
    pd = G.lib()
    base, cnt = _qp(1000, 500, 1000), 20
    rng = np.random.default_rng(3)
    C, B = base.c + 0.1 * rng.standard_normal((cnt, base.n)), np.tile(base.b, (cnt, 1))
    out = {}
    for nt in (256, 0):
        h = pd.family_from_base(base, C, B)
        try:
            x = np.zeros(cnt * base.n)
            _, info = pd.pdqp_solve(h, pd.pdqp_default_options(precision=1, spmv_threads=nt, max_iter=130, eps=0.0),
                                    x_out=x)
            out[nt] = (x, info.spmv_threads)
        finally:
            pd.pdqp_destroy(h)
    assert out[0][1] == 3
    np.testing.assert_array_equal(out[0][0], out[256][0])


@pytest.mark.parametrize("precision,n,m", [(0, 100, 10000), (0, 40, 11500), (1, 40, 24000), (0, 7600, 0), (1, 15900, 0)])
def test_asked_for_within_its_limit(precision, n, m):
    """Up to 3n + 2m values in 200 KB the chunk runs where it is asked for, whatever the shape."""
    G.lib()
    inst = _qp(n, m, 4, seed=5) if n >= 100 and m else None
    if inst is None and m == 0:
        inst = qpgen.diagonal_box_qp(qpgen.SEED_BASE + 8100, n=n)
    if inst is None:
        rng = np.random.default_rng(6)
        cols = (rng.integers(0, n, (m, 1)) + np.arange(3)) % n
        A = sp.csr_matrix((rng.standard_normal(3 * m) / np.sqrt(m), (np.repeat(np.arange(m), 3), cols.ravel())), (m, n))
        inst = qpgen.QPInstance("tall", n, m, 0, _as32(sp.identity(n)), _as32(A), rng.standard_normal(n),
                                np.asarray(A @ np.full(n, 0.1)).ravel() - 0.1, np.full(n, -1.0), np.full(n, 1.0))
    a = G.solve(inst, precision=precision, spmv_threads=256, max_iter=70, eps=0.0)
    b = G.solve(inst, precision=precision, spmv_threads=2, max_iter=70, eps=0.0)
    assert b[1].spmv_threads == 2 and a[0] == b[0]
    np.testing.assert_array_equal(a[2], b[2])
    np.testing.assert_array_equal(a[3], b[3])
