"""The slice layout of large instances (reported as variant 5): sizes around a
slice (32 rows), rows of no, one and odd numbers of entries and of a whole row
block, bit for bit against the row-block kernels; rows too uneven keep these."""
import numpy as np
import pytest
import scipy.sparse as sp

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _qp(n, m, a_row, long_rows, stride, seed):
    """Diagonal Q, a_row entries in every row of A (none in every seventh) and
    `long_rows` rows of 2000, one every `stride` rows."""
    rng = np.random.default_rng(seed)
    cnt = np.full(m, a_row)
    cnt[6::7] = 0
    cnt[:long_rows * stride:stride] = 2000
    rows = np.repeat(np.arange(m), cnt)
    cols = np.concatenate([np.sort(rng.choice(n, k, replace=False)) if k > 50 else
                           (rng.integers(0, n) + np.arange(k) * 977) % n for k in cnt])
    A = sp.csr_matrix((rng.standard_normal(rows.size), (rows, cols)), shape=(m, n))
    A.sort_indices()
    Q = sp.diags(rng.uniform(0.5, 2.0, n)).tocsr()
    x0 = rng.uniform(-0.5, 0.5, n)
    as32 = lambda S: sp.csr_matrix((S.data, S.indices.astype(np.int32), S.indptr.astype(np.int32)), shape=S.shape)
    return qpgen.QPInstance("slices", n, m, m // 2, as32(Q), as32(A), rng.standard_normal(n),
                            A @ x0 - np.where(np.arange(m) < m // 2, 0.0, 0.1), np.full(n, -1.0), np.full(n, 1.0))


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n,m,a_row,long_rows,stride,taken", [
    (140_001, 220_031, 9, 0, 1, True),       # one row in the last slice of P
    (160_000, 130_000, 16, 40, 1, True),     # 40 rows of 2000 side by side
    (60_000, 60_000, 33, 1500, 40, False),   # one in most slices: nearly all pads
])
def test_slices_match_row_blocks(n, m, a_row, long_rows, stride, taken, precision):
    """Every candidate, the slices among them, runs eight iterations of a handle's
    first solve while it is timed."""
    pd = G.lib()
    inst = _qp(n, m, a_row, long_rows, stride, n)
    out, variants = [], set()
    for nt in (256, 0, 0):
        h = G.handle(inst)
        try:
            x, y = np.zeros(n), np.zeros(m)
            st, info = pd.pdqp_solve(h, pd.pdqp_default_options(precision=precision, spmv_threads=nt, max_iter=192,
                                                                eps=0.0), x_out=x, y_out=y)
            out.append((st, x, y))
            variants.add(info.spmv_threads)
        finally:
            pd.pdqp_destroy(h)
    assert taken or 5 not in variants
    for o in out[1:]:
        assert o[0] == out[0][0]
        np.testing.assert_array_equal(o[1], out[0][1])
        np.testing.assert_array_equal(o[2], out[0][2])
