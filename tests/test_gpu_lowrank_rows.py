"""The low-rank kernels that read the factor once are taken where every row of P
is short: a variable in few enough rows of A keeps them, one in hundreds goes to
the general kernels; the iterates are bit for bit the same."""
import numpy as np
import pytest
import scipy.sparse as sp

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("rows,fused", [(189, True), (190, False), (1500, False)])   # P's row: Q, two dense rows, these
def test_a_long_row_of_P_takes_the_general_kernels(rows, fused, precision):
    G.lib()
    base = qpgen.portfolio_qp(qpgen.SEED_BASE + 8300, n=2000, r=16)
    rng = np.random.default_rng(rows)
    k = np.arange(rows)
    extra = sp.csr_matrix((np.concatenate([np.full(rows, 0.5), 0.1 * rng.random(rows)]),
                           (np.concatenate([k, k]), np.concatenate([np.full(rows, 7), 8 + k]))), shape=(rows, base.n))
    A = sp.vstack([base.A, extra]).tocsr()
    A.sort_indices()
    A = sp.csr_matrix((A.data, A.indices.astype(np.int32), A.indptr.astype(np.int32)), shape=A.shape)
    inst = qpgen.QPInstance("portfolio_long_row", base.n, base.m + rows, base.m_eq, base.Q, A, base.c,
                            np.concatenate([base.b, np.full(rows, -0.01)]), base.l, base.u, F=base.F)
    a, b = (G.solve(inst, precision=precision, spmv_threads=nt, max_iter=130, eps=0.0) for nt in (256, 0))
    assert (b[1].spmv_threads == 4) == fused
    np.testing.assert_array_equal(a[2], b[2])
    np.testing.assert_array_equal(a[3], b[3])
