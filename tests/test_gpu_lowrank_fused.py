"""The low-rank half-step that reads F once (variant 4, chosen for a low-rank
term over short rows of P) against the general kernels, bit for bit: ranks with
and without 16-byte rows, the smallest and largest, tiles with a remainder."""
import numpy as np
import pytest

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n,r", [(40, 1), (257, 3), (1000, 8), (1000, 33), (3001, 64), (600, 255)])
def test_fused_lowrank_is_bitwise_the_general_kernels(n, r, precision):
    pd = G.lib()
    inst = qpgen.portfolio_qp(seed=qpgen.SEED_BASE + 7400 + n + r, n=n, r=r)
    runs = {nt: G.solve(inst, precision=precision, spmv_threads=nt, max_iter=330) for nt in (256, 0)}
    fits = not (precision == 0 and r == 255)      # 200 rows of 255 float64 values exceed a CTA's shared memory
    assert (runs[0][1].spmv_threads == 4) == fits and runs[256][1].spmv_threads == 256
    assert runs[0][1].iterations == runs[256][1].iterations
    np.testing.assert_array_equal(runs[0][2], runs[256][2])
    np.testing.assert_array_equal(runs[0][3], runs[256][3])


def test_fused_lowrank_partial_chunks():
    G.lib()
    inst = qpgen.portfolio_qp(seed=qpgen.SEED_BASE + 7500, n=700, r=16)
    for iters in (1, 64, 97):
        a = G.state_after(inst, iters, precision=0, spmv_threads=256)
        b = G.state_after(inst, iters, precision=0, spmv_threads=0)
        for k in a:
            np.testing.assert_array_equal(b[k], a[k])


def test_relkkt_of_rows_longer_than_a_row_block():
    """The check's segment sums of dense rows (of A, and of P through a dense
    column) against float64 products on the host; each sum has at most 3e4
    terms, so 1e-11 relative covers any order."""
    import scipy.sparse as sp
    pd = G.lib()
    rng = np.random.default_rng(7600)
    n, m = 6000, 5000
    A = sp.random(m, n, 2e-4, random_state=1, format="lil")
    A[0, :] = rng.standard_normal(n)
    A[4, :2049] = rng.standard_normal(2049)
    A[:, 7] = rng.standard_normal((m, 1))
    A = sp.csr_matrix(A)
    A.sort_indices()
    Q = sp.diags(rng.uniform(1, 2, n)).tolil()
    v = rng.standard_normal(3000) * 1e-3
    Q[11, 100:3100] = v
    Q[100:3100, 11] = v.reshape(-1, 1)
    Q = sp.csr_matrix(Q)
    Q.sort_indices()
    inst = qpgen.QPInstance("long", n, m, m // 2, sp.csr_matrix((Q.data, Q.indices.astype(np.int32), Q.indptr.astype(np.int32)), Q.shape),
                            sp.csr_matrix((A.data, A.indices.astype(np.int32), A.indptr.astype(np.int32)), A.shape),
                            rng.standard_normal(n), rng.standard_normal(m), np.full(n, -3.0), np.full(n, 3.0))
    x, y = np.clip(rng.standard_normal(n), -3, 3), rng.standard_normal(m)
    h = G.handle(inst)
    try:
        got = pd.pdqp_kkt(h, x, y)
    finally:
        pd.pdqp_destroy(h)
    from oracle import rapdhg as R
    want = R.kkt_parts(R.problem_from_instance(inst), x, y)
    for k, key in enumerate(("r_primal", "r_dual", "r_gap", "rel_kkt", "primal_obj", "dual_obj")):
        assert got[k] == pytest.approx(want[key], rel=1e-11, abs=1e-13), key
