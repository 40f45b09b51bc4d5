"""pdqp_kkt_noalloc at the edge between its one-cluster kernel (rows that fill at
most eight blocks of 512 threads) and the kernel with a block counter: 32 and 2
lanes per row, with and without rows of A."""
import pytest

import qpgen
from oracle import rapdhg as R
from tests import gpu_util as G
from tests.test_zz_no_alloc import KEYS, TOL, _noalloc, _point

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [
    (1, 0), (16, 1), (17, 16), (64, 64), (64, 65), (128, 0), (129, 0),    # dense rows: 16 rows a block
])
def test_dense_rows(n, m):
    inst = qpgen.tiny_qp(n + m, n=n, m=m, m_eq=m // 2, bounds="mixed")
    _check(inst, 7 * n + m)


@pytest.mark.parametrize("n", [255, 256, 2048, 2049])    # one nonzero per row: 256 rows a block
def test_diagonal(n):
    _check(qpgen.diagonal_box_qp(3, n), n)


def _check(inst, seed):
    x, y = _point(inst, seed)
    got = _noalloc(G.lib(), inst, x, y)
    ref = R.kkt_parts(R.problem_from_instance(inst), x, y)
    for k, key in enumerate(KEYS):
        assert got[k] == pytest.approx(ref[key], rel=TOL, abs=1e-13), (key, got[k], ref[key])
