"""Small families take the one-launch chunk, large ones the interleaved kernels:
on both sides of the line the chosen variant's iterates are bit for bit the
row-block kernels'."""
import numpy as np
import pytest

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("count,variant", [(2, 2), (200, 2), (1000, 2), (1001, 3)])   # 300 rows a member
def test_family_choice(count, variant, precision):
    pd = G.lib()
    fam = qpgen.family_qp(n=200, m=100)
    C, B = fam.params(11, count)
    out = []
    for nt in (256, 0):
        h = pd.family_from_base(fam.base, C, B)
        try:
            x, y = np.zeros(count * 200), np.zeros(count * 100)
            st, info = pd.pdqp_solve(h, pd.pdqp_default_options(precision=precision, spmv_threads=nt, max_iter=200),
                                     x_out=x, y_out=y)
            out.append((st, [(i.status, i.iterations) for i in pd.pdqp_batch_info(h)], x, y))
        finally:
            pd.pdqp_destroy(h)
    assert info.spmv_threads == variant
    assert out[0][:2] == out[1][:2]
    np.testing.assert_array_equal(out[0][2], out[1][2])
    np.testing.assert_array_equal(out[0][3], out[1][3])
