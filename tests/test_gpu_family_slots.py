"""The interleaved vectors of a family hold its running members densely: member
counts at the edges of a lane (4), of a warp (128) and of the slot scan (1024),
members that stop at different checks and a short check period, bit for bit
against the row-block kernels."""
import numpy as np
import pytest

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("count,period", [(1, 64), (5, 6), (127, 64), (129, 6), (1025, 64)])
def test_dense_slots(count, period, precision):
    pdqp = G.lib()
    fam = qpgen.family_qp(n=60, m=30)
    C, B = fam.params(3, count)
    out = []
    for nt in (256, 3):
        h = pdqp.family_from_base(fam.base, C, B)
        try:
            x, y = np.zeros(count * 60), np.zeros(count * 30)
            st, info = pdqp.pdqp_solve(h, pdqp.pdqp_default_options(precision=precision, spmv_threads=nt,
                                                                    check_period=period), x_out=x, y_out=y)
            out.append((st, [(i.status, i.iterations) for i in pdqp.pdqp_batch_info(h)], x, y))
        finally:
            pdqp.pdqp_destroy(h)
    assert out[0][:2] == out[1][:2] and out[0][0] == pdqp.PDQP_OK
    np.testing.assert_array_equal(out[0][2], out[1][2])
    np.testing.assert_array_equal(out[0][3], out[1][3])
