"""A family on the interleaved kernels whose check period is longer than the block
of iterations whose step scalars it holds at a time: bit for bit the row-block
kernels, at the block's edges and past an iteration limit inside one."""
import numpy as np
import pytest

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("period,limit", [(256, 512), (258, 600), (1024, 1500)])
def test_period_longer_than_the_step_block(period, limit, precision):
    pd = G.lib()
    fam = qpgen.family_qp(qpgen.SEED_BASE + 8600, n=60, m=30)
    C, B = fam.params(2, 7)
    out = []
    for nt in (256, 3):
        h = pd.family_from_base(fam.base, C, B)
        try:
            x, y = np.zeros(7 * 60), np.zeros(7 * 30)
            pd.pdqp_solve(h, pd.pdqp_default_options(precision=precision, spmv_threads=nt, check_period=period,
                                                     max_iter=limit, eps=0.0), x_out=x, y_out=y)
            out.append((x, y))
        finally:
            pd.pdqp_destroy(h)
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
