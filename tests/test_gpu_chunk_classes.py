"""The one-launch chunk launches once per class of instances (by what shares an SM)
however the classes lie along the order of sizes: a batch of wide and sparse
problems beside narrow and dense ones of about as many entries."""
import numpy as np
import pytest

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def test_a_mixed_batch_takes_a_few_launches_a_chunk():
    pd = G.lib()
    insts = []
    for i in range(160):
        insts.append(qpgen.diagonal_box_qp(qpgen.SEED_BASE + 8200 + i, n=1800 + 9 * i))
        insts.append(qpgen.tiny_qp(qpgen.SEED_BASE + 8400 + i, n=64, m=1 + i % 23, m_eq=0, density=0.5))
    N = sum(i.n for i in insts)
    out, launches = {}, []
    h = pd.batch_from_instances(insts)
    try:
        for nt, iters in ((256, 128), (0, 64), (0, 128)):
            x = np.zeros(N)
            before = pd.pdqp_launch_count()
            _, info = pd.pdqp_solve(h, pd.pdqp_default_options(precision=1, spmv_threads=nt, max_iter=iters, eps=0.0,
                                                               no_graphs=1), x_out=x)
            launches.append(pd.pdqp_launch_count() - before)
            out[nt] = (x, info.spmv_threads)
    finally:
        pd.pdqp_destroy(h)
    assert out[0][1] == 2
    np.testing.assert_array_equal(out[0][0], out[256][0])
    # one chunk and its check (about a dozen kernels) more
    assert launches[2] - launches[1] <= 20, launches
