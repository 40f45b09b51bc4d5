"""The one-launch chunk with clusters of unequal sizes: fewer instances than SMs
whose horizons differ, from one CTA to sixteen for an instance, in both precisions
in turn on one handle, bit for bit against the row-block kernels."""
import numpy as np
import pytest

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("horizons", [
    [2 + 3 * k for k in range(30)],            # small and large ones: clusters of many sizes
    [40] * 90,                                 # equal ones, more than half as many as SMs
    list(range(1, 151)),                       # nearly as many instances as SMs
    [1, 100],
], ids=["uneven30", "equal90", "uneven150", "two"])
def test_uneven_clusters(horizons):
    pd = G.lib()
    insts = [qpgen.mpc_qp(qpgen.SEED_BASE + 9100 + i, T=T) for i, T in enumerate(horizons)]
    N, M = sum(i.n for i in insts), sum(i.m for i in insts)
    out = {}
    for nt in (256, 0):
        h = pd.batch_from_instances(insts)
        try:
            got = []
            for precision in (1, 0):
                x, y = np.zeros(N), np.zeros(M)
                _, info = pd.pdqp_solve(h, pd.pdqp_default_options(spmv_threads=nt, precision=precision, max_iter=300),
                                        x_out=x, y_out=y)
                assert info.spmv_threads == nt or nt == 0
                got.append((x, y, [(i.iterations, i.status) for i in pd.pdqp_batch_info(h)]))
            out[nt] = got
        finally:
            pd.pdqp_destroy(h)
    for a, b in zip(out[0], out[256]):
        assert a[2] == b[2]
        np.testing.assert_array_equal(a[0], b[0])
        np.testing.assert_array_equal(a[1], b[1])
