"""A row per thread on the slice layout (variant 5) is what the tuning chooses for a
large float64 problem (52 us an iteration against 85 with the row-block kernels at
this size), and its iterates are theirs bit for bit."""
import numpy as np
import pytest

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def test_variant_5_runs():
    G.lib()
    inst = qpgen.large_sparse_qp(qpgen.SEED_BASE + 8700, n=300_007)
    a, b = (G.solve(inst, precision=0, spmv_threads=nt, max_iter=192, eps=0.0) for nt in (256, 0))
    assert b[1].spmv_threads == 5
    np.testing.assert_array_equal(a[2], b[2])
    np.testing.assert_array_equal(a[3], b[3])
