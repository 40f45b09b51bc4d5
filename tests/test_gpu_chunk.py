"""The one-launch chunk (a CTA or a cluster per instance, the matrices in 32-row
slices of 16-bit columns) against the per-iteration row-block kernels, bit for
bit: at the edges of the slices and of the entry pairs, without rows, on
batches whose instances share SMs and stop apart, on clusters, and where part
of the matrix streams from global memory."""
import numpy as np
import pytest

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu
SEED = qpgen.SEED_BASE + 7300


def edge_instances():
    """Rows and variables around multiples of 32, dense rows of odd and even length, no rows."""
    out = [qpgen.tiny_qp(SEED + 17 * n + m, n=n, m=m, m_eq=m // 2, bounds="mixed", density=d)
           for n in (1, 2, 31, 32, 33, 64, 65) for m, d in ((1, 1.0), (31, 0.5), (33, 1.0))]
    return out + [qpgen.diagonal_box_qp(SEED, n=n) for n in (1, 32, 45)]


def control_instances(count, T):
    return [qpgen.mpc_qp(SEED + 100 + i, T=T[i % len(T)]) for i in range(count)]


CASES = {
    "edges": edge_instances,
    # more than two instances an SM: one CTA each, two or four to an SM, the largest beside small ones
    "shared_sms": lambda: control_instances(320, (3, 5, 8, 12)) + control_instances(1, (120,)),
    # fewer instances than SMs: clusters
    "clusters": lambda: control_instances(21, (4, 30)),
    # more matrix than the shared memory of a cluster: the rest streams from global memory
    "streamed": lambda: [qpgen.tiny_qp(SEED + 500 + i, n=330 + i, m=165, m_eq=80, bounds="box") for i in range(20)],
}


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("case", sorted(CASES))
def test_chunk_is_bitwise_the_row_block_kernels(case, precision):
    pd = G.lib()
    insts = CASES[case]()
    N, M = sum(i.n for i in insts), sum(i.m for i in insts)
    res = {}
    for nt in (256, 0):
        h = pd.batch_from_instances(insts)
        try:
            x, y = np.zeros(N), np.zeros(M)
            _, info = pd.pdqp_solve(h, pd.pdqp_default_options(spmv_threads=nt, precision=precision, max_iter=700),
                                    x_out=x, y_out=y)
            res[nt] = (x, y, [(i.iterations, i.status) for i in pd.pdqp_batch_info(h)], info.spmv_threads)
        finally:
            pd.pdqp_destroy(h)
    assert res[0][3] == 2 and res[256][3] == 256
    assert res[0][2] == res[256][2]
    np.testing.assert_array_equal(res[0][0], res[256][0])
    np.testing.assert_array_equal(res[0][1], res[256][1])


def test_chunk_after_a_solve_of_the_other_precision_and_partial_chunks():
    """One handle, both precisions in turn, an iteration limit inside a period:
    the plan's two value arrays and launches do not mix."""
    pd = G.lib()
    insts = control_instances(30, (2, 9))
    N = sum(i.n for i in insts)
    out = {}
    for nt in (256, 0):
        h = pd.batch_from_instances(insts)
        try:
            got = []
            for precision, iters in ((1, 100), (0, 65), (1, 3), (0, 128)):
                x = np.zeros(N)
                pd.pdqp_solve(h, pd.pdqp_default_options(spmv_threads=nt, precision=precision, max_iter=iters, eps=0.0),
                              x_out=x)
                got.append(x)
            out[nt] = got
        finally:
            pd.pdqp_destroy(h)
    for a, b in zip(out[0], out[256]):
        np.testing.assert_array_equal(a, b)
