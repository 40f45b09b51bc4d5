"""A float64 batch at an iteration limit that ends its last chunk after an odd
number of iterations: the members that stopped in an earlier period return the
y they stopped with, in every iteration-kernel variant (the handle's y then is
the other half of the double buffer, which a stopped member's later chunks do
not write), and so does a state saved there."""
import numpy as np
import pytest

import qpgen
from oracle import rapdhg as R
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _members():
    out = [qpgen.mpc_qp(qpgen.SEED_BASE + 7900 + i, T=3 + i % 6) for i in range(24)]
    # the all-zero start is optimal: stops before the first chunk
    z = qpgen.tiny_qp(qpgen.SEED_BASE + 7950, n=20, m=8, m_eq=4, bounds="box")
    z.c = np.zeros(z.n)
    z.b = np.concatenate([np.zeros(4), np.full(4, -1.0)])
    return out[:11] + [z] + out[11:]


def _solve(pd, h, sizes, **opts):
    x, y = np.full(sizes[0], np.nan), np.full(sizes[1], np.nan)
    pd.pdqp_solve(h, pd.pdqp_default_options(precision=0, accelerate=0, **opts), x_out=x, y_out=y)
    return x, y, pd.pdqp_batch_info(h)


@pytest.mark.parametrize("nt", [0, 1, 2, 256, 512])
def test_stopped_members_return_the_iterate_they_stopped_with(nt):
    pd = G.lib()
    insts = _members()
    sizes = sum(i.n for i in insts), sum(i.m for i in insts)
    xo, yo = np.cumsum([0] + [i.n for i in insts]), np.cumsum([0] + [i.m for i in insts])
    h = pd.batch_from_instances(insts)
    try:
        long = _solve(pd, h, sizes, spmv_threads=nt, max_iter=20000, eps=1e-4)[2]
        its = sorted(i.iterations for i in long if i.status == pd.PDQP_OK)
        limit = its[len(its) // 2] + 1              # after half of the members' last checks, odd
        assert limit % 2 == 1 and its[-1] > limit
        x, y, infos = _solve(pd, h, sizes, spmv_threads=nt, max_iter=limit, eps=1e-4)
        stopped = [k for k, i in enumerate(infos) if i.status == pd.PDQP_OK]
        assert 0 < len(stopped) < len(insts) and infos[11].iterations == 0 and 11 in stopped
        blob = pd.pdqp_get_state(h)
    finally:
        pd.pdqp_destroy(h)
    for k in stopped:
        parts = R.kkt_parts(R.problem_from_instance(insts[k]), x[xo[k]:xo[k + 1]], y[yo[k]:yo[k + 1]])
        # the device's own value of the same iterate: float64 sums of a few dozen terms
        assert parts["rel_kkt"] == pytest.approx(infos[k].rel_kkt, rel=1e-6, abs=1e-12), k
    h = pd.batch_from_instances(insts)
    try:
        pd.pdqp_set_state(h, blob)
        x2, y2, infos2 = _solve(pd, h, sizes, spmv_threads=nt, max_iter=limit + 64, eps=1e-4)
    finally:
        pd.pdqp_destroy(h)
    for k in stopped:
        np.testing.assert_array_equal(x2[xo[k]:xo[k + 1]], x[xo[k]:xo[k + 1]])
        np.testing.assert_array_equal(y2[yo[k]:yo[k + 1]], y[yo[k]:yo[k + 1]])


@pytest.mark.parametrize("nt", [0, 3])
def test_stopped_members_of_a_family(nt):
    pd = G.lib()
    fam = qpgen.family_qp(qpgen.SEED_BASE + 7960, n=420, m=210)
    cnt, base = 12, fam.base
    n, m = base.n, base.m
    C, B = fam.params(0, cnt)
    C[7] = 0.0                                      # the all-zero start is optimal
    B[7] = np.where(np.arange(m) < base.m_eq, 0.0, -1.0)
    h = pd.family_from_base(base, C, B)
    try:
        long = _solve(pd, h, (cnt * n, cnt * m), spmv_threads=nt, max_iter=50000, eps=1e-5)[2]
        its = sorted(i.iterations for i in long if i.status == pd.PDQP_OK)
        limit = its[len(its) // 2] + 1
        assert limit % 2 == 1 and its[-1] > limit
        x, y, infos = _solve(pd, h, (cnt * n, cnt * m), spmv_threads=nt, max_iter=limit, eps=1e-5)
    finally:
        pd.pdqp_destroy(h)
    stopped = [k for k, i in enumerate(infos) if i.status == pd.PDQP_OK]
    assert 0 < len(stopped) < cnt
    for k in stopped:
        inst = qpgen.QPInstance("member", n, m, base.m_eq, base.Q, base.A, C[k], B[k], base.l, base.u)
        parts = R.kkt_parts(R.problem_from_instance(inst), x[k * n:(k + 1) * n], y[k * m:(k + 1) * m])
        assert parts["rel_kkt"] == pytest.approx(infos[k].rel_kkt, rel=1e-6, abs=1e-12), k
