"""The norm estimates of instances of two to four chunks of row blocks (33 to 128
row blocks of P) in a batch whose vector-update grid runs in several waves: the
chunk sums of v'w that one warp reads and those of |r|^2 that another chunk closes
in the same launch must not be the same memory, so every copy's norms are the
standalone ones bit for bit, whatever the order of the blocks."""
import pytest

import qpgen
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_norms_of_several_chunks_match_standalone_in_a_batch_of_several_waves(precision):
    P = G.lib()
    kinds = [qpgen.large_sparse_qp(qpgen.SEED_BASE + 7800 + n, n=n) for n in (4500, 6000, 8500, 12000)]
    o = P.pdqp_default_options(precision=precision, max_iter=2, eps=0.0)
    want = []
    for inst in kinds:
        blocks = (inst.Q.nnz + inst.A.nnz) / 2048
        assert 33 <= blocks and blocks * 1.05 <= 128        # two to four chunks of 32
        h = G.handle(inst)
        try:
            info = P.pdqp_solve(h, o)[1]
        finally:
            P.pdqp_destroy(h)
        want.append((info.norm_A, info.norm_Q, info.norm_iters))
    assert min(w[2] for w in want) > 8
    order = [(7 * i) % len(kinds) for i in range(240)]      # about 2000 blocks of eight warps
    h = P.batch_from_instances([kinds[k] for k in order])
    try:
        for _ in range(3):
            P.pdqp_solve(h, o)
            got = [(i.norm_A, i.norm_Q, i.norm_iters) for i in P.pdqp_batch_info(h)]
            assert got == [want[k] for k in order]
    finally:
        P.pdqp_destroy(h)
