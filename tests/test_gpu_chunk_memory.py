"""A batch whose second copy of the matrices (the one-launch chunk's layout) does
not fit the memory that is left solves without it, with the same results; a
process of its own, since it fills the device's memory with one allocation."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = """
import numpy as np, torch
import qpgen
from tests import gpu_util as G
pd = G.lib()
kinds = [qpgen.large_sparse_qp(qpgen.SEED_BASE + 8000 + s, n=2000) for s in range(4)]
insts = [kinds[s % 4] for s in range(600)]
N = sum(i.n for i in insts)
torch.zeros(1, device="cuda")
def run(leave):
    h = pd.batch_from_instances(insts)
    fill = None
    try:
        if leave:
            fill = torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")
        x = np.zeros(N)
        st, info = pd.pdqp_solve(h, pd.pdqp_default_options(precision=0, max_iter=128, eps=0.0), x_out=x)
        return st, info.spmv_threads, x
    finally:
        pd.pdqp_destroy(h)
        del fill
        torch.cuda.empty_cache()
a = run(320 << 20)       # the layout: 31 million nonzeros, 10 bytes each and the pads
b = run(0)
assert a[0] == b[0] == pd.PDQP_ITER_LIMIT, (a[0], b[0])
assert a[1] != 2 and b[1] == 2, (a[1], b[1])
assert np.array_equal(a[2], b[2])
print("ok")
"""


def test_batch_without_room_for_the_layout():
    r = subprocess.run([sys.executable, "-c", SCRIPT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-500:] + r.stderr[-2000:]
