"""Edges of the network's kernels: the fitted statistics at the ends of their
row ranges, with odd feature counts and for values outside the float32 pairs'
range."""
import numpy as np
import pytest

from tests.gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 2, 63, 64, 65, 129, 1000])
@pytest.mark.parametrize("n,m", [(5, 0), (257, 33)])
def test_fit_statistics(n, m, count):
    """Against float64 numpy.  The outputs are float32 roundings (2^-24
    relative) of values whose own error is below 1e-9 relative (offsets of at
    most 1e4 deviations: 2^-46 of the offset)."""
    pd = lib()
    rng = np.random.default_rng(1000 * count + n)
    scale = 10.0 ** rng.uniform(-3, 3, n + m)
    data = [rng.standard_normal((count, k)) * s + o for k, s, o in
            ((n, scale[:n], 100 * scale[:n]), (m, scale[n:], 0.0), (n, scale[:n], -1e4 * scale[:n]), (m, scale[n:], scale[n:]))]
    data[0][:, 0] *= 1e25                        # squares beyond float32
    data[2][:, 1] = 3.25                         # constant
    w = pd.pdqp_ws_create(n, m, 8, 8, 1, 8)
    try:
        pd.pdqp_ws_fit(w, *data)
        got = pd.pdqp_ws_get_normalization(w, n + m)
    finally:
        pd.pdqp_ws_destroy(w)
    v, t = np.concatenate(data[:2], 1), np.concatenate(data[2:], 1)
    std = lambda a: np.where(a.std(0) < 1e-8, 1.0, a.std(0))
    want = dict(in_mean=v.mean(0), in_scale=1 / std(v), out_mean=t.mean(0), out_std=std(t), out_inv=1 / std(t))
    for k, x in want.items():
        np.testing.assert_allclose(got[k], x, rtol=1.3e-7, atol=0, err_msg=k)
