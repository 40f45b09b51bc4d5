"""The fitted statistics of columns whose deviations lie around the ends of the
float32 pairs' range: single squares below float32's largest value whose sum over
a range of rows is above it, and values far below and above."""
import numpy as np
import pytest

from tests.gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [64, 200])
def test_fit_statistics_across_the_pairs_range(count):
    """Float32 roundings (2^-24 relative) of values whose own error is below 1e-9
    relative."""
    pd = lib()
    rng = np.random.default_rng(count)
    scales = 2.0 ** np.array([-60.0, -52, -50, -48, 0, 50, 57, 58, 59, 60, 61, 62, 63, 64, 65, 70, 100])
    n = scales.size
    # every value near the scale: the squares of a range sum to 50 times the scale's
    data = [rng.choice([-1.0, 1.0], (count, n)) * rng.uniform(0.9, 1.0, (count, n)) * scales for _ in range(2)]
    empty = np.zeros((count, 0))
    w = pd.pdqp_ws_create(n, 0, 8, 8, 1, 8)
    try:
        pd.pdqp_ws_fit(w, data[0], empty, data[1], empty)
        got = pd.pdqp_ws_get_normalization(w, n)
    finally:
        pd.pdqp_ws_destroy(w)
    std = [np.where(d.std(0) < 1e-8, 1.0, d.std(0)) for d in data]
    err = np.abs(got["in_mean"] - data[0].mean(0))      # a mean near zero: relative to the values
    assert (err <= 1.3e-7 * np.abs(data[0].mean(0)) + 1e-12 * scales).all()
    np.testing.assert_allclose(got["in_scale"], 1 / std[0], rtol=1.3e-7)
    np.testing.assert_allclose(got["out_std"], std[1], rtol=1.3e-7)
    np.testing.assert_allclose(got["out_inv"], 1 / std[1], rtol=1.3e-7)
