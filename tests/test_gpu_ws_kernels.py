"""Edges of the network's kernels: the fitted statistics at the ends of their
row ranges and for values outside the float32 pairs' range, the elementwise
kernels with odd feature counts, and the GEMM on CTA pairs at the edges of its
tiles and widths."""
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


@pytest.mark.parametrize("M,N,K,ld", [
    (129, 256, 8, 8),          # one pair, its second CTA a single row; one ragged k-tile
    (255, 257, 72, 72),        # a last tile of one column
    (256, 512, 64, 64),        # whole tiles
    (300, 1000, 520, 528),     # several tiles, ragged everywhere
    (1100, 2048, 136, 136),    # more tiles than one wave of narrow ones
    (513, 30001, 64, 64),      # many tiles, odd N
])
@pytest.mark.parametrize("epilogue", ["plain", "bias_relu_mask_bf16"])
def test_gemm_pairs(M, N, K, ld, epilogue):
    """|D - ref| <= 4 K 2^-24 |A||B|' as a float32 sum of exact products in any
    order; a bf16 output adds half an ulp (2^-8 of the value covers it)."""
    import torch
    pd = lib()
    g = torch.Generator(device="cuda").manual_seed(M * N + K)
    A = torch.randn(M, ld, generator=g, device="cuda").bfloat16()
    B = torch.randn(N, ld, generator=g, device="cuda").bfloat16()
    ref = A[:, :K].double() @ B[:, :K].double().T
    bound = 4 * K * 2.0 ** -24 * (A[:, :K].double().abs() @ B[:, :K].double().abs().T) + 1e-30
    if epilogue == "plain":
        D = torch.full((M, N), float("nan"), device="cuda")
        pd.pdqp_gemm_bf16(A, B, D_f32=D, K=K)
    else:
        bias = torch.randn(N, generator=g, device="cuda")
        mask = torch.randn(M, N, generator=g, device="cuda").bfloat16()
        D = torch.full((M, N), float("nan"), device="cuda", dtype=torch.bfloat16)
        pd.pdqp_gemm_bf16(A, B, bias=bias, relu=True, mask=mask, D_bf16=D, K=K)
        ref = torch.relu(ref + bias.double())
        ref[~(mask > 0)] = 0.0
        bound = bound + 2.0 ** -8 * ref.abs() + 2.0 ** -23 * bias.double().abs()
    assert pd.pdqp_gemm_bf16_check() == 0
    err = (D.double() - ref).abs()
    assert bool((err <= bound).all()), float((err / bound).max())
