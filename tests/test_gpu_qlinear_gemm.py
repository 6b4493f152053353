"""The tiled float32 linear kernel (five and more rows) at the edges of its tiles, thread groups and clusters.  Bound: each
output is a float32 sum of K rounded products in some order, so |delta| <= (K + 2) 2^-24 s_n sum_k |w x|, plus the rounding
of the scaled sum and of the bias.  The sums meet in a fixed order: the same bits twice."""
import numpy as np
import pytest

from oracle import aiq_oracle as O
from gpu_util import binding, to_dev

pytestmark = pytest.mark.gpu


# every tile (64x64, 64x32, 32x32, 64x8, 32x16 channels x rows), whole and ragged; K below one slice, at its edge and odd;
# one block per tile up to clusters of eight; both sides of 2^26 products (without workspace the rest runs here too)
@pytest.mark.parametrize("bits", [4, 8, 16, 32])
@pytest.mark.parametrize("N,K,M", [(1, 1, 5), (31, 33, 7), (33, 31, 9), (70, 8190, 5), (64, 4096, 16), (300, 1001, 17),
                                   (2048, 96, 17), (4097, 65, 33), (9473, 40, 64), (9472, 32, 65), (1024, 129, 256),
                                   (4096, 2049, 8), (512, 512, 256), (513, 513, 255)])
def test_gemm_bound(bits, N, K, M):
    import torch
    aiq = binding()
    rng = np.random.default_rng(N + K + M)
    W = rng.standard_normal((N, K)).astype(np.float32)
    x = rng.standard_normal((M, K)).astype(np.float32)
    bias = rng.standard_normal(N).astype(np.float32) if N % 2 else None
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, bits)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(to_dev(W), bits, packed, scales)
    ys = []
    for _ in range(2):
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        aiq.aiq_qlinear(packed, scales, to_dev(bias) if bias is not None else None, N, K, bits, to_dev(x), y)
        ys.append(y.cpu().numpy())
    assert np.array_equal(ys[0], ys[1])
    v, s = O.quantize_rows(W, bits)
    w = v.astype(np.float64) * np.asarray(s, np.float64)[:, None]
    want = x.astype(np.float64) @ w.T + (0 if bias is None else bias.astype(np.float64))
    bound = (K + 2) * 2.0 ** -24 * (np.abs(x).astype(np.float64) @ np.abs(w).T) + 2.0 ** -22 * np.abs(want) + 1e-30
    assert np.all(np.abs(ys[0] - want) <= bound)


@pytest.mark.parametrize("bits", [4, 16])
@pytest.mark.parametrize("N,K,M", [(8192, 777, 64), (8192, 777, 6), (1001, 1999, 256), (9473, 4096, 72), (4800, 2100, 33)])
def test_gemm_rounding_error(bits, N, K, M):
    """Long chains of additions are broken up.  n additions in sequence leave about 2^-25 sqrt(n / 2) of the result's norm; a
    lane's share of K / 32 products, or two levels of fewer, stays below 2^-24 (1.5 + sqrt(K) / 20); one chain of K / 2 does not."""
    import torch
    aiq = binding()
    g = torch.Generator(device="cuda").manual_seed(N + K + M)
    W = torch.randn(N, K, generator=g, device="cuda")
    x = torch.randn(M, K, generator=g, device="cuda")
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, bits)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(W, bits, packed, scales)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    aiq.aiq_qlinear(packed, scales, None, N, K, bits, x, y)
    if bits == 16:
        w = packed.view(torch.float16)[:, :K].double()
    else:
        codes = torch.stack([packed & 15, packed >> 4], 2).reshape(N, -1)[:, :K].to(torch.int16)
        w = torch.where(codes > 7, codes - 16, codes).double() * scales.double()[:, None]
    want = x.double() @ w.T
    error = ((y.double() - want).norm() / want.norm()).item()
    assert error <= 2.0 ** -24 * (1.5 + K ** 0.5 / 20)


# the kernel of four rows: one launch chained and unchained, rows of x aligned and not, five to eight rows as two of four
@pytest.mark.parametrize("bits", [4, 8, 16, 32])
@pytest.mark.parametrize("N,K,M", [(512, 512, 3), (513, 511, 4), (3000, 2900, 4), (2600, 3301, 3), (1100, 8023, 1), (1200, 8023, 2),
                                   (601, 1001, 2), (330, 288, 5), (1535, 509, 8), (1000, 1280, 7), (4801, 3600, 6), (6200, 516, 5)])
def test_rows_of_four_bound(bits, N, K, M):
    import torch
    aiq = binding()
    rng = np.random.default_rng(N + K + M)
    W = rng.standard_normal((N, K)).astype(np.float32)
    x = rng.standard_normal((M, K)).astype(np.float32)
    bias = rng.standard_normal(N).astype(np.float32) if N % 2 else None
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, bits)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(to_dev(W), bits, packed, scales)
    ys = []
    for _ in range(2):
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        aiq.aiq_qlinear(packed, scales, to_dev(bias) if bias is not None else None, N, K, bits, to_dev(x), y)
        ys.append(y.cpu().numpy())
    assert np.array_equal(ys[0], ys[1])
    v, s = O.quantize_rows(W, bits)
    w = v.astype(np.float64) * np.asarray(s, np.float64)[:, None]
    want = x.astype(np.float64) @ w.T + (0 if bias is None else bias.astype(np.float64))
    bound = (K + 2) * 2.0 ** -24 * (np.abs(x).astype(np.float64) @ np.abs(w).T) + 2.0 ** -22 * np.abs(want) + 1e-30
    assert np.all(np.abs(ys[0] - want) <= bound)
