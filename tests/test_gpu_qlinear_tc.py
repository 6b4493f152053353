"""The tcgen05 linear layer at the edges of its pipeline: one to several weight tiles per CTA, a tile cut off by the end of a
split, one split to many, pairs of CTAs and odd splits, ragged channels, batch rows on both sides of 128 and 256, activations
of very different magnitude per row.  Bound for 4 / 8 / 16 bits: an activation enters with 2^-22 of itself or 2^-39 of its
row's maximum; the tensor cores add K products (and up to 64 partial sums) in float32 with at most 2^-22 of the sum of
magnitudes each 16, so |delta| <= (K / 16 + 80) 2^-22 s_n sum_k |w x| is ample.  32 bits: 2^-16 for the split operands."""
import numpy as np
import pytest

from oracle import aiq_oracle as O
from gpu_util import binding, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [4, 8, 16, 32])
@pytest.mark.parametrize("N,K,M", [(8192, 8192, 9), (5000, 1480, 16), (7000, 712, 33), (4096, 4096, 17), (2000, 8184, 65),
                                   (4000, 1000, 128), (4001, 1000, 129), (1100, 520, 144), (900, 2048, 256),
                                   (40, 8192, 257), (2200, 648, 300), (513, 328, 600)])
def test_tc_bound(bits, N, K, M):
    import torch
    aiq = binding()
    nbytes = aiq.aiq_qlinear_workspace_bytes(N, K, bits, M)
    assert nbytes > 0
    rng = np.random.default_rng(N + K + M)
    W = rng.standard_normal((N, K)).astype(np.float32)
    x = (rng.standard_normal((M, K)) * np.exp(rng.uniform(-20, 20, (M, 1)))).astype(np.float32)
    x[:, 3::11] *= 1e-3
    x[M // 2] = 0
    bias = rng.standard_normal(N).astype(np.float32) if N % 2 else None
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, bits)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(to_dev(W), bits, packed, scales)
    y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    ws = torch.full((nbytes,), 255, dtype=torch.uint8, device="cuda")
    aiq.aiq_qlinear(packed, scales, to_dev(bias) if bias is not None else None, N, K, bits, to_dev(x), y, workspace=ws)
    got = y.cpu().numpy()
    assert int(ws[-16:-12].cpu().numpy().view(np.int32)[0]) == 0            # no wait expired
    v, s = O.quantize_rows(W, bits)
    w = v.astype(np.float64) * np.asarray(s, np.float64)[:, None]
    want = x.astype(np.float64) @ w.T + (0 if bias is None else bias.astype(np.float64))
    mags = np.abs(x).astype(np.float64) @ np.abs(w).T
    tol = 2.0 ** -16 if bits == 32 else 0.0
    bound = ((K / 16 + 80) * 2.0 ** -22 + tol) * mags + 2.0 ** -22 * np.abs(want) + 1e-30
    bound += 2.0 ** -39 * np.abs(x).max(axis=1)[:, None].astype(np.float64) * np.abs(w).sum(axis=1)[None, :]
    assert np.all(np.abs(got - want) <= bound)


@pytest.mark.parametrize("N,K,M,limit", [(8192, 8192, 16, 2.0e-6), (8192, 8192, 256, 6.3e-6), (8192, 4096, 256, 3.7e-6),
                                         (4096, 4096, 64, 5.0e-7), (2048, 2048, 64, 2.5e-7)])
def test_tc_rounding_error_at_8_bits(N, K, M, limit):
    """The tensor cores drop what a product has below the accumulator's last bit.  Limits: below what bfloat16 pairs give
    (2.6e-6, 6.4e-6, 3.8e-6, 2.5e-6, 2.5e-6 of the result's norm), and at short sums what the activations' 22 bits allow."""
    import torch
    aiq = binding()
    g = torch.Generator(device="cuda").manual_seed(N + K + M)
    W = torch.randn(N, K, generator=g, device="cuda") * 0.02
    x = torch.randn(M, K, generator=g, device="cuda")
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, 8)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(W, 8, packed, scales)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    ws = torch.empty(aiq.aiq_qlinear_workspace_bytes(N, K, 8, M), dtype=torch.uint8, device="cuda")
    aiq.aiq_qlinear(packed, scales, None, N, K, 8, x, y, workspace=ws)
    want = x.double() @ (packed.view(torch.int8)[:, :K].double() * scales.double()[:, None]).T
    assert ((y.double() - want).norm() / want.norm()).item() <= limit
