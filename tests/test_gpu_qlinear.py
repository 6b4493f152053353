"""CUDA small-batch quantized linear layer against the oracle."""
import numpy as np
import pytest

from aiq_workloads import gen_linear_case
from oracle import aiq_oracle as O
from gpu_util import binding, to_dev, assert_logits_close

pytestmark = pytest.mark.gpu


def _run(aiq, W, x, bits, bias=None, use_workspace=True):
    import torch
    N, K = W.shape
    rb = aiq.aiq_packed_row_bytes(K, bits)
    packed = torch.empty((N, rb), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(to_dev(W), bits, packed, scales)
    y = torch.full((x.shape[0], N), float("nan"), dtype=torch.float32, device="cuda")
    ws_bytes = aiq.aiq_qlinear_workspace_bytes(N, K, bits, x.shape[0]) if use_workspace else 0
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda") if ws_bytes else None
    aiq.aiq_qlinear(packed, scales, to_dev(bias) if bias is not None else None, N, K, bits, to_dev(x), y,
                    workspace=ws)
    torch.cuda.synchronize()
    v, s = O.quantize_rows(W, bits)
    return y.cpu().numpy(), O.qlinear(v, s, bias, bits, x)


@pytest.mark.parametrize("bits", [4, 8, 16, 32])
@pytest.mark.parametrize("N,K,M", [(1280, 320, 1), (1280, 320, 4), (1280, 320, 16), (10, 64, 64),
                                   (1000, 1280, 5), (37, 100, 3), (5, 27, 2), (4096, 4096, 1),
                                   (2048, 4096, 4), (300, 2052, 7), (1, 1, 1),
                                   # shapes on the warp-level tensor-core path (K % 512 == 0, N*K >= 2^20)
                                   (4100, 512, 16), (1000, 1536, 3), (2050, 1024, 9), (8192, 8192, 2),
                                   (1030, 1024, 1), (4100, 8192, 2), (2048, 3072, 2),
                                   # batches on the tcgen05 path (M >= 9, K % 8 == 0): ragged N, K and M tails,
                                   # several batch blocks, K split over CTAs
                                   (4096, 4096, 256), (1280, 320, 256), (1000, 1280, 37), (2050, 1024, 300),
                                   (130, 72, 16), (33, 64, 9), (4100, 520, 64)])
def test_qlinear_matches_oracle(bits, N, K, M):
    aiq = binding()
    W, x = gen_linear_case(N, K, M, seed=3234 + N + K + M)
    bias = np.random.default_rng(N).standard_normal(N).astype(np.float32) if N % 2 == 0 else None
    got, ref = _run(aiq, W, x, bits, bias)
    assert_logits_close(got, ref, f"N={N} K={K} M={M} bits={bits}")
    if aiq.aiq_qlinear_workspace_bytes(N, K, bits, M):        # the same shape on the plain kernel
        got, ref = _run(aiq, W, x, bits, bias, use_workspace=False)
        assert_logits_close(got, ref, f"plain N={N} K={K} M={M} bits={bits}")


@pytest.mark.parametrize("bits", [4, 8])
def test_qlinear_exact_on_integers(bits):
    """Integer weights and activations: every product and partial sum is exact in float32,
    so the result must equal the integer answer exactly (s = 1)."""
    aiq = binding()
    rng = np.random.default_rng(1)
    qmax = 2 ** (bits - 1) - 1
    # plain / int8 warp-level (M = 5 and M = 2) / tcgen05
    for shape_w, m in (((96, 200), 4), ((2176, 512), 5), ((2176, 2048), 2), ((300, 520), 20)):
        W = rng.integers(-qmax, qmax + 1, shape_w).astype(np.float32)
        W[:, 0] = qmax
        x = rng.integers(-8, 9, (m, shape_w[1])).astype(np.float32)
        got, ref = _run(aiq, W, x, bits)
        want = x.astype(np.int64) @ W.astype(np.int64).T
        assert np.array_equal(got.astype(np.int64), want)
        assert np.array_equal(ref.astype(np.int64), want)


@pytest.mark.parametrize("bits", [16, 32])
def test_qlinear_two_piece_path_exact_on_integers(bits):
    """16- and 32-bit weights on the tcgen05 kernel enter as two bfloat16 pieces.  Small integer
    weights and activations make every product and sum exact, so any dropped, repeated or stale
    tile shows up as a wrong integer.  Shapes with many K chunks per CTA, several batch blocks and
    K splits; each shape is run three times (a race would not repeat)."""
    aiq = binding()
    for (N, K, M) in ((128, 64, 16), (256, 512, 32), (4096, 4096, 128), (2048, 2048, 256), (4096, 4096, 256),
                      (1000, 1288, 300)):
        rng = np.random.default_rng(N + K + M + bits)
        W = rng.integers(-3, 4, (N, K)).astype(np.float32)
        x = rng.integers(-2, 3, (M, K)).astype(np.float32)
        want = x.astype(np.int64) @ W.astype(np.int64).T
        for trial in range(3):
            got, ref = _run(aiq, W, x, bits)
            assert np.array_equal(got.astype(np.int64), want), (N, K, M, bits, trial)


@pytest.mark.parametrize("N,K,M", [(512, 512, 16), (4096, 4096, 1), (2048, 1024, 6), (4096, 4096, 64), (8192, 64, 9)])
def test_qlinear_refuses_a_misaligned_workspace(N, K, M):
    """Wherever a kernel with scratch exists for the shape, also where another one runs; elsewhere the workspace is ignored."""
    import torch
    aiq = binding()
    W, x = gen_linear_case(N, K, M, seed=5)
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, 4)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(to_dev(W), 4, packed, scales)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
    with pytest.raises(aiq.AiqError) as e:
        aiq.aiq_qlinear(packed, scales, None, N, K, 4, to_dev(x), y, workspace=ws[4:])
    assert e.value.status == aiq.ERR_INVALID_ARG
    aiq.aiq_qlinear(packed, scales, None, N, K, 4, to_dev(x), y, workspace=ws)
    small = torch.empty((30, aiq.aiq_packed_row_bytes(100, 4)), dtype=torch.uint8, device="cuda")
    aiq.aiq_quantize_layer(torch.randn((30, 100), device="cuda"), 4, small, scales[:30])
    aiq.aiq_qlinear(small, scales[:30], None, 30, 100, 4, torch.zeros((M, 100), device="cuda"), y.view(-1)[:30 * M].view(M, 30), workspace=ws[4:])


@pytest.mark.parametrize("N,K", [(13000, 8192), (100001, 1024), (51000, 2048)])
@pytest.mark.parametrize("M", [1, 2, 3, 4])
def test_large_4_bit_layer_with_scratch(N, K, M):
    """Above 3 x 2^25 weights the kernel with scratch takes up to four rows.  Integers beside activations that only the fourth
    digit holds (j 2^-26 where the largest of every 512 is 1 and meets a zero weight): every sum is exact, with and without
    the workspace.  An infinity makes its own row not finite."""
    import torch
    aiq = binding()
    g = torch.Generator(device="cuda").manual_seed(N + K + M)
    W = torch.randint(-7, 8, (N, K), generator=g, device="cuda").float()
    W[:, 1] = 7
    W[:, ::64] = 0
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, 4)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(W, 4, packed, scales)
    ws = torch.empty(aiq.aiq_qlinear_workspace_bytes(N, K, 4, M), dtype=torch.uint8, device="cuda")
    assert ws.numel() > 0
    j = torch.randint(-63, 64, (M, K), generator=g, device="cuda")
    x = j.float() * 2.0 ** -26
    x[:, ::64] = 1.0
    j[:, ::64] = 0
    want = j.double() @ W.double().T
    for workspace in (ws, None):
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        aiq.aiq_qlinear(packed, scales, None, N, K, 4, x, y, workspace=workspace)
        assert torch.equal(y.double() * 2.0 ** 26, want)
    x[M - 1, 700] = float("inf")
    aiq.aiq_qlinear(packed, scales, None, N, K, 4, x, y, workspace=ws)
    assert torch.equal(y[:M - 1].double() * 2.0 ** 26, want[:M - 1])
    assert not bool(torch.isfinite(y[M - 1]).any())


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("N,K,M", [(33000, 512, 5), (18000, 1024, 8), (8200, 2048, 6)])
def test_digit_kernel_extreme_activations(bits, N, K, M):
    """Five to eight rows with scratch: infinities and NaN make their rows not finite, and slices of denormals count, in rows
    beside ordinary ones; integers, so that what is finite is exact, but for what float atomics flush: denormal addends and
    sums, less than 2^-126 each, three digits and up to K / 512 slices an output."""
    import torch
    aiq = binding()
    g = torch.Generator(device="cuda").manual_seed(N + K + M)
    W = torch.randint(-7, 8, (N, K), generator=g, device="cuda").float()
    W[:, 1] = 7 if bits == 4 else 127
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, bits)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(W, bits, packed, scales)
    ws = torch.empty(aiq.aiq_qlinear_workspace_bytes(N, K, bits, M), dtype=torch.uint8, device="cuda")
    assert ws.numel() > 0
    unit = torch.ones(M, 1, device="cuda")
    unit[1] = 2.0 ** -132
    x = torch.randint(-63, 64, (M, K), generator=g, device="cuda").float() * unit
    x[2, K - 1] = float("inf")
    x[M - 1, 17] = float("nan")
    y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    aiq.aiq_qlinear(packed, scales, None, N, K, bits, x, y, workspace=ws)
    want = (torch.where(x.isfinite(), x, 0).double() @ W.double().T).float()
    assert not bool(torch.isfinite(y[[2, M - 1]]).any())
    assert float((y[1].double() - want[1].double()).abs().max()) <= 2 * 3 * (K // 512) * 2.0 ** -126
    rest = [m for m in range(M) if m not in (1, 2, M - 1)]
    assert torch.equal(y[rest], want[rest])
