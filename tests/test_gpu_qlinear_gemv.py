"""The one-kernel linear layer for up to four rows, at its edges: rows whose packed length is no multiple of a chunk or of 32
elements, fewer and more channels than a unit per SM, one warp to sixteen warps per unit, the longest row, one to four
batch rows, activations over a wide range of magnitudes.  Bound: the integer sums are exact; the digits hold x to 2^-27 of
the largest |x| of its slice, digit sums and the at most 16 partial sums round to 2^-24 each, so
|delta| <= 2^-20 s_n sum_k |code| max|x| is ample (random errors average out far below it; that all four digits take part
is a test of its own).  Integer inputs come out exactly.  The kernel needs no workspace and gives the same bits twice."""
import numpy as np
import pytest

from oracle import aiq_oracle as O
from gpu_util import binding, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("N,K,M", [(1024, 520, 1), (1030, 777, 2), (40, 8192, 3), (2999, 1000, 4), (520, 8190, 1),
                                   (9000, 4100, 4), (20000, 512, 2)])
def test_gemv_bound(bits, N, K, M):
    import torch
    aiq = binding()
    rng = np.random.default_rng(N + K + M)
    W = rng.standard_normal((N, K)).astype(np.float32)
    x = (rng.standard_normal((M, K)) * np.exp(rng.uniform(-12, 4, (M, K)))).astype(np.float32)
    x[:, :: 7] = 0
    bias = rng.standard_normal(N).astype(np.float32)
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, bits)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(to_dev(W), bits, packed, scales)
    ys = []
    for _ in range(2):
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        aiq.aiq_qlinear(packed, scales, to_dev(bias), N, K, bits, to_dev(x), y)
        ys.append(y.cpu().numpy())
    assert np.array_equal(ys[0], ys[1])
    v, s = O.quantize_rows(W, bits)
    want = x.astype(np.float64) @ (v.astype(np.float64) * np.asarray(s, np.float64)[:, None]).T + bias.astype(np.float64)
    bound = 2.0 ** -20 * (np.abs(x).max(axis=1)[:, None] * (np.abs(v).sum(axis=1) * s)[None, :]) + 2.0 ** -22 * np.abs(want)
    assert np.all(np.abs(ys[0] - want) <= bound)


@pytest.mark.parametrize("bits", [4, 8])
def test_gemv_exact_on_integers_and_nonfinite_rows(bits):
    import torch
    aiq = binding()
    rng = np.random.default_rng(bits)
    qmax = 2 ** (bits - 1) - 1
    N, K, M = 1200, 2050, 4
    W = rng.integers(-qmax, qmax + 1, (N, K)).astype(np.float32)
    W[:, 0] = qmax
    x = rng.integers(-8, 9, (M, K)).astype(np.float32)
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, bits)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(to_dev(W), bits, packed, scales)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    aiq.aiq_qlinear(packed, scales, None, N, K, bits, to_dev(x), y)
    assert np.array_equal(y.cpu().numpy().astype(np.int64), x.astype(np.int64) @ W.astype(np.int64).T)
    x[2, 11] = np.inf
    x[3, 1999] = np.nan
    aiq.aiq_qlinear(packed, scales, None, N, K, bits, to_dev(x), y)
    got = y.cpu().numpy()
    assert np.isfinite(got[:2]).all() and not np.isfinite(got[2:]).any()


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("N,K,M", [(1030, 777, 2), (2999, 1000, 4), (40, 8190, 3), (2500, 4096, 1)])
def test_gemv_infinite_activations(bits, N, K, M):
    """An infinite activation gives an infinity of the code's sign, or a NaN where the code is zero or two infinities
    meet, as float32 products do; rows without one are as accurate as ever."""
    import torch
    aiq = binding()
    rng = np.random.default_rng(N + K + M + bits)
    W = rng.standard_normal((N, K)).astype(np.float32)
    x = rng.standard_normal((M, K)).astype(np.float32)
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, bits)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(to_dev(W), bits, packed, scales)
    v, s = O.quantize_rows(W, bits)
    w = v.astype(np.float64) * np.asarray(s, np.float64)[:, None]
    cases = [[(0, 5, np.inf)], [(0, K - 1, -np.inf), (M - 1, 600, np.inf)], [(M - 1, 3, np.inf), (M - 1, K - 2, np.inf)],
             [(M - 1, 1, -np.inf), (0, 2, np.nan)]]
    for case in cases:
        xi = x.copy()
        for m, k, val in case:
            xi[m, k] = val
        y = torch.zeros((M, N), dtype=torch.float32, device="cuda")
        aiq.aiq_qlinear(packed, scales, None, N, K, bits, to_dev(xi), y)
        got = y.cpu().numpy()
        fin = np.where(np.isfinite(xi), xi, 0).astype(np.float64)
        want = fin @ w.T
        bound = 2.0 ** -20 * np.abs(fin).max() * np.abs(w).sum(axis=1)[None, :] + 2.0 ** -22 * np.abs(want)
        with np.errstate(invalid="ignore"):
            for m, k, val in case:
                want[m] += float(val) * w[:, k]
            assert np.array_equal(np.isnan(got), np.isnan(want))
            inf = np.isinf(want)
            assert inf.any() or np.isnan(want).any()
            assert np.array_equal(np.isinf(got), inf) and np.array_equal(np.sign(got[inf]), np.sign(want[inf]))
            fine = np.isfinite(want)
            assert np.all(np.abs(got[fine] - want[fine]) <= np.broadcast_to(bound, want.shape)[fine])


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("N,K,M", [(1024, 1536, 1), (600, 4100, 2), (1200, 8192, 3), (3000, 777, 4)])
def test_gemv_fourth_digit(bits, N, K, M):
    """Activations of j 2^-26, |j| < 64, beside ones of 1 that meet zero weights: with the largest |x| of every slice at 1 the
    fourth digit counts 2^-26, so it alone holds them, and every sum is exact."""
    import torch
    aiq = binding()
    qmax = 2 ** (bits - 1) - 1
    g = torch.Generator(device="cuda").manual_seed(N + K)
    W = torch.randint(-qmax, qmax + 1, (N, K), generator=g, device="cuda").float()
    W[:, 1] = qmax
    W[:, ::64] = 0
    j = torch.randint(-63, 64, (M, K), generator=g, device="cuda")
    x = j.float() * 2.0 ** -26
    x[:, ::64] = 1.0
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, bits)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(W, bits, packed, scales)
    assert bool((scales == 1).all())
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    aiq.aiq_qlinear(packed, scales, None, N, K, bits, x, y)
    j[:, ::64] = 0
    want = j.double() @ W.double().T
    assert bool((want != 0).any()) and torch.equal(y.double() * 2.0 ** 26, want)


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("N,K,M", [(12000, 8192, 1), (12000, 8192, 3), (20003, 4100, 4), (20003, 4100, 2), (30001, 1030, 1)])
def test_gemv_many_units_per_block(bits, N, K, M):
    """More units than a block forms outputs of at a time (eight) and than its ring has slots: partial sums, slots and parities
    are used again.  Integers: every sum is exact."""
    import torch
    aiq = binding()
    qmax = 2 ** (bits - 1) - 1
    g = torch.Generator(device="cuda").manual_seed(N + K + M)
    W = torch.randint(-qmax, qmax + 1, (N, K), generator=g, device="cuda").float()
    W[:, 0] = qmax
    x = torch.randint(-8, 9, (M, K), generator=g, device="cuda").float()
    packed = torch.empty((N, aiq.aiq_packed_row_bytes(K, bits)), dtype=torch.uint8, device="cuda")
    scales = torch.empty(N, dtype=torch.float32, device="cuda")
    aiq.aiq_quantize_layer(W, bits, packed, scales)
    want = x.double() @ W.double().T
    for _ in range(2):
        y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
        aiq.aiq_qlinear(packed, scales, None, N, K, bits, x, y)
        assert torch.equal(y.double(), want)
