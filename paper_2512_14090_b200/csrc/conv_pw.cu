// Pointwise (1x1, stride 1) convolution on the tcgen05 tensor cores.
//
// A 1x1 convolution over split activations is a plain GEMM over all (padded) pixels.  A pixel is stored as
// [hi(Cs) | lo(Cs)] bfloat16, so it is one row of K2 = 2 Cs elements, and element k meets weight column k mod Cs:
//   D[128 pixels][Nt channels] += A[128][64 k] * B[Nt][64 k]^T   per chunk of 64 consecutive k of the pixel row.
// The layer is bound by its activation bytes (MobileNetV2: 4 (Cin + Cout) bytes and 2 Cin Cout operations per pixel),
// so the kernel is built to keep them moving:
//   - a block owns Nt output channels of one job, expands their packed weights to bfloat16 once, and then streams
//     pixel tiles (the kernel before expanded them again for every tile of 128 pixels);
//   - A chunks are dense whatever the channel count (hi and lo of a 32-channel pixel share one chunk);
//   - every epilogue warp works by itself on units of 32 pixels x 32 channels: accumulators -> scale, bias, residual,
//     activation -> split into hi / lo -> its own 4 KB of shared memory -> one TMA store of both halves.  No barrier
//     joins the warps, so the stores of one overlap the arithmetic of the others;
//   - two blocks per SM where their weights fit: one block's set-up and last tiles overlap the other's stream.
// Warps: 0 TMA producer, 1 MMA issuer, then EW epilogue warps.  Two accumulator buffers in tensor memory.
//
// STREAM variant, for layers with so many input channels that resident weights leave no room: the weights of 64
// channels travel through the ring beside the hi and lo chunk of the pixels, expanded by eight more warps.  A block
// can then hold more output channels, so that the pixels (the large tensor of such a layer) are read fewer times, and
// has more bytes in flight.
#include "tc_ptx.cuh"

#include <algorithm>
#include <type_traits>

namespace aiq {

namespace {

constexpr int kPrChunkBytes = 128 * 128;             // 128 pixels x 64 bfloat16
constexpr int kPrUnitBytes = 4096;                   // 32 pixels x 32 channels, hi then lo
constexpr int kPrMaxStages = 8;
constexpr int kPrExpWarps = 8;                       // weight expander warps of the STREAM variant

struct PrParams {
  int P;                    // padded pixels of the batch: B * (H + 2) * W
  int H, W;
  uint32_t w_magic, h_magic;   // 2^32 / W and 2^32 / (H + 2), rounded up (see div_by)
  int Cs_in, Cout, Cs_out, kpad;
  int Nt, n_ntiles;         // output channels per block, tiles of them
  int splits, tiles_per_cta, n_tiles;
  int act, n_stages, n_bufs;   // n_bufs: store buffers per epilogue warp, 1 or 2
  int tmem_cols;
  long long ver_pixels;     // pixels per version of the input slot
  int32_t* error_flag;
};

// shared memory: ring | store buffers | B (pieces x Cs_in / 8 planes of Nt rows x 16 bytes) | scale, bias | barriers
// A ring stage is one chunk of A, or in the STREAM variant the hi and the lo chunk of 64 channels and their weights.
__host__ __device__ inline int pr_stage_bytes(bool stream, int Nt, int pieces) {
  return stream ? 2 * kPrChunkBytes + pieces * Nt * 128 : kPrChunkBytes;
}
__host__ __device__ inline int pr_b_bytes(bool stream, int Nt, int Cs_in, int pieces) { return stream ? 0 : pieces * Nt * Cs_in * 2; }
__host__ __device__ inline int pr_smem_bytes(bool stream, int Nt, int Cs_in, int pieces, int ew, int stages, int bufs) {
  return stages * pr_stage_bytes(stream, Nt, pieces) + ew * bufs * kPrUnitBytes + pr_b_bytes(stream, Nt, Cs_in, pieces) + 2 * Nt * 4 +
         (3 * kPrMaxStages + 4) * 8 + 16;
}

// n / d with magic = floor(2^32 / d) + 1: the product is exact or one too high for any 32-bit n
__device__ __forceinline__ uint32_t div_by(uint32_t n, uint32_t d, uint32_t magic) {
  if (d == 1) return n;
  const uint32_t q = __umulhi(n, magic);
  return q * d > n ? q - 1 : q;
}

// 16 packed bytes of one weight row (32 bytes at 32 bits) -> bfloat16 planes: plane j of this row goes to dst + j * plane
template <int PIECES>
struct PrRaw { uint4 v[PIECES]; };
template <int PIECES>
__device__ __forceinline__ PrRaw<PIECES> pr_fetch(const uint8_t* __restrict__ src, int bits) {
  PrRaw<PIECES> r;
  r.v[0] = __ldg(reinterpret_cast<const uint4*>(src));
  if (PIECES == 2) r.v[PIECES - 1] = bits == 32 ? __ldg(reinterpret_cast<const uint4*>(src) + 1) : make_uint4(0u, 0u, 0u, 0u);
  return r;
}
template <int PIECES>
__device__ __forceinline__ void pr_expand(const PrRaw<PIECES>& raw, int bits, int n_planes, uint8_t* dst, int plane, int piece) {
  uint32_t o[4];
  if (PIECES == 1) {
    const uint4 r = raw.v[0];
    if (bits == 8) {
      expand8_bf16(make_uint2(r.x, r.y), 8, o);
      *reinterpret_cast<uint4*>(dst) = make_uint4(o[0], o[1], o[2], o[3]);
      if (n_planes > 1) {
        expand8_bf16(make_uint2(r.z, r.w), 8, o);
        *reinterpret_cast<uint4*>(dst + plane) = make_uint4(o[0], o[1], o[2], o[3]);
      }
    } else {
      const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j < n_planes) {
          expand8_bf16(make_uint2(w[j], 0u), 4, o);
          *reinterpret_cast<uint4*>(dst + j * plane) = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
  } else {
    // w = hi + lo, hi = bf16(w), lo = bf16(w - hi): exact for a half, within 2^-17 of a float32 weight
    float w[8];
    if (bits == 16) {
      const uint4 r = raw.v[0];
      const __half2* h2 = reinterpret_cast<const __half2*>(&r);
#pragma unroll
      for (int j = 0; j < 4; ++j) { const float2 f = __half22float2(h2[j]); w[2 * j] = f.x; w[2 * j + 1] = f.y; }
    } else {
      const uint4 a = raw.v[0], b = raw.v[PIECES - 1];
      w[0] = __uint_as_float(a.x); w[1] = __uint_as_float(a.y); w[2] = __uint_as_float(a.z); w[3] = __uint_as_float(a.w);
      w[4] = __uint_as_float(b.x); w[5] = __uint_as_float(b.y); w[6] = __uint_as_float(b.z); w[7] = __uint_as_float(b.w);
    }
    uint32_t l[4];
#pragma unroll
    for (int j = 0; j < 8; j += 2) split_pair(w[j], w[j + 1], o[j >> 1], l[j >> 1]);
    *reinterpret_cast<uint4*>(dst) = make_uint4(o[0], o[1], o[2], o[3]);
    *reinterpret_cast<uint4*>(dst + piece) = make_uint4(l[0], l[1], l[2], l[3]);
  }
}

// F32: the output is stored as floats (ConvGeom::out_f32) with the values that the hi / lo pairs would have had.
template <int EW, int PIECES, bool STREAM, bool F32>
__global__ void __launch_bounds__((2 + EW + (STREAM ? kPrExpWarps : 0)) * 32, EW == 12 && !STREAM ? 2 : 1)
conv_pw_kernel(const __grid_constant__ CUtensorMap in_map, const __grid_constant__ CUtensorMap out_map, PrParams p,
               const LayerJob* __restrict__ jobs) {
  constexpr int THREADS = (2 + EW + (STREAM ? kPrExpWarps : 0)) * 32;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  // blocks that read the same pixels (the channel tiles of a range) are neighbours: the later ones find them in L2
  const int ntile = (int)blockIdx.x % p.n_ntiles;
  const int split = ((int)blockIdx.x / p.n_ntiles) % p.splits;
  const LayerJob job = jobs[(int)blockIdx.x / (p.n_ntiles * p.splits)];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int Nt = p.Nt, n0 = ntile * Nt, stages = p.n_stages;
  const int stage_bytes = pr_stage_bytes(STREAM, Nt, PIECES);
  uint8_t* staging = smem + stages * stage_bytes;
  uint8_t* bsm = staging + EW * p.n_bufs * kPrUnitBytes;
  float* s_scale = reinterpret_cast<float*>(bsm + pr_b_bytes(STREAM, Nt, p.Cs_in, PIECES));
  float* s_bias = s_scale + Nt;
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_bias + Nt);
  const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8 * kPrMaxStages;
  const uint32_t bar_b_full = bar_empty + 8 * kPrMaxStages;     // STREAM: the expanders finished the weights of a stage
  const uint32_t bar_acc_full = bar_b_full + 8 * kPrMaxStages, bar_acc_empty = bar_acc_full + 16;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(bars + 3 * kPrMaxStages + 4);
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
  const int tile0 = split * p.tiles_per_cta, tile1 = min(tile0 + p.tiles_per_cta, p.n_tiles);
  const int K2 = 2 * p.Cs_in, n_chunks = STREAM ? (p.Cs_in + 63) >> 6 : (K2 + 63) >> 6;
  const int groups = (min(Nt, p.Cs_out - n0) + 31) >> 5;      // units of 32 channels of this block

  if (tid == 0) {
    for (int i = 0; i < stages; ++i) {
      mbar_init(bar_full + 8 * i, 1);
      mbar_init(bar_empty + 8 * i, 1);
      mbar_init(bar_b_full + 8 * i, kPrExpWarps);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_acc_full + 8 * i, 1);
      mbar_init(bar_acc_empty + 8 * i, EW);                    // one arrival per epilogue warp and tile
    }
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(s_tmem), (uint32_t)p.tmem_cols);
    tmem_relinquish();
  }
  for (int i = tid; i < Nt; i += THREADS) {
    const int n = n0 + i;
    s_scale[i] = n < p.Cout ? job.scale[n] : 0.f;              // padded channels come out as zeros
    s_bias[i] = n < p.Cout ? job.bias[n] : 0.f;
  }
  // weights -> B operand (K-major, no swizzle: plane of 8 channels, row, 16 bytes); consecutive threads take
  // consecutive rows, so their 16-byte stores are contiguous
  const int plane = Nt * 16;
  const int ppu = PIECES == 2 ? 1 : (job.bits == 8 ? 2 : 4);     // planes per 16 packed bytes (16 / 32 bits: one plane)
  const size_t wrow = (size_t)p.kpad * job.bits / 8;
  if (!STREAM) {
    const int piece = (p.Cs_in >> 3) * plane;
    const int uk = ((p.Cs_in >> 3) + ppu - 1) / ppu;
    const int n_units = Nt * uk;
#pragma unroll 4
    for (int u = tid; u < n_units; u += THREADS) {
      const int j = u / Nt, r = u - j * Nt, n = n0 + r;
      uint8_t* dst = bsm + (size_t)(j * ppu) * plane + r * 16;
      const int planes = min(ppu, (p.Cs_in >> 3) - j * ppu);
      if (n < p.Cout) {
        pr_expand<PIECES>(pr_fetch<PIECES>(job.w + (size_t)n * wrow + (size_t)j * ppu * job.bits, job.bits), job.bits, planes, dst, plane, piece);
      } else {
        for (int i = 0; i < planes; ++i) {
          *reinterpret_cast<uint4*>(dst + i * plane) = make_uint4(0u, 0u, 0u, 0u);
          if (PIECES == 2) *reinterpret_cast<uint4*>(dst + piece) = make_uint4(0u, 0u, 0u, 0u);
        }
      }
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // expanded weights -> visible to the MMA
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  chain_release();                                 // tensor memory is allocated (see launch_chained)
  const uint32_t tmem_base = *s_tmem;
  bool alive = true;

  if (warp == 0) {
    // ---- TMA producer -----------------------------------------------------------------------
    chain_wait();
    uint32_t stage = 0, phase = 0, issued = 0, issued_phase = 0;
    for (int tile = tile0; tile < tile1 && alive; ++tile) {
      const int pix = (int)(job.in_version * p.ver_pixels) + tile * 128;
      for (int c = 0; c < n_chunks; ++c) {
        alive = mbar_wait_warp(bar_empty + 8 * stage, phase ^ 1u, s_abort, p.error_flag);
        if (!alive) break;
        const uint32_t dst = smem_u32(smem) + stage * stage_bytes;
        if (STREAM) tma_fill2_2d(dst, &in_map, bar_full + 8 * stage, kPrChunkBytes, c * 64, c * 64 + p.Cs_in, pix);   // 64 channels: hi, lo
        else tma_fill_2d(dst, &in_map, bar_full + 8 * stage, kPrChunkBytes, c * 64, pix);
        issued |= 1u << stage;
        issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
        if (++stage == (uint32_t)stages) { stage = 0; phase ^= 1u; }
      }
    }
    for (int i = 0; i < stages; ++i)               // copies in flight must land before the CTA exits
      if (issued & (1u << i)) {
        const long long t0 = clock64();
        while (!mbar_try_wait(bar_full + 8 * i, (issued_phase >> i) & 1u) && clock64() - t0 < kWaitLimitCycles) {}
      }
  } else if (warp == 1) {
    // ---- MMA issuer: all 32 lanes converged, one elected lane issues (see umma_bf16) ------------
    // Nothing to do before: asleep instead of polling for the first chunk beside the kernel before, whose issue slots that took
    // (MobileNetV2-CIFAR, one image 279.5 -> 276.1 us; the other kernels of the chain gained nothing from it).
    chain_wait();
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(Nt >> 3) << 17) | ((128u >> 4) << 24);
    constexpr uint32_t A_HI = (uint32_t)(1024 >> 4) | (1u << 14) | (2u << 29);   // SBO 1024, version 1, 128-byte swizzle
    constexpr uint32_t B_HI = (uint32_t)(128 >> 4) | (1u << 14);                 // 128 bytes between groups of 8 rows; no swizzle
    const uint32_t b_lo0 = (smem_u32(bsm) >> 4) | ((uint32_t)Nt << 16);          // plane stride Nt * 16 bytes
    const uint32_t b_step = 2u * (uint32_t)Nt, b_piece = (uint32_t)(p.Cs_in >> 3) * (uint32_t)Nt;
    const int steps = p.Cs_in >> 4;                // 16-channel steps per half of the pixel
    uint32_t stage = 0, phase = 0;
    int it = 0;
    for (int tile = tile0; tile < tile1 && alive; ++tile, ++it) {
      const int buf = it & 1;
      alive = mbar_wait_warp(bar_acc_empty + 8 * buf, ((it >> 1) & 1) ^ 1u, s_abort, p.error_flag);
      if (!alive) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + (uint32_t)(buf * Nt);
      int ks = 0;                                  // step inside the half: weight column = 16 ks
      uint32_t accumulate = 0;
      for (int c = 0; c < n_chunks; ++c) {
        alive = mbar_wait_warp(bar_full + 8 * stage, phase, s_abort, p.error_flag);
        if (!alive) break;
        tc_fence_after();
        const uint32_t a_lo = ((smem_u32(smem) + stage * stage_bytes) >> 4) | (1u << 16);
        if constexpr (STREAM) {
          alive = mbar_wait_warp(bar_b_full + 8 * stage, phase, s_abort, p.error_flag);
          if (!alive) break;
          tc_fence_after();
          const uint32_t b_st = ((smem_u32(smem) + stage * stage_bytes + 2 * kPrChunkBytes) >> 4) | ((uint32_t)Nt << 16);
          const int kmax = min(4, steps - c * 4);
#pragma unroll
          for (int part = 0; part < 2; ++part)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              if (kk < kmax) {
                const uint64_t adesc = ((uint64_t)A_HI << 32) | (uint64_t)(a_lo + part * (kPrChunkBytes >> 4) + kk * 2);
                const uint32_t b_lo = b_st + (uint32_t)kk * b_step;
                umma_bf16(d_tmem, adesc, ((uint64_t)B_HI << 32) | (uint64_t)b_lo, idesc, accumulate);
                accumulate = 1;
                if (PIECES == 2) umma_bf16(d_tmem, adesc, ((uint64_t)B_HI << 32) | (uint64_t)(b_lo + 8u * (uint32_t)Nt), idesc, 1u);
              }
        } else {
        const int kmax = min(4, (K2 >> 4) - c * 4);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          if (kk < kmax) {
            const uint64_t adesc = ((uint64_t)A_HI << 32) | (uint64_t)(a_lo + kk * 2);
            const uint32_t b_lo = b_lo0 + (uint32_t)ks * b_step;
            umma_bf16(d_tmem, adesc, ((uint64_t)B_HI << 32) | (uint64_t)b_lo, idesc, accumulate);
            accumulate = 1;
            if (PIECES == 2) umma_bf16(d_tmem, adesc, ((uint64_t)B_HI << 32) | (uint64_t)(b_lo + b_piece), idesc, 1u);
            if (++ks == steps) ks = 0;
          }
        }
        }
        umma_commit(bar_empty + 8 * stage);
        if (++stage == (uint32_t)stages) { stage = 0; phase ^= 1u; }
      }
      if (alive) umma_commit(bar_acc_full + 8 * buf);
    }
  } else if (STREAM && warp >= 2 + EW) {
    // ---- STREAM weight expanders: packed rows -> the stage's B planes (8 of Nt rows per piece).  The packed words come
    // from L2 one chunk ahead, so that their latency hides behind the expansion and the wait for a free stage.
    constexpr int XT = kPrExpWarps * 32, UPT = 4;
    const int et = tid - (2 + EW) * 32;
    const int upr = 8 / ppu, n_units = Nt * upr;               // units of 16 packed bytes (32 at 32 bits) per chunk
    PrRaw<PIECES> cur[UPT], nxt[UPT];
    auto fetch = [&](int c, PrRaw<PIECES>* r) {
#pragma unroll
      for (int i = 0; i < UPT; ++i) {
        const int u = et + i * XT, j = u / Nt, n = n0 + u - j * Nt, pl = c * 8 + j * ppu;
        if (u < n_units && n < p.Cout && pl < (p.Cs_in >> 3)) {
          r[i] = pr_fetch<PIECES>(job.w + (size_t)n * wrow + (size_t)pl * job.bits, job.bits);
        } else {
#pragma unroll
          for (int k = 0; k < PIECES; ++k) r[i].v[k] = make_uint4(0u, 0u, 0u, 0u);
        }
      }
    };
    uint32_t stage = 0, phase = 0;
    fetch(0, cur);
    for (int tile = tile0; tile < tile1 && alive; ++tile) {
      for (int c = 0; c < n_chunks; ++c) {
        fetch(c + 1 < n_chunks ? c + 1 : 0, nxt);
        alive = mbar_wait_warp(bar_empty + 8 * stage, phase ^ 1u, s_abort, p.error_flag);
        if (!alive) break;
        uint8_t* bst = smem + stage * stage_bytes + 2 * kPrChunkBytes;
#pragma unroll
        for (int i = 0; i < UPT; ++i) {
          const int u = et + i * XT;
          if (u < n_units) {
            const int j = u / Nt, r = u - j * Nt;
            pr_expand<PIECES>(cur[i], job.bits, ppu, bst + (size_t)(j * ppu) * plane + r * 16, plane, 8 * plane);
          }
          cur[i] = nxt[i];
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> visible to the MMA
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_b_full + 8 * stage);
        if (++stage == (uint32_t)stages) { stage = 0; phase ^= 1u; }
      }
    }
  } else {
    // ---- epilogue: TMEM lanes 32q .. 32q+31 (pixels of the tile) belong to the warps with index mod 4 = q; the
    // HW warps of a quarter take the units (tile, group of 32 channels) in turn.  Every warp sees every tile, also
    // one it has no unit of: the parities it waits for would not be consecutive otherwise
    constexpr int HW = EW / 4;
    const int q = warp & 3, h = (warp - 2) >> 2;
    uint8_t* my_buf = staging + (size_t)(warp - 2) * p.n_bufs * kPrUnitBytes;
    const uint32_t my_buf_u32 = smem_u32(my_buf);
    // F32 rows are 128 bytes: 16-byte unit ^ (row mod 8); else two of 64 bytes: unit ^ (row / 2 mod 4)
    const uint32_t key = F32 ? (uint32_t)lane & 7u : (uint32_t)(lane >> 1) & 3u;
    int buf_idx = 0, g = h % groups, skip = h / groups;        // next group of this warp, tiles until then
    chain_wait();                                              // the residual and the output slot
    for (int tile = tile0, it = 0; tile < tile1 && alive; ++tile, ++it) {
      const int buf = it & 1;
      if (skip > 0) {                                          // nothing of this tile
        --skip;
        alive = mbar_wait_warp(bar_acc_full + 8 * buf, (it >> 1) & 1, s_abort, p.error_flag);
        if (lane == 0 && alive) mbar_arrive(bar_acc_empty + 8 * buf);
        continue;
      }
      const int pix0 = tile * 128 + q * 32, pix = pix0 + lane;
      const uint32_t row = div_by((uint32_t)pix, (uint32_t)p.W, p.w_magic);
      const int yp = (int)(row - div_by(row, (uint32_t)(p.H + 2), p.h_magic) * (uint32_t)(p.H + 2));
      const bool interior = pix < p.P && yp >= 1 && yp <= p.H, all_interior = __all_sync(0xffffffffu, interior);
      const int g0 = g;
      for (; g < groups; g += HW) {
      const int c0 = g * 32;
      const int nv = min(32, p.Cs_out - n0 - c0);              // stored channels of the unit: 32 or 16
      uint8_t* dst = my_buf + buf_idx * kPrUnitBytes + lane * (F32 ? 128 : 64);
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * Nt + c0);
      if (g == g0) {
        alive = mbar_wait_warp(bar_acc_full + 8 * buf, (it >> 1) & 1, s_abort, p.error_flag);
        if (!alive) break;
        tc_fence_after();
      }
      // the store that last read this buffer must be done with it
      if (lane == 0) {
        if (p.n_bufs == 2) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        else asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      }
      __syncwarp();
#pragma unroll 1
      for (int half = 0; half < 2 && half * 16 < nv; ++half) {   // 16 channels at a time: registers for more warps
        uint32_t v[16];
        tmem_ld16(taddr + 16 * half, v);
        uint4 rh[2], rl[2];
        if (!F32 && job.res) {                                 // (a layer with a residual never stores floats)
          const __nv_bfloat16* res = static_cast<const __nv_bfloat16*>(job.res) + (size_t)pix * (2 * p.Cs_out) + n0 + c0 + 16 * half;
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (interior) {
              rh[j] = ld_chain(reinterpret_cast<const uint4*>(res) + j);
              rl[j] = ld_chain(reinterpret_cast<const uint4*>(res + p.Cs_out) + j);
            } else {
              rh[j] = rl[j] = make_uint4(0u, 0u, 0u, 0u);
            }
        }
        tmem_ld_wait();
        if (g + HW >= groups && (half == 1 || nv <= 16)) {     // this warp's last accumulators of the tile
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_acc_empty + 8 * buf);
        }
        auto finish = [&](auto act, auto res) {
          if constexpr (F32) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int cc = c0 + 16 * half + 4 * j;
              ulonglong2 o = finish4<decltype(act)::value>(v + 4 * j, s_scale + cc, s_bias + cc);
              if (!all_interior && !interior) o = make_ulonglong2(0ull, 0ull);
              *reinterpret_cast<ulonglong2*>(dst + (((uint32_t)(4 * half + j) ^ key) << 4)) = o;
            }
            return;
          }
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            uint32_t hi[4], lo[4];
            const int cc = c0 + 16 * half + 8 * j;
            finish8<decltype(act)::value, decltype(res)::value>(v + 8 * j, s_scale + cc, s_bias + cc, rh[j], rl[j], hi, lo);
            if (!all_interior && !interior) {                  // border rows are zeros
#pragma unroll
              for (int i = 0; i < 4; ++i) hi[i] = lo[i] = 0u;
            }
            const uint32_t off = ((uint32_t)(2 * half + j) ^ key) << 4;
            *reinterpret_cast<uint4*>(dst + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4*>(dst + 2048 + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
          }
        };
        auto finish_act = [&](auto res) {
          if (p.act == AIQ_ACT_RELU6) finish(std::integral_constant<int, AIQ_ACT_RELU6>(), res);
          else if (p.act == AIQ_ACT_RELU) finish(std::integral_constant<int, AIQ_ACT_RELU>(), res);
          else finish(std::integral_constant<int, AIQ_ACT_NONE>(), res);
        };
        if (F32 || !job.res) finish_act(std::false_type()); else finish_act(std::true_type());
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        // channels past Cs_out and pixels past the slot's capacity are clipped by the tensor map
        if (pix0 < p.P)
          asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
                       ::"l"(reinterpret_cast<uint64_t>(&out_map)), "r"(my_buf_u32 + buf_idx * kPrUnitBytes), "r"(n0 + c0), "r"(pix0), "r"(0),
                       "r"(job.out_version)
                       : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
      if (++buf_idx == p.n_bufs) buf_idx = 0;
      }
      g -= groups;                                             // counted on into the next tiles
      while (g >= groups) { g -= groups; ++skip; }
    }
    // all stores must have left shared memory (and be complete) before the CTA retires
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    __syncwarp();
  }

  // ---- teardown -------------------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
}

// Launch shape: variant, channel tile, blocks per SM, ring depth, pixel splits.  Every channel tile but the last is a
// multiple of the 32 channels of a store unit.  Costs are in SM clocks: a tile of 128 pixels takes the longest of its
// MMAs ((128 + Nt) / 4 clocks per 16-channel step), its input (40 bytes per clock and SM, less where the ring holds fewer
// than about 1,600 clocks of that), its epilogue (about 12 clocks per channel) and, streamed, the expansion of its
// weights; a block adds a set-up that grows with the weights it expands.  Blocks fill the GPU in waves.
struct PrConfig { bool stream; int Nt, ew, stages, bufs, splits, tiles_per_cta, smem; };
// streamed: 0 / 1 restricts the search to that variant, -1 does not.
bool pr_search(const ConvGeom& g, int n_jobs, int pieces, const DeviceProps& props, int streamed, PrConfig* out) {
  const long long n_tiles = ((long long)g.B * (g.H + 2) * g.W + 127) / 128;   // of the nominal batch: may pass 2^31 pixels
  const double K2 = 2.0 * g.Cs_in;
  double best = 1e300;
  for (int nt = 32; nt <= 256; nt += 32) {
    const int Nt = g.Cs_out <= nt ? g.Cs_out : nt;             // the last candidate: one tile, any multiple of 16
    const int ntiles = (g.Cs_out + Nt - 1) / Nt;
    for (int variant = 0; variant < 4; ++variant) {
      // two blocks per SM, one with 12 or 24 epilogue warps, one with streamed weights
      const bool stream = variant == 3;
      const int occ = variant == 0 ? 2 : 1, ew = stream ? 8 : variant == 2 ? 24 : 12;
      if (streamed >= 0 && stream != (streamed == 1)) continue;
      if (occ == 2 && Nt > 128) continue;                      // tensor memory: 2 Nt columns per block
      if (stream && (Nt * 8 / (pieces == 2 ? 1 : 2) > 4 * kPrExpWarps * 32 || 2 * Nt > 512)) continue;
      const int limit = occ == 2 ? (props.smem_optin + 1024) / 2 - 1024 : props.smem_optin;
      auto need = [&](int st, int bf) { return pr_smem_bytes(stream, Nt, g.Cs_in, pieces, ew, st, bf) + 1024; };
      if (need(2, 1) > limit) continue;
      int st = 2, bf = 1;
      while (st < 4 && need(st + 1, bf) <= limit) ++st;
      if (need(st, 2) <= limit) bf = 2;
      while (st < kPrMaxStages && need(st + 1, bf) <= limit) ++st;
      const double in_flight = (double)occ * st * (stream ? 2 : 1) * kPrChunkBytes;
      const double c_mma = K2 / 16 * pieces * (128 + Nt) / 4.0;
      const double c_in = 128.0 * K2 * 2 / std::min(40.0, in_flight / 1600.0);
      const double c_epi = (ew < 24 && occ == 1 ? 18.0 : 12.0) * Nt;
      const double c_exp = stream ? Nt * (double)g.Cs_in * pieces * 0.06 : 0.0;
      const double tile = std::max(std::max(c_mma, c_in), std::max(c_epi, c_exp));
      const double setup = 3000.0 + (stream ? 0.0 : Nt * (double)g.Cs_in * pieces / 16.0);
      const int pairs = n_jobs * ntiles;
      for (int wave = 1; wave <= 5; ++wave) {
        long long splits = wave == 5 ? n_tiles : wave * occ * props.n_sms / pairs;
        if (splits < 1) splits = 1;
        if (splits > n_tiles) splits = n_tiles;
        const long long tpc = (n_tiles + splits - 1) / splits;
        splits = (n_tiles + tpc - 1) / tpc;
        const long long ctas = splits * pairs;
        const long long full = ctas / (occ * props.n_sms), rem = ctas - full * occ * props.n_sms;
        const double one = occ * tpc * tile + setup;
        const double cost = full * one + (rem > props.n_sms ? one : rem > 0 ? tpc * tile + setup : 0.0);
        if (cost < best * 0.999) {
          best = cost;
          *out = {stream, Nt, ew, st, bf, (int)splits, (int)tpc, need(st, bf)};
        }
        if (ctas >= n_tiles * pairs) break;
      }
    }
    if (Nt == g.Cs_out) break;
  }
  return best < 1e300;
}
bool pr_config(const ConvGeom& g, int n_jobs, int pieces, const DeviceProps& props, PrConfig* out) {
  static thread_local ConfigMemo<PrConfig, 8> memo;
  const int key[8] = {g.B, g.H, g.W, g.Cs_in, g.Cs_out, n_jobs, pieces, props.dev};
  return memo.get(key, out, [&](PrConfig* c) {
    // The variants add the hi and lo products of a pixel in different orders.  Which one a layer takes is decided at a
    // nominal batch, so that an image's result depends neither on the batch around it nor on the number of jobs.
    ConvGeom nominal = g;
    nominal.B = 256;
    PrConfig v;
    return pr_search(nominal, 1, pieces, props, -1, &v) && pr_search(g, n_jobs, pieces, props, v.stream ? 1 : 0, c);
  });
}

template <int EW, int PIECES, bool STREAM, bool F32>
aiq_status_t launch_pr(const LaunchScope& scope, const DeviceProps& props, const PrConfig& c, const PrParams& p, const CUtensorMap& m,
                       const CUtensorMap& mo, const LayerJob* jobs_dev, int n_jobs, cudaStream_t s) {
  AIQ_ENSURE_DYNAMIC_SMEM((conv_pw_kernel<EW, PIECES, STREAM, F32>), props.smem_optin);
  AIQ_CUDA_TRY(launch_chained(scope.chain, conv_pw_kernel<EW, PIECES, STREAM, F32>, dim3((unsigned)(n_jobs * p.splits * p.n_ntiles)),
                              dim3((2 + EW + (STREAM ? kPrExpWarps : 0)) * 32), c.smem, s, m, mo, p, jobs_dev));
  return AIQ_OK;
}

}  // namespace

bool conv_pw_eligible(const ConvGeom& g) {
  if (g.in_is_nchw || g.act_format != ACT_SPLIT) return false;
  return g.ks == 1 && g.pad == 0 && g.stride == 1 && g.Cin % 8 == 0 && g.Cin >= 16;
}

aiq_status_t conv_pw_encode_maps(const ConvGeom& g, const void* in_slot, int in_versions, const void* out_slot, int out_versions,
                                 int batch_capacity, void* maps_out /* 2 x 128 bytes */) {
  EncodeTiledFn enc = encode_tiled_fn();
  if (!enc) return set_error(AIQ_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
  CUtensorMap* maps = static_cast<CUtensorMap*>(maps_out);
  const cuuint64_t pixels = (cuuint64_t)batch_capacity * (g.H + 2) * g.W;
  const cuuint32_t one[4] = {1, 1, 1, 1};
  {
    // (element of the pixel row [hi | lo], pixel over all versions)
    cuuint64_t dims[2] = {2ull * g.Cs_in, pixels * in_versions};
    cuuint64_t strides[1] = {4ull * g.Cs_in};
    cuuint32_t box[2] = {64u, 128u};
    const CUresult r = enc(&maps[0], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(in_slot), dims, strides, box, one,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(AIQ_ERR_CUDA, "cuTensorMapEncodeTiled (pointwise) failed with code %d", (int)r);
  }
  {
    // (channel within a half, pixel of a version, hi | lo, version)
    cuuint64_t dims[4] = {(cuuint64_t)g.Cs_out, pixels, 2, (cuuint64_t)out_versions};
    cuuint64_t strides[3] = {4ull * g.Cs_out, 2ull * g.Cs_out, 4ull * g.Cs_out * pixels};
    cuuint32_t box[4] = {32u, 32u, 2u, 1u};
    if (g.out_f32) { dims[2] = 1; strides[1] = 4ull * g.Cs_out; box[2] = 1; }       // 32 channels: 128 bytes of floats
    const CUresult r = enc(&maps[1], g.out_f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4,
                           const_cast<void*>(out_slot), dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           g.out_f32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(AIQ_ERR_CUDA, "cuTensorMapEncodeTiled (pointwise store) failed with code %d", (int)r);
  }
  return AIQ_OK;
}

aiq_status_t launch_conv_pw(const ConvGeom& g, const void* maps, const LayerJob* jobs_dev, int n_jobs, int batch_capacity,
                            int32_t* error_flag, double weight_bytes, int weight_bits, cudaStream_t s) {
  DeviceProps props;
  if (aiq_status_t st = current_device_props(&props)) return st;
  const int pieces = weight_bits > 8 ? 2 : 1;
  PrConfig c = {};
  if (!pr_config(g, n_jobs, pieces, props, &c)) return set_error(AIQ_ERR_SHAPE, "conv_pw: no launch shape fits shared memory");
  PrParams p = {};
  p.P = g.B * (g.H + 2) * g.W; p.H = g.H; p.W = g.W;
  p.w_magic = (uint32_t)(0x100000000ull / (uint32_t)g.W + 1); p.h_magic = (uint32_t)(0x100000000ull / (uint32_t)(g.H + 2) + 1);
  p.Cs_in = g.Cs_in; p.Cout = g.Cout; p.Cs_out = g.Cs_out; p.kpad = padded_k(g.Cin);
  p.Nt = c.Nt; p.n_ntiles = (g.Cs_out + c.Nt - 1) / c.Nt;
  p.splits = c.splits; p.tiles_per_cta = c.tiles_per_cta; p.n_tiles = (p.P + 127) / 128;
  p.act = g.act; p.n_stages = c.stages; p.n_bufs = c.bufs;
  p.tmem_cols = 32;
  while (p.tmem_cols < 2 * p.Nt) p.tmem_cols <<= 1;
  p.ver_pixels = (long long)batch_capacity * (g.H + 2) * g.W;
  p.error_flag = error_flag;
  const CUtensorMap* m = static_cast<const CUtensorMap*>(maps);
  LaunchScope scope(AIQ_KERNEL_CONV_TC, s, 2.0 * g.B * g.Ho * g.Wo * g.Cout * (double)g.Cin * n_jobs,
                    weight_bytes + 4.0 * n_jobs * ((double)g.B * g.Cin * g.H * g.W + (double)g.B * g.Ho * g.Wo * g.Cout));
#define AIQ_PW(EW_, P_, S_) (g.out_f32 ? launch_pr<EW_, P_, S_, true>(scope, props, c, p, m[0], m[1], jobs_dev, n_jobs, s) \
                                       : launch_pr<EW_, P_, S_, false>(scope, props, c, p, m[0], m[1], jobs_dev, n_jobs, s))
  aiq_status_t st;
  if (c.stream) st = pieces == 1 ? AIQ_PW(8, 1, true) : AIQ_PW(8, 2, true);
  else if (c.ew == 12) st = pieces == 1 ? AIQ_PW(12, 1, false) : AIQ_PW(12, 2, false);
  else st = pieces == 1 ? AIQ_PW(24, 1, false) : AIQ_PW(24, 2, false);
#undef AIQ_PW
  if (st != AIQ_OK) return st;
  AIQ_LAUNCH_CHECK("conv_pw");
  return AIQ_OK;
}

}  // namespace aiq
