// Quantized linear layer at batch sizes where it is a dense contraction (M >= 9), on the
// tcgen05 tensor cores.  Included by conv_tc.cu (shares its PTX wrappers); not a stand-alone
// translation unit.
//
//   y[m][n] = s_n * sum_k code[n][k] * x[m][k] + bias[n]
//
// The weight matrix is the M operand of the MMA (128 output channels per CTA) and the batch
// is its N operand (up to 256 batch rows per CTA), so the packed weights - the bytes that
// bound the layer at small batch - are read from memory exactly once:
//   D[128 n][Mt m] += A[128 n][64 k] * B[Mt m][64 k]^T     per chunk of 64 k.
// 4, 8 and 16 bits: both operands are halves.  A = the integer codes as halves (exact), or the
// stored halves themselves: a TMA tile of 16-bit weights is the A operand as it lands.  B = the
// activations times a power of two per batch row that brings the row's largest |x| into [2^14,
// 2^15), as the sum of two halves (hi + lo: 22 bits of each value - 20 at 8 bits and long sums, see the
// pre-pass - or 2^-39 of the row's maximum where that is coarser); the power of two is taken out of the sums again, exactly.
// 32 bits: both operands are bfloat16 sums hi + lo (a float32 weight has no bounded exponent).
// A pre-pass writes the two planes of x into the caller's workspace; the main kernel starts under programmatic dependent launch, so its
// weight prefetch overlaps the pre-pass.
//   warp 0      TMA producer of the B tiles (Mt rows x 64 k, 128-byte swizzle)
//   warp 1      MMA issuer (converged warp, elected lane)
//   warps 2-5   epilogue: sums TMEM -> shared memory.  Before that, warp 2
//               is the TMA producer of the packed weights: 128 rows x 128 bytes at a time, so that
//               every row is read from memory in whole 128-byte lines, running as far ahead of
//               the MMAs as its own ring allows
//   warps 6-21  (4, 8, 32 bits) weight expanders: packed tile in shared memory -> A tile in tensor
//               memory, so that the expanded weights cost shared memory neither room nor bandwidth
// A CTA owns one (128-channel block, K split, 256-row batch block) and runs once.  The parts of a split K
// range meet in y by atomics (it is zeroed by the pre-pass); two neighbours of a large batch are a cluster and first add
// up, each half of the batch rows, over both shared memories.
// Bound at 16 rows by the weight stream (16 bits: 5.9 TB/s in the steady state) or by one MMA warp's 64 k steps (4 / 8 bits),
// plus 7 us for two launches, the pre-pass and the first loads; at 256 rows by the activations every CTA reads from L2 (64 KB
// per 64 k: 1,180 cycles a step, 1,024 of them MMA time).
// On the device, before (bfloat16, expanded into shared memory, atomics from the accumulators) and now: 8192 x 8192, 16
// rows: 4 bits 53 -> 26 us, 8 bits 47 -> 26, 16 bits 51 -> 31, 32 bits 77 -> 50; 256 rows: 8 bits 72 -> 57, 16 bits 123 ->
// 66, 32 bits 153 -> 107; 4096 x 4096, 16 bits, 16 rows 18 -> 11.4.  Steps of it: halves instead of bfloat16 pairs (16
// bits: half the MMAs, no expansion), A in tensor memory (-2 us), one copy per step issued by a converged warp (-3 us).
#pragma once

namespace aiq {
namespace {

constexpr int kQtExpWarps = 16;                      // weight expander warps: four (128 rows) on each chunk
constexpr int kQtAStages = kQtExpWarps / 4;          // A tiles in flight, one per group of expander warps
constexpr int kQtChunk = 64;                         // k per stage
constexpr int kQtWTile = 128 * 128;                  // 16 KB: 128 channels x 128 packed bytes
constexpr int kQtACols = kQtChunk / 2;               // tensor memory columns of an A tile of 16-bit values
constexpr int kQtMaxWStages = 12;
constexpr int kQtMaxBStages = 24;

template <int BITS>
struct QtKind {
  static constexpr bool DIRECT = BITS == 16;         // the packed tile is the A operand
  static constexpr int PIECES = BITS == 32 ? 2 : 1;  // 16-bit pieces per weight
  static constexpr int CPW = BITS == 4 ? 4 : BITS == 8 ? 2 : 1;   // chunks per packed tile (128 bytes of a row)
  static constexpr int TPC = BITS == 32 ? 2 : 1;     // packed tiles per chunk
  static constexpr int A_STAGES = DIRECT ? 0 : kQtAStages;
  static constexpr int A_COLS = A_STAGES * PIECES * kQtACols;
  static constexpr int THREADS = (6 + kQtExpWarps) * 32;   // DIRECT: the expander warps only take part in the last step
};

struct QtParams {
  int N, K, M;
  int Mt;                   // batch rows per CTA tile (multiple of 16, <= 256)
  int m_block;              // batch rows per blockIdx.z: 256 or 128
  int n_chunks;             // ceil(K / 64)
  int chunks_per_split;
  int cluster;              // K splits that are one cluster (blockIdx.x = 128-channel block * cluster + rank)
  int atomic;               // several clusters (blockIdx.y) per block of y: it is zeroed by the pre-pass
  int b_stages;             // activation units in flight (a ring of its own: TMA loads with a long round trip)
  int w_stages;             // packed weight tiles in flight
  int stack;                // 1: hi and lo rows of B are one unit, an operand of N = 2 Mt (Mt <= 128); 0: a unit each
  int a_col;                // first tensor memory column of the A tiles (behind the sums)
  int tmem_cols;
  int32_t* error_flag;      // optional
};

__host__ __device__ inline int qt_b_unit_bytes(int Mt, int stack) { return (stack ? 2 : 1) * Mt * kQtChunk * 2; }
// the rings; afterwards the sums of the tile, [batch row][128 channels]
__host__ __device__ inline int qt_ring_bytes(int Mt, int stack, int b_stages, int w_stages) {
  const int rings = b_stages * qt_b_unit_bytes(Mt, stack) + w_stages * kQtWTile, sums = Mt * 128 * 4;
  return rings > sums ? rings : sums;
}
inline int qt_smem_bytes(int a_stages, int Mt, int stack, int b_stages, int w_stages) {
  return qt_ring_bytes(Mt, stack, b_stages, w_stages) + (2 * a_stages + 2 * b_stages + 2 * w_stages + 1) * 8 + 24 + (Mt + 256) * 4;
}

// x [M][K] float32 -> planes hi [M][K], lo [M][K]; one block per batch row.
//   HALF: x 2^-e = hi + lo in halves, 2^e in down[row] (PERM4: each 8 k in the order 0 4 1 5 2 6 3 7, in which the expanders
//   unpack 4-bit codes); else hi + lo in bfloat16 (2^-17 of each value), down[row] = 1.
//   HI8: hi keeps 8 of its 11 bits and lo takes the rest (2^-20 of each value instead of 2^-22).  The tensor cores drop what
//   a product has below the accumulator's last bit; with 8-bit codes and long sums that costs more than it gains: error
//   against 64 bits at 8192 x 8192, 8 bits, 16 / 256 rows 3.6e-6 / 8.4e-6 with 11 bits, 1.0e-6 / 5.9e-6 with 8 (bfloat16
//   pairs: 2.6e-6 / 6.4e-6); 4096 x 4096, 16 rows 7.0e-7 and 3.6e-7; 2048 x 2048, short sums, 1.7e-7 and 3.2e-7.
// Optionally y = 0 (the split-K partial sums are added atomically); the status word starts at 0.
template <bool HALF, bool PERM4, bool HI8>
__global__ void __launch_bounds__(512)
qlinear_split_x_kernel(const float* __restrict__ x, int K, int M, uint16_t* __restrict__ planes, float* __restrict__ down,
                       float* __restrict__ y, long long y_elems, int32_t* __restrict__ status) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ int s_max[16];
  const int row = blockIdx.x, tid = threadIdx.x;
  if (row == 0 && tid == 0 && status) *status = 0;
  const float* xr = x + (size_t)row * K;
  float up = 1.f;
  if (HALF) {
    int top = 0;
    for (int k = tid * 4; k < K; k += 512 * 4) {
      const float4 v = *reinterpret_cast<const float4*>(xr + k);
      top = max(max(top, max(__float_as_int(v.x) & 0x7FFFFFFF, __float_as_int(v.y) & 0x7FFFFFFF)),
                max(__float_as_int(v.z) & 0x7FFFFFFF, __float_as_int(v.w) & 0x7FFFFFFF));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    if ((tid & 31) == 0) s_max[tid >> 5] = top;
    __syncthreads();
    top = s_max[tid & 15];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    const float xmax = __int_as_float(top);
    int e = 15;
    if (top != 0 && top < 0x7F800000) frexpf(xmax, &e);          // xmax = f 2^e, f in [0.5, 1)
    const int sh = min(15 - e, 126);
    up = ldexpf(1.f, sh);
    if (tid == 0) down[row] = ldexpf(1.f, -sh);
  } else if (tid == 0) {
    down[row] = 1.f;
  }
  uint16_t* hi_row = planes + (size_t)row * K;
  uint16_t* lo_row = hi_row + (size_t)M * K;
  for (int k = tid * 8; k < K; k += 512 * 8) {                   // K is a multiple of 8
    const float4 v0 = *reinterpret_cast<const float4*>(xr + k), v1 = *reinterpret_cast<const float4*>(xr + k + 4);
    uint32_t h[4], l[4];
    if (HALF) {
      float f[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float a = f[PERM4 ? j : 2 * j] * up, b = f[PERM4 ? j + 4 : 2 * j + 1] * up;
        float ha = a, hb = b;
        if (HI8) {                                               // the leading 8 bits, rounded to nearest
          const float ta = __fmul_rn(a, 65537.f), tb = __fmul_rn(b, 65537.f);
          ha = __fsub_rn(ta, __fsub_rn(ta, a));
          hb = __fsub_rn(tb, __fsub_rn(tb, b));
        }
        const __half2 hh = __floats2half2_rn(ha, hb);
        const float2 back = __half22float2(hh);
        const __half2 ll = __floats2half2_rn(a - back.x, b - back.y);
        h[j] = *reinterpret_cast<const uint32_t*>(&hh);
        l[j] = *reinterpret_cast<const uint32_t*>(&ll);
      }
    } else {
      split_pair(v0.x, v0.y, h[0], l[0]); split_pair(v0.z, v0.w, h[1], l[1]);
      split_pair(v1.x, v1.y, h[2], l[2]); split_pair(v1.z, v1.w, h[3], l[3]);
    }
    *reinterpret_cast<uint4*>(hi_row + k) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(lo_row + k) = make_uint4(l[0], l[1], l[2], l[3]);
  }
  const long long step = (long long)gridDim.x * 512;
  for (long long i = (long long)row * 512 + tid; i < y_elems; i += step) y[i] = 0.f;
}

__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
// eight codes -> eight halves (a code plus 1024 and its offset is a half's mantissa); 4 bits in the order 0 4 1 5 2 6 3 7
template <int BITS>
__device__ __forceinline__ void expand8_half(uint2 raw, uint32_t* o) {
  const uint32_t off = BITS == 4 ? 0x64086408u : 0x64806480u;    // 1024 + 8, 1024 + 128
  const __half2 off2 = *reinterpret_cast<const __half2*>(&off);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint32_t u;
    if (BITS == 4) u = ((raw.x >> (4 * j)) & 0x000F000Fu) ^ 0x64086408u;
    else u = __byte_perm((j < 2 ? raw.x : raw.y) ^ 0x80808080u, 0x64646464u, (j & 1) ? 0x4342 : 0x4140);
    const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&u), off2);
    o[j] = *reinterpret_cast<const uint32_t*>(&r);
  }
}

template <int BITS>
__global__ void __launch_bounds__(QtKind<BITS>::THREADS, 1)
qlinear_tc_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap w_map, QtParams p,
                  const float* __restrict__ scale, const float* __restrict__ bias, const float* down, float* __restrict__ y) {
  using T = QtKind<BITS>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = blockIdx.x % p.cluster, split = blockIdx.y * p.cluster + rank;
  const int n0 = (int)(blockIdx.x / p.cluster) * 128, m0 = blockIdx.z * p.m_block;
  constexpr int stages = T::A_STAGES;
  const int b_stages = p.b_stages, Mt = p.Mt, w_stages = p.w_stages;
  const int b_unit = qt_b_unit_bytes(Mt, p.stack), units = p.stack ? 1 : 2;
  const int c_begin = min(p.n_chunks, split * p.chunks_per_split);
  const int c_end = min(p.n_chunks, c_begin + p.chunks_per_split);

  // shared memory: B ring | packed weight ring (then the sums) | barriers (every tile 1024-aligned) | row factors, scales, biases
  uint8_t* bring = smem;
  uint8_t* wring = bring + b_stages * b_unit;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + qt_ring_bytes(Mt, p.stack, b_stages, w_stages));
  const uint32_t bar_a_full = smem_u32(bars);               // expanders finished an A tile
  const uint32_t bar_a_empty = bar_a_full + 8 * stages;     // the MMAs that read an A tile have retired
  const uint32_t bar_b_full = bar_a_empty + 8 * stages;     // TMA bytes of an activation unit have landed
  const uint32_t bar_b_empty = bar_b_full + 8 * b_stages;   // the MMAs that read it have retired
  const uint32_t bar_w_full = bar_b_empty + 8 * b_stages;   // a packed weight tile has landed
  const uint32_t bar_w_empty = bar_w_full + 8 * w_stages;   // the expanders (16 bits: the MMAs) are done with it
  const uint32_t bar_acc_full = bar_w_empty + 8 * w_stages;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(bars + 2 * stages + 2 * b_stages + 2 * w_stages + 1);
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
  float* s_down = reinterpret_cast<float*>(s_tmem + 6);   // 16-byte aligned: an odd number of barriers lies before s_tmem
  float* s_scale = s_down + Mt;                             // [128], then the biases

  if (tid == 0) {
    for (int i = 0; i < stages; ++i) {
      mbar_init(bar_a_full + 8 * i, 4);             // one arrival per expander warp of the chunk
      mbar_init(bar_a_empty + 8 * i, 1);
    }
    for (int i = 0; i < b_stages; ++i) {
      mbar_init(bar_b_full + 8 * i, 1);
      mbar_init(bar_b_empty + 8 * i, 1);
    }
    for (int i = 0; i < w_stages; ++i) {
      mbar_init(bar_w_full + 8 * i, 1);
      mbar_init(bar_w_empty + 8 * i, T::DIRECT ? 1 : 4 * T::CPW);
    }
    mbar_init(bar_acc_full, 1);
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (warp == 1) {
    tmem_alloc(smem_u32(s_tmem), (uint32_t)p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  bool alive = true;

  if (warp == 0) {
    // ---- TMA producer of the activation units (the planes are written by the pre-pass) -----------
    // A unit is one copy: the box holds both planes when hi and lo are one operand.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    uint32_t stage = 0, phase = 0, issued = 0, issued_phase = 0, dst = smem_u32(bring), c0 = (uint32_t)c_begin * kQtChunk, plane = 0;
    for (int i = (c_end - c_begin) * units; i > 0; --i) {
      alive = mbar_wait_warp(bar_b_empty + 8 * stage, phase ^ 1u, s_abort, p.error_flag);
      if (!alive) break;
      tma_fill_3d(dst, &x_map, bar_b_full + 8 * stage, (uint32_t)b_unit, (int)c0, m0, (int)plane);
      issued |= 1u << stage;
      issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
      dst += b_unit;
      if (++stage == (uint32_t)b_stages) { stage = 0; phase ^= 1u; dst = smem_u32(bring); }
      if (p.stack || plane) { c0 += kQtChunk; plane = 0; } else plane = 1;
    }
    for (int i = 0; i < b_stages; ++i)             // copies in flight must land before the CTA exits
      if (issued & (1u << i)) {
        const long long t0 = clock64();
        while (!mbar_try_wait(bar_b_full + 8 * i, (issued_phase >> i) & 1u) && clock64() - t0 < kWaitLimitCycles) {}
      }
  } else if (!T::DIRECT && warp >= 6) {
    // ---- weight expanders: packed tile -> A tile in tensor memory (128 lanes x 32 columns) ---------
    // The packed tile holds 128 bytes of each of the 128 rows, 16-byte units XOR-swizzled by the row
    // (the tensor map's 128-byte swizzle): a warp reads one unit of 32 rows at a time, free of bank
    // conflicts, and writes the quarter of the lanes that is its own.  Four warps make a group; the
    // groups work on different chunks, since a chunk is a chain of waits, loads and stores.  (Every
    // group meets every phase of the barriers it waits on: see the ring sizes in the launcher.)
    const int group = (warp - 6) >> 2, quarter = warp & 3;
    const uint32_t r7 = lane & 7, wrow = smem_u32(wring) + (uint32_t)(quarter * 32 + lane) * 128;
    const uint32_t atile = tmem_base + p.a_col + group * T::PIECES * kQtACols + ((uint32_t)(quarter * 32) << 16);
    const int n = c_end - c_begin;
    uint32_t phase = 0;
    for (int idx = group; idx < n && alive; idx += kQtAStages, phase ^= 1u) {
      uint32_t tile_stage[T::TPC];
#pragma unroll
      for (int t = 0; t < T::TPC; ++t) {
        const uint32_t ti = (uint32_t)(idx / T::CPW * T::TPC + t), round = ti / (uint32_t)w_stages;
        tile_stage[t] = ti - round * w_stages;
        alive = alive && mbar_wait_warp(bar_w_full + 8 * tile_stage[t], round & 1u, s_abort, p.error_flag);
      }
      if (!alive) break;
      if (BITS == 32) {                                         // 32 k of a row per packed tile
        alive = mbar_wait_warp(bar_a_empty + 8 * group, phase ^ 1u, s_abort, p.error_flag);
        if (!alive) break;
        tc_fence_after();
#pragma unroll
        for (int t = 0; t < T::TPC; ++t) {
          const uint32_t src = wrow + tile_stage[t] * kQtWTile;
          uint32_t h[16], l[16];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint4 r = lds128(src + ((j ^ r7) << 4));
            split_pair(__uint_as_float(r.x), __uint_as_float(r.y), h[2 * j], l[2 * j]);
            split_pair(__uint_as_float(r.z), __uint_as_float(r.w), h[2 * j + 1], l[2 * j + 1]);
          }
          tmem_st16(atile + t * 16, h);
          tmem_st16(atile + kQtACols + t * 16, l);
        }
      } else {
        const uint32_t src = wrow + tile_stage[0] * kQtWTile, u0 = idx % T::CPW * (BITS / 2);
        uint4 raw[BITS / 2];
#pragma unroll
        for (int j = 0; j < BITS / 2; ++j) raw[j] = lds128(src + (((u0 + j) ^ r7) << 4));
        alive = mbar_wait_warp(bar_a_empty + 8 * group, phase ^ 1u, s_abort, p.error_flag);
        if (!alive) break;
        tc_fence_after();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t v[16];
#pragma unroll
          for (int j = 0; j < 4; ++j) {                         // 8 weights each
            const uint4 r = raw[BITS == 4 ? half : half * 2 + (j >> 1)];
            if (BITS == 4) expand8_half<4>(make_uint2(j == 0 ? r.x : j == 1 ? r.y : j == 2 ? r.z : r.w, 0u), v + 4 * j);
            else expand8_half<8>((j & 1) ? make_uint2(r.z, r.w) : make_uint2(r.x, r.y), v + 4 * j);
          }
          tmem_st16(atile + half * 16, v);
        }
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      // The packed tiles are released only now, after their words have been used: every lane's loads
      // have then returned.  (Released right after the loads were issued, a refill by the TMA reached
      // shared memory before the last loads of a warp had read it: wrong weights in 2-4 adjacent rows,
      // a few times per million outputs.)
      if (lane == 0) {
        for (int t = 0; t < T::TPC; ++t) mbar_arrive(bar_w_empty + 8 * tile_stage[t]);
        mbar_arrive(bar_a_full + 8 * group);
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer: all 32 lanes converged, one elected lane issues (see umma_bf16) ------------
    // Up to Mt = 128 the hi and the lo tile (adjacent in shared memory) are one B operand of
    // 2 Mt rows: half as many MMAs, the two partial products land in separate accumulator
    // columns and are added in the epilogue.  Small MMAs cost more to issue than to execute.
    // Above that each is a unit of its own, freed and refilled by itself.
    const int mma_n = p.stack ? 2 * Mt : Mt;
    const uint32_t types = BITS == 32 ? (1u << 7) | (1u << 10) : 0u;   // bfloat16 : half
    const uint32_t idesc = (1u << 4) | types | ((uint32_t)(mma_n >> 3) << 17) | ((128u >> 4) << 24);
    constexpr uint32_t DESC_HI = (uint32_t)(1024 >> 4) | (1u << 14) | (2u << 29);   // SBO 1024, version 1, 128-byte swizzle
    constexpr uint32_t LBO_FIELD = 1u << 16;
    const uint32_t a_full = T::DIRECT ? bar_w_full : bar_a_full, a_empty = T::DIRECT ? bar_w_empty : bar_a_empty;
    const uint32_t a_stages = T::DIRECT ? w_stages : stages;
    // One step = one activation unit.  Whether the next step's operands are there is asked before this step's MMAs are issued.
    uint32_t stage = 0, phase = 0, bstage = 0, bphase = 0, accumulate = 0;
    bool first_unit = true, ready = false;
    for (int i = (c_end - c_begin) * units; i > 0; --i) {
      if (!ready) {
        alive = mbar_wait_warp(a_full + 8 * stage, phase, s_abort, p.error_flag) &&
                mbar_wait_warp(bar_b_full + 8 * bstage, bphase, s_abort, p.error_flag);
        if (!alive) break;
      }
      tc_fence_after();
      const uint32_t a_done = a_empty + 8 * stage, a_tile = stage;
      const uint32_t b_lo = ((smem_u32(bring) + bstage * b_unit) >> 4) | LBO_FIELD, b_done = bar_b_empty + 8 * bstage;
      const bool last_unit = p.stack || !first_unit;
      if (last_unit && ++stage == a_stages) { stage = 0; phase ^= 1u; }
      if (++bstage == (uint32_t)b_stages) { bstage = 0; bphase ^= 1u; }
      first_unit = last_unit;
      ready = mbar_test(a_full + 8 * stage, phase) & mbar_test(bar_b_full + 8 * bstage, bphase);
      const uint64_t bdesc = ((uint64_t)DESC_HI << 32) | (uint64_t)b_lo;
      if (T::DIRECT) {
        umma_k64(tmem_base, ((uint64_t)DESC_HI << 32) | (uint64_t)(((smem_u32(wring) + a_tile * kQtWTile) >> 4) | LBO_FIELD), bdesc, idesc, accumulate);
      } else {
        const uint32_t a_tmem = tmem_base + p.a_col + a_tile * T::PIECES * kQtACols;
        umma_k64_ta(tmem_base, a_tmem, bdesc, idesc, accumulate);
        if (T::PIECES == 2) umma_k64_ta(tmem_base, a_tmem + kQtACols, bdesc, idesc, 1u);
      }
      accumulate = 1;
      umma_commit(b_done);
      if (last_unit) umma_commit(a_done);
      ready = __all_sync(0xffffffffu, ready);
    }
    if (alive) umma_commit(bar_acc_full);
  } else {
    // ---- epilogue: warp q owns TMEM lanes 32q .. 32q+31 = output channels n0 + 32q + lane ---------
    const int q = warp & 3;
    if (warp == 2) {
      // packed weight tiles: independent of the pre-pass, requested as early as the ring allows
      uint32_t wst = 0, wphase = 0, w_issued = 0, w_issued_phase = 0;
      int byte = c_begin * kQtChunk * BITS / 8;
      bool ok = true;
      for (int i = (c_end - c_begin + T::CPW - 1) / T::CPW * T::TPC; i > 0; --i) {   // 128 bytes of 128 rows
        ok = mbar_wait_warp(bar_w_empty + 8 * wst, wphase ^ 1u, s_abort, p.error_flag);
        if (!ok) break;
        tma_fill_2d(smem_u32(wring) + wst * kQtWTile, &w_map, bar_w_full + 8 * wst, kQtWTile, byte, n0);
        w_issued |= 1u << wst;
        w_issued_phase = (w_issued_phase & ~(1u << wst)) | (wphase << wst);
        byte += 128;
        if (++wst == (uint32_t)w_stages) { wst = 0; wphase ^= 1u; }
      }
      if (!ok)                                     // copies in flight must land before the CTA exits
        for (int i = 0; i < w_stages; ++i)
          if (w_issued & (1u << i)) {
            const long long t0 = clock64();
            while (!mbar_try_wait(bar_w_full + 8 * i, (w_issued_phase >> i) & 1u) && clock64() - t0 < kWaitLimitCycles) {}
          }
      __syncwarp();
    }
    const int ch = q * 32 + lane, n = n0 + ch;
    s_scale[ch] = n < p.N ? scale[n] : 0.f;
    s_scale[128 + ch] = (n < p.N && bias && blockIdx.y == 0) ? bias[n] : 0.f;
    asm volatile("griddepcontrol.wait;" ::: "memory");       // y is zeroed, `down` written by the pre-pass
    for (int i = tid - 64; i < Mt; i += 128) s_down[i] = m0 + i < p.M ? ld_chain(down + m0 + i) : 0.f;
    // after the last MMA the rings are free: every copy has landed and been read
    alive = mbar_wait_warp(bar_acc_full, 0, s_abort, p.error_flag);
    if (alive) {
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16);
      float* sums = reinterpret_cast<float*>(smem) + ch;
      for (int c0 = 0; c0 < Mt; c0 += 16) {
        if (m0 + c0 >= p.M) break;
        uint32_t v[16], v2[16];
        tmem_ld16(taddr + c0, v);
        if (p.stack) tmem_ld16(taddr + Mt + c0, v2);       // the lo half's partial products
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          float f = __uint_as_float(v[j]);
          if (p.stack) f += __uint_as_float(v2[j]);
          sums[(c0 + j) * 128] = c_begin < c_end ? f : 0.f;
        }
      }
    }
  }

  // ---- sums of the cluster -> y, a row of 128 channels per warp -----------------------------------
  tc_fence_before();
  if (p.cluster > 1) {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
  const int rows = min(Mt, p.M - m0), n = n0 + lane * 4;
  const float4 s = *reinterpret_cast<const float4*>(s_scale + lane * 4), b = *reinterpret_cast<const float4*>(s_scale + 128 + lane * 4);
  const bool vec = (p.N & 3) == 0 && (((uintptr_t)y) & 15) == 0;
  if (!vec) {
    // rows of y that are not 16-byte aligned: neighbouring lanes take neighbouring channels (four channels a lane here too
    // quadrupled the transactions: 5671 x 608, 8 bits, 256 rows 20.6 us in the first version of this epilogue, 24.7 then, 20.6 now)
    for (int r = rank + warp * p.cluster; r < rows; r += (T::THREADS / 32) * p.cluster)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int ch = lane + 32 * j;
        const uint32_t mine = smem_u32(smem) + (uint32_t)(r * 128 + ch) * 4;
        float v = 0.f;
        for (int q = 0; q < p.cluster; ++q) {
          uint32_t theirs;
          float part;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(theirs) : "r"(mine), "r"(q));
          asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(part) : "r"(theirs) : "memory");
          v += part;
        }
        if (n0 + ch >= p.N) continue;
        v = fmaf(v * s_down[r], s_scale[ch], s_scale[128 + ch]);
        float* dst = y + (size_t)(m0 + r) * p.N + n0 + ch;
        if (p.atomic) atomicAdd(dst, v); else *dst = v;
      }
  } else
  for (int r = rank + warp * p.cluster; r < rows; r += (T::THREADS / 32) * p.cluster) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t mine = smem_u32(smem) + (uint32_t)(r * 128 + lane * 4) * 4;
    for (int q = 0; q < p.cluster; ++q) {
      uint32_t theirs;
      float4 part;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(theirs) : "r"(mine), "r"(q));
      asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(part.x), "=f"(part.y), "=f"(part.z), "=f"(part.w) : "r"(theirs) : "memory");
      v.x += part.x; v.y += part.y; v.z += part.z; v.w += part.w;
    }
    const float d = s_down[r];
    v.x = fmaf(v.x * d, s.x, b.x); v.y = fmaf(v.y * d, s.y, b.y); v.z = fmaf(v.z * d, s.z, b.z); v.w = fmaf(v.w * d, s.w, b.w);
    float* dst = y + (size_t)(m0 + r) * p.N + n;
    if (n < p.N) {
      if (p.atomic) asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
      else *reinterpret_cast<float4*>(dst) = v;
    }
  }
  if (p.cluster > 1) {                                       // no CTA leaves while another reads its sums
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
}

static size_t qt_down_offset(int K, int M) { return align_up((size_t)2 * M * K * 2, 16); }

template <int BITS>
aiq_status_t launch_qlinear_tc_bits(const LayerJob& job, int N, int K, int M, void* workspace, int32_t* status, cudaStream_t s) {
  using T = QtKind<BITS>;
  DeviceProps props;
  if (aiq_status_t st = current_device_props(&props)) return st;
  const int smem_limit = props.smem_optin, n_sms = props.n_sms;
  AIQ_ENSURE_DYNAMIC_SMEM(qlinear_tc_kernel<BITS>, smem_limit);
  EncodeTiledFn enc = encode_tiled_fn();
  if (!enc) return set_error(AIQ_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
  QtParams p = {};
  p.N = N; p.K = K; p.M = M; p.error_flag = status;
  // Two A tiles per stage leave room for activation tiles of 128 rows.  At 16 bits a small layer takes those too: a tile of 256
  // rows spends its time in set-up and epilogue (256 rows, 1000 x 1280 18.6 us with tiles of 256, 13.0 of 128; 8192 x 512 20.5 |
  // 14.5; but 8192 x 8192, 192 rows, 56.5 | 64.6, and 4096 x 4096, 129 rows, 22.7 | 24.6).
  p.m_block = T::PIECES == 2 || (T::DIRECT && M > 128 && (long long)N * K <= (1ll << 23)) ? 128 : 256;
  p.Mt = M >= p.m_block ? p.m_block : (M + 15) / 16 * 16;
  const int m_blocks = (M + p.m_block - 1) / p.m_block, row_blocks = (N + 127) / 128;
  p.n_chunks = (K + kQtChunk - 1) / kQtChunk;
  int splits = n_sms / (row_blocks * m_blocks);
  if (splits < 1) splits = 1;
  if (splits > p.n_chunks) splits = p.n_chunks;
  p.chunks_per_split = (p.n_chunks + splits - 1) / splits;
  splits = (p.n_chunks + p.chunks_per_split - 1) / p.chunks_per_split;
  // A pair halves the additions to y, or saves them and zeroing it (4096 x 4096, 8 bits, 256 rows 28.4 us -> 23.6), which
  // pays for the cluster launch only where y is large; larger clusters do not fill the GPCs with one CTA per SM (2048 x
  // 2048, 8 bits, 64 rows, clusters of eight: 8.1 us -> 14).
  p.cluster = splits % 2 == 0 && M > 64 ? 2 : 1;
  const int groups = splits / p.cluster;
  p.atomic = groups > 1;
  p.stack = p.Mt <= 128 ? 1 : 0;
  // The weight and the activation ring (memory, L2) grow in turn, so that both reach equally many chunks ahead.  The weight
  // ring's length is a multiple of the packed tiles between two visits of an expander group, so that a group meets every
  // phase of its barriers.
  const int units = p.stack ? 1 : 2;
  constexpr int w_step = T::A_STAGES * T::TPC > T::CPW ? T::A_STAGES * T::TPC / T::CPW : 1;
  auto fits = [&](int b, int w) { return qt_smem_bytes(T::A_STAGES, p.Mt, p.stack, b, w) + 1024 <= smem_limit; };
  int b_stages = 2, w_stages = w_step > 2 ? w_step : 2;
  if (!fits(b_stages, w_stages))
    return set_error(AIQ_ERR_SHAPE, "qlinear_tc: %d bytes of shared memory needed",
                     qt_smem_bytes(T::A_STAGES, p.Mt, p.stack, b_stages, w_stages) + 1024);
  for (bool more = true; more;) {
    const int w_ahead = w_stages * T::CPW / T::TPC, b_ahead = b_stages / units;
    const bool w_can = w_stages + w_step <= kQtMaxWStages && w_ahead < p.chunks_per_split && fits(b_stages, w_stages + w_step);
    const bool b_can = b_stages < kQtMaxBStages && b_ahead < p.chunks_per_split && fits(b_stages + 1, w_stages);
    if (w_can && (w_ahead <= b_ahead || !b_can)) w_stages += w_step;
    else if (b_can) ++b_stages;
    else more = false;
  }
  p.b_stages = b_stages;
  p.w_stages = w_stages;
  p.a_col = p.stack ? 2 * p.Mt : p.Mt;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.a_col + T::A_COLS) p.tmem_cols <<= 1;

  // activation planes in the workspace: (k, batch row, hi | lo)
  uint16_t* planes = static_cast<uint16_t*>(workspace);
  float* down = reinterpret_cast<float*>(static_cast<uint8_t*>(workspace) + qt_down_offset(K, M));
  CUtensorMap x_map;
  cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)M, 2};
  cuuint64_t strides[2] = {2ull * K, 2ull * K * M};
  cuuint32_t box[3] = {(cuuint32_t)kQtChunk, (cuuint32_t)p.Mt, p.stack ? 2u : 1u};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(&x_map, CU_TENSOR_MAP_DATA_TYPE_UINT16, 3, planes, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(AIQ_ERR_CUDA, "cuTensorMapEncodeTiled (linear layer) failed with code %d", (int)r);

  // packed weights: (byte of a row, row); rows past N and bytes past the row arrive as zeros
  CUtensorMap w_map;
  {
    const cuuint64_t wrow = (cuuint64_t)row_bytes(K, BITS);
    cuuint64_t wdims[2] = {wrow, (cuuint64_t)N};
    cuuint64_t wstrides[1] = {wrow};
    cuuint32_t wbox[2] = {128u, 128u};
    cuuint32_t westr[2] = {1, 1};
    r = enc(&w_map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(job.w), wdims, wstrides, wbox, westr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(AIQ_ERR_CUDA, "cuTensorMapEncodeTiled (packed weights) failed with code %d", (int)r);
  }

  const float* x = static_cast<const float*>(job.in);
  float* y = static_cast<float*>(job.out);
  LaunchScope scope(AIQ_KERNEL_QLINEAR, s, 2.0 * M * N * K,
                    (double)N * row_bytes(K, BITS) + 4.0 * N + 4.0 * M * ((double)K + N));
  const auto split_x = BITS == 8 && p.chunks_per_split * kQtChunk >= 1024 ? qlinear_split_x_kernel<BITS != 32, BITS == 4, BITS == 8>
                                                                          : qlinear_split_x_kernel<BITS != 32, BITS == 4, false>;
  split_x<<<M, 512, 0, s>>>(x, K, M, planes, down, y, p.atomic ? (long long)M * N : 0ll, status);
  AIQ_LAUNCH_CHECK("qlinear_split_x");
  const int smem = qt_smem_bytes(T::A_STAGES, p.Mt, p.stack, b_stages, w_stages) + 1024;
  AIQ_CUDA_TRY(launch_chained_cluster(true, p.cluster, qlinear_tc_kernel<BITS>, dim3(row_blocks * p.cluster, groups, m_blocks), dim3(T::THREADS), smem, s,
                              x_map, w_map, p, job.scale, job.bias, (const float*)down, y));
  AIQ_LAUNCH_CHECK("qlinear_tc");
  return AIQ_OK;
}

}  // namespace

bool qlinear_tc_applicable(int N, int K, int bits, int M) {
  if (!bits_ok(bits)) return false;
  if (M < 9) return false;                         // smaller batches: the warp-level kernels
  if (K % 8 != 0 || K < 64 || N < 32) return false;
  return true;
}

size_t qlinear_tc_workspace_bytes(int K, int M) { return align_up(qt_down_offset(K, M) + (size_t)M * 4, 16); }

aiq_status_t launch_qlinear_tc(const LayerJob& job, int N, int K, int M, void* workspace, int32_t* status, cudaStream_t s) {
  switch (job.bits) {
    case 4: return launch_qlinear_tc_bits<4>(job, N, K, M, workspace, status, s);
    case 8: return launch_qlinear_tc_bits<8>(job, N, K, M, workspace, status, s);
    case 16: return launch_qlinear_tc_bits<16>(job, N, K, M, workspace, status, s);
    case 32: return launch_qlinear_tc_bits<32>(job, N, K, M, workspace, status, s);
  }
  return set_error(AIQ_ERR_UNSUPPORTED_BITS, "qlinear_tc: bits=%d", job.bits);
}

}  // namespace aiq
