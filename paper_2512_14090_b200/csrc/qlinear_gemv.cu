// Quantized linear layer for 4- and 8-bit weights and up to four batch rows, in one kernel.
//
//   y[m][n] = s_n * sum_k code[n][k] * x[m][k] + bias[n]
//
// The weight stream bounds the layer (8192 x 8192 at 4 bits: 33.6 MB, 5.2 us at the copy bandwidth), so everything is
// arranged around having it in flight from the first instruction on:
//   - one block per SM; a block takes 8 output channels at a time (a unit) over the whole K, and requests as many units as
//     fit its shared memory (about 180 KB) as soon as its first activation loads are under way, by one bulk copy per row;
//   - meanwhile every warp turns its slice of the activations (at most 512 k) into int8 digits with a shared exponent,
//     x = 2^(e-6) (d1 + d2 / 2^7 + d3 / 2^14 + d4 / 2^21), an image of x to 28 bits below the slice's largest |x|, and
//     keeps them in registers as the A operand of mma.m16n8k32 (row 4 m + d = digit d of batch row m) for the whole
//     kernel;
//   - the packed words are the B operand (column = output channel): 8-bit words as they are, a 4-bit word as its even
//     and its odd nibbles (one AND, one shift-AND; the +8 of the offset-binary nibbles leaves again exactly, as 8 times
//     the digit sum); the k order inside a fragment follows from that on both operands;
//   - the integer sums are exact; a warp scales them with its slice's exponent, and the warps' partial sums meet in shared
//     memory in a fixed order: no second kernel, no workspace, no atomics, run-to-run identical;
//   - nothing joins the warps inside the stream: they wait for a unit's copies only, and the output of up to eight units
//     is formed together after it (a block barrier and an output per unit cost 0.5 us each).
// The two kernels this replaces at these sizes (a digit pass over x with three digits, then the matrix with its K slices
// meeting in y through atomics), on the device, calls back to back, one and four rows, before -> now: 8192 x 8192, 4 bits
// 13.4 -> 12.4 and 16.5 -> 16.7 us, 8 bits 18.4 -> 14.0 and 22.3 -> 18.2; 2048 x 8192, 4 bits 10.2 -> 5.6 and 12.4 -> 10.8.
#include "tc_ptx.cuh"

#include <algorithm>

namespace aiq {

namespace {

constexpr int kGvWarps = 16;
constexpr int kGvFrags = 16;                         // k32 fragments of a warp's slice at most: 512 k
constexpr int kGvMaxSlots = 16;
constexpr int kGvEpoch = 8;                          // units per warp between two outputs
constexpr int kGvMaxRows = 4;                        // batch rows
constexpr int kGvRowWords = 128 + 32;                // digit words of 128 k of a batch row
constexpr int kGvDigWords = 2 * kGvRowWords;
static_assert(kGvEpoch * kGvMaxRows * 8 <= kGvDigWords, "the partial sums take the place of the digit words");
__device__ __forceinline__ int gv_dig(int k) { return k + (k >> 4) * 4; }
// max(a, |b|), a NaN if either is one
__device__ __forceinline__ float max_abs_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(fabsf(b)));
  return r;
}

struct GvParams {
  int N, K, M;
  int rb;                   // bytes of a packed row
  int stride;               // of a row in shared memory: 64 modulo 128, so that eight rows x 4 units of 16 bytes spread over all banks
  int kw;                   // warps that share a unit's K
  int cw;                   // 64-byte chunks of a row per warp
  int slots, slot_bytes;
  int slack;                // bytes behind the ring: a row's last chunk may reach past the last slot
};

__device__ __forceinline__ void gv_mma(int* d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Batch rows with an infinity or a NaN have no digits.  After the stream a block works out its channels of those rows (bit m
// of `rows`) again from products in float32, with the results of the plain kernel: 0 x infinity is a NaN.  (Inside the stream,
// slice by slice, the call cost four rows at 4 bits 12 to 19 % in spilled registers.)
template <int BITS>
__device__ __noinline__ void gv_nonfinite_rows(const uint8_t* __restrict__ w, const float* __restrict__ scale,
                                               const float* __restrict__ bias, const float* x, float* y, GvParams p, uint32_t rows) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, ug = kGvWarps / p.kw;
  for (int u0 = (int)blockIdx.x * ug; u0 * 8 < p.N; u0 += (int)gridDim.x * ug)
    for (int n = u0 * 8 + warp; n < min((u0 + ug) * 8, p.N); n += kGvWarps)
      for (int m = 0; m < p.M; ++m) {
        if (!(rows >> m & 1u)) continue;
        const uint8_t* row = w + (size_t)n * p.rb;
        float sum = 0.f;
        for (int k = lane; k < p.K; k += 32) {
          const int b = row[BITS == 4 ? k >> 1 : k];
          const int code = BITS == 4 ? (((b >> (4 * (k & 1))) & 0xF) ^ 8) - 8 : (int)(int8_t)b;
          sum = fmaf((float)code, x[(size_t)m * p.K + k], sum);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) y[(size_t)m * p.N + n] = fmaf(sum, scale[n], bias ? bias[n] : 0.f);
      }
}

// ROWS: batch rows at most, 1, 2 or 4.
template <int BITS, int ROWS>
__global__ void __launch_bounds__(kGvWarps * 32, 1)
qlinear_gemv_kernel(const uint8_t* __restrict__ w, const float* __restrict__ scale, const float* __restrict__ bias,
                    const float* x, float* y, GvParams p) {
  constexpr int HALVES = ROWS > 2 ? 2 : 1;           // of the 16 digit rows of an MMA
  constexpr int RP = ROWS > 1 ? 2 : 1;               // batch rows converted at a time
  constexpr int QP = 2 / RP;                         // and parts of 128 k of each
  constexpr int CHUNK_K = 512 / BITS;                // k of a 64-byte chunk: 128 / 64
  constexpr int LANE_K = CHUNK_K / 4;                // k of a lane's 16 bytes of it: 32 / 16
  constexpr int MPC = CHUNK_K / 32;                  // MMAs per chunk: 4 / 2
  constexpr int MAX_CW = kGvFrags / MPC;             // chunks per warp at most: 4 / 8
  extern __shared__ __align__(128) uint8_t gsm[];
  uint8_t* ring = gsm;
  uint32_t* s_dig = reinterpret_cast<uint32_t*>(gsm + p.slots * p.slot_bytes + p.slack);   // [warp] digit words, then
  float* s_part = reinterpret_cast<float*>(s_dig);                                        // [kGvEpoch][warp][row][8] partial sums
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_dig + kGvWarps * kGvDigWords);
  volatile int* s_abort = reinterpret_cast<volatile int*>(bars + 2 * kGvMaxSlots);
  uint32_t* s_bad = reinterpret_cast<uint32_t*>(bars + 2 * kGvMaxSlots) + 1;              // batch rows that are not finite
  const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8 * kGvMaxSlots;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int ug = kGvWarps / p.kw;                    // units a block works on at a time
  const int n_units = (p.N + 7) >> 3;
  const int per_step = (int)gridDim.x * ug;
  const int n_steps = ((int)blockIdx.x * ug < n_units) ? (n_units - 1 - (int)blockIdx.x * ug) / per_step + 1 : 0;
  const int kwi = warp % p.kw, ugi = warp / p.kw;

  if (tid == 0) {
    for (int i = 0; i < p.slots; ++i) { mbar_init(bar_full + 8 * i, 1); mbar_init(bar_empty + 8 * i, kGvWarps); }
    *s_abort = 0;
    *s_bad = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  chain_release();
  chain_wait();

  const int slice_k = p.cw * CHUNK_K, k0 = kwi * slice_k;
  const bool vec = (p.K & 3) == 0 && (((uintptr_t)x) & 15) == 0;
  auto load_x = [&](int m, int j) {                  // four elements of row m: k = 128 j + 4 lane of the slice
    const float* xr = x + (size_t)m * p.K;
    const int kl = j * 128 + lane * 4, k = k0 + kl;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (m < p.M && kl < slice_k) {
      if (vec && k + 4 <= p.K) q = *reinterpret_cast<const float4*>(xr + k);
      else {
        if (k < p.K) q.x = xr[k];
        if (k + 1 < p.K) q.y = xr[k + 1];
        if (k + 2 < p.K) q.z = xr[k + 2];
        if (k + 3 < p.K) q.w = xr[k + 3];
      }
    }
    return q;
  };
  float4 xv[RP][4];                                  // ahead of the weights, which would queue in front of it
#pragma unroll
  for (int r = 0; r < RP; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) xv[r][j] = load_x(r, j);

  // rows of step i -> slot i mod slots, by one warp.  (Issuing a bulk copy takes about 50 ns: one warp alone needed 2.5 us for
  // the 48 first ones, so each first slot has a warp of its own.)
  auto issue = [&](int i) {
    const int row0 = (i * per_step + (int)blockIdx.x * ug) * 8;
    const int rows = min(8 * ug, p.N - row0);
    const uint32_t bar = bar_full + 8 * (i % p.slots), dst = smem_u32(ring) + (i % p.slots) * p.slot_bytes;
    if (lane == 0) mbar_expect_tx(bar, (uint32_t)(rows * p.rb));
    __syncwarp();
    for (int r = lane; r < rows; r += 32) bulk_load(dst + r * p.stride, w + (size_t)(row0 + r) * p.rb, (uint32_t)p.rb, bar);
  };
  if (warp < p.slots && warp < n_steps) issue(warp);

  // ---- activations of this warp's slice -> digit fragments in registers ---------------------------------
  uint32_t a[kGvFrags][2 * HALVES];                  // per fragment: k 0-15 and 16-31 of row g (and of row g + 8)
  float down[HALVES];                                // value of one unit of this lane's digit row
  int corr[HALVES];                                  // 4 bits: 8 x the digit sum of the row
#pragma unroll
  for (int f = 0; f < kGvFrags; ++f)
#pragma unroll
    for (int i = 0; i < 2 * HALVES; ++i) a[f][i] = 0u;
#pragma unroll
  for (int h = 0; h < HALVES; ++h) { down[h] = 0.f; corr[h] = 0; }
  // Two batch rows at a time, 128 k of both, so that every lane has a row to gather from; the arithmetic is packed float32.
  // (Issue slots bound it.  One row at a time and scalar it was 2.1 us a row; 4 bits, 8192 x 8192, four rows 18.5 -> 16.7 us,
  // 2048 x 8192 12.7 -> 10.8, two rows 7.9 -> 6.6; 8 bits, 8192 x 8192, four rows 20.7 -> 18.2.)
  uint32_t* my_dig = s_dig + warp * kGvDigWords;     // word k at gv_dig(k): four words of padding per 16, against bank conflicts
  const uint32_t d = g & 3, sel = d | ((d + 4u) << 4);            // byte d of two words
  const uint64_t magic = pack2(12582912.f, 12582912.f), m128 = pack2(128.f, 128.f);
#pragma unroll 1
  for (int m0 = 0; m0 < (ROWS > 2 ? p.M : 1); m0 += RP) {
    float up[RP];
    int e_mine = 0;                                               // exponent of this lane's row, m0 + (g >> 2)
    bool finite_mine = true;
#pragma unroll
    for (int r = 0; r < RP; ++r) {
      float top = 0.f;                                            // a NaN stays one
#pragma unroll
      for (int j = 0; j < 4; ++j)
        top = max_abs_nan(max_abs_nan(max_abs_nan(max_abs_nan(top, xv[r][j].x), xv[r][j].y), xv[r][j].z), xv[r][j].w);
      const uint32_t mx = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
      // 2^(e-1) <= largest |x| < 2^e; slices of zeros and of denormals share the smallest exponent
      const int e = max((int)(mx >> 23) - 126, -90);
      const bool finite = mx < 0x7F800000u;
      if (!finite && lane == 0) atomicOr(s_bad, 1u << (m0 + r));  // its digits are never used
      up[r] = __int_as_float((6 - min(e, 128) + 127) << 23);
      if (RP == 1 || (g >> 2) == r) { e_mine = e; finite_mine = finite; }
    }
    uint32_t sum = 0;
#pragma unroll
    for (int j0 = 0; j0 < 4; j0 += QP) {
      if (128 * j0 >= slice_k) break;
#pragma unroll
      for (int part = 0; part < 2; ++part) {                      // row m0 + part, or the part of 128 k after j0
        const int r = RP == 2 ? part : 0, j = RP == 2 ? j0 : j0 + part;
        if (RP == 2 ? m0 + r >= p.M : 128 * j >= slice_k) break;
        uint32_t word[4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          // |v| < 64; every step below is exact.  rint without the conversion unit (a quarter of the rate): adding 1.5 x 2^23
          // leaves the rounded integer in the low bits
          uint64_t v = mul2(i ? pack2(xv[r][j].z, xv[r][j].w) : pack2(xv[r][j].x, xv[r][j].y), pack2(up[r], up[r]));
          float2 q4[4];
#pragma unroll
          for (int dd = 0; dd < 4; ++dd) {
            const uint64_t q = add2(v, magic);
            q4[dd] = unpack2(q);
            if (dd < 3) v = mul2(sub2(v, sub2(q, magic)), m128);
          }
          auto bytes = [](float a, float b, float c, float e) {
            return __byte_perm(__byte_perm(__float_as_uint(a), __float_as_uint(b), 0x0040),
                               __byte_perm(__float_as_uint(c), __float_as_uint(e), 0x0040), 0x5410);
          };
          word[2 * i] = bytes(q4[0].x, q4[1].x, q4[2].x, q4[3].x);
          word[2 * i + 1] = bytes(q4[0].y, q4[1].y, q4[2].y, q4[3].y);
        }
        *reinterpret_cast<uint4*>(my_dig + part * kGvRowWords + gv_dig(lane * 4)) = make_uint4(word[0], word[1], word[2], word[3]);
        if (ROWS > 2) xv[r][j] = load_x(m0 + 2 + r, j);           // the next pair
      }
      __syncwarp();
      // lane (g, t) gathers digit g & 3 of batch row m0 + (g >> 2) into fragment row g = 4 (m & 1) + digit, half m0 >> 1
      if (m0 + (g >> 2) < p.M) {
#pragma unroll
        for (int c = 0; c < QP * 128 / CHUNK_K; ++c) {
          if (j0 * (128 / CHUNK_K) + c >= p.cw) break;
#pragma unroll
          for (int i = 0; i < MPC; ++i) {
            // the eight k of this lane in MMA i of the chunk: 4 bits: 8 i ..: even ones, then odd ones; 8 bits: 8 i ..: in order
            const uint32_t* src = my_dig + (RP == 2 ? (g >> 2) * kGvRowWords : 0) + gv_dig(c * CHUNK_K + t * LANE_K + 8 * i);
            const uint4 lo = *reinterpret_cast<const uint4*>(src), hi = *reinterpret_cast<const uint4*>(src + 4);
            uint32_t f0, f1;
            if (BITS == 4) {
              f0 = __byte_perm(__byte_perm(lo.x, lo.z, sel), __byte_perm(hi.x, hi.z, sel), 0x5410);
              f1 = __byte_perm(__byte_perm(lo.y, lo.w, sel), __byte_perm(hi.y, hi.w, sel), 0x5410);
            } else {
              f0 = __byte_perm(__byte_perm(lo.x, lo.y, sel), __byte_perm(lo.z, lo.w, sel), 0x5410);
              f1 = __byte_perm(__byte_perm(hi.x, hi.y, sel), __byte_perm(hi.z, hi.w, sel), 0x5410);
            }
            sum = (uint32_t)__dp4a((int)f0, 0x01010101, (int)sum);
            sum = (uint32_t)__dp4a((int)f1, 0x01010101, (int)sum);
            const int f = (j0 * (128 / CHUNK_K) + c) * MPC + i;
#pragma unroll
            for (int h = 0; h < HALVES; ++h)
              if ((m0 >> 1) == h) { a[f][2 * h] = f0; a[f][2 * h + 1] = f1; }
          }
        }
      }
      __syncwarp();
    }
    if (m0 + (g >> 2) < p.M) {
#pragma unroll
      for (int h = 0; h < HALVES; ++h)
        if ((m0 >> 1) == h) {
          corr[h] = BITS == 4 ? 8 * (int)sum : 0;
          down[h] = finite_mine ? __int_as_float((e_mine - 6 - 7 * (int)d + 127) << 23) : 0.f;
        }
    }
  }
#pragma unroll
  for (int h = 0; h < HALVES; ++h) {                 // digit sums of the row: its four lanes hold a quarter each
    corr[h] += __shfl_xor_sync(0xffffffffu, corr[h], 1);
    corr[h] += __shfl_xor_sync(0xffffffffu, corr[h], 2);
  }

  __syncthreads();                                   // the digit words make room for the partial sums
  // ---- the weight stream --------------------------------------------------------------------------------
  const uint32_t lane_off = (uint32_t)((ugi * 8 + g) * p.stride + kwi * p.cw * 64 + t * 16);
  bool alive = true;
  int issued = min(p.slots, n_steps);                // steps requested so far (followed by every warp)
  for (int e0 = 0; e0 < n_steps; e0 += kGvEpoch) {
  const int e1 = min(e0 + kGvEpoch, n_steps);
  // the scale and bias of this thread's first output of the epoch, ahead of their use
  const int n_out = (e1 - e0) * ug * p.M * 8;
  auto channel = [&](int o) { return ((e0 + (o >> 3) / (p.M * ug)) * per_step + (int)blockIdx.x * ug + (o >> 3) / p.M % ug) * 8 + (o & 7); };
  float sc = 0.f, bi = 0.f;
  if (tid < n_out && channel(tid) < p.N) {
    sc = __ldg(scale + channel(tid));
    if (bias) bi = __ldg(bias + channel(tid));
  }
  for (int i = e0; i < e1 && alive; ++i) {
    const int slot = i % p.slots;
    alive = mbar_wait_warp(bar_full + 8 * slot, (uint32_t)(i / p.slots) & 1u, s_abort, nullptr);
    if (!alive) break;
    const uint8_t* src = ring + slot * p.slot_bytes + lane_off;
    int acc2[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};     // two chains of dependent MMAs
#pragma unroll
    for (int c = 0; c < MAX_CW; ++c) {
      if (c >= p.cw) break;
      uint4 q = *reinterpret_cast<const uint4*>(src + c * 64);
      if (BITS == 4) { q.x ^= 0x88888888u; q.y ^= 0x88888888u; q.z ^= 0x88888888u; q.w ^= 0x88888888u; }
      const uint32_t words[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < MPC; ++j) {
        const uint32_t b0 = BITS == 4 ? words[j] & 0x0F0F0F0Fu : words[2 * j];
        const uint32_t b1 = BITS == 4 ? (words[j] >> 4) & 0x0F0F0F0Fu : words[2 * j + 1];
        const int f = c * MPC + j;
        gv_mma(acc2[f & 1], a[f][0], HALVES == 2 ? a[f][2 * HALVES - 2] : 0u, a[f][1], HALVES == 2 ? a[f][2 * HALVES - 1] : 0u, b0, b1);
      }
    }
    // the words have been used (the sums below depend on them): hand the slot back
    asm volatile("" ::"r"(acc2[0][0]), "r"(acc2[1][0]) : "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(bar_empty + 8 * slot);
    int acc[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j] = acc2[0][j] + acc2[1][j];
    // lane (g, t): rows g (and g + 8), output channels 2 t and 2 t + 1 of the unit; the four digits of a batch row sit in
    // the lanes with equal g >> 2
    float* part = s_part + ((i - e0) * kGvWarps + warp) * kGvMaxRows * 8;
#pragma unroll
    for (int h = 0; h < HALVES; ++h) {
      float v0 = (float)(acc[2 * h] - corr[h]) * down[h], v1 = (float)(acc[2 * h + 1] - corr[h]) * down[h];
      v0 += __shfl_xor_sync(0xffffffffu, v0, 4);
      v1 += __shfl_xor_sync(0xffffffffu, v1, 4);
      v0 += __shfl_xor_sync(0xffffffffu, v0, 8);
      v1 += __shfl_xor_sync(0xffffffffu, v1, 8);
      if ((g & 3) == 0) *reinterpret_cast<float2*>(part + (2 * h + (g >> 2)) * 8 + 2 * t) = make_float2(v0, v1);
    }
    // one step later, so that the other warps are through with it as well, warp 0 refills the slot of the step before
    if (i > 0 && issued < n_steps && issued == i - 1 + p.slots) {
      if (warp == 0) {
        alive = mbar_wait_warp(bar_empty + 8 * ((i - 1) % p.slots), (uint32_t)((i - 1) / p.slots) & 1u, s_abort, nullptr);
        if (alive) issue(issued);
      }
      ++issued;
    }
  }
  __syncthreads();                                   // the epoch's partial sums are in place
  if (*s_abort) break;
  for (int o = tid; o < n_out; o += kGvWarps * 32) {
    const int n = channel(o), m = (o >> 3) % p.M, u = (o >> 3) / p.M % ug, st = (o >> 3) / (p.M * ug);
    if (n >= p.N) continue;
    if (o != tid) { sc = __ldg(scale + n); bi = bias ? __ldg(bias + n) : 0.f; }
    const float* sp = s_part + (st * kGvWarps + u * p.kw) * kGvMaxRows * 8 + m * 8 + (o & 7);
    float sum = 0.f;
    for (int k = 0; k < p.kw; ++k) sum += sp[k * kGvMaxRows * 8];
    y[(size_t)m * p.N + n] = fmaf(sum, sc, bi);
  }
  __syncthreads();                                   // before the next epoch's partial sums
  }
  if (*s_abort) {
    // a wait expired: let the copies in flight land (bounded as well) and make the failure visible in the result
    if (tid == 0)
      for (int j = 0; j < p.slots && j < issued; ++j) {
        const int u = issued - 1 - (issued - 1 - j) % p.slots;             // last step issued to slot j
        const long long t0 = clock64();
        while (!mbar_try_wait(bar_full + 8 * j, (uint32_t)(u / p.slots) & 1u) && clock64() - t0 < kWaitLimitCycles) {}
      }
    for (int i = tid; i < p.M * p.N; i += kGvWarps * 32) y[i] = __int_as_float(0x7FC00000);
  } else if (*s_bad) {
    gv_nonfinite_rows<BITS>(w, scale, bias, x, y, p, *s_bad);    // after the stream's own outputs (barrier above)
  }
}

}  // namespace

// Up to four rows and rows of at most 8,192 elements (16 warps x 512); at least 256 bytes a row and 2^18 elements:
// below, both this and the plain kernel take less time than a call's host side (512 x 512: 5.8 us a call with either), while
// at 1000 x 1280 the plain kernel needs 10 us and this one 5.9.  Three and four short rows of a small layer are the plain
// kernel's (1280 x 320, 8 bits, 3 rows 5.4 us here, 3.7 there; 512 x 512 5.5 | 3.8; but 1000 x 1280 5.3 | 8.0).
bool qlinear_gemv_applicable(int N, int K, int bits, int M) {
  if ((bits != 4 && bits != 8) || M < 1 || M > kGvMaxRows || K > 8192) return false;
  if (M > 2 && K < 768 && (long long)N * K < (1 << 19)) return false;
  return row_bytes(K, bits) >= 256 && (long long)N * K >= (1 << 18);
}

aiq_status_t launch_qlinear_gemv(const LayerJob& job, int N, int K, int M, cudaStream_t s) {
  DeviceProps props;
  if (aiq_status_t st = current_device_props(&props)) return st;
  GvParams p = {};
  p.N = N; p.K = K; p.M = M;
  p.rb = (int)row_bytes(K, job.bits);
  p.stride = (p.rb + 127) / 128 * 128 + 64;
  const int chunks = (p.rb + 63) / 64, max_cw = job.bits == 4 ? 4 : 8;
  // as few warps per unit as its K needs; more of them where there are fewer units than that leaves warps for
  p.kw = 1;
  const int units = (N + 7) / 8;
  while (p.kw < kGvWarps && ((chunks + p.kw - 1) / p.kw > max_cw || (p.kw < chunks && units * p.kw < props.n_sms * kGvWarps))) p.kw <<= 1;
  p.cw = (chunks + p.kw - 1) / p.kw;
  const int ug = kGvWarps / p.kw;
  p.slot_bytes = (8 * ug * p.stride + 127) / 128 * 128;
  p.slack = (std::max(0, 64 * p.cw * p.kw - p.stride) + 127) / 128 * 128;
  const int fixed = p.slack + kGvWarps * kGvDigWords * 4 + 2 * kGvMaxSlots * 8 + 16;
  const int steps = (units + props.n_sms * ug - 1) / (props.n_sms * ug);
  p.slots = std::min(std::min(kGvMaxSlots, steps), (props.smem_optin - fixed) / p.slot_bytes);
  if (p.slots < 1) return set_error(AIQ_ERR_SHAPE, "qlinear_gemv: %d bytes per step do not fit shared memory", p.slot_bytes);
  const int smem = p.slots * p.slot_bytes + fixed;
  const int grid = std::min(props.n_sms, (units + ug - 1) / ug);
  const float* x = static_cast<const float*>(job.in);
  float* y = static_cast<float*>(job.out);
  LaunchScope scope(AIQ_KERNEL_QLINEAR, s, 2.0 * M * N * K, (double)N * p.rb + 4.0 * N + 4.0 * M * ((double)K + N));
#define AIQ_GEMV(B_, R_)                                                                                                  \
  do {                                                                                                                   \
    AIQ_ENSURE_DYNAMIC_SMEM((qlinear_gemv_kernel<B_, R_>), props.smem_optin);                                             \
    AIQ_CUDA_TRY(launch_chained(true, qlinear_gemv_kernel<B_, R_>, dim3(grid), dim3(kGvWarps * 32), smem, s, job.w, job.scale, \
                                job.bias, x, y, p));                                                                     \
  } while (0)
#define AIQ_GEMV_ROWS(B_) do { if (M == 1) AIQ_GEMV(B_, 1); else if (M == 2) AIQ_GEMV(B_, 2); else AIQ_GEMV(B_, 4); } while (0)
  if (job.bits == 4) AIQ_GEMV_ROWS(4); else AIQ_GEMV_ROWS(8);
#undef AIQ_GEMV_ROWS
#undef AIQ_GEMV
  AIQ_LAUNCH_CHECK("qlinear_gemv");
  return AIQ_OK;
}

}  // namespace aiq
