// Depthwise 3x3 convolution (stride 1 or 2, pad 1) with bias, residual and activation.
//
// The layer moves 8 bytes per output element for 18 FLOP: it is bound by memory traffic, so the
// kernel is organised around bytes in flight and instructions per element:
//   - input rows arrive in a ring of shared-memory stages by TMA, several rows ahead of their use (a
//     stage = one padded row of NI images x a column tile x a slab of Cb channels; columns outside
//     the map are filled with zeros, rows outside it are the physical padding rows of the tensor),
//     so the loads in flight do not depend on how many warps are resident;
//   - a thread owns 4 consecutive channels and COLS consecutive output columns of one image and walks
//     down the rows: each input row feeds the (up to three) output rows it belongs to, and an input value is
//     unpacked once per thread.  A block keeps its channel slab, whose expanded weights, scales and biases
//     sit in shared memory (beside three rows of accumulators they do not fit the registers);
//   - products are packed float32 pairs (two lanes per instruction).
// The kernels this one replaced loaded their inputs from global memory in each thread (one row per
// thread, or rows walked by a thread): 43 instructions per element and the loads of three blocks in
// flight, 2.7 TB/s on MobileNetV2-CIFAR at batch 256, and every block expanded the weights of all
// channels into shared memory first, which was most of the 13 us of a single-image launch.
// Rows 0 and Ho+1 of every output image (the physical padding rows) are written as zeros.
#include "tc_ptx.cuh"

#include <algorithm>
#include <type_traits>

namespace aiq {

namespace {

constexpr int kDwThreads = 224;                     // compute threads at most; one more warp issues the copies: eight warps
                                                    // per block, so that two blocks per SM have 128 registers a thread
constexpr int kDwMaxStages = 8;
constexpr int kDwMaxColGroups = 56;                 // column groups of a block: its input box stays within 256 columns

struct DwParams {
  int B, H, W, Ho, Wo, C, Cs, act;
  int Cb, CQ;               // channels of a slab, its quads
  int XG, n_ct;             // column groups of a block, column tiles of a row
  int NI, n_ig;             // images of a block, image groups
  int n_slabs, k;           // slabs (fastest in the grid), blocks per slab
  int rows, row_rem;        // output rows of a block, and how many blocks have one more
  int n_rb;                 // or: blocks per image column, each of `rows` rows (the last of fewer); 0: an equal share
  int Wb;                   // input columns of a stage
  int stages, box_bytes, stage_bytes;   // bytes a copy brings; stages start on 128-byte boundaries
  int batch_capacity;       // images per version of the input slot
  int32_t* error_flag;
};

// hi and lo halves of four channels -> two packed float pairs
__device__ __forceinline__ void join4(uint2 h, uint2 l, uint64_t* v) {
  v[0] = add2(widen2(h.x), widen2(l.x));
  v[1] = add2(widen2(h.y), widen2(l.y));
}

// Four channels of one pixel in shared memory: [hi(Cb) | lo(Cb)] bfloat16 or Cb floats.
// (By 32-bit address: through a pointer the compiler reads generically, with the latency of a global access.)
template <int FMT>
__device__ __forceinline__ void read4(uint32_t p, int Cb, uint64_t* v) {
  if (FMT == ACT_SPLIT) {
    uint2 h, l;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(h.x), "=r"(h.y) : "r"(p));
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(l.x), "=r"(l.y) : "r"(p + 2 * Cb));
    join4(h, l, v);
  } else {
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v[0]), "=l"(v[1]) : "r"(p));
  }
}

// The same four channels of a pixel in global memory (lo_off: bytes from the hi to the lo half).
template <int FMT>
__device__ __forceinline__ void load4(const uint8_t* p, uint32_t lo_off, uint64_t* v) {
  if (FMT == ACT_SPLIT) {
    join4(ld_chain(reinterpret_cast<const uint2*>(p)), ld_chain(reinterpret_cast<const uint2*>(p + lo_off)), v);
  } else {
    const float4 t = ld_chain(reinterpret_cast<const float4*>(p));
    v[0] = pack2(t.x, t.y); v[1] = pack2(t.z, t.w);
  }
}

template <int FMT>
__device__ __forceinline__ void store4(uint8_t* __restrict__ p, uint32_t lo_off, const float* v) {
  if (FMT == ACT_SPLIT) {
    uint2 h, l;
    split_pair(v[0], v[1], h.x, l.x);
    split_pair(v[2], v[3], h.y, l.y);
    *reinterpret_cast<uint2*>(p) = h;
    *reinterpret_cast<uint2*>(p + lo_off) = l;
  } else {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
}

// The output rows of a slab are one sequence: row of the image fastest, then column tile, image group.  A block owns an
// equal share of it, wherever that begins and ends, and walks it in pieces that stay inside one image; or, where a share
// would be less than an image, a piece of one image.
struct DwUnit { int ox0, oy0, n_out, img0; };           // ox0: first output column of the tile
template <int COLS>
__device__ __forceinline__ DwUnit dw_unit(const DwParams& p, int r, int r_end) {
  DwUnit d;
  const int col = r / p.Ho, ig = col / p.n_ct;
  d.oy0 = r - col * p.Ho;
  d.n_out = min(p.Ho - d.oy0, r_end - r);
  d.ox0 = (col - ig * p.n_ct) * p.XG * COLS;
  d.img0 = ig * p.NI;
  return d;
}

// COLS output columns per thread: 4 at stride 1 (small launches: 2, see dw_search_shape), 2 at stride 2.  Four columns share
// six input columns, two share four, two at stride 2 share five: an input value is read 1.5, 2 or 1.25 times.
// IFMT / FMT: pixel formats of the input and of the output; floats in, pairs out behind an expansion (ConvGeom::in_f32).
// What bounds it, at 256 x 32 x 32 x 192 channels (ncu, cold; two blocks of seven warps per SM, which is what the registers allow):
//   four columns, floats in   79 us, 31.6 M warp instructions, 0.42 per clock and scheduler, DRAM at 5.1 TB/s
//   four columns, pairs in    82 us, 39.2 M (a value is joined each time it is read), 0.47, 4.9 TB/s
//   stride 2, floats in       48 us, 11.2 M, 0.26, 5.2 TB/s
// so at these sizes DRAM first (a plain copy moves 6.5 TB/s), each warp then waiting for its next row; with two columns at
// stride 1 it had been instructions (37 per output element, 2.9 TB/s).  One image (two columns, seven warps per SM) is neither:
// 8 us of one row after the other, at 24 blocks as at 128.
template <int IFMT, int FMT, int STRIDE, int COLS, bool RES>
__global__ void __launch_bounds__(kDwThreads + 32, 2)
depthwise3x3_kernel(const __grid_constant__ CUtensorMap in_map, DwParams p, const LayerJob* __restrict__ jobs) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
  const LayerJob job = jobs[blockIdx.y];
  const int tid = threadIdx.x, lane = tid & 31;
  const int n_compute = (int)blockDim.x - 32;          // whole warps; the last warp issues the copies
  uint64_t* bars = reinterpret_cast<uint64_t*>(ring + p.stages * p.stage_bytes);
  const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8 * kDwMaxStages;
  volatile int* s_abort = reinterpret_cast<volatile int*>(bars + 2 * kDwMaxStages);
  float* s_w = reinterpret_cast<float*>(ring + p.stages * p.stage_bytes + (2 * kDwMaxStages + 2) * 8);   // [9 taps, scale, bias][Cb]
  const int share = (int)blockIdx.x / p.n_slabs, slab = (int)blockIdx.x - share * p.n_slabs;
  int r_begin = share * p.rows + min(share, p.row_rem), r_end = r_begin + p.rows + (share < p.row_rem ? 1 : 0);
  if (p.n_rb) {
    const int col = share / p.n_rb;
    r_begin = col * p.Ho + (share - col * p.n_rb) * p.rows;
    r_end = min(r_begin + p.rows, (col + 1) * p.Ho);
  }

  // expanded weights: a thread per channel of the slab
  for (int i = tid; i < p.Cb; i += (int)blockDim.x) {
    const int c = slab * p.Cb + i;
    const bool real = c < p.C;                           // padding channels: zero weights, scale and bias
    const uint8_t* row = job.w + (size_t)(real ? c : 0) * (32 * job.bits / 8);   // K = 9 pads to 32 elements
    uint4 r0 = __ldg(reinterpret_cast<const uint4*>(row)), r1 = r0, r2 = r0;
    if (job.bits >= 16) r1 = __ldg(reinterpret_cast<const uint4*>(row) + 1);
    if (job.bits == 32) r2 = __ldg(reinterpret_cast<const uint4*>(row) + 2);
    const uint32_t words[12] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w, r2.x, r2.y, r2.z, r2.w};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      float v;
      if (job.bits == 4) v = (float)((int)(((words[k >> 3] >> (4 * (k & 7))) & 0xFu) ^ 8u) - 8);
      else if (job.bits == 8) v = (float)(int)(int8_t)((words[k >> 2] >> (8 * (k & 3))) & 0xFFu);
      else if (job.bits == 16) v = __half2float(__ushort_as_half((unsigned short)((words[k >> 1] >> (16 * (k & 1))) & 0xFFFFu)));
      else v = __uint_as_float(words[k]);
      s_w[k * p.Cb + i] = real ? v : 0.f;
    }
    s_w[9 * p.Cb + i] = real ? __ldg(job.scale + c) : 0.f;
    s_w[10 * p.Cb + i] = real ? __ldg(job.bias + c) : 0.f;
  }
  if (tid == 0) {
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(bar_full + 8 * i, 1);
      mbar_init(bar_empty + 8 * i, n_compute / 32);
    }
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  chain_release();

  if (tid >= n_compute) {
    // ---- producer: padded input rows oy0 * STRIDE .. of every piece of this block, in order ----------
    chain_wait();
    bool alive = true;
    uint32_t stage = 0, phase = 0, issued = 0, issued_phase = 0;
    for (int r0 = r_begin; r0 < r_end && alive;) {
      const DwUnit d = dw_unit<COLS>(p, r0, r_end);
      r0 += d.n_out;
      const int n_rows = (d.n_out - 1) * STRIDE + 3;
      const int img = job.in_version * p.batch_capacity + d.img0;
      for (int r = 0; r < n_rows; ++r) {
        alive = mbar_wait_warp(bar_empty + 8 * stage, phase ^ 1u, s_abort, p.error_flag);
        if (!alive) break;
        issued |= 1u << stage;
        issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
        expect_tx_elect(bar_full + 8 * stage, (uint32_t)p.box_bytes);
        tma_load_5d_elect(smem_u32(ring) + stage * p.stage_bytes, &in_map, bar_full + 8 * stage, slab * p.Cb, 0,
                          d.ox0 * STRIDE - 1, d.oy0 * STRIDE + r, img);
        if (++stage == (uint32_t)p.stages) { stage = 0; phase ^= 1u; }
      }
    }
    for (int i = 0; i < p.stages; ++i)               // copies in flight must land before the CTA exits
      if (issued & (1u << i)) {
        const long long t0 = clock64();
        while (!mbar_try_wait(bar_full + 8 * i, (issued_phase >> i) & 1u) && clock64() - t0 < kWaitLimitCycles) {}
      }
    return;
  }

  // ---- compute: thread = (image of the group, column group, channel quad), quad fastest ---------------
  const int q = tid % p.CQ, xg = (tid / p.CQ) % p.XG, ni = tid / (p.CQ * p.XG);
  const bool worker = ni < p.NI;                         // the last warp may have idle lanes
  const int c = slab * p.Cb + q * 4;
  const size_t pix_bytes = (size_t)4 * p.Cs;             // [hi(Cs) | lo(Cs)] bfloat16 or Cs floats
  const uint32_t lo_off = 2u * p.Cs;
  const uint32_t ch_off = (uint32_t)c * (FMT == ACT_SPLIT ? 2u : 4u);
  const uint32_t out_pitch = (uint32_t)(p.Wo * pix_bytes);
  const uint32_t col_bytes = 4u * p.Cb;                  // a pixel of the slab in shared memory
  const bool clamp = p.act != AIQ_ACT_NONE;              // relu: [0, inf), relu6: [0, 6]
  const float act_hi = p.act == AIQ_ACT_RELU6 ? 6.0f : __int_as_float(0x7f800000);

  chain_wait();                                          // the output slot may still be read by an earlier kernel
  constexpr int IN_COLS = (COLS - 1) * STRIDE + 3;
  const uint32_t my_cols = smem_u32(ring) + (uint32_t)(worker ? ni * p.Wb + xg * COLS * STRIDE : 0) * col_bytes +
                           (uint32_t)q * (IFMT == ACT_SPLIT ? 8 : 16);
  uint32_t stage = 0, phase = 0;
  bool alive = true;
  const uint32_t my_w = smem_u32(s_w) + q * 16;
  auto coef = [&](int k, uint64_t (&v)[2]) {             // the four channels of row k of s_w
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v[0]), "=l"(v[1]) : "r"(my_w + k * p.Cb * 4));
  };
  // The next padded row: wait, accumulate it as tap row RA into `a`, RB into `b` and RC into `cc` (-1: not
  // at all; the first contribution to `cc` is written, not added) and hand the stage back.
  auto row = [&](auto ra, auto rb_, auto rc, uint64_t (&a)[COLS][2], uint64_t (&b)[COLS][2], uint64_t (&cc)[COLS][2]) -> bool {
    constexpr int RA = decltype(ra)::value, RB = decltype(rb_)::value, RC = decltype(rc)::value;
    alive = mbar_wait_warp(bar_full + 8 * stage, phase, s_abort, p.error_flag);
    if (!alive) return false;
    const uint32_t src = my_cols + stage * p.stage_bytes;
    uint64_t v[IN_COLS][2];
#pragma unroll
    for (int xx = 0; xx < IN_COLS; ++xx) read4<IFMT>(src + xx * col_bytes, p.Cb, v[xx]);
    auto tap_row = [&](auto r_, auto fresh, uint64_t (&s)[COLS][2]) {
      constexpr int R = decltype(r_)::value;
      constexpr bool FRESH = decltype(fresh)::value;
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        uint64_t w[2];
        coef(R * 3 + t, w);
#pragma unroll
        for (int x = 0; x < COLS; ++x)
#pragma unroll
          for (int i = 0; i < 2; ++i)
            s[x][i] = FRESH && t == 0 ? mul2(v[x * STRIDE + t][i], w[i]) : fma2(v[x * STRIDE + t][i], w[i], s[x][i]);
      }
    };
    if constexpr (RA >= 0) tap_row(ra, std::false_type(), a);
    if constexpr (RB >= 0) tap_row(rb_, std::false_type(), b);
    if constexpr (RC >= 0) tap_row(rc, std::true_type(), cc);
    // The stage is handed back once its words have been used, not merely loaded: the accumulators of this row (every
    // input column enters one of them) are operands of the empty statement before the arrival.
#pragma unroll
    for (int x = 0; x < COLS; ++x) {
      if (RA >= 0) asm volatile("" ::"l"(a[x][0]), "l"(a[x][1]) : "memory");
      else asm volatile("" ::"l"(cc[x][0]), "l"(cc[x][1]) : "memory");
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bar_empty + 8 * stage);
    if (++stage == (uint32_t)p.stages) { stage = 0; phase ^= 1u; }
    return true;
  };
  using I0 = std::integral_constant<int, 0>;
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  using IN = std::integral_constant<int, -1>;

  for (int r0 = r_begin; r0 < r_end && alive;) {
    const DwUnit d = dw_unit<COLS>(p, r0, r_end);
    r0 += d.n_out;
    const int b = d.img0 + ni, ox = d.ox0 + xg * COLS;
    const bool writes = worker && b < p.B && c < p.Cs && ox < p.Wo;
    uint8_t* outp = static_cast<uint8_t*>(job.out) + ch_off + (((size_t)b * (p.Ho + 2) + d.oy0 + 1) * p.Wo + ox) * pix_bytes;
    const uint8_t* resp = RES ? static_cast<const uint8_t*>(job.res) + (outp - static_cast<uint8_t*>(job.out)) : nullptr;
    // finish and store the next output row (rows are emitted in order) from its accumulators
    auto emit = [&](const uint64_t (&acc)[COLS][2]) {
      if (writes) {
        uint64_t sc[2], bi[2];
        coef(9, sc);
        coef(10, bi);
#pragma unroll
        for (int x = 0; x < COLS; ++x) {
          if (ox + x >= p.Wo) break;
          uint64_t r[2] = {fma2(acc[x][0], sc[0], bi[0]), fma2(acc[x][1], sc[1], bi[1])};
          if (RES) {
            uint64_t rs[2];
            load4<FMT>(resp + x * pix_bytes, lo_off, rs);
            r[0] = add2(r[0], rs[0]);
            r[1] = add2(r[1], rs[1]);
          }
          const float2 e0 = unpack2(r[0]), e1 = unpack2(r[1]);
          float v[4] = {e0.x, e0.y, e1.x, e1.y};
          if (clamp) {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = fminf(fmaxf(v[i], 0.f), act_hi);
          }
          store4<FMT>(outp + x * pix_bytes, lo_off, v);   // padding channels: zero weights and bias give zero
        }
      }
      outp += out_pitch;
      if (RES) resp += out_pitch;
    };
    if (STRIDE == 1) {
      // input row k of the block (padded row oy0 + k) is tap row 2 / 1 / 0 of output rows k - 2 / k - 1 / k
      uint64_t A[COLS][2], Bq[COLS][2], Cq[COLS][2];
#pragma unroll
      for (int x = 0; x < COLS; ++x) A[x][0] = A[x][1] = Bq[x][0] = Bq[x][1] = 0ull;
      const int n_rows = d.n_out + 2;
      for (int k = 0; k < n_rows; k += 3) {
        if (!row(I2(), I1(), I0(), A, Bq, Cq)) break;
        if (k >= 2) emit(A);
        if (k + 1 < n_rows) {
          if (!row(I2(), I1(), I0(), Bq, Cq, A)) break;
          if (k + 1 >= 2) emit(Bq);
        }
        if (k + 2 < n_rows) {
          if (!row(I2(), I1(), I0(), Cq, A, Bq)) break;
          emit(Cq);
        }
      }
    } else {
      // output row j takes padded rows 2 j, 2 j + 1, 2 j + 2; row 2 j + 2 is also the first of output j + 1
      uint64_t acc[COLS][2], next[COLS][2];
      row(IN(), IN(), I0(), acc, acc, next);
      for (int j = 0; j < d.n_out && alive; ++j) {
#pragma unroll
        for (int x = 0; x < COLS; ++x) { acc[x][0] = next[x][0]; acc[x][1] = next[x][1]; }
        if (!row(I1(), IN(), IN(), acc, acc, acc)) break;
        if (!row(I2(), IN(), I0(), acc, acc, next)) break;
        emit(acc);
      }
    }
    // the two physical padding rows of the image, by the pieces that hold the first and the last row
    if (writes) {
      const float zero[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        if (side == 0 ? d.oy0 != 0 : d.oy0 + d.n_out != p.Ho) continue;
        uint8_t* z = static_cast<uint8_t*>(job.out) + ch_off +
                     (((size_t)b * (p.Ho + 2) + (side == 0 ? 0 : p.Ho + 1)) * p.Wo + ox) * pix_bytes;
#pragma unroll
        for (int x = 0; x < COLS; ++x)
          if (ox + x < p.Wo) store4<FMT>(z + x * pix_bytes, lo_off, zero);
      }
    }
  }
}

// The part of the launch shape the tensor map depends on: slab width, column groups, images of a stage.
struct DwShape { int cols, Cb, XG, NI, Wb; };
DwShape dw_search_shape(const ConvGeom& g, int batch_capacity) {
  DwShape s = {};
  // Four columns per thread at stride 1 where that gives every resident thread a row, else two: a small launch is
  // bound by the chain of one row after the other, and half as many outputs per thread make a shorter one
  // (MobileNetV2-CIFAR, one image: 341 us per pass with four columns, 318 with two).
  s.cols = g.stride == 1 && (long long)batch_capacity * g.Ho * g.Wo * g.Cs_out >= 16ll * 65536 ? 4 : 2;
  const int xg = (g.Wo + s.cols - 1) / s.cols;
  // the slab width that keeps most of the threads on output columns that exist (ties: the widest, for long
  // contiguous runs of the tensor); narrow maps put several images side by side, 8 at most
  double best = 0.0;
  for (int cb = 16; cb <= 256 && cb <= g.Cs_out; cb += 16) {
    if (g.Cs_out % cb != 0 || cb / 4 > kDwThreads) continue;
    int w = std::min(xg, std::min(kDwMaxColGroups, kDwThreads / (cb / 4)));
    const int tiles = (xg + w - 1) / w;
    w = (xg + tiles - 1) / tiles;                              // column tiles of equal width
    const int ni = std::max(1, std::min(std::min(8, batch_capacity), kDwThreads / (cb / 4 * w)));
    const int wb = (w * s.cols - 1) * g.stride + 3;
    if (ni * wb * cb * 4 > 24 * 1024) continue;                // four rows in flight at two blocks per SM
    // (a 16-channel slab reads and writes runs of 32 bytes, a 32-channel one of 64)
    const double used = (double)(cb / 4) * w * ni * g.Wo / (tiles * w * s.cols) * (cb == 16 ? 0.75 : cb == 32 ? 0.9 : 1.0) *
                        batch_capacity / ((batch_capacity + ni - 1) / ni * ni);
    if (used >= best) { best = used; s.Cb = cb; s.XG = w; s.NI = ni; }
  }
  s.Wb = (s.XG * s.cols - 1) * g.stride + 3;
  return s;
}
DwShape dw_shape(const ConvGeom& g, int batch_capacity) {
  static thread_local ConfigMemo<DwShape, 5> memo;
  const int key[5] = {g.Cs_out, g.Ho, g.Wo, g.stride, batch_capacity};
  DwShape s;
  memo.get(key, &s, [&](DwShape* out) { *out = dw_search_shape(g, batch_capacity); return true; });
  return s;
}

// Blocks per slab, blocks per image column or 0, rows of a block (see launch_depthwise).
struct DwSplit { int k, n_rb, rows; };

}  // namespace

aiq_status_t depthwise_encode_map(const ConvGeom& g, const void* slot_base, int batch_capacity, int n_versions, void* map_out) {
  if (g.stride != 1 && g.stride != 2) return set_error(AIQ_ERR_SHAPE, "depthwise: stride %d is not supported", g.stride);
  EncodeTiledFn enc = encode_tiled_fn();
  if (!enc) return set_error(AIQ_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
  const DwShape s = dw_shape(g, batch_capacity);
  const bool split = g.act_format == ACT_SPLIT && !g.in_f32;
  // (channel, hi | lo, column, padded row, image over all versions); float32 pixels have one part
  const cuuint64_t pix = 4ull * g.Cs_in, row = pix * g.W;
  cuuint64_t dims[5] = {(cuuint64_t)g.Cs_in, split ? 2ull : 1ull, (cuuint64_t)g.W, (cuuint64_t)g.H + 2, (cuuint64_t)n_versions * batch_capacity};
  cuuint64_t strides[4] = {split ? 2ull * g.Cs_in : pix, pix, row, row * (g.H + 2)};
  cuuint32_t box[5] = {(cuuint32_t)s.Cb, split ? 2u : 1u, (cuuint32_t)s.Wb, 1u, (cuuint32_t)s.NI};
  cuuint32_t one[5] = {1, 1, 1, 1, 1};
  const CUresult r = enc(static_cast<CUtensorMap*>(map_out), split ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                         5, const_cast<void*>(slot_base), dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(AIQ_ERR_CUDA, "cuTensorMapEncodeTiled (depthwise) failed with code %d", (int)r);
  return AIQ_OK;
}

aiq_status_t launch_depthwise(const ConvGeom& g, const void* map, const LayerJob* jobs_dev, int n_jobs, int batch_capacity,
                              bool has_res, int32_t* error_flag, double weight_bytes, cudaStream_t s) {
  DeviceProps props;
  if (aiq_status_t st = current_device_props(&props)) return st;
  const DwShape sh = dw_shape(g, batch_capacity);
  DwParams p = {};
  p.B = g.B; p.H = g.H; p.W = g.W; p.Ho = g.Ho; p.Wo = g.Wo; p.C = g.Cout; p.Cs = g.Cs_out; p.act = g.act;
  p.Cb = sh.Cb; p.CQ = sh.Cb / 4; p.XG = sh.XG; p.NI = sh.NI; p.Wb = sh.Wb;
  const int col_groups = (g.Wo + sh.cols - 1) / sh.cols;
  p.n_ct = (col_groups + sh.XG - 1) / sh.XG;
  p.n_ig = (g.B + sh.NI - 1) / sh.NI;
  p.n_slabs = (g.Cs_out + sh.Cb - 1) / sh.Cb;
  p.batch_capacity = batch_capacity;
  p.error_flag = error_flag;
  p.box_bytes = sh.NI * sh.Wb * sh.Cb * 4;
  p.stage_bytes = (int)align_up((size_t)p.box_bytes, 128);
  const int threads = (p.CQ * p.XG * p.NI + 31) / 32 * 32 + 32;
  // two blocks per SM, each with as many rows in flight as fit (at most 8)
  const int per_cta = (props.smem_optin + 1024) / 2 - 1024;
  const int fixed = 128 + (2 * kDwMaxStages + 2) * 8 + 11 * sh.Cb * 4;
  p.stages = std::min(kDwMaxStages, (per_cta - fixed) / p.stage_bytes);
  if (p.stages < 2) return set_error(AIQ_ERR_SHAPE, "depthwise: %d bytes per input row do not fit shared memory", p.stage_bytes);
  // Blocks per slab.  Cost of a wave = input rows of a block, two halo rows per piece and a start-up of about six rows
  // included; a wave lasts as long however few blocks it has.  Equal shares keep every SM busy to the end (256 x 16 x 16 x
  // 384 channels: 228 blocks of two units each 54.7 us, 288 equal ones 47.5), pieces of one image save halo rows where a
  // share is shorter than an image (32 x 14 x 14 x 576: 15.7 us against 17).
  const int resident = 2 * props.n_sms;
  const long long columns = (long long)p.n_ig * p.n_ct, total = columns * g.Ho;   // output rows of a slab
  if (total >= (1ll << 31)) return set_error(AIQ_ERR_SHAPE, "depthwise: %lld rows of a channel slab", total);
  const int halo = 3 - g.stride;
  auto block_rows = [&](long long rows, bool one_piece) {
    return rows * g.stride + halo * (one_piece ? 1 : 1 + (rows + g.Ho - 2) / g.Ho);
  };
  static thread_local ConfigMemo<DwSplit, 8> memo;
  const int key[8] = {g.Ho, g.stride, p.n_ig, p.n_ct, p.n_slabs, n_jobs, resident, 0};
  DwSplit split;
  memo.get(key, &split, [&](DwSplit* out) {
    double best = 1e300;
    *out = {1, 0, (int)total};
    auto take = [&](long long k, long long rows, int n_rb) {
      const long long ctas = k * p.n_slabs * n_jobs;
      const double cost = (double)((ctas + resident - 1) / resident) * (block_rows(rows, n_rb > 0) + 6.0);
      if (cost < best * 0.999 && k * p.n_slabs < (1ll << 30)) { best = cost; *out = {(int)k, n_rb, (int)rows}; }
    };
    for (int n = 1; n <= g.Ho; n = n < 16 ? n + 1 : n + n / 8) {
      const int rb = (g.Ho + n - 1) / n, n_rb = (g.Ho + rb - 1) / rb;
      take(columns * n_rb, rb, n_rb);
    }
    for (int w = 1; w <= 6; ++w) {
      const long long k = std::max(1ll, std::min(total, (long long)w * resident / ((long long)p.n_slabs * n_jobs)));
      take(k, (total + k - 1) / k, 0);
    }
    return true;
  });
  p.k = split.k;
  p.n_rb = split.n_rb;
  p.rows = split.n_rb ? split.rows : (int)(total / p.k);
  p.row_rem = split.n_rb ? 0 : (int)(total % p.k);
  // no more stages than rows a block walks (small launches: what is left of the SM is the next kernel's)
  p.stages = (int)std::min<long long>(p.stages, std::max(2ll, block_rows(split.rows, split.n_rb > 0)));
  const int smem = p.stages * p.stage_bytes + fixed;
  const dim3 grid((unsigned)(p.k * p.n_slabs), n_jobs);
  LaunchScope scope(AIQ_KERNEL_DEPTHWISE, s, 18.0 * g.B * g.Ho * g.Wo * g.Cout * n_jobs,
                    weight_bytes + 4.0 * n_jobs * ((double)g.B * g.Cin * g.H * g.W +
                                                   (double)g.B * g.Ho * g.Wo * g.Cout));
  const CUtensorMap& m = *static_cast<const CUtensorMap*>(map);
#define AIQ_DW(IFMT_, FMT_, ST_, COLS_, RES_)                                                                   \
  do {                                                                                                          \
    AIQ_ENSURE_DYNAMIC_SMEM((depthwise3x3_kernel<IFMT_, FMT_, ST_, COLS_, RES_>), per_cta);                       \
    AIQ_CUDA_TRY(launch_chained(scope.chain, depthwise3x3_kernel<IFMT_, FMT_, ST_, COLS_, RES_>, grid, dim3(threads), smem, s, m, p, jobs_dev)); \
  } while (0)
#define AIQ_DW_SHAPE(IFMT_, FMT_, RES_)                                                                         \
  do {                                                                                                          \
    if (g.stride == 2) AIQ_DW(IFMT_, FMT_, 2, 2, RES_);                                                         \
    else if (sh.cols == 4) AIQ_DW(IFMT_, FMT_, 1, 4, RES_);                                                     \
    else AIQ_DW(IFMT_, FMT_, 1, 2, RES_);                                                                       \
  } while (0)
  if (g.act_format == ACT_SPLIT && g.in_f32) { if (has_res) AIQ_DW_SHAPE(ACT_F32, ACT_SPLIT, true); else AIQ_DW_SHAPE(ACT_F32, ACT_SPLIT, false); }
  else if (g.act_format == ACT_SPLIT) { if (has_res) AIQ_DW_SHAPE(ACT_SPLIT, ACT_SPLIT, true); else AIQ_DW_SHAPE(ACT_SPLIT, ACT_SPLIT, false); }
  else { if (has_res) AIQ_DW_SHAPE(ACT_F32, ACT_F32, true); else AIQ_DW_SHAPE(ACT_F32, ACT_F32, false); }
#undef AIQ_DW_SHAPE
#undef AIQ_DW
  AIQ_LAUNCH_CHECK("depthwise3x3");
  return AIQ_OK;
}

}  // namespace aiq
