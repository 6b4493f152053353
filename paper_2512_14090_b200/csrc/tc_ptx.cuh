// PTX wrappers shared by the tcgen05 kernels: mbarriers with bounded waits, TMA and bulk copies,
// tensor-memory allocation, MMA issue and accumulator loads.
#pragma once

#include "common.cuh"

#include <cuda.h>

namespace aiq {
namespace {

constexpr long long kWaitLimitCycles = 4000ll * 1000ll * 1000ll;  // every wait gives up after ~2 s of SM clocks
constexpr uint32_t kSpinLimit = 1u << 30;                         // and after this many polls at the latest

// cuTensorMapEncodeTiled of the driver (looked up once), or nullptr
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline EncodeTiledFn encode_tiled_fn() {
  static std::atomic<EncodeTiledFn> fn{nullptr};
  if (EncodeTiledFn f = fn.load(std::memory_order_acquire)) return f;
  void* sym = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess)
    return nullptr;
  fn.store(reinterpret_cast<EncodeTiledFn>(sym), std::memory_order_release);
  return reinterpret_cast<EncodeTiledFn>(sym);
}

// ---- PTX wrappers ------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// A look at a barrier without waiting.  Its answer takes about a hundred cycles to arrive, as that of a wait on a barrier
// that is already complete does: asked for one step ahead, it costs an issuing warp nothing.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false (and raises the abort flag) when `limit_cycles` SM clocks have
// passed, or another role has already aborted.
__device__ __forceinline__ bool mbar_wait_for(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                              int32_t* error_flag, long long limit_cycles) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (uint32_t i = 0; i < kSpinLimit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 255u) == 255u) {
      if (*abort_flag) return false;
      if (clock64() - t0 > limit_cycles) break;
    }
  }
  *abort_flag = 1;
  if (error_flag) atomicExch(error_flag, 1);
  return false;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int32_t* error_flag) {
  return mbar_wait_for(bar, parity, abort_flag, error_flag, kWaitLimitCycles);
}
// the same out of line: a loop that rarely waits stays small
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* error_flag) {
  return mbar_wait_for(bar, parity, abort_flag, error_flag, kWaitLimitCycles);
}
// bounded wait by a whole (converged) warp: the same answer in every lane.  (Polling from
// one elected lane and broadcasting the result was measured 40 % slower on the convolution.)
__device__ __forceinline__ bool mbar_wait_warp_inline(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* error_flag) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;      // one vote, a uniform branch
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, error_flag));
}
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               int32_t* error_flag) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;      // one vote, a uniform branch
  return __all_sync(0xffffffffu, mbar_wait_slow(bar, parity, abort_flag, error_flag));
}

// By a converged warp: one elected lane announces the bytes on the barrier and issues the copy.  (Inside `if (lane == 0)`
// a producer loop took 400 cycles for a copy; its descriptor and coordinates cannot stay in uniform registers there.)
__device__ __forceinline__ void tma_fill_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, uint32_t bytes, int c0, int c1, int c2) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%2], %3;\n\t"
      "@q cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%4, %5, %6}], [%2];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(bytes), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ void tma_fill_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, uint32_t bytes, int c0, int c1) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%2], %3;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%4, %5}], [%2];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(bytes), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void expect_tx_elect(uint32_t bar, uint32_t bytes) {
  asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}"
               ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_load_4d_elect(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
      "@q cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tma_load_5d_elect(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3, int c4) {
  asm volatile(
      "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
      "@q cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
      : "memory");
}
// two boxes of `half` bytes each on one barrier, the second at c0b
__device__ __forceinline__ void tma_fill2_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, uint32_t half, int c0, int c0b, int c1) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t.reg .b32 d, n;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "add.s32 n, %3, %3;\n\tadd.s32 d, %0, %3;\n\t"
      "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%2], n;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%4, %6}], [%2];\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [d], [%1, {%5, %6}], [%2];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(half), "r"(c0), "r"(c0b), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
               : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// The MMA-issuing warp runs its loop with all 32 lanes converged and lets one elected lane
// issue each tensor-core instruction (elect.sync picks the same lane every time, so the
// commits track the MMAs of that lane).  Converged code lets the compiler keep descriptors in
// uniform registers; a loop inside `if (lane == 0)` measured 50 cycles per MMA issued, this
// form 28 - 39, which matters here because the MMAs are small (8 - 32 cycles of math).
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
      ::"r"(bar) : "memory");
}
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// the four MMAs of 64 k whose operands lie in rows of 128 swizzled bytes (32 bytes further in both for each), one election
__device__ __forceinline__ void umma_k64(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "add.s64 a, %1, 2;\n\tadd.s64 b, %2, 2;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, 1;\n\t"
      "add.s64 a, %1, 4;\n\tadd.s64 b, %2, 4;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, 1;\n\t"
      "add.s64 a, %1, 6;\n\tadd.s64 b, %2, 6;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, 1;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// the same with A in tensor memory: two 16-bit values of a row (lane) per column, 8 columns for each 16 k
__device__ __forceinline__ void umma_k64_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b32 a;\n\t.reg .b64 b;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t"
      "add.s32 a, %1, 8;\n\tadd.s64 b, %2, 2;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, 1;\n\t"
      "add.s32 a, %1, 16;\n\tadd.s64 b, %2, 4;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, 1;\n\t"
      "add.s32 a, %1, 24;\n\tadd.s64 b, %2, 6;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, 1;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 16 columns of the 32 lanes of this warp's quarter; complete after tmem_st_wait
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}
// Two float32 lanes in one 64-bit register: one instruction for both, the roundings of the scalar operations.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// the two bfloat16 of a word as floats (a bfloat16 is the upper half of a float)
__device__ __forceinline__ uint64_t widen2(uint32_t w) { return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u)); }

// v = hi + lo with hi = bf16_rn(v), lo = bf16_rn(v - hi), two values at a time (one packed
// conversion per pair); the same roundings as split_bf16
__device__ __forceinline__ void split_pair(float u0, float u1, uint32_t& hi2, uint32_t& lo2) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(u0, u1);
  hi2 = *reinterpret_cast<const uint32_t*>(&h);
  const float2 d = unpack2(sub2(pack2(u0, u1), widen2(hi2)));
  const __nv_bfloat162 l = __floats2bfloat162_rn(d.x, d.y);
  lo2 = *reinterpret_cast<const uint32_t*>(&l);
}
// Eight finished accumulators of a pixel: scale, bias, residual (hi and lo words, or none), activation, split into four
// hi and four lo words.  ACT and RES are template arguments because the epilogues are bound by these instructions, and a
// residual or activation chosen inside is predicated, not skipped: its instructions issue all the same.  The pointwise
// layer 24 -> 144 (256 x 32 x 32) took 46 us so, 43.5 us with both chosen once per warp.
template <int ACT>
__device__ __forceinline__ float act_of(float v) {
  if (ACT == AIQ_ACT_RELU) return fmaxf(v, 0.0f);
  if (ACT == AIQ_ACT_RELU6) return fminf(fmaxf(v, 0.0f), 6.0f);
  return v;
}
template <int ACT, bool RES>
__device__ __forceinline__ void finish8(const uint32_t* v, const float* scale, const float* bias, uint4 rh, uint4 rl, uint32_t* hi,
                                        uint32_t* lo) {
  const uint32_t rhw[4] = {rh.x, rh.y, rh.z, rh.w}, rlw[4] = {rl.x, rl.y, rl.z, rl.w};
#pragma unroll
  for (int e = 0; e < 8; e += 4) {
    const ulonglong2 sc = *reinterpret_cast<const ulonglong2*>(scale + e), bi = *reinterpret_cast<const ulonglong2*>(bias + e);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int w = (e >> 1) + i;
      uint64_t u = fma2(pack2(__uint_as_float(v[2 * w]), __uint_as_float(v[2 * w + 1])), i ? sc.y : sc.x, i ? bi.y : bi.x);
      if (RES) u = add2(u, add2(widen2(rhw[w]), widen2(rlw[w])));
      const float2 f = unpack2(u);
      split_pair(act_of<ACT>(f.x), act_of<ACT>(f.y), hi[w], lo[w]);
    }
  }
}
// Four finished accumulators as floats, rounded as a stored hi / lo pair rounds them: the value of the pair itself.
template <int ACT>
__device__ __forceinline__ ulonglong2 finish4(const uint32_t* v, const float* scale, const float* bias) {
  const ulonglong2 sc = *reinterpret_cast<const ulonglong2*>(scale), bi = *reinterpret_cast<const ulonglong2*>(bias);
  ulonglong2 o;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float2 f = unpack2(fma2(pack2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])), i ? sc.y : sc.x, i ? bi.y : bi.x));
    uint32_t h, l;
    split_pair(act_of<ACT>(f.x), act_of<ACT>(f.y), h, l);
    (i ? o.y : o.x) = add2(widen2(h), widen2(l));
  }
  return o;
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Eight packed codes (4 bits: raw.x; 8 bits: raw.x, raw.y; two's complement) -> eight
// bfloat16, without the conversion unit: the offset-binary code is placed in the low
// mantissa bits of 2^23, one subtraction gives the integer as a float, and because
// |code| <= 128 has at most 8 significant bits the upper half of that float is the exact
// bfloat16.
__device__ __forceinline__ void expand8_bf16(uint2 raw, int bits, uint32_t* out) {
  float f[8];
  if (bits == 8) {
    const uint32_t w0 = raw.x ^ 0x80808080u, w1 = raw.y ^ 0x80808080u;
    f[0] = __uint_as_float(__byte_perm(w0, 0x4B000000u, 0x7540)) - 8388736.0f;
    f[1] = __uint_as_float(__byte_perm(w0, 0x4B000000u, 0x7541)) - 8388736.0f;
    f[2] = __uint_as_float(__byte_perm(w0, 0x4B000000u, 0x7542)) - 8388736.0f;
    f[3] = __uint_as_float(__byte_perm(w0, 0x4B000000u, 0x7543)) - 8388736.0f;
    f[4] = __uint_as_float(__byte_perm(w1, 0x4B000000u, 0x7540)) - 8388736.0f;
    f[5] = __uint_as_float(__byte_perm(w1, 0x4B000000u, 0x7541)) - 8388736.0f;
    f[6] = __uint_as_float(__byte_perm(w1, 0x4B000000u, 0x7542)) - 8388736.0f;
    f[7] = __uint_as_float(__byte_perm(w1, 0x4B000000u, 0x7543)) - 8388736.0f;
  } else {
    const uint32_t w = raw.x ^ 0x88888888u;
#pragma unroll
    for (int j = 0; j < 8; ++j) f[j] = __uint_as_float(((w >> (4 * j)) & 0xFu) | 0x4B000000u) - 8388616.0f;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) out[j] = __byte_perm(__float_as_uint(f[2 * j]), __float_as_uint(f[2 * j + 1]), 0x7632);
}

}  // namespace
}  // namespace aiq
