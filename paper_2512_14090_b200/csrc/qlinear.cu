// Small-batch quantized linear layer: y[m][n] = s_n * sum_k code[n][k] * x[m][k] + bias[n].
//
// The memory-bound case the method targets (Abstract; Section 5, Roofline paragraph): the
// packed weight matrix is streamed once with 128-bit loads, expanded to float32 in
// registers, multiplied against activations held in registers, and reduced across the
// warp with shuffles.  The per-channel scale multiplies the finished sum.
#include "tc_ptx.cuh"

#include <type_traits>

namespace aiq {

namespace {

constexpr int kRowsPerWarp = 4;
constexpr int kWarps = 8;

// 8 consecutive elements starting at element offset `e0` (a multiple of 8) inside a 16-byte
// packed chunk, as floats.
template <int BITS>
__device__ __forceinline__ void decode8(const uint4& q, int sub, float* f) {
  if (BITS == 4) {
    const uint32_t w = sub == 0 ? q.x : sub == 1 ? q.y : sub == 2 ? q.z : q.w;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      // offset-binary nibble in the mantissa of 2^23: exact integer-to-float without I2F
      const uint32_t u = (((w >> (4 * j)) & 0xFu) ^ 0x8u) | 0x4B000000u;
      f[j] = __uint_as_float(u) - 8388616.0f;
    }
  } else if (BITS == 8) {
    const uint32_t w0 = sub == 0 ? q.x : q.z;
    const uint32_t w1 = sub == 0 ? q.y : q.w;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t a = (((w0 >> (8 * j)) & 0xFFu) ^ 0x80u) | 0x4B000000u;
      const uint32_t b = (((w1 >> (8 * j)) & 0xFFu) ^ 0x80u) | 0x4B000000u;
      f[j] = __uint_as_float(a) - 8388736.0f;
      f[j + 4] = __uint_as_float(b) - 8388736.0f;
    }
  } else if (BITS == 16) {
    const __half2 h0 = *reinterpret_cast<const __half2*>(&q.x);
    const __half2 h1 = *reinterpret_cast<const __half2*>(&q.y);
    const __half2 h2 = *reinterpret_cast<const __half2*>(&q.z);
    const __half2 h3 = *reinterpret_cast<const __half2*>(&q.w);
    const float2 a = __half22float2(h0), b = __half22float2(h1), c = __half22float2(h2),
                 d = __half22float2(h3);
    f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y; f[4] = c.x; f[5] = c.y; f[6] = d.x; f[7] = d.y;
  }
}

// One warp: kRowsPerWarp output channels x MT batch rows.  Lanes stride over 16-byte chunks
// of the packed rows.  CHAIN: launched as a dependent of the kernel before (see launch_chained); x is then read by ordinary
// loads, else through the read-only path.
template <int BITS, int MT, bool CHAIN>
__global__ void __launch_bounds__(kWarps * 32)
qlinear_kernel(LayerJob job, int N, int K, int M) {
  constexpr int E = 128 / BITS;                 // elements per 16-byte chunk
  constexpr int SUBS = (E >= 8) ? E / 8 : 1;    // 8-element sub-chunks (fp32: one of 4)
  constexpr int SE = (E >= 8) ? 8 : 4;          // elements per sub-chunk
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int n0 = (blockIdx.x * kWarps + warp) * kRowsPerWarp;
  const int m0 = blockIdx.y * MT;
  if (CHAIN) {
    chain_release();
    chain_wait();
  }
  if (n0 >= N) return;
  const int Kpad = (K + 31) / 32 * 32;
  const size_t rb = (size_t)Kpad * BITS / 8;
  const int n_chunks = Kpad / E;
  const float* x = static_cast<const float*>(job.in);
  const bool xvec = ((K & 3) == 0) && ((((uintptr_t)x) & 15) == 0);

  float acc[kRowsPerWarp][MT];
#pragma unroll
  for (int r = 0; r < kRowsPerWarp; ++r)
#pragma unroll
    for (int m = 0; m < MT; ++m) acc[r][m] = 0.0f;

  const uint8_t* rows[kRowsPerWarp];
#pragma unroll
  for (int r = 0; r < kRowsPerWarp; ++r) rows[r] = job.w + (size_t)min(n0 + r, N - 1) * rb;

  for (int ci = lane; ci < n_chunks; ci += 32) {
    uint4 q[kRowsPerWarp];
#pragma unroll
    for (int r = 0; r < kRowsPerWarp; ++r) q[r] = __ldg(reinterpret_cast<const uint4*>(rows[r]) + ci);
#pragma unroll
    for (int sub = 0; sub < SUBS; ++sub) {
      const int k0 = ci * E + sub * SE;
      float xv[MT][SE];
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int mm = min(m0 + m, M - 1);
        const float* xp = x + (size_t)mm * K + k0;
        if (xvec && k0 + SE <= K) {
#pragma unroll
          for (int v = 0; v < SE / 4; ++v) {
            const float4* src = reinterpret_cast<const float4*>(xp) + v;
            const float4 t = CHAIN ? ld_chain(src) : __ldg(src);
            xv[m][4 * v] = t.x; xv[m][4 * v + 1] = t.y; xv[m][4 * v + 2] = t.z; xv[m][4 * v + 3] = t.w;
          }
        } else {
#pragma unroll
          for (int j = 0; j < SE; ++j) xv[m][j] = (k0 + j < K) ? (CHAIN ? ld_chain(xp + j) : __ldg(xp + j)) : 0.0f;
        }
      }
#pragma unroll
      for (int r = 0; r < kRowsPerWarp; ++r) {
        float wf[SE];
        if (BITS == 32) {
          wf[0] = __uint_as_float(q[r].x); wf[1] = __uint_as_float(q[r].y);
          wf[2] = __uint_as_float(q[r].z); wf[3] = __uint_as_float(q[r].w);
        } else {
          decode8<BITS>(q[r], sub, wf);
        }
#pragma unroll
        for (int j = 0; j < SE; ++j)
#pragma unroll
          for (int m = 0; m < MT; ++m) acc[r][m] = fmaf(wf[j], xv[m][j], acc[r][m]);
      }
    }
  }

#pragma unroll
  for (int r = 0; r < kRowsPerWarp; ++r)
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      float v = acc[r][m];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      acc[r][m] = v;
    }
  if (lane == 0) {
#pragma unroll
    for (int r = 0; r < kRowsPerWarp; ++r) {
      const int n = n0 + r;
      if (n >= N) break;
      const float s = job.scale[n];
      const float b = job.bias ? job.bias[n] : 0.0f;
#pragma unroll
      for (int m = 0; m < MT; ++m)
        if (m0 + m < M) static_cast<float*>(job.out)[(size_t)(m0 + m) * N + n] = fmaf(acc[r][m], s, b);
    }
  }
}

// ---------------------------------------------------------------------------------------
// Five and more batch rows: a tiled float32 GEMM.  The kernel above reads and expands the weights once per four rows;
// here a block expands a slice of BN channels x 32 k once for BM rows.  A thread owns 4 channels x 4 rows (channels
// tx + BN/4 i, rows ty + BM/4 j) and works on four k at a time from float4 reads of the untransposed slices (row pitch 36
// floats: eight rows cover all banks); products of neighbouring k are packed float32 pairs.  Small tiles leave threads
// over: they form KG groups that take every KG-th slice of K, and where the tiles are fewer than the blocks the chip holds
// a cluster of blocks shares a tile in the same way.  Their sums meet in shared memory, in a fixed order.
// Bound by shared-memory reads (two cycles of them per cycle of multiplications) and, for small layers, by the latency of
// a slice.  Measured, 4 bits, before (kernel above) and now: 8192 x 777, 5 rows 57.5 -> 8.6 us, 256 rows 1486 -> 124;
// 1001 x 1999, 64 rows 138 -> 15; 70 x 8190, 5 rows 140 -> 10.
// Against the tensor-core path (pre-pass, zeroed y, atomics), 8 bits: 512 x 512, 64 rows 10.6 -> 5.6; 1024 x 1024, 64
// rows 10.6 -> 9.2, 128 rows 13.6 | 14.5; 2048 x 2048, 16 rows 10.9 -> 9.3, 32 rows 12.4 | 15.
// Against the integer kernel with its pre-pass, 8 rows, 4 bits: 2048 x 2048 16.6 -> 7.5; 4096 x 4096 16.6 | 18.3.
// ---------------------------------------------------------------------------------------
constexpr int kGemmThreads = 256, kGemmBK = 32, kGemmPitch = kGemmBK + 4;

template <int BN, int BM>
struct GemmTile {
  static constexpr int T = (BN / 4) * (BM / 4), KG = kGemmThreads / T;
  static constexpr int BUF = (BN + BM) * kGemmPitch;             // floats of one slice
  static constexpr int SMEM = KG * 2 * BUF * 4;
  static constexpr int RESIDENT = SMEM > 113 * 1024 ? 1 : 2;     // blocks of an SM
};

// LONG: see the sums below.
template <int BITS, int BN, int BM, bool LONG>
__global__ void __launch_bounds__(kGemmThreads, (LONG ? GemmTile<BN, BM>::RESIDENT : 0))
qlinear_gemm_kernel(LayerJob single, const LayerJob* __restrict__ jobs, int N, int K, int M, int cluster) {
  using G = GemmTile<BN, BM>;
  constexpr int T = G::T, KG = G::KG;
  constexpr int XS = BM * kGemmBK / T;                           // activations a thread fetches per slice
  constexpr int WG = BN * (kGemmBK / 8) / T;                     // granules of 8 weights
  constexpr int RAW = BITS / 4;                                  // words of a granule: 1, 2, 4, 8
  extern __shared__ __align__(16) float gm_sm[];
  const LayerJob job = jobs ? jobs[blockIdx.z] : single;
  chain_release();
  chain_wait();
  const int kg = threadIdx.x / T, t = threadIdx.x % T;
  const int tx = t % (BN / 4), ty = t / (BN / 4);
  const int rank = blockIdx.x % cluster;                         // of the blocks that share a tile
  const int n0 = (int)(blockIdx.x / cluster) * BN, m0 = blockIdx.y * BM;
  const size_t rb = (size_t)((K + 31) / 32 * 32) * BITS / 8;
  const float* x = static_cast<const float*>(job.in);
  float* const buf0 = gm_sm + kg * 2 * G::BUF;
  const int n_slices = (K + kGemmBK - 1) / kGemmBK;

  float xr[XS];
  uint32_t wr[WG][RAW];
  auto fetch = [&](int s) {
#pragma unroll
    for (int i = 0; i < XS; ++i) {
      const int idx = t + i * T, m = m0 + idx / kGemmBK, k = s * kGemmBK + idx % kGemmBK;
      xr[i] = (m < M && k < K) ? ld_chain(x + (size_t)m * K + k) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < WG; ++i) {
      const int idx = t + i * T, n = n0 + idx / (kGemmBK / 8), gk = s * (kGemmBK / 8) + idx % (kGemmBK / 8);
#pragma unroll
      for (int j = 0; j < RAW; ++j) wr[i][j] = 0u;
      if (n < N) {                                               // rows are padded with zeros to whole slices
        const uint8_t* src = job.w + (size_t)n * rb + (size_t)gk * BITS;
        if (BITS == 4) {
          wr[i][0] = __ldg(reinterpret_cast<const uint32_t*>(src));
        } else if (BITS == 8) {
          const uint2 q = __ldg(reinterpret_cast<const uint2*>(src));
          wr[i][0] = q.x; wr[i][RAW > 1 ? 1 : 0] = q.y;
        } else {
#pragma unroll
          for (int j = 0; j < RAW / 4; ++j) {
            const uint4 q = __ldg(reinterpret_cast<const uint4*>(src) + j);
            wr[i][4 * j] = q.x; wr[i][4 * j + 1] = q.y; wr[i][4 * j + 2] = q.z; wr[i][4 * j + 3] = q.w;
          }
        }
      }
    }
  };
  auto stash = [&](int b) {
    float* ws = buf0 + b * G::BUF;
    float* xs = ws + BN * kGemmPitch;
#pragma unroll
    for (int i = 0; i < XS; ++i) {
      const int idx = t + i * T;
      xs[(idx / kGemmBK) * kGemmPitch + idx % kGemmBK] = xr[i];
    }
#pragma unroll
    for (int i = 0; i < WG; ++i) {
      const int idx = t + i * T;
      float f[8];
      if (BITS == 32) {
#pragma unroll
        for (int j = 0; j < 8; ++j) f[j] = __uint_as_float(wr[i][j < RAW ? j : 0]);
      } else if (BITS == 16) {
        decode8<16>(make_uint4(wr[i][0], wr[i][RAW > 1 ? 1 : 0], wr[i][RAW > 2 ? 2 : 0], wr[i][RAW > 3 ? 3 : 0]), 0, f);
      } else {
        decode8<BITS>(make_uint4(wr[i][0], wr[i][RAW > 1 ? 1 : 0], 0u, 0u), 0, f);
      }
      float* dst = ws + (idx / (kGemmBK / 8)) * kGemmPitch + (idx % (kGemmBK / 8)) * 8;
      *reinterpret_cast<float4*>(dst) = make_float4(f[0], f[1], f[2], f[3]);
      *reinterpret_cast<float4*>(dst + 4) = make_float4(f[4], f[5], f[6], f[7]);
    }
  };
  auto group_sync = [&]() {                                      // the threads of this K group
    if (T == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + kg), "n"(T) : "memory");
  };

  // LONG: a sum per slice, then the sum of those.  One chain over all slices of a group had up to three times the rounding
  // error of the kernel above, whose lanes add K / 32 products each (8192 x 777, 256 rows: 3.5e-7 of the result's norm
  // against 1.1e-7, now 1.2e-7).  It costs 1 to 5 % of the time, so it runs only where the chain, K / 2 over the groups of
  // the tile, is longer than that lane's and than two slices.
  float sum[4][4];                                               // [channel][row]
  uint64_t acc[4][4];                                            // sums over even and over odd k; LONG: of one slice
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) { sum[i][j] = 0.f; acc[i][j] = 0ull; }
  auto add_up = [&]() {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) { const float2 f = unpack2(acc[i][j]); sum[i][j] += f.x + f.y; }
  };
  int b = 0;
  const int first = rank * KG + kg, step = cluster * KG;
  if (first < n_slices) { fetch(first); stash(0); }
  for (int s = first; s < n_slices; s += step) {
    group_sync();                                                // slice s is in place; slice s - step's buffer is free
    if (s + step < n_slices) fetch(s + step);
    const float* ws = buf0 + b * G::BUF;
    const float* xs = ws + BN * kGemmPitch;
#pragma unroll
    for (int k = 0; k < kGemmBK; k += 4) {
      ulonglong2 w[4], v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = *reinterpret_cast<const ulonglong2*>(ws + (tx + i * (BN / 4)) * kGemmPitch + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = *reinterpret_cast<const ulonglong2*>(xs + (ty + j * (BM / 4)) * kGemmPitch + k);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma2(w[i].y, v[j].y, LONG && k == 0 ? mul2(w[i].x, v[j].x) : fma2(w[i].x, v[j].x, acc[i][j]));
    }
    if (LONG) add_up();
    b ^= 1;
    if (s + step < n_slices) stash(b);
  }
  if (!LONG) add_up();
  auto put = [&](int i, float v) {
    const int n = n0 + tx + (i >> 2) * (BN / 4), m = m0 + ty + (i & 3) * (BM / 4);
    if (n < N && m < M) static_cast<float*>(job.out)[(size_t)m * N + n] = fmaf(v, job.scale[n], job.bias ? job.bias[n] : 0.0f);
  };
  if (KG == 1 && cluster == 1) {
#pragma unroll
    for (int i = 0; i < 16; ++i) put(i, sum[i >> 2][i & 3]);
    return;
  }
  __syncthreads();                                               // every group is through with its slices
  float* red = gm_sm;                                            // [group][16][T]; group 0's part then holds the block's sums
#pragma unroll
  for (int i = 0; i < 16; ++i) red[(kg * 16 + i) * T + t] = sum[i >> 2][i & 3];
  __syncthreads();
  for (int i = kg; i < 16; i += KG) {                            // each group adds up a part of the 16 sums of a position
    float v = 0.f;
#pragma unroll
    for (int q = 0; q < KG; ++q) v += red[(q * 16 + i) * T + t];
    if (cluster == 1) put(i, v);
    else red[i * T + t] = v;
  }
  if (cluster > 1) {
    asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");   // releases: the block's sums are in place
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    for (int i = rank * KG + kg; i < 16; i += step) {
      float v = 0.f;
      const uint32_t mine = smem_u32(red + i * T + t);
      for (int q = 0; q < cluster; ++q) {
        uint32_t theirs;
        float part;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(theirs) : "r"(mine), "r"(q));
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(part) : "r"(theirs) : "memory");
        v += part;
      }
      put(i, v);
    }
    asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");   // no block leaves while another reads its sums
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  }
}

// Clusters of `size` blocks that the device holds at a time: they form inside a GPC, so fewer than the SMs would hold one by
// one.  (2228 x 6400, 16 bits, 5 rows: 35 clusters of four ran in two waves, 31.4 us.)  Asked once per kernel, device and size.
template <typename K>
aiq_status_t resident_clusters(K* kernel, int smem, int size, std::atomic<int> (&known)[64], int* out) {
  int dev = 0;
  AIQ_CUDA_TRY(cudaGetDevice(&dev));
  const bool cached = dev >= 0 && dev < 64;
  *out = cached ? known[dev].load(std::memory_order_acquire) : 0;
  if (*out) return AIQ_OK;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(size); cfg.blockDim = dim3(kGemmThreads); cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = size; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  AIQ_CUDA_TRY(cudaOccupancyMaxActiveClusters(out, kernel, &cfg));
  if (cached) known[dev].store(*out, std::memory_order_release);
  return AIQ_OK;
}

template <int BITS, int BN, int BM>
aiq_status_t launch_gemm_tile(const LaunchScope& scope, const LayerJob* jobs_dev, const LayerJob& single, int n_jobs, int N, int K, int M,
                              int n_sms, cudaStream_t s, int fixed_cluster) {
  using G = GemmTile<BN, BM>;
  const dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, n_jobs);
  const long long blocks = (long long)grid.x * grid.y * grid.z;
  const int n_slices = (K + kGemmBK - 1) / kGemmBK;
  AIQ_ENSURE_DYNAMIC_SMEM((qlinear_gemm_kernel<BITS, BN, BM, false>), (G::SMEM));
  // blocks per tile: doubled while all blocks stay resident and a group of threads has more than one slice
  int cluster = fixed_cluster ? fixed_cluster : 1;
  while (!fixed_cluster && cluster < 8 && blocks * cluster * 2 <= G::RESIDENT * n_sms && n_slices > cluster * G::KG) {
    const int next = cluster * 2;
    if (G::RESIDENT == 1) {                                      // with two blocks per SM a second wave has not been seen
      static std::atomic<int> known[3][64];
      int fit = 0;
      if (aiq_status_t st = resident_clusters(qlinear_gemm_kernel<BITS, BN, BM, false>, G::SMEM, next, known[next >> 2], &fit)) return st;
      if (blocks > fit) break;
    }
    cluster = next;
  }
  auto launch = [&](auto kernel) {
    return launch_chained_cluster(scope.chain, cluster, kernel, dim3(grid.x * cluster, grid.y, grid.z), dim3(kGemmThreads), G::SMEM, s,
                                  single, jobs_dev, N, K, M, cluster);
  };
  if (!jobs_dev && cluster * G::KG < 16 && n_slices > 2 * cluster * G::KG) {
    AIQ_ENSURE_DYNAMIC_SMEM((qlinear_gemm_kernel<BITS, BN, BM, true>), (G::SMEM));
    AIQ_CUDA_TRY(launch(qlinear_gemm_kernel<BITS, BN, BM, true>));
  } else {
    AIQ_CUDA_TRY(launch(qlinear_gemm_kernel<BITS, BN, BM, false>));
  }
  return AIQ_OK;
}

// Five to eight rows on the kernel of four, twice, instead of the tile of 64 channels.  Measured, gemm | plain: short rows
// (16 bits 512 x 512 5.3 | 3.7 us, 1280 x 320 5.1 | 3.9, 1000 x 1280 7.0 | 5.9, 32 bits 901 x 288 5.6 | 3.6, 8 bits 330 x 288 5.1 | 3.5; but 623 x
// 212, 8 bits, 3.7 | 4.2, 2629 x 139 3.6 | 6.1); 16 bits, where a large layer gives every SM enough and its rows are aligned
// (4096 x 4096 19.6 | 17.6, 5823 x 6184 52.3 | 45.9, 8192 x 8192 68.9 | 64.8; but 2048 x 8192 19.8 | 29.4); 32 bits, where the
// tiles occupy half to two thirds of the SMs, one each (5823 x 6184 57.0 | 40.5, 6223 x 1492 16.8 | 13.0; 7522 x 4384 43.2 | 51.4).
bool plain_rows8(int bits, int N, int K, int M, int n_sms) {
  if (M > 8 || bits == 4) return false;
  if (K >= 256 && K <= 512 && N <= 1536) return true;
  if (bits == 16 && K <= 1280 && N >= 768 && N <= 1536) return true;
  if (K % 4) return false;
  if (bits == 16) return N > 16 * n_sms && (long long)N * K >= (1ll << 24);
  const int tiles = (N + 63) / 64;
  return bits == 32 && 2 * tiles > n_sms && 3 * tiles <= 2 * n_sms;
}

template <int BITS>
aiq_status_t launch_bits(const LayerJob* jobs_dev, const LayerJob& single, int n_jobs, int N, int K,
                         int M, cudaStream_t s) {
  DeviceProps props;
  if (aiq_status_t st = current_device_props(&props)) return st;
  const int gx = (N + kWarps * kRowsPerWarp - 1) / (kWarps * kRowsPerWarp);
  LaunchScope scope(AIQ_KERNEL_QLINEAR, s, 2.0 * M * N * K * n_jobs,
                    n_jobs * ((double)N * row_bytes(K, BITS) + 4.0 * N + 4.0 * M * ((double)K + N)));
  if (jobs_dev) {
    // A classifier inside a model: one tile, and a split of K that depends on the layer alone, so that an image's logits
    // depend neither on the batch around it nor on the number of jobs.
    const int n_tiles = (N + 31) / 32, n_slices = (K + kGemmBK - 1) / kGemmBK;
    int cluster = 1;
    while (cluster < 8 && n_tiles * cluster * 2 <= 64 && n_slices > cluster * GemmTile<32, 16>::KG) cluster *= 2;
    if (aiq_status_t st = launch_gemm_tile<BITS, 32, 16>(scope, jobs_dev, single, n_jobs, N, K, M, props.n_sms, s, cluster)) return st;
  } else if (M > 4 && !plain_rows8(BITS, N, K, M, props.n_sms)) {
    // The largest tile that still gives every SM a block; smaller ones split K over more thread groups.  The tile of 8 rows
    // leaves out the work of rows that are not there (8191 x 8191, 5 rows, 4 bits: 72 us against 94 with the tile of 16).
    auto blocks = [&](int bn, int bm) { return (long long)((N + bn - 1) / bn) * ((M + bm - 1) / bm); };
    auto args = [&](auto launch) { return launch(scope, nullptr, single, 1, N, K, M, props.n_sms, s, 0); };
    aiq_status_t st;
    if (M > 32 && blocks(64, 64) >= props.n_sms) st = args(launch_gemm_tile<BITS, 64, 64>);
    else if (M > 16 && blocks(64, 32) >= props.n_sms) st = args(launch_gemm_tile<BITS, 64, 32>);
    else if (M > 16 && blocks(32, 32) >= props.n_sms / 2) st = args(launch_gemm_tile<BITS, 32, 32>);
    else if (M <= 8) st = args(launch_gemm_tile<BITS, 64, 8>);
    else st = args(launch_gemm_tile<BITS, 32, 16>);
    if (st != AIQ_OK) return st;
  } else {
    // Chained, but for two kinds of launch.  The blocks of the next call settle on the SMs that this one leaves idle; where
    // those are less than half, two on one, and a long stream of three or four rows then waits for them (16 bits, 4 rows: 4096
    // x 4096 18.2 us chained, 16.4 not, 3063 x 4147 40.9 | 35.0; 4096 x 1024 6.8 | 8.2, 8192 x 4096 19.5 | 20.7).  And rows of x
    // that are not 16-byte aligned are read by element, for which the read-only path is the faster one (32 bits, 2 rows: 8099 x
    // 8023 79 | 62, 543 x 3814 27.7 | 26.0, but 723 x 1593 13.3 | 13.8; 16 bits, 1 / 2 rows: 47.6 / 65 | 41.5 / 49.4, but 543 x 3814 16.0 / 20.2 | 18.1 / 22.2).
    const bool large = (long long)N * row_bytes(K, BITS) > (16ll << 20);
    const bool by_element = (K & 3) != 0 || (((uintptr_t)single.in) & 15) != 0;
    const bool chain = M > 4 || (M > 2 ? !(large && 2 * gx > props.n_sms && gx < props.n_sms) : !(by_element && (BITS == 32 ? M == 2 && K >= 3500 : large)));
    const dim3 grid(gx, M > 4 ? 2 : 1);
    auto launch = [&](auto kernel) { return launch_chained(chain && scope.chain, kernel, grid, dim3(kWarps * 32), 0, s, single, N, K, M); };
    auto pick = [&](auto chained) {
      constexpr bool CH = decltype(chained)::value;
      return M == 1 ? launch(qlinear_kernel<BITS, 1, CH>) : M == 2 ? launch(qlinear_kernel<BITS, 2, CH>) : launch(qlinear_kernel<BITS, 4, CH>);
    };
    AIQ_CUDA_TRY(chain && scope.chain ? pick(std::true_type()) : pick(std::false_type()));
  }
  AIQ_LAUNCH_CHECK("qlinear");
  return AIQ_OK;
}

}  // namespace

aiq_status_t launch_qlinear(const LayerJob* jobs_dev, const LayerJob* single_host, int n_jobs, int N,
                            int K, int M, cudaStream_t s) {
  LayerJob single = {};
  int bits;
  if (jobs_dev) {
    // all jobs of one launch share a bit-width: the caller groups them
    bits = single_host->bits;
  } else {
    single = *single_host;
    bits = single.bits;
  }
  switch (bits) {
    case 4: return launch_bits<4>(jobs_dev, single, n_jobs, N, K, M, s);
    case 8: return launch_bits<8>(jobs_dev, single, n_jobs, N, K, M, s);
    case 16: return launch_bits<16>(jobs_dev, single, n_jobs, N, K, M, s);
    case 32: return launch_bits<32>(jobs_dev, single, n_jobs, N, K, M, s);
  }
  return set_error(AIQ_ERR_UNSUPPORTED_BITS, "qlinear: bits=%d", bits);
}

}  // namespace aiq

// Up to 2^26 products the one launch of the float32 kernel (from five rows on) beats the pre-pass and the atomics of the
// kernels below; see the figures at qlinear_gemm_kernel.  Long rows leave it few tiles with many slices each (128 x 8192,
// 40 rows: 14.2 us against 7.6 on the tensor cores): from K = 4096 up to 2^24.  Below 32 bits the tensor cores take a part
// of that range too, with halves that lose next to nothing (error 1e-7 to 3.5e-7 of the result's norm): K > 4096 from 2^22 on
// (64 x 8192, 12 rows, 8 bits: 10.1 | 8.3), K >= 1024 from 2^25 on (1000 x 1280, 40 rows, 8 bits: 12.5 | 8.3; 1360 x 3000, 9
// rows 12.6 | 11.1; 2048 x 2048, 9 rows 9.6 | 8.3).
static bool small_gemm(int N, int K, int bits, int M) {
  const long long products = (long long)N * K * M;
  if (M <= 4 || products > (K > 4096 && M > 8 ? 1ll << 24 : 1ll << 26)) return false;
  return bits == 32 || M <= 8 || !(products > (K > 4096 ? 1ll << 22 : K >= 1024 ? 1ll << 25 : 1ll << 26));
}

// The kernel of a call, and of the size query: SCRATCH_* ones need the workspace, and without it GEMV or PLAIN runs in their place.
enum QlinearPath { QL_PLAIN, QL_GEMV, QL_SCRATCH_MMA, QL_SCRATCH_TC };
static QlinearPath qlinear_path(int N, int K, int bits, int M) {
  // 4 bits above 3 x 2^25 weights: the kernel of up to four rows needs twice the MMAs of the one with scratch (its weights are
  // the narrow operand) and no longer streams at the memory's rate.  One / four rows, on the device: 16384 x 8192 21.6 / 26.4
  // us there, 18.7 / 23.7 here; 32768 x 8192 41.0 / 46.5 | 30.0 / 40.0; at 8192 x 8192 calls take 12.2 / 16.9 us and 14.2 / 16.6.
  if (bits == 4 && M <= 4 && (long long)N * K > (3ll << 25) && aiq::qlinear_mma_applicable(N, K, bits, M)) return QL_SCRATCH_MMA;
  if (aiq::qlinear_gemv_applicable(N, K, bits, M)) return QL_GEMV;
  if (small_gemm(N, K, bits, M)) return QL_PLAIN;
  if (aiq::qlinear_tc_applicable(N, K, bits, M)) return QL_SCRATCH_TC;
  return aiq::qlinear_mma_applicable(N, K, bits, M) ? QL_SCRATCH_MMA : QL_PLAIN;
}

extern "C" size_t aiq_qlinear_workspace_bytes(int N, int K, int bits, int M) {
  if (N <= 0 || K <= 0 || M <= 0) return 0;
  switch (qlinear_path(N, K, bits, M)) {
    case QL_SCRATCH_TC: return aiq::qlinear_tc_workspace_bytes(K, M) + 16;   // + status word
    case QL_SCRATCH_MMA: return aiq::qlinear_mma_workspace_bytes(K, M);
    // the kernel of up to four rows touches none; callers that size one buffer by the smallest call keep their answer
    case QL_GEMV: return aiq::qlinear_mma_applicable(N, K, bits, M) ? aiq::qlinear_mma_workspace_bytes(K, M) : 0;
    default: return 0;
  }
}

extern "C" aiq_status_t aiq_qlinear(const void* packed, const float* scales, const float* bias, int N,
                                    int K, int bits, const float* x, int M, float* y, void* workspace,
                                    size_t workspace_bytes, void* stream) {
  if (!aiq::bits_ok(bits)) return aiq::set_error(AIQ_ERR_UNSUPPORTED_BITS, "aiq_qlinear: bits=%d", bits);
  if (!packed || !scales || !x || !y) return aiq::set_error(AIQ_ERR_INVALID_ARG, "aiq_qlinear: null pointer");
  if (N <= 0 || K <= 0 || M <= 0)
    return aiq::set_error(AIQ_ERR_INVALID_ARG, "aiq_qlinear: N=%d K=%d M=%d", N, K, M);
  if (((uintptr_t)packed) & 15)
    return aiq::set_error(AIQ_ERR_INVALID_ARG, "aiq_qlinear: packed not 16-byte aligned");
  aiq_status_t st = aiq::check_device_sm100();
  if (st != AIQ_OK) return st;
  aiq::LayerJob job = {};
  job.in = x;
  job.out = y;
  job.w = static_cast<const uint8_t*>(packed);
  job.scale = scales;
  job.bias = bias;
  job.bits = bits;
  // a misaligned workspace is refused wherever a kernel with scratch exists for the shape, whichever kernel then runs
  if (workspace && (((uintptr_t)workspace) & 15) && (aiq::qlinear_tc_applicable(N, K, bits, M) || aiq::qlinear_mma_applicable(N, K, bits, M)))
    return aiq::set_error(AIQ_ERR_INVALID_ARG, "aiq_qlinear: workspace not 16-byte aligned");
  const QlinearPath path = qlinear_path(N, K, bits, M);
  // the tensor-core kernels need scratch for the converted activations
  if (path == QL_SCRATCH_TC && workspace) {
    const size_t scratch = aiq::qlinear_tc_workspace_bytes(K, M);
    if (workspace_bytes >= scratch + 16) {
      // device status word behind the scratch: 0 (set by the pre-pass), or 1 once a bounded wait of the kernel expired
      int32_t* status = reinterpret_cast<int32_t*>(static_cast<uint8_t*>(workspace) + scratch);
      return aiq::launch_qlinear_tc(job, N, K, M, workspace, status, (cudaStream_t)stream);
    }
  }
  if (path == QL_SCRATCH_MMA && workspace && workspace_bytes >= aiq::qlinear_mma_workspace_bytes(K, M))
    return aiq::launch_qlinear_mma(job, N, K, M, workspace, (cudaStream_t)stream);
  if (aiq::qlinear_gemv_applicable(N, K, bits, M)) return aiq::launch_qlinear_gemv(job, N, K, M, (cudaStream_t)stream);
  return aiq::launch_qlinear(nullptr, &job, 1, N, K, M, (cudaStream_t)stream);
}
