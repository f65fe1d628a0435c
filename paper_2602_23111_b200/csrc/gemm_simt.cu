// General FMA GEMM: any leading dimensions and alignments, fp32 / bf16 elements, fp32
// accumulation.  It serves the fp32 storage path, the small dense products of the basis fit
// and any operand layout the TMA-fed tensor-core kernels cannot take.
//
// What bounds it: the products of an fp32 layer are small (2048 x 512 by 512 x 32 is 67 Mflop,
// 1 us of the chip's FMA rate) and one of their dimensions is the narrow k + r, so tiles alone
// leave most SMs idle and each of them with a serial walk over K.  K is therefore cut twice:
// among the thread groups of a CTA (SL slices of BK rows per step, summed through shared memory)
// and among the CTAs of a cluster (2, 4 or 8 pieces, summed through distributed shared memory,
// so no workspace is needed).  Both sums run in a fixed order.  Measured against the 64 x 64 tiles
// with one serial walk over K that this replaced (fp32 layer, N = 2048, d = d_out = 512, k = r = 16):
// compress and weight gradient 207 -> 32 us, the refit step 1089 -> 642 us by this alone (23 and 434 us with
// what the launches and the rest of the fit have gained since).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "per_device.h"
#include "ptx.cuh"

namespace prac {
namespace {

constexpr int BK = 16, THREADS = 256;

struct DevGemm {
  int M, N, K;
  const void* A; long long lda; int bf16_a, vec_a;      // vec: groups of four elements are aligned
  const void* B; long long ldb; int bf16_b, vec_b;
  void* C; long long ldc; int bf16_c, vec_c;
  float alpha, beta;
  int kscale_from; float kscale;
  int tiles_n;
  int symmetric;        // C = A^T A: only the tiles that reach the upper triangle, mirrored
  int parts;            // CTAs per cluster: each takes every parts-th step along K
  const int* run_if; int run_if_mask;   // optional: do nothing unless *run_if & run_if_mask
  long long ext_a, ext_b, ext_c;        // elements the three buffers span (used by the bounds-checking build)
};

__device__ __forceinline__ float bf16_bits(uint32_t lo16) { return __uint_as_float(lo16 << 16); }

// Elements (slow, fast .. fast + 3) of a row-major matrix, zeros outside slow_end x fast_end.  As they
// are stored (four bf16 in x and y): nothing touches a fetched value before it is needed, or the loads of
// a step would wait for one another.
__device__ __forceinline__ float4 load4(const void* base, int bf16, int vec, long long ld, long long ext, int slow, int fast,
                                        int slow_end, int fast_end) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (slow >= slow_end || fast >= fast_end) return v;
  const long long idx = static_cast<long long>(slow) * ld + fast;
  if (vec && fast + 4 <= fast_end && PRAC_IN(idx + 3, ext)) {
    if (!bf16) return *reinterpret_cast<const float4*>(static_cast<const float*>(base) + idx);
    const float2 w = *reinterpret_cast<const float2*>(static_cast<const __nv_bfloat16*>(base) + idx);
    v.x = w.x; v.y = w.y;
    return v;
  }
  if (!bf16) {
    const float* p = static_cast<const float*>(base) + idx;
    if (PRAC_IN(idx, ext)) v.x = *p;
    if (fast + 1 < fast_end && PRAC_IN(idx + 1, ext)) v.y = p[1];
    if (fast + 2 < fast_end && PRAC_IN(idx + 2, ext)) v.z = p[2];
    if (fast + 3 < fast_end && PRAC_IN(idx + 3, ext)) v.w = p[3];
  } else {
    const unsigned short* p = static_cast<const unsigned short*>(base) + idx;
    uint32_t e[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (fast + i < fast_end && PRAC_IN(idx + i, ext)) e[i] = p[i];
    v.x = __uint_as_float(e[0] | (e[1] << 16));
    v.y = __uint_as_float(e[2] | (e[3] << 16));
  }
  return v;
}
__device__ __forceinline__ float4 as_floats(const float4& v, int bf16) {
  if (!bf16) return v;
  const uint32_t a = __float_as_uint(v.x), b = __float_as_uint(v.y);
  return make_float4(bf16_bits(a & 0xffffu), __uint_as_float(a & 0xffff0000u), bf16_bits(b & 0xffffu), __uint_as_float(b & 0xffff0000u));
}

// One CTA: a TM x TN tile of C over its share of K.  SL groups of 256 / SL threads; group g of CTA
// `part` takes the K rows [(step * parts + part) * SL + g] * BK ... + BK.  A thread owns 4 MI rows
// (blocks of four, 4 TY apart) by 8 columns (two blocks of four, 4 TX apart).
template <int TM, int TN, int SL>
struct Shape {
  static constexpr int GT = THREADS / SL;              // threads of a group
  static constexpr int TX = TN / 8, TY = GT / TX;      // a group's threads along N and M
  static constexpr int MI = TM / (4 * TY);             // row blocks per thread
  static constexpr int PA = TM + 4, PB = TN + 4;       // pitches of the staged operands [k][m], [k][n]
  static constexpr int STAGE = BK * (PA + PB);         // floats of one buffer of one group
  static constexpr int RED_P = TN + 4;                 // pitch of the tiles the slices are summed from
  static constexpr int FLOATS_LOOP = 2 * SL * STAGE, FLOATS_RED = SL * TM * RED_P;
  static constexpr int SMEM = (FLOATS_LOOP > FLOATS_RED ? FLOATS_LOOP : FLOATS_RED) * 4;
  static constexpr int QA = TM * BK / 4 / GT, QB = TN * BK / 4 / GT;   // groups of four a thread fetches per step
  static_assert(TY * TX == GT && MI * 4 * TY == TM && QA * 4 * GT == TM * BK && QB * 4 * GT == TN * BK, "thread layout");
};

template <int TM, int TN, int SL, bool TRANS_A, bool TRANS_B>
__global__ void __launch_bounds__(THREADS, 2) gemm_simt_kernel(const DevGemm g) {
  using S = Shape<TM, TN, SL>;
  extern __shared__ __align__(16) float sm[];
  grid_dep_wait();
  if (g.run_if != nullptr && (*reinterpret_cast<const volatile int*>(g.run_if) & g.run_if_mask) == 0) return;
  const int group = threadIdx.x / S::GT, t = threadIdx.x % S::GT;
  const int tx = t % S::TX, ty = t / S::TX;
  const int part = blockIdx.x % g.parts;
  int tile = blockIdx.x / g.parts, ti, tj;
  if (!g.symmetric) {
    ti = tile / g.tiles_n; tj = tile % g.tiles_n;
  } else {                                   // square tiles, row ti keeps the columns tj >= ti
    ti = 0;
    while (tile >= g.tiles_n - ti) { tile -= g.tiles_n - ti; ++ti; }
    tj = ti + tile;
  }
  const int m0 = ti * TM, n0 = tj * TN;
  float* stage = sm + group * 2 * S::STAGE;

  float4 fa[S::QA], fb[S::QB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int e = 0; e < S::QA; ++e) {
      const int q = t + S::GT * e;
      if (!TRANS_A) fa[e] = load4(g.A, g.bf16_a, g.vec_a, g.lda, g.ext_a, m0 + (q >> 2), k0 + (q & 3) * 4, g.M, g.K);
      else fa[e] = load4(g.A, g.bf16_a, g.vec_a, g.lda, g.ext_a, k0 + q / (TM / 4), m0 + (q % (TM / 4)) * 4, g.K, g.M);
    }
#pragma unroll
    for (int e = 0; e < S::QB; ++e) {
      const int q = t + S::GT * e;
      if (TRANS_B) fb[e] = load4(g.B, g.bf16_b, g.vec_b, g.ldb, g.ext_b, n0 + (q >> 2), k0 + (q & 3) * 4, g.N, g.K);
      else fb[e] = load4(g.B, g.bf16_b, g.vec_b, g.ldb, g.ext_b, k0 + q / (TN / 4), n0 + (q % (TN / 4)) * 4, g.K, g.N);
    }
  };
  auto put = [&](float* s, int k0) {         // what fetch(k0) brought
#pragma unroll
    for (int e = 0; e < S::QA; ++e) {
      const int q = t + S::GT * e;
      float4 v = as_floats(fa[e], g.bf16_a);
      if (!TRANS_A) {
        const int kq = k0 + (q & 3) * 4;
        if (kq + 3 >= g.kscale_from) {
          if (kq >= g.kscale_from) v.x *= g.kscale;
          if (kq + 1 >= g.kscale_from) v.y *= g.kscale;
          if (kq + 2 >= g.kscale_from) v.z *= g.kscale;
          v.w *= g.kscale;
        }
        float* o = s + (q & 3) * 4 * S::PA + (q >> 2);
        o[0] = v.x; o[S::PA] = v.y; o[2 * S::PA] = v.z; o[3 * S::PA] = v.w;
      } else {
        if (k0 + q / (TM / 4) >= g.kscale_from) { v.x *= g.kscale; v.y *= g.kscale; v.z *= g.kscale; v.w *= g.kscale; }
        *reinterpret_cast<float4*>(s + (q / (TM / 4)) * S::PA + (q % (TM / 4)) * 4) = v;
      }
    }
    float* sb = s + BK * S::PA;
#pragma unroll
    for (int e = 0; e < S::QB; ++e) {
      const int q = t + S::GT * e;
      const float4 v = as_floats(fb[e], g.bf16_b);
      if (TRANS_B) {
        float* o = sb + (q & 3) * 4 * S::PB + (q >> 2);
        o[0] = v.x; o[S::PB] = v.y; o[2 * S::PB] = v.z; o[3 * S::PB] = v.w;
      } else {
        *reinterpret_cast<float4*>(sb + (q / (TN / 4)) * S::PB + (q % (TN / 4)) * 4) = v;
      }
    }
  };

  float acc[S::MI][4][8];
#pragma unroll
  for (int b = 0; b < S::MI; ++b)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[b][i][j] = 0.f;

  // every group of every CTA of the cluster walks the same number of steps (zeros past K)
  const int per_step = g.parts * SL * BK;
  const int steps = (g.K + per_step - 1) / per_step;
  const int first = (part * SL + group) * BK;
  fetch(first);
  put(stage, first);
  __syncthreads();
  for (int st = 0; st < steps; ++st) {
    if (st + 1 < steps) fetch(first + (st + 1) * per_step);
    const float* s = stage + (st & 1) * S::STAGE;
    const float* sb = s + BK * S::PA;
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[S::MI][4], b[8];
#pragma unroll
      for (int i = 0; i < S::MI; ++i)
        *reinterpret_cast<float4*>(a[i]) = *reinterpret_cast<const float4*>(s + kk * S::PA + 4 * ty + 4 * S::TY * i);
      *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(sb + kk * S::PB + 4 * tx);
      *reinterpret_cast<float4*>(b + 4) = *reinterpret_cast<const float4*>(sb + kk * S::PB + 4 * tx + 4 * S::TX);
#pragma unroll
      for (int r = 0; r < S::MI; ++r)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[r][i][j] = fmaf(a[r][i], b[j], acc[r][i][j]);
    }
    if (st + 1 < steps) put(stage + ((st + 1) & 1) * S::STAGE, first + (st + 1) * per_step);
    __syncthreads();
  }

  // ---- the slices of this CTA, then those of the cluster, added in order through shared memory
  // (the last barrier of the loop: nobody reads the staged operands any more)
  float* red = sm + group * TM * S::RED_P;
#pragma unroll
  for (int r = 0; r < S::MI; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float* o = red + (4 * ty + 4 * S::TY * r + i) * S::RED_P + 4 * tx;
      *reinterpret_cast<float4*>(o) = make_float4(acc[r][i][0], acc[r][i][1], acc[r][i][2], acc[r][i][3]);
      *reinterpret_cast<float4*>(o + 4 * S::TX) = make_float4(acc[r][i][4], acc[r][i][5], acc[r][i][6], acc[r][i][7]);
    }
  __syncthreads();
  constexpr int ROW4 = TN / 4;
  if (SL > 1 && g.parts > 1) {
    for (int q = threadIdx.x; q < TM * ROW4; q += THREADS) {
      float* o = sm + (q / ROW4) * S::RED_P + (q % ROW4) * 4;
      float4 v = *reinterpret_cast<const float4*>(o);
#pragma unroll
      for (int h = 1; h < SL; ++h) {
        const float4 w = *reinterpret_cast<const float4*>(o + h * TM * S::RED_P);
        v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
      }
      *reinterpret_cast<float4*>(o) = v;
    }
  }
  if (g.parts > 1) ptx::cluster_sync_all();
  const int rows = TM / g.parts;             // this CTA closes the rows [part * rows, + rows) of the tile
  if (g.vec_c && !g.symmetric) {             // fp32 rows on the 16-byte grid: four columns per thread
    for (int q = threadIdx.x; q < rows * ROW4; q += THREADS) {
      const int row = part * rows + q / ROW4, col = (q % ROW4) * 4;
      const float* o = sm + row * S::RED_P + col;
      float4 v;
      if (g.parts > 1) {
        v = ptx::cluster_ld_f32x4(ptx::cluster_addr(o, 0));
        for (int h = 1; h < g.parts; ++h) {
          const float4 w = ptx::cluster_ld_f32x4(ptx::cluster_addr(o, h));
          v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
        }
      } else {
        v = *reinterpret_cast<const float4*>(o);
#pragma unroll
        for (int h = 1; h < SL; ++h) {
          const float4 w = *reinterpret_cast<const float4*>(o + h * TM * S::RED_P);
          v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
        }
      }
      const int gi = m0 + row, gj = n0 + col;
      if (gi >= g.M || gj >= g.N) continue;
      const long long idx = static_cast<long long>(gi) * g.ldc + gj;
      float e[4] = {g.alpha * v.x, g.alpha * v.y, g.alpha * v.z, g.alpha * v.w};
      float* c = static_cast<float*>(g.C) + idx;
      if (gj + 4 <= g.N && PRAC_IN(idx + 3, g.ext_c)) {
        if (g.beta != 0.f) {
          const float4 old = *reinterpret_cast<const float4*>(c);
          e[0] = fmaf(g.beta, old.x, e[0]); e[1] = fmaf(g.beta, old.y, e[1]);
          e[2] = fmaf(g.beta, old.z, e[2]); e[3] = fmaf(g.beta, old.w, e[3]);
        }
        *reinterpret_cast<float4*>(c) = make_float4(e[0], e[1], e[2], e[3]);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (gj + i >= g.N || !PRAC_IN(idx + i, g.ext_c)) continue;
          c[i] = g.beta != 0.f ? fmaf(g.beta, c[i], e[i]) : e[i];
        }
      }
    }
  } else {
    // one column per thread, so that a warp's stores to a row off the grid are one run of addresses
    for (int q = threadIdx.x; q < rows * TN; q += THREADS) {
      const int row = part * rows + q / TN, col = q % TN;
      const int gi = m0 + row, gj = n0 + col;
      const float* o = sm + row * S::RED_P + col;
      float v;
      if (g.parts > 1) {
        v = ptx::cluster_ld_f32(ptx::cluster_addr(o, 0));
        for (int h = 1; h < g.parts; ++h) v += ptx::cluster_ld_f32(ptx::cluster_addr(o, h));
      } else {
        v = *o;
#pragma unroll
        for (int h = 1; h < SL; ++h) v += o[h * TM * S::RED_P];
      }
      if (gi >= g.M || gj >= g.N) continue;
      const long long idx = static_cast<long long>(gi) * g.ldc + gj;
      if (!PRAC_IN(idx, g.ext_c)) continue;
      float e = g.alpha * v;
      if (g.symmetric) {
        // (a diagonal tile gives its upper triangle to both halves: the result is exactly symmetric)
        if (gi > gj) continue;
        float* c = static_cast<float*>(g.C);
        c[idx] = e;
        c[static_cast<long long>(gj) * g.ldc + gi] = e;
      } else if (g.bf16_c) {
        __nv_bfloat16* c = static_cast<__nv_bfloat16*>(g.C) + idx;
        if (g.beta != 0.f) e = fmaf(g.beta, __bfloat162float(*c), e);
        *c = __float2bfloat16_rn(e);
      } else {
        float* c = static_cast<float*>(g.C) + idx;
        if (g.beta != 0.f) e = fmaf(g.beta, *c, e);
        *c = e;
      }
    }
  }
  if (g.parts > 1) ptx::cluster_sync_all();           // a CTA's shared memory is read until its peers are done
}

template <int TM, int TN, int SL, bool TA, bool TB>
int launch_shape(DevGemm d, long long tiles, cudaStream_t stream) {
  using S = Shape<TM, TN, SL>;
  auto kern = gemm_simt_kernel<TM, TN, SL, TA, TB>;
  static DeviceOnce attr_set;      // the attribute belongs to the device that was current
  int dev = -1;
  PRAC_CUDA_TRY(cudaGetDevice(&dev));
  if (!attr_set.done(dev)) {
    PRAC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM));
    attr_set.mark(dev);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(tiles * d.parts));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = S::SMEM;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(d.parts); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1] = dependent_launch_attr();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  count_launch();
  PRAC_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, d));
  return PRAC_OK;
}
template <int TM, int TN, int SL>
int launch_trans(const DevGemm& d, int ta, int tb, long long tiles, cudaStream_t stream) {
  if (ta && tb) return PRAC_EINVAL;        // (nothing asks for it)
  if (ta) return launch_shape<TM, TN, SL, true, false>(d, tiles, stream);
  return tb ? launch_shape<TM, TN, SL, false, true>(d, tiles, stream) : launch_shape<TM, TN, SL, false, false>(d, tiles, stream);
}

// CTAs of a shape that can be resident at once in clusters of `parts` (two per SM without clusters; larger
// clusters do not fill every group of SMs: 33 of 4 and 16 of 8 at one CTA per SM); 0 where the device has no
// room for such a cluster (a part of a GPU may not).
template <int TM, int TN, int SL>
int resident_ctas(int parts, int sms) {
  using S = Shape<TM, TN, SL>;
  if (parts == 1) return 2 * sms;
  static DeviceValue cached[3];    // parts 2, 4, 8
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 0; }
  DeviceValue& slot = cached[parts == 2 ? 0 : (parts == 4 ? 1 : 2)];
  if (slot.get(dev) > 0) return slot.get(dev);
  auto kern = gemm_simt_kernel<TM, TN, SL, false, false>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(sms / parts * parts));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = S::SMEM;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(parts); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
    cudaGetLastError();
    return 0;
  }
  slot.set(dev, n * parts);
  return n * parts;
}

}  // namespace

PRAC_BOUNDS_READER(bounds_violations_simt)

#ifdef PRAC_DEBUG_BOUNDS
// The bounds-checking build only: every product takes this tile (0, 1, 2: see `cand` below) and this number of
// K pieces (1, 2, 4, 8) instead of those of the rule; tile < 0 gives the rule back.
static int g_forced_tile = -1, g_forced_parts = 1;
extern "C" void prac_debug_force_product(int tile, int parts) { g_forced_tile = tile; g_forced_parts = parts; }
#endif

int gemm_general(const GemmArgs& g, cudaStream_t stream) {
  if (g.M < 0 || g.N < 0 || g.K < 0) return PRAC_EINVAL;
  if (g.M == 0 || g.N == 0) return PRAC_OK;
  if (g.M > 65535ll * 64 || g.N > 0x7fffff00 || g.K > 0x7fff0000) return PRAC_EINVAL;
  const bool symmetric = g.symmetric != 0;
  if (symmetric && (g.A != g.B || g.M != g.N || !g.trans_a || g.trans_b || g.type_c != ET_F32 || g.beta != 0.0)) return PRAC_EINVAL;
  auto vec = [](const void* p, int type, int64_t ld) {
    return (reinterpret_cast<uintptr_t>(p) & (type == ET_BF16 ? 7u : 15u)) == 0 && ld % 4 == 0;
  };
  DevGemm d{};
  d.M = static_cast<int>(g.M); d.N = static_cast<int>(g.N); d.K = static_cast<int>(g.K);
  d.A = g.A; d.lda = g.lda; d.bf16_a = g.type_a == ET_BF16; d.vec_a = vec(g.A, g.type_a, g.lda);
  d.B = g.B; d.ldb = g.ldb; d.bf16_b = g.type_b == ET_BF16; d.vec_b = vec(g.B, g.type_b, g.ldb);
  d.C = g.C; d.ldc = g.ldc; d.bf16_c = g.type_c == ET_BF16; d.vec_c = !d.bf16_c && vec(g.C, ET_F32, g.ldc);
  d.alpha = static_cast<float>(g.alpha); d.beta = static_cast<float>(g.beta);
  d.kscale_from = (g.kscale_from < 0 || g.kscale_from > g.K) ? d.K : static_cast<int>(g.kscale_from);
  if (d.kscale_from == d.K) d.kscale_from = 0x7fffffff;
  d.kscale = static_cast<float>(g.kscale);
  d.symmetric = symmetric;
  d.run_if = g.run_if; d.run_if_mask = g.run_if_mask;
  // what a row-major buffer of these dimensions spans: (rows - 1) * ld + cols elements
  d.ext_a = g.trans_a ? (g.K - 1) * g.lda + g.M : (g.M - 1) * g.lda + g.K;
  d.ext_b = g.trans_b ? (g.N - 1) * g.ldb + g.K : (g.K - 1) * g.ldb + g.N;
  d.ext_c = (g.M - 1) * g.ldc + g.N;
  // Tile and number of K pieces: the smallest estimated time, in us, from what was measured over products of
  // 0.02 to 8.6 Gflop: a step of a CTA takes `alone` by itself on its SM and two CTAs that share one take
  // `shared` for a step of both (a tile gets about half of the FMA rate; the small one loads more per
  // FMA), a round of CTAs costs 2 to 5 more the larger its clusters.  The rule with one cost per step
  // that it replaces took 39, 103 and 83 us for Gram products of 2048 x 512, 5561 x 482 and an inner
  // product of 8192 x 1024 by 128, this one 25, 67 and 69.
  struct Cand { int tm, tn, sl; double alone, shared; };
  static const Cand cand[3] = {{128, 128, 1, 2.0, 3.5}, {64, 64, 4, 2.45, 4.0}, {32, 32, 8, 1.3, 2.65}};
  int sms = tc_num_sms();
  if (sms <= 0) sms = 148;
  int best = 2, parts = 1;
  long long best_tiles = 0;
  double best_t = -1.0;
  for (int c = 0; c < 3; ++c) {
    const long long tm = (g.M + cand[c].tm - 1) / cand[c].tm, tn = (g.N + cand[c].tn - 1) / cand[c].tn;
    const long long tiles = symmetric ? tn * (tn + 1) / 2 : tm * tn;
    for (int p = 1; p <= 8; p *= 2) {
      if (tiles * p > 0x7fffffff) break;
      const long long steps = (g.K + BK * cand[c].sl * p - 1) / (BK * cand[c].sl * p);
      if (p > 1 && (steps < 2 || g.run_if != nullptr)) break;    // (an optional launch stays off the cluster barrier)
      const int fit = c == 0 ? resident_ctas<128, 128, 1>(p, sms) : (c == 1 ? resident_ctas<64, 64, 4>(p, sms) : resident_ctas<32, 32, 8>(p, sms));
      if (fit < p) break;
      const double rounds = tiles * p > fit ? static_cast<double>(tiles * p) / fit : 1.0;     // of up to two CTAs per SM
      const double step = tiles * p <= fit / 2 ? cand[c].alone : cand[c].shared;
      const double est = rounds * (steps * step + (p == 1 ? 2.0 : (p == 2 ? 3.0 : (p == 4 ? 4.0 : 5.0))));
      if (best_t < 0.0 || est < best_t) { best_t = est; best = c; parts = p; best_tiles = tiles; }
    }
  }
  if (best_t < 0.0) return PRAC_EINVAL;
#ifdef PRAC_DEBUG_BOUNDS
  if (g_forced_tile >= 0) {
    best = g_forced_tile; parts = g.run_if != nullptr ? 1 : g_forced_parts;
    const long long tm = (g.M + cand[best].tm - 1) / cand[best].tm, tn = (g.N + cand[best].tn - 1) / cand[best].tn;
    best_tiles = symmetric ? tn * (tn + 1) / 2 : tm * tn;
  }
#endif
  d.parts = parts;
  d.tiles_n = static_cast<int>((g.N + cand[best].tn - 1) / cand[best].tn);
  if (best == 0) return launch_trans<128, 128, 1>(d, g.trans_a, g.trans_b, best_tiles, stream);
  if (best == 1) return launch_trans<64, 64, 4>(d, g.trans_a, g.trans_b, best_tiles, stream);
  return launch_trans<32, 32, 8>(d, g.trans_a, g.trans_b, best_tiles, stream);
}

}  // namespace prac
