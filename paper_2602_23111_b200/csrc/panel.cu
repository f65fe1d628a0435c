// Small-matrix kernels of the basis fit: the counter-based Gaussian draw, the one-sided block
// Jacobi eigen-solver of the Rayleigh-Ritz step, and format conversions.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "act.cuh"
#include "grid_barrier.cuh"
#include "internal.h"
#include "per_device.h"
#include "ptx.cuh"

namespace prac {
namespace {

// ------------------------------------------------------------------ Philox4x32-10
// Salmon, Moraes, Dror, Shaw (SC'11).  One call turns a 128-bit counter and a 64-bit key
// into four 32-bit words.
__device__ __forceinline__ uint4 philox4x32_10(uint4 ctr, uint2 key) {
  constexpr uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const uint32_t hi0 = __umulhi(M0, ctr.x), lo0 = M0 * ctr.x;
    const uint32_t hi1 = __umulhi(M1, ctr.z), lo1 = M1 * ctr.z;
    ctr = make_uint4(hi1 ^ ctr.y ^ key.x, lo1, hi0 ^ ctr.w ^ key.y, lo0);
    key.x += W0;
    key.y += W1;
  }
  return ctr;
}

__device__ __forceinline__ uint4 draw_block(uint64_t seed, uint64_t draw_counter, uint64_t blk) {
  const uint4 ctr = make_uint4(static_cast<uint32_t>(blk), static_cast<uint32_t>(blk >> 32),
                               static_cast<uint32_t>(draw_counter), static_cast<uint32_t>(draw_counter >> 32));
  const uint2 key = make_uint2(static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32));
  return philox4x32_10(ctr, key);
}

__global__ void philox_words_kernel(uint64_t seed, uint64_t dc, long long n, uint32_t* __restrict__ out) {
  grid_dep_wait();
  grid_dep_launch();
  const long long blk = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  const long long e0 = blk * 4;
  if (e0 >= n) return;
  const uint4 w = draw_block(seed, dc, static_cast<uint64_t>(blk));
  if (e0 + 4 <= n && (reinterpret_cast<uintptr_t>(out + e0) & 15u) == 0) {
    *reinterpret_cast<uint4*>(out + e0) = w;
  } else {
    const uint32_t v[4] = {w.x, w.y, w.z, w.w};
    for (int e = 0; e < 4 && e0 + e < n; ++e)
      if (PRAC_IN(e0 + e, n)) out[e0 + e] = v[e];
  }
}

// 23-bit uniform at a cell midpoint: (2 (w >> 9) + 1) / 2^24, never 0 or 1.
__device__ __forceinline__ double word_to_uniform(uint32_t w) {
  return (2.0 * static_cast<double>(w >> 9) + 1.0) * (1.0 / 16777216.0);
}

// Box-Muller on lane pairs (0,1) and (2,3); evaluated in double, stored as float.
__global__ void gaussian_kernel(uint64_t seed, uint64_t dc, long long d, long long r,
                                float* __restrict__ S, long long lds) {
  grid_dep_wait();
  const long long blk = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  const long long n = d * r;
  const long long e0 = blk * 4;
  if (e0 >= n) return;
  const uint4 w = draw_block(seed, dc, static_cast<uint64_t>(blk));
  const uint32_t wa[2] = {w.x, w.z}, wb[2] = {w.y, w.w};
  float z[4];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const double rad = sqrt(-2.0 * log(word_to_uniform(wa[h])));
    double sn, cs;
    sincospi(2.0 * word_to_uniform(wb[h]), &sn, &cs);
    z[2 * h] = static_cast<float>(rad * cs);
    z[2 * h + 1] = static_cast<float>(rad * sn);
  }
  for (int e = 0; e < 4 && e0 + e < n; ++e) {
    const long long idx = e0 + e;
    if (PRAC_IN((idx / r) * lds + (idx % r), (d - 1) * lds + r)) S[(idx / r) * lds + (idx % r)] = z[e];
  }
}

// ------------------------------------------------------------------ Jacobi eigen-solver
// Dominant eigenvectors of a small symmetric positive semi-definite matrix B by one-sided
// (Hestenes) block Jacobi.  With A = B + sigma I (sigma > 0 small), plane rotations applied to the
// columns of A make them mutually orthogonal: A J = J (Lambda + sigma I).  The column norms then
// order the eigenvalues and the normalised columns are the eigenvectors, so no eigenvector
// matrix is accumulated and a null space of B comes out as an orthonormal set.  (Rotating a
// Cholesky factor of A instead was measured: it saved no sweep and cost a factorisation.)
// The columns (stored as rows of At) are grouped in blocks of b.  In one outer step the
// round-robin schedule gives each CTA a pair of blocks: it loads the 2b columns into shared
// memory, runs one full inner sweep over them (2b - 1 steps of b disjoint rotations, one warp
// per rotation) and writes them back; the CTAs then meet at a grid barrier.  One outer sweep =
// (number of blocks - 1) barriers instead of the (n - 1) of element-wise Jacobi.
constexpr int JAC_MAX_SWEEPS = 30;
// A sweep that met no squared cosine above JAC_DONE_COS2 is the last one: what the result may lack of
// orthogonality has been measured, at the level that fp32 keeps.  (Convergence is quadratic only between well
// separated eigenvalues.  Columns of nearly equal norm turn by large angles however small their cosines are,
// and a sweep shrinks those by a small factor only: a rule that stopped after cosines of 3e-4 and trusted the
// square left |U^T U - I| at 2e-3 for 64 columns on a spectrum of 0.1 % spread, where this one leaves 1e-6.
// The sweep that confirms is one of seven or eight on a power law.)
// Sweeps that run out are an error only where a cosine of 1e-4 is left (JAC_FAIL_COS2).
constexpr float JAC_DONE_COS2 = 1e-13f, JAC_FAIL_COS2 = 1e-8f;
// A finishing step (jacobi_finish) is tried after a sweep that met cosines up to JAC_NEAR; it turns all columns at once where
// no column's angles add up to more than JAC_STEP_TURN, by a rotation that is orthogonal to JAC_TURN_REST.  The last step, like
// the last sweep, is one that met no squared cosine above JAC_DONE_COS2.  (The angles alone say too little: two short
// columns beside a long one keep the product of their cosines with it, however small the angles towards it are.)
// Pairs with a squared cosine below JAC_ALONE_COS2 are left alone, as in the kernel for larger problems: 1e-9 is far below
// what the fp32 result keeps, and below what a rounding of B in fp32 does to two columns so close that the pair would
// still turn by a large angle.
constexpr int JAC_MAX_FINISH = 8;
constexpr float JAC_NEAR_COS2 = 1e-4f, JAC_STEP_TURN = 0.2f, JAC_TURN_REST = 1e-10f, JAC_ALONE_COS2 = 1e-18f;
struct JacobiInfo {
  GridBarrierState bar;             // zeroed before the launch
  int sweeps;
  double inv_scale;                 // 1 / largest diagonal entry of B (written by jacobi_prepare_kernel)
  int rotations[JAC_MAX_SWEEPS];    // rotations applied in each outer sweep
  int max_cos2[JAC_MAX_SWEEPS];     // largest squared cosine rotated away in each sweep (float bits)
  int fin_cos2[JAC_MAX_FINISH], fin_turn[JAC_MAX_FINISH];    // the same, and the largest sum of a column's angles, of each finishing step
  double norms[128];                // squared norms of the columns in a finishing step
  int late[JAC_MAX_SWEEPS];         // a wait for a visit's columns gave up in this sweep
};

// Pair i of step `step` of the round-robin schedule on m (even) items, as p < q.
__device__ __forceinline__ void rr_pair(int m, int step, int i, int& p, int& q) {
  int a, b;
  if (i == 0) { a = m - 1; b = step; }
  else {                       // (modulo m - 1, without a division: it is on the way from one visit to the next)
    a = step + i; if (a >= m - 1) a -= m - 1;
    b = step - i; if (b < 0) b += m - 1;
  }
  p = a < b ? a : b;
  q = a < b ? b : a;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// At (n x n, n a multiple of 16) = symmetrised B (ell x ell, leading dimension ldb) + sigma I,
// padded with 0.5 sigma on the diagonal; sigma = 2^-15 * largest diagonal entry of B (1 if B = 0):
// above the rounding noise that B inherits from its fp32 factors (so that null directions of B
// get columns of a definite size), and harmless, since a shift moves no eigenvector.
__global__ void __launch_bounds__(256) jacobi_prepare_kernel(const double* B, long long ldb, int ell,
                                                             double* __restrict__ At, int n, JacobiInfo* info) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ double red[256];
  if (blockIdx.x == 0) {       // the solver's barrier counter and sweep records start at zero
    int* words = reinterpret_cast<int*>(info);
    for (int i = threadIdx.x; i < static_cast<int>(sizeof(JacobiInfo) / sizeof(int)); i += blockDim.x) words[i] = 0;
  }
  double m = 0.0;
  for (int i = threadIdx.x; i < ell; i += blockDim.x) m = fmax(m, fabs(B[static_cast<long long>(i) * ldb + i]));
  red[threadIdx.x] = m;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
    __syncthreads();
  }
  const double sigma = red[0] > 0.0 ? red[0] * (1.0 / 32768.0) : 1.0;
  if (blockIdx.x == 0 && threadIdx.x == 0) info->inv_scale = red[0] > 0.0 ? 1.0 / red[0] : 1.0;
  for (long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; idx < static_cast<long long>(n) * n;
       idx += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int i = static_cast<int>(idx / n), j = static_cast<int>(idx % n);
    double v = 0.0;
    if (i < ell && j < ell) {
      v = 0.5 * (B[static_cast<long long>(i) * ldb + j] + B[static_cast<long long>(j) * ldb + i]);
      if (i == j) v += sigma;
    } else if (i == j) {
      v = 0.5 * sigma;
    }
    At[idx] = v;
  }
}

// One rotation of the shared-memory columns cp, cq (length n) by one warp.  With R > 0 each lane
// keeps its R elements of both columns in registers between the dot products and the update, so
// a rotation reads and writes shared memory once; R = 0 re-reads (any n).  scale brings squared column
// norms into the range of fp32.  Returns 1 if rotated.
template <int R>
__device__ __forceinline__ int rotate_pair(double* cp, double* cq, int n, int lane, double tol, double scale, float& max_cos2) {
  double alpha = 0.0, beta = 0.0, gamma = 0.0;
  double xr[R > 0 ? R : 1], yr[R > 0 ? R : 1];
  if (R > 0) {
#pragma unroll
    for (int e = 0; e < R; ++e) {
      const int r = lane + 32 * e;
      xr[e] = r < n ? cp[r] : 0.0;
      yr[e] = r < n ? cq[r] : 0.0;
      alpha = fma(xr[e], xr[e], alpha); beta = fma(yr[e], yr[e], beta); gamma = fma(xr[e], yr[e], gamma);
    }
  } else {
    for (int r = lane; r < n; r += 32) {
      const double x = cp[r], y = cq[r];
      alpha = fma(x, x, alpha); beta = fma(y, y, beta); gamma = fma(x, y, gamma);
    }
  }
  alpha = warp_sum(alpha); beta = warp_sum(beta); gamma = warp_sum(gamma);
  if (!(gamma * gamma > tol * tol * alpha * beta)) return 0;    // warp-uniform
  max_cos2 = fmaxf(max_cos2, static_cast<float>(gamma * gamma / (alpha * beta)));
  // The angle only has to shrink the inner product, so tan is taken in fp32 (double-precision
  // divisions and square roots are slow here); cos and sin are then formed in double from that
  // tangent, which keeps the rotation orthogonal to double accuracy.
  const float zeta = static_cast<float>((beta - alpha) * scale) / (2.f * static_cast<float>(gamma * scale));
  const float az = fabsf(zeta);
  const float t32 = (az > 1e15f) ? 0.5f / zeta : copysignf(1.f, zeta) / (az + sqrtf(1.f + az * az));
  const double t = static_cast<double>(t32);
  const double c = rsqrt(1.0 + t * t), s = c * t;
  if (R > 0) {
#pragma unroll
    for (int e = 0; e < R; ++e) {
      const int r = lane + 32 * e;
      if (r < n) { cp[r] = c * xr[e] - s * yr[e]; cq[r] = s * xr[e] + c * yr[e]; }
    }
  } else {
    for (int r = lane; r < n; r += 32) {
      const double x = cp[r], y = cq[r];
      cp[r] = c * x - s * y;
      cq[r] = s * x + c * y;
    }
  }
  return 1;
}

// blockDim = 32 * b; dynamic shared memory = 2 b n doubles; R: see rotate_pair (32 R >= n).
// A block's own column pairs are rotated in the first visit of each sweep in which the block
// takes part (a full inner sweep over the 2b columns); every other visit rotates only the b*b
// pairs that cross the two blocks (b steps of b disjoint rotations).
template <int R>
__global__ void jacobi_kernel(double* At, int n, int b, int max_sweeps, double tol, JacobiInfo* info,
                              int* dev_status, unsigned poll_limit) {
  extern __shared__ double cols[];          // [2b][n]
  const int nb = n / b;
  const int nbr = nb + (nb & 1);            // an odd count plays with a bye
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = 2 * b;
  const unsigned nctas = gridDim.x;
  const double inv_scale = info->inv_scale;
  unsigned bar = 0;
  bool alive = true, converged = false;
  float mc2 = 1.f;
  int sweep = 0;
  for (; alive && sweep < max_sweeps && !converged; ++sweep) {
    for (int step = 0; alive && step < nbr - 1; ++step) {
      int I, J;
      rr_pair(nbr, step, blockIdx.x, I, J);
      if (J < nb) {                          // J == nb: bye
        // each warp moves whole columns, all of a lane's loads in flight together
        for (int lc = warp; lc < m; lc += b) {
          const double* src = At + static_cast<long long>(lc < b ? I * b + lc : J * b + (lc - b)) * n;
          double* dst = cols + lc * n;
          if (R > 0) {
            double v[R > 0 ? R : 1];
#pragma unroll
            for (int e = 0; e < R; ++e) { const int r = lane + 32 * e; v[e] = r < n ? __ldcg(&src[r]) : 0.0; }
#pragma unroll
            for (int e = 0; e < R; ++e) { const int r = lane + 32 * e; if (r < n) dst[r] = v[e]; }
          } else {
            for (int r = lane; r < n; r += 32) dst[r] = __ldcg(&src[r]);
          }
        }
        __syncthreads();
        // with a bye in the schedule, the block that sat out step 0 is first seen in step 1
        bool full = (step == 0);
        if (nbr != nb && step == 1) {
          int I0, J0;
          for (int c = 0; c < nbr / 2; ++c) {
            rr_pair(nbr, 0, c, I0, J0);
            if (J0 == nb && (I0 == I || I0 == J)) full = true;
          }
        }
        int rotated = 0;
        float max_cos2 = 0.f;
        if (full) {
          for (int is = 0; is < m - 1; ++is) {
            int p, q;
            rr_pair(m, is, warp, p, q);
            rotated += rotate_pair<R>(cols + p * n, cols + q * n, n, lane, tol, inv_scale * inv_scale, max_cos2);
            __syncthreads();
          }
        } else {
          for (int is = 0; is < b; ++is) {
            const int p = warp, q = b + (warp + is) % b;
            rotated += rotate_pair<R>(cols + p * n, cols + q * n, n, lane, tol, inv_scale * inv_scale, max_cos2);
            __syncthreads();
          }
        }
        if (lane == 0 && rotated) {
          atomicAdd(&info->rotations[sweep], rotated);
          atomicMax(&info->max_cos2[sweep], __float_as_int(max_cos2));   // non-negative floats order as ints
        }
        for (int lc = warp; lc < m; lc += b) {
          double* dstg = At + static_cast<long long>(lc < b ? I * b + lc : J * b + (lc - b)) * n;
          const double* srcs = cols + lc * n;
          for (int r = lane; r < n; r += 32) dstg[r] = srcs[r];
        }
      }
      alive = grid_barrier(&info->bar, ++bar * nctas, poll_limit);
    }
    // Every CTA reads the same values after the barrier of the sweep's last step.
    if (alive) {
      const int rot = *reinterpret_cast<volatile int*>(&info->rotations[sweep]);
      mc2 = __int_as_float(*reinterpret_cast<volatile int*>(&info->max_cos2[sweep]));
      converged = (rot == 0) || (mc2 < JAC_DONE_COS2);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    info->sweeps = sweep;
    if (!alive && dev_status) atomicOr(dev_status, DEV_WAIT_EXPIRED);
    else if (!converged && mc2 >= JAC_FAIL_COS2 && dev_status) atomicOr(dev_status, DEV_JACOBI_NOCONV);
  }
}

// ------------------------------------------------------------------ block Jacobi through the Gram matrix
constexpr int JG_B = 8;          // columns per block
constexpr int JG_M = 2 * JG_B;   // columns a CTA holds
constexpr int JG_P = JG_M + 1;   // pitch of the small matrices

// Rotation coefficients of one column within a round: new column x = self * x + other * partner(x).
struct JgCoef { double self, other; int partner; int pad; };

// Same sweeps, visits and rotation order as jacobi_kernel, for 8-column blocks and 256 threads, but a
// visit works on the 16 x 16 Gram matrix G of its columns: G is formed once (tensor cores), each
// round's eight disjoint rotations are read off G and applied to G and to the accumulated
// rotation J (16 x 16, one element per thread), and the columns are multiplied by J once at the
// end (tensor cores).  The long vectors are touched twice per visit instead of twice per round.
// A cooperative launch with the bounded software barrier; it serves n > 256 (jacobi_stream_kernel below).
__global__ void __launch_bounds__(256) jacobi_gram_kernel(double* At, int n, int max_sweeps, double tol, JacobiInfo* info,
                                                          int* dev_status, unsigned poll_limit) {
  extern __shared__ double jsm[];
  const int ns = n + 4;                                   // column pitch: keeps the fragment loads off one bank
  double* cols = jsm;                                     // [16][ns]
  double (*G0)[JG_P] = reinterpret_cast<double (*)[JG_P]>(cols + JG_M * ns);
  double (*G1)[JG_P] = G0 + JG_M;
  double (*J0)[JG_P] = G1 + JG_M;
  double (*J1)[JG_P] = J0 + JG_M;
  double* part = reinterpret_cast<double*>(J1 + JG_M);    // [8 warps][3 tiles][64]
  JgCoef* coef = reinterpret_cast<JgCoef*>(part + 8 * 3 * 64);   // [16]
  __shared__ int visit_rotated;

  const int b = JG_B, m = JG_M;
  const int nb = n / b;
  const int nbr = nb + (nb & 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, q4 = lane & 3;
  const int ei = threadIdx.x >> 4, ej = threadIdx.x & 15;   // this thread's element of the 16 x 16 matrices
  const unsigned nctas = gridDim.x;
  const double inv_scale = info->inv_scale;                 // (G is scaled with it: its entries are taken to fp32)
  unsigned bar = 0;
  bool alive = true, converged = false;
  float mc2 = 1.f;
  int sweep = 0;
  for (; alive && sweep < max_sweeps && !converged; ++sweep) {
    for (int step = 0; alive && step < nbr - 1; ++step) {
      int I, J;
      rr_pair(nbr, step, blockIdx.x, I, J);
      if (J < nb) {
        for (int lc = warp; lc < m; lc += 8) {
          const double* src = At + static_cast<long long>(lc < b ? I * b + lc : J * b + (lc - b)) * n;
          double* dst = cols + lc * ns;
          for (int r0 = lane; r0 < n; r0 += 32 * 12) {    // up to twelve loads in flight per lane
            double v[12];
#pragma unroll
            for (int e = 0; e < 12; ++e) { const int r = r0 + 32 * e; v[e] = r < n ? __ldcg(&src[r]) : 0.0; }
#pragma unroll
            for (int e = 0; e < 12; ++e) { const int r = r0 + 32 * e; if (r < n) dst[r] = v[e]; }
          }
        }
        if (threadIdx.x == 0) visit_rotated = 0;
        __syncthreads();
        // ---- G = A^T A: each warp sums a slice of the rows, the slices are added in warp order
        {
          double t00[2] = {0.0, 0.0}, t01[2] = {0.0, 0.0}, t11[2] = {0.0, 0.0};
          const int ks_total = n / 4, kpw = (ks_total + 7) / 8;
          const int ks_end = min(ks_total, (warp + 1) * kpw);
          for (int ks = warp * kpw; ks < ks_end; ++ks) {
            const int r = ks * 4 + q4;
            const double a0 = cols[g * ns + r], a1 = cols[(8 + g) * ns + r];
            ptx::dmma_884(t00, a0, a0);
            ptx::dmma_884(t01, a0, a1);
            ptx::dmma_884(t11, a1, a1);
          }
          double* pw = part + warp * 192 + g * 8 + 2 * q4;
          pw[0] = t00[0]; pw[1] = t00[1];
          pw[64] = t01[0]; pw[65] = t01[1];
          pw[128] = t11[0]; pw[129] = t11[1];
        }
        __syncthreads();
        {
          // element (ei, ej): tile 00, 01 (or its transpose) or 11
          int tile, r, c;
          if (ei < 8 && ej < 8) { tile = 0; r = ei; c = ej; }
          else if (ei < 8) { tile = 1; r = ei; c = ej - 8; }
          else if (ej < 8) { tile = 1; r = ej; c = ei - 8; }
          else { tile = 2; r = ei - 8; c = ej - 8; }
          double sum = 0.0;
#pragma unroll
          for (int w8 = 0; w8 < 8; ++w8) sum += part[w8 * 192 + tile * 64 + r * 8 + c];
          G0[ei][ej] = sum * inv_scale * inv_scale;
          J0[ei][ej] = (ei == ej) ? 1.0 : 0.0;
        }
        __syncthreads();
        // with a bye in the schedule, the block that sat out step 0 is first seen in step 1
        bool full = (step == 0);
        if (nbr != nb && step == 1) {
          int I0, J0b;
          for (int c = 0; c < nbr / 2; ++c) {
            rr_pair(nbr, 0, c, I0, J0b);
            if (J0b == nb && (I0 == I || I0 == J)) full = true;
          }
        }
        const int rounds = full ? m - 1 : b;
        int rotated = 0;
        float max_cos2 = 0.f;
        double (*Gc)[JG_P] = G0; double (*Gn)[JG_P] = G1;
        double (*Jc)[JG_P] = J0; double (*Jn)[JG_P] = J1;
        for (int is = 0; is < rounds; ++is) {
          if (threadIdx.x < b) {
            int p, q;
            if (full) rr_pair(m, is, threadIdx.x, p, q);
            else { p = threadIdx.x; q = b + (threadIdx.x + is) % b; }
            const double alpha = Gc[p][p], beta = Gc[q][q], gamma = Gc[p][q];
            double c = 1.0, sn = 0.0;
            if (gamma * gamma > tol * tol * alpha * beta) {
              ++rotated;
              max_cos2 = fmaxf(max_cos2, static_cast<float>(gamma * gamma) / static_cast<float>(alpha * beta));
              // The angle only has to shrink the inner product, so cos and sin are taken in fp32;
              // one Newton step on their norm in double then makes the rotation orthogonal to
              // double accuracy (the fp32 pair is off the unit circle by ~1e-7, the step squares that).
              const float zeta = static_cast<float>(beta - alpha) / (2.f * static_cast<float>(gamma));
              const float az = fabsf(zeta);
              const float t32 = (az > 1e15f) ? 0.5f / zeta : copysignf(1.f, zeta) / (az + sqrtf(1.f + az * az));
              const float c32 = rsqrtf(fmaf(t32, t32, 1.f));
              c = static_cast<double>(c32);
              sn = static_cast<double>(c32 * t32);
              const double fix = fma(-0.5, fma(c, c, sn * sn), 1.5);
              c *= fix;
              sn *= fix;
            }
            // column p' = c p - s q,  column q' = s p + c q
            coef[p].self = c; coef[p].other = -sn; coef[p].partner = q;
            coef[q].self = c; coef[q].other = sn;  coef[q].partner = p;
          }
          __syncthreads();
          {
            const JgCoef ci = coef[ei], cj = coef[ej];
            const int pi = ci.partner, pj = cj.partner;
            // G <- R^T G R and J <- J R for the round's rotation R (block diagonal after permutation)
            const double row_i = fma(cj.self, Gc[ei][ej], cj.other * Gc[ei][pj]);
            const double row_p = fma(cj.self, Gc[pi][ej], cj.other * Gc[pi][pj]);
            Gn[ei][ej] = fma(ci.self, row_i, ci.other * row_p);
            Jn[ei][ej] = fma(cj.self, Jc[ei][ej], cj.other * Jc[ei][pj]);
          }
          __syncthreads();
          double (*tg)[JG_P] = Gc; Gc = Gn; Gn = tg;
          double (*tj)[JG_P] = Jc; Jc = Jn; Jn = tj;
        }
        if (threadIdx.x < b && rotated) {
          atomicAdd(&visit_rotated, rotated);
          atomicAdd(&info->rotations[sweep], rotated);
          atomicMax(&info->max_cos2[sweep], __float_as_int(max_cos2));   // non-negative floats order as ints
        }
        __syncthreads();
        if (visit_rotated) {
          // ---- columns <- columns * J, eight rows at a time; a warp reads only the rows it writes
          double b0[4], b1[4];
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) { b0[kk] = Jc[kk * 4 + q4][g]; b1[kk] = Jc[kk * 4 + q4][8 + g]; }
          for (int band = warp; band < n / 8; band += 8) {
            const int r = band * 8 + g;
            double o0[2] = {0.0, 0.0}, o1[2] = {0.0, 0.0};
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              const double a = cols[(kk * 4 + q4) * ns + r];
              ptx::dmma_884(o0, a, b0[kk]);
              ptx::dmma_884(o1, a, b1[kk]);
            }
            cols[(2 * q4) * ns + r] = o0[0];
            cols[(2 * q4 + 1) * ns + r] = o0[1];
            cols[(8 + 2 * q4) * ns + r] = o1[0];
            cols[(8 + 2 * q4 + 1) * ns + r] = o1[1];
          }
          __syncthreads();
          for (int lc = warp; lc < m; lc += 8) {
            double* dstg = At + static_cast<long long>(lc < b ? I * b + lc : J * b + (lc - b)) * n;
            const double* srcs = cols + lc * ns;
            for (int r = lane; r < n; r += 32) dstg[r] = srcs[r];
          }
        }
      }
      alive = grid_barrier(&info->bar, ++bar * nctas, poll_limit);
    }
    if (alive) {
      const int rot = *reinterpret_cast<volatile int*>(&info->rotations[sweep]);
      mc2 = __int_as_float(*reinterpret_cast<volatile int*>(&info->max_cos2[sweep]));
      converged = (rot == 0) || (mc2 < JAC_DONE_COS2);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    info->sweeps = sweep;
    if (!alive && dev_status) atomicOr(dev_status, DEV_WAIT_EXPIRED);
    else if (!converged && mc2 >= JAC_FAIL_COS2 && dev_status) atomicOr(dev_status, DEV_JACOBI_NOCONV);
  }
}

// ------------------------------------------------------------------ the same for n <= 256, rotations streamed
// What bounded jacobi_gram_kernel at n = 128 (6.5 us per visit, 120 visits): the eight rounds' dependent
// fp64 chains with two block barriers each (3.2 us), then the columns' trip into shared memory, through
// the accumulated rotation and out again.  Here 64 threads walk the rounds on the visit's 16 x 16 Gram
// matrix alone (in double; the angles are fp32, each rotation is made orthogonal to double accuracy
// before it touches a column): thread (u, v)
// holds the 2 x 2 block where pairs u and v meet and works out both pairs' angles itself, so a round
// is one barrier of two warps.  ROWS other threads hold one row each of the sixteen columns in registers
// and apply the rounds in double as their angles are published: the update costs nothing beyond the
// rounds.
// (With G in fp32 and the rotations of G not on the unit circle a round takes 360 cycles, but the diagonal of
// G then drifts by more than the columns of a cluster differ by: 18 to 30 sweeps there instead of 7 to 14.)
//
// Pairs of a round as slots: the first visit of a sweep plays the full round robin on 16 items (item 15
// fixed, the others y[0..14] moving up by one per round: (15, y[0]), (y[i], y[15 - i])); every other
// visit the 64 pairs that cross the two blocks ((i, 8 + y[i]), y moving up by one).  After the last
// round every item is back in its place.
//
// CLUSTER: the whole grid is one thread-block cluster.  The columns never leave its shared memory: after a visit the
// row threads store them where the next visit wants them, in the second buffer of the CTA before or after this one, whose
// mbarrier counts their bytes (a visit's columns through global memory: 2350 cycles from the last round to the next Gram
// matrix, and 1350 to form it from loads that go to L2, of 7400).  A buffer is free when it is stored to again two visits
// later: the columns that this CTA needed meanwhile came from its two neighbours' visit after they had read it.  Only at the
// end of a sweep do the CTAs meet at the hardware cluster barrier: every CTA runs the same
// number of steps and sweeps (the stopping test reads values that are final before the barrier it
// follows), so each barrier is reached by all of them.  A wait for columns is bounded, in polls and in time (a poll may itself
// block for a while).  A CTA that gives up sends its columns, such as they are, to the end of the sweep, so that nobody
// waits for them in vain, but waits no more and arms its barriers no more (the one it gave up on is still in a phase that
// must not be armed twice); at the end of the sweep all of them stop, and it waits for every byte that was sent to it before
// it leaves.  Otherwise a cooperative launch with the bounded software barrier, the columns in global memory.
constexpr int JS_G_THREADS = 256;      // form the Gram matrix; the first 64 walk the rounds
constexpr int JS_R_THREADS = 64;
constexpr int JS_MAX_ROWS = 256;
constexpr uint64_t JS_WAIT_NS = 2000000000ull;   // what a wait for columns may last
// (the warp has to be converged at these barriers)
__device__ __forceinline__ void named_sync(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ float rsqrt_fast(float x) { float r; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }

// Items (a, b) of pair u in round `is` (see above).
__device__ __forceinline__ void stream_pair(bool full, int is, int u, int& a, int& b) {
  if (!full) { a = u; b = JG_B + ((u + is) & (JG_B - 1)); return; }
  if (u == 0) { a = JG_M - 1; b = is; return; }
  a = is + u; if (a >= JG_M - 1) a -= JG_M - 1;
  b = is - u; if (b < 0) b += JG_M - 1;
}

// a' = c a + o b, b' = c b - o a make the columns orthogonal: with d = |b|^2 - |a|^2 and g = 2 a.b the smaller such angle has
// cos 2t = |d| / |(d, g)|, sin 2t = sign(d) g / |(d, g)|; c = sqrt((1 + cos 2t) / 2), o = -sin 2t / (2 c).  (The hardware's
// approximations, two in a row: the angle only has to shrink the inner product.  A shift of |d| by 1e-18 keeps the angle of
// two zero columns zero.)
__device__ __forceinline__ float2 stream_angle(double aa, double bb, double ab) {
  const float d = static_cast<float>(bb - aa), g = 2.f * static_cast<float>(ab);
  const float ad = fabsf(d) + 1e-18f;
  const float ih = rsqrt_fast(fmaf(ad, ad, g * g));
  const float c2 = fmaf(0.5f * ad, ih, 0.5f);
  const float rc = rsqrt_fast(c2);
  return make_float2(c2 * rc, -0.5f * copysignf(1.f, d) * g * ih * rc);
}

// Where block X of m (even) is in step `step` of the round-robin schedule: CTA and slot (0: the lower block of the pair).
__device__ __forceinline__ void rr_where(int m, int step, int X, int& cta, int& slot) {
  int partner;
  if (X == m - 1) { cta = 0; partner = step; }
  else if (X == step) { cta = 0; partner = m - 1; }
  else {
    int d = X - step;
    if (d < 0) d += m - 1;
    const bool first = d <= m / 2 - 1;
    cta = first ? d : m - 1 - d;
    partner = first ? step - cta : step + cta;
    if (partner < 0) partner += m - 1;
    if (partner >= m - 1) partner -= m - 1;
  }
  slot = X < partner ? 0 : 1;
}

// A finishing step on the columns of all CTAs (16 each; up to ROWS of them), once they are nearly orthogonal:
// the whole Gram matrix, and then, where the rotation angles T_ij = g_ij / (g_jj - g_ii) of all pairs are small, one rotation for
// all of them, A <- A exp(T), else nothing, because columns of nearly equal norm still turn by large angles.  Pairs that
// are orthogonal already are left alone, however close their norms.  It converges as the sweeps do at the end,
// quadratically: of the cosines it leaves products of two.
// T is antisymmetric to the last bit (both CTAs of a pair add the same products in the same order), so exp(T) is a rotation
// and A = B J keeps an orthogonal J, without which orthogonal columns need not be eigenvectors: I + T alone, off by T^2, turned
// single eigenvectors of power laws by up to 1e-3 (64 and 128 columns), exp(T) by what fp32 leaves, as the sweeps do.
// The series is summed until what is cut off is below JAC_TURN_REST: one to seven terms A T^m / m!, some 4000 cycles
// each at 128 columns, after 8000 for the Gram matrix, where a sweep takes 100 000.
// Called by all threads of all CTAs; returns 0: no step, 1: one step, 2: the last step, -1: a barrier gave up.
// CLUSTER: cols are this CTA's columns and term0, term1 two buffers for its columns of the terms, in shared memory (term0 holds
// the Gram matrix before).  Else the columns are in At, as the next sweep's first step pairs them, the terms in terms (2 n x n), and
// term0 holds the Gram matrix.  The norms pass through info.
template <bool CLUSTER, int ROWS>
__device__ __noinline__ int jacobi_finish(double (*cols)[ROWS + 2], double* At, double* terms, int n, double (*T)[ROWS + 2],
                                          double (*term0)[ROWS + 2], double (*term1)[ROWS + 2], double scale2, JacobiInfo* info,
                                          int attempt, unsigned& bar, unsigned poll_limit) {
  __shared__ double norms[ROWS];
  __shared__ int worst[2];
  constexpr int WARPS = (JS_G_THREADS + ROWS) / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q4 = lane & 3;
  const int ctas = gridDim.x, rank = blockIdx.x;
  // column e of CTA c: where it starts in At
  auto column = [&](int c, int e) {
    int I, J;
    rr_pair(2 * ctas, 0, c, I, J);
    return At + static_cast<long long>(e < JG_B ? I * JG_B + e : J * JG_B + e - JG_B) * n;
  };
  auto meet = [&]() {
    if (CLUSTER) { ptx::cluster_sync_all(); return true; }
    return grid_barrier(&info->bar, ++bar * gridDim.x, poll_limit);
  };
  // ---- Gp[i][j] = column i of this CTA times column j of all
  double (*const Gp)[ROWS + 2] = term0;
  for (int job = warp; job < 2 * ctas; job += WARPS) {
    const int e = 8 * (job & 1) + g;
    const uint32_t other = CLUSTER ? ptx::cluster_addr(&cols[e][q4], job >> 1) : 0u;
    const double* const in_mem = CLUSTER ? nullptr : column(job >> 1, e) + q4;
    const double* const own0 = CLUSTER ? &cols[g][q4] : column(rank, g) + q4;
    const double* const own1 = CLUSTER ? &cols[8 + g][q4] : column(rank, 8 + g) + q4;
    double acc0[2] = {0.0, 0.0}, acc1[2] = {0.0, 0.0};
#pragma unroll 8
    for (int ks = 0; ks < ROWS / 4; ++ks) {
      double a0, a1, b;
      if (CLUSTER) {
        b = ptx::cluster_ld_f64(other + ks * 32);
        a0 = own0[4 * ks]; a1 = own1[4 * ks];
      } else {                         // (n is a multiple of 16)
        const bool in = 4 * ks < n;
        b = in ? __ldcg(in_mem + 4 * ks) : 0.0;
        a0 = in ? __ldcg(own0 + 4 * ks) : 0.0; a1 = in ? __ldcg(own1 + 4 * ks) : 0.0;
      }
      ptx::dmma_884(acc0, a0, b);
      ptx::dmma_884(acc1, a1, b);
    }
#pragma unroll
    for (int e2 = 0; e2 < 2; ++e2) {
      Gp[g][8 * job + 2 * q4 + e2] = acc0[e2] * scale2;
      Gp[8 + g][8 * job + 2 * q4 + e2] = acc1[e2] * scale2;
    }
  }
  if (threadIdx.x < 2) worst[threadIdx.x] = 0;
  __syncthreads();
  if (threadIdx.x < JG_M) info->norms[JG_M * rank + threadIdx.x] = Gp[threadIdx.x][JG_M * rank + threadIdx.x];
  if (!meet()) return -1;
  for (int j = threadIdx.x; j < n; j += blockDim.x) norms[j] = __ldcg(&info->norms[j]);
  __syncthreads();
  // ---- T: the angle by which column j of this CTA takes up column i; turn: the sum of a column's angles
  float cos2 = 0.f, turn = 0.f;
  for (int j = warp; j < JG_M; j += WARPS) {
    const int jj = JG_M * rank + j;
    float sum = 0.f;
    for (int i = lane; i < n; i += 32) {
      const double v = Gp[j][i], di = norms[i], dj = norms[jj];
      const float c2 = i == jj ? 0.f : static_cast<float>(v * v / (di * dj));
      double t = 0.0;
      if (c2 > JAC_ALONE_COS2) {
        t = v / (dj - di);
        cos2 = fmaxf(cos2, fminf(c2, 1.f));
        sum += fabsf(static_cast<float>(t));
      }
      T[j][i] = t;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    turn = fmaxf(turn, fminf(sum, 1e30f));
  }
  const int w0 = __reduce_max_sync(0xffffffffu, __float_as_int(cos2)), w1 = __reduce_max_sync(0xffffffffu, __float_as_int(turn));
  if (lane == 0) { atomicMax(&worst[0], w0); atomicMax(&worst[1], w1); }   // (non-negative floats order as ints)
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicMax(&info->fin_cos2[attempt], worst[0]);
    atomicMax(&info->fin_turn[attempt], worst[1]);
  }
  if (!meet()) return -1;
  cos2 = __int_as_float(*reinterpret_cast<volatile int*>(&info->fin_cos2[attempt]));
  turn = __int_as_float(*reinterpret_cast<volatile int*>(&info->fin_turn[attempt]));
  if (!(turn <= JAC_STEP_TURN)) return 0;
  // ---- columns of this CTA += all columns times T, times T^2 / 2, ..; a term is the product of the one before it, eight
  // rows at a time.  turn is the 1-norm of T (and, T being antisymmetric, its infinity norm), so the terms after the m-th
  // add up to turn^(m + 1) / (m + 1)! and a little
  bool last = false;
  float rest = turn;
  for (int m = 1; !last; ++m) {
    rest *= turn / static_cast<float>(m + 1);
    last = rest <= JAC_TURN_REST;
    double (*const from)[ROWS + 2] = m == 1 ? cols : ((m & 1) ? term1 : term0);
    double (*const to)[ROWS + 2] = (m & 1) ? term0 : term1;
    const long long nn = static_cast<long long>(n) * n;
    const double* const from_mem = terms + ((m & 1) ? nn : 0);
    double* const to_mem = terms + ((m & 1) ? 0 : nn) + static_cast<long long>(JG_M) * rank * n;
    const double scale = 1.0 / m;
    for (int band = warp; 8 * band < n; band += WARPS) {
      double acc0[2] = {0.0, 0.0}, acc1[2] = {0.0, 0.0};
      const int r = 8 * band + g;
      for (int c = 0; c < ctas; ++c) {
        const uint32_t other = CLUSTER ? ptx::cluster_addr(&from[q4][r], c) : 0u;
#pragma unroll
        for (int ks = 0; ks < JG_M / 4; ++ks) {
          const int e = 4 * ks + q4;
          const double a = CLUSTER ? ptx::cluster_ld_f64(other + ks * 4 * (ROWS + 2) * 8)
                                   : __ldcg(m == 1 ? column(c, e) + r : from_mem + static_cast<long long>(JG_M * c + e) * n + r);
          ptx::dmma_884(acc0, a, T[g][JG_M * c + e]);
          ptx::dmma_884(acc1, a, T[8 + g][JG_M * c + e]);
        }
      }
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int e = 8 * (h >> 1) + 2 * q4 + (h & 1);
        const double v = scale * (h < 2 ? acc0[h] : acc1[h - 2]);
        if (CLUSTER) to[e][r] = v;
        else to_mem[e * n + r] = v;
      }
    }
    if (!meet()) return -1;            // (this term is complete, and nobody reads the one before it any more)
    for (int idx = threadIdx.x; idx < JG_M * n; idx += blockDim.x) {
      const int e = idx / n, r = idx % n;
      if (CLUSTER) {
        cols[e][r] += to[e][r];
      } else {
        double* const o = column(rank, e) + r;
        *o = __ldcg(o) + __ldcg(&to_mem[idx]);
      }
    }
  }
  if (!meet()) return -1;
  return cos2 < JAC_DONE_COS2 ? 2 : 1;
}

template <bool CLUSTER, int ROWS>   // ROWS = 128 or 256 >= n
__global__ void __launch_bounds__(JS_G_THREADS + ROWS, 1) jacobi_stream_kernel(
    double* At, double* terms, int n, int max_sweeps, JacobiInfo* info, int* dev_status, unsigned poll_limit) {
  grid_dep_wait();
  constexpr unsigned VISIT_BYTES = JG_M * ROWS * 8;   // what a CTA receives per visit
  __shared__ double part[8][3][64];
  __shared__ double G[2][JG_M][JG_P];
  __shared__ float2 coef[JG_M][JG_B];            // every round of the visit, per pair: c, o
  __shared__ double2 unit[ROWS / 32][2][JG_B];   // two rounds of them on the unit circle, per row warp
  // CLUSTER: the sixteen columns of this visit and of the next, which the CTAs of this visit store here
  extern __shared__ __align__(16) double jacobi_cols[];
  __shared__ uint64_t arrived[2];                // all of a buffer's columns are there
  typedef double (*Cols)[ROWS + 2];
  const int b = JG_B;
  const int nb = n / b;                          // even: n is a multiple of 16
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, q4 = lane & 3;
  const bool row_thread = threadIdx.x >= JS_G_THREADS;
  const unsigned nctas = gridDim.x;
  const double inv_scale = info->inv_scale;
  unsigned bar = 0;
  bool alive = true, converged = false;
  float mc2 = 1.f;
  int sweep = 0;
  unsigned visit = 0;
  bool late = false;                             // (lane 0 of each warp)
  unsigned late_visit = 0;                       // the visit after which it gave up
  __shared__ int gave_up;
  int attempt = 0, refused = 0;
  if (CLUSTER) {
    if (threadIdx.x < 2) ptx::mbar_init(&arrived[threadIdx.x], 1);
    if (threadIdx.x == 0) gave_up = 0;
    ptx::fence_mbar_init();
    int I, J;
    rr_pair(nb, 0, blockIdx.x, I, J);
    for (int e = warp; e < JG_M; e += (JS_G_THREADS + ROWS) / 32)
      for (int r = lane; r < ROWS; r += 32)
        reinterpret_cast<Cols>(jacobi_cols)[e][r] = r < n ? __ldcg(At + static_cast<long long>((e < b ? I * b + e : J * b + e - b)) * n + r) : 0.0;
    __syncthreads();
    ptx::cluster_sync_all();                 // (every CTA of the cluster has started)
  }
  for (; alive && sweep < max_sweeps && !converged; ++sweep) {
    for (int step = 0; alive && step < nb - 1; ++step) {
      int I, J;
      rr_pair(nb, step, blockIdx.x, I, J);
      double* const colI = At + static_cast<long long>(I) * b * n;
      double* const colJ = At + static_cast<long long>(J) * b * n;
      const unsigned turn = visit & 1;
      Cols const here = reinterpret_cast<Cols>(jacobi_cols) + turn * JG_M, there = reinterpret_cast<Cols>(jacobi_cols) + (turn ^ 1) * JG_M;
      if (CLUSTER && threadIdx.x == 0 && !late) ptx::mbar_arrive_expect_tx(&arrived[turn ^ 1], VISIT_BYTES);
      const bool full = step == 0;
      const int rounds = full ? JG_M - 1 : JG_B;
      if (row_thread) {
        const int r = threadIdx.x - JS_G_THREADS;
        double2 (*un)[JG_B] = unit[warp - JS_G_THREADS / 32];
        double x[JG_M];
#pragma unroll
        for (int e = 0; e < JG_B; ++e) {
          if (CLUSTER) {
            x[e] = here[e][r];
            x[JG_B + e] = here[JG_B + e][r];
          } else {
            x[e] = r < n ? __ldcg(colI + e * n + r) : 0.0;
            x[JG_B + e] = r < n ? __ldcg(colJ + e * n + r) : 0.0;
          }
        }
        auto rotate = [&](const double2 co, int a, int bq) {
          const double xa = x[a], xb = x[bq];
          x[a] = fma(co.x, xa, co.y * xb);
          x[bq] = fma(co.x, xb, -(co.y * xa));
        };
#pragma unroll 1
        for (int is = 0; is < rounds; is += 2) {
          named_sync(2 + (is >> 1), JS_R_THREADS + ROWS);
          // the angles of two rounds, put on the unit circle by one Newton step in double
          if (lane < 2 * JG_B) {
            const float2 co = coef[is + (lane >> 3)][lane & 7];
            const double c = static_cast<double>(co.x), o = static_cast<double>(co.y);
            const double fix = fma(-0.5, fma(c, c, o * o), 1.5);
            un[lane >> 3][lane & 7] = make_double2(c * fix, o * fix);
          }
          __syncwarp();
          if (!full) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
#pragma unroll
              for (int u = 0; u < JG_B; ++u) rotate(un[h][u], u, JG_B + ((u + h) & (JG_B - 1)));
            }
            const double y0 = x[JG_B], y1 = x[JG_B + 1];
#pragma unroll
            for (int e = JG_B; e < JG_M - 2; ++e) x[e] = x[e + 2];
            x[JG_M - 2] = y0; x[JG_M - 1] = y1;
          } else {
#pragma unroll 1
            for (int h = 0; h < 2 && is + h < rounds; ++h) {
              rotate(un[h][0], JG_M - 1, 0);
#pragma unroll
              for (int u = 1; u < JG_B; ++u) rotate(un[h][u], u, JG_M - 1 - u);
              const double first = x[0];
#pragma unroll
              for (int e = 0; e < JG_M - 2; ++e) x[e] = x[e + 1];
              x[JG_M - 2] = first;
            }
          }
          __syncwarp();
        }
        if (CLUSTER) {
          const int next = step + 1 < nb - 1 ? step + 1 : 0;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            int cta, slot;
            rr_where(nb, next, h ? J : I, cta, slot);
            const uint32_t to = ptx::cluster_addr(&there[JG_B * slot][r], cta), bar = ptx::cluster_addr(&arrived[turn ^ 1], cta);
#pragma unroll
            for (int e = 0; e < JG_B; ++e) ptx::cluster_st_async(to + e * (ROWS + 2) * 8, x[JG_B * h + e], bar);
          }
        } else if (r < n) {
#pragma unroll
          for (int e = 0; e < JG_B; ++e) {
            colI[e * n + r] = x[e];
            colJ[e * n + r] = x[JG_B + e];
          }
        }
      } else {
        // ---- G = A^T A: warp w takes the 16-row groups w, w + 8; lane (g, q4) the rows 4 q4 .. 4 q4 + 3 of
        // a group of the columns g of both blocks, straight from global memory in fragment layout
        {
          double t00[2] = {0.0, 0.0}, t01[2] = {0.0, 0.0}, t11[2] = {0.0, 0.0};
          double2 v[ROWS / 128][4];
#pragma unroll
          for (int h = 0; h < ROWS / 128; ++h) {
            const int r = (warp + 8 * h) * 16 + 4 * q4;
            const double2 zero = make_double2(0.0, 0.0);
            if (CLUSTER) {
              const double2* p0 = reinterpret_cast<const double2*>(&here[g][r]);
              const double2* p1 = reinterpret_cast<const double2*>(&here[JG_B + g][r]);
              v[h][0] = p0[0]; v[h][1] = p0[1]; v[h][2] = p1[0]; v[h][3] = p1[1];
            } else {
              const double2* p0 = reinterpret_cast<const double2*>(colI + g * n + r);
              const double2* p1 = reinterpret_cast<const double2*>(colJ + g * n + r);
              v[h][0] = r < n ? __ldcg(p0) : zero; v[h][1] = r < n ? __ldcg(p0 + 1) : zero;
              v[h][2] = r < n ? __ldcg(p1) : zero; v[h][3] = r < n ? __ldcg(p1 + 1) : zero;
            }
          }
#pragma unroll
          for (int h = 0; h < ROWS / 128; ++h) {
            const double a0[4] = {v[h][0].x, v[h][0].y, v[h][1].x, v[h][1].y};
            const double a1[4] = {v[h][2].x, v[h][2].y, v[h][3].x, v[h][3].y};
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
              ptx::dmma_884(t00, a0[ks], a0[ks]);
              ptx::dmma_884(t01, a0[ks], a1[ks]);
              ptx::dmma_884(t11, a1[ks], a1[ks]);
            }
          }
          const int o = g * 8 + 2 * q4;
          part[warp][0][o] = t00[0]; part[warp][0][o + 1] = t00[1];
          part[warp][1][o] = t01[0]; part[warp][1][o + 1] = t01[1];
          part[warp][2][o] = t11[0]; part[warp][2][o + 1] = t11[1];
        }
        named_sync(1, JS_G_THREADS);
        {
          // element (ei, ej): tile 00, 01 (or its transpose) or 11
          const int ei = threadIdx.x >> 4, ej = threadIdx.x & 15;
          int tile, r, c;
          if (ei < 8 && ej < 8) { tile = 0; r = ei; c = ej; }
          else if (ei < 8) { tile = 1; r = ei; c = ej - 8; }
          else if (ej < 8) { tile = 1; r = ej; c = ei - 8; }
          else { tile = 2; r = ei - 8; c = ej - 8; }
          double sum = 0.0;
#pragma unroll
          for (int w8 = 0; w8 < 8; ++w8) sum += part[w8][tile][r * 8 + c];
          G[0][ei][ej] = sum * inv_scale * inv_scale;
        }
        named_sync(1, JS_G_THREADS);
        if (threadIdx.x < JS_R_THREADS) {
          const int u = threadIdx.x >> 3, v = threadIdx.x & 7;
          double* Gc = &G[0][0][0];
          double* Gn = &G[1][0][0];
          int au, bu, av, bv;
          stream_pair(full, 0, u, au, bu);
          stream_pair(full, 0, v, av, bv);
#pragma unroll 1
          for (int is = 0; is < rounds; ++is) {
            const int ra = au * JG_P, rb = bu * JG_P, sa = av * JG_P, sb = bv * JG_P;
            const double uaa = Gc[ra + au], ubb = Gc[rb + bu], uab = Gc[ra + bu];
            const double vaa = Gc[sa + av], vbb = Gc[sb + bv], vab = Gc[sa + bv];
            const double x = Gc[ra + av], y = Gc[ra + bv], z = Gc[rb + av], w = Gc[rb + bv];
            const float2 cu = stream_angle(uaa, ubb, uab), cv = stream_angle(vaa, vbb, vab);
            const double uc = cu.x, uo = cu.y, vc = cv.x, vo = cv.y;
            // (both pairs' Newton step towards the unit circle, beside the products: without it the diagonal
            // drifts by 2^-22 per round, more than the columns of a cluster differ by)
            const double fix = fma(-0.5, fma(uc, uc, uo * uo), 1.5) * fma(-0.5, fma(vc, vc, vo * vo), 1.5);
            // the block of R_u^T G R_v
            const double x1 = fma(vc, x, vo * y), y1 = fma(vc, y, -vo * x);
            const double z1 = fma(vc, z, vo * w), w1 = fma(vc, w, -vo * z);
            Gn[ra + av] = fix * fma(uc, x1, uo * z1);
            Gn[rb + av] = fix * fma(uc, z1, -uo * x1);
            Gn[ra + bv] = fix * fma(uc, y1, uo * w1);
            Gn[rb + bv] = fix * fma(uc, w1, -uo * y1);
            if (u == v) coef[is][u] = cu;
            // (the next round's items are worked out before the barrier)
            stream_pair(full, is + 1, u, au, bu);
            stream_pair(full, is + 1, v, av, bv);
            double* t = Gc; Gc = Gn; Gn = t;
            named_sync(1, JS_R_THREADS);
            if ((is & 1) == 1 || is == rounds - 1) named_arrive(2 + (is >> 1), JS_R_THREADS + ROWS);
          }
        } else if (threadIdx.x >= 128) {
          // meanwhile: the largest cosine between columns that this visit is about to rotate (four more warps;
          // G[0] is intact until the second round has begun to write it, so its copy is taken from `part`)
          const int e = threadIdx.x - 128;           // the 64 entries of the crossing tile, the pairs within the blocks
          float c2 = 0.f;
          const int i = (e >> 3) & 7, j = e & 7;
          double ii = 0.0, jj = 0.0, ij = 0.0;
          if (e < 64) {
#pragma unroll
            for (int w8 = 0; w8 < 8; ++w8) { ii += part[w8][0][i * 9]; jj += part[w8][2][j * 9]; ij += part[w8][1][i * 8 + j]; }
            c2 = static_cast<float>(ij * ij / (ii * jj));
          } else if (full && i < j) {
            double jj2 = 0.0, kk2 = 0.0, jk2 = 0.0;
#pragma unroll
            for (int w8 = 0; w8 < 8; ++w8) {
              ii += part[w8][0][i * 9]; jj += part[w8][0][j * 9]; ij += part[w8][0][i * 8 + j];
              jj2 += part[w8][2][i * 9]; kk2 += part[w8][2][j * 9]; jk2 += part[w8][2][i * 8 + j];
            }
            c2 = static_cast<float>(fmax(ij * ij / (ii * jj), jk2 * jk2 / (jj2 * kk2)));
          }
          c2 = c2 > 0.f ? fminf(c2, 1.f) : 0.f;      // (NaN counts as nothing to rotate)
          const int bits = __reduce_max_sync(0xffffffffu, __float_as_int(c2));   // non-negative floats order as ints
          if (lane == 0) atomicMax(&info->max_cos2[sweep], bits);
        }
      }
      if (CLUSTER) {
        // (the whole CTA has to be through with this visit's angles; and warps that polled meanwhile would slow those that
        // work: a round 457 -> 540 cycles)
        __syncthreads();
        if (lane == 0 && !late) {
          unsigned polls = 0;
          uint64_t since = 0;
          while (!ptx::mbar_try_wait(&arrived[turn ^ 1], (visit >> 1) & 1u)) {
            late = ++polls >= poll_limit;
            if ((polls & 63u) == 0u) {
              const uint64_t now = ptx::globaltimer_ns();
              if (since == 0) since = now;
              late = late || now - since > JS_WAIT_NS || *reinterpret_cast<volatile int*>(&gave_up);
            }
            if (!late) continue;
            *reinterpret_cast<volatile int*>(&gave_up) = 1;
            atomicOr(&info->late[sweep], 1);
            late_visit = visit;
            break;
          }
        }
        __syncwarp();
        ++visit;
        if (step == nb - 2) ptx::cluster_sync_all();         // the sweep's largest cosine is complete
      } else {
        alive = grid_barrier(&info->bar, ++bar * nctas, poll_limit);
      }
    }
    if (CLUSTER) alive = *reinterpret_cast<volatile int*>(&info->late[sweep]) == 0;     // (final before that barrier)
    if (alive) {
      mc2 = __int_as_float(*reinterpret_cast<volatile int*>(&info->max_cos2[sweep]));
      converged = mc2 < JAC_DONE_COS2;
      if (ROWS == 128) {               // (128 columns: 449 -> 391 us in all; a step's three matrices of 256 columns do not fit beside the buffers)
        while (alive && !converged && mc2 < JAC_NEAR_COS2 && attempt < JAC_MAX_FINISH && refused < 3) {
          Cols const buf = reinterpret_cast<Cols>(jacobi_cols);
          const int r = jacobi_finish<CLUSTER, ROWS>(buf + (visit & 1) * JG_M, At, terms, n, buf + ((visit & 1) ^ 1) * JG_M, buf + 2 * JG_M,
                                                     buf + 3 * JG_M, inv_scale * inv_scale, info, attempt++, bar, poll_limit);
          alive = r >= 0;
          converged = r == 2;
          if (r == 0) { ++refused; break; }
        }
      }
    }
  }
  if (CLUSTER && late && threadIdx.x == 0) {
    // what has been sent here since the wait that gave up: the rest of that visit's columns, for which the barrier was armed,
    // and those of the visits up to the end of the sweep (all sent by now), for which it was not; the other barrier's likewise
    const uint64_t since = ptx::globaltimer_ns();
    auto drained = [&](unsigned v) {
      while (!ptx::mbar_try_wait(&arrived[(v & 1) ^ 1], (v >> 1) & 1u))
        if (ptx::globaltimer_ns() - since > JS_WAIT_NS) return false;
      return true;
    };
    bool ok = drained(late_visit);
    for (unsigned v = late_visit + 1; ok && v <= late_visit + 2 && v < visit; ++v) {
      ptx::mbar_arrive_expect_tx(&arrived[(v & 1) ^ 1], (visit - v + 1) / 2 * VISIT_BYTES);
      ok = drained(v);
    }
  }
  if (CLUSTER) {                       // (the columns lie as the next sweep's first step has them)
    int I, J;
    rr_pair(nb, 0, blockIdx.x, I, J);
    for (int e = warp; e < JG_M; e += (JS_G_THREADS + ROWS) / 32)
      for (int r = lane; r < n; r += 32)
        At[static_cast<long long>((e < b ? I * b + e : J * b + e - b)) * n + r] = (reinterpret_cast<Cols>(jacobi_cols) + (visit & 1) * JG_M)[e][r];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    info->sweeps = sweep;
    if (!alive && dev_status) atomicOr(dev_status, DEV_WAIT_EXPIRED);
    else if (!converged && mc2 >= JAC_FAIL_COS2 && dev_status) atomicOr(dev_status, DEV_JACOBI_NOCONV);
  }
}

// norms[i] = || column i of A || (row i of At): the shifted eigenvalues.
__global__ void __launch_bounds__(128) jacobi_norms_kernel(const double* At, int n, double* __restrict__ norms) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ double red[4];
  const double* row = At + static_cast<long long>(blockIdx.x) * n;
  double s = 0.0;
  for (int r = threadIdx.x; r < n; r += blockDim.x) s = fma(row[r], row[r], s);
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) norms[blockIdx.x] = sqrt(red[0] + red[1] + red[2] + red[3]);
}

// Rank the eigenvalues and gather the unit eigenvectors of the k largest into Wsel (ell x k,
// float), largest first; ties go to the lower index.  One CTA per eigenvalue.
__global__ void __launch_bounds__(128) select_topk_kernel(const double* At, const double* norms,
                                                          int n, int ell, int k, float* __restrict__ Wsel) {
  grid_dep_wait();
  grid_dep_launch();
  const int i = blockIdx.x;
  const double li = norms[i];
  __shared__ int rank_sh;
  if (threadIdx.x == 0) rank_sh = 0;
  __syncthreads();
  int cnt = 0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double lj = norms[j];
    if (lj > li || (lj == li && j < i)) ++cnt;
  }
  atomicAdd(&rank_sh, cnt);
  __syncthreads();
  const int rank = rank_sh;
  if (rank >= k) return;
  const double inv = li > 0.0 ? 1.0 / li : 0.0;
  for (int a = threadIdx.x; a < ell; a += blockDim.x)
    if (PRAC_IN(static_cast<long long>(a) * k + rank, static_cast<long long>(ell) * k))
      Wsel[static_cast<long long>(a) * k + rank] = static_cast<float>(At[static_cast<long long>(i) * n + a] * inv);
}

// x = hi + mid + lo, each piece a bf16 (round to nearest); the remainders are exact in fp32.
__device__ __forceinline__ void split3_one(float x, __nv_bfloat16& hi, __nv_bfloat16& mid, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(x);
  x -= __bfloat162float(hi);
  mid = __float2bfloat16_rn(x);
  x -= __bfloat162float(mid);
  lo = __float2bfloat16_rn(x);
}

// Pb[i][j] = bf16(P[i][j]);  PTb[j][i] = bf16(P[i][j]); 32 x 32 tiles through shared memory.  P3 (optional):
// the three pieces of P, rows3 rows apart.
__global__ void __launch_bounds__(256) make_bf16_copies_kernel(const float* P, long long ldp,
                                                               long long d, long long s,
                                                               __nv_bfloat16* __restrict__ Pb, long long ldpb,
                                                               __nv_bfloat16* __restrict__ PTb, long long ldptb,
                                                               __nv_bfloat16* __restrict__ Pcb, long long k, float c,
                                                               __nv_bfloat16* __restrict__ P3, long long rows3) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ float tile[32][33];
  const long long i0 = static_cast<long long>(blockIdx.y) * 32, j0 = static_cast<long long>(blockIdx.x) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  for (int r = ty; r < 32; r += 8) {
    const long long i = i0 + r, j = j0 + tx;
    const float v = (i < d && j < s) ? P[i * ldp + j] : 0.f;
    tile[r][tx] = v;
    if (i < d && j < s && PRAC_IN(i * ldpb + j, (d - 1) * ldpb + s)) {
      Pb[i * ldpb + j] = __float2bfloat16_rn(v);
      Pcb[i * ldpb + j] = __float2bfloat16_rn(j >= k ? c * v : v);   // [U | c Q]: operand of the rebuilt input
      if (P3) split3_one(v, P3[i * ldpb + j], P3[(rows3 + i) * ldpb + j], P3[(2 * rows3 + i) * ldpb + j]);
    }
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    const long long j = j0 + r, i = i0 + tx;
    if (i < d && j < s && PRAC_IN(j * ldptb + i, (s - 1) * ldptb + d)) PTb[j * ldptb + i] = __float2bfloat16_rn(tile[tx][r]);
  }
}

// One thread per 8 consecutive elements of a destination row (ldd is a multiple of 8).
__global__ void __launch_bounds__(256) split3_kernel(const float* src, long long lds, long long rows,
                                                     long long cols, __nv_bfloat16* __restrict__ dst,
                                                     long long rows_pad, long long ldd) {
  grid_dep_wait();
  grid_dep_launch();
  const long long groups = ldd / 8;
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= rows_pad * groups) return;
  const long long i = idx / groups, j0 = (idx - i * groups) * 8;
  float x[8];
  const float* s = src + i * lds + j0;
  if (i < rows && j0 + 8 <= cols && (reinterpret_cast<uintptr_t>(s) & 15u) == 0) {
    const float4 a = *reinterpret_cast<const float4*>(s), b = *(reinterpret_cast<const float4*>(s) + 1);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = (i < rows && j0 + e < cols) ? s[e] : 0.f;
  }
  __align__(16) __nv_bfloat16 hi[8], mid[8], lo[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) split3_one(x[e], hi[e], mid[e], lo[e]);
  const long long o = i * ldd + j0, plane = rows_pad * ldd;
  *reinterpret_cast<uint4*>(dst + o) = *reinterpret_cast<const uint4*>(hi);
  *reinterpret_cast<uint4*>(dst + plane + o) = *reinterpret_cast<const uint4*>(mid);
  *reinterpret_cast<uint4*>(dst + 2 * plane + o) = *reinterpret_cast<const uint4*>(lo);
}

// The transpose of scale * src (rows x cols, fp32) as three bf16 pieces side by side: dst[j][l],
// dst[j][kp + l], dst[j][2 kp + l] = leading, middle and last piece of scale * src[l][j]; l >= rows
// is filled with zeros.  (A small matrix: the K-major second operand of a panel product.)
__global__ void __launch_bounds__(256) split3_transposed_kernel(const float* src, long long lds, long long rows,
                                                                long long cols, float scale,
                                                                __nv_bfloat16* __restrict__ dst, long long kp) {
  grid_dep_wait();
  grid_dep_launch();
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= cols * kp) return;
  const long long j = idx / kp, l = idx - j * kp;
  float x = 0.f;
  if (l < rows && PRAC_IN(l * lds + j, (rows - 1) * lds + cols)) x = scale * src[l * lds + j];
  __nv_bfloat16 hi, mid, lo;
  split3_one(x, hi, mid, lo);
  __nv_bfloat16* o = dst + j * 3 * kp + l;
  o[0] = hi; o[kp] = mid; o[2 * kp] = lo;
}

// The three pieces of a row side by side: dst[i] = [hi_i | mid_i | lo_i], each kp wide.
__global__ void __launch_bounds__(256) split3_cols_kernel(const float* src, long long lds, long long rows,
                                                          long long cols, __nv_bfloat16* __restrict__ dst, long long kp) {
  grid_dep_wait();
  grid_dep_launch();
  const long long groups = kp / 8;
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= rows * groups) return;
  const long long i = idx / groups, j0 = (idx - i * groups) * 8;
  float x[8];
  const float* s = src + i * lds + j0;
  if (j0 + 8 <= cols && (reinterpret_cast<uintptr_t>(s) & 15u) == 0) {
    const float4 a = *reinterpret_cast<const float4*>(s), b = *(reinterpret_cast<const float4*>(s) + 1);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = (j0 + e < cols) ? s[e] : 0.f;
  }
  __align__(16) __nv_bfloat16 hi[8], mid[8], lo[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) split3_one(x[e], hi[e], mid[e], lo[e]);
  __nv_bfloat16* o = dst + i * 3 * kp + j0;
  *reinterpret_cast<uint4*>(o) = *reinterpret_cast<const uint4*>(hi);
  *reinterpret_cast<uint4*>(o + kp) = *reinterpret_cast<const uint4*>(mid);
  *reinterpret_cast<uint4*>(o + 2 * kp) = *reinterpret_cast<const uint4*>(lo);
}

// dX = dY * f'(Xh), element-wise (fp32 storage).
__global__ void __launch_bounds__(256) act_backward_f32_kernel(const float* Xh, long long ldxh,
                                                               const float* dY, long long lddy,
                                                               float* __restrict__ dX, long long lddx,
                                                               long long rows, long long cols, int act) {
  grid_dep_wait();
  grid_dep_launch();
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= rows * cols) return;
  const long long i = idx / cols, j = idx % cols;
  if (!PRAC_IN(i * lddx + j, (rows - 1) * lddx + cols) || !PRAC_IN(i * lddy + j, (rows - 1) * lddy + cols) ||
      !PRAC_IN(i * ldxh + j, (rows - 1) * ldxh + cols)) return;
  dX[i * lddx + j] = dY[i * lddy + j] * act_derivative(Xh[i * ldxh + j], act);
}

// Column sums of the pass-1 partials, shared by the two reductions below: a CTA closes 32 columns.
// Thread (g, q) adds, for the four columns 4q .. 4q + 3 of the CTA's 32, the partials of the 32-row
// blocks b = g, g + 32, ... (16-byte loads when the rows of col_part allow it); the 32 subtotals
// of a column are then combined in a fixed order, so the result does not depend on timing.
// Returns the column total in the threads with g == 0 && q < 8 as four values (columns 4q + e).
__device__ __forceinline__ void column_totals(const float* col_part, long long blocks, long long N,
                                              long long col0, float (&sub)[32][33], float (&tot)[4]) {
  const int g = threadIdx.x >> 3, q = threadIdx.x & 7;
  const long long c = col0 + 4 * q;
  float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
  const bool vec = (N % 4 == 0) && ((reinterpret_cast<uintptr_t>(col_part) & 15u) == 0) && c + 4 <= N;
  if (vec) {
#pragma unroll 16
    for (long long b = g; b < blocks; b += 32) {
      const float4 v = *reinterpret_cast<const float4*>(col_part + b * N + c);
      a0 += v.x; a1 += v.y; a2 += v.z; a3 += v.w;
    }
  } else {
    for (long long b = g; b < blocks; b += 4 * 32) {       // (four blocks' loads in flight together)
      float v[4][4];
#pragma unroll
      for (int h = 0; h < 4; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const long long bb = b + 32 * h < blocks ? b + 32 * h : b, cc = c + e < N ? c + e : N - 1;
          v[h][e] = col_part[bb * N + cc];
        }
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (b + 32 * h >= blocks) break;
        a0 += v[h][0]; a1 += v[h][1]; a2 += v[h][2]; a3 += v[h][3];
      }
    }
  }
  __syncthreads();                // an earlier call's readers are done with `sub`
  sub[g][4 * q] = a0; sub[g][4 * q + 1] = a1; sub[g][4 * q + 2] = a2; sub[g][4 * q + 3] = a3;
  __syncthreads();
  tot[0] = tot[1] = tot[2] = tot[3] = 0.f;
  if (g == 0) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float t = 0.f;
#pragma unroll 8
      for (int h = 0; h < 32; ++h) t += sub[h][4 * q + e];
      tot[e] = t;
    }
  }
}

// After pass 1 of the RMSNorm backward.  The first ceil(M / 256) CTAs close the row sums (one
// thread per token); each of the others closes 32 column sums (column_totals).
__global__ void __launch_bounds__(256) rms_reduce_kernel(const float* row_part, int parts,
                                                         const float* col_part, long long blocks,
                                                         const float* rstd, long long M, long long N,
                                                         float* __restrict__ row_b, float* __restrict__ dgain) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ float sub[32][33];
  const long long row_ctas = (M + 255) / 256;
  if (blockIdx.x < row_ctas) {
    const long long idx = blockIdx.x * 256ll + threadIdx.x;
    if (idx < M) {
      float u = 0.f;
#pragma unroll 16
      for (int p = 0; p < parts; ++p) u += row_part[static_cast<long long>(p) * M + idx];
      const float rs = rstd[idx];
      row_b[idx] = rs * rs * rs * u / static_cast<float>(N);
    }
    return;
  }
  const long long col0 = (blockIdx.x - row_ctas) * 32;
  float tot[4];
  column_totals(col_part, blocks, N, col0, sub, tot);
  if (threadIdx.x < 8) {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (col0 + 4 * threadIdx.x + e < N) dgain[col0 + 4 * threadIdx.x + e] = tot[e];
  }
}

// LayerNorm backward, the part that does not need the rebuilt input: per column i the sums over
// 512 tokens of dY[t][i] and of rstd[t] mean[t] dY[t][i].  Grid (ceil(N / 256), ceil(M / 512)).
// Thread (g, q) takes the eight columns 8q .. 8q + 7 of the CTA's 256 (one 16-byte load per row
// when VEC: rows of dY 16-byte aligned and padded to a multiple of 8) and the rows g, g + 8, ...
// of its 512; the eight subtotals of a column are combined in order.  An ordinary launch, which waits for the
// end of the kernel before it, so that the inputs may be read through the non-coherent path (4096 x 1179, the
// whole backward: 57 us on padded rows and 70 on contiguous ones, with an early launch 65 and 98).
template <bool VEC>
__global__ void __launch_bounds__(256) ln_colsum_partial_kernel(const __nv_bfloat16* __restrict__ dY, long long lddy,
                                                                const float* __restrict__ mean, const float* __restrict__ rstd,
                                                                long long M, long long N, float* __restrict__ part_plain,
                                                                float* __restrict__ part_w) {
  __shared__ float sp[8][257], sw[8][257];
  const int g = threadIdx.x >> 5, q = threadIdx.x & 31;
  const long long c0 = blockIdx.x * 256ll + 8 * q;
  const long long r0 = blockIdx.y * 512ll, r1 = (r0 + 512 < M) ? r0 + 512 : M;
  float ap[8], aw[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) ap[e] = aw[e] = 0.f;
  if (c0 < N) {
#pragma unroll 4
    for (long long t = r0 + g; t < r1; t += 8) {
      const float wgt = __ldg(rstd + t) * __ldg(mean + t);
      const __nv_bfloat16* row = dY + t * lddy + c0;
      if (VEC) {
        // (a group of eight that straddles the last column is still inside the padded row)
        const uint4 raw = __ldg(reinterpret_cast<const uint4*>(row));
        const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&raw);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float v = __bfloat162float(h[e]);
          ap[e] += v;
          aw[e] = fmaf(wgt, v, aw[e]);
        }
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          if (c0 + e < N && PRAC_IN(t * lddy + c0 + e, (M - 1) * lddy + N)) {
            const float v = __bfloat162float(row[e]);
            ap[e] += v;
            aw[e] = fmaf(wgt, v, aw[e]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) { sp[g][8 * q + e] = ap[e]; sw[g][8 * q + e] = aw[e]; }
  __syncthreads();
  const long long col = blockIdx.x * 256ll + threadIdx.x;
  if (col < N) {
    float tp = 0.f, tw = 0.f;
#pragma unroll
    for (int h = 0; h < 8; ++h) { tp += sp[h][threadIdx.x]; tw += sw[h][threadIdx.x]; }
    part_plain[blockIdx.y * N + col] = tp;
    part_w[blockIdx.y * N + col] = tw;
  }
}

// After pass 1 of the LayerNorm backward (layout as rms_reduce_kernel).  Rows: with S = sum_i a x,
// A = sum_i a (a = gain dY): u = rstd (S - mean A); row_b = rstd^2 u / N; row_c = -rstd A / N + row_b mean.
// Columns: dgain = sum of the pass-1 column partials - sum of the weighted partials; dbias = sum
// of the plain partials.
__global__ void __launch_bounds__(256) ln_reduce_kernel(const float* row_part, const float* row_part2,
                                                        int parts, const float* col_part, long long blocks,
                                                        const float* part_plain, const float* part_w,
                                                        long long groups, const float* mean,
                                                        const float* rstd, long long M, long long N,
                                                        float* __restrict__ row_b, float* __restrict__ row_c,
                                                        float* __restrict__ dgain, float* __restrict__ dbias) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ float sub[32][33];
  const long long row_ctas = (M + 255) / 256;
  if (blockIdx.x < row_ctas) {
    const long long idx = blockIdx.x * 256ll + threadIdx.x;
    if (idx < M) {
      float S = 0.f, A = 0.f;
      for (int p = 0; p < parts; ++p) {
        S += row_part[static_cast<long long>(p) * M + idx];
        A += row_part2[static_cast<long long>(p) * M + idx];
      }
      const float rs = rstd[idx], mu = mean[idx], inv = 1.f / static_cast<float>(N);
      const float u = rs * (S - mu * A);
      const float rb = rs * rs * u * inv;
      row_b[idx] = rb;
      row_c[idx] = fmaf(rb, mu, -rs * A * inv);
    }
    return;
  }
  const long long col0 = (blockIdx.x - row_ctas) * 32;
  float tot[4], tw[4], tp[4];
  column_totals(col_part, blocks, N, col0, sub, tot);
  column_totals(part_w, groups, N, col0, sub, tw);
  column_totals(part_plain, groups, N, col0, sub, tp);
  if (threadIdx.x < 8) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const long long col = col0 + 4 * threadIdx.x + e;
      if (col < N) {
        dgain[col] = tot[e] - tw[e];
        dbias[col] = tp[e];
      }
    }
  }
}

// fp32 storage, one CTA per token: A = sum a, S = sum a xn (a = gain dY, xn = (x - mean) rstd), then
// dX = rstd (a - A / N - xn S / N).
__global__ void __launch_bounds__(256) ln_rows_f32_kernel(const float* Xh, long long ldxh,
                                                          const float* dY, long long lddy,
                                                          const float* mean, const float* rstd,
                                                          const float* gain, float* __restrict__ dX,
                                                          long long lddx, long long N) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ double ra[256], rb[256];
  const long long t = blockIdx.x;
  const float* x = Xh + t * ldxh;
  const float* y = dY + t * lddy;
  const float mu = mean[t], rs = rstd[t];
  double A = 0.0, S = 0.0;
  for (long long i = threadIdx.x; i < N; i += blockDim.x) {
    const double a = static_cast<double>(gain[i]) * y[i];
    A += a;
    S += a * ((x[i] - mu) * rs);
  }
  ra[threadIdx.x] = A; rb[threadIdx.x] = S;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) { ra[threadIdx.x] += ra[threadIdx.x + o]; rb[threadIdx.x] += rb[threadIdx.x + o]; }
    __syncthreads();
  }
  const float mA = static_cast<float>(ra[0] / static_cast<double>(N)), mS = static_cast<float>(rb[0] / static_cast<double>(N));
  for (long long i = threadIdx.x; i < N; i += blockDim.x)
    dX[t * lddx + i] = rs * (gain[i] * y[i] - mA - (x[i] - mu) * rs * mS);
}
// fp32 storage: dgain_i = sum_t dY_ti xn_ti, dbias_i = sum_t dY_ti; one thread per column, rows in order.
__global__ void __launch_bounds__(256) ln_cols_f32_kernel(const float* Xh, long long ldxh,
                                                          const float* dY, long long lddy,
                                                          const float* mean, const float* rstd,
                                                          float* __restrict__ dgain, float* __restrict__ dbias,
                                                          long long M, long long N) {
  grid_dep_wait();
  grid_dep_launch();
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (i >= N) return;
  double sg = 0.0, sb = 0.0;
  for (long long t = 0; t < M; ++t) {
    const double y = dY[t * lddy + i];
    sg += y * ((Xh[t * ldxh + i] - mean[t]) * rstd[t]);
    sb += y;
  }
  dgain[i] = static_cast<float>(sg);
  dbias[i] = static_cast<float>(sb);
}

// fp32 storage, one CTA per token: u = sum_i gain_i dY_i x_i, then dX = rstd gain dY - rstd^3 u / N x.
__global__ void __launch_bounds__(256) rms_rows_f32_kernel(const float* Xh, long long ldxh,
                                                           const float* dY, long long lddy,
                                                           const float* rstd, const float* gain,
                                                           float* __restrict__ dX, long long lddx, long long N) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ double red[256];
  const long long t = blockIdx.x;
  const float* x = Xh + t * ldxh;
  const float* y = dY + t * lddy;
  double u = 0.0;
  for (long long i = threadIdx.x; i < N; i += blockDim.x) u += static_cast<double>(gain[i]) * y[i] * x[i];
  red[threadIdx.x] = u;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  const float rs = rstd[t];
  const float coef = static_cast<float>(static_cast<double>(rs) * rs * rs * red[0] / static_cast<double>(N));
  for (long long i = threadIdx.x; i < N; i += blockDim.x) dX[t * lddx + i] = rs * gain[i] * y[i] - coef * x[i];
}
// fp32 storage: dgain_i = sum_t dY_ti x_ti rstd_t, one thread per column, rows in order.
__global__ void __launch_bounds__(256) rms_cols_f32_kernel(const float* Xh, long long ldxh,
                                                           const float* dY, long long lddy,
                                                           const float* rstd, float* __restrict__ dgain,
                                                           long long M, long long N) {
  grid_dep_wait();
  grid_dep_launch();
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (i >= N) return;
  double sacc = 0.0;
  for (long long t = 0; t < M; ++t) sacc += static_cast<double>(dY[t * lddy + i]) * Xh[t * ldxh + i] * rstd[t];
  dgain[i] = static_cast<float>(sacc);
}

// dst (bf16) = src with columns from `from` on multiplied by scale.
__global__ void __launch_bounds__(256) scale_to_bf16_kernel(const float* src, long long lds,
                                                            long long rows, long long cols, long long from, float scale,
                                                            __nv_bfloat16* __restrict__ dst, long long ldd) {
  grid_dep_wait();
  grid_dep_launch();
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= rows * cols) return;
  const long long i = idx / cols, j = idx % cols;
  if (!PRAC_IN(i * lds + j, (rows - 1) * lds + cols) || !PRAC_IN(i * ldd + j, (rows - 1) * ldd + cols)) return;
  const float v = src[i * lds + j];
  dst[i * ldd + j] = __float2bfloat16_rn(j >= from ? scale * v : v);
}

__global__ void copy2d_kernel(const float* src, long long lds, float* __restrict__ dst,
                              long long ldd, long long rows, long long cols) {
  grid_dep_wait();
  grid_dep_launch();
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= rows * cols) return;
  const long long i = idx / cols, j = idx % cols;
  if (!PRAC_IN(i * lds + j, (rows - 1) * lds + cols) || !PRAC_IN(i * ldd + j, (rows - 1) * ldd + cols)) return;
  dst[i * ldd + j] = src[i * lds + j];
}

// dst (rows x cols bf16, leading dimension ldd: rows 16-byte aligned, zero beyond cols up to ldd)
// = src (rows x cols bf16, any leading dimension, 2-byte aligned).  One thread per 8 destination
// elements: eight 2-byte loads (coalesced across the warp), one 16-byte store.
__global__ void __launch_bounds__(256) repack_rows_bf16_kernel(const __nv_bfloat16* src, long long lds,
                                                               long long rows, long long cols,
                                                               __nv_bfloat16* __restrict__ dst, long long ldd) {
  grid_dep_wait();
  grid_dep_launch();
  const long long groups = ldd / 8;
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= rows * groups) return;
  const long long i = idx / groups, j0 = (idx - i * groups) * 8;
  const unsigned short* s16 = reinterpret_cast<const unsigned short*>(src + i * lds + j0);
  unsigned short v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) v[e] = (j0 + e < cols) ? s16[e] : static_cast<unsigned short>(0);
  if (!PRAC_IN(i * ldd + j0 + 7, rows * ldd)) return;
  uint4 o;
  o.x = v[0] | (static_cast<uint32_t>(v[1]) << 16);
  o.y = v[2] | (static_cast<uint32_t>(v[3]) << 16);
  o.z = v[4] | (static_cast<uint32_t>(v[5]) << 16);
  o.w = v[6] | (static_cast<uint32_t>(v[7]) << 16);
  *reinterpret_cast<uint4*>(dst + i * ldd + j0) = o;
}

inline unsigned nblocks(long long work, int threads) {
  return static_cast<unsigned>((work + threads - 1) / threads);
}

}  // namespace

PRAC_BOUNDS_READER(bounds_violations_panel)

int launch_repack_rows_bf16(const __nv_bfloat16* src, int64_t lds, int64_t rows, int64_t cols, __nv_bfloat16* dst,
                            int64_t ldd, cudaStream_t stream) {
  if (rows <= 0 || cols <= 0) return PRAC_OK;
  if (ldd % 8 != 0 || ldd < cols || (reinterpret_cast<uintptr_t>(dst) & 15u) != 0) return PRAC_EALIGN;
  PRAC_LAUNCH(repack_rows_bf16_kernel, dim3(nblocks(rows * (ldd / 8), 256)), dim3(256), 0, stream, src, lds, rows, cols, dst, ldd);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_philox_words(uint64_t seed, uint64_t dc, int64_t n, uint32_t* out, cudaStream_t stream) {
  if (n <= 0) return PRAC_OK;
  PRAC_LAUNCH(philox_words_kernel, dim3(nblocks((n + 3) / 4, 256)), dim3(256), 0, stream, seed, dc, n, out);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_gaussian(uint64_t seed, uint64_t dc, int64_t d, int64_t r, float* S, int64_t lds,
                    cudaStream_t stream) {
  if (d <= 0 || r <= 0) return PRAC_OK;
  PRAC_LAUNCH(gaussian_kernel, dim3(nblocks((d * r + 3) / 4, 256)), dim3(256), 0, stream, seed, dc, d, r, S, lds);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

// Eigen-solver workspace: At n*n double | norms n double | info   (n = ell rounded up to 16)
namespace {
struct JacWs { double* At; double* norms; JacobiInfo* info; double* terms; size_t bytes; int64_t n; };
JacWs carve_jac(void* ws, int64_t ell) {
  JacWs j;
  j.n = round_up(ell, 16);
  size_t off = 0;
  auto take = [&](size_t b) { size_t o = off; off += (b + 255) / 256 * 256; return o; };
  const size_t o1 = take(j.n * j.n * 8), o2 = take(j.n * 8), o3 = take(sizeof(JacobiInfo));
  const size_t o4 = take(j.n <= 128 ? 2 * j.n * j.n * 8 : 0);
  char* b = static_cast<char*>(ws);
  j.At = reinterpret_cast<double*>(b + o1); j.norms = reinterpret_cast<double*>(b + o2);
  j.info = reinterpret_cast<JacobiInfo*>(b + o3); j.terms = reinterpret_cast<double*>(b + o4);
  j.bytes = off;
  return j;
}
}  // namespace

size_t jacobi_ws_bytes(int64_t ell) { return ell > 0 ? carve_jac(nullptr, ell).bytes : 0; }

int jacobi_read_sweeps(void* ws, int64_t ell, int* sweeps, cudaStream_t stream) {
  if (!ws || ell <= 0 || !sweeps) return PRAC_EINVAL;
  const JacWs j = carve_jac(ws, ell);
  PRAC_CUDA_TRY(cudaStreamSynchronize(stream));
  JacobiInfo h;
  PRAC_CUDA_TRY(cudaMemcpy(&h, j.info, sizeof(JacobiInfo), cudaMemcpyDeviceToHost));
  *sweeps = h.sweeps;
  return PRAC_OK;
}

int jacobi_topk(const double* B, int64_t ldb, int64_t ell, int64_t k, float* Wsel, void* ws, size_t ws_bytes,
                int* dev_status, cudaStream_t stream) {
  if (ell <= 0 || k <= 0 || k > ell || ldb < ell) return PRAC_EINVAL;
  const JacWs j = carve_jac(ws, ell);
  if (ws == nullptr || ws_bytes < j.bytes) return PRAC_EWORKSPACE;
  const int n = static_cast<int>(j.n);
  // columns per block: as many as fit in shared memory, two blocks per CTA, at least two blocks
  // 8 columns per block = 256 threads per CTA: measured faster than 16 (more CTAs share the
  // rotations, and the 20-element register variant fits the register file)
  int bcols = 8;
  while (bcols > 4 && static_cast<size_t>(2 * bcols) * n * 8 > 200u * 1024u) bcols /= 2;
  const size_t smem = static_cast<size_t>(2 * bcols) * n * 8;
  if (smem > 200u * 1024u) return PRAC_EINVAL;
  void (*kern)(double*, int, int, int, double, JacobiInfo*, int*, unsigned) =
      n <= 32 * 12 ? jacobi_kernel<12> : (n <= 32 * 20 ? jacobi_kernel<20> : jacobi_kernel<0>);
  int sms = 0, dev = 0, per_sm = 0;
  PRAC_CUDA_TRY(cudaGetDevice(&dev));
  static DeviceOnce attr_set;      // function attributes belong to the device that was current
  if (!attr_set.done(dev)) {
    PRAC_CUDA_TRY(cudaFuncSetAttribute(jacobi_kernel<12>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    PRAC_CUDA_TRY(cudaFuncSetAttribute(jacobi_kernel<20>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    PRAC_CUDA_TRY(cudaFuncSetAttribute(jacobi_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    attr_set.mark(dev);
  }
  const int nb = n / bcols;
  const int grid = (nb + (nb & 1)) / 2;
  PRAC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // 8-column blocks take a Gram-matrix kernel (rotations streamed to the threads that hold the rows up to
  // n = 256, the most rows they can hold); narrower blocks (very long columns) the plain one
  const bool gram = (bcols == JG_B), stream_rows = gram && n <= JS_MAX_ROWS;
  const size_t gram_smem = (static_cast<size_t>(JG_M) * (n + 4) + 4 * JG_M * JG_P + 8 * 3 * 64) * 8 + JG_M * sizeof(JgCoef);
  if (gram && !stream_rows) {
    static DeviceOnce gram_attr;
    if (!gram_attr.done(dev)) {
      PRAC_CUDA_TRY(cudaFuncSetAttribute(jacobi_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
      gram_attr.mark(dev);
    }
    PRAC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, jacobi_gram_kernel, 256, gram_smem));
  } else if (!gram) {
    PRAC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * bcols, smem));
  } else {
    per_sm = 1;                                                // at most 16 CTAs
  }
  if (per_sm < 1 || grid > per_sm * sms) return PRAC_EINVAL;   // the barrier needs every CTA resident
  PRAC_LAUNCH(jacobi_prepare_kernel, dim3(64), dim3(256), 0, stream, B, ldb, static_cast<int>(ell), j.At, n, j.info);
  count_launch();
  double* at = j.At;
  int ni = n, bi = bcols, max_sweeps = JAC_MAX_SWEEPS;
  // (larger problems) a pair of columns whose cosine is below this is left alone: far below what the fp32
  // result keeps
  double tol = 1e-9;
  JacobiInfo* info = j.info;
  unsigned poll_limit = barrier_poll_limit();
  if (stream_rows) {
    // Up to 16 CTAs (eigenproblems up to 256 columns: the Rayleigh-Ritz windows of k <= 512) run as
    // one cluster on the hardware barrier (more than 8 CTAs is a cluster size the device has to
    // allow and be able to place: the occupancy query below decides), unless a test has shortened
    // the software barrier's poll limit, which only that barrier can honour.
    void (*const on_cluster)(double*, double*, int, int, JacobiInfo*, int*, unsigned) =
        n <= 128 ? jacobi_stream_kernel<true, 128> : jacobi_stream_kernel<true, 256>;
    void (*const on_grid)(double*, double*, int, int, JacobiInfo*, int*, unsigned) =
        n <= 128 ? jacobi_stream_kernel<false, 128> : jacobi_stream_kernel<false, 256>;
    const unsigned threads = JS_G_THREADS + (n <= 128 ? 128 : 256);
    const int cols_smem = (n <= 128 ? 4 : 2) * JG_M * ((n <= 128 ? 128 : 256) + 2) * 8;
    bool as_cluster = poll_limit == GRID_BARRIER_POLLS;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = cols_smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = grid;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = dependent_launch_attr();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if (as_cluster) {
      static DeviceOnce smem_attr[2];
      DeviceOnce& once = smem_attr[n <= 128 ? 0 : 1];
      if (!once.done(dev)) {
        PRAC_CUDA_TRY(cudaFuncSetAttribute(on_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, cols_smem));
        once.mark(dev);
      }
    }
    if (as_cluster && grid > 8) {
      static DeviceOnce wide_attr;
      if (!wide_attr.done(dev)) {
        if (cudaFuncSetAttribute(on_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
          (void)cudaGetLastError();
          as_cluster = false;
        } else {
          wide_attr.mark(dev);
        }
      }
    }
    if (as_cluster) {
      int clusters = 0;
      if (cudaOccupancyMaxActiveClusters(&clusters, on_cluster, &cfg) != cudaSuccess || clusters < 1) {
        (void)cudaGetLastError();
        as_cluster = false;
      }
    }
    if (as_cluster) {
      PRAC_CUDA_TRY(cudaLaunchKernelEx(&cfg, on_cluster, at, j.terms, ni, max_sweeps, info, dev_status, column_poll_limit()));
    } else {
      double* terms = j.terms;
      void* sargs[] = {&at, &terms, &ni, &max_sweeps, &info, &dev_status, &poll_limit};
      static DeviceOnce grid_attr;
      if (n <= 128 && !grid_attr.done(dev)) {
        PRAC_CUDA_TRY(cudaFuncSetAttribute(on_grid, cudaFuncAttributeMaxDynamicSharedMemorySize, cols_smem));
        grid_attr.mark(dev);
      }
      PRAC_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(on_grid), dim3(grid), dim3(threads), sargs,
                                                n <= 128 ? cols_smem : 0, stream));   // (a finishing step's matrices)
    }
  } else if (gram) {
    void* gargs[] = {&at, &ni, &max_sweeps, &tol, &info, &dev_status, &poll_limit};
    PRAC_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(jacobi_gram_kernel), dim3(grid), dim3(256),
                                              gargs, gram_smem, stream));
  } else {
    void* args[] = {&at, &ni, &bi, &max_sweeps, &tol, &info, &dev_status, &poll_limit};
    PRAC_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(kern), dim3(grid), dim3(32 * bcols), args,
                                              smem, stream));
  }
  count_launch();
  PRAC_LAUNCH(jacobi_norms_kernel, dim3(n), dim3(128), 0, stream, j.At, n, j.norms);
  count_launch();
  PRAC_LAUNCH(select_topk_kernel, dim3(n), dim3(128), 0, stream, j.At, j.norms, n, static_cast<int>(ell), static_cast<int>(k), Wsel);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_make_bf16_copies(const float* P, int64_t ldp, int64_t d, int64_t s, int64_t k, double c,
                            __nv_bfloat16* Pcb, __nv_bfloat16* Pb, int64_t ldpb,
                            __nv_bfloat16* PTb, int64_t ldptb, __nv_bfloat16* P3, int64_t rows3, cudaStream_t stream) {
  dim3 grid(static_cast<unsigned>((s + 31) / 32), static_cast<unsigned>((d + 31) / 32));
  PRAC_LAUNCH(make_bf16_copies_kernel, dim3(grid), dim3(256), 0, stream,
              P, ldp, d, s, Pb, ldpb, PTb, ldptb, Pcb, k, static_cast<float>(c), P3, rows3);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_split3(const float* src, int64_t lds, int64_t rows, int64_t cols, __nv_bfloat16* dst,
                  int64_t rows_pad, int64_t ldd, cudaStream_t stream) {
  if (rows <= 0 || cols <= 0) return PRAC_OK;
  if (ldd % 8 != 0 || (reinterpret_cast<uintptr_t>(dst) & 15u) != 0) return PRAC_EALIGN;
  PRAC_LAUNCH(split3_kernel, dim3(nblocks(rows_pad * (ldd / 8), 256)), dim3(256), 0, stream, src, lds, rows, cols, dst, rows_pad, ldd);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_split3_transposed(const float* src, int64_t lds, int64_t rows, int64_t cols, float scale,
                             __nv_bfloat16* dst, int64_t kp, cudaStream_t stream) {
  if (rows <= 0 || cols <= 0) return PRAC_OK;
  if (kp < rows) return PRAC_EINVAL;
  PRAC_LAUNCH(split3_transposed_kernel, dim3(nblocks(cols * kp, 256)), dim3(256), 0, stream, src, lds, rows, cols, scale, dst, kp);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_split3_cols(const float* src, int64_t lds, int64_t rows, int64_t cols, __nv_bfloat16* dst, int64_t kp,
                       cudaStream_t stream) {
  if (rows <= 0 || cols <= 0) return PRAC_OK;
  if (kp % 8 != 0 || kp < cols || (reinterpret_cast<uintptr_t>(dst) & 15u) != 0) return PRAC_EALIGN;
  PRAC_LAUNCH(split3_cols_kernel, dim3(nblocks(rows * (kp / 8), 256)), dim3(256), 0, stream, src, lds, rows, cols, dst, kp);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_rms_reduce(const float* row_part, int parts, const float* col_part, int64_t blocks, const float* rstd,
                      int64_t M, int64_t N, float* row_b, float* dgain, cudaStream_t stream) {
  const unsigned ctas = nblocks(M, 256) + nblocks(N, 32);
  PRAC_LAUNCH(rms_reduce_kernel, dim3(ctas), dim3(256), 0, stream, row_part, parts, col_part, blocks, rstd, M, N, row_b, dgain);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_ln_colsum_partial(const __nv_bfloat16* dY, int64_t lddy, const float* mean, const float* rstd, int64_t M,
                             int64_t N, float* part_plain, float* part_w, cudaStream_t stream) {
  dim3 grid(nblocks(N, 256), nblocks(M, 512));
  const bool vec = (reinterpret_cast<uintptr_t>(dY) & 15u) == 0 && lddy % 8 == 0 && lddy >= (N + 7) / 8 * 8;
  if (vec) ln_colsum_partial_kernel<true><<<grid, 256, 0, stream>>>(dY, lddy, mean, rstd, M, N, part_plain, part_w);
  else ln_colsum_partial_kernel<false><<<grid, 256, 0, stream>>>(dY, lddy, mean, rstd, M, N, part_plain, part_w);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_ln_reduce(const float* row_part, const float* row_part2, int parts, const float* col_part, int64_t blocks,
                     const float* part_plain, const float* part_w, int64_t groups, const float* mean, const float* rstd,
                     int64_t M, int64_t N, float* row_b, float* row_c, float* dgain, float* dbias, cudaStream_t stream) {
  const unsigned ctas = nblocks(M, 256) + nblocks(N, 32);
  PRAC_LAUNCH(ln_reduce_kernel, dim3(ctas), dim3(256), 0, stream,
              row_part, row_part2, parts, col_part, blocks, part_plain, part_w, groups, mean, rstd, M, N, row_b, row_c,
              dgain, dbias);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_ln_backward_f32(const float* Xh, int64_t ldxh, const float* dY, int64_t lddy, const float* mean,
                           const float* rstd, const float* gain, float* dX, int64_t lddx, float* dgain, float* dbias,
                           int64_t M, int64_t N, cudaStream_t stream) {
  PRAC_LAUNCH(ln_rows_f32_kernel, dim3(static_cast<unsigned>(M)), dim3(256), 0, stream, Xh, ldxh, dY, lddy, mean, rstd, gain, dX, lddx, N);
  count_launch();
  PRAC_LAUNCH(ln_cols_f32_kernel, dim3(nblocks(N, 256)), dim3(256), 0, stream, Xh, ldxh, dY, lddy, mean, rstd, dgain, dbias, M, N);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_rms_backward_f32(const float* Xh, int64_t ldxh, const float* dY, int64_t lddy, const float* rstd,
                            const float* gain, float* dX, int64_t lddx, float* dgain, int64_t M, int64_t N,
                            cudaStream_t stream) {
  PRAC_LAUNCH(rms_rows_f32_kernel, dim3(static_cast<unsigned>(M)), dim3(256), 0, stream, Xh, ldxh, dY, lddy, rstd, gain, dX, lddx, N);
  count_launch();
  PRAC_LAUNCH(rms_cols_f32_kernel, dim3(nblocks(N, 256)), dim3(256), 0, stream, Xh, ldxh, dY, lddy, rstd, dgain, M, N);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_scale_to_bf16(const float* src, int64_t lds, int64_t rows, int64_t cols, int64_t from, float scale,
                         __nv_bfloat16* dst, int64_t ldd, cudaStream_t stream) {
  if (rows <= 0 || cols <= 0) return PRAC_OK;
  PRAC_LAUNCH(scale_to_bf16_kernel, dim3(nblocks(rows * cols, 256)), dim3(256), 0, stream, src, lds, rows, cols, from, scale, dst, ldd);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_act_backward_f32(const float* Xh, int64_t ldxh, const float* dY, int64_t lddy, float* dX, int64_t lddx,
                            int64_t rows, int64_t cols, int act, cudaStream_t stream) {
  if (rows <= 0 || cols <= 0) return PRAC_OK;
  PRAC_LAUNCH(act_backward_f32_kernel, dim3(nblocks(rows * cols, 256)), dim3(256), 0, stream,
              Xh, ldxh, dY, lddy, dX, lddx, rows, cols, act);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

int launch_copy2d(const float* src, int64_t lds, float* dst, int64_t ldd, int64_t rows, int64_t cols,
                  cudaStream_t stream) {
  if (rows <= 0 || cols <= 0) return PRAC_OK;
  PRAC_LAUNCH(copy2d_kernel, dim3(nblocks(rows * cols, 256)), dim3(256), 0, stream, src, lds, dst, ldd, rows, cols);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

}  // namespace prac
