// Orthonormalisation of tall fp32 panels by Cholesky-QR, three launches per pass:
//   1. G = V^T V accumulated in double over slices of the rows (atb_f64_partial_kernel) and
//      summed in a fixed order (reduce_partials_kernel);
//   2. R = chol(G) and R^-1 in one cooperative kernel (chol_inv_kernel), all in double;
//   3. V_out = V_in * R^-1: on the tensor cores for panels big enough to fill their tiles (both
//      operands as three bf16 pieces, six chained cross terms: fp32 accuracy), else a general
//      fp32 GEMM.
// R has a positive diagonal, so V R^-1 is the unique thin-QR Q factor.  The same
// transposed-product kernel serves every small "tall^T x tall" product of the basis fit.
#include <cuda_runtime.h>

#include "internal.h"
#include "per_device.h"

namespace prac {
namespace {

inline unsigned nblocks(long long work, int threads) {
  return static_cast<unsigned>((work + threads - 1) / threads);
}

// ------------------------------------------------------------------ Out = A^T B, double accumulation
constexpr int AT_T = 64;     // output tile
constexpr int AT_K = 16;     // rows per staging step

struct AtbArgs {
  const float* A; long long lda;   // d x m
  const float* B; long long ldb;   // d x n
  int m, n;
  long long d;
  int splits;                      // row slices
  int tiles_m, tiles_n, num_tiles;
  int symmetric;                   // A == B, m == n: only tiles reaching the upper triangle
  double* partial;                 // [splits][m][n]
  const int* run_if;               // optional: the kernel does nothing unless *run_if & run_if_mask
  int run_if_mask;
};

// Kernels of an optional pass are always launched and look at a device word to see whether
// they have anything to do (the host does not wait for the device to find out).
__device__ __forceinline__ bool pass_is_off(const int* run_if, int mask) {
  return run_if != nullptr && (*reinterpret_cast<const volatile int*>(run_if) & mask) == 0;
}

__device__ __forceinline__ void atb_tile(const AtbArgs& g, int tile, int& ti, int& tj) {
  if (!g.symmetric) { ti = tile / g.tiles_n; tj = tile % g.tiles_n; return; }
  int row = 0, rest = tile;
  while (true) {
    const int cnt = g.tiles_n - row;
    if (rest < cnt) { ti = row; tj = row + rest; return; }
    rest -= cnt;
    ++row;
  }
}

// One double-precision tensor-core product: D (8 x 8) += A (8 x 4, row-major fragment) * B (4 x 8,
// column-major fragment).  Lane L holds A[L / 4][L % 4], B[L % 4][L / 4] and D[L / 4][2 (L % 4) + {0, 1}].
__device__ __forceinline__ void dmma_884(double (&d)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
               : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

// A 64 x 64 output tile over one slice of the rows: 16 rows at a time are widened to double in
// shared memory (the next 16 are already on their way in registers), warp w multiplies 16 columns
// of A (w / 2) by 32 columns of B (w % 2) on the fp64 tensor cores: six fragment loads for eight
// products (the kernel waits on its shared-memory loads; 8 x 64 per warp took nine).
__global__ void __launch_bounds__(256) atb_f64_partial_kernel(const AtbArgs g) {
  grid_dep_wait();
  __shared__ double As[AT_K][AT_T + 2];
  __shared__ double Bs[AT_K][AT_T + 2];
  if (pass_is_off(g.run_if, g.run_if_mask)) return;
  int ti, tj;
  atb_tile(g, blockIdx.x, ti, tj);
  const int split = blockIdx.y;
  const long long r0 = g.d * split / g.splits, r1 = g.d * (split + 1) / g.splits;
  const int t = threadIdx.x;
  const int warp = t >> 5, lane = t & 31, gq = lane >> 2, q4 = lane & 3;
  const int m0 = ti * AT_T, n0 = tj * AT_T;
  const int wa = (warp >> 1) * 16, wb = (warp & 1) * 32;   // this warp's columns of A and of B within the tile
  double acc[2][4][2];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < 4; ++c) { acc[h][c][0] = 0.0; acc[h][c][1] = 0.0; }
  // staging: row lr of the chunk, columns lc, lc + 16, lc + 32, lc + 48: the 16 threads of a row write
  // 16 consecutive doubles per store (one shared-memory wavefront per row; four columns per thread
  // side by side made every store an eight-way bank conflict)
  const int lr = t >> 4, lc = t & 15;
  // two chunks of 16 rows are on their way in registers while a third is multiplied (one was not
  // enough to cover the loads' latency: the long slices of a wide panel took 2 us per chunk)
  float ra[2][4], rb[2][4];
  auto fetch = [&](long long k0, float (&fa)[4], float (&fb)[4]) {
    const long long row = k0 + lr;
    const bool in_k = row < r1;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int ca = m0 + lc + 16 * e, cb = n0 + lc + 16 * e;
      fa[e] = (in_k && ca < g.m && PRAC_IN(row * g.lda + ca, (g.d - 1) * g.lda + g.m)) ? g.A[row * g.lda + ca] : 0.f;
      fb[e] = (in_k && cb < g.n && PRAC_IN(row * g.ldb + cb, (g.d - 1) * g.ldb + g.n)) ? g.B[row * g.ldb + cb] : 0.f;
    }
  };
  fetch(r0, ra[0], rb[0]);
  fetch(r0 + AT_K, ra[1], rb[1]);
  int cur = 0;
  for (long long k0 = r0; k0 < r1; k0 += AT_K, cur ^= 1) {
    // (cur is 0, 1, 0, ...: both branches below are the same code on the two register sets)
    if (cur == 0) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        As[lr][lc + 16 * e] = static_cast<double>(ra[0][e]);
        Bs[lr][lc + 16 * e] = static_cast<double>(rb[0][e]);
      }
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        As[lr][lc + 16 * e] = static_cast<double>(ra[1][e]);
        Bs[lr][lc + 16 * e] = static_cast<double>(rb[1][e]);
      }
    }
    __syncthreads();
    if (cur == 0) fetch(k0 + 2 * AT_K, ra[0], rb[0]);
    else fetch(k0 + 2 * AT_K, ra[1], rb[1]);
#pragma unroll
    for (int kk = 0; kk < AT_K / 4; ++kk) {
      const double a0 = As[kk * 4 + q4][wa + gq], a1 = As[kk * 4 + q4][wa + 8 + gq];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const double bv = Bs[kk * 4 + q4][wb + c * 8 + gq];
        dmma_884(acc[0][c], a0, bv);
        dmma_884(acc[1][c], a1, bv);
      }
    }
    __syncthreads();
  }
  double* out = g.partial + static_cast<long long>(split) * g.m * g.n;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int gi = m0 + wa + h * 8 + gq;
    if (gi >= g.m) continue;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int gj = n0 + wb + c * 8 + 2 * q4 + i;
        if (gj < g.n && PRAC_IN(static_cast<long long>(gi) * g.n + gj, static_cast<long long>(g.m) * g.n))
          out[static_cast<long long>(gi) * g.n + gj] = acc[h][c][i];
      }
    }
  }
}

// out[i][j] = alpha * sum_s partial[s][i][j], slices added in order.  symmetric: entries
// below the diagonal are read from their mirror image (tiles below the diagonal were
// not computed).  TOut = float or double.
template <typename TOut>
__global__ void reduce_partials_kernel(const double* partial, int splits, int m, int n,
                                       int symmetric, double alpha, TOut* __restrict__ out, long long ldo,
                                       const int* run_if, int run_if_mask, int* zero_words, int zero_count) {
  grid_dep_wait();
  if (pass_is_off(run_if, run_if_mask)) return;
  // state that the next kernel on the stream expects zeroed (its grid-barrier counter)
  if (blockIdx.x == 0 && static_cast<int>(threadIdx.x) < zero_count) zero_words[threadIdx.x] = 0;
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= static_cast<long long>(m) * n) return;
  const int i = static_cast<int>(idx / n), j = static_cast<int>(idx % n);
  const long long src = (symmetric && i > j) ? static_cast<long long>(j) * n + i : static_cast<long long>(i) * n + j;
  // (eight loads in flight at a time: with many slices and few entries, as for the Rayleigh-Ritz
  // matrix, the kernel is a chain of loads otherwise; the slices are still added one by one, in order)
  const long long mn = static_cast<long long>(m) * n;
  double s = 0.0;
  int sp = 0;
  for (; sp + 8 <= splits; sp += 8) {
    double v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = partial[(sp + e) * mn + src];
#pragma unroll
    for (int e = 0; e < 8; ++e) s += v[e];
  }
  for (; sp < splits; ++sp) s += partial[sp * mn + src];
  if (PRAC_IN(static_cast<long long>(i) * ldo + j, static_cast<long long>(m - 1) * ldo + n))
    out[static_cast<long long>(i) * ldo + j] = static_cast<TOut>(alpha * s);
}

// ------------------------------------------------------------------ Cholesky + inverse, one launch
constexpr int CB = 32;       // block size of the factorisation
// Shared-memory pitch of a block, in doubles: 36 = 8 banks (mod 32) per row, so that the rows a
// tensor-core fragment load touches (four rows of eight consecutive doubles, or eight rows of four)
// fall into two wavefronts, the least a 64-bit load of a warp can take.  (33, the pitch that keeps a
// walk down a column free of conflicts, made those loads four-way conflicts: 168 -> 154 us per launch
// at 320 columns.)
constexpr int CP = CB + 4;
constexpr int CHOL_SMEM = 12 * CB * CP * 8;  // six staging blocks for each group of a worker (the chain's CTA uses eight)
// What a launch asks for: more than half of an SM's shared memory, so that no two CTAs of this
// kernel (of this or of another factorisation running beside it) land on one SM.  The kernel is a
// chain of dependent steps that issues instructions most of the time: two of its CTAs on one SM
// take nearly twice as long, and every barrier waits for the slowest.
constexpr int CHOL_SMEM_ASK = 116 * 1024;
static_assert(CHOL_SMEM_ASK >= CHOL_SMEM && 2 * CHOL_SMEM_ASK > 227 * 1024, "one CTA per SM");

// How the CTAs of a factorisation meet: diagonal blocks published, (worker, step) pairs done, blocks that
// the chain needs next brought up to date (two per step).
struct CholSync { unsigned chain, work, next; int abort; };

struct CholArgs {
  double* G;        // n x n, symmetric on entry; its trailing blocks are updated in place
  double* R;        // n x n: the off-diagonal blocks of the upper factor (row j, columns right of j)
  double* Dinv;     // [nb][CB][CB]: inverses of the diagonal blocks of R
  double* X;        // n x n scratch: R^-1 in double
  double* diag0;    // n: the diagonal of G on entry
  float* Rinv;      // n x n output: R^-1 (upper triangular, zeros below); or, where Rt3 is given,
  __nv_bfloat16* Rt3;  // n x 3 kp: row j = column j of R^-1 as three bf16 pieces side by side, zeros past j
  int kp;
  long long ldr;
  int n, nb;
  int* dev_status;
  int flag_bit;
  CholSync* sync;          // zeroed before the launch
  unsigned poll_limit;
  int run_if_mask;         // != 0: the kernel does nothing unless *dev_status has one of these bits
};

// Element (i, j) of the n x n matrix padded to nb*CB with the identity.
__device__ __forceinline__ double ld_pad(const double* M, int n, int i, int j) {
  return (i < n && j < n) ? __ldcg(&M[static_cast<long long>(i) * n + j]) : (i == j ? 1.0 : 0.0);
}

// A group of 256 threads works on blocks together (a CTA has one or two such groups).
__device__ __forceinline__ int group_tid() { return threadIdx.x & 255; }

// C (CB x CB, shared) = products of two CB x CB blocks, all 256 threads of a group: warp w owns the 8-row
// band w / 2 and the two 8-column tiles 2 (w % 2), 2 (w % 2) + 1 of C.
//   MODE 0:  C  = A^T * B
//   MODE 1:  C -= A^T * B
//   MODE 2:  C  = A * B
//   MODE 3:  C -= A * B
__device__ __forceinline__ void blk_mm(double (*C)[CP], const double (*A)[CP], const double (*B)[CP], int mode) {
  const int warp = group_tid() >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, q = lane & 3;
  const int row0 = (warp >> 1) * 8, col0 = (warp & 1) * 16;
  double acc0[2] = {0.0, 0.0}, acc1[2] = {0.0, 0.0};
#pragma unroll
  for (int ks = 0; ks < CB / 4; ++ks) {
    const double a = (mode >= 2) ? A[row0 + g][ks * 4 + q] : A[ks * 4 + q][row0 + g];
    const double b0 = B[ks * 4 + q][col0 + g];
    const double b1 = B[ks * 4 + q][col0 + 8 + g];
    dmma_884(acc0, a, b0);
    dmma_884(acc1, a, b1);
  }
  double* c0 = &C[row0 + g][col0 + 2 * q];
  double* c1 = &C[row0 + g][col0 + 8 + 2 * q];
  if (mode == 1 || mode == 3) {
    c0[0] -= acc0[0]; c0[1] -= acc0[1]; c1[0] -= acc1[0]; c1[1] -= acc1[1];
  } else {
    c0[0] = acc0[0]; c0[1] = acc0[1]; c1[0] = acc1[0]; c1[1] = acc1[1];
  }
}

__device__ __forceinline__ void blk_load(double (*S)[CP], const double* M, int n, int bi, int bj) {
  for (int idx = group_tid(); idx < CB * CB; idx += 256) {
    const int i = idx / CB, j = idx % CB;
    S[i][j] = ld_pad(M, n, bi * CB + i, bj * CB + j);
  }
}
__device__ __forceinline__ void blk_store(const double (*S)[CP], double* M, int n, int bi, int bj) {
  for (int idx = group_tid(); idx < CB * CB; idx += 256) {
    const int i = bi * CB + idx / CB, j = bj * CB + idx % CB;
    if (i < n && j < n) M[static_cast<long long>(i) * n + j] = S[idx / CB][idx % CB];
  }
}

// The 8 x 8 diagonal sub-block of a diagonal block, by one warp in registers: lane (r, c) holds
// M[r][2c], M[r][2c + 1] (the accumulator layout of dmma_884).  Elimination without square roots and
// without a division: on return row r of the triangular matrix T = S L^-1, M = L diag(pv) L^T, S a diagonal
// matrix of positive scales, is in the strictly lower part of M and S_r in `scale`; `pivot` is S_r pv_r, so that
// M = T^-1 diag(pivot * scale) T^-T.  (An identity kept in the lower triangle is eliminated along
// with M.)  Only the upper triangle is read.  A pivot that is not safely positive relative to the column's
// original squared norm is replaced by a guard value.
//
// This is the careful form, one column at a time with S = 1, for sub-blocks in which a pivot is bad.
__device__ __noinline__ void sub_chol_guarded(double& m0, double& m1, const double* guard, double& scale, double& pivot,
                                              int* dev_status, int flag_bit) {
  const int lane = threadIdx.x & 31, r = lane >> 2, c = lane & 3;
  scale = 1.0;
#pragma unroll 1
  for (int j = 0; j < 8; ++j) {
    const int row = j << 2;
    double pv = __shfl_sync(0xffffffffu, (j & 1) ? m1 : m0, row | (j >> 1));
    const double rj0 = __shfl_sync(0xffffffffu, m0, row | c), rj1 = __shfl_sync(0xffffffffu, m1, row | c);
    const double t0 = __shfl_sync(0xffffffffu, m0, row | (r >> 1)), t1 = __shfl_sync(0xffffffffu, m1, row | (r >> 1));
    if (!(pv > guard[j])) {                                      // warp-uniform
      pv = guard[j];
      if (lane == 0 && flag_bit && dev_status) atomicOr(dev_status, flag_bit);
    }
    if (r == j) pivot = pv;
    const double m = ((r & 1) ? t1 : t0) / pv;                   // M[j][r] / pv
    const double u0 = fma(-m, rj0, m0), u1 = fma(-m, rj1, m1);
    // U part, and L^-1 columns before j: updated; L^-1 column j starts here; the rest waits
    const int l0 = 2 * c, l1 = 2 * c + 1;
    const double n0 = (l0 >= r || l0 < j) ? u0 : ((l0 == j) ? -m : m0);
    const double n1 = (l1 >= r || l1 < j) ? u1 : ((l1 == j) ? -m : m1);
    m0 = r > j ? n0 : m0;
    m1 = r > j ? n1 : m1;
  }
}

// The same with neither a division nor a test in the dependent chain.  Column j turns every later row r into
// (pv_j M[r] - M[j][r] M[j]) 2^-e, e the exponent of the new scale: rows keep a common scale S in [1, 2) instead
// of being divided by the pivot, and a column is a shuffle and three operations (with a reciprocal
// approximation and its refinement in the chain it took 165 cycles).  Returns whether all pivots were good; where
// not, the caller repeats the sub-block in the careful form.
__device__ __forceinline__ bool sub_chol(double& m0, double& m1, const double* guard, double& scale, double& pivot) {
  const int lane = threadIdx.x & 31, r = lane >> 2, c = lane & 3;
  const int l0 = 2 * c, l1 = 2 * c + 1;
  bool good = true;
  double S = 1.0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int row = j << 2;
    const double pv = __shfl_sync(0xffffffffu, (j & 1) ? m1 : m0, row | (j >> 1));
    good = good && pv > guard[j] * S;                            // (false for NaN)
    if (r == j) { scale = S; pivot = pv; }
    if (j == 7) break;
    const double rj0 = __shfl_sync(0xffffffffu, m0, row | c), rj1 = __shfl_sync(0xffffffffu, m1, row | c);
    const double t0 = __shfl_sync(0xffffffffu, m0, row | (r >> 1)), t1 = __shfl_sync(0xffffffffu, m1, row | (r >> 1));
    const double t = (r & 1) ? t1 : t0;                          // M[j][r]
    const double Sp = S * pv;
    // 2^-e with e the exponent of Sp (a good pivot is a positive normal number)
    const double two = __hiloint2double(0x7fe00000 - (__double2hiint(Sp) & 0x7ff00000), 0);
    const double u0 = fma(pv, m0, -(t * rj0)) * two, u1 = fma(pv, m1, -(t * rj1)) * two;
    const double start = -(t * S) * two;                         // column j of T begins (its diagonal entry is S)
    S = Sp * two;
    const double n0 = (l0 >= r || l0 < j) ? u0 : ((l0 == j) ? start : m0);
    const double n1 = (l1 >= r || l1 < j) ? u1 : ((l1 == j) ? start : m1);
    m0 = r > j ? n0 : m0;
    m1 = r > j ? n1 : m1;
  }
  return good;
}

// 1 / x for a positive normal x: 1 / x = x0 (1 + e + e^2 + ..), e = 1 - x x0; the hardware's x0 is good to 20 bits, so the
// terms up to e^2 leave a relative error below 2^-60.
__device__ __forceinline__ double rcp_f64(double x) {
  double x0;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x0) : "d"(x));
  const double e = fma(-x, x0, 1.0);
  return fma(x0, fma(e, e, e), x0);
}

// The 256 threads that compute (the chain's CTA has more, see chol_inv_kernel).
constexpr int CHOL_MAIN = 256, CHOL_HELP = 256;
// (a warp has to be converged at these barriers)
__device__ __forceinline__ void bar_sync(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void main_sync() { bar_sync(1, CHOL_MAIN); }

// What a diagonal block's factorisation leaves in shared memory beside the block: limits below which a pivot is
// replaced, scaled pivots, their inverse square roots.
struct CholDiag { double guard[CB], pi[CB], rs[CB]; };
__device__ __forceinline__ double pivot_guard(double diagonal_on_entry) {
  return diagonal_on_entry > 0.0 ? 1e-13 * diagonal_on_entry : 1.0;
}

// In shared memory: D (CB x CB, symmetric positive definite on entry, upper triangle used) -> I = R^-1
// (upper), where R^T R = D, by the 256 main threads, which have met at a barrier since D and x.guard were written.  The
// chain of 32 dependent column steps is what this costs, so
// it runs in one warp's registers, eight columns at a time (one block barrier per column over all
// 256 threads took 330 cycles each); the other 8 x 8 tiles are brought up to date on the fp64 tensor
// cores by the other warps, one tile each, beside the next sub-block's chain.  With T = S L_ss^-1 of sub-block s (sub_chol),
// pi = pivot * scale, U_q = T D_sq, V_q = diag(1/pi) U_q:
// D_pq -= V_p^T U_q, and the same elimination applied to an identity (E) gives the block rows of S L^-1:
// Lin_sc = T E_sc (E_ss = 1), E_pc -= V_p^T Lin_sc.  R^-1 = (S L^-1)^T diag(1/sqrt(pi)).
// W: scratch, rows 0..7 U, 8..15 V (columns 8 q ..), 16..23 T, two in turn.  emit(r, c, v0, v1): elements (r, c), (r, c + 1) of
// R^-1, which are written to I too.
template <typename Emit>
__device__ __forceinline__ void blk_chol_inv(double (*D)[CP], double (*I)[CP], double (*Lin)[CP], double (*E)[CP], double (*W)[CP],
                                             CholDiag& x, int* dev_status, int flag_bit, Emit emit) {
  static_assert(CB == 32, "four sub-blocks of eight columns");
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, g = lane >> 2, q4 = lane & 3;
  double (*U)[CP] = W; double (*V)[CP] = W + 8; double (*T)[CP] = W + 16;
  double m0 = 0.0, m1 = 0.0;
  if (warp == 0) { m0 = D[g][2 * q4]; m1 = D[g][2 * q4 + 1]; }
#pragma unroll 1
  for (int s = 0; s < CB / 8; ++s) {
    const int o = 8 * s;
    const int tc = 8 * (s & 1);                    // T of this sub-block: W[16 ..][tc ..]
    double t0 = 0.0, t1 = 0.0, pi = 1.0;
    if (warp == 0) {
      const double k0 = m0, k1 = m1;
      double scale = 1.0, pivot = 1.0;
      if (!sub_chol(m0, m1, x.guard + o, scale, pivot)) {     // (the lanes agree)
        m0 = k0; m1 = k1;
        sub_chol_guarded(m0, m1, x.guard + o, scale, pivot, dev_status, flag_bit);
      }
      t0 = 2 * q4 < g ? m0 : (2 * q4 == g ? scale : 0.0);
      t1 = 2 * q4 + 1 < g ? m1 : (2 * q4 + 1 == g ? scale : 0.0);
      pi = pivot * scale;
      T[g][tc + 2 * q4] = t0; T[g][tc + 2 * q4 + 1] = t1;
      Lin[o + g][o + 2 * q4] = t0; Lin[o + g][o + 2 * q4 + 1] = t1;
      if (q4 == 0) x.pi[o + g] = pi;
    }
    main_sync();
    if (warp == 0) {
      // the next diagonal sub-block, on its own and in registers (the others make U and V of block column s + 1
      // again): a fragment of A may name its columns in any order that B's rows follow, so T goes in as it lies;
      // U comes back with its rows over the lanes and is turned by shuffles
      if (s + 1 < CB / 8) {
        const int p = o + 8;
        double acc[2] = {0.0, 0.0};
        dmma_884(acc, t0, D[o + 2 * q4][p + g]);
        dmma_884(acc, t1, D[o + 2 * q4 + 1][p + g]);
        const double xi = rcp_f64(pi);
        double upd[2] = {0.0, 0.0};
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
          const int from = ((4 * kk + q4) << 2) | (g >> 1);
          const double u0 = __shfl_sync(0xffffffffu, acc[0], from), u1 = __shfl_sync(0xffffffffu, acc[1], from);
          const double u = (g & 1) ? u1 : u0;      // U[4 kk + q4][g]
          dmma_884(upd, u * __shfl_sync(0xffffffffu, xi, (4 * kk + q4) << 2), u);
        }
        m0 = D[p + g][p + 2 * q4] - upd[0];
        m1 = D[p + g][p + 2 * q4 + 1] - upd[1];
      }
    } else {
      if (warp == 7 && lane < 8) x.rs[o + lane] = rsqrt(x.pi[o + lane]);
      // three tiles: U_q, q > s, and Lin_sc, c < s
      if (warp < 4) {
        const int q = warp - 1 < s ? warp - 1 : warp;
        double (*B)[CP] = q < s ? E : D;
        double acc[2] = {0.0, 0.0};
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) dmma_884(acc, T[g][tc + 4 * kk + q4], B[o + 4 * kk + q4][8 * q + g]);
        if (q < s) {
          Lin[o + g][8 * q + 2 * q4] = acc[0]; Lin[o + g][8 * q + 2 * q4 + 1] = acc[1];
        } else {
          const double xi = rcp_f64(x.pi[o + g]);
          U[g][8 * q + 2 * q4] = acc[0]; U[g][8 * q + 2 * q4 + 1] = acc[1];
          V[g][8 * q + 2 * q4] = xi * acc[0]; V[g][8 * q + 2 * q4 + 1] = xi * acc[1];
        }
      }
      bar_sync(8, CHOL_MAIN - 32);
      // trailing tiles D_pq (s < p <= q, without the one warp 0 has) and E_pc (c <= s < p), in one list
      const int rest = CB / 8 - 1 - s, nd = rest * (rest + 1) / 2 - 1, ne = rest * (s + 1);
      for (int u = warp - 1; u < nd + ne; u += 7) {
        double acc[2] = {0.0, 0.0};
        int p, q;
        if (u < nd) {                              // tile u + 1 of the upper triangle, by rows (tile 0 is warp 0's)
          int left = u + 1;
          p = s + 1;
          while (left >= CB / 8 - p) { left -= CB / 8 - p; ++p; }
          q = p + left;
        } else {
          p = s + 1 + (u - nd) / (s + 1);
          q = (u - nd) % (s + 1);
        }
        double (*B)[CP] = u < nd ? U : Lin + o;
        double (*C)[CP] = u < nd ? D : E;
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) dmma_884(acc, V[4 * kk + q4][8 * p + g], B[4 * kk + q4][8 * q + g]);
        double* o0 = &C[8 * p + g][8 * q + 2 * q4];
        const bool fresh = u >= nd && q == s;      // (E_ps starts from zero)
        o0[0] = (fresh ? 0.0 : o0[0]) - acc[0];
        o0[1] = (fresh ? 0.0 : o0[1]) - acc[1];
      }
    }
  }
  main_sync();
#pragma unroll
  for (int e = 0; e < CB * CB / 2 / CHOL_MAIN; ++e) {
    const int r = (t + CHOL_MAIN * e) / (CB / 2), c = 2 * (t % (CB / 2));
    const double v0 = r <= c ? Lin[c][r] * x.rs[c] : 0.0, v1 = r <= c + 1 ? Lin[c + 1][r] * x.rs[c + 1] : 0.0;
    *reinterpret_cast<double2*>(&I[r][c]) = make_double2(v0, v1);
    emit(r, c, v0, v1);
  }
}

// Up to three blocks fetched in one round trip: all of a thread's loads are issued before the first store.
__device__ __forceinline__ void blk_load3(double (*A)[CP], const double* MA, int ai, int aj, double (*B)[CP], const double* MB,
                                          int bi, int bj, double (*C)[CP], const double* MC, int ci, int cj, int n) {
  double v[3][CB * CB / 256];
#pragma unroll
  for (int e = 0; e < CB * CB / 256; ++e) {
    const int i = (group_tid() + 256 * e) / CB, j = group_tid() % CB;
    v[0][e] = A ? ld_pad(MA, n, ai * CB + i, aj * CB + j) : 0.0;
    v[1][e] = B ? ld_pad(MB, n, bi * CB + i, bj * CB + j) : 0.0;
    v[2][e] = C ? ld_pad(MC, n, ci * CB + i, cj * CB + j) : 0.0;
  }
#pragma unroll
  for (int e = 0; e < CB * CB / 256; ++e) {
    const int i = (group_tid() + 256 * e) / CB, j = group_tid() % CB;
    if (A) A[i][j] = v[0][e];
    if (B) B[i][j] = v[1][e];
    if (C) C[i][j] = v[2][e];
  }
}

// Block (p, q), p <= q, of the result R^-1, from shared memory into the outputs (see CholArgs): the fp32
// matrix, or the transposed matrix as three bf16 pieces.
__device__ __forceinline__ void chol_emit(const CholArgs& a, const double (*S)[CP], int p, int q) {
  for (int idx = group_tid(); idx < CB * CB; idx += 256) {
    if (!a.Rt3) {
      const int i = p * CB + idx / CB, j = q * CB + idx % CB;
      if (i < a.n && j < a.n) a.Rinv[static_cast<long long>(i) * a.ldr + j] = static_cast<float>(S[idx / CB][idx % CB]);
    } else {
      const int j = q * CB + idx / CB, l = p * CB + idx % CB;
      if (j < a.n && l < a.kp) {
        float x = l < a.n ? static_cast<float>(S[idx % CB][idx / CB]) : 0.f;
        __nv_bfloat16* o = a.Rt3 + static_cast<long long>(j) * 3 * a.kp + l;
        const __nv_bfloat16 hi = __float2bfloat16_rn(x);
        x -= __bfloat162float(hi);
        const __nv_bfloat16 mid = __float2bfloat16_rn(x);
        x -= __bfloat162float(mid);
        o[0] = hi; o[a.kp] = mid; o[2 * a.kp] = __float2bfloat16_rn(x);
      }
    }
  }
}
// What lies below the diagonal blocks of R^-1 (and the padding of the transposed pieces) is zero.
__device__ __forceinline__ void chol_emit_zeros(const CholArgs& a, int worker, int workers) {
  for (int row = worker; row < a.n; row += workers) {
    const int from = (row / CB) * CB;              // first row or column of the diagonal block of this row
    if (!a.Rt3) {
      for (int j = group_tid(); j < from; j += 256) a.Rinv[static_cast<long long>(row) * a.ldr + j] = 0.f;
    } else {
      __nv_bfloat16* o = a.Rt3 + static_cast<long long>(row) * 3 * a.kp;
      for (int l = from + CB + group_tid(); l < a.kp; l += 256) {
        o[l] = o[a.kp + l] = o[2 * a.kp + l] = __float2bfloat16_rn(0.f);
      }
    }
  }
}

// Waits until *word >= target (words only grow).  Bounded: after poll_limit polls, or when another
// waiter has given up, the wait ends with false.  One thread.
__device__ __forceinline__ bool chol_wait(CholSync* sy, const unsigned* word, unsigned target, unsigned poll_limit) {
  // (plain volatile polls and one fence at the end: an acquiring load per poll disturbs the SM's other warps)
  unsigned polls = 0;
  while (*reinterpret_cast<const volatile unsigned*>(word) < target) {
    if (++polls >= poll_limit) { atomicExch(&sy->abort, 1); return false; }
    if ((polls & 63u) == 0u && *reinterpret_cast<volatile int*>(&sy->abort)) return false;
  }
  __threadfence();
  return true;
}

// R = chol(G) and R^-1, blocks of 32, right-looking.  CTA 0 walks the chain of diagonal blocks and nothing
// else: it brings block (j, j) up to date with row j - 1, factors it and publishes R_jj^-1 (sync->chain = j + 1);
// the other CTAs (the workers) then do the rest of step j, the trailing blocks
// G_pq -= R_jp^T R_jq and the products of the inverse, and count themselves in sync->work (and the two blocks
// that the chain needs next in sync->next).  While the
// chain is at block j the workers are at step j - 1.  What the chain needs of their results (blocks
// (j, j + 1) and (j + 1, j + 1), up to date with step j - 1) eight helper warps of CTA 0 wait for and fetch
// while block j is being factored, and they publish it, so that the chain itself is two products and a
// factorisation per block and never waits for global memory.  320 columns: 132 us when every CTA factored
// the diagonal block itself and then did its blocks between grid barriers, 103 us with a grid barrier per
// block and CTA 0 on the chain, 76 us now.
//
// Every wait on another CTA is bounded; a CTA that gives up (or sees that another did) reports it and
// leaves; nothing asynchronous is in flight here, so the early exit is clean.
__global__ void __launch_bounds__(CHOL_MAIN + CHOL_HELP) chol_inv_kernel(const CholArgs a) {
  if (a.run_if_mask && pass_is_off(a.dev_status, a.run_if_mask)) return;
  extern __shared__ __align__(16) double chol_smem[];
  __shared__ int ok_sh[2];
  __shared__ CholDiag diag;
  double (*S0)[CP] = reinterpret_cast<double (*)[CP]>(chol_smem);
  double (*S1)[CP] = S0 + CB;
  double (*S2)[CP] = S1 + CB;
  double (*S3)[CP] = S2 + CB;
  double (*S4)[CP] = S3 + CB;
  double (*S5)[CP] = S4 + CB;
  const int n = a.n, nb = a.nb;
  const unsigned workers = 2 * (gridDim.x - 1);      // groups of 256 threads
  CholSync* const sy = a.sync;

  if (blockIdx.x == 0) {
    // barriers between the main threads and the helpers: 2 and 6 in turn = a block's inverse is stored
    // (the main threads may arrive for the next block before the helpers have left this one's barrier),
    // 3 = the next two blocks are fetched, 4 = their buffers may be filled
    double (*F0)[CP] = S5 + CB;                    // G_j,j+1
    double (*FD)[CP] = F0 + CB;                    // G_j+1,j+1: takes turns with S0 as the block being factored
    if (threadIdx.x >= CHOL_MAIN) {
      const int t = threadIdx.x - CHOL_MAIN;
      for (int j = 0; j < nb; ++j) {
        if (j + 1 < nb) {
          bar_sync(4, CHOL_MAIN + CHOL_HELP);
          if (t == 0) ok_sh[0] = chol_wait(sy, &sy->next, 2u * static_cast<unsigned>(j), a.poll_limit) ? 1 : 0;
          bar_sync(5, CHOL_HELP);
          const bool ok = ok_sh[0] != 0;
          if (ok) {
            double (*D)[CP] = (j & 1) ? S0 : FD;   // (block j itself is in the other one)
            double v[2][CB * CB / CHOL_HELP];
#pragma unroll
            for (int e = 0; e < CB * CB / CHOL_HELP; ++e) {
              const int i = (t + CHOL_HELP * e) / CB, c = t % CB;
              v[0][e] = ld_pad(a.G, n, j * CB + i, (j + 1) * CB + c);
              v[1][e] = ld_pad(a.G, n, (j + 1) * CB + i, (j + 1) * CB + c);
            }
#pragma unroll
            for (int e = 0; e < CB * CB / CHOL_HELP; ++e) {
              const int i = (t + CHOL_HELP * e) / CB, c = t % CB;
              F0[i][c] = v[0][e];
              D[i][c] = v[1][e];
            }
          }
          bar_arrive(3, CHOL_MAIN + CHOL_HELP);
          if (!ok) return;
        }
        bar_sync(2 + 4 * (j & 1), CHOL_MAIN + CHOL_HELP);
        if (t == 0) {
          __threadfence();
          atomicExch(&sy->chain, static_cast<unsigned>(j + 1));
        }
        __syncwarp();
      }
      return;
    }
    // the diagonal on entry (read by this CTA only, before any block is updated)
    for (int i = threadIdx.x; i < n; i += CHOL_MAIN) a.diag0[i] = __ldcg(&a.G[static_cast<long long>(i) * n + i]);
    blk_load(S0, a.G, n, 0, 0);
    main_sync();
    for (int j = 0; j < nb; ++j) {
      double (*D)[CP] = (j & 1) ? FD : S0;
      if (j > 0) {
        bar_sync(3, CHOL_MAIN + CHOL_HELP);
        if (!ok_sh[0]) {
          if (threadIdx.x == 0 && a.dev_status) atomicOr(a.dev_status, DEV_WAIT_EXPIRED);
          return;
        }
        blk_mm(S4, S1, F0, 0);                     // R_j-1,j = R_j-1,j-1^-T G_j-1,j
        main_sync();
        blk_mm(D, S4, S4, 1);
        blk_store(S4, a.R, n, j - 1, j);
        main_sync();
      }
      if (j + 1 < nb) bar_arrive(4, CHOL_MAIN + CHOL_HELP);
      if (threadIdx.x < CB) {                      // (warp 0, which alone reads the limits)
        const int i = j * CB + threadIdx.x;
        diag.guard[threadIdx.x] = pivot_guard(i < n ? a.diag0[i] : 1.0);
        __syncwarp();
      }
      double* const inv = a.Dinv + static_cast<long long>(j) * CB * CB;
      blk_chol_inv(D, S1, S2, S3, S5, diag, a.dev_status, a.flag_bit,
                   [&](int r, int c, double v0, double v1) { *reinterpret_cast<double2*>(&inv[r * CB + c]) = make_double2(v0, v1); });
      main_sync();
      bar_arrive(2 + 4 * (j & 1), CHOL_MAIN + CHOL_HELP);
    }
    return;
  }

  // ---- workers: two groups of 256 threads per CTA, each with its own blocks
  const int group = threadIdx.x / CHOL_MAIN, t = group_tid(), bar = 1 + 6 * group;
  S0 += group * 6 * CB; S1 += group * 6 * CB; S2 += group * 6 * CB; S3 += group * 6 * CB; S4 += group * 6 * CB; S5 += group * 6 * CB;
  const int worker = static_cast<int>(blockIdx.x) - 1 + group * (static_cast<int>(gridDim.x) - 1);   // (one group per SM first)
  auto sync = [&]() { bar_sync(bar, CHOL_MAIN); };
  auto wait = [&](const unsigned* word, unsigned target) {
    if (t == 0) ok_sh[group] = chol_wait(sy, word, target, a.poll_limit) ? 1 : 0;
    sync();
    const bool ok = ok_sh[group] != 0;
    sync();
    if (!ok && t == 0 && a.dev_status) atomicOr(a.dev_status, DEV_WAIT_EXPIRED);
    return ok;
  };
  chol_emit_zeros(a, worker, static_cast<int>(workers));
  for (int j = 0; j < nb; ++j) {
    // Trailing blocks (p, q), j < p <= q < nb, without (j + 1, j + 1), then the tasks of the inverse, dealt
    // round-robin.  A block's owner recomputes the two blocks of row j of R it needs:
    // R_jp = R_jj^-T G_jp,  R_jq = R_jj^-T G_jq,  then G_pq -= R_jp^T R_jq.  The owner of a diagonal block
    // also stores R_jp (into R, not over G_jp, which other workers are still reading).
    const int rem = nb - j - 1;
    const int ntile = rem > 0 ? rem * (rem + 1) / 2 - 1 : 0;
    const int width = nb - j, ntask = j * width;
    auto tile_of = [&](int item, int& p, int& q) {
      int row = 0, rest = item + 1;
      while (rest >= rem - row) { rest -= rem - row; ++row; }
      p = j + 1 + row; q = p + rest;
    };
    auto fetch_tile = [&](int p, int q) {
      blk_load3(S2, a.G, j, p, q != p ? S3 : nullptr, a.G, j, q, S5, a.G, p, q, n);
    };
    // every worker is done with step j - 1: this one's first blocks can be on their way while the chain is
    // still at block j
    if (!wait(&sy->work, workers * static_cast<unsigned>(j))) return;
    int p = 0, q = 0;
    if (worker < ntile) { tile_of(worker, p, q); fetch_tile(p, q); }
    // R_jj^-1 is published (with it row j - 1 of R is complete)
    if (!wait(&sy->chain, static_cast<unsigned>(j + 1))) return;
    for (int idx = t; idx < CB * CB; idx += CHOL_MAIN)
      S1[idx / CB][idx % CB] = __ldcg(&a.Dinv[static_cast<long long>(j) * CB * CB + idx]);
    for (int item = worker; item < ntile + ntask; item += static_cast<int>(workers)) {
      if (item < ntile) {
        if (item != worker) { sync(); tile_of(item, p, q); fetch_tile(p, q); }
        sync();
        blk_mm(S4, S1, S2, 0);                 // S4 = R_jj^-T G_jp = R_jp
        if (q != p) blk_mm(S0, S1, S3, 0);     // S0 = R_jq
        sync();
        blk_mm(S5, S4, (q != p) ? S0 : S4, 1); // G_pq -= R_jp^T R_jq
        sync();
        blk_store(S5, a.G, n, p, q);
        if (q == p) blk_store(S4, a.R, n, j, p);
        if (q == j + 2) {                      // (j + 1, j + 2) and (j + 2, j + 2): the chain is waiting for them
          sync();
          if (t == 0) { __threadfence(); atomicAdd(&sy->next, 1u); }
        }
      } else {
        // X = R^-1 grows with the factorisation: X_pq = -(sum_{p <= c < q} X_pc R_cq) R_qq^-1, X_pp = R_pp^-1.
        // Step j adds the c = j - 1 terms (X_p,j-1 and row j - 1 of R are finished) to the running sums kept
        // in the blocks (p, q), q >= j, of X, and closes block column j with R_jj^-1.  j (nb - j) tasks of
        // one product each.
        const int u = item - ntile, pu = u / width, qu = j + u % width;
        sync();
        if (pu == j - 1) {
          for (int idx = t; idx < CB * CB; idx += CHOL_MAIN) {
            S2[idx / CB][idx % CB] = __ldcg(&a.Dinv[static_cast<long long>(pu) * CB * CB + idx]);
            S0[idx / CB][idx % CB] = 0.0;
          }
          blk_load(S3, a.R, n, j - 1, qu);
        } else {
          blk_load3(S2, a.X, pu, j - 1, S0, a.X, pu, qu, S3, a.R, j - 1, qu, n);   // (S0: the running sum, negated)
        }
        sync();
        blk_mm(S0, S2, S3, 3);                 // S0 -= X_p,j-1 R_j-1,q
        sync();
        if (qu == j) {
          blk_mm(S4, S0, S1, 2);               // X_pj = S0 R_jj^-1
          sync();
          blk_store(S4, a.X, n, pu, j);
          chol_emit(a, S4, pu, j);
        } else {
          blk_store(S0, a.X, n, pu, qu);
        }
      }
    }
    sync();
    if (t == 0 && j + 1 < nb) {
      __threadfence();
      atomicAdd(&sy->work, 1u);
    }
    if (worker == static_cast<int>(workers) - 1) { chol_emit(a, S1, j, j); sync(); }
  }
}

// ------------------------------------------------------------------ the same on one cluster, up to 16 blocks of columns
// Shared memory of another CTA of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void* own, unsigned rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(own))), "r"(rank));
  return r;
}
__device__ __forceinline__ double2 cluster_ld(uint32_t addr) {
  double2 v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_st(uint32_t addr, double x, double y) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(addr), "d"(x), "d"(y) : "memory");
}
__device__ __forceinline__ void cluster_st_flag(uint32_t addr, int v) {
  asm volatile("st.release.cluster.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_flag(const int* own) {
  int v;
  asm volatile("ld.acquire.cluster.shared::cta.s32 %0, [%1];" : "=r"(v)
               : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(own))) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

constexpr int CC_MAX = 16;                       // blocks of columns = CTAs of the cluster
constexpr int CC_GROUPS = 2;                     // groups of 256 threads in a CTA
// What the CTAs tell one another; every word is written by one CTA and only grows.
struct ChainWords {
  int row_done[CC_MAX];      // [x]: blocks (c, x), c < row_done[x], of R are final in CTA x
  int inv_done[CC_MAX];      // [x]: 8 when the inverse of diagonal block x is final in CTA x (x before this one: stored here by CTA x's eight warps)
  int abort;                 // a wait gave up
};

// Column blocks of G and block rows of the inverse stay in shared memory for the whole factorisation: CTA q of
// the cluster holds the blocks (p, q), p <= q, of G, which become those of R, and row q of X = R^-1.  Step c, once R_cc^-1
// is known: the CTAs right of c form R_cq = R_cc^-T G_cq and subtract R_cp^T R_cq from their blocks (p, q), p > c; the others
// close X_qc = X_qc R_cc^-1 and subtract X_qc R_cx from their running sums X_qx, x > c.  The blocks R_cx of another CTA are
// fetched from its shared memory when its flag says that they are final; nothing is ever overwritten that another
// CTA may still want.  CTA c + 1, whose diagonal block the chain waits for, has nothing else to do in step c: R_cc^-1 is
// stored into its shared memory as it is formed, and two products later it factors.
//
// The chain of diagonal blocks is what this costs.  A factorisation whose CTAs met through flags in global memory
// (chol_inv_kernel) took 13 400 cycles a block, most of them the way of a block through L2 and back.
//
// Every wait on another CTA is bounded; a CTA that gives up tells the others, and all of them meet at the
// cluster's barrier before any leaves, so that nobody's shared memory goes away under a reader.
__global__ void __launch_bounds__(256 * CC_GROUPS, 1) chol_cluster_kernel(const CholArgs a) {
  grid_dep_wait();
  if (a.run_if_mask && pass_is_off(a.dev_status, a.run_if_mask)) return;
  extern __shared__ __align__(16) double chol_smem[];
  __shared__ CholDiag diag;
  __shared__ ChainWords words;
  typedef double (*Blk)[CP];
  const int n = a.n, nb = a.nb, q = static_cast<int>(blockIdx.x);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, group = tid >> 8, gt = tid & 255;
  const int g = lane >> 2, q4 = lane & 3;
  auto block = [&](int i) { return reinterpret_cast<Blk>(chol_smem + static_cast<size_t>(i) * CB * CP); };
  auto col = [&](int p) { return block(p); };                 // (p, q) of G, then of R
  auto inv = [&](int x) { return block(x + 1); };             // (q, x) of R^-1, x >= q
  Blk const Lin = block(nb + 1), E = block(nb + 2), W = block(nb + 3), Dprev = block(nb + 4), Dfar = block(nb + 5);
  Blk const stage = block(nb + 6 + group);
  bool fail = false;

  if (tid < static_cast<int>(sizeof(words) / sizeof(int))) reinterpret_cast<int*>(&words)[tid] = 0;
  __syncthreads();
  cluster_arrive();
  // this CTA's column of G, padded with the identity
  for (int idx = tid; idx < (q + 1) * CB * CB; idx += 256 * CC_GROUPS) {
    const int i = idx / CB, j = idx % CB;
    col(i / CB)[i % CB][j] = ld_pad(a.G, n, i, q * CB + j);
  }
  for (int idx = tid; idx < (nb - 1 - q) * CB * CP; idx += 256 * CC_GROUPS)      // the running sums
    inv(q + 1)[idx / CP][idx % CP] = 0.0;
  if (group == 1) chol_emit_zeros(a, q, nb);
  cluster_wait();
  __syncthreads();
  if (tid < CB) diag.guard[tid] = pivot_guard(col(q)[tid][tid]);
  __syncthreads();

  auto give_up = [&]() {
    fail = true;
    for (int x = 0; x < nb; ++x) cluster_st_flag(cluster_addr(&words.abort, x), 1);
  };
  // One lane of a warp polls a word of this CTA's shared memory; where it gives up the caller carries on with what it
  // has, until the CTA next meets and leaves together.
  auto wait_word = [&](const int* word, int target) {
    if (lane == 0 && !fail) {
      unsigned polls = 0;
      while (ld_flag(word) < target) {
        if (++polls >= a.poll_limit) { give_up(); break; }
        if ((polls & 63u) == 0u && ld_flag(&words.abort)) { fail = true; break; }
      }
    }
    __syncwarp();
  };
  // the pairs (row, 2 columns) of a block that a thread of a group moves
  auto pull = [&](uint32_t from, double2 (&v)[2]) {
#pragma unroll
    for (int e = 0; e < 2; ++e)
      v[e] = cluster_ld(from + (((gt + 256 * e) >> 4) * CP + 2 * (gt & 15)) * 8);
  };
  auto put = [&](Blk to, const double2 (&v)[2]) {
#pragma unroll
    for (int e = 0; e < 2; ++e) *reinterpret_cast<double2*>(&to[(gt + 256 * e) >> 4][2 * (gt & 15)]) = v[e];
  };

  for (int c = 0; c < nb; ++c) {
    if (c == q) {
      if (group == 0) {
        const bool next = q + 1 < nb;
        const uint32_t far = next ? cluster_addr(Dprev, q + 1) : 0u;
        blk_chol_inv(col(q), inv(q), Lin, E, W, diag, a.dev_status, a.flag_bit, [&](int r, int cc, double v0, double v1) {
          if (next) cluster_st(far + (r * CP + cc) * 8, v0, v1);
        });
        // (each warp says that its part is there: inv_done counts them)
        __syncwarp();
        if (next && lane == 0) {
          asm volatile("red.release.cluster.shared::cluster.add.u32 [%0], 1;" ::"r"(cluster_addr(&words.inv_done[q], q + 1)) : "memory");
        }
      }
      __syncthreads();
      // the CTA after this one counts the eight warps above, the others wait for this word
      if (warp == 8 && lane < nb && lane != q && lane != q + 1) cluster_st_flag(cluster_addr(&words.inv_done[q], lane), 8);
    } else {
      // ---- R_cc^-1, then this CTA's own block of step c
      Blk D = Dfar;
      wait_word(&words.inv_done[c], 8);
      if (c == q - 1) {
        D = Dprev;
      } else {
        const int r = tid >> 4, cc = 2 * (tid & 15);
        const double2 v = cluster_ld(cluster_addr(&block(c + 1)[r][cc], c));
        *reinterpret_cast<double2*>(&Dfar[r][cc]) = v;
        __syncthreads();
      }
      const int r0 = (warp >> 2) * 8, c0 = (warp & 3) * 8;    // a tile per warp
      double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
      Blk const mine = c < q ? col(c) : inv(c);
      // (R_cc^-1 is upper triangular: the products end where it does)
      const int ks_end = c < q ? 2 * (warp >> 2) + 2 : 2 * (warp & 3) + 2;
#pragma unroll
      for (int ks = 0; ks < CB / 4; ++ks) {
        if (ks >= ks_end) break;
        const double x = c < q ? D[ks * 4 + q4][r0 + g] : mine[r0 + g][ks * 4 + q4];
        const double y = c < q ? mine[ks * 4 + q4][c0 + g] : D[ks * 4 + q4][c0 + g];
        dmma_884(acc[ks & 1], x, y);
      }
      __syncthreads();
      *reinterpret_cast<double2*>(&mine[r0 + g][c0 + 2 * q4]) = make_double2(acc[0][0] + acc[1][0], acc[0][1] + acc[1][1]);
    }
    // every thread leaves here if one has given up
    if (__syncthreads_or(fail)) { fail = true; break; }

    if (c < q) {
      if (warp == 15 && lane < nb && lane != q) cluster_st_flag(cluster_addr(&words.row_done[q], lane), c + 1);
      Blk const R = col(c);
      if (c == q - 1) {
        // the diagonal block, at once: the upper 8 x 8 tiles, by the threads that factor it next
        if (group == 0) {
          for (int u = warp; u < 10; u += 8) {
            int p = 0, left = u;
            while (left >= 4 - p) { left -= 4 - p; ++p; }
            const int r0 = 8 * p, c0 = 8 * (p + left);
            double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
            for (int ks = 0; ks < CB / 4; ++ks) dmma_884(acc[ks & 1], R[ks * 4 + q4][r0 + g], R[ks * 4 + q4][c0 + g]);
            double2* o = reinterpret_cast<double2*>(&col(q)[r0 + g][c0 + 2 * q4]);
            const double2 old = *o;
            *o = make_double2(old.x - (acc[0][0] + acc[1][0]), old.y - (acc[0][1] + acc[1][1]));
          }
          main_sync();
        }
      } else {
        // blocks (p, q), c < p <= q, dealt to the groups, (q, q) first: it needs nobody else's block
        if (group == 0) blk_mm(col(q), R, R, 1);
        double2 v[2];
        int p = c + 1 + (1 - group);
        if (p < q) { wait_word(&words.row_done[p], c + 1); pull(cluster_addr(R, p), v); }
        for (; p < q; p += CC_GROUPS) {
          bar_sync(1 + group, 256);            // the block before this one is done with
          put(stage, v);
          bar_sync(1 + group, 256);
          if (p + CC_GROUPS < q) { wait_word(&words.row_done[p + CC_GROUPS], c + 1); pull(cluster_addr(R, p + CC_GROUPS), v); }
          blk_mm(col(p), stage, R, 1);
        }
      }
    } else {
      // row q of the inverse: X_qx -= X_qc R_cx, x > c
      Blk const X = inv(c);
      double2 v[2];
      int x = c + 1 + group;
      if (x < nb) { wait_word(&words.row_done[x], c + 1); pull(cluster_addr(block(c), x), v); }
      if (group == 1) chol_emit(a, X, q, c);
      for (; x < nb; x += CC_GROUPS) {
        bar_sync(1 + group, 256);
        put(stage, v);
        bar_sync(1 + group, 256);
        if (x + CC_GROUPS < nb) { wait_word(&words.row_done[x + CC_GROUPS], c + 1); pull(cluster_addr(block(c), x + CC_GROUPS), v); }
        blk_mm(inv(x), X, stage, 3);
      }
    }
    // (the next step reads what the other group has brought up to date; the diagonal block is group 0's own)
    if (c != q - 1) __syncthreads();
  }
  if (fail && lane == 0 && a.dev_status) atomicOr(a.dev_status, DEV_WAIT_EXPIRED);
  cluster_arrive();
  cluster_wait();
}

size_t chol_cluster_smem(int nb) {
  const size_t need = static_cast<size_t>(nb + 6 + CC_GROUPS) * CB * CP * 8;
  return need > static_cast<size_t>(CHOL_SMEM_ASK) ? need : static_cast<size_t>(CHOL_SMEM_ASK);
}

void chol_cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], int nb, cudaStream_t stream) {
  cfg = {};
  cfg.gridDim = dim3(nb);
  cfg.blockDim = dim3(256 * CC_GROUPS);
  cfg.dynamicSmemBytes = chol_cluster_smem(nb);
  cfg.stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = nb;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1] = dependent_launch_attr();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
}

// Whether the current device can place a cluster of nb CTAs of chol_cluster_kernel (asked once per device and size).
bool chol_cluster_fits(int nb) {
  if (nb < 1 || nb > CC_MAX) return false;
  static DeviceValue known[CC_MAX + 1];          // 1: no, 2: yes
  static DeviceOnce attrs;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return false; }
  const int v = known[nb].get(dev);
  if (v != 0) return v == 2;
  bool ok = true;
  if (!attrs.done(dev)) {
    ok = cudaFuncSetAttribute(chol_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(chol_cluster_smem(CC_MAX))) == cudaSuccess &&
         cudaFuncSetAttribute(chol_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    if (ok) attrs.mark(dev);
  }
  if (ok) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    chol_cluster_config(cfg, attr, nb, nullptr);
    int clusters = 0;
    ok = cudaOccupancyMaxActiveClusters(&clusters, chol_cluster_kernel, &cfg) == cudaSuccess && clusters >= 1;
  }
  if (!ok) (void)cudaGetLastError();
  known[nb].set(dev, ok ? 2 : 1);
  return ok;
}

cudaError_t chol_smem_attr() {
  static DeviceOnce done;      // the attribute belongs to the device that was current
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (done.done(dev)) return cudaSuccess;
  e = cudaFuncSetAttribute(chol_inv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, CHOL_SMEM_ASK);
  if (e == cudaSuccess) done.mark(dev);
  return e;
}

int pick_row_splits(int num_tiles, int64_t d) {
  tc_init();
  int sms = tc_num_sms();
  if (sms <= 0) sms = 148;
  int s = (2 * sms) / (num_tiles > 0 ? num_tiles : 1);
  const int64_t max_by_rows = d / 64 > 0 ? d / 64 : 1;
  if (s > max_by_rows) s = static_cast<int>(max_by_rows);
  if (s < 1) s = 1;
  if (s > 64) s = 64;
  return s;
}

}  // namespace

PRAC_BOUNDS_READER(bounds_violations_cholqr)

// ------------------------------------------------------------------ host side
namespace {
int atb_tiles(int64_t m, int64_t n, int symmetric) {
  const int tm = static_cast<int>((m + AT_T - 1) / AT_T), tn = static_cast<int>((n + AT_T - 1) / AT_T);
  return symmetric ? tn * (tn + 1) / 2 : tm * tn;
}
}  // namespace

size_t atb_ws_bytes(int64_t m, int64_t n, int64_t d, int symmetric) {
  if (m <= 0 || n <= 0 || d <= 0) return 0;
  return static_cast<size_t>(pick_row_splits(atb_tiles(m, n, symmetric), d)) * m * n * sizeof(double);
}

int atb_f64(const float* A, int64_t lda, const float* B, int64_t ldb, int64_t d, int64_t m, int64_t n,
            int symmetric, double alpha, void* out, int64_t ldo, int out_double, void* ws, size_t ws_bytes,
            cudaStream_t stream, const int* run_if, int run_if_mask, void* zero_after, int zero_bytes) {
  if (m <= 0 || n <= 0) return PRAC_OK;
  if (d <= 0 || (symmetric && (A != B || m != n))) return PRAC_EINVAL;
  AtbArgs g{};
  g.A = A; g.lda = lda; g.B = B; g.ldb = ldb;
  g.m = static_cast<int>(m); g.n = static_cast<int>(n); g.d = d;
  g.tiles_m = static_cast<int>((m + AT_T - 1) / AT_T);
  g.tiles_n = static_cast<int>((n + AT_T - 1) / AT_T);
  g.symmetric = symmetric;
  g.num_tiles = atb_tiles(m, n, symmetric);
  g.splits = pick_row_splits(g.num_tiles, d);
  const size_t need = static_cast<size_t>(g.splits) * m * n * sizeof(double);
  if (!ws || ws_bytes < need) return PRAC_EWORKSPACE;
  g.partial = static_cast<double*>(ws);
  g.run_if = run_if; g.run_if_mask = run_if_mask;
  PRAC_LAUNCH(atb_f64_partial_kernel, dim3(static_cast<unsigned>(g.num_tiles), static_cast<unsigned>(g.splits)), dim3(256), 0, stream, g);
  count_launch();
  if (out_double)
    PRAC_LAUNCH(reduce_partials_kernel<double>, dim3(nblocks(m * n, 256)), dim3(256), 0, stream,
                g.partial, g.splits, g.m, g.n, symmetric, alpha, static_cast<double*>(out), ldo, run_if, run_if_mask,
                static_cast<int*>(zero_after), zero_bytes / 4);
  else
    PRAC_LAUNCH(reduce_partials_kernel<float>, dim3(nblocks(m * n, 256)), dim3(256), 0, stream,
                g.partial, g.splits, g.m, g.n, symmetric, alpha, static_cast<float*>(out), ldo, run_if, run_if_mask,
                static_cast<int*>(zero_after), zero_bytes / 4);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

// Workspace of one Cholesky-QR pass on n columns (all 256-byte aligned):
//   G n*n double | R n*n double | X n*n double | Dinv nb*CB*CB double | diag0 n double | Rinv n*n float |
//   slices of the transposed product
namespace {
// Both operands as three bf16 pieces, side by side in rows of 3 kp: the segments of the chained
// product mid*mid, lo*hi, hi*lo, mid*hi, hi*mid, hi*hi: everything down to 2^-24 of the product, the
// small cross terms first so that they add up among themselves before the leading term arrives.
TcSegments six_cross_terms(int64_t kp) {
  TcSegments segs{};
  segs.n = 6;
  const int64_t pa[6] = {1, 2, 0, 1, 0, 0}, pb[6] = {1, 0, 2, 0, 1, 0};
  for (int q = 0; q < 6; ++q) { segs.off_a[q] = pa[q] * kp; segs.off_b[q] = pb[q] * kp; }
  segs.rows_a = 3 * kp;
  segs.rows_b = 3 * kp;
  return segs;
}

struct CholWs { double* G; double* R; double* X; double* Dinv; double* diag0; float* Rinv; void* part; size_t part_bytes; size_t bytes;
                __nv_bfloat16* V3; __nv_bfloat16* Rt3; int64_t kp; bool tensor; CholSync* sync; };
// V R^-1 runs on the tensor cores (operands as three bf16 pieces each, six cross terms: fp32
// accuracy) when the panel is big enough to fill their tiles.
inline bool vr_on_tensor_cores(int64_t n, int64_t d) { return d >= 256 && n >= 64; }
CholWs carve_chol(void* ws, int64_t n, int64_t d) {
  CholWs c;
  const int64_t nb = (n + CB - 1) / CB;
  size_t off = 0;
  auto take = [&](size_t b) { size_t o = off; off += (b + 255) / 256 * 256; return o; };
  const size_t oG = take(n * n * 8), oRR = take(n * n * 8), oX = take(n * n * 8), oD = take(nb * CB * CB * 8), o0 = take(n * 8);
  const size_t oR = take(n * n * 4);
  c.part_bytes = atb_ws_bytes(n, n, d, 1);
  const size_t oP = take(c.part_bytes);
  c.tensor = vr_on_tensor_cores(n, d);
  c.kp = (n + 63) / 64 * 64;
  const size_t oV3 = take(c.tensor ? static_cast<size_t>(d) * 3 * c.kp * 2 : 0);
  const size_t oR3 = take(c.tensor ? static_cast<size_t>(n) * 3 * c.kp * 2 : 0);
  const size_t oBar = take(sizeof(CholSync));
  char* b = static_cast<char*>(ws);
  c.sync = reinterpret_cast<CholSync*>(b + oBar);
  c.G = reinterpret_cast<double*>(b + oG); c.R = reinterpret_cast<double*>(b + oRR); c.X = reinterpret_cast<double*>(b + oX);
  c.Dinv = reinterpret_cast<double*>(b + oD); c.diag0 = reinterpret_cast<double*>(b + o0);
  c.Rinv = reinterpret_cast<float*>(b + oR); c.part = b + oP;
  c.V3 = reinterpret_cast<__nv_bfloat16*>(b + oV3); c.Rt3 = reinterpret_cast<__nv_bfloat16*>(b + oR3);
  c.bytes = off;
  return c;
}
}  // namespace

size_t cholqr_ws_bytes(int64_t n, int64_t d) { return n > 0 ? carve_chol(nullptr, n, d).bytes : 0; }

int cholqr_pass(const float* Vin, int64_t ldin, float* Vout, int64_t ldout, int64_t d, int64_t n, void* ws,
                size_t ws_bytes, int* dev_status, int flag_bit, cudaStream_t stream, int run_if_mask) {
  if (n <= 0) return PRAC_OK;
  if (d < n || Vin == Vout || n > 40000) return PRAC_EINVAL;   // (the kernel indexes n x n with 32 bits)
  if (run_if_mask && !dev_status) return PRAC_EINVAL;
  const CholWs c = carve_chol(ws, n, d);
  if (ws == nullptr || ws_bytes < c.bytes) return PRAC_EWORKSPACE;
  const int* run_if = run_if_mask ? dev_status : nullptr;
  // (the reduction kernel also zeroes the grid-barrier state of the factorisation that follows it)
  int st = atb_f64(Vin, ldin, Vin, ldin, d, n, n, 1, 1.0, c.G, n, 1, c.part, c.part_bytes, stream, run_if, run_if_mask,
                   c.sync, static_cast<int>(sizeof(CholSync)));
  if (st != PRAC_OK) return st;
  CholArgs a{};
  a.G = c.G; a.R = c.R; a.Dinv = c.Dinv; a.X = c.X; a.diag0 = c.diag0; a.Rinv = c.Rinv; a.ldr = n;
  a.n = static_cast<int>(n); a.nb = static_cast<int>((n + CB - 1) / CB);
  a.dev_status = dev_status; a.flag_bit = flag_bit;
  a.sync = c.sync; a.poll_limit = barrier_poll_limit(); a.run_if_mask = run_if_mask;
  // an optional pass (run_if_mask != 0) is rare and small: it takes the general product
  const bool tensor = run_if_mask == 0 && c.tensor && tc_init() == PRAC_OK && aligned16(Vout) && (ldout % 4) == 0;
  a.Rt3 = tensor ? c.Rt3 : nullptr;
  a.kp = static_cast<int>(c.kp);
  if (chol_cluster_fits(a.nb)) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    chol_cluster_config(cfg, attr, a.nb, stream);
    PRAC_CUDA_TRY(cudaLaunchKernelEx(&cfg, chol_cluster_kernel, a));
  } else {
    const int rem = a.nb - 1;
    // one group of 256 threads per task of the busiest step (trailing blocks plus the products of the
    // inverse), two groups per CTA
    int want = rem * (rem + 1) / 2;
    for (int j = 1; j < a.nb; ++j) {
      const int w = a.nb - j;
      const int tasks = (w - 1) * w / 2 + j * w;
      if (tasks > want) want = tasks;
    }
    int grid = (want < 1 ? 1 : (want + 1) / 2) + 1;    // at least one CTA of workers, and CTA 0, which walks the diagonal
    // ... and at most a quarter of the SMs, an SM each: a transformer block fits the bases of its four
    // distinct inputs side by side (four streams), and factorisations whose CTAs share SMs hold one
    // another up (their waits are as long as the slowest CTA)
    {
      const int sms = tc_num_sms();
      const int quarter = sms >= 8 ? sms / 4 : 2;
      if (grid > quarter) grid = quarter;
    }
    const int smem = CHOL_SMEM_ASK;
    void* args[] = {const_cast<CholArgs*>(&a)};
    PRAC_CUDA_TRY(chol_smem_attr());
    // cooperative launch: CTAs wait for one another, so all have to be resident
    PRAC_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(chol_inv_kernel), dim3(grid), dim3(CHOL_MAIN + CHOL_HELP), args,
                                              smem, stream));
  }
  count_launch();
  if (tensor) {
    st = launch_split3_cols(Vin, ldin, d, n, c.V3, c.kp, stream);
    if (st != PRAC_OK) return st;
    const TcSegments segs = six_cross_terms(c.kp);
    return tc_gemm_kmajor(c.V3, 3 * c.kp, c.Rt3, 3 * c.kp, d, n, c.kp, Vout, ldout, ET_F32, 0, dev_status, stream, &segs);
  }
  GemmArgs g{};
  g.M = d; g.N = n; g.K = n;
  g.A = Vin; g.lda = ldin; g.type_a = ET_F32; g.trans_a = 0;
  g.B = c.Rinv; g.ldb = n; g.type_b = ET_F32; g.trans_b = 0;
  g.C = Vout; g.ldc = ldout; g.type_c = ET_F32;
  g.alpha = 1.0; g.beta = 0.0; g.symmetric = 0; g.kscale_from = -1; g.kscale = 1.0;
  g.run_if = run_if; g.run_if_mask = run_if_mask;
  return gemm_general(g, stream);
}

namespace {
__global__ void copy2d_if_kernel(const float* src, long long lds, float* __restrict__ dst, long long ldd,
                                 long long rows, long long cols, const int* status, int run_if_mask) {
  grid_dep_wait();
  grid_dep_launch();
  if (pass_is_off(status, run_if_mask)) return;
  // a small fixed grid striding over the matrix: the launch is almost always a no-op and should cost one
  for (long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; idx < rows * cols;
       idx += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long i = idx / cols, j = idx % cols;
    if (!PRAC_IN(i * lds + j, (rows - 1) * lds + cols) || !PRAC_IN(i * ldd + j, (rows - 1) * ldd + cols)) continue;
    dst[i * ldd + j] = src[i * lds + j];
  }
}
// Runs alone after every kernel of the optional pass has read the word.
__global__ void clear_status_bits_kernel(int* status, int clear_bits) {
  grid_dep_wait();
  grid_dep_launch();
  atomicAnd(status, ~clear_bits);
}
}  // namespace

int launch_copy2d_if(const float* src, int64_t lds, float* dst, int64_t ldd, int64_t rows, int64_t cols,
                     int* status, int run_if_mask, int clear_bits, cudaStream_t stream) {
  if (!status) return PRAC_EINVAL;
  if (rows > 0 && cols > 0) {
    const unsigned want = nblocks(rows * cols, 256);
    PRAC_LAUNCH(copy2d_if_kernel, dim3(want < 296u ? want : 296u), dim3(256), 0, stream,
                src, lds, dst, ldd, rows, cols, status, run_if_mask);
    count_launch();
  }
  PRAC_LAUNCH(clear_status_bits_kernel, dim3(1), dim3(1), 0, stream, status, clear_bits);
  count_launch();
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

// C (d x n, fp32) = [C +] scale * A (d x kd, fp32) * B (kd x n, fp32) to fp32 accuracy on the tensor
// cores: A row by row and B transposed are cut into three bf16 pieces each and the six leading
// cross terms are chained into one accumulator.  Panels too small for the tensor-core tiles take
// the general kernel.  Workspace: the pieces of A (d x 3 kp) and of B^T (n x 3 kp), kp = kd up to 64.
size_t panel_mm3_ws_bytes(int64_t d, int64_t kd, int64_t n) {
  const int64_t kp = (kd + 63) / 64 * 64;
  return (static_cast<size_t>(d) * 3 * kp * 2 + 255) / 256 * 256 + (static_cast<size_t>(n) * 3 * kp * 2 + 255) / 256 * 256;
}
int panel_mm3(const float* A, int64_t lda, const float* B, int64_t ldb, int64_t d, int64_t kd, int64_t n, float scale,
              float* C, int64_t ldc, int accumulate, void* ws, size_t ws_bytes, int* dev_status, cudaStream_t stream) {
  if (d <= 0 || kd <= 0 || n <= 0) return PRAC_OK;
  if (!(d >= 256 && n >= 64 && kd >= 64) || ws == nullptr || ws_bytes < panel_mm3_ws_bytes(d, kd, n)) {
    GemmArgs g{};
    g.M = d; g.N = n; g.K = kd;
    g.A = A; g.lda = lda; g.type_a = ET_F32; g.trans_a = 0;
    g.B = B; g.ldb = ldb; g.type_b = ET_F32; g.trans_b = 0;
    g.C = C; g.ldc = ldc; g.type_c = ET_F32;
    g.alpha = scale; g.beta = accumulate ? 1.0 : 0.0; g.symmetric = 0; g.kscale_from = -1; g.kscale = 1.0;
    return gemm_general(g, stream);
  }
  const int64_t kp = (kd + 63) / 64 * 64;
  __nv_bfloat16* A3 = static_cast<__nv_bfloat16*>(ws);
  __nv_bfloat16* Bt3 = reinterpret_cast<__nv_bfloat16*>(static_cast<char*>(ws) +
                                                        (static_cast<size_t>(d) * 3 * kp * 2 + 255) / 256 * 256);
  int st = launch_split3_cols(A, lda, d, kd, A3, kp, stream);
  if (st != PRAC_OK) return st;
  st = launch_split3_transposed(B, ldb, kd, n, scale, Bt3, kp, stream);
  if (st != PRAC_OK) return st;
  const TcSegments segs = six_cross_terms(kp);
  return tc_gemm_kmajor(A3, 3 * kp, Bt3, 3 * kp, d, n, kp, C, ldc, ET_F32, accumulate, dev_status, stream, &segs);
}

int cholqr_final(const float* Vin, int64_t ldin, float* Vout, int64_t ldout, float* tmp, int64_t d, int64_t n,
                 void* ws, size_t ws_bytes, int* dev_status, cudaStream_t stream) {
  if (n <= 0) return PRAC_OK;
  if (!dev_status || tmp == Vout || tmp == Vin) return PRAC_EINVAL;
  int st = cholqr_pass(Vin, ldin, Vout, ldout, d, n, ws, ws_bytes, dev_status, DEV_CHOL_RETRY, stream);
  if (st != PRAC_OK) return st;
  // A bad pivot means the panel was (numerically) rank deficient: the guarded column of Vout is
  // amplified rounding noise, a direction of its own but neither normalised nor orthogonal to
  // the rest.  One more pass orthonormalises it; only if that pass breaks down too is the
  // failure reported.
  st = cholqr_pass(Vout, ldout, tmp, n, d, n, ws, ws_bytes, dev_status, DEV_CHOL_PIVOT, stream, DEV_CHOL_RETRY);
  if (st != PRAC_OK) return st;
  return launch_copy2d_if(tmp, n, Vout, ldout, d, n, dev_status, DEV_CHOL_RETRY, DEV_CHOL_RETRY, stream);
}

}  // namespace prac
