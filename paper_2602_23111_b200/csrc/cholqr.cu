// Orthonormalisation of tall fp32 panels by Cholesky-QR, three launches per pass:
//   1. G = V^T V accumulated in double over slices of the rows that are summed in a fixed order (atb_f64_kernel);
//   2. R = chol(G) and R^-1 in one kernel, all in double: a cluster up to 512 columns (chol_cluster_kernel), a cooperative
//      launch above (chol_inv_kernel);
//   3. V_out = V_in * R^-1: on the tensor cores for panels big enough to fill their tiles (both
//      operands as three bf16 pieces, six chained cross terms: fp32 accuracy), else a general
//      fp32 GEMM.
// R has a positive diagonal, so V R^-1 is the unique thin-QR Q factor.  The same
// transposed-product kernel serves every small "tall^T x tall" product of the basis fit.
#include <cuda_runtime.h>

#include "internal.h"
#include "per_device.h"
#include "ptx.cuh"

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
  int tiles_n;
  int symmetric;                   // A == B, m == n: only tiles reaching the upper triangle, mirrored
  double alpha;
  void* out; long long ldo;
  int out_double;                  // out is double, else float
  const int* run_if;               // optional: the kernel does nothing unless *run_if & run_if_mask
  int run_if_mask;
  int* zero_words; int zero_count; // words that the next kernel on the stream expects zeroed
};

// Kernels of an optional pass are always launched and look at a device word to see whether
// they have anything to do (the host does not wait for the device to find out).
__device__ __forceinline__ bool pass_is_off(const int* run_if, int mask) {
  return run_if != nullptr && (*reinterpret_cast<const volatile int*>(run_if) & mask) == 0;
}

// A barrier for one event: an arrival, or, where bytes > 0, that many bytes stored by ptx::cluster_st_async.
__device__ __forceinline__ void cluster_bar_init(uint64_t* own, unsigned bytes) {
  ptx::mbar_init(own, 1);
  if (bytes) ptx::mbar_arrive_expect_tx(own, bytes);
}
__device__ __forceinline__ bool cluster_try_wait(uint64_t* own) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred P;\n\t"
      "mbarrier.try_wait.parity.relaxed.cluster.shared::cta.b64 P, [%1], 0;\n\t"
      "selp.b32 %0, 1, 0, P;\n\t}"
      : "=r"(ok) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(own))) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool cluster_try_wait_acquire(uint64_t* own) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred P;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 P, [%1], 0;\n\t"
      "selp.b32 %0, 1, 0, P;\n\t}"
      : "=r"(ok) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(own))) : "memory");
  return ok != 0;
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

// A 64 x 64 output tile by one cluster: each CTA takes a slice of the rows, 16 at a time, three chunks ahead of the
// products by asynchronous copies; warp w multiplies 16 columns
// of A (w / 2) by 32 columns of B (w % 2) on the fp64 tensor cores: six fragment loads, widened to double, for eight
// products.  Then every CTA adds up its rows of the
// slices' tiles from the others' shared memory, in the order of the slices, and writes them.  (Slices that went through
// global memory, 15 MB of them at 320 columns, took a second kernel of 8 us.)  The loops are short on purpose: most of these
// launches last a few microseconds, and an SM fetches instructions that it has not seen at 270 cycles per 128 bytes.
constexpr int AT_STAGES = 4;
constexpr int AT_P = AT_T + 8;      // pitch of a row in shared memory: what four rows of a fragment load read lies in 32 banks
__global__ void __launch_bounds__(256) atb_f64_kernel(const AtbArgs g) {
  grid_dep_wait();
  __shared__ __align__(16) double tile[AT_T * AT_P];        // the chunks in flight (fp32), then the slice's tile
  static_assert(AT_STAGES * 2 * AT_K * AT_P * sizeof(float) <= sizeof(tile), "the tile takes the place of the chunks");
  if (pass_is_off(g.run_if, g.run_if_mask)) return;
  float* const raw = reinterpret_cast<float*>(tile);
  int ti, tj;
  atb_tile(g, blockIdx.x, ti, tj);
  const int rank = blockIdx.y, slices = gridDim.y;          // (the cluster is 1 x slices)
  const int r0 = static_cast<int>(g.d * rank / slices), r1 = static_cast<int>(g.d * (rank + 1) / slices);
  const int t = threadIdx.x;
  const int warp = t >> 5, lane = t & 31, gq = lane >> 2, q4 = lane & 3;
  const int m0 = ti * AT_T, n0 = tj * AT_T;
  const int wa = (warp >> 1) * 16, wb = (warp & 1) * 32;   // this warp's columns of A and of B within the tile
  if (blockIdx.x == 0 && rank == 0)
    for (int i = t; i < g.zero_count; i += 256) g.zero_words[i] = 0;
  double acc[2][4][2];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < 4; ++c) { acc[h][c][0] = 0.0; acc[h][c][1] = 0.0; }
  // a thread copies column t % 64 of four rows of A's chunk and of B's (past the slice, or the matrix: zeros)
  const int lr = t >> 6, lc = t & 63;
  const bool in_a = m0 + lc < g.m, in_b = n0 + lc < g.n;
  const float* pa = g.A + static_cast<long long>(r0 + lr) * g.lda + (in_a ? m0 + lc : 0);
  const float* pb = g.B + static_cast<long long>(r0 + lr) * g.ldb + (in_b ? n0 + lc : 0);
  const uint32_t to = static_cast<uint32_t>(__cvta_generic_to_shared(raw)) + (lr * AT_P + lc) * 4;
  int next = r0 + lr;                                       // this thread's next row
  auto fetch = [&](int stage) {
    const uint32_t dst = to + stage * (2 * AT_K * AT_P * 4);
#pragma unroll
    for (int e = 0; e < AT_K / 4; ++e) {
      const bool in = next < r1;
      const bool ok_a = in && in_a && PRAC_IN(pa - g.A, (g.d - 1) * g.lda + g.m), ok_b = in && in_b && PRAC_IN(pb - g.B, (g.d - 1) * g.ldb + g.n);
      const float* const sa = ok_a ? pa : g.A;
      const float* const sb = ok_b ? pb : g.B;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + e * (4 * AT_P * 4)), "l"(sa), "r"(ok_a ? 4 : 0) : "memory");
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + (AT_K + 4 * e) * (AT_P * 4)), "l"(sb), "r"(ok_b ? 4 : 0) : "memory");
      pa += 4 * g.lda; pb += 4 * g.ldb; next += 4;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll 1
  for (int s = 0; s < AT_STAGES - 1; ++s) fetch(s);
  int stage = 0;
#pragma unroll 1
  for (int k0 = r0; k0 < r1; k0 += AT_K) {
    asm volatile("cp.async.wait_group %0;" ::"n"(AT_STAGES - 2) : "memory");
    __syncthreads();                 // everybody's part of this chunk is there, and the chunk before it has been read
    fetch((stage + AT_STAGES - 1) % AT_STAGES);
    const float* const As = raw + stage * (2 * AT_K * AT_P) + q4 * AT_P + gq;
#pragma unroll 2
    for (int kk = 0; kk < AT_K / 4; ++kk) {
      const float* const a = As + kk * 4 * AT_P + wa;
      const float* const b = As + (AT_K + kk * 4) * AT_P + wb;
      const double a0 = a[0], a1 = a[8];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const double bv = b[c * 8];
        ptx::dmma_884(acc[0][c], a0, bv);
        ptx::dmma_884(acc[1][c], a1, bv);
      }
    }
    stage = (stage + 1) % AT_STAGES;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < 4; ++c)
      *reinterpret_cast<double2*>(&tile[(wa + h * 8 + gq) * AT_P + wb + c * 8 + 2 * q4]) = make_double2(acc[h][c][0], acc[h][c][1]);
  ptx::cluster_arrive();
  ptx::cluster_wait();
  // rows [64 rank / slices, 64 (rank + 1) / slices) of the tile
  const int rows = AT_T / slices;
#pragma unroll 1
  for (int idx = t; idx < rows * AT_T; idx += 256) {
    const int r = rows * rank + idx / AT_T, c = idx % AT_T;
    const int i = m0 + r, j = n0 + c;
    double v = 0.0;
#pragma unroll 4
    for (int s = 0; s < slices; ++s) v += ptx::cluster_ld_f64(ptx::cluster_addr(&tile[r * AT_P + c], s));
    v *= g.alpha;
    if (i >= g.m || j >= g.n || (g.symmetric && i > j)) continue;
    const int copies = g.symmetric && i != j ? 2 : 1;
#pragma unroll 1
    for (int e = 0; e < copies; ++e) {
      const long long o = e ? static_cast<long long>(j) * g.ldo + i : static_cast<long long>(i) * g.ldo + j;
      if (!PRAC_IN(o, static_cast<long long>(g.m - 1) * g.ldo + g.n)) continue;
      if (g.out_double) static_cast<double*>(g.out)[o] = v;
      else static_cast<float*>(g.out)[o] = static_cast<float>(v);
    }
  }
  ptx::cluster_arrive();                  // (nobody's tile goes away under a reader)
  ptx::cluster_wait();
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
  int flag_bit;            // set for a bad pivot
  int weak_bit;            // set for a weak column (0: not looked at)
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
    ptx::dmma_884(acc0, a, b0);
    ptx::dmma_884(acc1, a, b1);
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

__device__ __forceinline__ double pivot_guard(double diagonal_on_entry) {
  return diagonal_on_entry > 0.0 ? 1e-13 * diagonal_on_entry : 1.0;
}

// Where a diagonal block is factored, all in shared memory.  D: the block (upper triangle); guard: limits below which a
// pivot is replaced.  Lin: the block rows of R^-T, D = R^T R (zero right of the diagonal tiles on entry).  E: the
// identity under the same elimination.  W: eight rows of R at a time, rows 0..7 and 8..15 in turn.
struct CholBlock { double (*D)[CP]; double (*Lin)[CP]; double (*E)[CP]; double (*W)[CP]; const double* guard; };

// The column of a sub-block's row that a lane carries through the elimination: tile `lane / 8` of four (the
// identity, the tiles of D right of the diagonal, those of E left of it), column lane % 8.
struct CholLane { int column; bool unit, of_d; };
__device__ __forceinline__ CholLane chol_lane(int s) {
  const int lane = threadIdx.x & 31, i = lane >> 3;
  CholLane l;
  l.unit = i == 0;
  l.of_d = i > 0 && s + i < CB / 8;
  l.column = 8 * (l.unit ? s : (l.of_d ? s + i : s + i - CB / 8)) + (lane & 7);
  return l;
}
__device__ __forceinline__ double chol_lane_load(const CholBlock& b, const CholLane& l, int s, int k) {
  if (l.unit) return (threadIdx.x & 7) == k ? 1.0 : 0.0;
  return (l.of_d ? b.D : b.E)[8 * s + k][l.column];
}
__device__ __forceinline__ double* chol_lane_out(const CholBlock& b, const CholLane& l, int s) {
  return l.of_d ? &b.W[8 * (s & 1)][l.column] : &b.Lin[8 * s][l.column];
}

// Sub-block s in the careful form, for one in which a pivot is not safely positive relative to the
// column's original squared norm: such a pivot is replaced by a guard value (and reported).  One warp; the
// diagonal tile is overwritten.
__device__ __noinline__ void sub_chol_guarded(const CholBlock b, int s, int* dev_status, int flag_bit) {
  const int lane = threadIdx.x & 31, o = 8 * s;
  const CholLane l = chol_lane(s);
  double* const out = chol_lane_out(b, l, s);
  double rhs[8];
  for (int k = 0; k < 8; ++k) rhs[k] = chol_lane_load(b, l, s, k);
  for (int j = 0; j < 8; ++j) {
    __syncwarp();
    double pv = b.D[o + j][o + j];
    if (!(pv > b.guard[o + j])) {
      pv = b.guard[o + j];
      if (lane == 0 && flag_bit && dev_status) atomicOr(dev_status, flag_bit);
    }
    for (int r = j + 1; r < 8; ++r) rhs[r] = fma(-(b.D[o + j][o + r] / pv), rhs[j], rhs[r]);
    for (int i = lane; i < 64; i += 32) {
      const int r = i >> 3, c = i & 7;
      if (r > j && c >= r) b.D[o + r][o + c] = fma(-(b.D[o + j][o + r] / pv), b.D[o + j][o + c], b.D[o + r][o + c]);
    }
    out[j * CP] = rhs[j] * rsqrt(pv);
  }
}

// a / b by one step of the hyperpower iteration of order three (Altman, Pacific J. Math. 10, 1960, for inverses of
// operators) on the hardware's approximation x0 of 1 / b, which is good to 20 bits: with e = 1 - b x0, 1 / b = x0 (1 + e + e^2)
// up to e^3 = 2^-60, and the three roundings of the quotient.  b has to be a normal number with a normal reciprocal.
struct CubicQuotient {
  double x0, corr;
  __device__ __forceinline__ explicit CubicQuotient(double b) {
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x0) : "d"(b));
    const double e = fma(-b, x0, 1.0);
    corr = fma(e, e, e);
  }
  __device__ __forceinline__ double operator()(double a) const {
    const double q = a * x0;
    return fma(q, corr, q);
  }
};

// The same without the tests.  Every lane eliminates the 8 x 8 tile in its own registers (no exchange between the
// dependent steps: pivot, reciprocal, multiplier, next pivot; with the tile spread over the lanes and rows
// passed by shuffles a column took 165 cycles, here 115 with its loads and stores) and takes its own column along, so that the
// whole block row s of R and of R^-T comes out with it.  The multipliers, on the way from one pivot to the next, are quotients
// by the cubic iteration (a division took 12 us more per factorisation of 320 columns); the square root is not on that way.
// Returns whether all pivots were good.
__device__ __forceinline__ bool sub_chol(const CholBlock& b, int s) {
  const int o = 8 * s;
  const CholLane l = chol_lane(s);
  double* const out = chol_lane_out(b, l, s);
  double m[8][8], rhs[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
#pragma unroll
    for (int j = i & ~1; j < 8; j += 2) {
      const double2 v = *reinterpret_cast<const double2*>(&b.D[o + i][o + j]);
      if (j >= i) m[i][j] = v.x;
      m[i][j + 1] = v.y;
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) rhs[k] = chol_lane_load(b, l, s, k);
  bool good = true;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const double pv = m[j][j];
    const CubicQuotient by_pivot(pv);
#pragma unroll
    for (int r = j + 1; r < 8; ++r) {
      const double f = by_pivot(m[j][r]);
#pragma unroll
      for (int c = r; c < 8; ++c) m[r][c] = fma(-f, m[j][c], m[r][c]);
      rhs[r] = fma(-f, rhs[j], rhs[r]);
    }
    out[j * CP] = rhs[j] * rsqrt(pv);
    good = good && pv > b.guard[o + j];                           // (false for NaN)
  }
  return good;
}

// C (8 x 8 tile) = [C] - R_p^T B_q, the k = 8 rows of a sub-block.
__device__ __forceinline__ void sub_update(double (*C)[CP], int p, int q, const double (*R)[CP], const double (*B)[CP], bool fresh) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q4 = lane & 3;
  double2* const o = reinterpret_cast<double2*>(&C[8 * p + g][8 * q + 2 * q4]);
  const double2 old = *o;
  double a0[2] = {0.0, 0.0}, a1[2] = {0.0, 0.0};
  ptx::dmma_884(a0, R[q4][8 * p + g], B[q4][8 * q + g]);
  ptx::dmma_884(a1, R[4 + q4][8 * p + g], B[4 + q4][8 * q + g]);
  *o = make_double2((fresh ? 0.0 : old.x) - (a0[0] + a1[0]), (fresh ? 0.0 : old.y) - (a0[1] + a1[1]));
}

// D (CB x CB, symmetric positive definite on entry, upper triangle used) -> Lin = R^-T (lower), where R^T R = D, by
// the 256 main threads, which have met at a barrier since D and the limits were written.  The
// chain of 32 dependent column steps is what this costs, so one warp walks it, eight columns at a time, each lane on
// its own (sub_chol); the other warps bring the 8 x 8 tiles below up to date on the fp64 tensor cores, those of the
// next row first.  With R_s the eight rows of R from sub-block s: D_pq -= R_sp^T R_sq, and the same elimination applied
// to an identity (E) gives the block rows of R^-T: E_pc -= R_sp^T Lin_sc.
// rows_done(s): rows 8 s .. 8 s + 7 of Lin, final, are visible to warps 4..7, which call it (after the last, warps 0..3).
template <typename RowsDone>
__device__ __forceinline__ void blk_chol_inv(const CholBlock& b, int* dev_status, int flag_bit, RowsDone rows_done) {
  static_assert(CB == 32, "four sub-blocks of eight columns");
  const int warp = threadIdx.x >> 5;
#pragma unroll 1
  for (int s = 0; s < CB / 8; ++s) {
    double (*R)[CP] = b.W + 8 * (s & 1);
    const double (*L)[CP] = b.Lin + 8 * s;
    if (warp == 0 && !sub_chol(b, s)) sub_chol_guarded(b, s, dev_status, flag_bit);     // (the lanes agree)
    main_sync();
    if (s + 1 == CB / 8) break;
    // row s + 1, the four tiles that the next sub-block starts from: its part of D (warp 0 the diagonal tile) and of E
    if (warp < 4) {
      const int q = s + 1 + warp;
      const bool of_d = q < CB / 8;
      sub_update(of_d ? b.D : b.E, s + 1, of_d ? q : q - CB / 8, R, of_d ? R : L, q - CB / 8 == s);   // (E_ps starts from zero)
      bar_sync(8, 128);
    } else {
      rows_done(s);
      // the rows below, beside the next sub-block's chain
      const int rest = CB / 8 - 2 - s, nd = rest * (rest + 1) / 2, ne = rest * (s + 1);
      for (int u = warp - 4; u < nd + ne; u += 4) {
        if (u < nd) {
          int p = s + 2, left = u;
          while (left >= CB / 8 - p) { left -= CB / 8 - p; ++p; }
          sub_update(b.D, p, p + left, R, R, false);
        } else {
          const int c = (u - nd) % (s + 1);
          sub_update(b.E, s + 2 + (u - nd) / (s + 1), c, R, L, c == s);
        }
      }
    }
  }
  if (warp < 4) rows_done(CB / 8 - 1);
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
// matrix, or the transposed matrix as three bf16 pieces.  transposed: S holds the block's transpose.
__device__ __forceinline__ void chol_emit(const CholArgs& a, const double (*S)[CP], int p, int q, bool transposed = false) {
  for (int idx = group_tid(); idx < CB * CB; idx += 256) {
    if (!a.Rt3) {
      const int i = p * CB + idx / CB, j = q * CB + idx % CB;
      if (i < a.n && j < a.n) a.Rinv[static_cast<long long>(i) * a.ldr + j] = static_cast<float>(transposed ? S[idx % CB][idx / CB] : S[idx / CB][idx % CB]);
    } else {
      const int j = q * CB + idx / CB, l = p * CB + idx % CB;
      if (j < a.n && l < a.kp) {
        float x = l < a.n ? static_cast<float>(transposed ? S[idx / CB][idx % CB] : S[idx % CB][idx / CB]) : 0.f;
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
// A column is weak where the columns before it leave less than 1e-3 of its squared norm.  The fp32 product V R^-1 is then off
// orthonormal by 2^-24 times a condition number of 30 and more, and what is left of that decides how well the panel spans what it should: a
// few weak columns in the null space of a rank-deficient input (noise, as many vectors as it has dimensions) turned the dominant
// space by 1e-3 in 6 % of such fits and left U off orthonormal by up to 0.7.  inv: the column's entry of R^-1 on the diagonal.
__device__ __forceinline__ void chol_report_weak(const CholArgs& a, double inv, double diagonal_on_entry) {
  if (a.weak_bit && inv * inv * diagonal_on_entry > 1e3) atomicOr(a.dev_status, a.weak_bit);
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
// factorisation per block and never waits for global memory.  On 320 columns, which it served before
// chol_cluster_kernel, a factorisation took 132 us when every CTA factored the diagonal block itself and then did its blocks between
// grid barriers, 103 us with a grid barrier per block and CTA 0 on the chain, 76 us in this form.  Draws before and after the
// lane-wise elimination (sub_chol) and A^T B on clusters, together: 2048 x 640 328 and 325 us, 5461 x 513 401 and 398, 5461 x 640 407 and 412.
//
// Every wait on another CTA is bounded; a CTA that gives up (or sees that another did) reports it and
// leaves; nothing asynchronous is in flight here, so the early exit is clean.
__global__ void __launch_bounds__(CHOL_MAIN + CHOL_HELP) chol_inv_kernel(const CholArgs a) {
  if (a.run_if_mask && pass_is_off(a.dev_status, a.run_if_mask)) return;
  extern __shared__ __align__(16) double chol_smem[];
  __shared__ int ok_sh[2];
  __shared__ double guard[CB];
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
        guard[threadIdx.x] = pivot_guard(i < n ? a.diag0[i] : 1.0);
        __syncwarp();
      }
      double* const inv = a.Dinv + static_cast<long long>(j) * CB * CB;
      blk_chol_inv(CholBlock{D, S2, S3, S5, guard}, a.dev_status, a.flag_bit, [](int) {});
      for (int idx = threadIdx.x; idx < CB * CB; idx += CHOL_MAIN) {
        const int r = idx / CB, c = idx % CB;
        inv[idx] = S1[r][c] = r <= c ? S2[c][r] : 0.0;
      }
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
    if (worker == static_cast<int>(workers) - 1) {
      chol_emit(a, S1, j, j);
      if (t < CB && j * CB + t < n) chol_report_weak(a, S1[t][t], __ldcg(&a.diag0[j * CB + t]));
      sync();
    }
  }
}

// ------------------------------------------------------------------ the same on one cluster, up to 16 blocks of columns
constexpr int CC_MAX = 16;                       // blocks of columns = CTAs of the cluster
constexpr int CC_GROUPS = 2;                     // groups of 256 threads in a CTA
constexpr uint64_t CC_WAIT_NS = 2000000000ull;   // what a wait may last
// What the CTAs tell one another: barriers in the shared memory of the CTA that waits, each for one event.
struct ChainWords {
  uint64_t row[CC_MAX][CC_MAX];   // [c][x]: block (c, x) of R is final in CTA x
  uint64_t diag[CC_MAX];          // [c]: R_cc^-T is final in CTA c
  uint64_t band[CB / 8];          // rows 8 s .. 8 s + 7 of R_cc^-T from the CTA before this one have arrived here
  int abort;                      // a wait gave up
};

// Column blocks of G and block rows of the inverse stay in shared memory for the whole factorisation: CTA q of
// the cluster holds the blocks (p, q), p <= q, of G, which become those of R, and row q of X = R^-1 (its diagonal block
// transposed).  Step c, once R_cc^-1
// is known: the CTAs right of c form R_cq = R_cc^-T G_cq and subtract R_cp^T R_cq from their blocks (p, q), p > c; the others
// close X_qc = X_qc R_cc^-1 and subtract X_qc R_cx from their running sums X_qx, x > c.  The blocks R_cx of another CTA are
// fetched from its shared memory when it has said that they are final; nothing is ever overwritten that another
// CTA may still want.  CTA c + 1, whose diagonal block the chain waits for, has nothing else to do in step c: the rows of
// R_cc^-T are stored into its shared memory as they are formed, eight at a time, and its threads form the same rows of
// R_c,c+1 and take their part off the diagonal block while the next eight are on their way.
//
// The chain of diagonal blocks is what this costs.  A factorisation whose CTAs met through flags in global memory
// (chol_inv_kernel) took 13 400 cycles a block, most of them the way of a block through L2 and back.
//
// Every wait on another CTA is bounded, in polls and in time (a poll may itself block for a while); a CTA that gives up tells the
// others.  Then every CTA that has not sent its rows of R_cc^-T sends zeros in their place, every CTA waits for all the rows
// that it is to receive (that wait ends, since they have all been sent; it is bounded too), and all meet at the cluster's
// barrier before any leaves: nobody's shared memory goes away under a reader or under a store on its way.
//
// A CTA walks most of this code once, with its instructions not in the SM's cache yet (270 cycles per 128 bytes).  A dry run
// of the chain's part of a step on an identity, while the product before this kernel was still running, was no gain: the
// product fills the GPU at 160 columns and more, and below that the dry run's own time shows (draws of 320 columns 104 us with
// it, 96 without; fits of 2048 x 256 1559 and 1526, of the small fp32 layer 390 and 383; four fits side by side the same).
__global__ void __launch_bounds__(256 * CC_GROUPS, 1) chol_cluster_kernel(const CholArgs a) {
  extern __shared__ __align__(16) double chol_smem[];
  __shared__ double guard[CB];
  __shared__ ChainWords words;
  typedef double (*Blk)[CP];
  const int n = a.n, nb = a.nb, q = static_cast<int>(blockIdx.x);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, group = tid >> 8, gt = tid & 255;
  const int g = lane >> 2, q4 = lane & 3;
  auto block = [&](int i) { return reinterpret_cast<Blk>(chol_smem + static_cast<size_t>(i) * CB * CP); };
  auto col = [&](int p) { return block(p); };                 // (p, q) of G, then of R
  auto inv = [&](int x) { return block(x + 1); };             // (q, x) of R^-1, x >= q
  Blk const W = block(nb + 1), Dprev = block(nb + 2), Dfar = block(nb + 3);
  Blk const stage = block(nb + 4 + group);
  Blk const E = block(nb + 4);                                // (group 0's: it factors or it fetches)
  bool fail = false, sent = false;               // sent: this CTA's rows are on their way to the next one

  // After a poll in vain: whether to give up, because this wait has lasted too long (the others are told) or another gave up.
  auto gives_up = [&](unsigned polls, uint64_t& since) {
    bool late = polls >= a.poll_limit;
    if ((polls & 63u) == 0u) {
      if (*reinterpret_cast<volatile int*>(&words.abort)) return true;
      const uint64_t now = ptx::globaltimer_ns();
      if (since == 0) since = now;
      late = late || now - since > CC_WAIT_NS;
    }
    if (late)
      for (int x = 0; x < nb; ++x) ptx::cluster_st_release(ptx::cluster_addr(&words.abort, x), 1);
    return late;
  };
  // Every lane waits for a barrier of its own (or none): cheap polls, and one that acquires (it takes 400 cycles) once
  // all of them are through.  Where a lane gives up the caller carries on with what it has, until the CTA next meets and leaves together.
  auto wait_for = [&](uint64_t* bar) {
    if (bar != nullptr && !fail) {
      unsigned polls = 0;
      uint64_t since = 0;
      while (!cluster_try_wait(bar))
        if (gives_up(++polls, since)) { fail = true; break; }
    }
    __syncwarp();
    if (bar != nullptr && !fail) (void)cluster_try_wait_acquire(bar);
    __syncwarp();
  };
  // (what arrives by cluster_st_async is visible to who has seen its barrier complete)
  auto wait_rows = [&](uint64_t* bar) {
    if (lane == 0 && !fail) {
      unsigned polls = 0;
      uint64_t since = 0;
      while (!ptx::mbar_try_wait(bar, 0))
        if (gives_up(++polls, since)) { fail = true; break; }
    }
    __syncwarp();
  };
  // Rows 8 s .. 8 s + 7 of R_qq^-T up to the diagonal tile, to the next CTA (128 threads): rows(r, cc) is the pair at column cc.
  const uint32_t far = q + 1 < nb ? ptx::cluster_addr(Dprev, q + 1) : 0u, far_bar = q + 1 < nb ? ptx::cluster_addr(words.band, q + 1) : 0u;
  auto send_rows = [&](int s, auto rows) {
    const int i = tid & 127, r = 8 * s + (i & 7), cc = 2 * (i >> 3);
    if (cc < 8 * (s + 1)) ptx::cluster_st_async(far + (r * CP + cc) * 8, rows(r, cc), far_bar + 8 * s);
  };
  // the pairs (row, 2 columns) of a block that a thread of a group moves
  auto pull = [&](uint32_t from, double2 (&v)[2]) {
#pragma unroll
    for (int e = 0; e < 2; ++e)
      v[e] = ptx::cluster_ld_f64x2(from + (((gt + 256 * e) >> 4) * CP + 2 * (gt & 15)) * 8);
  };
  auto put = [&](Blk to, const double2 (&v)[2]) {
#pragma unroll
    for (int e = 0; e < 2; ++e) *reinterpret_cast<double2*>(&to[(gt + 256 * e) >> 4][2 * (gt & 15)]) = v[e];
  };

  grid_dep_wait();
  if (a.run_if_mask && pass_is_off(a.dev_status, a.run_if_mask)) return;
  if (tid < CC_MAX * CC_MAX) cluster_bar_init(&words.row[0][0] + tid, 0);
  else if (tid < CC_MAX * CC_MAX + CC_MAX) cluster_bar_init(&words.diag[tid - CC_MAX * CC_MAX], 0);
  else if (tid < CC_MAX * CC_MAX + CC_MAX + CB / 8) {
    const int s = tid - CC_MAX * CC_MAX - CC_MAX;
    cluster_bar_init(&words.band[s], q > 0 ? 8 * 8 * (s + 1) * 8 : 0);          // eight rows up to the diagonal tile, in bytes
  }
  if (tid == 511) words.abort = 0;
  ptx::fence_mbar_init();
  __syncthreads();
  ptx::cluster_arrive();
  // this CTA's column of G, padded with the identity
  for (int i0 = tid / CB; i0 < (q + 1) * CB; i0 += 8 * (256 * CC_GROUPS / CB)) {           // (eight loads in flight)
    double v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int i = i0 + e * (256 * CC_GROUPS / CB), j = q * CB + tid % CB;
      v[e] = i == j ? 1.0 : 0.0;
      if (i < n && j < n) v[e] = __ldcg(&a.G[static_cast<long long>(i) * n + j]);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int i = i0 + e * (256 * CC_GROUPS / CB);
      if (i < (q + 1) * CB) col(i / CB)[i % CB][tid % CB] = v[e];
    }
  }
  for (int idx = tid; idx < (nb - q) * CB * CP; idx += 256 * CC_GROUPS)          // the running sums
    inv(q)[0][idx] = 0.0;
  if (group == 1) chol_emit_zeros(a, q, nb);
  ptx::cluster_wait();
  __syncthreads();
  if (tid < CB) guard[tid] = pivot_guard(col(q)[tid][tid]);
  __syncthreads();

  // c = -1: CTA 0 factors its block; then the steps
  for (int c = -1; c < nb; ++c) {
    if (c == q - 1) {
      // ---- the chain: block (c, q) of R and the diagonal block, by rows of R_cc^-T as they come; then the factorisation
      Blk const Dq = col(q), Rbuf = Dfar;
      if (c == -1) {
        // (CTA 0: nothing to take off)
      } else if (group == 1) {
        for (int s = (warp >> 2) & 1; s < CB / 8; s += 2) {
          wait_rows(&words.band[s]);
          Blk const mine = col(c);
          const int r0 = 8 * s, c0 = 8 * (warp & 3);
          double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 2
          for (int ks = 0; ks < 2 * s + 2; ks += 2) {
            ptx::dmma_884(acc[0], Dprev[r0 + g][ks * 4 + q4], mine[ks * 4 + q4][c0 + g]);
            ptx::dmma_884(acc[1], Dprev[r0 + g][ks * 4 + 4 + q4], mine[ks * 4 + 4 + q4][c0 + g]);
          }
          *reinterpret_cast<double2*>(&Rbuf[r0 + g][c0 + 2 * q4]) = make_double2(acc[0][0] + acc[1][0], acc[0][1] + acc[1][1]);
          bar_arrive(9 + s, 128 + 256);
        }
      } else {
        // a tile of the upper triangle per warp, two for the last two
        const int u0 = warp, u1 = warp >= 6 ? warp + 2 : -1;
        auto tile = [](int u, int& p, int& x) {
          p = 0;
          while (u >= 4 - p) { u -= 4 - p; ++p; }
          x = p + u;
        };
        int p0, x0, p1 = 0, x1 = 0;
        tile(u0, p0, x0);
        if (u1 >= 0) tile(u1, p1, x1);
        double acc[2][2][2] = {};
#pragma unroll 1
        for (int s = 0; s < CB / 8; ++s) {
          bar_sync(9 + s, 128 + 256);
          const double (*R)[CP] = Rbuf + 8 * s;
          ptx::dmma_884(acc[0][0], R[q4][8 * p0 + g], R[q4][8 * x0 + g]);
          ptx::dmma_884(acc[0][1], R[4 + q4][8 * p0 + g], R[4 + q4][8 * x0 + g]);
          if (u1 >= 0) {
            ptx::dmma_884(acc[1][0], R[q4][8 * p1 + g], R[q4][8 * x1 + g]);
            ptx::dmma_884(acc[1][1], R[4 + q4][8 * p1 + g], R[4 + q4][8 * x1 + g]);
          }
        }
        double2* o = reinterpret_cast<double2*>(&Dq[8 * p0 + g][8 * x0 + 2 * q4]);
        double2 old = *o;
        *o = make_double2(old.x - (acc[0][0][0] + acc[0][1][0]), old.y - (acc[0][0][1] + acc[0][1][1]));
        if (u1 >= 0) {
          o = reinterpret_cast<double2*>(&Dq[8 * p1 + g][8 * x1 + 2 * q4]);
          old = *o;
          *o = make_double2(old.x - (acc[1][0][0] + acc[1][1][0]), old.y - (acc[1][0][1] + acc[1][1][1]));
        }
        main_sync();
      }
      if (group == 0) {
        Blk const Lin = inv(q);
        const bool next = q + 1 < nb;
        blk_chol_inv(CholBlock{Dq, Lin, E, W, guard}, a.dev_status, a.flag_bit, [&](int s) {
          if (next) send_rows(s, [&](int r, int cc) { return *reinterpret_cast<const double2*>(&Lin[r][cc]); });
        });
      } else if (c >= 0) {
        bar_sync(2, 256);                        // (Rbuf is complete)
        double2 v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) v[e] = *reinterpret_cast<const double2*>(&Rbuf[(gt + 256 * e) >> 4][2 * (gt & 15)]);
        put(col(c), v);
        bar_sync(2, 256);
        if (warp == 15 && lane < nb && lane != q) ptx::mbar_arrive_cluster(ptx::cluster_addr(&words.row[c][q], lane));
      }
      sent = true;
      // every thread leaves here if one has given up
      if (__syncthreads_or(fail)) { fail = true; break; }
      if (warp == 8 && lane < nb && lane != q) ptx::mbar_arrive_cluster(ptx::cluster_addr(&words.diag[q], lane));
    }
    if (c >= 0 && c != q - 1) {
      const bool left = c < q;
      Blk const own = left ? col(c) : inv(c);
      // ---- R_cc^-T, then this CTA's own block of step c
      if (c != q) {
        wait_for(lane == 0 ? &words.diag[c] : nullptr);
        {
          const int r = tid >> 4, cc = 2 * (tid & 15);
          const double2 v = ptx::cluster_ld_f64x2(ptx::cluster_addr(&block(c + 1)[r][cc], c));
          *reinterpret_cast<double2*>(&Dfar[r][cc]) = v;
        }
        __syncthreads();
        const int r0 = (warp >> 2) * 8, c0 = (warp & 3) * 8;    // a tile per warp
        double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
        // (R_cc^-T is lower triangular: the products end where it does)
        const int ks_end = left ? 2 * (warp >> 2) + 2 : 2 * (warp & 3) + 2;
#pragma unroll 2
        for (int ks = 0; ks < ks_end; ks += 2) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int k = (ks + e) * 4 + q4;
            ptx::dmma_884(acc[e], left ? Dfar[r0 + g][k] : own[r0 + g][k], left ? own[k][c0 + g] : Dfar[c0 + g][k]);
          }
        }
        __syncthreads();
        *reinterpret_cast<double2*>(&own[r0 + g][c0 + 2 * q4]) = make_double2(acc[0][0] + acc[1][0], acc[0][1] + acc[1][1]);
        if (__syncthreads_or(fail)) { fail = true; break; }
        if (left && warp == 15 && lane < nb && lane != q) ptx::mbar_arrive_cluster(ptx::cluster_addr(&words.row[c][q], lane));
      }
      // ---- the blocks it brings up to date, dealt to the groups: (p, q), c < p <= q, of G, (q, q) first, which needs nobody
      // else's block; or (q, x), x > c, of the inverse
      if (left && group == 0) blk_mm(col(q), own, own, 1);
      if (!left && group == 1) {
        chol_emit(a, own, q, c, c == q);
        if (c == q && gt < CB) chol_report_weak(a, own[gt][gt], 1e13 * guard[gt]);       // (a zero column is a bad pivot anyway)
      }
      const int first = c + 1 + (left ? 1 - group : group), end = left ? q : nb;
      Blk const from = block(c);
      double2 v[2];
      if (first < end) {
        const int mine = first + CC_GROUPS * lane;
        wait_for(mine < end ? &words.row[c][mine] : nullptr);
        pull(ptx::cluster_addr(from, first), v);
      }
      for (int x = first; x < end; x += CC_GROUPS) {
        bar_sync(1 + group, 256);            // the block before this one is done with
        put(stage, v);
        bar_sync(1 + group, 256);
        if (x + CC_GROUPS < end) pull(ptx::cluster_addr(from, x + CC_GROUPS), v);
        Blk const C = left ? col(x) : inv(x);
        if (left) blk_mm(C, stage, own, 1);
        else blk_mm(C, own, stage, c == q ? 1 : 3);
      }
      __syncthreads();
    }
  }
  fail = __syncthreads_or(fail) != 0;
  if (fail) {
    if (tid == 0 && a.dev_status) atomicOr(a.dev_status, DEV_WAIT_EXPIRED);
    if (!sent && q + 1 < nb && tid < 128)
      for (int s = 0; s < CB / 8; ++s) send_rows(s, [](int, int) { return make_double2(0.0, 0.0); });
    if (tid == 0 && q > 0) {
      const uint64_t since = ptx::globaltimer_ns();
      for (int s = 0; s < CB / 8; ++s)
        while (!ptx::mbar_try_wait(&words.band[s], 0) && ptx::globaltimer_ns() - since <= 2 * CC_WAIT_NS) {}
    }
    __syncthreads();
  }
  ptx::cluster_arrive();
  ptx::cluster_wait();
}

size_t chol_cluster_smem(int nb) {
  const size_t need = static_cast<size_t>(nb + 4 + CC_GROUPS) * CB * CP * 8;
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

// Whether a cluster of nb CTAs of chol_cluster_kernel can be placed where this stream's kernels run.  Asked for every
// launch (0.3 us), as what a process may use can shrink; where the answer is no, chol_inv_kernel serves.
bool chol_cluster_fits(int nb, cudaStream_t stream) {
  if (nb < 1 || nb > CC_MAX || cooperative_cholesky_forced()) return false;
  static DeviceOnce attrs;
  int dev = -1;
  bool ok = cudaGetDevice(&dev) == cudaSuccess;
  if (ok && !attrs.done(dev)) {
    ok = cudaFuncSetAttribute(chol_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(chol_cluster_smem(CC_MAX))) == cudaSuccess &&
         cudaFuncSetAttribute(chol_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    if (ok) attrs.mark(dev);
  }
  if (ok) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    chol_cluster_config(cfg, attr, nb, stream);
    int clusters = 0;
    ok = cudaOccupancyMaxActiveClusters(&clusters, chol_cluster_kernel, &cfg) == cudaSuccess && clusters >= 1;
  }
  if (!ok) (void)cudaGetLastError();
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

void atb_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], int tiles, int slices, cudaStream_t stream) {
  cfg = {};
  cfg.gridDim = dim3(tiles, slices);
  cfg.blockDim = dim3(256);
  cfg.stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = slices;
  attr[0].val.clusterDim.z = 1;
  attr[1] = dependent_launch_attr();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
}

// Slices of the rows = CTAs of a tile's cluster: what lets the busiest SM go through the fewest chunks of 16 rows.  A chunk takes
// 0.7 us whether one or several CTAs share the SM (the fp64 rate), a launch 5 to 7 us beside that, at every number of
// slices.  Clusters have to lie within a group of SMs: with a CTA per SM the device holds 74, 33, 15 and 7 clusters of 2, 4, 8 and 16, so on
// 148, 132, 120 and 112 SMs.  Up to three CTAs per SM the SMs with one more set the time, above that it evens out.  Where the count is the
// same 8 is taken, the fastest or within 5 % of it.  Symmetric, us with 4 / 8 / 16 slices: 2048 x 128 28.4 / 16.8 / 11.3, x 256
// 29.0 / 17.1 / 16.9, x 320 29.0 / 17.3 / 21.7, x 384 29.3 / 27.3 / 22.3, x 512 48.4 / 37.4 / 33.2, x 640 49.4 / 47.7 / 48.9; 5461 x 512
// 118 / 89.0 / 76.7, x 640 120 / 116 / 117.  Whether the cluster can be placed is asked for every launch (see chol_cluster_fits).
int atb_slices(int tiles, int64_t d, cudaStream_t stream) {
  static DeviceOnce wide;                      // (16 is more than the portable cluster size)
  int dev = -1;
  bool ok = cudaGetDevice(&dev) == cudaSuccess;
  if (ok && !wide.done(dev)) {
    ok = cudaFuncSetAttribute(atb_f64_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    if (ok) wide.mark(dev);
  }
  if (!ok) (void)cudaGetLastError();           // (then 16 cannot be placed)
  tc_init();
  const int sms = tc_num_sms() > 0 ? tc_num_sms() : 148;
  int best = 0;
  long long least = 0;
  for (const int s : {8, 16, 4, 2, 1}) {
    const int room = s <= 2 ? sms : sms * (s == 4 ? 132 : (s == 8 ? 120 : 112)) / 148;
    const long long ctas = static_cast<long long>(tiles) * s, rows = (d + AT_K * s - 1) / (AT_K * s);
    const long long chunks = ctas <= 3ll * room ? (ctas + room - 1) / room * rows : (ctas * rows + room - 1) / room;
    if (best == 0 || chunks < least) { least = chunks; best = s; }
  }
  for (; best > 1; best /= 2) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    atb_config(cfg, attr, tiles, best, stream);
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, atb_f64_kernel, &cfg) == cudaSuccess && clusters >= 1) break;
    (void)cudaGetLastError();
  }
  return best;
}

__global__ void quotients_kernel(const double* a, const double* b, double* q, long long n) {
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (i < n) q[i] = CubicQuotient(b[i])(a[i]);
}

}  // namespace

PRAC_BOUNDS_READER(bounds_violations_cholqr)

// ------------------------------------------------------------------ host side
int atb_f64(const float* A, int64_t lda, const float* B, int64_t ldb, int64_t d, int64_t m, int64_t n,
            int symmetric, double alpha, void* out, int64_t ldo, int out_double, cudaStream_t stream, const int* run_if,
            int run_if_mask, void* zero_words, int zero_bytes) {
  if (m <= 0 || n <= 0) return PRAC_OK;
  if (d <= 0 || (symmetric && (A != B || m != n))) return PRAC_EINVAL;
  AtbArgs g{};
  g.A = A; g.lda = lda; g.B = B; g.ldb = ldb;
  g.m = static_cast<int>(m); g.n = static_cast<int>(n); g.d = d;
  const int tiles_m = static_cast<int>((m + AT_T - 1) / AT_T);
  g.tiles_n = static_cast<int>((n + AT_T - 1) / AT_T);
  g.symmetric = symmetric;
  g.alpha = alpha;
  g.out = out; g.ldo = ldo; g.out_double = out_double;
  g.run_if = run_if; g.run_if_mask = run_if_mask;
  g.zero_words = static_cast<int*>(zero_words); g.zero_count = zero_bytes / 4;
  const int tiles = symmetric ? g.tiles_n * (g.tiles_n + 1) / 2 : tiles_m * g.tiles_n;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  atb_config(cfg, attr, tiles, atb_slices(tiles, d, stream), stream);
  PRAC_CUDA_TRY(cudaLaunchKernelEx(&cfg, atb_f64_kernel, g));
  count_launch();
  return PRAC_OK;
}

// Workspace of one Cholesky-QR pass on n columns (all 256-byte aligned):
//   G n*n double | R n*n double | X n*n double | Dinv nb*CB*CB double | diag0 n double | Rinv n*n float
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

struct CholWs { double* G; double* R; double* X; double* Dinv; double* diag0; float* Rinv; size_t bytes;
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
  c.tensor = vr_on_tensor_cores(n, d);
  c.kp = (n + 63) / 64 * 64;
  const size_t oV3 = take(c.tensor ? static_cast<size_t>(d) * 3 * c.kp * 2 : 0);
  const size_t oR3 = take(c.tensor ? static_cast<size_t>(n) * 3 * c.kp * 2 : 0);
  const size_t oBar = take(sizeof(CholSync));
  char* b = static_cast<char*>(ws);
  c.sync = reinterpret_cast<CholSync*>(b + oBar);
  c.G = reinterpret_cast<double*>(b + oG); c.R = reinterpret_cast<double*>(b + oRR); c.X = reinterpret_cast<double*>(b + oX);
  c.Dinv = reinterpret_cast<double*>(b + oD); c.diag0 = reinterpret_cast<double*>(b + o0);
  c.Rinv = reinterpret_cast<float*>(b + oR);
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
  // (the product's kernel also zeroes the state of the factorisation that follows it)
  int st = atb_f64(Vin, ldin, Vin, ldin, d, n, n, 1, 1.0, c.G, n, 1, stream, run_if, run_if_mask,
                   c.sync, static_cast<int>(sizeof(CholSync)));
  if (st != PRAC_OK) return st;
  CholArgs a{};
  a.G = c.G; a.R = c.R; a.Dinv = c.Dinv; a.X = c.X; a.diag0 = c.diag0; a.Rinv = c.Rinv; a.ldr = n;
  a.n = static_cast<int>(n); a.nb = static_cast<int>((n + CB - 1) / CB);
  a.dev_status = dev_status; a.flag_bit = flag_bit;
  a.weak_bit = dev_status && flag_bit == DEV_CHOL_RETRY ? flag_bit : 0;
  a.sync = c.sync; a.poll_limit = barrier_poll_limit(); a.run_if_mask = run_if_mask;
  // an optional pass (run_if_mask != 0) is rare and small: it takes the general product
  const bool tensor = run_if_mask == 0 && c.tensor && tc_init() == PRAC_OK && aligned16(Vout) && (ldout % 4) == 0;
  a.Rt3 = tensor ? c.Rt3 : nullptr;
  a.kp = static_cast<int>(c.kp);
  if (chol_cluster_fits(a.nb, stream)) {
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
  // the rest.  A weak column (chol_report_weak) is not as orthogonal to the rest as fp32 allows.  One more pass
  // orthonormalises them; only if that pass breaks down is the failure reported.
  st = cholqr_pass(Vout, ldout, tmp, n, d, n, ws, ws_bytes, dev_status, DEV_CHOL_PIVOT, stream, DEV_CHOL_RETRY);
  if (st != PRAC_OK) return st;
  return launch_copy2d_if(tmp, n, Vout, ldout, d, n, dev_status, DEV_CHOL_RETRY, DEV_CHOL_RETRY, stream);
}

}  // namespace prac

extern "C" int prac_debug_quotients(const double* a, const double* b, double* q, int64_t n, void* stream) {
  if (!a || !b || !q || n <= 0) return PRAC_EINVAL;
  prac::quotients_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(a, b, q, n);
  PRAC_CUDA_TRY(cudaGetLastError());
  return PRAC_OK;
}

extern "C" size_t prac_debug_cholqr_ws_bytes(int64_t d, int64_t n) { return d > 0 && n > 0 ? prac::cholqr_ws_bytes(n, d) : 0; }
extern "C" int prac_debug_cholqr(const float* V, float* Q, int64_t d, int64_t n, void* ws, size_t ws_bytes, int32_t* word, void* stream) {
  if (!V || !Q || !ws || !word || d <= 0 || n <= 0) return PRAC_EINVAL;
  return prac::cholqr_pass(V, n, Q, n, d, n, ws, ws_bytes, word, prac::DEV_CHOL_PIVOT, static_cast<cudaStream_t>(stream));
}
