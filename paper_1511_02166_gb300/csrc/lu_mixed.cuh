// lu_mixed.cuh -- declarations shared by the FP32 factorisations of the
// mixed-precision path (k_solve_mixed.cu: one block per airfoil; k_lu_large.cu:
// the step-synchronous blocked factor of large airfoils) and the refinement.
#pragma once
#include "panel_common.cuh"

namespace panel {

constexpr int kSmemM = 230;  // largest m = n + 1 of a Gauss-Jordan inverse in shared memory
constexpr int kGjM = 288;    // m up to this: Gauss-Jordan inverse (k_gj_mixed.cu)
constexpr int kLargeM = 640; // m above this takes the step-synchronous blocked factor
constexpr int kSmemLuM = 222; // m up to this: LU with the whole matrix in shared memory
constexpr int kNB = 32;      // panel width
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

struct SolveArgs {
  Batch bt;
  const float* A_hi;
  const float* A_lo;
  float* LU;
  int32_t* piv;
  const double* rhs;
  const double* vinf;
  const double* chord;
  double* u;         // forward solution (may be NULL: no forward system)
  double* lam;       // transposed solution (may be NULL: no transposed system)
  int max_iter;
  double tol;
  int32_t* info;
  int32_t* iters;
  int inverse;       // m <= kGjM: Gauss-Jordan inverse (k_gj_mixed.cu) instead of the LU
  int n_cap;         // the caller's n_max (bt.n_max may be lowered to size a kernel)
  int rhs_kind;      // forward right-hand side: 0 rhs, 1 v m_y, 2 -v m_x (polar basis)
  int ir_shape;      // refinement block shape: 0 by size, 1..4 = 128x8, 256x4, 512x2, 1024x1
  int lu_kind;       // LU of m <= kSmemLuM: 2 whole matrix in shared memory, 1 through L2
  // Transposed right-hand side of a vector-Jacobian product (vjp != 0):
  // w_cl[b] dCl/du + w_u + w_cp dCp/du (each may be NULL = 0), with the
  // strengths u_in of the forward solution; vjp == 0 is dCl/du alone.
  int vjp;
  const double* w_cl;
  const double* w_u;   // [sum m_b], packed like u (gamma, C)
  const double* w_cp;  // [sum n_b], packed like the nodes
  const double* u_in;  // [sum m_b]
};

// Magnitude of an FP64 value as an integer that orders like it (0 for NaN, which a
// maximum passes over).
__device__ __forceinline__ unsigned long long magnitude_bits(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  return u <= 0x7ff0000000000000ull ? u : 0ull;
}
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32) == hi ? (unsigned)v : 0u);
  return ((unsigned long long)hi << 32) | lo;
}

// The refinement's stopping test of the systems q with run[q], by the whole block:
// dm[q], xm[q] are the thread's maxima (magnitude_bits) of the correction just applied
// and of the solution; dprev is the test's own memory (2 shared words); conv[q] is set once
// system q has converged.  red: 4 words of 64 bits per warp and one more.
// Converged when the correction just applied is below tol |x|, or when the contraction
// seen over the last two corrections (rho = |d_k| / |d_{k-1}| <= 1/8) predicts the next
// one, |d_k| rho, below tol |x|: the error left in x_{k+1} is about that next
// correction.  The correction of iteration 1 comes from the double-float residual, so
// the first test waits for iteration 2, and the sizes before iteration 1 are not needed.
// Ends with a barrier of the block.
// Sizes, tolerance and rule are FP64; only the maxima go over the integer pipe, and the
// rule is one warp's work per system, without the division: FP64 maxima in every thread
// were 12 % of a 100-panel refinement.  (Corrections pass through float32, so their
// squares neither overflow nor underflow in FP64.)
__device__ __forceinline__ void block_converged(const unsigned long long (&dm)[2],
                                                const unsigned long long (&xm)[2],
                                                const bool (&run)[2], int it, double tol,
                                                double* dprev, bool (&conv)[2], double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (it == 0) {
    __syncthreads();
    return;
  }
  unsigned long long* w = reinterpret_cast<unsigned long long*>(red);
  int* flag = reinterpret_cast<int*>(w + 4 * nw);
  unsigned long long d[2] = {0, 0}, x[2] = {0, 0};
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (run[q]) {
      d[q] = warp_max_u64(dm[q]);
      x[q] = warp_max_u64(xm[q]);
    }
  __syncthreads();  // (red may still be in use)
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      w[q * nw + warp] = d[q];
      w[(2 + q) * nw + warp] = x[q];
    }
  __syncthreads();
  if (warp < 2 && (warp == 0 ? run[0] : run[1])) {
    const double dmax = __longlong_as_double(
        (long long)warp_max_u64(lane < nw ? w[warp * nw + lane] : 0ull));
    if (it >= 2) {
      const double lim = tol * __longlong_as_double((long long)warp_max_u64(
                                   lane < nw ? w[(2 + warp) * nw + lane] : 0ull));
      const double dp = dprev[warp];
      const bool c = dmax <= lim || (dmax <= 0.125 * dp && dmax * dmax <= lim * dp);
      if (lane == 0) flag[warp] = c ? 1 : 0;
    }
    __syncwarp();
    if (lane == 0) dprev[warp] = dmax;
  }
  if (it == 1) return;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (run[q] && flag[q] != 0) conv[q] = true;
}
// Doubles of block_converged's scratch in a block of nt threads (block_sum needs 32; a
// whole number of 16-byte words).
__host__ __device__ constexpr int converged_words(int nt) {
  return nt / 8 + 2 > 32 ? nt / 8 + 2 : 32;
}

// border scale s = mean |A_jj| over the influence block (hi plane)
__device__ __forceinline__ double border_scale(const float* Ah, int n, int m, double* red) {
  double sdiag = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) sdiag += fabs((double)Ah[j * m + j]);
  return block_sum(sdiag, red) / n;
}

// ---------------------------------------------------------------------------
// Inverted diagonal blocks, in place: X = L_dd^{-1} (unit lower) replaces the
// part below the diagonal, Y = U_dd^{-1} (upper) the rest.  Each is one warp's
// work, lane j computing column j of the inverse in registers by substitution
// against the unit vector e_j, right-looking: once entry k of the column is
// final, it is multiplied into every later entry (L: rows below k, U: rows
// above k) at once, so each step is 31 independent FMAs on broadcast loads
// instead of a dependent dot product.  The two parts read and write disjoint
// entries (strictly below / on and above the diagonal): two warps may do them
// at the same time.  Every index into the register column is a compile-time
// constant (fully unrolled loops); kb <= 32 is the block size, B its first
// element, ld the row stride, all lanes of the warp call.
// ---------------------------------------------------------------------------
__device__ inline void invert_lower_unit(float* B, int ld, int kb) {
  const int j = threadIdx.x & 31;
  float acc[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i] = (i == j) ? 1.0f : 0.0f;
#pragma unroll
  for (int k = 0; k < 31; ++k) {
    if (k < kb) {
      const float xk = acc[k];  // X[k][j], final
#pragma unroll
      for (int i = k + 1; i < 32; ++i)
        if (i < kb) acc[i] = fmaf(-B[i * ld + k], xk, acc[i]);
    }
  }
  __syncwarp();
#pragma unroll
  for (int i = 1; i < 32; ++i)
    if (i < kb && j < i) B[i * ld + j] = acc[i];
  __syncwarp();
}

__device__ inline void invert_upper(float* B, int ld, int kb) {
  const int j = threadIdx.x & 31;
  float acc[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i] = (i == j) ? 1.0f : 0.0f;
#pragma unroll
  for (int k = 31; k >= 0; --k) {
    if (k < kb) {
      const float yk = acc[k] / B[k * ld + k];  // Y[k][j], final
      acc[k] = yk;
#pragma unroll
      for (int i = 0; i < k; ++i) acc[i] = fmaf(-B[i * ld + k], yk, acc[i]);
    }
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (i < kb && j >= i && j < kb) B[i * ld + j] = acc[i];
  __syncwarp();
}

__device__ inline void invert_block(float* B, int ld, int kb) {
  invert_lower_unit(B, ld, kb);
  invert_upper(B, ld, kb);
}

// Substitution against a 32 x 32 triangle, right-looking, a right-hand side per thread
// in x: SCALE, x <- x U^{-1} (a row); else x <- L^{-1} x (a column, unit L).  tab: row q
// of U or column q of L from the diagonal outwards (tab[q][s] = U(q, q + 1 + s) or
// L(q + 1 + s, q), 0 beyond the block) in shared memory, 16-byte aligned; rinv: the
// reciprocals of U's diagonal (SCALE).  Each final entry goes to out(q, value).  The
// entries rotate down the registers as they are updated (x[0] is the current one), in
// four groups of eight steps whose updates narrow from 31 to 7 entries: 608
// multiply-adds a thread for the 496 of the triangle, and a loop body short enough to
// stay in the instruction cache (the fully unrolled form with one scalar load per
// multiply-add took 8-12 thousand cycles a panel, bound by its shared-memory loads).
template <int W, bool SCALE, class Out>
__device__ __forceinline__ void tri_group(float (&x)[32], const float* tab, const float* rinv,
                                          const Out& out) {
#pragma unroll 1
  for (int lq = 0; lq < 8; ++lq) {
    const int q = 32 - W + lq;
    const float4* m = reinterpret_cast<const float4*>(tab + q * 32);
    const float xq = SCALE ? x[0] * rinv[q] : x[0];
    out(q, xq);
#pragma unroll
    for (int t4 = 0; t4 < W / 4; ++t4) {
      const float4 f = m[t4];
      x[4 * t4] = fmaf(-xq, f.x, x[4 * t4 + 1]);
      x[4 * t4 + 1] = fmaf(-xq, f.y, x[4 * t4 + 2]);
      x[4 * t4 + 2] = fmaf(-xq, f.z, x[4 * t4 + 3]);
      x[4 * t4 + 3] = (4 * t4 + 4 < W) ? fmaf(-xq, f.w, x[(4 * t4 + 4) & 31]) : 0.0f;
    }
  }
}
template <bool SCALE, class Out>
__device__ __forceinline__ void tri_subst(float (&x)[32], const float* tab, const float* rinv,
                                          const Out& out) {
  tri_group<32, SCALE>(x, tab, rinv, out);
  tri_group<24, SCALE>(x, tab, rinv, out);
  tri_group<16, SCALE>(x, tab, rinv, out);
  tri_group<8, SCALE>(x, tab, rinv, out);
}

cudaError_t launch_lu_large(const SolveArgs& a, cudaStream_t s);
cudaError_t launch_gj_mixed(const SolveArgs& a, cudaStream_t s);
// Kernels of the two for airfoils of at most mv unknowns.
int lu_large_launches(int mv);
int gj_launches(int mv);
long long set_wait_limit(long long polls);
size_t lu_large_min_m();

}  // namespace panel
