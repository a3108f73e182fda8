// k_solve_mixed.cu -- FP32 LU with partial pivoting + double-float iterative
// refinement for the bordered panel system (the mixed-precision path).
//
// The factor is of the rescaled matrix Mt = S_r M S_c, where S_c multiplies the
// C column and S_r the Kutta row by s = mean |A_jj| (the self-influence scale);
// this balances the border against the influence coefficients and lowers the
// condition number seen by the FP32 factor.  Refinement (Wilkinson/Moler):
//   x_0 = solve(b);  r_k = b - M x_k  with products and sums exact to ~2^-70
//   against the stored planes A_hi + A_lo;  x_{k+1} = x_k + solve(r_k), until
//   |dx|_inf <= tol |x|_inf, or until the contraction of the last two
//   corrections predicts the next one below that.  The transposed system
//   M^T lambda = g (g = dCl/du) is refined in the same kernel.
//
// The FP32 factor depends on the size m = n + 1 and the launch's choices:
//   PANEL_INVERSE, m <= kGjM (288)   explicit inverse by blocked Gauss-Jordan
//                                    (k_gj_mixed.cu); a correction is one GEMV;
//   m <= kSmemLuM (222)              k_lu_smem below: LU with the whole matrix in
//                                    shared memory (PANEL_TUNE_LU(2)), or
//                                    k_lu_global (PANEL_TUNE_LU(1)); by default
//                                    by batch and size (lu_kind_by_size);
//   m <= kLargeM (640)               k_lu_global below: one block per airfoil,
//                                    blocked right-looking LU, the trailing
//                                    matrix in the caller's LU buffer through L2;
//   m > kLargeM                      the step-synchronous blocked LU
//                                    (k_lu_large.cu, k_update_tc.cu).
// All LU variants pivot inside the current diagonal block and replace the
// 32 x 32 diagonal blocks of L and U by their inverses, so that the triangular
// solves below are sequences of matrix-vector products.  The LU buffer
// therefore holds a library-internal layout (an inverse, or an LU with
// inverted diagonal blocks: row-major up to kLargeM, above it the tiled layout
// of the blocked factor, tl_layout.cuh).
//  k_ir_mixed  one block per airfoil: the corrections with the stored factor
//    (read through L1/L2) and the refinement residuals (for m <= kFuseM one
//    pass over the matrix for both systems, else one over the rows for M u and
//    one over the columns for M^T lambda).
#include <type_traits>

#include "df.cuh"
#include "tl_layout.cuh"

namespace panel {

// ---------------------------------------------------------------------------
// LU with partial pivoting of one kb x kb diagonal block (kb <= 32) by one
// warp, register-resident: lane r holds row r (x = its 32 columns, zero beyond
// the block); rows keep their lanes and `pos` tracks their current position, so
// an exchange of positions q and p is bookkeeping plus one ipiv entry.  The
// pivot of column q is the largest |x_q| among the rows not yet pivotal, the
// lowest lane (row of the block before its exchanges) among equals.
//
// One warp walks a chain of kb dependent steps, so a step's latency is what
// counts.  The next column is brought up to date first, and its pivot searched (a
// REDUX for the magnitude, a vote for the lane; every lane takes the reciprocal of its
// own entry) between the updates of the other columns: one airfoil of 200 panels, in
// shared memory, 88 us (91 with a search of 18-bit magnitudes, the lane in the key's
// low bits, at the head of the step), of 100, through L2, 39 (40).  A REDUX more, for
// the lowest position among equals, took 96 and 43 us, a branch for it 92 and 43.
// The columns rotate down the registers as they are updated (x[0] is the current
// one), so that the step loop stays rolled with constant register indices; each
// finished entry goes to the row's own place in `blk`.  Four groups of eight steps
// narrow the update from 31 to 7 columns.
// ipiv[q] receives base + the position of column q's pivot row.  On return `fz`
// is 0, or q + 1 for the first exactly zero (or NaN) pivot column q, after which
// the block's contents have no meaning.
// ---------------------------------------------------------------------------
// 1 / a by one Newton-Raphson step on the hardware approximation: the correctly
// rounded reciprocal for every |a| below 2^126, infinite ones included (compared with
// __frcp_rn on all of them; beyond, where it is subnormal, 5 magnitudes differ in the
// last bit).
__device__ __forceinline__ float rcp_newton(float a) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(a));
  const float v = fmaf(r, fmaf(-a, r, 1.0f), r);
  return v == v ? v : r;
}

// The pivot of a column, x the lane's entry: largest() and vote(), apart (a warp keeps
// the order of such operations, and the second waits for the first).
struct PivotSearch {
  unsigned key, mx;  // the lane's magnitude (0: no candidate), the largest
  int lane;
  float rcp;         // of the lane's own entry
  __device__ __forceinline__ void largest(float x, bool done) {
    key = (!done && x == x) ? __float_as_uint(x) & 0x7fffffffu : 0u;
    mx = __reduce_max_sync(0xffffffffu, key);
    rcp = rcp_newton(x);
  }
  __device__ __forceinline__ void vote() {
    lane = __ffs(__ballot_sync(0xffffffffu, key == mx)) - 1;
  }
};

template <int W, class Blk>
__device__ __forceinline__ void warp_block_lu_group(float (&x)[32], const Blk& blk, int& pos,
                                                    bool& done, int& fz, int kb, int* ipiv,
                                                    int base, PivotSearch& s) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int lq = 0; lq < 8; ++lq) {
    const int q = 32 - W + lq;
    const int pl = s.lane;
    const bool ok = s.mx != 0u;  // a nonzero pivot
    const float l = x[0] * __shfl_sync(0xffffffffu, s.rcp, pl);
    const bool elim = ok && !done && lane != pl;
    const float le = elim ? l : 0.0f;
    if (lane < kb && q < kb) blk(lane, q) = elim ? l : x[0];
    if (ok && lane == pl) done = true;
    x[0] = fmaf(-le, __shfl_sync(0xffffffffu, x[1], pl), x[1]);
    s.largest(x[0], done);
#pragma unroll
    for (int t = 2; t < W; ++t) {
      x[t - 1] = fmaf(-le, __shfl_sync(0xffffffffu, x[t], pl), x[t]);
      if (t == (W < 16 ? W - 2 : 14)) s.vote();
    }
    x[W - 1] = 0.0f;
    // bookkeeping, off the chain
    const int pm = __shfl_sync(0xffffffffu, pos, pl);
    if (ok) {
      if (lane == 0) ipiv[q] = base + pm;
      if (pos == q) pos = pm;
      if (lane == pl) pos = q;
    } else if (q < kb && fz == 0) {
      fz = q + 1;
    }
  }
}

template <class Blk>
__device__ __forceinline__ void warp_block_lu(float (&x)[32], const Blk& blk, int& pos, bool& done,
                                              int& fz, int kb, int* ipiv, int base) {
  PivotSearch s;
  s.largest(x[0], done);
  s.vote();
  warp_block_lu_group<32>(x, blk, pos, done, fz, kb, ipiv, base, s);
  if (kb > 8) warp_block_lu_group<24>(x, blk, pos, done, fz, kb, ipiv, base, s);
  if (kb > 16) warp_block_lu_group<16>(x, blk, pos, done, fz, kb, ipiv, base, s);
  if (kb > 24) warp_block_lu_group<8>(x, blk, pos, done, fz, kb, ipiv, base, s);
}

// ---------------------------------------------------------------------------
// The factored diagonal block as the other steps of a panel read it, in shared
// memory: row q of U and column q of L from the diagonal outwards (u[q][s] =
// U(q, q + 1 + s), l[q][s] = L(q + 1 + s, q), 0 beyond the block) and the
// reciprocals of U's diagonal.  A substitution step then reads its 31
// multipliers as eight broadcast vector loads at the same register indices in
// every step, so that the step loop stays rolled.
// ---------------------------------------------------------------------------
struct alignas(16) DiagTab {
  float u[32 * 32];
  float l[32 * 32];
  float rinv[32];
  int bperm[32];  // final row q of the block = row bperm[q] before its exchanges
  int fz;         // 0, or the first zero pivot column + 1
  int moved;      // some row of the block was exchanged
  int pad[2];
};

// LU of the kb x kb diagonal block by the calling warp into the table; blk(r, t)
// are the block's entries, overwritten.  The pivots go to ipiv[0 .. kb) (+ base).
template <class Blk>
__device__ __forceinline__ void diag_lu(const Blk& blk, int kb, int* ipiv, int base, DiagTab& d) {
  const int lane = threadIdx.x & 31;
  float x[32];
#pragma unroll
  for (int t = 0; t < 32; ++t) x[t] = (lane < kb && t < kb) ? blk(lane, t) : 0.0f;
  int pos = lane;
  bool done = lane >= kb;  // already a pivot row (or outside the block)
  int fz = 0;
  warp_block_lu(x, blk, pos, done, fz, kb, ipiv, base);
  // the lane's row sits at `pos` of the block (rows beyond kb: zero, unit pivot)
  float* ur = d.u + pos * 31 - 1;  // U(pos, t) at ur + pos + t
  float* lc = d.l + pos - 1;       // L(pos, t) at lc + 31 t
#pragma unroll 4
  for (int t = 0; t < 32; ++t) {
    const float v = (lane < kb && t < kb) ? blk(lane, t) : 0.0f;
    if (t != pos) *(t > pos ? ur + t : lc + 31 * t) = v;
  }
  const float dia = lane < kb ? blk(lane, pos) : 1.0f;
  d.rinv[pos] = 1.0f / dia;
  d.bperm[pos] = lane;
  const bool moved = __any_sync(0xffffffffu, pos != lane);
  if (lane == 0) {
    d.fz = fz;
    d.moved = moved ? 1 : 0;
  }
}

// The entries beyond the block's triangles, once per kernel (all threads).
__device__ __forceinline__ void diag_tab_init(DiagTab& d) {
  for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x)
    if ((e & 31) >= 31 - (e >> 5)) d.u[e] = d.l[e] = 0.0f;
}

template <bool SCALE, class Out>
__device__ __forceinline__ void tri_subst(float (&x)[32], const DiagTab& d, const Out& out) {
  tri_subst<SCALE>(x, SCALE ? d.u : d.l, d.rinv, out);
}

// ---------------------------------------------------------------------------
// The LU kernel, factor in global memory (kSmemLuM < m <= kLargeM, or every
// m <= kLargeM with PANEL_TUNE_LU(1)): blocked right-looking with the current
// panel of 32 columns staged in shared memory, transposed (panel column q at
// PT[q ldt + row]: the update reads eight rows' multipliers with two broadcast
// vector loads), the row exchanges, U12 and the rank-32 update applied to the
// factor in the caller's LU buffer through L2.  Shared memory stays small (the
// panel plus a 128-column slab of U12), so several airfoils share an SM and
// hide each other's latencies.  A step has two phases:
//   A  a warp per 32 rows: the panel's tile in, L21, and out to the factor; a
//      warp per 32 columns: U12, the first slab of it kept for the update; the
//      inverses of the diagonal block's triangles; the exchanges to the left;
//   B  warp 0 updates the next diagonal block and factors it (look-ahead) while
//      the others update everything else.
// The first step reads the hi plane and writes the factor.  What bounded the
// kernel were its chains of L2 and DRAM round trips, not the products: a copy of
// the plane ahead of the first step, one load after the other, was 27-30 % of its
// time, the unhidden diagonal blocks 28 % (201 unknowns) to 8 % (601), and moving
// the panel between barriers of its own another 8-15 %.
// ---------------------------------------------------------------------------
constexpr int kSlabW = 128;  // columns of U12 staged at a time

// What a step reads the trailing matrix from: the factor, or (first step) the hi
// plane, whose border the reader then scales by sf (after all of its loads: a
// choice per load waits for each).
struct LuSource {
  const float* p;
  int m;
  float sf;
  bool first;
  __device__ __forceinline__ float operator()(int r, int c) const { return p[r * m + c]; }
  __device__ __forceinline__ void scale(float& v, int r, int c) const {
    if (r == m - 1 || c == m - 1) v *= sf;
  }
};

// (d.x, d.y) + a (b, b), each rounded once.
__device__ __forceinline__ void fma2(float2& d, float ax, float ay, float b) {
  asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %4};\n\t"
      "mov.b64 d, {%0, %1};\n\tfma.rn.f32x2 d, a, b, d;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "+f"(d.x), "+f"(d.y)
      : "f"(ax), "f"(ay), "f"(b));
}

// A22 -= L21 U12 over the columns [cc, cc + 32 J) of the staged slab of -U12: the w-th
// of nw warps takes the 8-row tiles w, w + nw, ...; lane l the columns cc + l + 32 j.
// lt: row k1 of the transposed panel.  The next diagonal block (rows and columns
// below k2) is warp 0's.
template <int J>
__device__ __forceinline__ void update_tiles(const LuSource& S, float* F,
                                             const float* __restrict__ lt, int ldt,
                                             const float* __restrict__ U, int k1, int k2, int cc,
                                             int nrt, int w, int nw) {
  constexpr int R = 8;
  const int lane = threadIdx.x & 31, m = S.m;
  for (int rt = w; rt < nrt; rt += nw) {
    const int r0 = k1 + R * rt;
    float2 acc[R / 2][J];
#pragma unroll
    for (int aa = 0; aa < R; ++aa)
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const int r = r0 + aa, c = cc + lane + 32 * j;
        const float v = (r < m && c < m) ? S(r, c) : 0.0f;
        if (aa & 1)
          acc[aa / 2][j].y = v;
        else
          acc[aa / 2][j].x = v;
      }
    if (S.first)
#pragma unroll
      for (int aa = 0; aa < R; ++aa)
#pragma unroll
        for (int j = 0; j < J; ++j)
          S.scale((aa & 1) ? acc[aa / 2][j].y : acc[aa / 2][j].x, r0 + aa, cc + lane + 32 * j);
    const float* l0 = lt + R * rt;
#pragma unroll 2
    for (int q = 0; q < 32; ++q) {
      float uv[J];
#pragma unroll
      for (int j = 0; j < J; ++j) uv[j] = U[q * kSlabW + lane + 32 * j];
#pragma unroll
      for (int a4 = 0; a4 < R / 4; ++a4) {
        const float4 l = *reinterpret_cast<const float4*>(l0 + q * ldt + 4 * a4);
#pragma unroll
        for (int j = 0; j < J; ++j) {
          fma2(acc[2 * a4][j], l.x, l.y, uv[j]);
          fma2(acc[2 * a4 + 1][j], l.z, l.w, uv[j]);
        }
      }
    }
    const int c0 = r0 < k2 ? k2 : 0;
#pragma unroll
    for (int aa = 0; aa < R; ++aa)
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const int r = r0 + aa, c = cc + lane + 32 * j;
        if (r < m && c < m && c >= c0) F[r * m + c] = (aa & 1) ? acc[aa / 2][j].y : acc[aa / 2][j].x;
      }
  }
}

// Row stride of the transposed panel: the rows below the first block, padded to
// whole 8-row tiles and to whole 32-row tiles of phase A, and 4 mod 32, so that 4
// rows x 8 columns moved by a warp touch all banks.
__host__ __device__ constexpr int lu_panel_ld(int m) {
  return (((m > 32 ? m - 32 : 1) + 31) & ~31) + 4;
}

// Barriers of k_lu_global's phase B: the seven updating warps among themselves, and
// (arrive / sync) warp 0's last read of the first slab.
__device__ __forceinline__ void lu_update_sync() {
  asm volatile("bar.sync 1, %0;\n" ::"n"(kThreads - 32) : "memory");
}
__device__ __forceinline__ void lu_slab_read() {
  asm volatile("bar.arrive 2, %0;\n" ::"n"(kThreads) : "memory");
}
__device__ __forceinline__ void lu_slab_wait() {
  asm volatile("bar.sync 2, %0;\n" ::"n"(kThreads) : "memory");
}

template <int MINB>
__global__ void __launch_bounds__(kThreads, MINB) k_lu_global(SolveArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int NB = 32;
  const Batch& bt = a.bt;
  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b);
  const int m = n + 1;
  if (a.info[b] != 0) return;
  if (m <= kGjM && a.inverse) return;  // taken by k_gj_mixed
  if (n > a.n_cap) {
    if (threadIdx.x == 0) a.info[b] = PANEL_INFO_TOO_LARGE;
    return;
  }
  if (m > kLargeM) return;  // taken by the blocked factor (k_lu_large.cu)
  if (m <= kSmemLuM && a.lu_kind != 1) return;  // taken by k_lu_smem
  const int mv = bt.n_max + 1;
  DiagTab& dt = *reinterpret_cast<DiagTab*>(smraw);
  float* U = reinterpret_cast<float*>(smraw + sizeof(DiagTab));  // NB x kSlabW slab of U12
  double* red = reinterpret_cast<double*>(U + NB * kSlabW);      // 32
  float* PT = reinterpret_cast<float*>(red + 32);                // NB x ldt panel, transposed
  const int ldt = lu_panel_ld(mv);
  float* D = PT + NB * ldt;                                      // NB x 33 diagonal block
  int* ipiv = reinterpret_cast<int*>(D + NB * 33);               // mv

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t moff = bt.mat_off[b];
  const float* Ah = a.A_hi + moff;
  float* F = a.LU + moff;
  diag_tab_init(dt);
  LuSource S{Ah, m, (float)border_scale(Ah, n, m, red), true};
  auto diag = [&](int k, int kb) {
    diag_lu([&](int r, int t) -> float& { return D[r * 33 + t]; }, kb, ipiv + k, k, dt);
  };
  if (warp == 0) {
    const int kb = min(NB, m);
#pragma unroll
    for (int r = 0; r < NB; ++r)
      if (r < kb && lane < kb) D[r * 33 + lane] = S(r, lane);
    if (m <= NB && lane < m) {  // the block holds the border
      D[n * 33 + lane] *= S.sf;
      if (lane < n) D[lane * 33 + n] *= S.sf;
    }
    __syncwarp();
    diag(0, kb);
  }
  __syncthreads();

  const int pc = lane & 7, pr = lane >> 3;  // panel moves: 8 columns x 4 rows per warp
  for (int k0 = 0;; k0 += NB) {
    if (dt.fz != 0) {
      if (tid == 0) {
        a.info[b] = k0 + dt.fz;
        if (a.iters) a.iters[b] = 0;
      }
      return;
    }
    const int kb = min(NB, m - k0);
    const int k1 = k0 + kb;
    // ---- A: L21 = A21 U11^{-1}, a row per thread, in place in PT; U12 = L11^{-1}
    // A12, a column per thread, the rows read through the block's exchanges; and
    // the two inverses of the diagonal block the refinement takes, U11^{-1} as 32
    // more rows (of the identity) and L11^{-1} as 32 more columns.  A warp takes
    // 32 rows or columns (rows below the block only beside a full block) ----
    const int nw = (m - k1 + 31) >> 5;
    for (int w = warp; w < 2 * nw + 2; w += kWarps) {
      float x[32];
      if (w == 0) {
#pragma unroll
        for (int t = 0; t < 32; ++t) x[t] = (t == lane) ? 1.0f : 0.0f;
        float* G = F + (k0 + lane) * m + k0;
        tri_subst<true>(x, dt, [&](int q, float v) {
          if (lane < kb && q < kb && q >= lane) G[q] = v;
        });
      } else if (w == 1) {
#pragma unroll
        for (int t = 0; t < 32; ++t) x[t] = (t == lane) ? 1.0f : 0.0f;
        float* G = F + k0 * m + k0 + lane;
        tri_subst<false>(x, dt, [&](int q, float v) {
          if (q < kb && q > lane) G[q * m] = v;
        });
      } else if (w < 2 + nw) {
        // the tile in, 32 loads a lane in flight, through the warp's own part of PT
        const int rw = 32 * (w - 2);
        float* T = PT + rw;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const int r = 4 * (i >> 2) + pr, t = 8 * (i & 3) + pc;
          x[i] = (k1 + rw + r < m) ? S(k1 + rw + r, k0 + t) : 0.0f;
        }
        if (S.first)
#pragma unroll
          for (int i = 0; i < 32; ++i)
            S.scale(x[i], k1 + rw + 4 * (i >> 2) + pr, k0 + 8 * (i & 3) + pc);
#pragma unroll
        for (int i = 0; i < 32; ++i) T[(8 * (i & 3) + pc) * ldt + 4 * (i >> 2) + pr] = x[i];
        __syncwarp();
#pragma unroll
        for (int t = 0; t < 32; ++t) x[t] = T[t * ldt + lane];
        tri_subst<true>(x, dt, [&](int q, float v) { T[q * ldt + lane] = v; });
        __syncwarp();
        float* G = F + (k1 + rw) * m + k0;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const int r = 4 * (i >> 2) + pr, t = 8 * (i & 3) + pc;
          if (k1 + rw + r < m) G[r * m + t] = T[t * ldt + r];
        }
      } else {
        const int cu = 32 * (w - 2 - nw) + lane, c = k1 + cu;
        const bool ok = c < m, slab = cu < kSlabW;
#pragma unroll
        for (int t = 0; t < 32; ++t) x[t] = ok ? S(k0 + dt.bperm[t], c) : 0.0f;
        if (S.first && c == n)  // (the block's rows are not the last one)
#pragma unroll
          for (int t = 0; t < 32; ++t) x[t] *= S.sf;
        float* G = F + k0 * m + c;
        tri_subst<false>(x, dt, [&](int q, float v) {
          if (ok) G[q * m] = v;
          if (slab) U[q * kSlabW + cu] = -v;
        });
      }
    }
    // the exchanges of this block's rows on the columns left of it: composed
    // into bperm, all loads of a column in flight at once
    if (dt.moved)
      for (int c = tid; c < k0; c += kThreads) {
        float v[NB];
#pragma unroll
        for (int q = 0; q < NB; ++q) v[q] = (q < kb) ? F[(k0 + dt.bperm[q]) * m + c] : 0.0f;
#pragma unroll
        for (int q = 0; q < NB; ++q)
          if (q < kb) F[(k0 + q) * m + c] = v[q];
      }
    __syncthreads();
    if (k1 >= m) break;
    // ---- B: A22 -= L21 U12, 128-column slabs of U12 staged in shared memory (the
    // first one is there) ----
    const int k2 = min(k1 + NB, m);
    if (warp == 0) {
      const int kb2 = k2 - k1;
      float x[32];
#pragma unroll
      for (int r = 0; r < NB; ++r) x[r] = (r < kb2 && lane < kb2) ? S(k1 + r, k1 + lane) : 0.0f;
      if (S.first)
#pragma unroll
        for (int r = 0; r < NB; ++r) S.scale(x[r], k1 + r, k1 + lane);
#pragma unroll 2
      for (int q = 0; q < NB; ++q) {
        const float uq = U[q * kSlabW + lane];
#pragma unroll
        for (int r4 = 0; r4 < 8; ++r4) {
          const float4 l = *reinterpret_cast<const float4*>(PT + q * ldt + 4 * r4);
          x[4 * r4] = fmaf(l.x, uq, x[4 * r4]);
          x[4 * r4 + 1] = fmaf(l.y, uq, x[4 * r4 + 1]);
          x[4 * r4 + 2] = fmaf(l.z, uq, x[4 * r4 + 2]);
          x[4 * r4 + 3] = fmaf(l.w, uq, x[4 * r4 + 3]);
        }
      }
      lu_slab_read();
#pragma unroll
      for (int r = 0; r < NB; ++r) D[r * 33 + lane] = x[r];
      __syncwarp();
      diag(k1, kb2);
    } else {
      const int nrt = k2 < m ? (m - k1 + 7) >> 3 : 0;
      for (int cc = k1; cc < m; cc += kSlabW) {
        if (cc > k1) {
          for (int t = warp - 1; t < NB; t += kWarps - 1)
#pragma unroll
            for (int j = 0; j < kSlabW / 32; ++j) {
              const int c = cc + lane + 32 * j;
              U[t * kSlabW + lane + 32 * j] = (c < m) ? -F[(k0 + t) * m + c] : 0.0f;
            }
          lu_update_sync();
        }
        // register tiles 8 rows x 32 J columns, J = 1..4 by the width of the slab
        const int J = min(kSlabW / 32, (m - cc + 31) >> 5);
        if (J == 4)
          update_tiles<4>(S, F, PT, ldt, U, k1, k2, cc, nrt, warp - 1, kWarps - 1);
        else if (J == 3)
          update_tiles<3>(S, F, PT, ldt, U, k1, k2, cc, nrt, warp - 1, kWarps - 1);
        else if (J == 2)
          update_tiles<2>(S, F, PT, ldt, U, k1, k2, cc, nrt, warp - 1, kWarps - 1);
        else
          update_tiles<1>(S, F, PT, ldt, U, k1, k2, cc, nrt, warp - 1, kWarps - 1);
        if (cc == k1)
          lu_slab_wait();
        else
          lu_update_sync();
      }
    }
    S.p = F;
    S.first = false;
    __syncthreads();
  }
  int32_t* gpiv = a.piv + vec_off(bt, b);
  for (int k = tid; k < m; k += kThreads) gpiv[k] = ipiv[k];
}

// ---------------------------------------------------------------------------
// The LU kernel with the whole matrix in shared memory (3 <= m <= kSmemLuM):
// one block of NT threads per airfoil.  The algorithm, its operations and their
// order are those of k_lu_global, so the two kernels store the same factor bit
// for bit.  Here every step works on the scaled matrix staged once in shared
// memory (odd row stride: conflict-free columns) and the factor goes to the
// caller's buffer once: one read of the hi plane and one write of the factor
// per airfoil.  One (m > 160 or so) or a few airfoils have the SM to themselves,
// so the steps are arranged to keep the warps busy:
//   A  the first half of the threads: L21, a row each, also kept transposed in
//      LT so that the update reads eight rows' multipliers with two broadcast
//      vector loads, and the rows of U11^{-1}; the second half: U12, a column
//      each, and the columns of L11^{-1}; the inverses replace the block;
//   B  the update of the next panel's 32 columns;
//   C  warp 0 factors the next diagonal block (look-ahead) while the others
//      update the remaining columns.
// ---------------------------------------------------------------------------
// A22 -= L21 U12 on rows [r0, r0 + 8) x columns cc + lane + 32 j (j < J): the
// multipliers of the 8 rows from LT (panel column q at LT[q ldt + r - k1]),
// U12 from the matrix rows k0..k0 + 32.
template <int J>
__device__ __forceinline__ void smem_update_tile(float* __restrict__ F, int ld,
                                                 const float* __restrict__ LT, int ldt, int m,
                                                 int k0, int k1, int r0, int cc) {
  const int lane = threadIdx.x & 31;
  float acc[8][J];
#pragma unroll
  for (int aa = 0; aa < 8; ++aa)
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int r = r0 + aa, c = cc + lane + 32 * j;
      acc[aa][j] = (r < m && c < m) ? F[r * ld + c] : 0.0f;
    }
  const float* lt = LT + (r0 - k1);
#pragma unroll 4
  for (int q = 0; q < 32; ++q) {
    const float4 la = *reinterpret_cast<const float4*>(lt + q * ldt);
    const float4 lb = *reinterpret_cast<const float4*>(lt + q * ldt + 4);
    const float lv[8] = {la.x, la.y, la.z, la.w, lb.x, lb.y, lb.z, lb.w};
    float uv[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int c = cc + lane + 32 * j;
      uv[j] = (c < m) ? F[(k0 + q) * ld + c] : 0.0f;
    }
#pragma unroll
    for (int aa = 0; aa < 8; ++aa)
#pragma unroll
      for (int j = 0; j < J; ++j) acc[aa][j] = fmaf(-lv[aa], uv[j], acc[aa][j]);
  }
#pragma unroll
  for (int aa = 0; aa < 8; ++aa)
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int r = r0 + aa, c = cc + lane + 32 * j;
      if (r < m && c < m) F[r * ld + c] = acc[aa][j];
    }
}

// Update tasks of 8 rows x 32 J columns over the columns [c0, c1) of the rows
// [k1, m), shared by the calling warps: the w-th of nw.
__device__ __forceinline__ void smem_update(float* F, int ld, const float* LT, int ldt, int m,
                                            int k0, int k1, int c0, int c1, int w, int nw,
                                            int cw) {
  if (c1 <= c0) return;
  const int nrt = (m - k1 + 7) >> 3, ncs = (c1 - c0 + cw - 1) / cw;
  for (int task = w; task < nrt * ncs; task += nw) {
    const int r0 = k1 + 8 * (task / ncs), cc = c0 + cw * (task % ncs);
    const int J = min(cw / 32, (min(c1, m) - cc + 31) >> 5);
    if (J >= 4)
      smem_update_tile<4>(F, ld, LT, ldt, m, k0, k1, r0, cc);
    else if (J == 3)
      smem_update_tile<3>(F, ld, LT, ldt, m, k0, k1, r0, cc);
    else if (J == 2)
      smem_update_tile<2>(F, ld, LT, ldt, m, k0, k1, r0, cc);
    else
      smem_update_tile<1>(F, ld, LT, ldt, m, k0, k1, r0, cc);
  }
}

// Row stride of the transposed panel: the rows below the first block, in whole
// 8-row tiles.
__host__ __device__ constexpr int lu_smem_ldt(int m) { return m > 32 ? (m - 32 + 7) & ~7 : 8; }

template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_lu_smem(SolveArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int NB = 32, NW = NT / 32;
  const Batch& bt = a.bt;
  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b);
  const int m = n + 1;
  if (a.info[b] != 0) return;
  if (m <= kGjM && a.inverse) return;  // taken by k_gj_mixed
  if (n > a.n_cap) {
    if (threadIdx.x == 0) a.info[b] = PANEL_INFO_TOO_LARGE;
    return;
  }
  if (m > kSmemLuM || a.lu_kind == 1) return;  // taken by k_lu_global or the blocked factor
  const int ld = m | 1;
  const int mv = bt.n_max + 1;
  const int ldt = lu_smem_ldt(mv);
  DiagTab& dt = *reinterpret_cast<DiagTab*>(smraw);
  double* red = reinterpret_cast<double*>(smraw + sizeof(DiagTab));  // 32
  float* LT = reinterpret_cast<float*>(red + 32);                    // NB x ldt
  int* ipiv = reinterpret_cast<int*>(LT + NB * ldt);                 // mv
  float* F = reinterpret_cast<float*>(ipiv + mv);                    // m x ld

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t moff = bt.mat_off[b];
  const float* Ah = a.A_hi + moff;
  // the hi plane in by asynchronous copies (every element of the thread in
  // flight at once; rows of stride m are only 4-byte aligned), a warp per row
  for (int rr = warp; rr < m; rr += NW)
    for (int cc = lane; cc < m; cc += 32) {
      const unsigned dst = (unsigned)__cvta_generic_to_shared(F + rr * ld + cc);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(Ah + rr * m + cc)
                   : "memory");
    }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  diag_tab_init(dt);
  const float sf = (float)border_scale(Ah, n, m, red);
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  // the C column and the Kutta row scaled by sf
  for (int k = tid; k < m; k += NT) {
    F[n * ld + k] *= sf;
    if (k < n) F[k * ld + n] *= sf;
  }
  __syncthreads();
  auto diag = [&](int k, int kb) {
    float* P = F + k * ld + k;
    diag_lu([&](int r, int t) -> float& { return P[r * ld + t]; }, kb, ipiv + k, k, dt);
  };
  if (warp == 0) diag(0, min(NB, m));
  __syncthreads();

  for (int k0 = 0;; k0 += NB) {
    if (dt.fz != 0) {
      if (tid == 0) {
        a.info[b] = k0 + dt.fz;
        if (a.iters) a.iters[b] = 0;
      }
      return;
    }
    const int kb = min(NB, m - k0);
    const int k1 = k0 + kb;
    const int nw = (m - k1 + 31) >> 5;
    // ---- A ---- (the warps of either half take 32 rows / columns each)
    if (warp < NW / 2) {
      for (int w = warp; w < nw + 1; w += NW / 2) {
        float x[32];
        if (w == 0) {
#pragma unroll
          for (int t = 0; t < 32; ++t) x[t] = (t == lane) ? 1.0f : 0.0f;
          float* G = F + (k0 + lane) * ld + k0;
          tri_subst<true>(x, dt, [&](int q, float v) {
            if (lane < kb && q < kb && q >= lane) G[q] = v;
          });
        } else {
          const int r = k1 + 32 * (w - 1) + lane;
          const bool ok = r < m;
          float* G = F + (ok ? r : k0) * ld + k0;
          float* T = LT + (r - k1);
#pragma unroll
          for (int t = 0; t < 32; ++t) x[t] = ok ? G[t] : 0.0f;
          tri_subst<true>(x, dt, [&](int q, float v) {
            if (ok) {
              G[q] = v;
              T[q * ldt] = v;
            }
          });
        }
      }
    } else {
      for (int w = warp - NW / 2; w < nw + 1; w += NW / 2) {
        float x[32];
        if (w == 0) {
#pragma unroll
          for (int t = 0; t < 32; ++t) x[t] = (t == lane) ? 1.0f : 0.0f;
          float* G = F + k0 * ld + k0 + lane;
          tri_subst<false>(x, dt, [&](int q, float v) {
            if (q < kb && q > lane) G[q * ld] = v;
          });
        } else {
          const int c = k1 + 32 * (w - 1) + lane;
          const bool ok = c < m;
          float* G = F + k0 * ld + (ok ? c : k0);
#pragma unroll
          for (int t = 0; t < 32; ++t) x[t] = ok ? G[dt.bperm[t] * ld] : 0.0f;
          tri_subst<false>(x, dt, [&](int q, float v) {
            if (ok) G[q * ld] = v;
          });
        }
      }
    }
    // the exchanges on the columns left of the panel
    if (dt.moved)
      for (int c = tid; c < k0; c += NT) {
        float v[NB];
#pragma unroll
        for (int q = 0; q < NB; ++q) v[q] = (q < kb) ? F[(k0 + dt.bperm[q]) * ld + c] : 0.0f;
#pragma unroll
        for (int q = 0; q < NB; ++q)
          if (q < kb) F[(k0 + q) * ld + c] = v[q];
      }
    __syncthreads();
    if (k1 >= m) break;
    const int kb2 = min(NB, m - k1);
    // ---- B: the next panel's columns [k1, k1 + kb2) ----
    smem_update(F, ld, LT, ldt, m, k0, k1, k1, k1 + kb2, warp, NW, 32);
    __syncthreads();
    // ---- C: the next diagonal block (warp 0) | the remaining columns ----
    // (warp 0 has its scheduler to itself: every fourth warp stays out)
    if (warp == 0)
      diag(k1, kb2);
    else if (warp & 3)
      smem_update(F, ld, LT, ldt, m, k0, k1, k1 + kb2, m, warp - 1 - (warp >> 2), 3 * NW / 4, 128);
    __syncthreads();
  }
  float* G = a.LU + moff;
  for (int rr = warp; rr < m; rr += NW)
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int cc = lane + 32 * u;
      if (cc < m) G[rr * m + cc] = F[rr * ld + cc];
    }
  int32_t* gpiv = a.piv + vec_off(bt, b);
  for (int k = tid; k < m; k += NT) gpiv[k] = ipiv[k];
}
static_assert(kSmemLuM <= 256, "k_lu_smem writes rows of at most 8 x 32 columns");

static size_t lu_smem_smem(int n_max) {
  const size_t mv = (size_t)n_max + 1, ldv = mv | 1;
  return sizeof(DiagTab) + 32 * 8 + 32 * (size_t)lu_smem_ldt((int)mv) * 4 + mv * 4 + mv * ldv * 4;
}

static size_t lu_global_smem(int n_max) {
  const size_t mv = (size_t)n_max + 1;
  return sizeof(DiagTab) + 32 * (size_t)kSlabW * 4 + 32 * 8 +
         32 * (size_t)lu_panel_ld((int)mv) * 4 + 32 * 33 * 4 + mv * 4;
}

// ---------------------------------------------------------------------------
// Triangular solves with the stored factor (global memory, the 32 x 32
// diagonal blocks inverted) on float vectors in shared memory: the forward
// system y <- U^{-1} L^{-1} y and the transposed system z <- L^{-T} U^{-T} z,
// one of them or both at once.  Both go over the 32-row groups of the factor
// top-down (L, U^T) and then bottom-up (U, L^T), two block barriers per group:
//   phase A  forward: t_i = y_i - (row i of L or U outside the group) . y, a
//            few rows per warp, lanes along the rows (left-looking, coalesced);
//            transposed: the previous group's columns of U^T (rows of U), or
//            of L^T, applied to the rest of z, a thread per column
//            (right-looking, coalesced across the threads); the group's own
//            entries go to its scratch (32 floats of 64) instead of z;
//   phase B  the group's diagonal block: y_i = sum X_iq t_q, z_i = sum X_qi t_q
//            (a few rows / columns per warp).
// Solving both systems, every warp takes its share of both in each phase (the
// two share the barriers, and a warp done with its forward rows goes on to its
// transposed columns while others are still loading); each system's
// arithmetic is the same as when it is solved alone.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums over the lanes of R values per lane (R = 1, 2, 4, 8): log2 R halving exchanges
// (each lane keeps half of the values and adds the partner's copies of them), then
// butterflies; the total of value r is in the lanes l with l / (32 / R) == r.  R = 8
// takes 9 shuffles instead of 40.
template <int R>
__device__ __forceinline__ float lane_sums(float (&v)[R], int lane) {
  int o = 16;
#pragma unroll
  for (int h = R / 2; h >= 1; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int r = 0; r < h; ++r) {
      const float keep = up ? v[r + h] : v[r], send = up ? v[r] : v[r + h];
      v[r] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  float s = v[0];
#pragma unroll
  for (int k = 16 / R; k >= 1; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
  return s;
}

// acc[r] += sum over the chunks c in [c0, c1) of p[r rs + c cs] y[32 c] for R rows (p and
// y already offset by the lane): per chunk R loads, one shared read of y, R
// multiply-adds; U chunks' loads in flight.
template <int R, int U>
__device__ __forceinline__ void rows_dot(float (&acc)[R], const float* __restrict__ p, int rs,
                                         int cs, const float* y, int c0, int c1) {
  int c = c0;
  for (; c + U <= c1; c += U) {
    float v[U][R];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) v[u][r] = __ldg(p + (c + u) * cs + r * rs);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float yy = y[32 * (c + u)];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = fmaf(v[u][r], yy, acc[r]);
    }
  }
  if (U > 1)
    for (; c < c1; ++c) {
      const float yy = y[32 * c];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = fmaf(__ldg(p + c * cs + r * rs), yy, acc[r]);
    }
}

// The same over the columns [c0, c1) of R rows stored row-major (stride m, from F):
// full chunks, then one masked chunk.
template <int R, int U>
__device__ __forceinline__ void rows_dot_range(float (&acc)[R], const float* __restrict__ F, int m,
                                               const float* y, int c0, int c1, int lane) {
  const int full = (c1 - c0) >> 5;
  rows_dot<R, U>(acc, F + c0 + lane, m, 32, y + c0 + lane, 0, full);
  const int c = c0 + 32 * full + lane;
  if (c < c1) {
    const float yy = y[c];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = fmaf(__ldg(F + c + r * m), yy, acc[r]);
  }
}

// z -= the 32 (or kb) rows p, p + step, .. of a group, times the group's values g
// (16-byte aligned), for one column.
template <int U>
__device__ __forceinline__ float column_update(const float* __restrict__ p, int step, int kb,
                                               const float* g, float acc) {
  if (kb == 32) {
#pragma unroll 1
    for (int t = 0; t < 32; t += U) {
      float v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = __ldg(p + (t + u) * step);
#pragma unroll
      for (int u = 0; u < U; u += 4) {
        const float4 q = *reinterpret_cast<const float4*>(g + t + u);
        acc = fmaf(-v[u], q.x, acc);
        acc = fmaf(-v[u + 1], q.y, acc);
        acc = fmaf(-v[u + 2], q.z, acc);
        acc = fmaf(-v[u + 3], q.w, acc);
      }
    }
  } else {
    for (int t = 0; t < kb; ++t) acc = fmaf(-__ldg(p + t * step), g[t], acc);
  }
  return acc;
}

// The factor of an airfoil of at most kLargeM - 1 panels: row-major, ld m,
// groups of 32 rows from row 0.
struct RmFactor {
  const float* F;
  int m;
  __device__ int groups() const { return (m + 31) >> 5; }
  __device__ int k0(int d) const { return 32 * d; }
  __device__ int kb(int d) const { return min(32, m - 32 * d); }
  // lane shares of rows i .. i + R - 1 (of group d) . y over the columns before /
  // after the group; i + R - 1 may run past the group's (and the matrix's) last row:
  // the caller asks for existing rows only (R full rows, or one at a time)
  template <int R, int U>
  __device__ void dot_left(float (&acc)[R], int i, int d, const float* y, int lane) const {
    rows_dot<R, U>(acc, F + i * m + lane, m, 32, y + lane, 0, d);
  }
  template <int R, int U>
  __device__ void dot_right(float (&acc)[R], int i, int d, const float* y, int lane) const {
    rows_dot_range<R, U>(acc, F + i * m, m, y, 32 * d + kb(d), m, lane);
  }
  // row i's entries in the columns of group d, and the distance between rows
  __device__ const float* diag_row(int d, int i) const { return F + (int64_t)i * m + 32 * d; }
  __device__ int diag_step(int) const { return m; }
  // z_r -= sum_t M[k0 + t][r] g_t (group d's rows, its values g) for the columns r
  // after group d; those of group d + 1 go to nx.  Thread tid of nth.
  template <int U>
  __device__ void update_right(int d, float* z, const float* g, float* nx, int tid, int nth) const {
    const int k0 = 32 * d, kb = this->kb(d), c0 = k0 + kb;
    for (int r = c0 + tid; r < m; r += nth) {
      const float acc = column_update<U>(F + k0 * m + r, m, kb, g, z[r]);
      if (r < c0 + 32)
        nx[r - c0] = acc;
      else
        z[r] = acc;
    }
  }
  // the same for the columns before group d; those of group d - 1 go to nx
  template <int U>
  __device__ void update_left(int d, float* z, const float* g, float* nx, int tid, int nth) const {
    const int k0 = 32 * d, kb = this->kb(d);
    for (int r = tid; r < k0; r += nth) {
      const float acc = column_update<U>(F + k0 * m + r, m, kb, g, z[r]);
      if (r >= k0 - 32)
        nx[r - (k0 - 32)] = acc;
      else
        z[r] = acc;
    }
  }
};

// The factor of an airfoil of more than kLargeM - 1 panels, in the layout the
// blocked LU (k_lu_large.cu) leaves: the tiled layout of tl_layout.cuh with
// every full tile in row chunks.  Block row 0 (the first e rows) is row-major
// (ld m); in block row I >= 1 the columns below e sit in the ragged tile (I, 0)
// (row-major, ld e, split at the head) and column e + 32 ch + c of row rr at
// tile(I, 1) + 4096 ch + 32 rr + c: a row is a run of 32-float chunks 4096
// floats apart.  The 32-row groups follow the tiles: ceil(e / 32) groups in
// block row 0, then four per full block row, and the diagonal blocks inverted
// are those of these groups.  In the transposed updates of block row I >= 1
// the threads of a warp take the 32 columns of one chunk.
struct CrFactor;
// The ragged tile (I, 0) of block row I >= 1: element (rr, c), c < e, is float
// rr e + c of the tile, which sits at span(I) up to the head and after the full
// tiles beyond it.
struct CrRag {
  const float* p;  // the block row's span
  int hh, e;
  int jump;        // the full tiles' floats
  __device__ CrRag(const float* F, const TlGeom& g, int I)
      : p(F + g.span(I)), hh(g.head(I)), e(g.e), jump((g.T - 1) * kTlTile) {}
  __device__ float operator()(int rr, int c) const {
    const int idx = rr * e + c;
    return __ldg(p + (idx < hh ? idx : idx + jump));
  }
};

struct CrFactor {
  const float* F;  // the airfoil's matrix
  TlGeom g;
  int m;
  int G0;          // groups of block row 0
  int nch;         // chunks of a full block row: 4 (T - 1)
  __device__ void init(const float* F_, int m_, int64_t moff) {
    F = F_;
    m = m_;
    g.init(m_, moff);
    G0 = (g.e + 31) >> 5;
    nch = 4 * (g.T - 1);
  }
  __device__ int groups() const { return G0 + nch; }
  __device__ int k0(int d) const { return d < G0 ? 32 * d : g.e + 32 * (d - G0); }
  __device__ int kb(int d) const { return d < G0 ? min(32, g.e - 32 * d) : 32; }
  // row rr of block row I >= 1: its chunk 0 (add 4096 ch + the column in the chunk)
  __device__ const float* chunk_row(int I, int rr) const {
    return F + g.tile(I, 1) + (int64_t)rr * kTlC;
  }
  // rows i .. i + R - 1 of group d, as RmFactor
  template <int R, int U>
  __device__ void dot_left(float (&acc)[R], int i, int d, const float* y, int lane) const {
    if (d < G0) {
      rows_dot<R, U>(acc, F + i * m + lane, m, 32, y + lane, 0, d);
      return;
    }
    const int e = g.e, I = 1 + ((i - e) >> 7), rr = (i - e) & (kTlB - 1);
    const CrRag rag(F, g, I);
#pragma unroll 1
    for (int c = lane; c < e; c += 32) {
      const float yy = y[c];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = fmaf(rag(rr + r, c), yy, acc[r]);
    }
    rows_dot<R, U>(acc, chunk_row(I, rr) + lane, kTlC, kTlChunk, y + e + lane, 0, d - G0);
  }
  template <int R, int U>
  __device__ void dot_right(float (&acc)[R], int i, int d, const float* y, int lane) const {
    if (d < G0) {
      rows_dot_range<R, U>(acc, F + i * m, m, y, k0(d) + kb(d), m, lane);
      return;
    }
    const int e = g.e, I = 1 + ((i - e) >> 7), rr = (i - e) & (kTlB - 1);
    rows_dot<R, U>(acc, chunk_row(I, rr) + lane, kTlC, kTlChunk, y + e + lane, d - G0 + 1, nch);
  }
  __device__ const float* diag_row(int d, int i) const {
    if (d < G0) return F + (int64_t)i * m + 32 * d;
    const int h = d - G0, rr = (i - g.e) & (kTlB - 1);
    return chunk_row(1 + (h >> 2), rr) + (int64_t)h * kTlChunk;
  }
  __device__ int diag_step(int d) const { return d < G0 ? m : kTlC; }
  template <int U>
  __device__ void update_right(int d, float* z, const float* gv, float* nx, int tid, int nth) const {
    const int k0 = this->k0(d), kb = this->kb(d), c0 = k0 + kb;
    const int c1 = c0 + this->kb(d + 1);  // end of group d + 1 (d + 1 < groups())
    if (d < G0) {
      for (int r = c0 + tid; r < m; r += nth) {
        const float acc = column_update<U>(F + k0 * m + r, m, kb, gv, z[r]);
        if (r < c1)
          nx[r - c0] = acc;
        else
          z[r] = acc;
      }
    } else {
      const int h = d - G0, e = g.e;
      const float* p = chunk_row(1 + (h >> 2), 32 * (h & 3));  // row k0 of the group
      for (int c = 32 * (h + 1) + tid; c < 32 * nch; c += nth) {
        const float* pc = p + (c >> 5) * kTlChunk + (c & 31);
        const float acc = column_update<U>(pc, kTlC, 32, gv, z[e + c]);
        if (e + c < c1)
          nx[e + c - c0] = acc;
        else
          z[e + c] = acc;
      }
    }
  }
  template <int U>
  __device__ void update_left(int d, float* z, const float* gv, float* nx, int tid, int nth) const {
    const int k0 = this->k0(d), kb = this->kb(d);
    const int p0 = this->k0(d - 1);  // start of group d - 1 (d >= 1)
    if (d < G0) {
      for (int r = tid; r < k0; r += nth) {
        const float acc = column_update<U>(F + k0 * m + r, m, kb, gv, z[r]);
        if (r >= p0)
          nx[r - p0] = acc;
        else
          z[r] = acc;
      }
    } else {
      const int h = d - G0, I = 1 + (h >> 2), rr0 = 32 * (h & 3), e = g.e;
      // columns below e: the ragged tile (I, 0)
      const CrRag rag(F, g, I);
      for (int r = tid; r < e; r += nth) {
        float acc = z[r];
#pragma unroll 16
        for (int t = 0; t < 32; ++t) acc = fmaf(-rag(rr0 + t, r), gv[t], acc);
        if (r >= p0)
          nx[r - p0] = acc;
        else
          z[r] = acc;
      }
      // columns e .. k0 - 1: the chunks before the group's
      const float* p = chunk_row(I, rr0);
      for (int c = tid; c < 32 * h; c += nth) {
        const float* pc = p + (c >> 5) * kTlChunk + (c & 31);
        const float acc = column_update<U>(pc, kTlC, 32, gv, z[e + c]);
        if (e + c >= p0)
          nx[e + c - p0] = acc;
        else
          z[e + c] = acc;
      }
    }
  }
};

// FWD: y <- U^{-1} L^{-1} y (scratch ty, 32 floats); TRN: z <- L^{-T} U^{-T} z (scratch
// tz, 64 floats, 16-byte aligned: the group's incoming values, then its results).
// Each of the block's 32 / R warps takes R neighbouring rows (columns) of a group,
// whose products share the reads of the vector and whose sums over the lanes are
// taken together (lane_sums): with one row after the other, the sums, masks and
// addresses were five times the instructions of the products, and the sweeps 61 % of
// the refinement of 4096 x 200 panels.
template <bool FWD, bool TRN, int R, class Fac>
__device__ void lu_sweeps(const Fac& f, float* y, float* z, float* ty, float* tz) {
  static_assert(FWD || TRN, "a system to solve");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tid = (int)threadIdx.x;
  constexpr int NT = 1024 / R;
  // loads in flight per lane: chunks of the rows (8 loads; 16 for the two rows of the
  // largest airfoils' blocks, 14.9 -> 14.6 ms on 304 of 1024..2048), and entries of a
  // column (8 where 8 blocks share an SM; 32 rather than 16 took 304 of 600 from 2022
  // to 1929 us)
  constexpr int U = R >= 8 ? 1 : R == 4 ? 2 : 16 / R;
  constexpr int UC = R >= 8 ? 8 : 32;
  const int G = f.groups();
  const int q0 = warp * R, sub = lane / (32 / R);  // the warp's rows; the lane's of them
  float* gz = tz + 32;
#pragma unroll 1
  for (int s = 0; s < 2 * G; ++s) {
    const bool down = s < G;
    const int d = down ? s : 2 * G - 1 - s;
    const int k0 = f.k0(d), kb = f.kb(d);
    if (FWD) {
      // t = y - (rows of L left of the group, of U right of it) . y
      if (q0 + R <= kb) {
        float acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = 0.0f;
        if (down)
          f.template dot_left<R, U>(acc, k0 + q0, d, y, lane);
        else
          f.template dot_right<R, U>(acc, k0 + q0, d, y, lane);
        const float v = lane_sums<R>(acc, lane);
        if ((lane & (32 / R - 1)) == 0) ty[q0 + sub] = y[k0 + q0 + sub] - v;
      } else {
        for (int q = q0; q < kb; ++q) {  // the last rows of a short group
          float acc[1] = {0.0f};
          if (down)
            f.template dot_left<1, 1>(acc, k0 + q, d, y, lane);
          else
            f.template dot_right<1, 1>(acc, k0 + q, d, y, lane);
          const float v = warp_sum_f(acc[0]);
          if (lane == 0) ty[q] = y[k0 + q] - v;
        }
      }
    }
    if (TRN) {
      if (s == 0 || s == G) {
        if (tid < 32) tz[tid] = (tid < kb) ? z[k0 + tid] : 0.0f;
      } else if (down) {
        f.template update_right<UC>(d - 1, z, gz, tz, tid, NT);
      } else {
        f.template update_left<UC>(d + 1, z, gz, tz, tid, NT);
      }
    }
    __syncthreads();
    if (FWD) {
      // down: y_i = t_i + sum_{k<i} X[i][k] t_k (X unit lower, stored below the
      // diagonal); up: y_i = sum_{k>=i} Y[i][k] t_k (Y upper with diagonal)
      const float t = (lane < kb) ? ty[lane] : 0.0f;
      const float* p = f.diag_row(d, k0) + lane;
      const int step = f.diag_step(d);
      float v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int q = q0 + r;
        const bool on = q < kb && lane < kb && (down ? lane < q : lane >= q);
        v[r] = on ? __ldg(p + q * step) * t : 0.0f;
      }
      const float w = lane_sums<R>(v, lane);
      const int q = q0 + sub;
      if ((lane & (32 / R - 1)) == 0 && q < kb) y[k0 + q] = down ? ty[q] + w : w;
    }
    if (TRN) {
      // down: z_i = sum_{k<=i} Y[k][i] t_k; up: z_i = t_i + sum_{k>i} X[k][i] t_k
      const float t = (lane < kb) ? tz[lane] : 0.0f;
      const float* p = f.diag_row(d, k0) + lane * f.diag_step(d);
      float v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int q = q0 + r;
        const bool on = q < kb && lane < kb && (down ? lane <= q : lane > q);
        v[r] = on ? __ldg(p + q) * t : 0.0f;
      }
      const float w = lane_sums<R>(v, lane);
      const int q = q0 + sub;
      if ((lane & (32 / R - 1)) == 0 && q < kb) {
        const float zi = down ? w : tz[q] + w;
        z[k0 + q] = zi;
        gz[q] = zi;
      }
    }
    __syncthreads();
  }
}

// The forward system (fw), the transposed one (tr) or both; ty: 32 floats, tz: 64.
// Both at once (COMBINE) or one after the other.
template <bool COMBINE, int R, class Fac>
__device__ void lu_solve(const Fac& f, bool fw, bool tr, float* y, float* z, float* ty,
                         float* tz) {
  if (COMBINE && fw && tr) {
    lu_sweeps<true, true, R>(f, y, z, ty, tz);
    return;
  }
  if (fw) lu_sweeps<true, false, R>(f, y, z, ty, tz);
  if (tr) lu_sweeps<false, true, R>(f, y, z, ty, tz);
}

// ---------------------------------------------------------------------------
// Double-float residuals against the stored planes
// ---------------------------------------------------------------------------
// Accumulator for sum_k (h_k + l_k)(xh_k + xl_k) with error ~2^-70 sum|p|:
// s1 collects the exact leading products h*xh through two_sum (their rounding
// errors go to s2), s2 (double-float) collects the ~2^-24 terms (the two_prod
// error of h*xh, h*xl, l*xh), summed error-free into one float per entry
// first, and s3 (float) the ~2^-48 terms (the errors of h*xl, l*xh and of
// that sum, and l*xl).  Every product is exact via two_prod.
// Corrections with the Gauss-Jordan inverse X = (P Mt)^{-1}: y <- X y (rows
// over the warps, 4 rows per pass, lanes along the row) and y <- X^T y (the
// rows split into 8 ranges, one per warp, a column per lane, partial sums in
// `part`, 8 x m floats).  `w` is an m-float shared scratch.
__device__ void gj_apply(const float* __restrict__ X, int m, float* y, float* w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i0 = 4 * warp; i0 < m; i0 += 4 * (int)(blockDim.x >> 5)) {
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int k = lane; k < m; k += 32) {
      const float yk = y[k];
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (i0 + r < m) acc[r] = fmaf(__ldg(X + (i0 + r) * m + k), yk, acc[r]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float v = warp_sum_f(acc[r]);
      if (lane == 0 && i0 + r < m) w[i0 + r] = v;
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < m; k += (int)blockDim.x) y[k] = w[k];
  __syncthreads();
}

__device__ void gj_apply_transposed(const float* __restrict__ X, int m, float* y, float* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rows = (m + (int)(blockDim.x >> 5) - 1) / (int)(blockDim.x >> 5);
  const int k0 = warp * rows, k1 = min(m, k0 + rows);
  for (int cb = 0; cb < m; cb += 32) {
    const int i = cb + lane;
    float acc = 0.0f;
    if (i < m) {
#pragma unroll 4
      for (int k = k0; k < k1; ++k) acc = fmaf(__ldg(X + k * m + i), y[k], acc);
    }
    if (i < m) part[warp * m + i] = acc;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += (int)blockDim.x) {
    float v = 0.0f;
#pragma unroll
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += part[w * m + i];
    y[i] = v;
  }
  __syncthreads();
}

struct ResAcc {
  float s1, s3;
  df2 s2;
};
__device__ __forceinline__ void resacc_init(ResAcc& a) {
  a.s1 = 0.0f;
  a.s3 = 0.0f;
  a.s2 = mkdf(0.0f);
}
__device__ __forceinline__ void resacc_add(ResAcc& a, float h, float l, float xh, float xl) {
  const df2 p1 = two_prod(h, xh);
  const df2 p2 = two_prod(h, xl);
  const df2 p3 = two_prod(l, xh);
  const df2 t = two_sum(a.s1, p1.hi);
  a.s1 = t.hi;
  // the four ~2^-24 terms summed error-free (u, v, w) before the one
  // double-float addition; the three sums' errors are ~2^-48 terms
  const df2 u = two_sum(t.lo, p1.lo);
  const df2 v = two_sum(p2.hi, p3.hi);
  const df2 w = two_sum(u.hi, v.hi);
  a.s2 = df_add_f(a.s2, w.hi);
  const float e1 = __fadd_rn(__fadd_rn(u.lo, v.lo), w.lo);
  const float e2 = __fadd_rn(__fadd_rn(p2.lo, p3.lo), __fmul_rn(l, xl));
  a.s3 = __fadd_rn(a.s3, __fadd_rn(e1, e2));
}
__device__ __forceinline__ void resacc_merge(ResAcc& a, const ResAcc& b) {
  const df2 t = two_sum(a.s1, b.s1);
  a.s1 = t.hi;
  a.s2 = df_add_f(a.s2, t.lo);
  a.s2 = df_add(a.s2, b.s2);
  a.s3 = __fadd_rn(a.s3, b.s3);
}
__device__ __forceinline__ ResAcc warp_sum_res(ResAcc a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ResAcc b;
    b.s1 = __shfl_xor_sync(0xffffffffu, a.s1, o);
    b.s2.hi = __shfl_xor_sync(0xffffffffu, a.s2.hi, o);
    b.s2.lo = __shfl_xor_sync(0xffffffffu, a.s2.lo, o);
    b.s3 = __shfl_xor_sync(0xffffffffu, a.s3, o);
    resacc_merge(a, b);
  }
  return a;
}
// c - acc in FP64 (c is FP64).
__device__ __forceinline__ double resacc_sub_from(double c, const ResAcc& a) {
  return ((c - (double)a.s1) - ((double)a.s2.hi + (double)a.s2.lo)) - (double)a.s3;
}

// The first residual of the refinement only has to carry the ~1e-4 error of
// the float32 solve to the next correction: a double-float sum of the products
// (each exact to ~2^-48 of itself, the sum to ~2^-44 of sum |p|) suffices there.
struct LiteAcc {
  df2 s;
};
__device__ __forceinline__ void resacc_init(LiteAcc& a) { a.s = mkdf(0.0f); }
__device__ __forceinline__ void resacc_add(LiteAcc& a, float h, float l, float xh, float xl) {
  const df2 p = two_prod(h, xh);
  const float e = __fmaf_rn(h, xl, __fmaf_rn(l, xh, p.lo));
  a.s = df_add(a.s, mkdf(p.hi, e));
}
__device__ __forceinline__ void resacc_merge(LiteAcc& a, const LiteAcc& b) { a.s = df_add(a.s, b.s); }
__device__ __forceinline__ LiteAcc warp_sum_res(LiteAcc a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    LiteAcc b;
    b.s.hi = __shfl_xor_sync(0xffffffffu, a.s.hi, o);
    b.s.lo = __shfl_xor_sync(0xffffffffu, a.s.lo, o);
    resacc_merge(a, b);
  }
  return a;
}
__device__ __forceinline__ double resacc_sub_from(double c, const LiteAcc& a) {
  return c - ((double)a.s.hi + (double)a.s.lo);
}

__device__ __forceinline__ ResAcc shfl_xor_acc(const ResAcc& a, int o) {
  ResAcc b;
  b.s1 = __shfl_xor_sync(0xffffffffu, a.s1, o);
  b.s2.hi = __shfl_xor_sync(0xffffffffu, a.s2.hi, o);
  b.s2.lo = __shfl_xor_sync(0xffffffffu, a.s2.lo, o);
  b.s3 = __shfl_xor_sync(0xffffffffu, a.s3, o);
  return b;
}
__device__ __forceinline__ LiteAcc shfl_xor_acc(const LiteAcc& a, int o) {
  LiteAcc b;
  b.s.hi = __shfl_xor_sync(0xffffffffu, a.s.hi, o);
  b.s.lo = __shfl_xor_sync(0xffffffffu, a.s.lo, o);
  return b;
}
__device__ __forceinline__ ResAcc sel_acc(bool c, const ResAcc& a, const ResAcc& b) {
  ResAcc r;
  r.s1 = c ? a.s1 : b.s1;
  r.s2.hi = c ? a.s2.hi : b.s2.hi;
  r.s2.lo = c ? a.s2.lo : b.s2.lo;
  r.s3 = c ? a.s3 : b.s3;
  return r;
}
__device__ __forceinline__ LiteAcc sel_acc(bool c, const LiteAcc& a, const LiteAcc& b) {
  LiteAcc r;
  r.s.hi = c ? a.s.hi : b.s.hi;
  r.s.lo = c ? a.s.lo : b.s.lo;
  return r;
}

// Residuals of a warp's rows j = first + step i (i = 0, 1, ...), four at a time:
// add() takes the lanes' shares of one row after the other.  Two halving exchanges
// (each lane keeps half of the rows) and three butterflies sum four rows over the
// lanes with 6 merges instead of 20, and the FP64 part (the right-hand side, the
// final subtraction) waits until every lane has a row of its own: on a pipe of 1/74
// of the FP32 rate it was one lane's chain of dependent operations per row.  QUAD
// false sums each row by itself (the fused pass has no registers for four).
template <class Acc, class Rhs, class RT, bool QUAD = true>
struct RowSums {
  Acc v[4], keep;
  int i = 0;  // rows taken
  const Rhs& b;
  RT* r;
  int first, step, m;
  __device__ RowSums(const Rhs& b_, RT* r_, int first_, int step_, int m_)
      : b(b_), r(r_), first(first_), step(step_), m(m_) {
#pragma unroll
    for (int t = 0; t < 4; ++t) resacc_init(v[t]);
    resacc_init(keep);
  }
  // b is kept by reference until finish(): a temporary would be gone by then
  RowSums(const Rhs&&, RT*, int, int, int) = delete;
  __device__ __forceinline__ void add(const Acc& a) {
    if constexpr (!QUAD) {
      keep = sel_acc((int)(threadIdx.x & 31) == (i & 31), warp_sum_res(a), keep);
      if ((++i & 31) == 0) flush(i - 32);
      return;
    }
    v[0] = v[1];
    v[1] = v[2];
    v[2] = v[3];
    v[3] = a;
    if ((++i & 3) == 0) reduce();
  }
  __device__ __forceinline__ void reduce() {
    const int lane = threadIdx.x & 31;
    const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0;
    Acc k0 = sel_acc(b4, v[2], v[0]), k1 = sel_acc(b4, v[3], v[1]);
    resacc_merge(k0, shfl_xor_acc(sel_acc(b4, v[0], v[2]), 16));
    resacc_merge(k1, shfl_xor_acc(sel_acc(b4, v[1], v[3]), 16));
    Acc k = sel_acc(b3, k1, k0);
    resacc_merge(k, shfl_xor_acc(sel_acc(b3, k0, k1), 8));
#pragma unroll 1
    for (int o = 4; o > 0; o >>= 1) resacc_merge(k, shfl_xor_acc(k, o));
    // the lanes l >> 3 == t hold row t of the four; lane l keeps the group l & 7
    keep = sel_acc((lane & 7) == ((i >> 2) - 1 & 7), k, keep);
    if ((i & 31) == 0) flush(i - 32);
  }
  __device__ __forceinline__ void flush(int i0) {
    const int lane = threadIdx.x & 31;
    const int row = i0 + (QUAD ? 4 * (lane & 7) + (lane >> 3) : lane);
    const int j = first + step * row;
    if (row < i && j < m) b.store(r, j, resacc_sub_from(b(j), keep));
  }
  __device__ __forceinline__ void finish() {
    const int n = i;
    if constexpr (QUAD) {
      Acc z;
      resacc_init(z);
      while (i & 3) add(z);
    }
    if (i & 31) {
      const int i0 = i & ~31;
      i = n;
      flush(i0);
    }
  }
};

// r_j = b_j - sum_i M_ji x_i for all rows j; x given as float pairs (xh, xl).
// A warp takes two neighbouring rows at a time and issues all loads of a
// 256-column chunk before accumulating.
template <class Acc, class Rhs, class RT>
__device__ void residual_rows(const float* __restrict__ Ah, const float* __restrict__ Al, int m,
                              const float* xh, const float* xl, const Rhs& b, RT* r) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
  RowSums<Acc, Rhs, RT> sums(b, r, warp, nw, m);
  for (int j0 = warp; j0 < m; j0 += 2 * nw) {
    Acc acc0, acc1;
    resacc_init(acc0);
    resacc_init(acc1);
    const int j1 = j0 + nw;
    const bool two = j1 < m;
    for (int c0 = 0; c0 < m; c0 += 256) {
      float h0[8], l0[8], h1[8], l1[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int c = c0 + lane + 32 * t;
        const bool ok = c < m;
        h0[t] = ok ? __ldg(Ah + j0 * m + c) : 0.0f;
        l0[t] = ok ? __ldg(Al + j0 * m + c) : 0.0f;
        h1[t] = (ok && two) ? __ldg(Ah + j1 * m + c) : 0.0f;
        l1[t] = (ok && two) ? __ldg(Al + j1 * m + c) : 0.0f;
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int c = c0 + lane + 32 * t;
        if (c < m) {
          const float xa = xh[c], xb = xl[c];
          resacc_add(acc0, h0[t], l0[t], xa, xb);
          resacc_add(acc1, h1[t], l1[t], xa, xb);
        }
      }
    }
    sums.add(acc0);
    sums.add(acc1);
  }
  sums.finish();
}

// r_i = g_i - sum_j M_ji x_j for all columns i: each warp owns 32 consecutive
// columns (one per lane) and walks all rows, 8 rows of loads in flight.
template <class Acc, class Rhs, class RT>
__device__ void residual_cols(const float* __restrict__ Ah, const float* __restrict__ Al, int m,
                              const float* xh, const float* xl, const Rhs& g, RT* r) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int cb = 32 * warp; cb < m; cb += (int)blockDim.x) {
    const int c = cb + lane;
    const bool ok = c < m;
    Acc acc;
    resacc_init(acc);
    for (int jb = 0; jb < m; jb += 8) {
      float h[8], l[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int j = jb + q;
        h[q] = (ok && j < m) ? __ldg(Ah + j * m + c) : 0.0f;
        l[q] = (ok && j < m) ? __ldg(Al + j * m + c) : 0.0f;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (jb + q < m) resacc_add(acc, h[q], l[q], xh[jb + q], xl[jb + q]);
    }
    if (ok) g.store(r, c, resacc_sub_from(g(c), acc));
  }
}

// Both residuals in one pass over the matrix (m <= kFuseM), each entry loaded
// once: warp w takes the rows j = w, w + 8, ...; lane l owns the columns
// c = l + 32 t.  The row sums (forward system, x) are reduced across the warp
// per row; the column sums (transposed system, lam) stay in per-lane
// accumulators and are merged across the warps through `part` ((int)(blockDim.x >> 5) x m).
constexpr int kFuseM = 288;
constexpr int kFuseT = (kFuseM + 31) / 32;
static_assert(kFuseM <= kLargeM, "KEEP launches never hold a blocked (tiled) factor");
template <class Acc, int FT = kFuseT, class Rhs, class RT>
__device__ void residual_both(const float* __restrict__ Ah, const float* __restrict__ Al, int m,
                              const float* xh, const float* xl, const float* yh, const float* yl,
                              const Rhs& b, const Rhs& g, RT* rf, RT* rt, Acc* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Acc cacc[FT];
#pragma unroll
  for (int t = 0; t < FT; ++t) resacc_init(cacc[t]);
  RowSums<Acc, Rhs, RT, false> sums(b, rf, warp, (int)(blockDim.x >> 5), m);
  for (int j = warp; j < m; j += (int)(blockDim.x >> 5)) {
    float h[FT], l[FT];
#pragma unroll
    for (int t = 0; t < FT; ++t) {
      const int c = lane + 32 * t;
      const bool ok = c < m;
      h[t] = ok ? __ldg(Ah + j * m + c) : 0.0f;
      l[t] = ok ? __ldg(Al + j * m + c) : 0.0f;
    }
    const float yjh = yh[j], yjl = yl[j];
    Acc racc;
    resacc_init(racc);
#pragma unroll
    for (int t = 0; t < FT; ++t) {
      const int c = lane + 32 * t;
      if (c < m) {
        resacc_add(racc, h[t], l[t], xh[c], xl[c]);
        resacc_add(cacc[t], h[t], l[t], yjh, yjl);
      }
    }
    sums.add(racc);
  }
  sums.finish();
#pragma unroll
  for (int t = 0; t < FT; ++t) {
    const int c = lane + 32 * t;
    if (c < m) part[warp * m + c] = cacc[t];
  }
  __syncthreads();
  for (int c = threadIdx.x; c < m; c += (int)blockDim.x) {
    Acc acc = part[c];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) resacc_merge(acc, part[w * m + c]);
    g.store(rt, c, resacc_sub_from(g(c), acc));
  }
}

// ---------------------------------------------------------------------------
// The refinement kernel: forward and/or transposed system of one airfoil
// ---------------------------------------------------------------------------
// Where the refinement keeps its vectors.  Launches of small airfoils
// (n_max + 1 <= kFuseM, KEEP) hold x, the residual r and the right-hand side
// in shared memory as doubles.  The others, whose shared memory bounds the
// airfoils per SM, keep x in the caller's output array, the residual as the
// float the correction solve takes (component n already times s) and evaluate
// the right-hand side where it is needed, once per row or column of a
// residual pass.
template <class RT>
struct IrSystem {
  double* x;   // m  current solution
  RT* r;       // m  residual
  float* xh;   // m  x as float pairs for the residual
  float* xl;   // m
};

// A stored right-hand side (KEEP): the residual is kept as is.
struct SmemRhs {
  const double* bb;
  __device__ double operator()(int k) const { return bb[k]; }
  __device__ void store(double* r, int k, double v) const { r[k] = v; }
};

// Right-hand side of system q (0: M u = b, 1: M^T lambda = g), evaluated; the
// residual is stored as the correction solve's float input.
struct IrRhs {
  const double* rhs;   // forward right-hand side (rhs_kind 0), at the airfoil's offset
  const double* nd;    // the airfoil's nodes
  const double* w_u;   // vector-Jacobian weights at the airfoil's offsets (or NULL)
  const double* w_cp;
  const double* u_in;
  double w_cl;
  int n, q, rhs_kind, vjp;
  double v, cc, s;
  __device__ void init(const SolveArgs& a, int b, int n_, int q_, double s_) {
    const int64_t vo = vec_off(a.bt, b);
    rhs = (a.rhs_kind == 0 && a.rhs) ? a.rhs + vo : nullptr;
    nd = a.bt.nodes + 2 * a.bt.node_off[b];
    w_u = a.w_u ? a.w_u + vo : nullptr;
    w_cp = a.w_cp ? a.w_cp + a.bt.node_off[b] : nullptr;
    u_in = a.u_in ? a.u_in + vo : nullptr;
    w_cl = a.w_cl ? a.w_cl[b] : 0.0;
    n = n_;
    q = q_;
    rhs_kind = a.rhs_kind;
    vjp = a.vjp;
    v = a.vinf ? a.vinf[b] : 1.0;
    cc = a.chord ? a.chord[b] : 1.0;
    s = s_;
  }
  __device__ double operator()(int k) const { return eval(k); }
  __device__ double eval(int k) const {
    if (q == 0) {
      if (rhs_kind == 0) return rhs[k];
      // the basis right-hand sides of a polar: b(alpha) = cos(alpha) b_y +
      // sin(alpha) b_x with b_y = v m_y, b_x = -v m_x (m the control point)
      if (k >= n) return 0.0;
      const int k1 = (k + 1 == n) ? 0 : k + 1;
      return (rhs_kind == 1) ? 0.5 * v * (nd[2 * k + 1] + nd[2 * k1 + 1])
                                : -0.5 * v * (nd[2 * k] + nd[2 * k1]);
    }
    double g = 0.0;
    if (k < n) {
      const int k1 = (k + 1 == n) ? 0 : k + 1;
      const double hx = nd[2 * k1] - nd[2 * k], hy = nd[2 * k1 + 1] - nd[2 * k + 1];
      g = 2.0 * sqrt(hx * hx + hy * hy) / (v * cc);  // dCl/dgamma_k
    }
    if (vjp) {
      // dL/du for L = w_cl Cl + w_u . u + w_cp . Cp, Cp_k = 1 - (gamma_k / v)^2
      g *= w_cl;
      if (w_u) g += w_u[k];
      if (w_cp && k < n) g += w_cp[k] * (-2.0 * u_in[k] / (v * v));
    }
    return g;
  }
  __device__ float scaled(int k, double r) const { return (float)((k == n) ? r * s : r); }
  __device__ void store(float* r, int k, double v) const { r[k] = scaled(k, v); }
};

// The float input of the correction solve from a residual component.
__device__ __forceinline__ float solve_input(double r, int k, int n, double s) {
  return (float)((k == n) ? r * s : r);
}
__device__ __forceinline__ float solve_input(float r, int, int, double) { return r; }

__device__ __forceinline__ int gpiv_first(const SolveArgs& a, int b) {
  return a.piv[vec_off(a.bt, b)];
}

// Row permutation of the factor, P y = y[perm], from its exchanges (by the whole
// block; ends with a barrier).  Every exchange stays inside its diagonal block
// (32 rows, or the blocks of the tiled layout), so the blocks' exchanges are
// composed side by side, a thread each, instead of one thread walking all m
// (~45 cycles a row: 20 k of a 200-panel airfoil's 600 k cycles).
__device__ __forceinline__ void factor_permutation(const int32_t* gpiv, int m, bool gj, int* perm) {
  for (int k = threadIdx.x; k < m; k += blockDim.x) perm[k] = k;
  __syncthreads();
  const bool tiled = !gj && m > kLargeM;
  const int blk = tiled ? kTlB : 32;
  const int e = tiled ? m - kTlB * ((m - 1) / kTlB) : 32;  // size of the first block
  const int k0 = threadIdx.x == 0 ? 0 : e + blk * ((int)threadIdx.x - 1);
  if (k0 < m) {
    const int k1 = min(m, threadIdx.x == 0 ? e : k0 + blk);
#pragma unroll 8
    for (int k = k0; k < k1; ++k) {
      const int p = gj ? -gpiv[k] - 1 : gpiv[k];
      if (p != k) {
        const int t = perm[k];
        perm[k] = perm[p];
        perm[p] = t;
      }
    }
  }
  __syncthreads();
}

// NT threads, MINB blocks per SM (see launch_ir_kernel).
template <int NT, int MINB, int FT, bool KEEP>
__global__ void __launch_bounds__(NT, MINB) k_ir_mixed(SolveArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const Batch& bt = a.bt;
  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b);
  const int m = n + 1;
  if (a.info[b] != 0 || n > bt.n_max) return;
  const int mv = bt.n_max + 1;
  using RT = typename std::conditional<KEEP, double, float>::type;
  double* red = reinterpret_cast<double*>(smraw);
  IrSystem<RT> sys[2];
  double* dp = red + converged_words(NT);
  double* bbs = dp;  // KEEP: x, r, bb of both systems (6 m doubles)
  if (KEEP) {
    for (int q = 0; q < 2; ++q) {
      sys[q].x = dp;
      sys[q].r = reinterpret_cast<RT*>(dp + mv);
      dp += 2 * mv;
    }
    bbs = dp;
    dp += 2 * mv;
  }
  float* y = reinterpret_cast<float*>(dp);  // m
  float* fp = y + mv;
  for (int q = 0; q < 2; ++q) {
    sys[q].xh = fp;
    sys[q].xl = fp + mv;
    fp += 2 * mv;
    if (!KEEP) {
      sys[q].r = reinterpret_cast<RT*>(fp);
      fp += mv;
    }
  }
  int* perm = reinterpret_cast<int*>(fp);  // m
  float* t32 = reinterpret_cast<float*>(perm + mv);  // 32
  // per-warp partial sums: of the inverse's products (floats, m <= kGjM), or of
  // the fused residual pass (ResAcc, launches with n_max + 1 <= kFuseM)
  double* dprev = reinterpret_cast<double*>(t32 + 32);  // 2
  float* part = reinterpret_cast<float*>(
      (reinterpret_cast<uintptr_t>(dprev + 2) + 15) & ~(uintptr_t)15);
  // The corrections: the forward one in y, the transposed one in z, which is
  // the transposed system's float copy of lambda (rewritten from lambda before
  // it is read again); the transposed sweeps' 64-float group scratch is `red`
  // (free while the sweeps run).
  float* z = sys[1].xh;
  float* t32z = reinterpret_cast<float*>(red);
  // the factor buffer holds an inverse (exchanges stored as -(row + 1)) or an LU
  const bool gj = gpiv_first(a, b) < 0;

  const int64_t moff = bt.mat_off[b];
  const float* Ah = a.A_hi + moff;
  const float* Al = a.A_lo + moff;
  const float* F = a.LU + moff;
  // above kLargeM - 1 panels: the blocked factor's tiled layout (never in a
  // KEEP launch: n_max + 1 <= kFuseM there)
  const bool cr = !KEEP && !gj && m > kLargeM;
  CrFactor crf;
  if constexpr (!KEEP) {
    if (cr) crf.init(F, m, moff);
  }
  const int32_t* gpiv = a.piv + vec_off(bt, b);
  const double s = border_scale(Ah, n, m, red);
  const bool act0 = a.u != nullptr, act1 = a.lam != nullptr;
  // the fused residual pass needs `part`, allocated when the launch's n_max fits
  const bool fuse = bt.n_max + 1 <= kFuseM;

  // right-hand sides: b, and g = dCl/du = 2 |h_k| / (v c) (0 for C); x = 0, r = b
  IrRhs rhs[2];
  for (int q = 0; q < 2; ++q) rhs[q].init(a, b, n, q, s);
  SmemRhs srhs[2];
  srhs[0].bb = bbs;
  srhs[1].bb = bbs + mv;
  if (!KEEP) {
    sys[0].x = act0 ? a.u + vec_off(bt, b) : nullptr;
    sys[1].x = act1 ? a.lam + vec_off(bt, b) : nullptr;
  }
  for (int k = threadIdx.x; k < m; k += (int)blockDim.x) {
    for (int q = 0; q < 2; ++q) {
      if (!(q == 0 ? act0 : act1)) continue;
      const double bk = rhs[q].eval(k);
      sys[q].x[k] = 0.0;
      if constexpr (KEEP) {
        bbs[q * mv + k] = bk;
        sys[q].r[k] = bk;
      } else {
        sys[q].r[k] = rhs[q].scaled(k, bk);
      }
    }
  }
  factor_permutation(gpiv, m, gj, perm);

  bool active[2] = {act0, act1};
  bool conv[2] = {!act0, !act1};
  int it = 0;
  for (;; ++it) {
    const bool run0 = active[0] && !conv[0], run1 = active[1] && !conv[1];
    // the corrections' right-hand sides: y = P S_r r (forward system; then
    // dx = S_c y) and z = S_c r (transposed system; then dlambda = S_r P^T z)
    for (int k = threadIdx.x; k < m; k += (int)blockDim.x) {
      if (run0) {
        const int src = perm[k];
        y[k] = solve_input(sys[0].r[src], src, n, s);
      }
      if (run1) z[k] = solve_input(sys[1].r[k], k, n, s);
    }
    __syncthreads();
    if (gj) {
      if (run0) gj_apply(F, m, y, part);
      if (run1) gj_apply_transposed(F, m, z, part);
    } else if constexpr (!KEEP) {
      if (cr)
        lu_solve<true, 1024 / NT>(crf, run0, run1, y, z, t32, t32z);
      else
        lu_solve<true, 1024 / NT>(RmFactor{F, m}, run0, run1, y, z, t32, t32z);
    } else {
      lu_solve<false, 1024 / NT>(RmFactor{F, m}, run0, run1, y, z, t32, t32z);
    }
    unsigned long long dm[2] = {0, 0}, xm[2] = {0, 0};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (!(q == 0 ? run0 : run1)) continue;
      IrSystem<RT>& S = sys[q];
      const float* w = (q == 0) ? y : z;
      for (int k = threadIdx.x; k < m; k += (int)blockDim.x) {
        const int dst = (q == 0) ? k : perm[k];
        const double d = (dst == n) ? (double)w[k] * s : (double)w[k];
        const double xn = S.x[dst] + d;
        S.x[dst] = xn;
        dm[q] = max(dm[q], magnitude_bits(d));
        xm[q] = max(xm[q], magnitude_bits(xn));
      }
    }
    const bool run[2] = {run0, run1};
    block_converged(dm, xm, run, it, a.tol, dprev, conv, red);
    if ((conv[0] && conv[1]) || it >= a.max_iter) break;
    for (int q = 0; q < 2; ++q) {
      if (!active[q] || conv[q]) continue;
      for (int k = threadIdx.x; k < m; k += (int)blockDim.x) {
        const df2 d = df_from_double(sys[q].x[k]);
        sys[q].xh[k] = d.hi;
        sys[q].xl[k] = d.lo;
      }
    }
    __syncthreads();
    const bool both = active[0] && !conv[0] && active[1] && !conv[1];
    auto residuals = [&](const auto& R0, const auto& R1) {
      if (it == 0) {
        if (both && fuse) {
          residual_both<LiteAcc, FT>(Ah, Al, m, sys[0].xh, sys[0].xl, sys[1].xh, sys[1].xl, R0,
                                     R1, sys[0].r, sys[1].r, reinterpret_cast<LiteAcc*>(part));
        } else {
          if (active[0] && !conv[0])
            residual_rows<LiteAcc>(Ah, Al, m, sys[0].xh, sys[0].xl, R0, sys[0].r);
          if (active[1] && !conv[1])
            residual_cols<LiteAcc>(Ah, Al, m, sys[1].xh, sys[1].xl, R1, sys[1].r);
        }
      } else if (both && fuse) {
        residual_both<ResAcc, FT>(Ah, Al, m, sys[0].xh, sys[0].xl, sys[1].xh, sys[1].xl, R0, R1,
                                  sys[0].r, sys[1].r, reinterpret_cast<ResAcc*>(part));
      } else {
        if (active[0] && !conv[0])
          residual_rows<ResAcc>(Ah, Al, m, sys[0].xh, sys[0].xl, R0, sys[0].r);
        if (active[1] && !conv[1])
          residual_cols<ResAcc>(Ah, Al, m, sys[1].xh, sys[1].xl, R1, sys[1].r);
      }
    };
    if constexpr (KEEP)
      residuals(srhs[0], srhs[1]);
    else
      residuals(rhs[0], rhs[1]);
    __syncthreads();
  }
  if (KEEP) {
    for (int k = threadIdx.x; k < m; k += (int)blockDim.x) {
      if (act0) a.u[vec_off(bt, b) + k] = sys[0].x[k];
      if (act1) a.lam[vec_off(bt, b) + k] = sys[1].x[k];
    }
  }
  if (threadIdx.x == 0) {
    if (a.iters && act0) a.iters[b] = it;
    if (!(conv[0] && conv[1])) a.info[b] = PANEL_INFO_NOCONV;
  }
}

// `part` (per-warp partial sums) serves the fused residual pass of launches with
// n_max + 1 <= kFuseM (nt/32 x m accumulators) and, in any launch, the
// Gauss-Jordan products of airfoils with m <= kGjM (nt/32 x m floats): the
// factor of a refinement launch may hold inverses whatever its n_max.
size_t ir_mixed_smem(int n_max, int nt) {
  const size_t mv = (size_t)n_max + 1;
  const size_t part = (mv <= (size_t)kFuseM) ? (size_t)(nt / 32) * mv * sizeof(ResAcc)
                                             : (size_t)(nt / 32) * kGjM * sizeof(float);
  // x, r and the right-hand side of both systems as doubles (KEEP), or r as floats
  const size_t vecs = (mv <= (size_t)kFuseM) ? 6 * mv * 8 + 5 * mv * 4 : 7 * mv * 4;
  return (size_t)converged_words(nt) * 8 + vecs + mv * 4 + 32 * 4 + 32 + part;
}

}  // namespace panel
#include "ir_cluster.cuh"
namespace panel {

static SolveArgs make_args(const Batch& bt, const float* A_hi, const float* A_lo, float* LU,
                           int32_t* piv, const double* rhs, const double* vinf,
                           const double* chord, double* u, double* lam, int max_iter, double tol,
                           int32_t* info, int32_t* iters) {
  SolveArgs a;
  a.bt = bt;
  a.A_hi = A_hi;
  a.A_lo = A_lo;
  a.LU = LU;
  a.piv = piv;
  a.rhs = rhs;
  a.vinf = vinf;
  a.chord = chord;
  a.u = u;
  a.lam = lam;
  a.max_iter = max_iter;
  a.tol = tol;
  a.info = info;
  a.iters = iters;
  a.inverse = 0;
  a.n_cap = bt.n_max;
  a.rhs_kind = 0;
  a.ir_shape = 0;
  a.lu_kind = 0;
  a.vjp = 0;
  a.w_cl = a.w_u = a.w_cp = a.u_in = nullptr;
  return a;
}

// Which one-block LU a launch of B airfoils of at most mv unknowns takes (1 through
// L2, 2 in shared memory).  Up to 64 unknowns the shared-memory form's blocks of 128
// threads, five on an SM, are the faster ones for any batch beyond three airfoils per
// SM (4096 of 40 panels 138 us against 202; one 20 / 20).  Above, one to three of its
// airfoils fit an SM and the L2-resident form is as fast or faster (4096 of 80 panels
// 365 / 360, 128 1358 / 678, 205 2426 / 1526), but for a single airfoil per SM above
// 160 unknowns, by its shorter steps (1 of 159 panels 57 / 54, of 160 65 / 68, of 205
// 89 / 96; 304 of 165 133 / 89).  A launch that also holds larger airfoils runs them all through L2
// at once.
static int lu_kind_by_size(int B, int mv, int sms) {
  if (mv > kSmemLuM) return 1;
  return mv <= 64 || (mv > 160 && B <= sms) ? 2 : 1;
}
// Whether a launch runs k_lu_smem and k_lu_global.
static bool runs_lu_smem(bool inverse, int lu_kind) { return !inverse && lu_kind != 1; }
static bool runs_lu_global(int mv, bool inverse, int lu_kind) {
  return (mv > kSmemLuM || lu_kind == 1) && (mv > kGjM || !inverse);
}
// Kernels of launch_lu_mixed.
int lu_mixed_launches(int B, int n_max, bool inverse, int lu_kind, int sms) {
  const int mv = n_max + 1;
  if (lu_kind == 0) lu_kind = lu_kind_by_size(B, mv, sms);
  return lu_large_launches(mv) + (runs_lu_smem(inverse, lu_kind) ? 1 : 0) +
         (runs_lu_global(mv, inverse, lu_kind) ? 1 : 0) + (inverse ? gj_launches(mv) : 0);
}

// Factor every airfoil: with `inverse` the Gauss-Jordan inverse for m <= kGjM;
// otherwise the one-block LU with the whole matrix in shared memory for m <=
// kSmemLuM (lu_kind 2, or 0 and lu_kind_by_size) or in the LU buffer through L2
// (lu_kind 1, and every m up to kLargeM); the step-synchronous blocked LU beyond.
cudaError_t launch_lu_mixed(const Batch& bt, const float* A_hi, float* LU, int32_t* piv,
                            int32_t* info, int32_t* iters, bool inverse, cudaStream_t s,
                            int lu_kind) {
  SolveArgs a = make_args(bt, A_hi, nullptr, LU, piv, nullptr, nullptr, nullptr, nullptr,
                          nullptr, 0, 0.0, info, iters);
  a.inverse = inverse ? 1 : 0;
  if (lu_kind == 0) lu_kind = lu_kind_by_size(bt.B, bt.n_max + 1, sm_count());
  a.lu_kind = lu_kind;
  cudaError_t e;
  if (bt.n_max + 1 > kLargeM) {
    e = launch_lu_large(a, s);
    if (e != cudaSuccess) return e;
  }
  if (runs_lu_smem(inverse, lu_kind)) {
    // airfoils up to kSmemLuM unknowns with the whole matrix in shared memory
    SolveArgs h = a;
    h.bt.n_max = min(bt.n_max, kSmemLuM - 1);
    const size_t hs = lu_smem_smem(h.bt.n_max);
    const int mv = h.bt.n_max + 1;
    auto go = [&](auto kernel, int nt) {
      const cudaError_t r = ensure_smem(kernel, hs);
      if (r != cudaSuccess) return r;
      kernel<<<bt.B, nt, hs, s>>>(h);
      return cudaGetLastError();
    };
    e = mv <= 64 ? go(k_lu_smem<128, 5>, 128)
                 : mv <= 128 ? go(k_lu_smem<256, 3>, 256) : go(k_lu_smem<512, 1>, 512);
    if (e != cudaSuccess) return e;
  }
  if (runs_lu_global(bt.n_max + 1, inverse, lu_kind)) {
    SolveArgs g = a;
    g.bt.n_max = min(bt.n_max, kLargeM - 1);
    const size_t smem = lu_global_smem(g.bt.n_max);
    auto go = [&](auto kernel) {
      const cudaError_t r = ensure_smem(kernel, smem);
      if (r != cudaSuccess) return r;
      kernel<<<bt.B, kThreads, smem, s>>>(g);
      return cudaGetLastError();
    };
    // three blocks per SM (80 registers, some spilled) where their shared memory fits
    // and the batch fills them, else two with 128 registers (4096 x 256 panels 2566 us
    // against 2781; 1216 x 400, whose panels leave room for two, 2510 against 2350; one
    // of 300 238 against 207)
    e = 3 * (smem + 1024) <= 228 * 1024 && bt.B > 2 * sm_count() ? go(k_lu_global<3>)
                                                                 : go(k_lu_global<2>);
    if (e != cudaSuccess) return e;
  }
  return launch_gj_mixed(a, s);
}

// lambda of a vector-Jacobian product: M^T lambda = w_cl dCl/du + w_u +
// w_cp dCp/du (refined), with the forward strengths u.
// Blocks of 128 threads, 8 per SM, while the shared memory of 8 fits in the SM's
// 228 KB (1 KB of it reserved per block; m <= 204) and the batch fills 8 blocks
// on every SM: more airfoils in flight to hide the latency of the dependent
// sweeps (a smaller batch is better served by more warps per airfoil).  Then 256
// threads, 4 per SM up to kFuseM unknowns (a few spilled registers), and above
// it the most warps per airfoil that shared memory allows: 4 x 256, 2 x 512 or
// 1 x 1024 threads (3 x 256 is the autotuner's fifth shape).
// FT: columns per lane of the fused residual pass (ceil(n_max + 1 / 32) at most;
// fewer registers for the smaller airfoils of the 128-thread shape, m <= 204).
template <int NT, int MINB, int FT = kFuseT>
static cudaError_t launch_ir_shape(const SolveArgs& a, cudaStream_t s) {
  const size_t smem = ir_mixed_smem(a.bt.n_max, NT);
  if (a.bt.n_max + 1 <= kFuseM) {
    const cudaError_t e = ensure_smem(k_ir_mixed<NT, MINB, FT, true>, smem);
    if (e != cudaSuccess) return e;
    k_ir_mixed<NT, MINB, FT, true><<<a.bt.B, NT, smem, s>>>(a);
  } else {
    const cudaError_t e = ensure_smem(k_ir_mixed<NT, MINB, FT, false>, smem);
    if (e != cudaSuccess) return e;
    k_ir_mixed<NT, MINB, FT, false><<<a.bt.B, NT, smem, s>>>(a);
  }
  return cudaGetLastError();
}

// Clusters of C blocks of k_ir_cluster the device holds at once, of the largest airfoil.
static int ir_cluster_capacity(int C) {
  return cluster_capacity(k_ir_cluster, C, kIrClThreads, ir_cluster_smem(PANEL_N_MAX));
}

// Blocks per airfoil of a refinement by clusters, or 0 for k_ir_mixed: the most that
// let every airfoil of the batch run at once.  Measured, both systems (us, the best
// block shape of k_ir_mixed / clusters): 1 airfoil of 200 panels 169 / 203, of 256 228 /
// 257; 8 blocks: 1 of 300 319 / 303, of 600 794 / 586, of 1024 2677 / 1331, of 2048 8526 /
// 3118; 4 blocks: 36 of 400 453 / 412, of 1024 3130 / 1721, of 2048 9863 / 5193; 2
// blocks: 76 of 300 323 / 348, of 400 522 / 509, of 600 926 / 876, of 1024 3218 / 2651;
// one block: 100 of 500 689 / 900, of 1024 3224 / 4005, so not taken.
static int ir_cluster_blocks(const SolveArgs& a) {
  const int mv = a.bt.n_max + 1;
  if (a.ir_shape != 0 || mv <= kFuseM) return 0;
  for (int C = 8; C >= 2; C >>= 1)
    if (a.bt.B <= ir_cluster_capacity(C)) return (C < 4 && mv <= 400) ? 0 : C;
  return 0;
}

static cudaError_t launch_ir_cluster(const SolveArgs& a, int C, cudaStream_t s) {
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = cluster_config(dim3(a.bt.B * C), dim3(C), kIrClThreads,
                                                ir_cluster_smem(a.bt.n_max), s, &at);
  return cudaLaunchKernelEx(&cfg, k_ir_cluster, a);
}

static cudaError_t launch_ir_kernel(const SolveArgs& a, cudaStream_t s) {
  const int n_max = a.bt.n_max;
  auto fits = [&](int nt, int blocks) {
    return (size_t)blocks * (ir_mixed_smem(n_max, nt) + 1024) <= 233472;
  };
  if (const int c = ir_cluster_blocks(a)) return launch_ir_cluster(a, c, s);
  // an explicit shape (autotuning), when one block of it fits the shared memory
  switch (a.ir_shape) {
    case 1:
      if (fits(128, 1) && n_max + 1 <= 7 * 32) return launch_ir_shape<128, 8, 7>(a, s);
      break;
    case 2:
      if (fits(kThreads, 1)) return launch_ir_shape<kThreads, 4>(a, s);
      break;
    case 3:
      if (fits(512, 1)) return launch_ir_shape<512, 2>(a, s);
      break;
    case 4:
      if (fits(1024, 1)) return launch_ir_shape<1024, 1>(a, s);
      break;
    case 5:
      if (fits(kThreads, 1)) return launch_ir_shape<kThreads, 3>(a, s);
      break;
    default:
      break;
  }
  // few airfoils per SM: more warps for each (us, both systems, 256 x 4 / 512 x 2 / 256 x
  // 3: 1 of 100 panels 90 / 87 / 85, 152 of 160 154 / 138 / 142, 304 of 200 283 / 279 /
  // 257, 608 of 256 644 / 790 / 702, 76 of 300 410 / 322 / 397)
  const int sms = sm_count(), mv = n_max + 1;
  // (an airfoil per SM, 512 x 2 / 1024 x 1: 100 of 300 355 / 353, of 500 709 / 689, of
  // 1024 3594 / 3224, forward system alone 2186 / 1996)
  if (mv > 400 && a.bt.B <= sms) return launch_ir_shape<1024, 1>(a, s);
  if (fits(512, 2) && ((mv > 128 && a.bt.B <= sms) || (mv > kFuseM && a.bt.B <= 2 * sms)))
    return launch_ir_shape<512, 2>(a, s);
  if (mv <= kFuseM && a.bt.B <= 3 * sms) return launch_ir_shape<kThreads, 3>(a, s);
  if (fits(128, 8) && n_max + 1 <= 7 * 32 && a.bt.B >= 8 * sm_count())
    return launch_ir_shape<128, 8, 7>(a, s);
  if (n_max + 1 <= kFuseM || fits(kThreads, 4)) return launch_ir_shape<kThreads, 4>(a, s);
  if (fits(512, 2)) return launch_ir_shape<512, 2>(a, s);
  return launch_ir_shape<1024, 1>(a, s);
}

cudaError_t launch_ir_vjp(const Batch& bt, const float* A_hi, const float* A_lo,
                          const float* LU, const int32_t* piv, const double* vinf,
                          const double* chord, const double* u, const double* w_cl,
                          const double* w_u, const double* w_cp, double* lam, int max_iter,
                          double tol, int32_t* info, cudaStream_t s) {
  SolveArgs a = make_args(bt, A_hi, A_lo, const_cast<float*>(LU), const_cast<int32_t*>(piv),
                          nullptr, vinf, chord, nullptr, lam, max_iter, tol, info, nullptr);
  a.vjp = 1;
  a.w_cl = w_cl;
  a.w_u = w_u;
  a.w_cp = w_cp;
  a.u_in = u;
  return launch_ir_kernel(a, s);
}

// Refine the forward (u) and/or transposed (lam) systems with the stored factor.
cudaError_t launch_ir_mixed(const Batch& bt, const float* A_hi, const float* A_lo,
                            const float* LU, const int32_t* piv, const double* rhs,
                            const double* vinf, const double* chord, double* u, double* lam,
                            int max_iter, double tol, int32_t* info, int32_t* iters,
                            cudaStream_t s, int rhs_kind, int ir_shape) {
  SolveArgs a = make_args(bt, A_hi, A_lo, const_cast<float*>(LU), const_cast<int32_t*>(piv),
                          rhs, vinf, chord, u, lam, max_iter, tol, info, iters);
  a.rhs_kind = rhs_kind;
  a.ir_shape = ir_shape;
  return launch_ir_kernel(a, s);
}

}  // namespace panel
