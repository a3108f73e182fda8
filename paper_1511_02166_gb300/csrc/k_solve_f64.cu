// k_solve_f64.cu -- plain FP64 path: LU with partial pivoting and solve.
//
// One block per airfoil.  Right-looking elimination with partial pivoting over the
// whole column (largest |a_rk|, the lowest row on ties, as in the oracle), physical
// row swap, multipliers, rank-1 update; then P b, forward substitution with the
// unit-lower factor and back substitution.  This is the "plain all-FP64
// per-airfoil" baseline; it does no refinement.
//
// The FP64 pipe issues 1/74 of the FP32 rate, so the m^3 / 3 multiply-adds bound a
// full step and the serial part (pivot search, reciprocal) must not wait beside
// them: warp 0 brings the next column up to date first, searches its pivot and takes
// its reciprocal while the other warps update the remaining columns, two block
// barriers per step.  A matrix of up to kSmemF64M unknowns stays in shared memory
// (100 panels: 436 us as four barriers a step on the matrix in L2).  The
// substitutions, one warp per system with its vector in shared memory, multiply by
// the reciprocals of U's diagonal formed beforehand.
#include <cooperative_groups.h>

#include "panel_common.cuh"

namespace panel {

cudaError_t launch_adjoint_prepare(const Batch&, const double*, const double*, const double*,
                                   const double*, const double*, const double*, double*,
                                   const int32_t*, bool, cudaStream_t);

constexpr int kSmemF64M = 160;  // 160 x 161 doubles = 206 KB
constexpr int kF64Threads = 512;  // most threads of a block (solve_f64_threads)

struct PivotF64 {
  int row;
  double value, inv;
};

// Warp 0: the pivot of column k over the rows k..m-1 (lane l the rows k + l + 32 t).
// Magnitudes compare as integers: the FP64 pipe is full of the other warps' updates,
// and every dependent FP64 operation here would queue behind them.
__device__ __forceinline__ void pivot_search_f64(const double* F, int ld, int m, int k,
                                                 PivotF64* p) {
  const int lane = threadIdx.x & 31;
  unsigned long long best = 0;  // |v| + 1 as bits; 0: no candidate (NaN)
  int bi = k;
  for (int r = k + lane; r < m; r += 32) {
    const unsigned long long v =
        (unsigned long long)__double_as_longlong(F[(int64_t)r * ld + k]) & 0x7fffffffffffffffull;
    if (v <= 0x7ff0000000000000ull && v + 1 > best) {
      best = v + 1;
      bi = r;
    }
  }
  const unsigned hi = (unsigned)(best >> 32), lo = (unsigned)best;
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  const int row = (int)__reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? (unsigned)bi : ~0u);
  if (lane == 0) {
    const double val = F[(int64_t)row * ld + k];
    p->row = row;
    p->value = val;
    p->inv = 1.0 / val;
  }
}

// Factor F (m x m, row stride ld) in place; returns 0 or k+1 for a zero pivot.
// rinv[k] = 1 / U_kk.
__device__ int lu_factor_f64(double* F, int ld, int32_t* piv, double* rinv, int m, PivotF64* sp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (warp == 0) pivot_search_f64(F, ld, m, 0, sp);
  __syncthreads();
  double pinv = 1.0;  // reciprocal of the previous pivot
  for (int k = 0; k < m; ++k) {
    const int p = sp->row;
    const double akk = sp->value, inv = sp->inv;
    if (akk == 0.0) return k + 1;  // uniform across the block
    double* fk = F + (int64_t)k * ld;
    double* fp = F + (int64_t)p * ld;
    if (threadIdx.x == 0) {
      piv[k] = p;
      rinv[k] = inv;
    }
    // the previous column becomes its multipliers as this step's rows are exchanged
    // (the thread of row k moves both of its entries)
    if (k > 0)
      for (int r = k + threadIdx.x; r < m; r += blockDim.x) {
        double* q = F + (int64_t)r * ld + k - 1;
        if (r == k) {
          const double t = *q * pinv;
          if (p != k) {
            *q = fp[k - 1] * pinv;
            fp[k - 1] = t;
          } else {
            *q = t;
          }
        } else if (r != p) {
          *q *= pinv;
        }
      }
    if (p != k)
      for (int c = threadIdx.x; c < m; c += blockDim.x) {
        if (c == k - 1) continue;
        const double t = fk[c];
        fk[c] = fp[c];
        fp[c] = t;
      }
    __syncthreads();
    // the multipliers, and with them the next column (warp 0, its own rows) and the
    // rest (the other warps: rows of their own, so each scales what it uses)
    if (warp == 0) {
      if (k + 1 < m) {
        const double u = fk[k + 1];
        for (int r = k + 1 + lane; r < m; r += 32) {
          double* fr = F + (int64_t)r * ld;
          fr[k + 1] = fma(-(fr[k] * inv), u, fr[k + 1]);
        }
        __syncwarp();
        pivot_search_f64(F, ld, m, k + 1, sp);
      }
    } else {
      // lane t takes the multiplier of the warp's row t of a batch of 32
      for (int r0 = k + warp; r0 < m; r0 += 32 * (nw - 1)) {
        const int rl = r0 + lane * (nw - 1);
        const double lv = rl < m ? F[(int64_t)rl * ld + k] * inv : 0.0;
        for (int t = 0; t < 32 && r0 + t * (nw - 1) < m; ++t) {
          double* fr = F + (int64_t)(r0 + t * (nw - 1)) * ld;
          const double l = __shfl_sync(0xffffffffu, lv, t);
          for (int c = k + 2 + lane; c < m; c += 32) fr[c] = fma(-l, fk[c], fr[c]);
        }
      }
    }
    __syncthreads();
    pinv = inv;
  }
  return 0;
}

// x <- (P^T L U)^{-1} x, i.e. solve M x = b with the factors, by one warp; x in
// shared memory.
__device__ void lu_solve_f64(const double* F, int ld, const int32_t* piv, const double* rinv,
                             int m, double* x) {
  const int lane = threadIdx.x & 31;
  if (lane == 0)
    for (int k = 0; k < m; ++k) {
      const int p = piv[k];
      if (p != k) { const double t = x[k]; x[k] = x[p]; x[p] = t; }
    }
  __syncwarp();
  for (int k = 0; k < m; ++k) {  // unit lower
    const double xk = x[k];
    for (int r = k + 1 + lane; r < m; r += 32) x[r] = fma(-F[(int64_t)r * ld + k], xk, x[r]);
    __syncwarp();
  }
  for (int k = m - 1; k >= 0; --k) {  // upper
    const double xk = x[k] * rinv[k];
    __syncwarp();
    if (lane == 0) x[k] = xk;
    for (int r = lane; r < k; r += 32) x[r] = fma(-F[(int64_t)r * ld + k], xk, x[r]);
    __syncwarp();
  }
}

// y <- M^{-T} y with M = P^T L U:  U^T z = y, L^T w = z, y = P^T w; by one warp.
__device__ void lu_solve_transposed_f64(const double* F, int ld, const int32_t* piv,
                                        const double* rinv, int m, double* y) {
  const int lane = threadIdx.x & 31;
  for (int k = 0; k < m; ++k) {  // U^T is lower triangular
    const double yk = y[k] * rinv[k];
    __syncwarp();
    if (lane == 0) y[k] = yk;
    for (int r = k + 1 + lane; r < m; r += 32) y[r] = fma(-F[(int64_t)k * ld + r], yk, y[r]);
    __syncwarp();
  }
  for (int k = m - 1; k >= 0; --k) {  // L^T unit upper
    const double yk = y[k];
    for (int r = lane; r < k; r += 32) y[r] = fma(-F[(int64_t)k * ld + r], yk, y[r]);
    __syncwarp();
  }
  if (lane == 0)
    for (int k = m - 1; k >= 0; --k) {
      const int p = piv[k];
      if (p != k) { const double t = y[k]; y[k] = y[p]; y[p] = t; }
    }
  __syncwarp();
}

// g = dCl/du: g_i = 2 |h_i| / (v_inf c) for the strengths, 0 for C.
__device__ void cl_sensitivity_f64(const double* nodes, int n, double v, double c, double* g) {
  const int m = n + 1;
  for (int k = threadIdx.x; k < m; k += blockDim.x) {
    if (k < n) {
      int k1 = (k + 1 == n) ? 0 : k + 1;
      double hx = nodes[2 * k1] - nodes[2 * k], hy = nodes[2 * k1 + 1] - nodes[2 * k + 1];
      g[k] = 2.0 * sqrt(hx * hx + hy * hy) / (v * c);
    } else {
      g[k] = 0.0;
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kF64Threads) k_solve_f64(
    Batch bt, const double* __restrict__ A, double* __restrict__ LU, int32_t* __restrict__ piv,
    const double* __restrict__ rhs, const double* __restrict__ vinf,
    const double* __restrict__ chord, double* __restrict__ u, double* __restrict__ lambda,
    int32_t* __restrict__ info, int32_t* __restrict__ iters, int smem_m) {
  extern __shared__ double sm[];
  __shared__ PivotF64 sp;
  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b);
  const int m = n + 1;
  if (info[b] != 0) return;
  if (n > bt.n_max) {
    if (threadIdx.x == 0) info[b] = PANEL_INFO_TOO_LARGE;
    return;
  }
  const int mv = bt.n_max + 1;
  double *x = sm, *y = sm + mv, *rinv = sm + 2 * mv;
  const double* Ab = A + bt.mat_off[b];
  double* Fg = LU + bt.mat_off[b];
  int32_t* pv = piv + vec_off(bt, b);
  const bool staged = m <= smem_m;  // the matrix in shared memory, odd row stride
  const int ld = staged ? (m | 1) : m;
  double* F = staged ? sm + 3 * mv : Fg;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int r = warp; r < m; r += nw)
    for (int c = lane; c < m; c += 32) F[(int64_t)r * ld + c] = Ab[(int64_t)r * m + c];
  for (int k = threadIdx.x; k < m; k += blockDim.x) x[k] = rhs[vec_off(bt, b) + k];
  if (lambda)
    cl_sensitivity_f64(bt.nodes + 2 * bt.node_off[b], n, vinf ? vinf[b] : 1.0,
                       chord ? chord[b] : 1.0, y);
  __syncthreads();
  const int st = lu_factor_f64(F, ld, pv, rinv, m, &sp);
  if (st != 0) {
    if (threadIdx.x == 0) { info[b] = st; if (iters) iters[b] = 0; }
    return;
  }
  // both systems at once, a warp each; the others store the staged factor
  if (warp == 0)
    lu_solve_f64(F, ld, pv, rinv, m, x);
  else if (warp == 1) {
    if (lambda) lu_solve_transposed_f64(F, ld, pv, rinv, m, y);
  } else if (staged) {
    for (int r = warp - 2; r < m; r += nw - 2)
      for (int c = lane; c < m; c += 32) Fg[(int64_t)r * m + c] = F[(int64_t)r * ld + c];
  }
  __syncthreads();
  for (int k = threadIdx.x; k < m; k += blockDim.x) {
    u[vec_off(bt, b) + k] = x[k];
    if (lambda) lambda[vec_off(bt, b) + k] = y[k];
  }
  if (threadIdx.x == 0 && iters) iters[b] = 0;
}

// Fewer threads for smaller airfoils, so that several share an SM (512 of 20 panels:
// 102 us with 512 threads each).
static int solve_f64_threads(int mv) { return mv <= 64 ? 128 : mv <= 128 ? 256 : kF64Threads; }

cudaError_t launch_solve_f64(const Batch& bt, const double* A, double* LU, int32_t* piv,
                             const double* rhs, const double* vinf, const double* chord, double* u,
                             double* lambda, int32_t* info, int32_t* iters, cudaStream_t s) {
  const size_t mv = (size_t)bt.n_max + 1;
  const int smem_m = mv <= (size_t)kSmemF64M ? (int)mv : 0;
  const size_t smem = (3 * mv + (smem_m ? mv * (mv | 1) : 0)) * sizeof(double);
  cudaError_t e = ensure_smem(k_solve_f64, smem);
  if (e != cudaSuccess) return e;
  k_solve_f64<<<bt.B, solve_f64_threads((int)mv), smem, s>>>(bt, A, LU, piv, rhs, vinf, chord, u,
                                                             lambda, info, iters, smem_m);
  return cudaGetLastError();
}

// lambda of M^T lambda = dCl/du with the stored factor, a block per airfoil.
__global__ void __launch_bounds__(128) k_lambda_f64(Batch bt, const double* __restrict__ LU,
                                                    const int32_t* __restrict__ piv,
                                                    const double* __restrict__ vinf,
                                                    const double* __restrict__ chord,
                                                    double* __restrict__ lambda,
                                                    const int32_t* __restrict__ info) {
  extern __shared__ double sm[];
  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b), m = n + 1;
  if ((info && info[b] != 0) || n > bt.n_max || n < 3) return;
  double *y = sm, *rinv = sm + bt.n_max + 1;
  const double* F = LU + bt.mat_off[b];
  cl_sensitivity_f64(bt.nodes + 2 * bt.node_off[b], n, vinf ? vinf[b] : 1.0,
                     chord ? chord[b] : 1.0, y);
  for (int k = threadIdx.x; k < m; k += blockDim.x) rinv[k] = 1.0 / F[(int64_t)k * m + k];
  __syncthreads();
  if (threadIdx.x < 32) lu_solve_transposed_f64(F, m, piv + vec_off(bt, b), rinv, m, y);
  __syncthreads();
  for (int k = threadIdx.x; k < m; k += blockDim.x) lambda[vec_off(bt, b) + k] = y[k];
}

// ---------------------------------------------------------------------------
// Adjoint contraction (plain FP64)
// ---------------------------------------------------------------------------
//
// With G(p; a, b) = (1/2pi) int_a^b log|p - s| ds, M_ji = -G(x_{j+1/2}; x_i, x_{i+1}),
// in the frame t = (b-a)/L, n = t rotated by +90 degrees, xi = (p-a).t,
// eta = (p-a).n, l1 = log|p-a|^2, l2 = log|p-b|^2, theta the subtended angle:
//   2pi dG/dp = (l1 - l2)/2 t + theta n
//   2pi dG/db = l2/2 t + ((l1 - l2)/2 eta - theta xi)/L n
//   dG/da     = -dG/dp - dG/db            (translation invariance)
// and dCl/dx_k = dCl/dx_k|_u + lambda^T (db/dx_k - (dM/dx_k) u) becomes
//   (2/(v c)) (gamma_{k-1} t_{k-1} - gamma_k t_k)
//   + v/2 (-sin a, cos a) (lambda_{k-1} + lambda_k)
//   + 1/2 (lambda_{k-1} P_{k-1} + lambda_k P_k) + u_k Acol_k + u_{k-1} Bcol_{k-1}
// with P_j = sum_i u_i dG_ji/dp, Acol_i = sum_j lambda_j dG_ji/da,
// Bcol_i = sum_j lambda_j dG_ji/db (indices mod n).  On the own panel (i = j)
// theta is ambiguous (+-pi); it cancels between the terms, so it is set to 0.
//
// Block (x, y) takes the rows [rows y, rows y + rows) of airfoil order[x] against all
// of its panels, so that a small batch still uses every SM's FP64 pipe, the bound
// here; a warp takes 31 panels (lane l the distance to node i0 + l: neighbouring
// panels share its logarithm) and windows of four rows, whose sums over the lanes
// take 6 additions instead of 20.  Above kFixedF64N panels k_adjoint_prepare writes the
// terms without pair sums first and everything else goes in by FP64 atomics, so the
// last bits vary between runs.  Up to kFixedF64N panels (FIXED) the row ranges of an
// airfoil are a cluster: each block keeps its sums by warp, and the block that owns a
// node adds them up through distributed shared memory, all in a fixed order.
constexpr int kFixedF64N = 64;  // at most 6 blocks of 12 rows, 3 column blocks
constexpr int kAdjF64Threads = 256;

__device__ __forceinline__ double rowsum4_f64(const double (&v)[4], int lane) {
  const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0;
  double k0 = b4 ? v[2] : v[0], k1 = b4 ? v[3] : v[1];
  k0 += __shfl_xor_sync(0xffffffffu, b4 ? v[0] : v[2], 16);
  k1 += __shfl_xor_sync(0xffffffffu, b4 ? v[1] : v[3], 16);
  double k = b3 ? k1 : k0;
  k += __shfl_xor_sync(0xffffffffu, b3 ? k0 : k1, 8);
  k += __shfl_xor_sync(0xffffffffu, k, 4);
  k += __shfl_xor_sync(0xffffffffu, k, 2);
  return k + __shfl_xor_sync(0xffffffffu, k, 1);
}

template <bool FIXED>
__global__ void __launch_bounds__(kAdjF64Threads) k_adjoint_f64(
    Batch bt, const double* __restrict__ u, const double* __restrict__ lambda,
    const double* __restrict__ alpha, const double* __restrict__ vinf,
    const double* __restrict__ chord, const double* __restrict__ grad_cl,
    double* __restrict__ grad, const int32_t* __restrict__ info, int rows) {
  extern __shared__ double sm[];  // the rows' control points, lambda, and P: 5 x rows
  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b);
  const int j0 = blockIdx.y * rows;
  double* gout = grad + 2 * bt.node_off[b];
  if ((info && info[b] != 0) || n > bt.n_max || n < 3) {  // (the whole cluster)
    if (FIXED)
      for (int k = blockIdx.y * kAdjF64Threads + threadIdx.x; k < 2 * n;
           k += gridDim.y * kAdjF64Threads)
        gout[k] = nan("");
    return;
  }
  if (!FIXED && j0 >= n) return;
  const int nr = max(0, min(rows, n - j0));
  double *px = sm, *py = sm + rows, *lam = sm + 2 * rows, *P = sm + 3 * rows;
  double* Pc = sm + 5 * rows;   // FIXED: P by column block, 3 x 2 rows
  double* T = Pc + 6 * rows;    // FIXED: 6 (rows + 1): P, A, B of a panel
  double* Cs = T + 6 * (rows + 1);  // FIXED: S, B by part and panel, 8 x 32 x 4
  const double* nodes = bt.nodes + 2 * bt.node_off[b];
  const double* ub = u + vec_off(bt, b);
  const double* lb = lambda + vec_off(bt, b);
  const double gscale = grad_cl ? grad_cl[b] : 1.0, w2pi = gscale * kInvTwoPi;
  for (int k = threadIdx.x; k < nr; k += kAdjF64Threads) {
    const int j = j0 + k, j1 = (j + 1 == n) ? 0 : j + 1;
    px[k] = 0.5 * (nodes[2 * j] + nodes[2 * j1]);
    py[k] = 0.5 * (nodes[2 * j + 1] + nodes[2 * j1 + 1]);
    lam[k] = lb[j];
    P[2 * k] = P[2 * k + 1] = 0.0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = kAdjF64Threads / 32;
  // 32 panels a warp, each with both of its logarithms, where that saves a whole group
  // of them (32, 63 and 64 panels; 4096 of 64 panels 5172 -> 4491 us)
  const int W = FIXED && (n == 32 || n > 62) ? 32 : 31;
  const int ncb = (n + W - 1) / W;
  // the warps: column blocks, and equal parts of the rows (whole windows) when there
  // are fewer column blocks than warps
  const int parts = max(1, min(nw / ncb, (nr + 3) >> 2));
  const int per = ((((nr + 3) >> 2) + parts - 1) / parts) * 4;
  for (int t = warp; t < ncb * parts; t += nw) {
    const int i = W * (t % ncb) + lane, r0 = (t / ncb) * per, r1 = min(nr, r0 + per);
    const bool ok = lane < W && i < n;
    const int k = i < n ? i : (i == n ? 0 : n - 1), k1 = (k + 1 == n) ? 0 : k + 1;  // x_n = x_0
    const double ax = nodes[2 * k], ay = nodes[2 * k + 1];
    const double hx = nodes[2 * k1] - ax, hy = nodes[2 * k1 + 1] - ay;
    const double L = sqrt(hx * hx + hy * hy), iL = 1.0 / L, tx = hx * iL, ty = hy * iL;
    const double ui = ok ? ub[i] : 0.0;
    double Sx = 0, Sy = 0, Bx = 0, By = 0;
    for (int w0 = r0; w0 < r1; w0 += 4) {
      double vx[4], vy[4];
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        double gx = 0.0, gy = 0.0;
        if (w0 + q < r1) {
          const int r = w0 + q;
          const double dx = px[r] - ax, dy = py[r] - ay;
          const double l1 = log(dx * dx + dy * dy);
          double l2 = __shfl_down_sync(0xffffffffu, l1, 1);
          if (FIXED && W == 32) {
            const double ex = px[r] - nodes[2 * k1], ey = py[r] - nodes[2 * k1 + 1];
            l2 = log(ex * ex + ey * ey);
          }
          const double xi = dx * tx + dy * ty, eta = dy * tx - dx * ty;
          const double th = (i == j0 + r) ? 0.0 : atan2(eta * L, xi * (xi - L) + eta * eta);
          const double hd = 0.5 * (l1 - l2);
          // dG/dp and dG/db (without the 1/2pi), in global coordinates
          gx = hd * tx - th * ty;
          gy = hd * ty + th * tx;
          const double cn = (hd * eta - th * xi) * iL, h2 = 0.5 * l2, lj = lam[r];
          Sx = fma(lj, gx, Sx);
          Sy = fma(lj, gy, Sy);
          Bx = fma(lj, h2 * tx - cn * ty, Bx);
          By = fma(lj, h2 * ty + cn * tx, By);
        }
        vx[0] = vx[1]; vx[1] = vx[2]; vx[2] = vx[3]; vx[3] = ui * gx;
        vy[0] = vy[1]; vy[1] = vy[2]; vy[2] = vy[3]; vy[3] = ui * gy;
      }
      const double sx = rowsum4_f64(vx, lane), sy = rowsum4_f64(vy, lane);
      const int r = w0 + (lane >> 3);
      if ((lane & 7) == 0 && r < r1) {
        if (FIXED) {
          double* q = Pc + 2 * ((t % ncb) * rows + r);
          q[0] = sx;
          q[1] = sy;
        } else {
          atomicAdd(&P[2 * r], sx);
          atomicAdd(&P[2 * r + 1], sy);
        }
      }
    }
    if (FIXED) {
      double* q = Cs + 4 * (32 * t + lane);
      q[0] = Sx;
      q[1] = Sy;
      q[2] = Bx;
      q[3] = By;
    } else if (ok) {
      // u_i A_i belongs to node i (start of panel i), u_i B_i to node i + 1;
      // A_i = -S_i - B_i
      const double f = w2pi * ui;
      atomicAdd(&gout[2 * i], -f * (Sx + Bx));
      atomicAdd(&gout[2 * i + 1], -f * (Sy + By));
      atomicAdd(&gout[2 * k1], f * Bx);
      atomicAdd(&gout[2 * k1 + 1], f * By);
    }
  }
  __syncthreads();
  if constexpr (FIXED) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int nz = gridDim.y, tid = threadIdx.x;
    // the column blocks of row `tid`; the parts of panel `tid`, into part 0's place
    if (tid < 2 * nr) {
      double v = Pc[tid];
      for (int q = 1; q < ncb; ++q) v += Pc[2 * q * rows + tid];
      P[tid] = v;
    }
    for (int e = tid; e < 4 * 32 * ncb; e += kAdjF64Threads)
      for (int q = 1; q < parts; ++q) Cs[e] += Cs[4 * 32 * ncb * q + e];
    cl.sync();
    // the sums of the panels j0 - 1 .. j0 + nr - 1, whose ends are the block's nodes
    for (int t = tid; t <= nr && nr > 0; t += kAdjF64Threads) {
      const int q = (j0 + t == 0) ? n - 1 : j0 + t - 1, at = 4 * (32 * (q / W) + q % W);
      double v[4];
      for (int e = 0; e < 4; ++e) {
        v[e] = cl.map_shared_rank(Cs, 0)[at + e];
        for (int z = 1; z < nz; ++z) v[e] += cl.map_shared_rank(Cs, z)[at + e];
      }
      const double* Pq = cl.map_shared_rank(P, q / rows) + 2 * (q % rows);
      double* o = T + 6 * t;
      o[0] = Pq[0];
      o[1] = Pq[1];
      o[2] = -(v[0] + v[2]);  // A_i = -S_i - B_i
      o[3] = -(v[1] + v[3]);
      o[4] = v[2];
      o[5] = v[3];
    }
    cl.sync();  // (a barrier of the block; and no block leaves while others read it)
    for (int t = tid; t < nr; t += kAdjF64Threads) {
      const int k = j0 + t, km = (k == 0) ? n - 1 : k - 1;
      const double *m = T + 6 * t, *o = m + 6;  // panels k - 1 and k
      double ex, ey, gx, gy;
      node_terms(nodes, ub, lb, n, k, vinf ? vinf[b] : 1.0, chord ? chord[b] : 1.0, alpha[b], ex,
                 ey, gx, gy);
      gx += kInvTwoPi * (0.5 * (lb[km] * m[0] + lb[k] * o[0]) + ub[k] * o[2] + ub[km] * m[4]);
      gy += kInvTwoPi * (0.5 * (lb[km] * m[1] + lb[k] * o[1]) + ub[k] * o[3] + ub[km] * m[5]);
      gout[2 * k] = gscale * (ex + gx);
      gout[2 * k + 1] = gscale * (ey + gy);
    }
  } else {
    for (int k = threadIdx.x; k < nr; k += kAdjF64Threads) {
      // lambda_j P_j / 2 belongs to the nodes j and j + 1 (the ends of panel j)
      const int j = j0 + k, j1 = (j + 1 == n) ? 0 : j + 1;
      const double f = 0.5 * w2pi * lam[k];
      atomicAdd(&gout[2 * j], f * P[2 * k]);
      atomicAdd(&gout[2 * j + 1], f * P[2 * k + 1]);
      atomicAdd(&gout[2 * j1], f * P[2 * k]);
      atomicAdd(&gout[2 * j1 + 1], f * P[2 * k + 1]);
    }
  }
}

// Kernels of launch_adjoint_f64 with a given lambda.
int adjoint_f64_launches(int n_max) { return n_max > kFixedF64N ? 2 : 1; }

cudaError_t launch_adjoint_f64(const Batch& bt, const double* LU, const int32_t* piv,
                               const double* u, const double* lambda_in, double* lambda_out,
                               const double* alpha, const double* vinf, const double* chord,
                               const double* grad_cl, double* grad, const int32_t* info,
                               cudaStream_t s) {
  const double* lam = lambda_in;
  cudaError_t e;
  if (!lam) {
    k_lambda_f64<<<bt.B, 128, 2 * ((size_t)bt.n_max + 1) * sizeof(double), s>>>(
        bt, LU, piv, vinf, chord, lambda_out, info);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    lam = lambda_out;
  }
  const int rows = f64_rows(bt.B, bt.n_max), nz = (bt.n_max + rows - 1) / rows;
  if (bt.n_max <= kFixedF64N) {
    const size_t smem = ((size_t)rows * 11 + 6 * (rows + 1) + 8 * 32 * 4) * sizeof(double);
    e = ensure_smem(k_adjoint_f64<true>, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg =
        cluster_config(dim3(bt.B, nz), dim3(1, nz), kAdjF64Threads, smem, s, &at);
    return cudaLaunchKernelEx(&cfg, k_adjoint_f64<true>, bt, u, lam, alpha, vinf, chord, grad_cl,
                              grad, info, rows);
  }
  e = launch_adjoint_prepare(bt, u, lam, alpha, vinf, chord, grad_cl, grad, info, false, s);
  if (e != cudaSuccess) return e;
  const size_t smem = (size_t)rows * 5 * sizeof(double);
  e = ensure_smem(k_adjoint_f64<false>, smem);
  if (e != cudaSuccess) return e;
  k_adjoint_f64<false><<<dim3(bt.B, nz), kAdjF64Threads, smem, s>>>(
      bt, u, lam, alpha, vinf, chord, grad_cl, grad, info, rows);
  return cudaGetLastError();
}

}  // namespace panel
