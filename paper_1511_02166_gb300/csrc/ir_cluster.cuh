// ir_cluster.cuh -- the refinement of a few airfoils: a thread-block cluster per
// airfoil (included by k_solve_mixed.cu, whose factor layouts, residual
// accumulators and right-hand sides it uses).
//
// k_ir_mixed gives an airfoil one block.  A batch of fewer airfoils than SMs then
// leaves most of the chip idle, and a large airfoil's sweeps wait on the loads of
// one SM (one of 1024 panels: 4.5 ms).  Here the C blocks of a cluster share the
// factor and the planes, and every block keeps the whole vectors, so that the
// short serial parts are done by each block for itself and only three kinds of
// results cross blocks, by remote shared-memory stores:
//   sweeps     per 32-row group, the 32 x S partial dot products of the forward
//              system (a row's columns are dealt out to S warps by groups) and
//              the 32 entries of the transposed one whose updates are complete (a
//              group's columns belong to one warp, which keeps their running
//              values); one cluster barrier, then every block forms the group's
//              32 results from the inverted diagonal block itself (one block
//              barrier).  The buffers alternate by group, so that a block may run
//              ahead into the next group's products;
//   residuals  rows go to warps in pairs; the 32-column chunks of the transposed
//              system are cut into row ranges when there are more warps than
//              chunks, their partial accumulators merged by the chunk's owner.
// Each sum's terms are those of k_ir_mixed in another grouping.
#pragma once
#include <cooperative_groups.h>

namespace panel {

namespace cg = cooperative_groups;

constexpr int kIrClThreads = 1024, kIrClWarps = kIrClThreads / 32;
constexpr int kIrClSlots = 32;  // 32-lane partial accumulators per block

// One lane's share of sum_k p[k stride] y[32 k] over the block's parts k = k0 + rank,
// k0 + rank + C, ... < k1 (of 32 columns each; p and y already offset by the lane,
// whose column 32 k + lane exists below `cols`).  Eight loads in flight: they sit in
// straight-line code, since a branch around each would leave one.
__device__ __forceinline__ float part_dot(const float* __restrict__ p, int64_t stride,
                                          const float* y, int k0, int k1, int C, int cols,
                                          int lane) {
  float a0 = 0.0f, a1 = 0.0f;
  for (int k = k0; k < k1; k += 8 * C) {
    float v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int kk = k + t * C;
      v[t] = (kk < k1 && 32 * kk + lane < cols) ? __ldg(p + kk * stride) : 0.0f;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int kk = k + t * C;
      if (kk < k1 && 32 * kk + lane < cols) {
        if (t & 1)
          a1 = fmaf(v[t], y[32 * kk], a1);
        else
          a0 = fmaf(v[t], y[32 * kk], a0);
      }
    }
  }
  return a0 + a1;
}

// Block `rank`'s share of row i (of group d) times y, over the columns before
// (down) or after the group.
__device__ __forceinline__ float row_part(const RmFactor& f, int d, int i, bool down,
                                          const float* y, int C, int rank, int lane) {
  const int c0 = down ? 0 : 32 * (d + 1), c1 = down ? 32 * d : f.m;
  return part_dot(f.F + (int64_t)i * f.m + c0 + lane, 32, y + c0 + lane, rank,
                  (c1 - c0 + 31) >> 5, C, c1 - c0, lane);
}
__device__ __forceinline__ float row_part(const CrFactor& f, int d, int i, bool down,
                                          const float* y, int C, int rank, int lane) {
  if (d < f.G0) {
    const int c0 = down ? 0 : f.k0(d) + f.kb(d), c1 = down ? 32 * d : f.m;
    return part_dot(f.F + (int64_t)i * f.m + c0 + lane, 32, y + c0 + lane, rank,
                    (c1 - c0 + 31) >> 5, C, c1 - c0, lane);
  }
  const int e = f.g.e, I = 1 + ((d - f.G0) >> 2), rr = (i - e) & (kTlB - 1), h = d - f.G0;
  float v = part_dot(f.chunk_row(I, rr) + lane, kTlChunk, y + e + lane,
                     (down ? 0 : h + 1) + rank, down ? h : f.nch, C, 1 << 30, lane);
  if (down) {
    const CrRag rag(f.F, f.g, I);
    for (int c = 32 * rank + lane; c < e; c += 32 * C) v = fmaf(rag(rr, c), y[c], v);
  }
  return v;
}

// acc - sum_{t < 8, t < pb} M[r0 + t][c] z[t] for the rows r0 + t of group d and
// column `lane` of group g (which exists), eight loads in flight.
__device__ __forceinline__ float col_part(const RmFactor& f, int d, int t0, int pb, int g,
                                          const float* z, float acc, int lane) {
  const float* p = f.F + (int64_t)(32 * d + t0) * f.m + 32 * g + lane;
  float v[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) v[t] = t < pb ? __ldg(p + (int64_t)t * f.m) : 0.0f;
#pragma unroll
  for (int t = 0; t < 8; ++t)
    if (t < pb) acc = fmaf(-v[t], z[t], acc);
  return acc;
}
__device__ __forceinline__ float col_part(const CrFactor& f, int d, int t0, int pb, int g,
                                          const float* z, float acc, int lane) {
  const bool rowmajor = d < f.G0;
  const int I = rowmajor ? 0 : 1 + ((d - f.G0) >> 2), rr = 32 * ((d - f.G0) & 3) + t0;
  float v[8];
  if (rowmajor || g >= f.G0) {
    const float* p = rowmajor ? f.F + (int64_t)(f.k0(d) + t0) * f.m + f.k0(g) + lane
                              : f.chunk_row(I, rr) + (int64_t)(g - f.G0) * kTlChunk + lane;
    const int step = rowmajor ? f.m : kTlC;
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = t < pb ? __ldg(p + (int64_t)t * step) : 0.0f;
  } else {
    const CrRag rag(f.F, f.g, I);
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = t < pb ? rag(rr + t, 32 * g + lane) : 0.0f;
  }
#pragma unroll
  for (int t = 0; t < 8; ++t)
    if (t < pb) acc = fmaf(-v[t], z[t], acc);
  return acc;
}

struct IrClSmem {
  double* red;   // converged_words
  double* dprev; // 2
  double* x[2];  // m each
  float *y, *z;  // m: the corrections
  float *xh[2], *xl[2], *r[2];  // m each
  int* perm;                    // m
  float* zp;                    // 4 x m: the transposed sweeps' running values
  float* ty;                    // 2 x 8 x 32: partial products of a group's rows
  float* tz;                    // 2 x 4 x 32: the parts of a group's running values
  ResAcc* part;                 // kIrClSlots x 32
};

__host__ __device__ inline size_t ir_cluster_smem(int n_max) {
  const size_t mv = (size_t)n_max + 1;
  return (size_t)(converged_words(kIrClThreads) + 2) * 8 + 2 * mv * 8 + 13 * mv * 4 + 2 * 8 * 32 * 4 + 2 * 4 * 32 * 4 + 16 +
         (size_t)kIrClSlots * 32 * sizeof(ResAcc);
}

// y <- U^{-1} L^{-1} y (fw) and / or z <- L^{-T} U^{-T} z (tr), by the cluster.
template <class Fac>
__device__ void cluster_sweeps(cg::cluster_group& cl, const Fac& f, bool fw, bool tr,
                               const IrClSmem& sm, int m, int C, int rank) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gw = rank * kIrClWarps + warp, GW = C * kIrClWarps;
  static_assert(kIrClWarps == 32, "a row of a group per warp");
  // forward: row `warp` of the group, the columns of the groups rank mod C
  // transposed: the rows [8 tp, 8 tp + 8) of the previous group, the columns of the
  // groups tg mod GW / 4; a running value per part
  const int tp = gw & 3, tg = gw >> 2, TG = GW >> 2;
  const int G = f.groups();
  float *y = sm.y, *z = sm.z, *zp = sm.zp + tp * m;
  for (int pass = 0; pass < 2; ++pass) {
    const bool down = pass == 0;
    if (tr) {
      for (int k = threadIdx.x; k < m; k += kIrClThreads) {
        sm.zp[k] = z[k];
        sm.zp[m + k] = sm.zp[2 * m + k] = sm.zp[3 * m + k] = 0.0f;
      }
      __syncthreads();
    }
    for (int s = 0; s < G; ++s) {
      const int d = down ? s : G - 1 - s;
      const int k0 = f.k0(d), kb = f.kb(d);
      float* ty = sm.ty + (s & 1) * 8 * 32;
      float* tz = sm.tz + (s & 1) * 4 * 32;
      // the group's diagonal block, needed after the barrier
      float xd = 0.0f, yd = 0.0f;
      if (warp < kb && lane < kb) {
        if (fw && (down ? lane < warp : lane >= warp)) xd = __ldg(f.diag_row(d, k0 + warp) + lane);
        if (tr && (down ? lane <= warp : lane > warp)) yd = __ldg(f.diag_row(d, k0 + lane) + warp);
      }
      if (fw && warp < kb) {
        float acc = warp_sum_f(row_part(f, d, k0 + warp, down, y, C, rank, lane));
        acc = (rank == 0 ? y[k0 + warp] : 0.0f) - acc;
        if (lane < C) *cl.map_shared_rank(ty + rank * 32 + warp, lane) = acc;
      }
      if (tr) {
        const int p = down ? d - 1 : d + 1;
        const int pk = s > 0 ? f.k0(p) + 8 * tp : 0, pb = s > 0 ? f.kb(p) - 8 * tp : 0;
        const int g1 = down ? G : d + 1;
        int g = tg;
        if (down && g < d) g += (d - g + TG - 1) / TG * TG;
        for (; g < g1; g += TG) {
          if (lane < f.kb(g)) {
            const int c = f.k0(g) + lane;
            float acc = zp[c];
            if (pb > 0) acc = col_part(f, p, 8 * tp, pb, g, z + pk, acc, lane);
            if (g == d)
              for (int k = 0; k < C; ++k) *cl.map_shared_rank(tz + tp * 32 + lane, k) = acc;
            else
              zp[c] = acc;
          }
        }
      }
      cl.sync();
      if (fw && warp < kb) {
        float t = 0.0f;
        for (int k = 0; k < C; ++k) t += ty[k * 32 + lane];
        // down: y_i = t_i + sum_{k<i} X[i][k] t_k (X unit lower); up: sum_{k>=i}
        const float tq = __shfl_sync(0xffffffffu, t, warp);
        const float v = warp_sum_f((lane < kb) ? xd * t : 0.0f);
        if (lane == 0) y[k0 + warp] = down ? tq + v : v;
      }
      if (tr && warp < kb) {
        const float t = (tz[lane] + tz[32 + lane]) + (tz[64 + lane] + tz[96 + lane]);
        const float tq = __shfl_sync(0xffffffffu, t, warp);
        const float v = warp_sum_f((lane < kb) ? yd * t : 0.0f);
        if (lane == 0) z[k0 + warp] = down ? v : tq + v;
      }
      __syncthreads();
    }
    // the last group's results are complete in every block; its buffers are
    // written again two groups later, beyond the next cluster barrier
    cl.sync();
  }
}

// Corrections with a Gauss-Jordan inverse X: y <- X y, z <- X^T z (w: m scratch).
__device__ inline void cluster_gj(cg::cluster_group& cl, const float* __restrict__ X, int m, bool fw,
                                  bool tr, float* y, float* z, float* w, int C, int rank) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gw = rank * kIrClWarps + warp, GW = C * kIrClWarps;
  for (int sys = 0; sys < 2; ++sys) {
    if (!(sys == 0 ? fw : tr)) continue;
    float* v = sys == 0 ? y : z;
    if (sys == 0) {
      for (int i = gw; i < m; i += GW) {
        float acc = 0.0f;
        for (int k = lane; k < m; k += 32) acc = fmaf(__ldg(X + i * m + k), v[k], acc);
        acc = warp_sum_f(acc);
        if (lane < C) *cl.map_shared_rank(w + i, lane) = acc;
      }
    } else {
      for (int cb = 32 * gw; cb < m; cb += 32 * GW) {
        const int i = cb + lane;
        float acc = 0.0f;
        if (i < m) {
#pragma unroll 4
          for (int k = 0; k < m; ++k) acc = fmaf(__ldg(X + k * m + i), v[k], acc);
          for (int c = 0; c < C; ++c) *cl.map_shared_rank(w + i, c) = acc;
        }
      }
    }
    cl.sync();
    for (int k = threadIdx.x; k < m; k += kIrClThreads) v[k] = w[k];
    cl.sync();
  }
}

// A right-hand side whose residuals go to every block.
struct ClusterRhs {
  const IrRhs& rhs;
  cg::cluster_group& cl;
  int C;
  __device__ double operator()(int k) const { return rhs(k); }
  __device__ void store(float* r, int k, double v) const {
    const float s = rhs.scaled(k, v);
    for (int c = 0; c < C; ++c) cl.map_shared_rank(r, c)[k] = s;
  }
};

// r0 = b - M x, r1 = g - M^T lambda (either system), into every block.
template <class Acc>
__device__ void cluster_residuals(cg::cluster_group& cl, const float* __restrict__ Ah,
                                  const float* __restrict__ Al, int m, bool fw, bool tr,
                                  const IrRhs& R0, const IrRhs& R1, const IrClSmem& sm, int C,
                                  int rank) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gw = rank * kIrClWarps + warp, GW = C * kIrClWarps;
  if (fw) {
    const float *xh = sm.xh[0], *xl = sm.xl[0];
    const ClusterRhs rhs{R0, cl, C};
    RowSums<Acc, ClusterRhs, float> sums(rhs, sm.r[0], gw, GW, m);
    for (int j = gw; j < m; j += GW) {
      Acc acc;
      resacc_init(acc);
      const float* h = Ah + (int64_t)j * m;
      const float* l = Al + (int64_t)j * m;
      for (int c0 = lane; c0 < m; c0 += 256) {
        float hv[8], lv[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const int c = c0 + 32 * t;
          hv[t] = c < m ? __ldg(h + c) : 0.0f;
          lv[t] = c < m ? __ldg(l + c) : 0.0f;
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const int c = c0 + 32 * t;
          if (c < m) resacc_add(acc, hv[t], lv[t], xh[c], xl[c]);
        }
      }
      sums.add(acc);
    }
    sums.finish();
  }
  if (tr) {
    const float *xh = sm.xh[1], *xl = sm.xl[1];
    const int nch = (m + 31) >> 5, own = (nch + C - 1) / C;
    const int S = max(1, min(min(16, GW / nch), kIrClSlots / own));  // row ranges per chunk
    Acc* part = reinterpret_cast<Acc*>(sm.part);
    for (int w = gw; w < nch * S; w += GW) {
      const int ch = w % nch, s = w / nch;
      const int c = 32 * ch + lane;
      const bool ok = c < m;
      const int j0 = (int)((int64_t)m * s / S), j1 = (int)((int64_t)m * (s + 1) / S);
      Acc acc;
      resacc_init(acc);
      for (int jb = j0; jb < j1; jb += 8) {
        float h[8], l[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const bool on = ok && jb + q < j1;
          h[q] = on ? __ldg(Ah + (int64_t)(jb + q) * m + c) : 0.0f;
          l[q] = on ? __ldg(Al + (int64_t)(jb + q) * m + c) : 0.0f;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (jb + q < j1) resacc_add(acc, h[q], l[q], xh[jb + q], xl[jb + q]);
      }
      if (S > 1) {
        *cl.map_shared_rank(part + ((ch / C) * S + s) * 32 + lane, ch % C) = acc;
      } else if (ok) {
        const float r = R1.scaled(c, resacc_sub_from(R1(c), acc));
        for (int k = 0; k < C; ++k) cl.map_shared_rank(sm.r[1], k)[c] = r;
      }
    }
    if (S > 1) {
      cl.sync();
      for (int o = warp; o * C + rank < nch; o += kIrClWarps) {
        const int c = 32 * (o * C + rank) + lane;
        if (c < m) {
          Acc acc = part[o * S * 32 + lane];
          for (int s = 1; s < S; ++s) resacc_merge(acc, part[(o * S + s) * 32 + lane]);
          const float r = R1.scaled(c, resacc_sub_from(R1(c), acc));
          for (int k = 0; k < C; ++k) cl.map_shared_rank(sm.r[1], k)[c] = r;
        }
      }
    }
  }
  cl.sync();
}

__global__ void __launch_bounds__(kIrClThreads, 1) k_ir_cluster(SolveArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const Batch& bt = a.bt;
  const int b = bt.order[blockIdx.x / C];
  const int n = airfoil_n(bt, b);
  const int m = n + 1;
  if (a.info[b] != 0 || n > bt.n_max) return;  // the whole cluster
  const int mv = bt.n_max + 1;
  IrClSmem sm;
  sm.red = reinterpret_cast<double*>(smraw);
  sm.dprev = sm.red + converged_words(kIrClThreads);
  sm.x[0] = sm.dprev + 2;
  sm.x[1] = sm.x[0] + mv;
  float* fp = reinterpret_cast<float*>(sm.x[1] + mv);
  sm.y = fp;
  sm.z = fp + mv;
  for (int q = 0; q < 2; ++q) {
    sm.xh[q] = fp + (2 + 3 * q) * mv;
    sm.xl[q] = fp + (3 + 3 * q) * mv;
    sm.r[q] = fp + (4 + 3 * q) * mv;
  }
  sm.perm = reinterpret_cast<int*>(fp + 8 * mv);
  sm.zp = fp + 9 * mv;
  sm.ty = fp + 13 * mv;
  sm.tz = sm.ty + 2 * 8 * 32;
  sm.part = reinterpret_cast<ResAcc*>(
      (reinterpret_cast<uintptr_t>(sm.tz + 2 * 4 * 32) + 15) & ~(uintptr_t)15);
  const int tid = threadIdx.x;
  const int64_t moff = bt.mat_off[b], vo = vec_off(bt, b);
  const float* Ah = a.A_hi + moff;
  const float* Al = a.A_lo + moff;
  const float* F = a.LU + moff;
  const int32_t* gpiv = a.piv + vo;
  const bool gj = gpiv_first(a, b) < 0;
  const bool cr = !gj && m > kLargeM;
  CrFactor crf;
  if (cr) crf.init(F, m, moff);
  const double s = border_scale(Ah, n, m, sm.red);
  const bool act[2] = {a.u != nullptr, a.lam != nullptr};
  IrRhs rhs[2];
  for (int q = 0; q < 2; ++q) rhs[q].init(a, b, n, q, s);
  for (int k = tid; k < m; k += kIrClThreads)
    for (int q = 0; q < 2; ++q)
      if (act[q]) {
        sm.x[q][k] = 0.0;
        sm.r[q][k] = rhs[q].scaled(k, rhs[q].eval(k));
      }
  factor_permutation(gpiv, m, gj, sm.perm);
  cl.sync();  // every block of the cluster runs before its memory is written

  bool conv[2] = {!act[0], !act[1]};
  int it = 0;
  for (;; ++it) {
    const bool run[2] = {!conv[0], !conv[1]};
    for (int k = tid; k < m; k += kIrClThreads) {
      if (run[0]) sm.y[k] = sm.r[0][sm.perm[k]];
      if (run[1]) sm.z[k] = sm.r[1][k];
    }
    __syncthreads();
    if (gj)
      cluster_gj(cl, F, m, run[0], run[1], sm.y, sm.z, sm.xh[0], C, rank);
    else if (cr)
      cluster_sweeps(cl, crf, run[0], run[1], sm, m, C, rank);
    else
      cluster_sweeps(cl, RmFactor{F, m}, run[0], run[1], sm, m, C, rank);
    unsigned long long dm[2] = {0, 0}, xm[2] = {0, 0};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (!run[q]) continue;
      const float* w = (q == 0) ? sm.y : sm.z;
      double* x = sm.x[q];
      for (int k = tid; k < m; k += kIrClThreads) {
        const int dst = (q == 0) ? k : sm.perm[k];
        const double d = (dst == n) ? (double)w[k] * s : (double)w[k];
        const double xn = x[dst] + d;
        x[dst] = xn;
        const df2 v = df_from_double(xn);
        sm.xh[q][dst] = v.hi;
        sm.xl[q][dst] = v.lo;
        dm[q] = max(dm[q], magnitude_bits(d));
        xm[q] = max(xm[q], magnitude_bits(xn));
      }
    }
    block_converged(dm, xm, run, it, a.tol, sm.dprev, conv, sm.red);  // as in k_ir_mixed
    if ((conv[0] && conv[1]) || it >= a.max_iter) break;
    if (it == 0)
      cluster_residuals<LiteAcc>(cl, Ah, Al, m, !conv[0], !conv[1], rhs[0], rhs[1], sm, C, rank);
    else
      cluster_residuals<ResAcc>(cl, Ah, Al, m, !conv[0], !conv[1], rhs[0], rhs[1], sm, C, rank);
  }
  __syncthreads();
  for (int k = rank * kIrClThreads + tid; k < m; k += C * kIrClThreads) {
    if (act[0]) a.u[vo + k] = sm.x[0][k];
    if (act[1]) a.lam[vo + k] = sm.x[1][k];
  }
  if (rank == 0 && tid == 0) {
    if (a.iters && act[0]) a.iters[b] = it;
    if (!(conv[0] && conv[1])) a.info[b] = PANEL_INFO_NOCONV;
  }
  cl.sync();  // no block leaves while another may still write to it
}

}  // namespace panel
