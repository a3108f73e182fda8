// k_assemble_df.cu -- mixed-precision assembly: the bordered system of Section 2
// in double-float, stored as two float32 planes A = A_hi + A_lo.
//
// k_assemble_df: one block per airfoil (launched in size order); further down the
// forms that spread an airfoil over several blocks (assemble_kind chooses).  Prologue: validate the
// geometry (FP64), build the per-panel constants in shared memory and stage the
// log/atan tables.  Main loop: pairs (j, i) in row-major order, consecutive
// threads on consecutive columns, so each warp writes contiguous runs of both
// planes.  The right-hand side phi_v(x_{j+1/2}) is FP64.
#include "panel_common.cuh"
#include "panel_df.cuh"

namespace panel {

__global__ void __launch_bounds__(256) k_assemble_df(Batch bt, const double* __restrict__ alpha,
                                                     const double* __restrict__ vinf,
                                                     float* __restrict__ A_hi,
                                                     float* __restrict__ A_lo,
                                                     double* __restrict__ rhs,
                                                     int32_t* __restrict__ info, int rounds) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int ld = bt.n_max;
  float4* tlog = reinterpret_cast<float4*>(smraw);                   // 257
  float2* tatan = reinterpret_cast<float2*>(tlog + 257);             // 33 (+1 pad)
  double* xs = reinterpret_cast<double*>(tatan + 34);                // n_max
  double* ys = xs + ld;                                              // n_max
  double* scratch = ys + ld;                                         // 32
  float* pc = reinterpret_cast<float*>(scratch + 32);                // 20 * n_max

  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b);
  const int m = n + 1;
  if (n > ld) {
    if (threadIdx.x == 0) info[b] = PANEL_INFO_TOO_LARGE;
    return;
  }
  const double* nodes = bt.nodes + 2 * bt.node_off[b];
  const int st = load_and_check_geometry(nodes, n, xs, ys, scratch);
  if (threadIdx.x == 0) info[b] = st;
  if (st != 0) return;
  df_stage_tables(tlog, tatan);
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const int k1 = (k + 1 == n) ? 0 : k + 1;
    panel_constants(pc, ld, k, xs[k], ys[k], xs[k1], ys[k1]);
  }
  const double v = vinf ? vinf[b] : 1.0;
  const double ca = cos(alpha[b]), sa = sin(alpha[b]);
  double* rb = rhs + vec_off(bt, b);
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    if (j < n) {
      const int j1 = (j + 1 == n) ? 0 : j + 1;
      rb[j] = v * (0.5 * (ys[j] + ys[j1]) * ca - 0.5 * (xs[j] + xs[j1]) * sa);
    } else {
      rb[j] = 0.0;
    }
  }
  __syncthreads();

  const int64_t base = bt.mat_off[b];
  float* Ah = A_hi + base;
  float* Al = A_lo + base;
  // border: C column of ones and the Kutta row (gamma_0 + gamma_{n-1} = 0)
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    if (j < n) {
      Ah[(int64_t)j * m + n] = 1.0f;
      Al[(int64_t)j * m + n] = 0.0f;
    }
    Ah[(int64_t)n * m + j] = (j == 0 || j == n - 1) ? 1.0f : 0.0f;
    Al[(int64_t)n * m + j] = 0.0f;
  }
  // pairs (j, i), j, i < n, row-major over the threads of the block, in rounds of
  // `rounds` pairs per thread: the far-field pairs are evaluated at once, the
  // near-field ones (|P| < 4 L) queued and then evaluated by all threads
  // together, so that no warp runs both forms for a mix of its lanes
  // (rounds == 0: both forms inline, for the largest airfoils, whose one block
  // per SM cannot afford the barriers)
  int* queue = reinterpret_cast<int*>(pc + kPanelFields * ld);  // blockDim.x * rounds
  int* qn = queue + blockDim.x * rounds;
  const int stride = blockDim.x;
  const int dj = stride / n, di = stride % n;
  int j = threadIdx.x / n, i = threadIdx.x % n;
  point3 pj = load_point(pc, ld, j < n ? j : 0);
  if (rounds == 0) {
    while (j < n) {
      const df2 g = panel_G_df<0>(pair_geom(pj, pc, ld, i), pc, ld, i, tlog, tatan);
      const int64_t e = (int64_t)j * m + i;
      Ah[e] = -g.hi;
      Al[e] = -g.lo;
      const int jo = j;
      i += di;
      j += dj;
      if (i >= n) {
        i -= n;
        ++j;
      }
      if (j != jo && j < n) pj = load_point(pc, ld, j);
    }
    return;
  }
  const int np = n * n;
  for (int p0 = 0; p0 < np; p0 += stride * rounds) {
    if (threadIdx.x == 0) *qn = 0;
    __syncthreads();
    for (int r = 0; r < rounds && j < n; ++r) {
      const PairGeom gm = pair_geom(pj, pc, ld, i);
      if (gm.far()) {
        const df2 g = panel_G_df<1>(gm, pc, ld, i, tlog, tatan);
        const int64_t e = (int64_t)j * m + i;
        Ah[e] = -g.hi;
        Al[e] = -g.lo;
      } else {
        queue[atomicAdd(qn, 1)] = j * n + i;
      }
      const int jo = j;
      i += di;
      j += dj;
      if (i >= n) {
        i -= n;
        ++j;
      }
      if (j != jo && j < n) pj = load_point(pc, ld, j);
    }
    __syncthreads();
    const int cnt = *qn;
    for (int t = threadIdx.x; t < cnt; t += stride) {
      const int pq = queue[t];
      const int jq = pq / n, iq = pq - jq * n;
      const PairGeom gm = pair_geom(load_point(pc, ld, jq), pc, ld, iq);
      const df2 g = panel_G_df<2>(gm, pc, ld, iq, tlog, tatan);
      const int64_t e = (int64_t)jq * m + iq;
      Ah[e] = -g.hi;
      Al[e] = -g.lo;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Several blocks per airfoil: k_assemble_prepare validates the geometry and
// writes info, the right-hand side and the border; then the pairs are spread
// over blocks that hold the constants of their own panels only (~120 FP64
// operations a panel, on a pipe of 1/74 of the FP32 rate).
// ---------------------------------------------------------------------------
constexpr int kPrepThreads = 128;
__global__ void __launch_bounds__(kPrepThreads) k_assemble_prepare(
    Batch bt, const double* __restrict__ alpha, const double* __restrict__ vinf,
    float* __restrict__ A_hi, float* __restrict__ A_lo, double* __restrict__ rhs,
    int32_t* __restrict__ info) {
  __shared__ double scratch[32];
  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b);
  const int m = n + 1;
  if (n > bt.n_max || n < 3) {
    if (threadIdx.x == 0) info[b] = n < 3 ? PANEL_INFO_FEW_NODES : PANEL_INFO_TOO_LARGE;
    return;
  }
  const double* nodes = bt.nodes + 2 * bt.node_off[b];
  const double v = vinf ? vinf[b] : 1.0;
  const double ca = cos(alpha[b]), sa = sin(alpha[b]);
  double* rb = rhs + vec_off(bt, b);
  float* Ah = A_hi + bt.mat_off[b];
  float* Al = A_lo + bt.mat_off[b];
  int bad = 0, zero = 0;
  double area = 0.0;
  for (int k = threadIdx.x; k < m; k += kPrepThreads) {
    if (k < n) {
      const int k1 = (k + 1 == n) ? 0 : k + 1;
      const double x = nodes[2 * k], y = nodes[2 * k + 1], x1 = nodes[2 * k1],
                   y1 = nodes[2 * k1 + 1];
      if (!(fabs(x) < kCoordLimit) || !(fabs(y) < kCoordLimit)) bad = 1;  // also NaN/inf
      if (x1 - x == 0.0 && y1 - y == 0.0) zero = 1;
      area += x * y1 - x1 * y;
      rb[k] = v * (0.5 * (y + y1) * ca - 0.5 * (x + x1) * sa);
      // the C column of ones and the Kutta row (gamma_0 + gamma_{n-1} = 0)
      Ah[(int64_t)k * m + n] = 1.0f;
      Al[(int64_t)k * m + n] = 0.0f;
    } else {
      rb[k] = 0.0;
    }
    Ah[(int64_t)n * m + k] = (k == 0 || k == n - 1) ? 1.0f : 0.0f;
    Al[(int64_t)n * m + k] = 0.0f;
  }
  bad = __syncthreads_or(bad);
  zero = __syncthreads_or(zero);
  area = block_sum(area, scratch);
  if (threadIdx.x == 0)
    info[b] = bad ? PANEL_INFO_NONFINITE
                  : zero ? PANEL_INFO_ZERO_PANEL : area > 0.0 ? 0 : PANEL_INFO_ORIENTATION;
}

// Small batches: block (x, y, z) takes the panels [64 y, 64 y + 64) of airfoil
// order[x] against the control points [16 z, 16 z + 16); warps 0 and 2 the first 32
// columns, 1 and 3 the others, on alternating rows.
constexpr int kAsmCols = 64, kAsmRows = 16, kAsmThreads = 128;

__global__ void __launch_bounds__(kAsmThreads) k_assemble_df_split(
    Batch bt, float* __restrict__ A_hi, float* __restrict__ A_lo,
    const int32_t* __restrict__ info) {
  __shared__ float4 tlog[257];
  __shared__ float2 tatan[34];
  __shared__ float pc[kPanelFields * kAsmCols];
  constexpr int rows = kAsmRows;
  __shared__ float pts[6 * rows];  // the split coordinates of the rows' points
  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b);
  const int m = n + 1;
  const int i0 = blockIdx.y * kAsmCols, j0 = blockIdx.z * rows;
  if (i0 >= n || j0 >= n || info[b] != 0) return;
  const double* nodes = bt.nodes + 2 * bt.node_off[b];
  df_stage_tables(tlog, tatan);
  const int nc = min(kAsmCols, n - i0), nr = min(rows, n - j0);
  for (int k = threadIdx.x; k < nc; k += kAsmThreads) {
    const int i = i0 + k, i1 = (i + 1 == n) ? 0 : i + 1;
    panel_constants(pc, kAsmCols, k, nodes[2 * i], nodes[2 * i + 1], nodes[2 * i1],
                    nodes[2 * i1 + 1]);
  }
  for (int k = threadIdx.x; k < nr; k += kAsmThreads) {
    const int j = j0 + k, j1 = (j + 1 == n) ? 0 : j + 1;
    const point3 p = make_point(0.5 * (nodes[2 * j] + nodes[2 * j1]),
                                0.5 * (nodes[2 * j + 1] + nodes[2 * j1 + 1]));
    pts[k] = p.xh;
    pts[rows + k] = p.xm;
    pts[2 * rows + k] = p.xl;
    pts[3 * rows + k] = p.yh;
    pts[4 * rows + k] = p.ym;
    pts[5 * rows + k] = p.yl;
  }
  float* Ah = A_hi + bt.mat_off[b];
  float* Al = A_lo + bt.mat_off[b];
  __syncthreads();
  const int il = threadIdx.x & (kAsmCols - 1);
  if (il >= nc) return;
  for (int k = threadIdx.x / kAsmCols; k < nr; k += kAsmThreads / kAsmCols) {
    point3 p;
    p.xh = pts[k];
    p.xm = pts[rows + k];
    p.xl = pts[2 * rows + k];
    p.yh = pts[3 * rows + k];
    p.ym = pts[4 * rows + k];
    p.yl = pts[5 * rows + k];
    const df2 g = panel_G_df<0>(pair_geom(p, pc, kAsmCols, il), pc, kAsmCols, il, tlog, tatan);
    const int64_t e = (int64_t)(j0 + k) * m + i0 + il;
    Ah[e] = -g.hi;
    Al[e] = -g.lo;
  }
}

// Each far-field pair's shared work done once for both of its entries.  For the
// control points c_j, c_i (the panel midpoints) the entries (j, i) and (i, j)
// have P = c_j - c_i and -P: |P|^2, 1/|P|^2, log|P| and P^2 are the same for
// both, exactly (the split coordinates make -P the exact negation of P); only the
// panel's orientation, length and scale differ (panel_G_far).  Every entry is
// computed by the same operations as in the other kernels, so all give the same
// matrix bit for bit.
//
// The panels are cut into chunks of C; block (x, p) takes the pair p = (I, J <= I)
// of chunks of airfoil order[x].  A warp takes 16 rows j x 32 columns i (lane =
// column) at a time and their mirror image: the row entries are written as they
// come, 128 bytes per warp; the mirror entries go through a 16-column staging
// tile, so that they too are written along rows (down a column each store is 32
// separate sectors, and the L2's write ports, not the arithmetic, were the limit
// with every SM at it).  Near-field entries (|P| < 4 L, decided per entry) are
// queued per warp and evaluated 32 at a time, so that no warp runs both forms
// for a mix of its lanes and no block barrier is needed.
constexpr int kTileRows = 16, kTileLd = kTileRows + 1, kTileQueue = 96;

template <int C>
constexpr size_t assemble_tiles_smem(int warps) {
  return 257 * 16 + 34 * 8 + (size_t)kPanelFields * 2 * C * 4 +
         (size_t)warps * (2 * 32 * kTileLd + kTileQueue) * 4;
}

template <int C, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_assemble_df_tiles(
    Batch bt, float* __restrict__ A_hi, float* __restrict__ A_lo,
    const int32_t* __restrict__ info) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int ld = 2 * C, NW = NT / 32, TC = C / 32;
  float4* tlog = reinterpret_cast<float4*>(smraw);        // 257
  float2* tatan = reinterpret_cast<float2*>(tlog + 257);  // 33 (+1 pad)
  float* pc = reinterpret_cast<float*>(tatan + 34);       // kPanelFields x (chunk I, chunk J)
  float* stage = pc + kPanelFields * ld;                  // per warp: 2 planes 32 x kTileLd
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* Th = stage + warp * (2 * 32 * kTileLd + kTileQueue);
  float* Tl = Th + 32 * kTileLd;
  unsigned* queue = reinterpret_cast<unsigned*>(Tl + 32 * kTileLd);

  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b);
  const int m = n + 1;
  int I = (int)((sqrtf(8.0f * blockIdx.y + 1.0f) - 1.0f) * 0.5f);
  if ((I + 1) * (I + 2) / 2 <= (int)blockIdx.y) ++I;
  if (I * (I + 1) / 2 > (int)blockIdx.y) --I;
  const int J = (int)blockIdx.y - I * (I + 1) / 2;
  const int i0 = I * C, j0 = J * C;
  if (i0 >= n || info[b] != 0) return;
  const double* nodes = bt.nodes + 2 * bt.node_off[b];
  df_stage_tables(tlog, tatan);
  const int jo = (I == J) ? 0 : C;  // chunk J's place in pc
  for (int t = threadIdx.x; t < (I == J ? C : ld); t += NT) {
    const int i = t < C ? i0 + t : j0 + t - C;
    if (i < n) {
      const int i1 = (i + 1 == n) ? 0 : i + 1;
      panel_constants(pc, ld, t, nodes[2 * i], nodes[2 * i + 1], nodes[2 * i1], nodes[2 * i1 + 1]);
    }
  }
  float* Ah = A_hi + bt.mat_off[b];
  float* Al = A_lo + bt.mat_off[b];
  __syncthreads();

  int cnt = 0;  // queued near-field entries of the warp
  auto flush = [&](int k) {  // evaluates the last k <= 32 of them
    __syncwarp();
    if (lane < k) {
      const unsigned code = queue[cnt - k + lane];
      const int rl = (int)(code & 0xffffu), cl = (int)(code >> 16);
      const int row = rl < C ? i0 + rl : j0 + rl - C, col = cl < C ? i0 + cl : j0 + cl - C;
      const df2 g = panel_G_df<2>(pair_geom(load_point(pc, ld, rl), pc, ld, cl), pc, ld, cl, tlog,
                                  tatan);
      Ah[(int64_t)row * m + col] = -g.hi;
      Al[(int64_t)row * m + col] = -g.lo;
    }
    cnt -= k;
    __syncwarp();
  };
  auto push = [&](bool on, unsigned code) {
    const unsigned mask = __ballot_sync(0xffffffffu, on);
    if (on) queue[cnt + __popc(mask & ((1u << lane) - 1u))] = code;
    cnt += __popc(mask);
  };

  for (int t = warp; t < 2 * TC * TC; t += NW) {
    const int ti = (t >> 1) / TC, tj = (t >> 1) % TC;
    const int jb = 32 * tj + kTileRows * (t & 1);  // first row within chunk J
    if ((I == J && tj > ti) || i0 + 32 * ti >= n || j0 + jb >= n) continue;
    const int il = 32 * ti + lane, i = i0 + il;
    const bool iok = i < n;
    const int ii = iok ? il : 32 * ti;
    const int jn = min(kTileRows, n - (j0 + jb));
    if (I == J && ti == tj) {  // a diagonal tile: every entry from its own row
      for (int r = 0; r < jn; ++r) {
        const int jl = jb + r;
        const PairGeom gm = pair_geom(load_point(pc, ld, jl), pc, ld, ii);
        const bool far = gm.far();
        if (__any_sync(0xffffffffu, far)) {
          const df2 g = panel_G_df<1>(gm, pc, ld, ii, tlog, tatan);
          if (iok && far) {
            const int64_t e = (int64_t)(j0 + jl) * m + i;
            Ah[e] = -g.hi;
            Al[e] = -g.lo;
          }
        }
        push(iok && !far, (unsigned)jl | ((unsigned)il << 16));
        while (cnt >= 32) flush(32);
      }
      continue;
    }
    const float Li = pc[kL * ld + ii];
    for (int r = 0; r < jn; ++r) {
      const int jl = jo + jb + r;
      const PairGeom gm = pair_geom(load_point(pc, ld, jl), pc, ld, ii);  // P = c_j - c_i
      const float Lj = pc[kL * ld + jl];
      const bool far_ji = gm.rho2.hi >= 16.0f * Li * Li;  // entry (j, i), panel i
      const bool far_ij = gm.rho2.hi >= 16.0f * Lj * Lj;  // entry (i, j), panel j
      // a near-field entry: NaN with a low word of 0 (an evaluated NaN has both)
      float th = __int_as_float(0x7fffffff), tl = 0.0f;
      if (__any_sync(0xffffffffu, far_ji || far_ij)) {
        const df2 X = df_sub(gm.px2, gm.py2);
        df2 Y = df_mul(gm.px, gm.py);
        Y.hi *= 2.0f;
        Y.lo *= 2.0f;
        const df2 inv = df_rcp(gm.rho2);
        const df2 inv2 = df_sqr(inv);
        df2 lg = df_log(gm.rho2, tlog);
        lg.hi *= 0.5f;
        lg.lo *= 0.5f;
        const df2 g = panel_G_far(X, Y, inv, inv2, lg, pc, ld, ii, Li);
        if (iok && far_ji) {
          const int64_t e = (int64_t)(j0 + jb + r) * m + i;
          Ah[e] = -g.hi;
          Al[e] = -g.lo;
        }
        const df2 h = panel_G_far(X, Y, inv, inv2, lg, pc, ld, jl, Lj);
        if (far_ij) {
          th = -h.hi;
          tl = -h.lo;
        }
      }
      Th[lane * kTileLd + r] = th;
      Tl[lane * kTileLd + r] = tl;
      if (__any_sync(0xffffffffu, iok && !(far_ji && far_ij))) {
        push(iok && !far_ji, (unsigned)jl | ((unsigned)il << 16));
        push(iok && !far_ij, (unsigned)il | ((unsigned)jl << 16));
        while (cnt >= 32) flush(32);
      }
    }
    __syncwarp();
    // the mirror entries along rows i: 2 rows x 16 columns per store
    const int jj = lane & (kTileRows - 1);
#pragma unroll 4
    for (int q = lane / kTileRows; q < 32; q += 32 / kTileRows) {
      const float th = Th[q * kTileLd + jj], tl = Tl[q * kTileLd + jj];
      if (jj < jn && i0 + 32 * ti + q < n && (th == th || tl != tl)) {
        const int64_t e = (int64_t)(i0 + 32 * ti + q) * m + j0 + jb + jj;
        Ah[e] = th;
        Al[e] = tl;
      }
    }
    __syncwarp();
  }
  flush(cnt);
}

// Pairs per thread between two near-field passes of k_assemble_df (the queue holds
// 256 x rounds pair indices, 16 KB); 0 above 1024 panels, where one block fits an
// SM and the barriers of the deferred pass cost more than the mixed branches.
// `sel` (the PANEL_TUNE_ROUNDS field of the flags) overrides it: 1 inline, 2..5
// rounds of 4, 8, 16 or 32 pairs.
static int assemble_rounds(int n_max, int sel) {
  static const int kSel[6] = {-1, 0, 4, 8, 16, 32};
  if (sel >= 1 && sel <= 5) return kSel[sel];
  return n_max <= 1024 ? 16 : 0;
}

static size_t assemble_df_smem(int n_max, int rounds) {
  return 257 * 16 + 34 * 8 + (size_t)(2 * n_max + 32) * 8 + (size_t)kPanelFields * n_max * 4 +
         ((size_t)256 * rounds + 1) * 4;
}

// Which kernel assembles a launch of B airfoils of at most n panels.  Measured (us,
// one block per airfoil / k_assemble_df_split / tiles of 64 / tiles of 128):
//   1 x 160  93 / 28 / 46 / 72      64 x 160  95 / 72 / 56 / 76
//   1 x 600  958 / 37 / 48 / 77     152 x 200  136 / 175 / 128 / 124
//   16 x 600  960 / 144 / 97 / 109  4096 x 200  2255 / - / 2737 / 2535
//   152 x 100  52 / 77 / 69 / 77    4096 x 256  3528 / - / 3455 / 3181
//   152 x 1024  2729 / 1750 / 1421 / 1369
// The split kernel fills the chip when even tiles of 64 leave SMs without a block;
// one block per airfoil is best for many airfoils of few panels, where most warps
// hold near-field pairs (one block / tiles of 64: 128 x 140  75 / 76, 140 x 140  74 / 81,
// 140 x 160  91 / 80); the pair-at-once tiles everywhere else.
enum AssembleKind { kAsmBlock, kAsmSplit, kAsmTiles64, kAsmTiles128 };
static AssembleKind assemble_kind(int B, int n_max, int sel, int sm_total) {
  if (sel >= 1 && sel <= 5) return kAsmBlock;
  if (sel == 6) return kAsmTiles128;
  if (n_max <= 64) return kAsmBlock;
  const long long sms = sm_total > 0 ? sm_total : 1;
  auto pairs = [&](int c) {
    const long long nch = (n_max + c - 1) / c;
    return B * (nch * (nch + 1) / 2);
  };
  if (pairs(64) <= sms) return kAsmSplit;
  if (n_max <= 128 || (n_max <= 144 && 4 * B > 3 * sms) || (n_max <= 224 && B > sms))
    return kAsmBlock;
  return pairs(128) <= 3 * sms ? kAsmTiles64 : kAsmTiles128;
}

// Kernels of launch_assemble_df.
int assemble_df_launches(int B, int n_max, int sel, int sms) {
  return assemble_kind(B, n_max, sel, sms) == kAsmBlock ? 1 : 2;
}

cudaError_t launch_assemble_df(const Batch& bt, const double* alpha, const double* vinf,
                               float* A_hi, float* A_lo, double* rhs, int32_t* info,
                               cudaStream_t s, int rounds_sel) {
  const AssembleKind kind = assemble_kind(bt.B, bt.n_max, rounds_sel, sm_count());
  if (kind == kAsmBlock) {
    int rounds = assemble_rounds(bt.n_max, rounds_sel);
    // a requested queue that does not fit the shared memory falls back to the default
    if (assemble_df_smem(bt.n_max, rounds) > 232448) rounds = assemble_rounds(bt.n_max, 0);
    const size_t smem = assemble_df_smem(bt.n_max, rounds);
    cudaError_t e = ensure_smem(k_assemble_df, smem);
    if (e != cudaSuccess) return e;
    k_assemble_df<<<bt.B, 256, smem, s>>>(bt, alpha, vinf, A_hi, A_lo, rhs, info, rounds);
    return cudaGetLastError();
  }
  k_assemble_prepare<<<bt.B, kPrepThreads, 0, s>>>(bt, alpha, vinf, A_hi, A_lo, rhs, info);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (kind == kAsmSplit) {
    const dim3 grid(bt.B, (bt.n_max + kAsmCols - 1) / kAsmCols,
                    (bt.n_max + kAsmRows - 1) / kAsmRows);
    k_assemble_df_split<<<grid, kAsmThreads, 0, s>>>(bt, A_hi, A_lo, info);
    return cudaGetLastError();
  }
  auto tiles = [&](auto kernel, int C, int nt, size_t smem) {
    const cudaError_t r = ensure_smem(kernel, smem);
    if (r != cudaSuccess) return r;
    const int nch = (bt.n_max + C - 1) / C;
    kernel<<<dim3(bt.B, nch * (nch + 1) / 2), nt, smem, s>>>(bt, A_hi, A_lo, info);
    return cudaGetLastError();
  };
  if (kind == kAsmTiles64)
    return tiles(k_assemble_df_tiles<64, 128, 6>, 64, 128, assemble_tiles_smem<64>(4));
  return tiles(k_assemble_df_tiles<128, 256, 3>, 128, 256, assemble_tiles_smem<128>(8));
}

// ---------------------------------------------------------------------------
// Diagnostic evaluation of the double-float primitives on arrays (panel_df_eval)
// ---------------------------------------------------------------------------
__global__ void k_df_eval(int op, int count, const double* __restrict__ a,
                          const double* __restrict__ b, double* __restrict__ out) {
  __shared__ float4 tlog[257];
  __shared__ float2 tatan[34];
  __shared__ float pc[kPanelFields * 256];  // 22.5 KB
  df_stage_tables(tlog, tatan);
  __syncthreads();
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  if (op == 0) {
    out[k] = df_to_double(df_log(df_from_double(a[k]), tlog));
  } else if (op == 1) {
    out[k] = df_to_double(df_atan2(df_from_double(a[k]), df_from_double(b[k]), tatan));
  } else {
    // op 2: A coefficient -G for control point a[2k..] and panel b[4k..4k+3]
    const int t = threadIdx.x;
    panel_constants(pc, 256, t, b[4 * k], b[4 * k + 1], b[4 * k + 2], b[4 * k + 3]);
    const df2 g = panel_G_df(make_point(a[2 * k], a[2 * k + 1]), pc, 256, t, tlog, tatan);
    out[k] = -df_to_double(g);
  }
}

cudaError_t launch_df_eval(int op, int count, const double* a, const double* b, double* out,
                           cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  k_df_eval<<<(count + 255) / 256, 256, 0, s>>>(op, count, a, b, out);
  return cudaGetLastError();
}

}  // namespace panel
