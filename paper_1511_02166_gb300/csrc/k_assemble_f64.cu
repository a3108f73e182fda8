// k_assemble_f64.cu -- plain FP64 assembly of the bordered panel system.
//
// Section 2 of the paper: A_ji = -F_i(x_{j+1/2}) / gamma_i with the closed-form
// panel integral, the C column of ones, the Kutta row gamma_0 + gamma_{n-1} = 0
// and b_j = v_inf (y_{j+1/2} cos a - x_{j+1/2} sin a).  The printed integral
// uses two log and two atan2 per pair; here the two atan2 of one pair are
// combined into one (their difference is the angle the panel subtends, always
// inside (-pi, pi)), and the logarithms are those of the distances to the two
// end nodes, which neighbouring panels share: one log and one atan2 per pair in
// native FP64.  The FP64 pipe (16 G log/s, 12 G atan2/s on the whole chip) is
// the bound; a block takes a range of rows, so that a batch of fewer airfoils
// than SMs still uses every SM's pipe.
#include "panel_common.cuh"

namespace panel {

// (1/2pi) * integral over the panel a->b of log|p - s| ds, in the panel frame
// xi = (p-a).t, eta = (p-a).n (n = t rotated by +90 degrees), L = |b-a|, with
// la = log|p-a|^2 and lb = log|p-b|^2:
//   G = (1/2pi) [ xi/2 la - (xi-L)/2 lb + eta*theta - L ],
//   theta = atan2(eta L, xi (xi - L) + eta^2).
__device__ __forceinline__ double panel_G_f64(double dx, double dy, double la, double lb,
                                              double tx, double ty, double L) {
  double xi = dx * tx + dy * ty;
  double eta = dy * tx - dx * ty;
  double xl = xi - L;
  double th = atan2(eta * L, xi * xl + eta * eta);
  return kInvTwoPi * (0.5 * xi * la - 0.5 * xl * lb + eta * th - L);
}

// Block (x, y): the rows [rows y, rows y + rows) of airfoil order[x].
__global__ void __launch_bounds__(256) k_assemble_f64(Batch bt, const double* __restrict__ alpha,
                                                      const double* __restrict__ vinf,
                                                      double* __restrict__ A,
                                                      double* __restrict__ rhs,
                                                      int32_t* __restrict__ info, int rows) {
  extern __shared__ double sm[];
  const int b = bt.order[blockIdx.x];
  const int n = airfoil_n(bt, b);
  const int m = n + 1;
  double* xs = sm;                 // nodes
  double* ys = xs + bt.n_max;
  double* txs = ys + bt.n_max;     // unit tangents of the panels
  double* tys = txs + bt.n_max;
  double* Ls = tys + bt.n_max;     // panel lengths
  double* mxs = Ls + bt.n_max;     // control points
  double* mys = mxs + bt.n_max;
  double* scratch = mys + bt.n_max;

  const double* nodes = bt.nodes + 2 * bt.node_off[b];
  const bool first = blockIdx.y == 0 && threadIdx.x == 0;
  if (n > bt.n_max) {
    if (first) info[b] = PANEL_INFO_TOO_LARGE;
    return;
  }
  const int j0 = blockIdx.y * rows;
  if (j0 > n && blockIdx.y > 0) return;
  int st = load_and_check_geometry(nodes, n, xs, ys, scratch);
  if (first) info[b] = st;
  if (st != 0) return;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    int k1 = (k + 1 == n) ? 0 : k + 1;
    double hx = xs[k1] - xs[k], hy = ys[k1] - ys[k];
    double L = sqrt(hx * hx + hy * hy);
    txs[k] = hx / L;
    tys[k] = hy / L;
    Ls[k] = L;
    mxs[k] = 0.5 * (xs[k] + xs[k1]);
    mys[k] = 0.5 * (ys[k] + ys[k1]);
  }
  __syncthreads();

  const double v = vinf ? vinf[b] : 1.0;
  const double ca = cos(alpha[b]), sa = sin(alpha[b]);
  double* Ab = A + bt.mat_off[b];
  double* rb = rhs + vec_off(bt, b);
  const int j1 = min(m, j0 + rows);
  for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x)
    rb[j] = (j < n) ? v * (mys[j] * ca - mxs[j] * sa) : 0.0;

  // the block's rows one after the other as n + 1 places each, the nodes and node 0
  // again; a warp takes 31 places at a time: lane l the distance to the node at place
  // s0 + l and, below lane 31, the panel from it to the next lane's node (by rows, 31
  // or fewer panels at a time, up to half of the lanes were idle: 4096 of 64 panels
  // 4424 us, now 3151; 3793 with two logarithms a panel and 32 at a time)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int places = (n + 1) * (min(j1, n) - j0);
  for (int s0 = 31 * warp; s0 < places; s0 += 31 * nw) {
    const int s = min(s0 + lane, places - 1), j = j0 + s / (n + 1), i = s % (n + 1);
    const int k = i < n ? i : 0;  // x_n = x_0
    const double dx = mxs[j] - xs[k], dy = mys[j] - ys[k];
    const double la = log(dx * dx + dy * dy);
    const double lb = __shfl_down_sync(0xffffffffu, la, 1);
    if (lane < 31 && i < n && s == s0 + lane)
      Ab[(int64_t)j * m + i] = -panel_G_f64(dx, dy, la, lb, txs[i], tys[i], Ls[i]);
  }
  for (int j = j0 + threadIdx.x; j < min(j1, n); j += blockDim.x) Ab[(int64_t)j * m + n] = 1.0;
  if (j1 == m)
    for (int i = threadIdx.x; i < m; i += blockDim.x)
      Ab[(int64_t)n * m + i] = (i == 0 || i == n - 1) ? 1.0 : 0.0;
}

size_t assemble_f64_smem(int n_max) { return (size_t)(7 * n_max + 32) * sizeof(double); }

cudaError_t launch_assemble_f64(const Batch& bt, const double* alpha, const double* vinf,
                                double* A, double* rhs, int32_t* info, cudaStream_t s) {
  size_t smem = assemble_f64_smem(bt.n_max);
  cudaError_t e = ensure_smem(k_assemble_f64, smem);
  if (e != cudaSuccess) return e;
  const int rows = f64_rows(bt.B, bt.n_max + 1);
  k_assemble_f64<<<dim3(bt.B, (bt.n_max + rows) / rows), 256, smem, s>>>(bt, alpha, vinf, A, rhs,
                                                                         info, rows);
  return cudaGetLastError();
}

}  // namespace panel
