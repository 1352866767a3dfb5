// Free-surface kernels (§3.1.1, §3.1.3, §3.3, §3.4 of arXiv 1512.02548), FP64, sm_103a.
//
//  * w̃ (eq. velocpot2).  On the tensor-product mesh the 2D mass is M = M_x ⊗ M_σ and
//    the σ-derivative (1/d)∂σΦ is continuous across x-element edges, so the surface row
//    of M⁻¹ S_z Φ reduces exactly to a per-column contraction
//        w̃(x_i) = Σ_l Σ_b c_{l,b} · (1/d_i) (2/Δσ_l) (D Φ_{i,l})_b,
//    with c_l = (Δσ_l/2) M · (M_σ⁻¹ e_top)|_layer l precomputed on the host.  No 2D mass
//    solve is needed; the result equals the global projection up to rounding.
//  * M' u = Σ_e Q_eᵀ R_e is solved by static condensation: the element interiors are
//    eliminated in the host tables (S_x f and the over-integrated Zakharov integrals are
//    formed condensed), the interface unknowns form a tridiagonal system (cyclic when
//    periodic) whose factors decay, so each block solves for its own elements from a
//    window of their neighbours (surface_device.cuh).
//  * The modal filter F = V̂SV̂⁻¹ acts per element on interior nodes only: the hat
//    modes are untouched, so shared end values are unchanged by construction.
#include "surface_device.cuh"

namespace semgb {

// The M' solves run per block of kRecElems elements: the block's window of condensed right-hand sides
// (its own elements and t.win + 1 more on either side) is enough for its interface unknowns
// (mass1d_window), so no block waits for another.
constexpr int kRecElems = 16, kRecThreads = 128, kRecCols = kRecThreads / 8;
__host__ __device__ static inline int rec_blocks(int Nx) { return (Nx + kRecElems - 1) / kRecElems; }

// Gradient recovery, latency bound, in one launch of two kinds of blocks.  The first nrec = Nx/16 take S_x of η
// and φ̃ (boundary rows for the whole window, kept in shared memory), the interface solves and their
// columns of ∂xη and ∂xφ̃; the others w̃ of 16 columns each: in the blocks of the solves it had made few
// blocks of high order work through hundreds of columns.  26×8, P = 12, called from the host: three launches
// 21 µs, w̃ in the solves' blocks 54, now 10; in a graph 16.6 and 11.3, 687×8 166 and 12.8.
__global__ void __launch_bounds__(kRecThreads) k_recover(SurfTables t, const double* __restrict__ Phi,
                                                         const double* __restrict__ eta,
                                                         const double* __restrict__ phis, double* __restrict__ w,
                                                         double* __restrict__ etax, double* __restrict__ phisx) {
  extern __shared__ double sm[];
  const int Nx = t.Nx, P = t.P, N = t.nif, W = t.win, nrec = rec_blocks(Nx);
  if ((int)blockIdx.x >= nrec) {
    const int col = ((int)blockIdx.x - nrec) * kRecCols + (threadIdx.x >> 3);
    wsurf_column8(t, Phi, eta, w, col < t.ncol ? col : -1, threadIdx.x & 7);
    return;
  }
  const int e0 = blockIdx.x * kRecElems, e1 = min(Nx, e0 + kRecElems), ne = e1 - e0;
  const int nwin = ne + 2 * W + 2;                    // elements e0 − W − 1 … e1 + W
  double* gl = sm;                                    // [2][nwin] left and right boundary rows
  double* gr = gl + 2 * nwin;
  double* ub = gr + 2 * nwin;                         // [2][kRecElems + 1]
  for (int k = threadIdx.x; k < 4 * nwin; k += blockDim.x) {
    const int i = k >> 2, fld = (k >> 1) & 1, end = k & 1;
    int ex = e0 - W - 1 + i;
    if (t.periodic) { ex %= Nx; if (ex < 0) ex += Nx; }
    const double v = (ex >= 0 && ex < Nx) ? sx_value(t, fld ? phis : eta, ex, end ? P : 0) : 0.0;
    (end ? gr : gl)[fld * nwin + i] = v;
  }
  const int c0 = e0 * P, c1 = e1 * P + ((!t.periodic && e1 == Nx) ? 1 : 0);
  __syncthreads();
  const int rh = threadIdx.x >> 5;
  if (rh < 2) {
    // unknown j of the window sits between its elements i = j − (e0 − W − 1) − 1 and i
    auto gfun = [&](int j) -> double {
      int d = j - (e0 - W);                           // position in the window, around the ring
      if (t.periodic) { d %= N; if (d < 0) d += N; }
      return gl[rh * nwin + d + 1] + gr[rh * nwin + d];
    };
    mass1d_window(t, gfun, e0, ne + 1, [&](int i, double u) { ub[rh * (kRecElems + 1) + i] = u; });
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 2 * (c1 - c0); k += blockDim.x) {
    const int fld = k >= c1 - c0 ? 1 : 0, col = c0 + k - fld * (c1 - c0);
    const int i = min((col - c0) / P, ne - 1), a = col - c0 - i * P;
    const double* u = ub + fld * (kRecElems + 1) + i;
    double v = a == 0 ? u[0] : u[1];
    if (a > 0 && a < P)
      v = sx_value(t, fld ? phis : eta, e0 + i, a) - (t.Z[a - 1] * u[0] + t.Z[P - 1 + a - 1] * u[1]);
    (fld ? phisx : etax)[col] = v;
  }
}

// M'u = Σ_e Q_eᵀ R_e from condensed right-hand sides, a block's columns from its own window.
__global__ void __launch_bounds__(kRecThreads) k_mass1d(SurfTables t, const double* __restrict__ R,
                                                        double* __restrict__ u0, double* __restrict__ u1) {
  __shared__ double ub[2 * (kRecElems + 1)];
  const int Nx = t.Nx, P = t.P, Q = P + 1;
  const int e0 = blockIdx.x * kRecElems, e1 = min(Nx, e0 + kRecElems), ne = e1 - e0;
  mass1d_windows(t, R, e0, e1, ub, kRecElems + 1);
  __syncthreads();
  const int c0 = e0 * P, nc = ne * P + ((!t.periodic && e1 == Nx) ? 1 : 0);
  for (int k = threadIdx.x; k < 2 * nc; k += blockDim.x) {
    const int fld = k >= nc ? 1 : 0, c = k - fld * nc;
    const int i = min(c / P, ne - 1);
    const double* u = ub + fld * (kRecElems + 1) + i;
    (fld ? u1 : u0)[c0 + c] = mass1d_value(t, R + ((size_t)fld * Nx + e0 + i) * Q, u[0], u[1], c - i * P);
  }
}

constexpr int kZakWarps = 4;

__global__ void __launch_bounds__(32 * kZakWarps) k_zak(SurfTables t, const double* __restrict__ eta,
                                                        const double* __restrict__ etax,
                                                        const double* __restrict__ phisx,
                                                        const double* __restrict__ w,
                                                        double* __restrict__ R) {
  __shared__ double sh[2 * kZakWarps][kSurfScratch];
  const int half = threadIdx.x >> 4, sub = threadIdx.x & 15, Q = t.P + 1;
  const int ex = blockIdx.x * 2 * kZakWarps + half;
  const bool active = ex < t.Nx;
  double* cv = sh[half] + 2 * kMaxQf;
  if (active && sub < Q) {
    const int c = scol(t, ex, sub);
    cv[sub] = eta[c];
    cv[Q + sub] = etax[c];
    cv[2 * Q + sub] = phisx[c];
    cv[3 * Q + sub] = w[c];
  }
  __syncwarp();
  zak_element16(t, R, ex, active, sub, sh[half]);
}

__global__ void k_filter(SurfTables t, double* __restrict__ q0, double* __restrict__ q1) {
  __shared__ double sh[kZakWarps][kSurfScratch];
  const int wid = threadIdx.x >> 5;
  const int ex = blockIdx.x * kZakWarps + wid;
  if (ex >= t.Nx) return;
  filter_element(t, q0, q1, ex, threadIdx.x & 31, sh[wid]);
}

__global__ void k_relax(SurfTables t, const double* __restrict__ eta, const double* __restrict__ phis,
                        double time, double inv_tau, double* __restrict__ de, double* __restrict__ dp) {
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= t.ncol) return;
  relax_column(t, eta, phis, time, inv_tau, de, dp, col);
}

__global__ void k_rk4(int stage, int n, double dt, double* __restrict__ eta, double* __restrict__ phis,
                      const double* __restrict__ ke, const double* __restrict__ kp,
                      double* __restrict__ ae, double* __restrict__ ap, double* __restrict__ se,
                      double* __restrict__ sp) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rk4_item(stage, dt, eta, phis, ke, kp, ae, ap, se, sp, i);
}

cudaError_t launch_recover(const SurfTables& t, const double* Phi, const double* eta, const double* phis, double* w,
                           double* etax, double* phisx, cudaStream_t s) {
  const size_t smem = sizeof(double) * (4 * (kRecElems + 2 * t.win + 2) + 2 * (kRecElems + 1));
  const int grid = rec_blocks(t.Nx) + (t.ncol + kRecCols - 1) / kRecCols;
  k_recover<<<grid, kRecThreads, smem, s>>>(t, Phi, eta, phis, w, etax, phisx);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_mass1d(const SurfTables& t, const double* R, double* u0, double* u1, cudaStream_t s) {
  k_mass1d<<<rec_blocks(t.Nx), kRecThreads, 0, s>>>(t, R, u0, u1);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_zakharov(const SurfTables& t, const double* eta, const double* etax,
                            const double* phisx, const double* w, double* R, cudaStream_t s) {
  k_zak<<<(t.Nx + 2 * kZakWarps - 1) / (2 * kZakWarps), 32 * kZakWarps, 0, s>>>(t, eta, etax, phisx, w, R);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_filter(const SurfTables& t, double* q0, double* q1, cudaStream_t s) {
  if (!t.filter_on) return cudaSuccess;
  k_filter<<<(t.Nx + kZakWarps - 1) / kZakWarps, 32 * kZakWarps, 0, s>>>(t, q0, q1);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_relax(const SurfTables& t, const double* eta, const double* phis, double time,
                         double inv_tau, double* de, double* dp, cudaStream_t s) {
  if (!(t.relax_left > 0.0) && !(t.relax_right > 0.0)) return cudaSuccess;
  k_relax<<<(t.ncol + 127) / 128, 128, 0, s>>>(t, eta, phis, time, inv_tau, de, dp);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rk4_stage(int stage, int n, double dt, double* eta, double* phis,
                             const double* keta, const double* kphis, double* acc_eta,
                             double* acc_phis, double* st_eta, double* st_phis, cudaStream_t s) {
  k_rk4<<<(n + 255) / 256, 256, 0, s>>>(stage, n, dt, eta, phis, keta, kphis, acc_eta, acc_phis,
                                        st_eta, st_phis);
  count_launch();
  return cudaGetLastError();
}

}  // namespace semgb
