// Device bodies of the free-surface operations (§3.1.1, §3.1.3, §3.3, §3.4, §2.2), shared by
// the stand-alone kernels (kernels_surface.cu) and the fused per-stage kernel
// (kernels_laplace.cu).  Each body computes one work item (a column, an element, a
// right-hand side); the callers decide which items a thread, warp or CTA takes.
#pragma once
#include "sem_internal.cuh"

namespace semgb {

constexpr int kMaxQf = 3 * kMaxP + 1;
// shared scratch of an element in the element bodies (zak, filter)
constexpr int kSurfScratch = 2 * kMaxQf + 4 * (kMaxP + 1);

__device__ __forceinline__ int scol(const SurfTables& t, int ex, int a) {
  int c = ex * t.P + a;
  return c >= t.ncol ? c - t.ncol : c;
}

// w̃ of column `col` by the 8 lanes of a warp with the same lane >> 3 (sub = lane & 7; every lane of the
// warp calls, col < 0: no column).  On the tensor-product mesh the 2D mass is M_x ⊗ M_σ and the
// σ-derivative (1/d)∂σΦ is continuous across x-element edges, so the surface row of
// M⁻¹S_zΦ (eq. velocpot2) is the per-column contraction
//     w̃ = (1/d) Σ_l Σ_b c_{l,b} (2/Δσ_l) (D Φ_l)_b,  c_l = (Δσ_l/2) M (M_σ⁻¹ e_top)|_l,
// whose weights are folded on the host into one weight per row, w̃ = (1/d) Σ_iz wrow_iz Φ_iz.
__device__ __forceinline__ void wsurf_column8(const SurfTables& t, const double* __restrict__ Phi,
                                              const double* __restrict__ eta, double* __restrict__ w,
                                              int col, int sub) {
  double acc = 0.0;
  if (col >= 0) {
    const double* phi = Phi + (size_t)col * t.nrow;
    for (int iz = sub; iz < t.nrow; iz += 8) acc = fma(t.wrow[iz], phi[iz], acc);
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (col >= 0 && sub == 0) w[col] = acc / (eta[col] + t.h[col]);
}

// The same by one thread (four partial sums: the chain of one would be Nrow FP64 latencies long).
__device__ __forceinline__ void wsurf_column1(const SurfTables& t, const double* __restrict__ Phi,
                                              const double* __restrict__ eta, double* __restrict__ w, int col) {
  const double* phi = Phi + (size_t)col * t.nrow;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  int iz = 0;
  for (; iz + 4 <= t.nrow; iz += 4)
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = fma(t.wrow[iz + q], phi[iz + q], a[q]);
  for (; iz < t.nrow; ++iz) a[0] = fma(t.wrow[iz], phi[iz], a[0]);
  w[col] = ((a[0] + a[1]) + (a[2] + a[3])) / (eta[col] + t.h[col]);
}

// M'u = Σ_e Q_eᵀ R_e (M' constant in time).  The element right-hand sides are stored condensed: the
// element interiors are eliminated on the host, in the tables, so that an item of an element's row a is
//   a = 0, P:      the boundary rows R_b − M_bi M_ii⁻¹ R_i (the interface right-hand side),
//   0 < a < P:     the particular interior part M_ii⁻¹ R_i,
// one dot product each.  Layout R[field][ex][a].

// S_x f = M·D f_e condensed (the Δx/2 and 2/Δx scales cancel in the boundary rows; the interior part
// takes 2/Δx); item k over [field][ex][a], two fields.
__device__ __forceinline__ double sx_value(const SurfTables& t, const double* __restrict__ f, int ex, int a) {
  const int Q = t.P + 1;
  double s = 0.0;
  for (int c = 0; c < Q; ++c) s = fma(t.SX[a * Q + c], __ldcg(f + scol(t, ex, c)), s);
  return (a == 0 || a == t.P) ? s : s * t.r2dx[ex];
}
__device__ __forceinline__ void sx_item(const SurfTables& t, const double* __restrict__ f0,
                                        const double* __restrict__ f1, double* __restrict__ R, int k) {
  const int Q = t.P + 1;
  const int fld = k / (t.Nx * Q), rem = k - fld * t.Nx * Q, ex = rem / Q, a = rem - ex * Q;
  R[k] = sx_value(t, fld == 0 ? f0 : f1, ex, a);
}

// Interface unknowns lo, lo+1, …, lo+cnt−1 (cyclic when periodic) of the condensed M' system, by one
// warp, from the right-hand side gfun(j), 0 ≤ j < N; store(i, u) receives unknown lo + i.
// The system's LDLᵀ factors decay, so the recurrences
//     y_j = g_j m_j − (e_{j−1} m_j) y_{j−1},        u_j = y_j − l_j u_{j+1}
// started t.win interfaces away from the first unknown wanted (and from zero) agree with the whole
// chain's.  For any element widths |l_j| = |e_j|/p_j ≤ |S01|/S00 = 1/(P+1), which makes (P+1)^−win < 1e-18
// for the second; the first has p_j ≥ Δx_{j−1}/2 (S11 − |S01|/(P+1)), so |e_{j−1}| m_j ≤ (P+1)/((P+1)² − 1): below 1e-18
// where the widths vary little, at most 7e-17 (order 2, every element far narrower than the one before it).
// Every CTA therefore solves for its own elements alone, without waiting for a solve of the whole chain
// elsewhere: an RK stage has four team barriers fewer and no 2049-unknown solve on two CTAs while the others wait.
// The periodic chain uses the cyclic factors (the fixed point of the pivot recurrence around the ring), no closure.
// Lanes hold chunks of c ≤ kWinRegs positions of the window; the composed affine maps are scanned
// over as many lanes as cover t.win positions.
constexpr int kWinRegs = 6;

template <class G, class Store>
__device__ __forceinline__ void mass1d_window(const SurfTables& t, G gfun, int lo, int cnt, Store store) {
  const int lane = threadIdx.x & 31, N = t.nif, W = t.win;
  const int len = cnt + 2 * W, c = (len + 31) >> 5;
  const unsigned full = 0xffffffffu;
  double al[kWinRegs], v[kWinRegs], cp[kWinRegs];
  int j = lo - W + lane * c;
  int jw = j;                                       // j around the ring
  if (t.periodic) { jw %= N; if (jw < 0) jw += N; }
#pragma unroll
  for (int q = 0; q < kWinRegs; ++q) {
    al[q] = v[q] = cp[q] = 0.0;
    if (q < c) {
      if (lane * c + q < len && jw >= 0 && jw < N) {
        al[q] = t.th_al[jw];
        v[q] = gfun(jw) * t.th_m[jw];
        cp[q] = -t.th_cp[jw];
      }
      ++jw;
      if (t.periodic && jw == N) jw = 0;
    }
  }
  double A = 1.0, B = 0.0;
#pragma unroll
  for (int q = 0; q < kWinRegs; ++q)
    if (q < c) { B = fma(al[q], B, v[q]); A *= al[q]; }
  for (int o = 1; o < 32 && o * c < W; o <<= 1) {
    const double Ap = __shfl_up_sync(full, A, o), Bp = __shfl_up_sync(full, B, o);
    if (lane >= o) { B = fma(A, Bp, B); A *= Ap; }
  }
  double y = __shfl_up_sync(full, B, 1);
  if (lane == 0) y = 0.0;
  A = 1.0;
#pragma unroll
  for (int q = 0; q < kWinRegs; ++q)
    if (q < c) { y = fma(al[q], y, v[q]); v[q] = y; }
  B = 0.0;
#pragma unroll
  for (int q = kWinRegs - 1; q >= 0; --q)
    if (q < c) { B = fma(cp[q], B, v[q]); A *= cp[q]; }
  for (int o = 1; o < 32 && o * c < W; o <<= 1) {
    const double An = __shfl_down_sync(full, A, o), Bn = __shfl_down_sync(full, B, o);
    if (lane + o < 32) { B = fma(A, Bn, B); A *= An; }
  }
  double x = __shfl_down_sync(full, B, 1);
  if (lane == 31) x = 0.0;
#pragma unroll
  for (int q = kWinRegs - 1; q >= 0; --q)
    if (q < c) {
      x = fma(cp[q], x, v[q]);
      const int i = lane * c + q - W;
      if (i >= 0 && i < cnt) store(i, x);
    }
}

// Interface unknowns e0 … e1 (both ends of every element e0 … e1−1) of both right-hand sides, by all
// warps of the CTA, from condensed right-hand sides R (read through L2: other CTAs wrote some of them);
// ub[rh·stride + i] receives unknown e0 + i.  The caller synchronises the CTA afterwards.
__device__ __forceinline__ void mass1d_windows(const SurfTables& t, const double* R, int e0, int e1, double* ub,
                                               int stride) {
  const int Q = t.P + 1, Nx = t.Nx, nw = blockDim.x >> 5;
  const int seg = 32 * kWinRegs - 2 * t.win, total = e1 - e0 + 1, nseg = (total + seg - 1) / seg;
  for (int k = threadIdx.x >> 5; k < 2 * nseg; k += nw) {
    const int rh = k & 1, i0 = (k >> 1) * seg;
    const double* Rr = R + (size_t)rh * Nx * Q;
    auto gfun = [&](int j) -> double {
      const int jl = j > 0 ? j - 1 : (t.periodic ? Nx - 1 : -1);
      return (j < Nx ? __ldcg(Rr + (size_t)j * Q) : 0.0) + (jl >= 0 ? __ldcg(Rr + (size_t)jl * Q + t.P) : 0.0);
    };
    double* o = ub + rh * stride + i0;
    mass1d_window(t, gfun, e0 + i0, min(seg, total - i0), [&](int i, double u) { o[i] = u; });
  }
}

// Value at local column a of element ex from its condensed rows Re and the interface unknowns ul, ur at
// its ends.
__device__ __forceinline__ double mass1d_value(const SurfTables& t, const double* Re, double ul, double ur, int a) {
  if (a == 0) return ul;
  if (a == t.P) return ur;
  return Re[a] - (t.Z[a - 1] * ul + t.Z[t.P - 1 + a - 1] * ur);
}

// Over-integrated Zakharov integrals of element ex: η, ηx, φ̃x, w̃ (cv: 4·Q coarse values in shared
// memory) are interpolated to the Pf+1 fine GLL nodes, the PDE integrands of eq. FSeqs evaluated
// pointwise and projected with Iᵀ M_f (Δx/2) (§3.1.1, §3.3).  R[0][ex][·] and R[1][ex][·] receive the
// condensed element right-hand sides of ∂tη and ∂tφ̃.  By the 16 lanes of half a warp (sub = 0..15),
// both halves in step (`active`: this half has an element): an FP64 instruction occupies the narrow pipe for a whole warp's
// time whatever its active lanes, and the fine nodes of the usual orders fit 16 lanes.
__device__ __forceinline__ void zak_element16(const SurfTables& t, double* __restrict__ R, int ex, bool active,
                                              int sub, double* sh) {
  const int Q = t.P + 1, Qf = t.Pf + 1;
  double* Fe = sh;
  double* Fp = Fe + kMaxQf;
  const double* cv = Fp + kMaxQf;
  if (active)
    for (int q = sub; q < Qf; q += 16) {
      const double* Iq = t.I + q * Q;
      double e = 0, ex_ = 0, px = 0, wv = 0;
      for (int c = 0; c < Q; ++c) {
        const double w = Iq[c];
        e = fma(w, cv[c], e);
        ex_ = fma(w, cv[Q + c], ex_);
        px = fma(w, cv[2 * Q + c], px);
        wv = fma(w, cv[3 * Q + c], wv);
      }
      const double s2 = fma(ex_, ex_, 1.0);
      Fe[q] = fma(wv, s2, -ex_ * px);
      Fp[q] = -t.g * e - 0.5 * fma(px, px, -wv * wv * s2);
    }
  __syncwarp();
  if (active) {
    const double se = t.se[ex];
    for (int k = sub; k < 2 * Q; k += 16) {
      const int fld = k >= Q ? 1 : 0, a = k - fld * Q;
      const double* Ba = t.ZB + a * Qf;
      const double* F = fld ? Fp : Fe;
      double s = 0.0;
      for (int q = 0; q < Qf; ++q) s = fma(Ba[q], F[q], s);
      // the interior part Δx/2 · (Δx/2 · M_ii)⁻¹: the scales cancel
      R[((size_t)fld * t.Nx + ex) * Q + a] = (a == 0 || a == t.P) ? se * s : s;
    }
  }
  __syncwarp();
}

// Modal filter of element ex on its interior nodes, two fields (one warp, `sh` scratch).  The
// hat modes are untouched, so the shared end values keep their value by construction.
__device__ __forceinline__ void filter_element(const SurfTables& t, double* q0, double* q1, int ex, int lane,
                                               double* sh) {
  const int P = t.P, Q = P + 1;
  double* v0 = sh;
  double* v1 = v0 + Q;
  if (lane < Q) {
    const int c = scol(t, ex, lane);
    v0[lane] = __ldcg(q0 + c);
    v1[lane] = q1 ? __ldcg(q1 + c) : 0.0;
  }
  __syncwarp();
  if (lane >= 1 && lane < P) {
    const double* Fa = t.F + lane * Q;
    double s0 = 0, s1 = 0;
    for (int c = 0; c < Q; ++c) {
      s0 = fma(Fa[c], v0[c], s0);
      s1 = fma(Fa[c], v1[c], s1);
    }
    const int c = scol(t, ex, lane);
    q0[c] = s0;
    if (q1) q1[c] = s1;
  }
  __syncwarp();
}

// Embedded penalty forcing of §2.2 at column `col`: q̇ += (1 − γ(x))(q_a(x,t) − q)/τ with
// γ = ξ²(3 − 2ξ) across each zone (1 outside); q_a is the linear superposition of the wave
// input in the left zone, rest in the right zone.
// Per time level, the component factors of the generated signal (§2.2): with A = ωt + θ and
// c = −g a/ω, wA = (a cos A, a sin A, c sin A, c cos A).  Items i = first, first + stride, ….
__device__ __forceinline__ void wave_angles(const SurfTables& t, double time, int first, int stride) {
  const int n = t.ncomp;
  const double* a = t.wave;
  const double* om = a + n;
  const double* th = om + 2 * n;
  for (int i = first; i < n; i += stride) {
    double sn, cs;
    sincos(fma(om[i], time, th[i]), &sn, &cs);
    const double c = -t.g * a[i] / om[i];
    t.wA[i] = a[i] * cs;
    t.wA[n + i] = a[i] * sn;
    t.wA[2 * n + i] = c * sn;
    t.wA[3 * n + i] = c * cs;
  }
}

// The generated η = Σ a cos(A − kx) and φ̃ = Σ c sin(A − kx) at left-zone column `col`, by one
// warp (lanes over the components, then a shuffle tree): cos(A − kx) = cos A cos kx + sin A sin kx,
// sin(A − kx) = sin A cos kx − cos A sin kx.  Written to wEP by lane 0.
__device__ __forceinline__ void wave_zone_column(const SurfTables& t, int col, int lane) {
  const int n = t.ncomp;
  const double* ck = t.wkx + (size_t)col * n * 2;
  double ea = 0.0, pa = 0.0;
  for (int i = lane; i < n; i += 32) {
    const double cb = ck[2 * i], sb = ck[2 * i + 1];
    ea = fma(t.wA[i], cb, fma(t.wA[n + i], sb, ea));
    pa = fma(t.wA[2 * n + i], cb, fma(-t.wA[3 * n + i], sb, pa));
  }
  for (int o = 16; o > 0; o >>= 1) {
    ea += __shfl_xor_sync(0xffffffffu, ea, o);
    pa += __shfl_xor_sync(0xffffffffu, pa, o);
  }
  if (lane == 0) {
    t.wEP[2 * col] = ea;
    t.wEP[2 * col + 1] = pa;
  }
}

// ep: the generated (η, φ̃) of the left-zone columns for this time (wave_zone_columns), or
// nullptr to sum the components here.
__device__ __forceinline__ void relax_column(const SurfTables& t, const double* __restrict__ eta,
                                             const double* __restrict__ phis, double time, double inv_tau,
                                             double* de, double* dp, int col, const double* ep = nullptr) {
  const double x = t.xcol[col];
  double gam = 1.0;
  const bool left = t.relax_left > 0.0 && x < t.x0 + t.relax_left;
  if (left) {
    const double xi = fmin(fmax((x - t.x0) / t.relax_left, 0.0), 1.0);
    gam = xi * xi * (3.0 - 2.0 * xi);
  }
  if (t.relax_right > 0.0 && x > t.x1 - t.relax_right) {
    const double xi = fmin(fmax((t.x1 - x) / t.relax_right, 0.0), 1.0);
    gam = fmin(gam, xi * xi * (3.0 - 2.0 * xi));
  }
  if (gam >= 1.0) return;
  double ea = 0.0, pa = 0.0;
  if (left && ep != nullptr && col < t.nzl) {
    ea = ep[2 * col];
    pa = ep[2 * col + 1];
  } else if (left) {
    const double* a = t.wave;
    const double* om = a + t.ncomp;
    const double* k = om + t.ncomp;
    const double* th = k + t.ncomp;
    for (int i = 0; i < t.ncomp; ++i) {
      double sn, cs;
      sincos(om[i] * time - k[i] * x + th[i], &sn, &cs);
      ea = fma(a[i], cs, ea);
      pa = fma(-t.g * a[i] / om[i], sn, pa);
    }
  }
  const double c = (1.0 - gam) * inv_tau;
  de[col] = fma(c, ea - eta[col], de[col]);
  dp[col] = fma(c, pa - phis[col], dp[col]);
}

// Classical RK4 stage bookkeeping at index i, with k = right-hand side of this stage:
//   stage 1: acc = k,   st = q + dt/2 k
//   stage 2: acc += 2k, st = q + dt/2 k
//   stage 3: acc += 2k, st = q + dt k
//   stage 4: q += dt/6 (acc + k)
__device__ __forceinline__ void rk4_item(int stage, double dt, double* eta, double* phis, const double* ke,
                                         const double* kp, double* ae, double* ap, double* se, double* sp,
                                         int i) {
  const double a = ke[i], b = kp[i];
  if (stage == 1) {
    ae[i] = a; ap[i] = b;
    se[i] = fma(0.5 * dt, a, eta[i]); sp[i] = fma(0.5 * dt, b, phis[i]);
  } else if (stage == 2 || stage == 3) {
    ae[i] = fma(2.0, a, ae[i]); ap[i] = fma(2.0, b, ap[i]);
    const double c = stage == 2 ? 0.5 * dt : dt;
    se[i] = fma(c, a, eta[i]); sp[i] = fma(c, b, phis[i]);
  } else {
    eta[i] = fma(dt / 6.0, ae[i] + a, eta[i]);
    phis[i] = fma(dt / 6.0, ap[i] + b, phis[i]);
  }
}

}  // namespace semgb
