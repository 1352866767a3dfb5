// Even-odd forms of the GLL derivative.  Included by laplace_device.cuh (order-templated, internal
// linkage).
//
// The GLL nodes are symmetric, so the derivative matrix satisfies D[P−i][P−j] = −D[i][j], and its
// weighted transpose H_ij = D_ji w_j as well.  With e_j = u_j + u_{P−j}, o_j = u_j − u_{P−j} (j < h = ⌊Q/2⌋)
//     S_i = Σ_j O_ij o_j,   T_i = Σ_j E_ij e_j (+ C_i u_mid),   (Du)_i = S_i + T_i,  (Du)_{P−i} = S_i − T_i,
//     (Du)_mid = Σ_j R_j o_j,    O, E = ½(D_ij ∓ D_{i,P−j}),  C_i = D_{i,mid},  R_j = D_{mid,j}:
// 36 operations for a line of 7 nodes instead of 49, 48 instead of 64 for 8 (even-odd decomposition,
// Solomonoff, J. Comput. Phys. 98, 1992).
#pragma once
#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

namespace semgb {

// Tables of the translation unit's order: O, E (h×h), C, R (h) of a matrix with that symmetry.
constexpr int kEoH = (kMaxP + 1) / 2;
// Rows of odd length: rows of whole 16-byte multiples would be loaded into registers as vectors, two tables
// of them through a loop (118 instead of 44 registers for two lines of 8), instead of being operands.
__host__ __device__ constexpr int eo_stride(int Q) { return Q / 2 | 1; }
template <class T>
struct EoTable {
  T O[kEoH * (kEoH | 1)], E[kEoH * (kEoH | 1)], C[kEoH], R[kEoH];
};
struct EoTables {
  EoTable<double> D64, T64, H64;     // D, Dᵀ and H = Dᵀ W
  EoTable<float> D32, T32;
  // the FP32 applies': s D and s' H, the weights w/(s s') taking the factors back (fill_scaled)
  EoTable<float> D32s, H32s;
  float w32s[kMaxP + 1];
};
static __constant__ EoTables c_eo;
template <class T> __device__ __forceinline__ const EoTable<T>& eo_D();
template <> __device__ __forceinline__ const EoTable<double>& eo_D<double>() { return c_eo.D64; }
template <> __device__ __forceinline__ const EoTable<float>& eo_D<float>() { return c_eo.D32; }
template <class T> __device__ __forceinline__ const EoTable<T>& eo_T();
template <> __device__ __forceinline__ const EoTable<double>& eo_T<double>() { return c_eo.T64; }
template <> __device__ __forceinline__ const EoTable<float>& eo_T<float>() { return c_eo.T32; }
template <class T> __device__ __forceinline__ const EoTable<T>& eo_Ds();
template <> __device__ __forceinline__ const EoTable<double>& eo_Ds<double>() { return c_eo.D64; }
template <> __device__ __forceinline__ const EoTable<float>& eo_Ds<float>() { return c_eo.D32s; }
template <class T> __device__ __forceinline__ const EoTable<T>& eo_Hs();
template <> __device__ __forceinline__ const EoTable<double>& eo_Hs<double>() { return c_eo.H64; }
template <> __device__ __forceinline__ const EoTable<float>& eo_Hs<float>() { return c_eo.H32s; }

template <int P, class T>
static void fill_eo(EoTable<T>& t, const double* M, double scale) {   // M: Q×Q, row-major
  constexpr int Q = P + 1, h = Q / 2;
  for (int i = 0; i < h; ++i) {
    for (int j = 0; j < h; ++j) {
      t.O[i * eo_stride(Q) + j] = (T)(scale * 0.5 * (M[i * Q + j] - M[i * Q + P - j]));
      t.E[i * eo_stride(Q) + j] = (T)(scale * 0.5 * (M[i * Q + j] + M[i * Q + P - j]));
    }
    t.C[i] = Q % 2 ? (T)(scale * M[i * Q + h]) : T(0);
    t.R[i] = Q % 2 ? (T)(scale * M[h * Q + i]) : T(0);
  }
}

// The FP32 applies' tables.  An even-odd line rounds its sums and differences too, which made the applies' errors
// of orders 2..6 up to a fifth larger than those of plain lines; the tables' own rounding, the same in every element,
// is taken back for that: of 2048 factors s and s' in [1, 2) those under which the entries of s D and s' H,
// and the weights w/(s s'), round best (relative root mean squares 4e-8 → 0.2..2e-8).
template <int P>
static double table_rounding(const double* M, double s) {
  EoTable<float> f{};
  EoTable<double> d{};
  fill_eo<P>(f, M, s);
  fill_eo<P>(d, M, s);
  constexpr int h = (P + 1) / 2, st = eo_stride(P + 1);
  double err = 0.0, sum = 0.0;
  auto add = [&](double v, float r) { err += (v - r) * (v - r); sum += v * v; };
  for (int i = 0; i < h; ++i) {
    for (int j = 0; j < h; ++j) { add(d.O[i * st + j], f.O[i * st + j]); add(d.E[i * st + j], f.E[i * st + j]); }
    add(d.C[i], f.C[i]);
    add(d.R[i], f.R[i]);
  }
  return err / sum;
}

template <int P>
static void fill_scaled(EoTables& eo, const double* D, const double* H, const double* w) {
  constexpr int kScales = 2048, kKeep = 32;
  std::pair<double, double> best[2][kKeep];            // (error, scale) of D and of H
  for (int m = 0; m < 2; ++m) {
    std::vector<std::pair<double, double>> all(kScales);
    for (int i = 0; i < kScales; ++i) {
      const double s = 1.0 + (double)i / kScales;
      all[i] = {table_rounding<P>(m ? H : D, s), s};
    }
    std::partial_sort_copy(all.begin(), all.end(), best[m], best[m] + kKeep);
  }
  double least = INFINITY, sD = 1.0, sH = 1.0;
  for (const auto& d : best[0])
    for (const auto& h : best[1]) {
      double e = 0.0;                                  // the weights come in twice
      for (int a = 0; a <= P; ++a) {
        const double v = w[a] / (d.second * h.second);
        e += ((float)v - v) / v * (((float)v - v) / v) * 2.0 / (P + 1);
      }
      if (d.first + h.first + e < least) { least = d.first + h.first + e; sD = d.second; sH = h.second; }
    }
  fill_eo<P>(eo.D32s, D, sD);
  fill_eo<P>(eo.H32s, H, sH);
  for (int a = 0; a <= P; ++a) eo.w32s[a] = (float)(w[a] / (sD * sH));
}

// out = D u for one line in registers, from differences against the middle value (the upper one of two): a
// derivative does not see a constant, so E takes e_j − 2 u_mid and C drops out.  e_j itself would round like the
// values, and the table's row sums like its entries: on smooth fields, whose derivatives are small beside
// them, that made the applies' errors up to 2.2 times those of plain lines (FP32 and FP64); the differences
// make them 0.01 to 0.6 times.  An operation a line more for 7 nodes (39), 6 for 8 (54).
template <int Q, class T>
__device__ __forceinline__ void eo_diff(const EoTable<T>& t, const T (&u)[Q], T (&out)[Q]) {
  constexpr int h = Q / 2, P = Q - 1;
  T e[h], o[h];
#pragma unroll
  for (int j = 0; j < h; ++j) {
    o[j] = u[j] - u[P - j];
    e[j] = P - j == h ? o[j] : (u[j] - u[h]) + (u[P - j] - u[h]);
  }
#pragma unroll
  for (int i = 0; i < h; ++i) {
    T S = t.O[i * eo_stride(Q)] * o[0], V = t.E[i * eo_stride(Q)] * e[0];
#pragma unroll
    for (int j = 1; j < h; ++j) { S = fmx(t.O[i * eo_stride(Q) + j], o[j], S); V = fmx(t.E[i * eo_stride(Q) + j], e[j], V); }
    out[i] = S + V;
    out[P - i] = S - V;
  }
  if constexpr (Q % 2) {
    T m = t.R[0] * o[0];
#pragma unroll
    for (int j = 1; j < h; ++j) m = fmx(t.R[j], o[j], m);
    out[h] = m;
  }
}

// out = M u for one line in registers.
template <int Q, class T>
__device__ __forceinline__ void eo_line(const EoTable<T>& t, const T (&u)[Q], T (&out)[Q]) {
  constexpr int h = Q / 2, P = Q - 1;
  T e[h], o[h];
#pragma unroll
  for (int j = 0; j < h; ++j) { e[j] = u[j] + u[P - j]; o[j] = u[j] - u[P - j]; }
#pragma unroll
  for (int i = 0; i < h; ++i) {
    T S = t.O[i * eo_stride(Q)] * o[0], V = t.E[i * eo_stride(Q)] * e[0];
#pragma unroll
    for (int j = 1; j < h; ++j) { S = fmx(t.O[i * eo_stride(Q) + j], o[j], S); V = fmx(t.E[i * eo_stride(Q) + j], e[j], V); }
    if constexpr (Q % 2) V = fmx(t.C[i], u[h], V);
    out[i] = S + V;
    out[P - i] = S - V;
  }
  if constexpr (Q % 2) {
    T m = t.R[0] * o[0];
#pragma unroll
    for (int j = 1; j < h; ++j) m = fmx(t.R[j], o[j], m);
    out[h] = m;
  }
}

}  // namespace semgb
