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
  EoTable<double> D64, T64, H64;        // D, Dᵀ and H = Dᵀ W
  EoTable<float> D32, T32, Dh32, H32;   // the same, and ½D
};
static __constant__ EoTables c_eo;
template <class T> __device__ __forceinline__ const EoTable<T>& eo_D();
template <> __device__ __forceinline__ const EoTable<double>& eo_D<double>() { return c_eo.D64; }
template <> __device__ __forceinline__ const EoTable<float>& eo_D<float>() { return c_eo.D32; }
template <class T> __device__ __forceinline__ const EoTable<T>& eo_T();
template <> __device__ __forceinline__ const EoTable<double>& eo_T<double>() { return c_eo.T64; }
template <> __device__ __forceinline__ const EoTable<float>& eo_T<float>() { return c_eo.T32; }
template <class T> __device__ __forceinline__ const EoTable<T>& eo_H();
template <> __device__ __forceinline__ const EoTable<double>& eo_H<double>() { return c_eo.H64; }
template <> __device__ __forceinline__ const EoTable<float>& eo_H<float>() { return c_eo.H32; }

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
