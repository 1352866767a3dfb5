// FP32 apply with one element per thread.  Included by laplace_device.cuh (order-templated, internal
// linkage).
#pragma once

namespace semgb {

// ------------------------------------------------------------------------------------
// FP32 apply y = 𝓛x, one element per thread (orders up to 8, up to 4 layers).
//
// The line-pass kernel (k_apply_tile) spends 142 instructions per node, two thirds of them moving
// lines between its three passes through shared memory.  Here a thread loads the (P+1)² values of its
// element once, keeps every intermediate in registers, and exchanges only the top row and the right
// column with its neighbours: about 43 FP32 operations per node.  What bounds it is the latency of a thread's long
// chains at 12 warps an SM (6 at order 8, 1 or 2 CTAs by registers and shared memory), 60% of the issue slots used.
// 65536×4, P = 6: 63.5 → 31.0 µs (2.5 TB/s of x and y); 8 M nodes of P = 3..8: 51–138 → 25–62 µs.
// A warp holds 32 consecutive elements of one layer; a CTA holds all layers of 32·G elements, the first
// of which is the element left of its tile, recomputed for the tile's first column.  x is staged by bulk
// copies, double-buffered as in k_apply_tile; y goes through the same buffer and leaves in contiguous
// 16-byte stores.  Sums have a fixed order that does not depend on the tiling.
template <int P, int NZ>
struct ElemTile {
  static constexpr int Q = P + 1, nrow = NZ * P + 1;
  static constexpr int G = NZ == 1 ? 4 : (NZ <= 3 ? 2 : 1);   // groups of 32 elements
  static constexpr int en = 32 * G, E = en - 1;               // elements computed, owned
  static constexpr int threads = 32 * NZ * G;
  // Floats between elements in the staging buffer.  Lanes read their elements at this stride: where it
  // would be a multiple of 8 words (8- or 16-way bank conflicts), the elements, then whole 16-byte
  // multiples, are copied one by one with 4 words between them (tanks of P = 5, three
  // layers: 52 → 26 µs at 8 M nodes).
  static constexpr int pe = P * nrow;
  static constexpr bool pad = pe % 8 == 0;
  static constexpr int se = pe + (pad ? 4 : 0);
  static constexpr int xbuf = ((en * se + nrow + 8 + 3) / 4) * 4;
  static constexpr int gbuf = 4 * en * Q, cbuf = 4 * en * NZ;   // floats: geometry, layer ratios (FP64)
  static constexpr size_t smem = 16 + 4 * (size_t)(2 * (xbuf + gbuf + cbuf) + NZ * (P + Q) * en);
  // CTAs per SM: 168 registers up to order 6, else 255, and as many as the shared memory holds (6, 1: two, 8, 1: one)
  static constexpr int reg_ctas = P <= 6 ? (threads <= 128 ? 3 : 2) : (threads <= 128 ? 2 : 1);
  static constexpr int smem_ctas = (int)((size_t)228 * 1024 / (smem + 1024 + 16));
  static constexpr int ctas = reg_ctas < smem_ctas ? reg_ctas : smem_ctas;
};

template <int P, int NZ>
__global__ void __launch_bounds__(ElemTile<P, NZ>::threads, ElemTile<P, NZ>::ctas)
    k_apply_elem(DevGeom g, const float* __restrict__ x, float* __restrict__ y, int bulk_ok, int vec_ok) {
  using L = ElemTile<P, NZ>;
  constexpr int Q = P + 1, h = Q / 2, nrow = L::nrow, E = L::E, en_max = L::en;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* mbar = reinterpret_cast<unsigned long long*>(smem_raw);   // [2]
  float* const Xb0 = reinterpret_cast<float*>(smem_raw + 16);
  float* const Gb0 = Xb0 + 2 * L::xbuf;                              // [en][Q][4] d, 1/d, ∂xh, ∂xd
  float* const Cb0 = Gb0 + 2 * L::gbuf;                              // [en][NZ][2] Δσ/Δx, Δx/Δσ (FP64)
  float* const Rrow = Cb0 + 2 * L::cbuf;                             // [NZ][P][en] top rows, a < P
  float* const Ccol = Rrow + NZ * P * en_max;                        // [NZ][Q][en] right columns
  __shared__ int s_ok;
  const int Nx = g.Nx, ncol = g.ncol;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = warp % NZ, el = (warp / NZ) * 32 + lane;             // layer, local element (0: left of the tile)
  if (threadIdx.x == 0) {
    mbar_init(&mbar[0]);
    mbar_init(&mbar[1]);
    mbar_init_fence();
    s_ok = 1;
  }
  float sg[Q];
#pragma unroll
  for (int b = 0; b < Q; ++b) sg[b] = (float)g.sig[l * P + b];
  __syncthreads();
  const int ntiles = (Nx + E - 1) / E;
  unsigned parity0 = 0u, parity1 = 0u;
  int pending0 = 0, pending1 = 0;
  auto issue = [&](int tile, int bf) {
    const int ex0 = tile * E, ne = min(E, Nx - ex0);
    long long lo;
    int count, shift;
    if (bulk_ok && tile_range<P, float>(g, ex0, ne, &lo, &count, &shift)) {
      // the elements ex0 − 1 … ex0 + ne − 1 (no wrap here): their nodes, geometry and layer ratios
      const unsigned bx = (L::pad ? (ne + 1) * L::pe + (nrow + 3) / 4 * 4 : count) * 4u, bg = (ne + 1) * Q * 16u, bc = (ne + 1) * NZ * 16u;
      fence_proxy_async_smem();
      mbar_expect(&mbar[bf], bx + bg + bc);
      float* dst = Xb0 + bf * L::xbuf;
      if constexpr (L::pad) {                    // (lo is the range's start: a multiple of 4)
        for (int e = 0; e <= ne; ++e) bulk_copy(dst + e * L::se, x + lo + (long long)e * L::pe, L::pe * 4u, &mbar[bf]);
        bulk_copy(dst + (ne + 1) * L::se, x + lo + (long long)(ne + 1) * L::pe, (nrow + 3) / 4 * 16u, &mbar[bf]);
      } else {
        bulk_copy(dst, x + lo, bx, &mbar[bf]);
      }
      bulk_copy(Gb0 + bf * L::gbuf, g.geo32 + (size_t)(ex0 - 1) * Q * 4, bg, &mbar[bf]);
      bulk_copy(Cb0 + bf * L::cbuf, g.cxz + (size_t)(ex0 - 1) * NZ * 2, bc, &mbar[bf]);
      if (bf) pending1 = 1;
      else pending0 = 1;
    }
  };
  if (threadIdx.x == 0 && (int)blockIdx.x < ntiles) issue(blockIdx.x, 0);

  int k = 0;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
    const int bf = k & 1, ex0 = tile * E, ne = min(E, Nx - ex0), en = ne + 1;
    long long lo;
    int count, shift;
    const bool bulk = bulk_ok && tile_range<P, float>(g, ex0, ne, &lo, &count, &shift);
    __syncthreads();                             // the previous tile's readers are done
    if (threadIdx.x == 0) {
      if (tile + (int)gridDim.x < ntiles) issue(tile + gridDim.x, bf ^ 1);
      const int pend = bf ? pending1 : pending0;
      if (pend) {
        const unsigned par = bf ? parity1 : parity0;
        if (!mbar_wait(&mbar[bf], par, kCopyTimeoutNs)) s_ok = 0;
        else if (bf) { parity1 ^= 1u; pending1 = 0; }
        else { parity0 ^= 1u; pending0 = 0; }
      }
    }
    float* const buf = Xb0 + bf * L::xbuf;
    float* X = buf;
    if (bulk) {
      X += shift;
    } else {
      for (int t = threadIdx.x; t < (en * P + 1) * nrow; t += L::threads) {
        const int j = t / nrow, r = t - j * nrow;
        int gc = (ex0 - 1) * P + j;
        if (gc < 0) gc = g.periodic ? gc + ncol : -1;
        else if (gc >= ncol) gc -= ncol;         // periodic: column Nx·P is column 0
        cp_async1(X + t + (L::pad ? j / P * (L::se - L::pe) : 0), x + (size_t)(gc < 0 ? 0 : gc) * nrow + r, gc >= 0);
      }
      cp_async_wait();
    }
    float4* const Gs = reinterpret_cast<float4*>(Gb0 + bf * L::gbuf);
    const double2* const Cs = reinterpret_cast<const double2*>(Cb0 + bf * L::cbuf);
    const bool on = el < en && (ex0 + el > 0 || g.periodic);   // walls: no element left of x = 0
    if (!bulk) {
      for (int t = threadIdx.x; t < en * Q; t += blockDim.x) {
        int ge = ex0 - 1 + t / Q;
        if (ge < 0) ge = g.periodic ? ge + Nx : 0;
        Gs[t] = reinterpret_cast<const float4*>(g.geo32)[(size_t)ge * Q + t % Q];
      }
      for (int t = threadIdx.x; t < en * NZ; t += blockDim.x) {
        int ge = ex0 - 1 + t / NZ;
        if (ge < 0) ge = g.periodic ? ge + Nx : 0;
        reinterpret_cast<double2*>(Cb0 + bf * L::cbuf)[t] = reinterpret_cast<const double2*>(g.cxz)[(size_t)ge * NZ + t % NZ];
      }
    }
    __syncthreads();
    if (!s_ok) break;                            // a copy did not complete: stop (status set below)
    float yv[Q][Q];                              // [a][b]: x even-odd sums of the result, then the result
    if (on) {
      const double2 cz = Cs[el * NZ + l];
      float c0, c0l, c1, c1l;
      split_ratio(cz.x, c0, c0l);
      split_ratio(cz.y, c1, c1l);
      float u[Q][Q];
      const float* Xe = X + el * L::se + l * P;
#pragma unroll
      for (int a = 0; a < Q; ++a)
#pragma unroll
        for (int b = 0; b < Q; ++b) u[a][b] = Xe[(a < P ? a * nrow : L::se) + b];
#pragma unroll
      for (int i = 0; i < h; ++i)                // u[i], u[P−i] ← e_i − 2 u_mid, o_i of the x-lines (eo_diff)
#pragma unroll
        for (int b = 0; b < Q; ++b) {
          const float p = u[i][b], q = u[P - i][b], m = u[h][b];
          u[P - i][b] = p - q;
          u[i][b] = P - i == h ? p - q : (p - m) + (q - m);
        }
#pragma unroll
      for (int a = 0; a < Q; ++a)
#pragma unroll
        for (int b = 0; b < Q; ++b) yv[a][b] = 0.f;
      const float* w = c_eo.w32s;
      // F1/w_a and F2/w_a of one column from u_r and u_t
      auto flux = [&](int a, const float (&ur)[Q], const float (&ut)[Q], float (&F1)[Q], float (&F2)[Q]) {
        const float4 q = Gs[el * Q + a];
        const float g11 = fmaf(c0, q.x, c0l * q.x), g22 = fmaf(c1, q.y, c1l * q.y);
#pragma unroll
        for (int b = 0; b < Q; ++b) {
          const float K12 = fmaf(-sg[b], q.w, q.z);
          F1[b] = w[b] * fmaf(g11, ur[b], K12 * ut[b]);   // the large products are not rounded by themselves
          F2[b] = fmaf(g22 * fmaf(K12, K12, 1.f), ut[b], K12 * ur[b]);
        }
      };
#pragma unroll
      for (int i = 0; i < h; ++i) {              // columns i and P−i together
        float r1[Q], r2[Q], t1[Q], t2[Q], F1a[Q], F2a[Q], F1b[Q], F2b[Q];
#pragma unroll
        for (int b = 0; b < Q; ++b) {
          float S = c_eo.D32s.O[i * eo_stride(Q)] * u[P][b], V = c_eo.D32s.E[i * eo_stride(Q)] * u[0][b];
#pragma unroll
          for (int j = 1; j < h; ++j) {
            S = fmaf(c_eo.D32s.O[i * eo_stride(Q) + j], u[P - j][b], S);
            V = fmaf(c_eo.D32s.E[i * eo_stride(Q) + j], u[j][b], V);
          }
          r1[b] = S + V;
          r2[b] = S - V;
        }
        float ua[Q], ub[Q];                          // the two columns again, from the staging buffer
#pragma unroll
        for (int b = 0; b < Q; ++b) {
          ua[b] = Xe[i * nrow + b];
          ub[b] = Xe[(P - i < P ? (P - i) * nrow : L::se) + b];
        }
        eo_diff<Q, float>(c_eo.D32s, ua, t1);
        eo_diff<Q, float>(c_eo.D32s, ub, t2);
        flux(i, r1, t1, F1a, F2a);
        flux(P - i, r2, t2, F1b, F2b);
#pragma unroll
        for (int b = 0; b < Q; ++b) {
          const float fe = F1a[b] + F1b[b], fo = F1a[b] - F1b[b];
#pragma unroll
          for (int c = 0; c < h; ++c) {
            yv[c][b] = fmaf(c_eo.H32s.O[c * eo_stride(Q) + i], fo, yv[c][b]);          // S_c
            yv[P - c][b] = fmaf(c_eo.H32s.E[c * eo_stride(Q) + i], fe, yv[P - c][b]);  // T_c
          }
          if constexpr (Q % 2) yv[h][b] = fmaf(c_eo.H32s.R[i], fo, yv[h][b]);
          const float p = F2a[b], q = F2b[b];
          F2a[b] = p + q;
          F2b[b] = p - q;
        }
        eo_line<Q, float>(c_eo.H32s, F2a, t1);
        eo_line<Q, float>(c_eo.H32s, F2b, t2);
        const float wh = 0.5f * w[i];
#pragma unroll
        for (int b = 0; b < Q; ++b) { yv[i][b] = fmaf(wh, t1[b], yv[i][b]); yv[P - i][b] = fmaf(wh, t2[b], yv[P - i][b]); }
      }
      if constexpr (Q % 2) {                     // the middle column
        float r[Q], t[Q], F1[Q], F2[Q];
#pragma unroll
        for (int b = 0; b < Q; ++b) {
          r[b] = c_eo.D32s.R[0] * u[P][b];
#pragma unroll
          for (int j = 1; j < h; ++j) r[b] = fmaf(c_eo.D32s.R[j], u[P - j][b], r[b]);
        }
        eo_diff<Q, float>(c_eo.D32s, u[h], t);
        flux(h, r, t, F1, F2);
        eo_line<Q, float>(c_eo.H32s, F2, t);
#pragma unroll
        for (int b = 0; b < Q; ++b) {
#pragma unroll
          for (int c = 0; c < h; ++c) yv[P - c][b] = fmaf(c_eo.H32s.C[c], F1[b], yv[P - c][b]);
          yv[h][b] = fmaf(w[h], t[b], yv[h][b]);
        }
      }
#pragma unroll
      for (int i = 0; i < h; ++i)
#pragma unroll
        for (int b = 0; b < Q; ++b) {
          const float S = yv[i][b], V = yv[P - i][b];
          yv[i][b] = S + V;
          yv[P - i][b] = S - V;
        }
#pragma unroll
      for (int a = 0; a < P; ++a)
        if (l < NZ - 1) Rrow[(l * P + a) * en_max + el] = yv[a][P];
#pragma unroll
      for (int b = 0; b < Q; ++b) Ccol[(l * Q + b) * en_max + el] = yv[P][b];
    } else if (el < en) {
#pragma unroll
      for (int b = 0; b < Q; ++b) Ccol[(l * Q + b) * en_max + el] = 0.f;   // nothing left of the wall
    }
    __syncthreads();                             // rows and columns exchanged; X is no longer read
    // the tile's own nodes a < P, b < P (b = P on the surface; a = P at the right wall): the layer
    // below, the element to the left, the element below left, in this order
    const long long out0 = (long long)ex0 * P * nrow;
    const int sh = (int)(out0 & 3);
    const bool last_wall = !g.periodic && ex0 + ne == Nx;
    if (on && el > 0) {
      float* Y = buf + sh + (el - 1) * L::se + l * P;
      float low[P];
#pragma unroll
      for (int a = 0; a < P; ++a) low[a] = l > 0 ? Rrow[((l - 1) * P + a) * en_max + el] : 0.f;
#pragma unroll
      for (int b = 0; b < Q; ++b) {
        if (b == P && l < NZ - 1) continue;
        float v = yv[0][b];
        if (b == 0) v += low[0];
        v += Ccol[(l * Q + b) * en_max + el - 1];
        if (b == 0 && l > 0) v += Ccol[((l - 1) * Q + P) * en_max + el - 1];
        Y[b] = -v;
#pragma unroll
        for (int a = 1; a < P; ++a) Y[a * nrow + b] = b == 0 ? -(yv[a][b] + low[a]) : -yv[a][b];
        if (last_wall && el == ne) {
          float r = yv[P][b];
          if (b == 0 && l > 0) r += Ccol[((l - 1) * Q + P) * en_max + el];
          Y[L::se + b] = -r;
        }
      }
    }
    __syncthreads();
    const int nout = (ne * P + (last_wall ? 1 : 0)) * nrow;
    float* yo = y + (out0 - sh);                 // 16-byte aligned where y is
    const float* ys = buf;
    if constexpr (L::pad) {                      // sh = 0: whole quads per element, then the wall's column
      if (vec_ok) {
        for (int t = threadIdx.x; t < ne * (L::pe / 4); t += L::threads) {
          const int e = t / (L::pe / 4);
          reinterpret_cast<float4*>(yo)[t] = reinterpret_cast<const float4*>(ys)[t + e];
        }
        for (int t = ne * L::pe + threadIdx.x; t < nout; t += L::threads) yo[t] = ys[t + 4 * ne];
      } else {
        for (int t = threadIdx.x; t < nout; t += L::threads) yo[t] = ys[t + t / L::pe * 4];
      }
    } else if (vec_ok) {
      const int v0 = sh ? 1 : 0, v1 = (sh + nout) >> 2;   // whole quads inside [sh, sh + nout)
      for (int t = v0 + threadIdx.x; t < v1; t += blockDim.x)
        reinterpret_cast<float4*>(yo)[t] = reinterpret_cast<const float4*>(ys)[t];
      if (sh && threadIdx.x >= sh && threadIdx.x < min(4, sh + nout)) yo[threadIdx.x] = ys[threadIdx.x];
      const int t = 4 * v1 + threadIdx.x;
      if (t < sh + nout) yo[t] = ys[t];
    } else {
      for (int t = sh + threadIdx.x; t < sh + nout; t += blockDim.x) yo[t] = ys[t];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {                        // a copy in flight lands before the shared memory is released
    if (!s_ok) atomicOr(g.status, ST_TIMEOUT);
    if (pending0 && !mbar_wait(&mbar[0], parity0, kCopyTimeoutNs)) atomicOr(g.status, ST_TIMEOUT);
    if (pending1 && !mbar_wait(&mbar[1], parity1, kCopyTimeoutNs)) atomicOr(g.status, ST_TIMEOUT);
  }
}

}  // namespace semgb
