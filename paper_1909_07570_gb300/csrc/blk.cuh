// Contractions of an nnTD sweep on shared-memory arrays, for the kernels that run whole
// fits of small tensors: one thread block per fit (small_batched.cu) or one cluster
// (ntd_cluster.cu). No sum depends on the block size.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace nnc {
namespace blk {

constexpr int kBlkMaxM = 16;
// Row pitch of a factor in shared memory: whole 16-byte pieces, from the tile widths that
// the passes are built for.
template <typename T>
__host__ __device__ inline int fpitch(int m) {
  if (sizeof(T) == 8 && m <= 6) return m <= 2 ? 2 : (m <= 4 ? 4 : 6);
  return m <= 4 ? 4 : (m <= 8 ? 8 : 16);
}
// Row pitch of T and P1 for N3 columns: 16-byte reads of eight consecutive rows
// fall on distinct banks (even 16-byte rows), single reads of 32 rows (odd).
template <typename T>
__host__ __device__ inline int rpitch(int n3) {
  constexpr int VL = 16 / (int)sizeof(T);
  if (n3 % VL) return n3 | 1;
  const int v = n3 / VL;
  return (v | 1) * VL;
}

template <typename T, int VL>
__device__ __forceinline__ void ldv(const T* p, T (&v)[VL]) {
  if constexpr (VL == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else if constexpr (VL == 2) {
    const double2 t = *reinterpret_cast<const double2*>(p);
    v[0] = t.x; v[1] = t.y;
  } else {
    v[0] = *p;
  }
}
template <typename T, int VL>
__device__ __forceinline__ void ldg_v(const T* p, T (&v)[VL]) {
  if constexpr (VL == 4) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else if constexpr (VL == 2) {
    const double2 t = __ldg(reinterpret_cast<const double2*>(p));
    v[0] = t.x; v[1] = t.y;
  } else {
    v[0] = __ldg(p);
  }
}
template <typename T, int VL>
__device__ __forceinline__ void stv(T* p, const T (&v)[VL]) {
  if constexpr (VL == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else if constexpr (VL == 2) *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  else *p = v[0];
}

// out[l, p, c] = sum_j F[j, p] X[l, j, c], p < Q (F: J x QP in shared memory,
// zero past Q), j in order, VL consecutive c per thread, over nc of the C columns of
// X. Column c = (j', k) of N3 entries per row k goes to
// out[((l Q + p) nc / N3 + j') cp + k].
template <typename T, int QP, int VL>
__device__ __forceinline__ void col_pass_impl(const T* __restrict__ X, int L, int J, int C, int nc,
                                              int N3, int cp, const T* F, int Q, T* out) {
  constexpr int VW = 16 / (int)sizeof(T);
  const int cv = nc / VL, rows = nc / N3;
  for (int t = threadIdx.x; t < L * cv; t += blockDim.x) {
    const int l = t / cv, c = (t - l * cv) * VL;
    const T* x = X + (int64_t)l * J * C + c;
    T acc[QP][VL];
#pragma unroll
    for (int p = 0; p < QP; ++p)
#pragma unroll
      for (int u = 0; u < VL; ++u) acc[p][u] = T(0);
    constexpr int U = VL == 4 ? 4 : 8;  // loads in flight
    int j = 0;
    for (; j + U <= J; j += U) {
      T v[U][VL];
#pragma unroll
      for (int q = 0; q < U; ++q) ldg_v<T, VL>(x + (int64_t)(j + q) * C, v[q]);
#pragma unroll
      for (int q = 0; q < U; ++q)
#pragma unroll
        for (int p = 0; p < QP; p += VW) {
          T w[VW];
          ldv<T, VW>(F + (j + q) * QP + p, w);
#pragma unroll
          for (int e = 0; e < VW; ++e)
#pragma unroll
            for (int u = 0; u < VL; ++u) acc[p + e][u] = fma(v[q][u], w[e], acc[p + e][u]);
        }
    }
    for (; j < J; ++j) {
      T v[VL];
      ldg_v<T, VL>(x + (int64_t)j * C, v);
#pragma unroll
      for (int p = 0; p < QP; p += VW) {
        T w[VW];
        ldv<T, VW>(F + j * QP + p, w);
#pragma unroll
        for (int e = 0; e < VW; ++e)
#pragma unroll
          for (int u = 0; u < VL; ++u) acc[p + e][u] = fma(v[u], w[e], acc[p + e][u]);
      }
    }
    const int jr = c / N3, k = c - jr * N3;
    T* o = out + ((int64_t)l * Q * rows + jr) * cp + k;
#pragma unroll
    for (int p = 0; p < QP; ++p)
      if (p < Q) stv<T, VL>(o + (int64_t)p * rows * cp, acc[p]);
  }
}

// f(width) with the tile width that fpitch gives Q.
template <typename T, int QM, typename F>
__device__ __forceinline__ void by_width(int Q, F f) {
  if (sizeof(T) == 8 && Q <= 2) f(std::integral_constant<int, 2>{});
  else if (Q <= 4) f(std::integral_constant<int, 4>{});
  else if (sizeof(T) == 8 && Q <= 6) f(std::integral_constant<int, 6>{});
  else if (Q <= 8) f(std::integral_constant<int, 8>{});
  else if constexpr (QM > 8) f(std::integral_constant<int, 16>{});
}

template <typename T, int QM>
__device__ void col_pass(const T* __restrict__ X, int L, int J, int C, int nc, int N3, int cp,
                         const T* F, int Q, bool vec, T* out) {
  constexpr int VL = 16 / (int)sizeof(T);
  by_width<T, QM>(Q, [&](auto w) {
    constexpr int QP = decltype(w)::value;
    if (vec) col_pass_impl<T, QP, VL>(X, L, J, C, nc, N3, cp, F, Q, out);
    else col_pass_impl<T, QP, 1>(X, L, J, C, nc, N3, cp, F, Q, out);
  });
}

// Y[row, q] = sum_k P[row cp + k] F[k, q], rows < R, q < Q, k < K in order (F:
// K x QP, zero past Q): one thread per row, all q.
template <typename T, int QP>
__device__ __forceinline__ void row_dots_impl(const T* P, int R, int cp, int K, const T* F, int Q,
                                              T* Y) {
  constexpr int VL = 16 / (int)sizeof(T);
  for (int r = threadIdx.x; r < R; r += blockDim.x) {
    T acc[QP];
#pragma unroll
    for (int q = 0; q < QP; ++q) acc[q] = T(0);
    const T* x = P + r * cp;
    auto add = [&](T v, const T* f) {
#pragma unroll
      for (int q = 0; q < QP; q += VL) {
        T w[VL];
        ldv<T, VL>(f + q, w);
#pragma unroll
        for (int e = 0; e < VL; ++e) acc[q + e] = fma(v, w[e], acc[q + e]);
      }
    };
    int k = 0;
    if (K % VL == 0) {  // cp is then a multiple of VL too
      for (; k < K; k += VL) {
        T v[VL];
        ldv<T, VL>(x + k, v);
#pragma unroll
        for (int u = 0; u < VL; ++u) add(v[u], F + (k + u) * QP);
      }
    } else {
#pragma unroll 4
      for (; k < K; ++k) add(x[k], F + k * QP);
    }
#pragma unroll
    for (int q = 0; q < QP; ++q)
      if (q < Q) Y[r * Q + q] = acc[q];
  }
}
template <typename T, int QM>
__device__ void row_dots(const T* P, int R, int cp, int K, const T* F, int Q, T* Y) {
  by_width<T, QM>(Q, [&](auto w) {
    row_dots_impl<T, decltype(w)::value>(P, R, cp, K, F, Q, Y);
  });
}

// S = F^T F (m x m; F: N rows of pitch fp): four lanes per entry, lane u adding
// the rows u, u + 4, ... in order, the four sums by a fixed shuffle tree.
template <typename T>
__device__ void gram4(const T* F, int N, int fp, int m, T* S) {
  const int u = threadIdx.x & 3;
  for (int e0 = 0; e0 < m * m; e0 += blockDim.x / 4) {
    const int e = e0 + (int)threadIdx.x / 4;
    T s = T(0);
    if (e < m * m) {
      const int a = e / m, b = e - a * m;
      for (int i = u; i < N; i += 4) s = fma(F[i * fp + a], F[i * fp + b], s);
    }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (e < m * m && u == 0) S[e] = s;
  }
}

// out[l, p, c] = sum_j A[p, j] in[l, j, c] for a symmetric A (J x J), all in
// shared memory (a core times a Gram along one mode).
template <typename T>
__device__ void core_gram(const T* in, int L, int J, int C, const T* A, T* out) {
  for (int e = threadIdx.x; e < L * J * C; e += blockDim.x) {
    const int c = e % C, lp = e / C, p = lp % J, l = lp / J;
    const T* x = in + l * J * C + c;
    T s = T(0);
    for (int j = 0; j < J; ++j) s = fma(A[p * J + j], x[j * C], s);
    out[e] = s;
  }
}

// out[i, a] = sum over l, c of Y[l, i, c] G[l, a, c] (out: row pitch op).
template <typename T>
__device__ void unfold_dots(const T* Y, const T* G, int L, int NI, int MA, int C, int op, T* out) {
  for (int e = threadIdx.x; e < NI * MA; e += blockDim.x) {
    const int i = e / MA, a = e - i * MA;
    T s = T(0);
    for (int l = 0; l < L; ++l) {
      const T* y = Y + (l * NI + i) * C;
      const T* g = G + (l * MA + a) * C;
      for (int c = 0; c < C; ++c) s = fma(y[c], g[c], s);
    }
    out[i * op + a] = s;
  }
}

// The MU step of a factor: Fn[i, a] from the old F, the numerators (pitch fp) and
// den = F H; Fn is another buffer, so every row of the old F stays readable.
template <typename T>
__device__ void mu_factor(const T* F, const T* num, const T* H, int N, int fp, int m, T eps,
                          T* Fn) {
  for (int e = threadIdx.x; e < N * m; e += blockDim.x) {
    const int i = e / m, a = e - i * m;
    const T* f = F + i * fp;
    T den = T(0);
    for (int w = 0; w < m; ++w) den = fma(f[w], H[w * m + a], den);
    const T v = f[a] * num[i * fp + a] / (den > eps ? den : eps);
    Fn[i * fp + a] = v > T(0) ? v : T(0);
  }
}


}  // namespace blk
}  // namespace nnc
