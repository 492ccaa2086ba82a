// nnTD of one small 3-way tensor by one thread-block cluster (Alg. 1, step 1):
// all sweeps of a fit in one launch.
//
// A sweep of a small tensor on the kernels of sweep.cu is a chain of eleven launches of
// a few microseconds each on a handful of blocks; its arithmetic would take one
// or two. Here the CTAs of a cluster share the sweep through distributed shared
// memory. CTA c owns the mode-1 slices i, the mode-2 slices j and the mode-3 slices k of
// its range and keeps a full copy of the factors, Grams and core; all CTAs hold the
// same bits. With S_k = F_k^T F_k, a sweep is
//   T  = X x_2 F2^T   on its i      Y1 = T x_3 F3^T,   Num1, H1, new rows F1[i]
//                                   -> every CTA                      (barrier 1)
//   P1 = X x_1 F1^T   on its j      Y2 = P1 x_3 F3^T,  Num2, H2, new rows F2[j]
//                     its share of Y3 = P1 x_2 F2^T (its j)
//                                   rows F2[j] -> every CTA           (barrier 2)
//   Y3 on its k       from every CTA's share;  Num3, H3, new rows F3[k]
//                     its share of M = Y3 x_3 F3^T (its k)
//                                   rows and share -> every CTA       (barrier 3)
//   G                 M added in CTA order, D = G x_k S_k: in every CTA alike
// and the trace entry sqrt(||X||^2 - 2 <M, G> + sum S1 .* H1^T) / ||X|| of the sweep,
// whose H1 the next sweep forms (FP64 sums, CTA 0). X is read twice per sweep, each CTA
// its slabs only, which it keeps in shared memory. Rows that a CTA sends land in the copy of the
// factor that no CTA reads any more (two copies, swapped at the barrier).
//
// What bounds it is the latency of its short contractions (about 15 intervals between
// block barriers and three cluster barriers a sweep), in FP64 also GB300's FP64
// rate on the cluster's SMs, hence the limits of ntd_cluster_fits.
#include <cooperative_groups.h>

#include <algorithm>

#include "blk.cuh"
#include "kernels.cuh"
#include "ntd.cuh"

namespace nnc {
namespace cg = cooperative_groups;
using namespace blk;
namespace {

// The last kClSide threads run what an interval does beside its main contraction.
constexpr int kClThreads = 512, kClSide = 128, kClMain = kClThreads - kClSide;
template <typename T>
constexpr int cl_ctas() { return sizeof(T) == 8 ? 16 : 8; }

template <typename T>
struct ClArgs {
  const T* X;
  int N[3], m[3];
  T* F[3];
  T* G;
  int iters;
  T eps;
  const double* x2;  // ||X||^2
  double* trace;     // may be NULL
  int* counter;      // trace_record's pair
};

// Offsets (elements) of one CTA's shared memory.
template <typename T>
struct ClSizes {
  int f, g, s, y, p, y3, num, mm, xi, xj, total;
  int fo[3], so[3];
  __host__ __device__ ClSizes(const int* N, const int* m, int ctas) {
    const int cp = rpitch<T>(N[2]);
    const int ni = (N[0] + ctas - 1) / ctas, nj = (N[1] + ctas - 1) / ctas,
              nk = (N[2] + ctas - 1) / ctas;
    f = s = num = mm = 0;
    for (int k = 0; k < 3; ++k) {
      fo[k] = f;
      f += (N[k] * fpitch<T>(m[k]) + 3) & ~3;
      so[k] = s;
      s += (m[k] * m[k] + 3) & ~3;
      const int rows = k == 0 ? ni : (k == 1 ? nj : nk);
      num = num > rows * fpitch<T>(m[k]) ? num : rows * fpitch<T>(m[k]);
      mm = m[k] * m[k] > mm ? m[k] * m[k] : mm;
    }
    num = (num + 3) & ~3;
    mm = (mm + 3) & ~3;
    g = (m[0] * m[1] * m[2] + 3) & ~3;
    const int y1 = ni * m[1] * m[2], y2 = m[0] * nj * m[2], y3k = m[0] * m[1] * nk;
    y = ((y1 > y2 ? (y1 > y3k ? y1 : y3k) : (y2 > y3k ? y2 : y3k)) + 3) & ~3;
    const int pa = ni * m[1] * cp, pb = m[0] * nj * cp;
    p = ((pa > pb ? pa : pb) + 3) & ~3;
    y3 = (m[0] * m[1] * N[2] + 3) & ~3;
    xi = (ni * N[1] * N[2] + 3) & ~3;
    xj = (N[0] * nj * N[2] + 3) & ~3;
    // F twice, G, W, W2, M, one share of M per CTA, S (S1 twice), Y, P, Y3's share, Num,
    // H, the slabs of X
    total = 2 * f + (4 + ctas) * g + s + ((m[0] * m[0] + 3) & ~3) + y + p + y3 + num + mm + xi + xj;
  }
};

// Thread t of a group of n (whole warps).
struct Grp {
  int t, n;
};

// out(e) = sum_{q < len} term(e, q, .) for e < nout: LS consecutive lanes share an output,
// lane u adds the terms u, u + LS, ... in order, a fixed shuffle tree the lanes. The
// contractions of a small fit are few and long chains; this keeps LS of them moving.
template <int LS, typename T, typename Term, typename Out>
__device__ __forceinline__ void dots_ls(Grp g, int nout, int len, Term term, Out out) {
  const int per = g.n / LS, u = g.t % LS;
  for (int e0 = 0; e0 < nout; e0 += per) {
    const int e = e0 + g.t / LS;
    T s = T(0);
    if (e < nout) {
#pragma unroll 4
      for (int q = u; q < len; q += LS) s = term(e, q, s);
    }
#pragma unroll
    for (int o = LS / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (e < nout && u == 0) out(e, s);
  }
}
// Lanes per output by the shape alone: 16 where the group has them, else 4.
template <typename T, typename Term, typename Out>
__device__ __forceinline__ void dots(Grp g, int nout, int len, Term term, Out out) {
  if (nout * 16 <= g.n && len > 16) dots_ls<16, T>(g, nout, len, term, out);
  else dots_ls<4, T>(g, nout, len, term, out);
}

template <typename T>
__device__ __forceinline__ void gram(Grp g, const T* F, int N, int fp, int m, T* S) {
  dots<T>(g, m * m, N, [&](int e, int i, T s) {
    const int x = e / m;
    return fma(F[i * fp + x], F[i * fp + e - x * m], s);
  }, [&](int e, T s) { S[e] = s; });
}

// out[l, p, c] = sum_j F[j, p] X[l, j, c], p < Q, c < C, X in shared memory (F: J x QP,
// zero past Q); column c = (j', k) of N3 entries per row goes to
// out[((l Q + p) C / N3 + j') cp + k]. LS lanes share a column: lane group u takes the rows
// j = u, u + LS, ..., and the sums are added by a fixed shuffle tree.
template <typename T, int QP, int LS>
__device__ __forceinline__ void slab_pass(Grp g, const T* X, int L, int J, int C, int N3, int cp,
                                          const T* F, int Q, T* out) {
  constexpr int VW = 16 / (int)sizeof(T), CW = 32 / LS;
  const int total = L * C, rows = C / N3;
  const int u = (g.t & 31) / CW, per = g.n / LS;
  for (int e0 = 0; e0 < total; e0 += per) {
    const int e = e0 + (g.t >> 5) * CW + (g.t & (CW - 1));
    const bool on = e < total;
    const int l = on ? e / C : 0, c = on ? e - l * C : 0;
    const T* x = X + l * J * C + c;
    T acc[QP];
#pragma unroll
    for (int p = 0; p < QP; ++p) acc[p] = T(0);
#pragma unroll 4
    for (int j = u; j < J; j += LS) {
      const T v = x[j * C];
#pragma unroll
      for (int p = 0; p < QP; p += VW) {
        T w[VW];
        ldv<T, VW>(F + j * QP + p, w);
#pragma unroll
        for (int b = 0; b < VW; ++b) acc[p + b] = fma(v, w[b], acc[p + b]);
      }
    }
#pragma unroll
    for (int p = 0; p < QP; ++p)
#pragma unroll
      for (int o = 16; o >= CW; o >>= 1) acc[p] += __shfl_xor_sync(0xffffffffu, acc[p], o);
    if (on) {
      const int jr = c / N3, k = c - jr * N3;
      T* o = out + (l * Q * rows + jr) * cp + k;
#pragma unroll
      for (int p = 0; p < QP; ++p)
        if (p < Q && (p & (LS - 1)) == u) o[p * rows * cp] = acc[p];
    }
  }
}
template <typename T>
__device__ __forceinline__ void slab_pass(Grp g, const T* X, int L, int J, int C, int N3, int cp,
                                          const T* F, int Q, T* out) {
  // Four lanes a column where one lane each would leave threads idle on long columns.
  const bool split = J >= 16 && L * C < 2 * g.n;
  by_width<T, 8>(Q, [&](auto w) {
    constexpr int QP = decltype(w)::value;
    if (split) slab_pass<T, QP, 4>(g, X, L, J, C, N3, cp, F, Q, out);
    else slab_pass<T, QP, 1>(g, X, L, J, C, N3, cp, F, Q, out);
  });
}

// core_gram (blk.cuh) on a group.
template <typename T>
__device__ __forceinline__ void core_gram_g(Grp g, const T* in, int L, int J, int C, const T* A,
                                            T* out) {
  for (int e = g.t; e < L * J * C; e += g.n) {
    const int c = e % C, lp = e / C, p = lp % J, l = lp / J;
    const T* x = in + l * J * C + c;
    T s = T(0);
#pragma unroll 4
    for (int j = 0; j < J; ++j) s = fma(A[p * J + j], x[j * C], s);
    out[e] = s;
  }
}

template <typename T>
__global__ void __launch_bounds__(kClThreads)
ntd_cluster_kernel(ClArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cg::cluster_group cl = cg::this_cluster();
  const int c = (int)cl.block_rank(), ctas = (int)cl.num_blocks();
  const int N1 = a.N[0], N2 = a.N[1], N3 = a.N[2];
  const int m1 = a.m[0], m2 = a.m[1], m3 = a.m[2], ng = m1 * m2 * m3;
  const ClSizes<T> z(a.N, a.m, ctas);
  const int p1 = fpitch<T>(m1), p2 = fpitch<T>(m2), p3 = fpitch<T>(m3), cp = rpitch<T>(N3);
  const int li = (N1 + ctas - 1) / ctas, lj = (N2 + ctas - 1) / ctas, lk = (N3 + ctas - 1) / ctas;
  const int i0 = min(c * li, N1), ni = min(li, N1 - i0);
  const int j0 = min(c * lj, N2), nj = min(lj, N2 - j0);
  const int k0 = min(c * lk, N3), nk = min(lk, N3 - k0);
  T* sm = reinterpret_cast<T*>(smem_raw);
  T* F[2] = {sm, sm + z.f};  // the two copies of all factors
  T* G = sm + 2 * z.f;
  T* W = G + z.g;
  T* W2 = W + z.g;
  T* M = W2 + z.g;
  T* Msh = M + z.g;  // [CTA][ng]
  T* S = Msh + ctas * z.g;
  T* Sa[2] = {S + z.so[0], S + z.s};  // S1 of this sweep and of the one before
  T* S1 = Sa[0];
  T* S2 = S + z.so[1];
  T* S3 = S + z.so[2];
  T* Y = S + z.s + ((m1 * m1 + 3) & ~3);
  T* P = Y + z.y;
  T* Y3 = P + z.p;  // this CTA's share, (m1, m2, N3)
  T* num = Y3 + z.y3;
  T* H = num + z.num;
  T* Xi = H + z.mm;  // X[i in this CTA's range]
  T* Xj = Xi + z.xi;  // X[:, j in this CTA's range]
  const T* X = a.X;
  const int tid = threadIdx.x;
  const Grp all{tid, kClThreads}, main{tid, kClMain}, side{tid - kClMain, kClSide};
  const Grp gramg{tid - kClMain, kClSide - 32};
  const bool is_main = tid < kClMain;

  for (int n = 0; n < 3; ++n) {
    const int fp = fpitch<T>(a.m[n]), mn = a.m[n];
    for (int e = tid; e < a.N[n] * fp; e += kClThreads) {
      const int i = e / fp, v = e - i * fp;
      F[0][z.fo[n] + e] = v < mn ? a.F[n][i * mn + v] : T(0);
      F[1][z.fo[n] + e] = T(0);
    }
  }
  for (int e = tid; e < ng; e += kClThreads) G[e] = a.G[e];
  for (int e = tid; e < ni * N2 * N3; e += kClThreads) Xi[e] = X[(int64_t)i0 * N2 * N3 + e];
  for (int e = tid; e < N1 * nj * N3; e += kClThreads) {
    const int i = e / (nj * N3), r = e - i * nj * N3;
    Xj[e] = X[((int64_t)i * N2 + j0) * N3 + r];
  }
  int cur[3] = {0, 0, 0};  // the copy of each factor in use
  auto fac = [&](int n) { return F[cur[n]] + z.fo[n]; };
  auto other = [&](int n) { return F[cur[n] ^ 1] + z.fo[n]; };
  __syncthreads();
  // (the same groups as in the sweeps, so that a resumed fit has the same bits)
  if (!is_main) {
    if (tid < kClThreads - 32) gram<T>(gramg, fac(0), N1, p1, m1, S1);
    gram<T>(side, fac(1), N2, p2, m2, S2);
  }
  gram<T>(all, fac(2), N3, p3, m3, S3);
  // No CTA sends before every CTA's copies are zeroed.
  cl.sync();

  // The MU step on this CTA's rows r0 .. r0 + rows - 1 of factor n (numerators num, pitch
  // fp, den = F H), sent to every CTA's other copy.
  auto send_rows = [&](int n, int r0, int rows, int fp, int mn) {
    const T* f = fac(n);
    T* dst = other(n);
    for (int e = tid; e < rows * mn; e += kClThreads) {
      const int i = e / mn, v = e - i * mn;
      const T* row = f + (r0 + i) * fp;
      T den = T(0);
      for (int w = 0; w < mn; ++w) den = fma(row[w], H[w * mn + v], den);
      T x = row[v] * num[i * fp + v] / (den > a.eps ? den : a.eps);
      x = x > T(0) ? x : T(0);
      T* o = dst + (r0 + i) * fp + v;
      for (int q = 0; q < ctas; ++q) *cl.map_shared_rank(o, q) = x;
    }
  };
  // H = unfold_n(W2) unfold_n(G)^T.
  auto h_of_1 = [&](Grp g) {
    dots<T>(g, m1 * m1, m2 * m3, [&](int e, int q, T x) {
      const int i = e / m1;
      return fma(W2[i * m2 * m3 + q], G[(e - i * m1) * m2 * m3 + q], x);
    }, [&](int e, T x) { H[e] = x; });
  };
  // The trace entry of the sweep before, by one warp of CTA 0: M and G are that sweep's, H
  // is H1 of its new core, S1 the copy `which` (FP64 sums in a fixed order).
  auto record = [&](int which) {
    if (c != 0) return;
    const int lane = tid & 31;
    const T* s1 = Sa[which];
    double mg = 0.0, gd = 0.0;
    for (int e = lane; e < ng; e += 32) mg += (double)M[e] * (double)G[e];
    for (int e = lane; e < m1 * m1; e += 32)
      gd += (double)s1[e] * (double)H[(e % m1) * m1 + e / m1];
    mg = warp_sum(mg);
    gd = warp_sum(gd);
    if (lane == 0) {
      const double xx = a.x2[0];
      double r2 = xx - 2.0 * mg + gd;
      const bool finite = isfinite(r2);
      if (r2 < 0.0) r2 = 0.0;
      trace_record(a.counter, a.trace, 1, sqrt(r2 / xx), finite);
    }
  };

  for (int it = 0; it < a.iters; ++it) {
    // ---- mode 1
    if (is_main)
      slab_pass<T>(main, Xi, ni, N2, N3, N3, cp, fac(1), m2, P);
    else core_gram_g(side, G, m1, m2, m3, S2, W);
    __syncthreads();
    if (is_main) {
      const T* f3 = fac(2);
      dots<T>(main, ni * m2 * m3, N3, [&](int e, int k, T x) {
        const int r = e / m3;
        return fma(P[r * cp + k], f3[k * p3 + e - r * m3], x);
      }, [&](int e, T x) { Y[e] = x; });
    } else {
      core_gram_g(side, W, m1 * m2, m3, 1, S3, W2);
    }
    __syncthreads();
    if (is_main)
      dots<T>(main, ni * m1, m2 * m3, [&](int e, int q, T x) {
        const int i = e / m1;
        return fma(Y[i * m2 * m3 + q], G[(e - i * m1) * m2 * m3 + q], x);
      }, [&](int e, T x) { num[(e / m1) * p1 + e % m1] = x; });
    else h_of_1(side);
    __syncthreads();
    send_rows(0, i0, ni, p1, m1);
    cl.sync();
    cur[0] ^= 1;
    // ---- mode 2
    if (is_main) {
      slab_pass<T>(main, Xj, 1, N1, nj * N3, N3, cp, fac(0), m1, P);
    } else {
      // The last warp records the sweep before (its S1 is the other copy).
      if (it > 0 && tid >= kClThreads - 32) record(it & 1);
      S1 = Sa[(it + 1) & 1];
      if (tid < kClThreads - 32) gram<T>(gramg, fac(0), N1, p1, m1, S1);
    }
    S1 = Sa[(it + 1) & 1];
    __syncthreads();
    if (is_main) {
      const T* f3 = fac(2);
      dots<T>(main, m1 * nj * m3, N3, [&](int e, int k, T x) {  // Y2 (m1, nj, m3)
        const int r = e / m3;
        return fma(P[r * cp + k], f3[k * p3 + e - r * m3], x);
      }, [&](int e, T x) { Y[e] = x; });
    } else {
      core_gram_g(side, G, 1, m1, m2 * m3, S1, W);
    }
    __syncthreads();
    if (is_main)
      dots<T>(main, nj * m2, m1 * m3, [&](int e, int q, T x) {
        const int j = e / m2, b = e - j * m2, aa = q / m3, cc = q - aa * m3;
        return fma(Y[(aa * nj + j) * m3 + cc], G[(aa * m2 + b) * m3 + cc], x);
      }, [&](int e, T x) { num[(e / m2) * p2 + e % m2] = x; });
    else core_gram_g(side, W, m1 * m2, m3, 1, S3, W2);
    __syncthreads();
    dots<T>(all, m2 * m2, m1 * m3, [&](int e, int q, T x) {
      const int i = e / m2, b = e - i * m2, aa = q / m3, cc = q - aa * m3;
      return fma(W2[(aa * m2 + i) * m3 + cc], G[(aa * m2 + b) * m3 + cc], x);
    }, [&](int e, T x) { H[e] = x; });
    __syncthreads();
    send_rows(1, j0, nj, p2, m2);
    __syncthreads();
    // ---- this CTA's share of Y3 = P1 x_2 F2^T (m1, m2, N3)
    {
      const T* f2 = other(1) + j0 * p2;
      for (int e = tid; e < m1 * m2 * N3; e += kClThreads) {
        const int k = e % N3, ab = e / N3, b = ab % m2, aa = ab / m2;
        const T* x = P + (int64_t)aa * nj * cp + k;
        T s = T(0);
#pragma unroll 4
        for (int j = 0; j < nj; ++j) s = fma(f2[j * p2 + b], x[j * cp], s);
        Y3[e] = s;
      }
    }
    cl.sync();
    cur[1] ^= 1;
    // ---- mode 3: Y3 on this CTA's k, shares in CTA order
    if (is_main) {
      for (int e = tid; e < m1 * m2 * nk; e += kClMain) {
        const int ab = e / nk, k = k0 + e - ab * nk;
        T v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q)
          v[q] = q < ctas ? cl.map_shared_rank(Y3, q)[ab * N3 + k] : T(0);
        T s = v[0];
#pragma unroll
        for (int q = 1; q < 16; ++q)
          if (q < ctas) s += v[q];
        Y[e] = s;
      }
    } else {
      gram<T>(side, fac(1), N2, p2, m2, S2);
    }
    __syncthreads();
    if (is_main)
      dots<T>(main, nk * m3, m1 * m2, [&](int e, int ab, T x) {
        const int k = e / m3;
        return fma(Y[ab * nk + k], G[ab * m3 + e - k * m3], x);
      }, [&](int e, T x) { num[(e / m3) * p3 + e % m3] = x; });
    else core_gram_g(side, W, m1, m2, m3, S2, W2);  // G x_1 S1 x_2 S2
    __syncthreads();
    dots<T>(all, m3 * m3, m1 * m2, [&](int e, int ab, T x) {
      const int i = e / m3;
      return fma(W2[ab * m3 + i], G[ab * m3 + e - i * m3], x);
    }, [&](int e, T x) { H[e] = x; });
    __syncthreads();
    send_rows(2, k0, nk, p3, m3);
    __syncthreads();
    // ---- this CTA's share of M = Y3 x_3 F3^T, to every CTA
    {
      const T* f3 = other(2) + k0 * p3;
      for (int e = tid; e < ng; e += kClThreads) {
        const int cc = e % m3, ab = e / m3;
        T s = T(0);
#pragma unroll 4
        for (int k = 0; k < nk; ++k) s = fma(Y[ab * nk + k], f3[k * p3 + cc], s);
        T* o = Msh + c * z.g + e;
        for (int q = 0; q < ctas; ++q) *cl.map_shared_rank(o, q) = s;
      }
    }
    cl.sync();
    cur[2] ^= 1;
    // ---- the core, in every CTA alike
    gram<T>(all, fac(2), N3, p3, m3, S3);
    __syncthreads();
    for (int e = tid; e < ng; e += kClThreads) {
      T mv = Msh[e];
      for (int q = 1; q < ctas; ++q) mv += Msh[q * z.g + e];
      M[e] = mv;
      const int cc = e % m3, ab = e / m3;
      T den = T(0);
      for (int w = 0; w < m3; ++w) den = fma(W2[ab * m3 + w], S3[w * m3 + cc], den);
      const T v = G[e] * mv / (den > a.eps ? den : a.eps);
      G[e] = v > T(0) ? v : T(0);
    }
    __syncthreads();
  }
  if (a.iters > 0) {  // the last sweep's trace entry
    core_gram_g(all, G, m1, m2, m3, S2, W);
    __syncthreads();
    core_gram_g(all, W, m1 * m2, m3, 1, S3, W2);
    __syncthreads();
    if (!is_main) h_of_1(side);
    __syncthreads();
    if (tid < 32) record(a.iters & 1);
  }
  if (c == 0) {
    for (int n = 0; n < 3; ++n) {
      const int fp = fpitch<T>(a.m[n]), mn = a.m[n];
      for (int e = tid; e < a.N[n] * mn; e += kClThreads)
        a.F[n][e] = fac(n)[(e / mn) * fp + e % mn];
    }
    for (int e = tid; e < ng; e += kClThreads) a.G[e] = G[e];
  }
  // No CTA leaves while another may still reach its shared memory.
  cl.sync();
}

template <typename T>
int launch(const ClArgs<T>& a, size_t smem, cudaStream_t s, bool probe = false) {
  auto kern = ntd_cluster_kernel<T>;
  NNC_CUDA_TRY(raise_smem_limit((const void*)kern, smem));
  if (cl_ctas<T>() > 8)
    NNC_CUDA_TRY(cudaFuncSetAttribute((const void*)kern,
                                      cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(cl_ctas<T>());
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cl_ctas<T>();
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (probe) {  // can the device place one such cluster?
    int n = 0;
    const bool ok = cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0;
    if (!ok) (void)cudaGetLastError();
    return ok ? NNC_OK : NNC_ERR_UNSUPPORTED;
  }
  NNC_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, a));
  note_launch(s);
  return NNC_OK;
}

}  // namespace

// Largest |X| (m1 + m2), the products of the two passes of a sweep, and largest multirank
// entry. us per sweep, the kernels of sweep.cu against this one (the call besides: 730
// against 240 us, no graph to capture):
//   FP32  5 x 61 x 201, m 3     55.6   17.1      FP64  5 x 61 x 201, m 3   133.4   51.7
//         40^3, m 5             42.8   17.0            11 x 64 x 64, m 3    85.5   25.8
//         33 x 47 x 51, m 10    42.3   45.8            40^3, m 5            73.4   52.3
//         20^3, m (16, 5, 16)   44.3   41.1
template <typename T>
constexpr int64_t kNtdClusterWork = sizeof(T) == 8 ? 800000 : 1200000;
constexpr int kNtdClusterM = 8;

template <typename T>
bool ntd_cluster_fits(const int64_t* dims, const int* m) {
  int64_t n = 1;
  for (int k = 0; k < 3; ++k) {
    if (dims[k] > 1 << 16 || m[k] > kNtdClusterM) return false;
    n *= dims[k];
    if (n > 1 << 24) return false;
  }
  if (n * (m[0] + m[1]) > kNtdClusterWork<T>) return false;
  const int N[3] = {(int)dims[0], (int)dims[1], (int)dims[2]};
  const size_t smem = (size_t)ClSizes<T>(N, m, cl_ctas<T>()).total * sizeof(T);
  if (smem > kSmemBudget) return false;
  return launch<T>(ClArgs<T>{}, smem, nullptr, true) == NNC_OK;
}

template <typename T>
int ntd_cluster_sweeps(const T* X, const int64_t* dims, const int* m, T* const* F, T* G, double eps,
                       int sweeps, const double* x2, double* trace, int* counter, cudaStream_t s) {
  ClArgs<T> a{};
  a.X = X;
  for (int k = 0; k < 3; ++k) {
    a.N[k] = (int)dims[k];
    a.m[k] = m[k];
    a.F[k] = F[k];
  }
  a.G = G;
  a.iters = sweeps;
  a.eps = (T)eps;
  a.x2 = x2;
  a.trace = trace;
  a.counter = counter;
  const size_t smem = (size_t)ClSizes<T>(a.N, a.m, cl_ctas<T>()).total * sizeof(T);
  return launch<T>(a, smem, s);
}

template bool ntd_cluster_fits<float>(const int64_t*, const int*);
template bool ntd_cluster_fits<double>(const int64_t*, const int*);
template int ntd_cluster_sweeps<float>(const float*, const int64_t*, const int*, float* const*,
                                       float*, double, int, const double*, double*, int*,
                                       cudaStream_t);
template int ntd_cluster_sweeps<double>(const double*, const int64_t*, const int*, double* const*,
                                        double*, double, int, const double*, double*, int*,
                                        cudaStream_t);

}  // namespace nnc
