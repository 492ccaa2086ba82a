// The lift A^(n) = F^(n) B^(n) and the one-pass reconstruction residual.
//
// recon_residual streams X once. The model is first reduced to rows U[t, :]
// (length K = m_d for Tucker, r for CP), t running over (i_1, ..., i_{d-1}):
//   Tucker: U = G x_1 F^(1) ... x_{d-1} F^(d-1)
//   CP:     U[t, q] = A^(1)[i_1, q] ... A^(d-1)[i_{d-1}, q]
// and X_hat[t, k] = sum_c U[t, c] F^(d)[k, c] (A^(d) for CP), by
// Eq. TD:matrix-format and Eq. CPD:matrix-format contracted mode by mode.
// The streaming kernel gives each thread one k (F^(d)[k, :] in registers) and
// a tile of rows (U rows in shared memory), forms X_hat in T and accumulates
// (x - x_hat)^2 and x^2 (FP32 per thread for float data, FP64 across threads
// and blocks); per-block partials are added in block order.
#include <type_traits>

#include "kernels.cuh"
#include "residual.cuh"

namespace nnc {
namespace {

template <typename T>
__global__ void lift_kernel(const T* __restrict__ F, const T* __restrict__ B, int64_t N, int M,
                            int r, T* __restrict__ A) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N * r;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / r;
    const int q = (int)(e % r);
    T s = T(0);
    for (int a = 0; a < M; ++a) s = fma(F[i * M + a], B[(int64_t)a * r + q], s);
    A[e] = s;
  }
}

// out[l, q, c] = sum_j A[q, j] Y[l, j, c] for any Q, J <= 64: a block takes 256
// flattened columns (l, c) and 16 outputs q, so an entry of Y serves 16 products and the
// writes of out, the largest array here, are whole rows of c. (One thread per output
// read Y once per product and divided for every output: the three products of a
// 128^3 x 64 fit, 134 MB written by the last, 400 -> 98 us.)
constexpr int kMpThreads = 256, kMpQ = 16;
template <typename T>
__global__ void __launch_bounds__(kMpThreads)
mode_product_any_kernel(const T* __restrict__ Y, int64_t L, int J, int64_t C, unsigned col_blocks,
                        const T* __restrict__ A, int Q, T* __restrict__ out) {
  __shared__ T as[64 * kMpQ];
  // Tiles of q and of columns in one grid dimension: a mode may have any length.
  const int q0 = (int)(blockIdx.x / col_blocks) * kMpQ, qn = Q - q0 < kMpQ ? Q - q0 : kMpQ;
  for (int e = threadIdx.x; e < J * kMpQ; e += kMpThreads) {
    const int j = e / kMpQ, q = e % kMpQ;
    as[e] = q < qn ? A[(int64_t)(q0 + q) * J + j] : T(0);
  }
  __syncthreads();
  const int64_t col = (int64_t)(blockIdx.x % col_blocks) * kMpThreads + threadIdx.x;
  if (col >= L * C) return;
  const int64_t l = col / C, c = col - l * C;
  const T* y = Y + l * J * C + c;
  T acc[kMpQ];
#pragma unroll
  for (int q = 0; q < kMpQ; ++q) acc[q] = T(0);
#pragma unroll 4
  for (int j = 0; j < J; ++j) {
    const T v = y[(int64_t)j * C];
#pragma unroll
    for (int q = 0; q < kMpQ; ++q) acc[q] = fma(as[j * kMpQ + q], v, acc[q]);
  }
  T* o = out + (l * Q + q0) * C + c;
#pragma unroll
  for (int q = 0; q < kMpQ; ++q)
    if (q < qn) o[q * C] = acc[q];
}

template <typename T>
__global__ void cp_rows_kernel(const T* __restrict__ A1, const T* __restrict__ A2, int64_t N1,
                               int64_t N2, int r, T* __restrict__ U) {
  const int64_t n = N1 * N2 * r;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int q = (int)(e % r);
    const int64_t j = (e / r) % N2;
    const int64_t i = e / (r * N2);
    U[e] = A1[i * r + q] * A2[j * r + q];
  }
}

constexpr int kResThreads = 128;
// U rows staged at a time (16 KB of FP32: a thread of a short-rowed X walks few of them).
__host__ __device__ constexpr int res_rows(int km) { return 4096 / km; }

// The k tile of a block: tx threads (a power of two, so that short rows of X use
// every thread) times KT columns each; rows per block.
template <typename T>
__host__ __device__ constexpr int res_kt(int km) { return sizeof(T) == 8 ? 1 : 64 / km; }
template <typename T>
inline int res_km(int K) { return K <= 16 ? 16 : (K <= 32 ? 32 : 64); }
struct ResGrid {
  int tx, rows;
  int64_t ktiles, blocks;
};
template <typename T>
ResGrid res_grid(int64_t R, int64_t N3, int K) {
  const int kt = res_kt<T>(res_km<T>(K));
  ResGrid g;
  g.tx = 1;
  while (g.tx < kResThreads && (int64_t)g.tx * kt < N3) g.tx *= 2;
  g.ktiles = ceil_div(N3, (int64_t)g.tx * kt);
  // A block loads its columns' rows of F^(d) once: as many rows as still leave several
  // blocks per SM.
  const int chunk = res_rows(res_km<T>(K));
  g.rows = 64;
  while (g.rows < 2 * chunk && g.ktiles * ceil_div(R, 2 * g.rows) >= 6LL * device_sm_count())
    g.rows *= 2;
  g.blocks = g.ktiles * ceil_div(R, (int64_t)g.rows);
  return g;
}

// Block (k tile, row tile). A thread keeps F3[k, :] of KT columns k = k0, k0 + tx, ...
// in registers (KM >= K entries, zero past K); the block's U rows sit in shared
// memory and are read in 16-byte broadcasts that serve KT products per entry
// (one column a thread, one row at a time: 512^3, K = 32, 519 us and 128^3 x 64, K = 16,
// 824 us, half of its threads past the row's end).
// Per element: x_hat = U[t, :] . F3[k, :] in T, then (x - x_hat)^2 and x^2. For T =
// float the thread adds at most 64 terms in one FP32 chain (rounded to nearest, so the errors
// are mostly unbiased; equal terms round alike, and 64 of them stay within 33 roundings), the chains
// of a chunk in a pair of floats with the error of every addition kept, the chunks in FP64:
// GB300's FP64 rate is far below its FP32 rate, and FP64 arithmetic per element would bound the
// pass (one FP64 addition and conversion a chain: 424 -> 446 us at 512^3, this 426 us). The block
// sums and the partials are FP64.
template <typename T, int KM, int KT>
__global__ void __launch_bounds__(kResThreads)
residual_stream_kernel(const T* __restrict__ X, int64_t R, int64_t N3, const T* __restrict__ U,
                       int K, const T* __restrict__ F3, int tx, int64_t ktiles, int rows,
                       double* __restrict__ part) {
  constexpr int kRows = res_rows(KM);
  __shared__ __align__(16) T us[kRows * KM];
  __shared__ double red[32];
  const int ty = kResThreads / tx, sub = threadIdx.x / tx;
  const int64_t k0 = (blockIdx.x % ktiles) * tx * KT + (threadIdx.x & (tx - 1));
  T f[KT][KM];
  bool act[KT];
#pragma unroll
  for (int u = 0; u < KT; ++u) {
    const int64_t k = k0 + (int64_t)u * tx;
    act[u] = k < N3;
#pragma unroll
    for (int c = 0; c < KM; ++c) f[u][c] = (act[u] && c < K) ? F3[k * K + c] : T(0);
  }
  const int64_t rb = (blockIdx.x / ktiles) * rows;
  const int64_t rend = rb + rows < R ? rb + rows : R;
  double td2 = 0.0, tx2 = 0.0;
  for (int64_t r0 = rb; r0 < rend; r0 += kRows) {
    const int nr = (int)(r0 + kRows < rend ? kRows : rend - r0);
    __syncthreads();
    for (int e = threadIdx.x; e < nr * KM; e += kResThreads) {
      const int row = e / KM, c = e % KM;
      us[e] = c < K ? U[(r0 + row) * K + c] : T(0);
    }
    __syncthreads();
    T d2 = T(0), x2 = T(0);
    T cd[2] = {T(0), T(0)}, cx[2] = {T(0), T(0)};  // sum and what its additions rounded off
    const T* xp = X + r0 * N3 + k0;
    // Four rows at a time, their entries of X requested one round ahead.
    constexpr int RU = 4, kRounds = 64 / (RU * KT);
    int rounds = 0;
    auto add = [](T (&c)[2], T v) {
      const T t = c[0] + v, b = t - c[0];
      c[1] += (c[0] - (t - b)) + (v - b);
      c[0] = t;
    };
    auto flush = [&]() {
      add(cd, d2);
      add(cx, x2);
      d2 = x2 = T(0);
    };
    T nx[RU][KT];
    auto fetch = [&](int row) {
#pragma unroll
      for (int q = 0; q < RU; ++q)
#pragma unroll
        for (int u = 0; u < KT; ++u)
          nx[q][u] = act[u] && row + q * ty < nr
                         ? __ldg(xp + (int64_t)(row + q * ty) * N3 + (int64_t)u * tx)
                         : T(0);
    };
    fetch(sub);
    for (int row = sub; row < nr; row += RU * ty) {
      T x[RU][KT];
#pragma unroll
      for (int q = 0; q < RU; ++q)
#pragma unroll
        for (int u = 0; u < KT; ++u) x[q][u] = nx[q][u];
      fetch(row + RU * ty);
#pragma unroll
      for (int q = 0; q < RU; ++q) {
        if (row + q * ty >= nr) break;
        T h0[KT], h1[KT];
#pragma unroll
        for (int u = 0; u < KT; ++u) h0[u] = h1[u] = T(0);
        const T* ur = us + (row + q * ty) * KM;
#pragma unroll
        for (int c = 0; c < KM; c += 4) {
          T w[4];
          if constexpr (sizeof(T) == 4) {
            const float4 t = *reinterpret_cast<const float4*>(ur + c);
            w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
          } else {
            const double2 t0 = *reinterpret_cast<const double2*>(ur + c);
            const double2 t1 = *reinterpret_cast<const double2*>(ur + c + 2);
            w[0] = t0.x; w[1] = t0.y; w[2] = t1.x; w[3] = t1.y;
          }
#pragma unroll
          for (int u = 0; u < KT; ++u) {
            h0[u] = fma(w[0], f[u][c], h0[u]);
            h1[u] = fma(w[1], f[u][c + 1], h1[u]);
            h0[u] = fma(w[2], f[u][c + 2], h0[u]);
            h1[u] = fma(w[3], f[u][c + 3], h1[u]);
          }
        }
#pragma unroll
        for (int u = 0; u < KT; ++u) {
          // (a column past the end has x = 0 and f = 0)
          const T dd = x[q][u] - (h0[u] + h1[u]);
          d2 = fma(dd, dd, d2);
          x2 = fma(x[q][u], x[q][u], x2);
        }
      }
      if (++rounds == kRounds) {
        flush();
        rounds = 0;
      }
    }
    flush();
    const double cd2 = (double)cd[0] + (double)cd[1], cx2 = (double)cx[0] + (double)cx[1];
    if (isfinite(cd2) && isfinite(cx2)) {
      td2 += cd2;
      tx2 += cx2;
    } else {
      // The FP32 terms overflowed (entries beyond about 1e19): these rows again
      // with FP64 terms. Non-finite data stays non-finite.
      for (int row = sub; row < nr; row += ty)
        for (int u = 0; u < KT; ++u) {
          const int64_t k = k0 + (int64_t)u * tx;
          if (k >= N3) continue;
          const double x = (double)xp[(int64_t)row * N3 + (int64_t)u * tx];
          double h = 0.0;
          for (int c = 0; c < K; ++c) h = fma((double)us[row * KM + c], (double)F3[k * K + c], h);
          const double dd = x - h;
          td2 += dd * dd;
          tx2 += x * x;
        }
    }
  }
  const double bd2 = block_sum(td2, red);
  const double bx2 = block_sum(tx2, red);
  if (threadIdx.x == 0) {
    part[2 * (int64_t)blockIdx.x] = bd2;
    part[2 * (int64_t)blockIdx.x + 1] = bx2;
  }
}

// The block partials added in block order; out (2 doubles) and/or rel_out
// (sqrt(d2 / x2), e.g. a trace slot) may be NULL.
__global__ void residual_final_kernel(const double* __restrict__ part, int64_t nblocks,
                                      double* out, double* rel_out) {
  __shared__ double red[32];
  double d2 = 0.0, x2 = 0.0;
  for (int64_t b = threadIdx.x; b < nblocks; b += blockDim.x) {
    d2 += part[2 * b];
    x2 += part[2 * b + 1];
  }
  d2 = block_sum(d2, red);
  x2 = block_sum(x2, red);
  if (threadIdx.x == 0) {
    if (out) {
      out[0] = d2;
      out[1] = x2;
    }
    if (rel_out) *rel_out = sqrt(d2 / x2);
  }
}

unsigned grid_cap(int64_t n, int threads) {
  int64_t b = ceil_div(n, threads);
  if (b > 8192) b = 8192;
  if (b < 1) b = 1;
  return (unsigned)b;
}

}  // namespace

template <typename T>
cudaError_t launch_lift(const T* F, const T* B, int64_t N, int M, int r, T* A, cudaStream_t s) {
  lift_kernel<T><<<grid_cap(N * r, 256), 256, 0, s>>>(F, B, N, M, r, A);
  note_launch(s);
  return cudaGetLastError();
}

template <typename T>
int residual_prepare(int d, const int64_t* dims, int model, const int* m, int r, Scratch& sc,
                     ResidualWork<T>* w) {
  if (d != 3 && d != 4) return NNC_ERR_INVALID_ARG;
  *w = ResidualWork<T>{};
  const int K = model == 0 ? m[d - 1] : r;
  int64_t R = 1;  // rows of U: N_1 ... N_{d-1}
  for (int k = 0; k < d - 1; ++k) R *= dims[k];
  NNC_TRY(sc.get(&w->U, (size_t)(R * K)));
  if (model == 0) {
    int64_t lead = 1, tail = 1;
    for (int k = 1; k < d; ++k) tail *= m[k];
    for (int k = 0; k < d - 2; ++k) {
      const int64_t n_out = lead * dims[k] * (tail);
      NNC_TRY(sc.get(&w->tmp[k & 1], (size_t)n_out));
      lead *= dims[k];
      tail /= m[k + 1];
    }
  } else {
    int64_t rows = dims[0];
    for (int k = 1; k < d - 2; ++k) {
      NNC_TRY(sc.get(&w->tmp[0], (size_t)(rows * dims[k] * r)));
      rows *= dims[k];
    }
  }
  w->nblocks = res_grid<T>(R, dims[d - 1], K).blocks;
  NNC_TRY(sc.get(&w->part, (size_t)(2 * w->nblocks)));
  return NNC_OK;
}

template <typename T>
int residual_run(const T* X, int d, const int64_t* dims, int model, const int* m, int r,
                 const T* const* factors, const T* G, const ResidualWork<T>& w, double* out2,
                 double* rel_out, cudaStream_t s) {
  const int K = model == 0 ? m[d - 1] : r;
  int64_t R = 1;
  for (int k = 0; k < d - 1; ++k) R *= dims[k];
  T* U = w.U;
  if (model == 0) {
    // Mode products of the core with F^(1) .. F^(d-1), the last one into U:
    // cur[t_<k, i_k, c_>k] = sum_a F^(k)[i_k, a] prev[t_<k, a, c_>k].
    int64_t lead = 1;  // N_1 ... N_{k-1}
    int64_t tail = 1;  // m_{k+1} ... m_d
    for (int k = 1; k < d; ++k) tail *= m[k];
    const T* src = G;
    for (int k = 0; k < d - 1; ++k) {
      T* dst = k < d - 2 ? w.tmp[k & 1] : U;
      const int64_t cols = ceil_div(lead * tail, kMpThreads);
      const int64_t qt = ceil_div(dims[k], kMpQ);
      if (m[k] > 64 || cols * qt > 0x7fffffffLL) return NNC_ERR_UNSUPPORTED;
      mode_product_any_kernel<T><<<(unsigned)(cols * qt), kMpThreads, 0, s>>>(
          src, lead, m[k], tail, (unsigned)cols, factors[k], (int)dims[k], dst);
      note_launch(s);
      src = dst;
      lead *= dims[k];
      tail /= m[k + 1];
    }
  } else {
    // U_k = U_{k-1} (.) A^(k) row by row: (rows of U_{k-1}) x N_k rows.
    int64_t rows = dims[0];
    const T* src = factors[0];
    for (int k = 1; k < d - 1; ++k) {
      T* dst = k < d - 2 ? w.tmp[0] : U;
      cp_rows_kernel<T><<<grid_cap(rows * dims[k] * r, 256), 256, 0, s>>>(src, factors[k], rows,
                                                                           dims[k], r, dst);
      note_launch(s);
      src = dst;
      rows *= dims[k];
    }
  }
  NNC_CUDA_TRY(cudaGetLastError());
  const T* Fd = factors[d - 1];  // F^(d) (Tucker) or A^(d) (CP): N_d x K
  const int64_t Nd = dims[d - 1];
  if (K > 64) return NNC_ERR_UNSUPPORTED;
  const ResGrid g = res_grid<T>(R, Nd, K);
  if (g.blocks > 0x7fffffffLL) return NNC_ERR_UNSUPPORTED;
  auto stream = [&](auto km) {
    constexpr int KM = decltype(km)::value;
    residual_stream_kernel<T, KM, res_kt<T>(KM)><<<(unsigned)g.blocks, kResThreads, 0, s>>>(
        X, R, Nd, U, K, Fd, g.tx, g.ktiles, g.rows, w.part);
  };
  if (K <= 16) stream(std::integral_constant<int, 16>{});
  else if (K <= 32) stream(std::integral_constant<int, 32>{});
  else stream(std::integral_constant<int, 64>{});
  note_launch(s);
  residual_final_kernel<<<1, 1024, 0, s>>>(w.part, w.nblocks, out2, rel_out);
  note_launch(s);
  NNC_CUDA_TRY(cudaGetLastError());
  return NNC_OK;
}

template <typename T>
int residual_device(const T* X, int d, const int64_t* dims, int model, const int* m, int r,
                    const T* const* factors, const T* G, double* out2, Scratch& sc,
                    cudaStream_t s) {
  ResidualWork<T> w;
  NNC_TRY(residual_prepare<T>(d, dims, model, m, r, sc, &w));
  return residual_run<T>(X, d, dims, model, m, r, factors, G, w, out2, nullptr, s);
}

template cudaError_t launch_lift<float>(const float*, const float*, int64_t, int, int, float*,
                                        cudaStream_t);
template cudaError_t launch_lift<double>(const double*, const double*, int64_t, int, int, double*,
                                         cudaStream_t);
template int residual_prepare<float>(int, const int64_t*, int, const int*, int, Scratch&,
                                     ResidualWork<float>*);
template int residual_prepare<double>(int, const int64_t*, int, const int*, int, Scratch&,
                                      ResidualWork<double>*);
template int residual_run<float>(const float*, int, const int64_t*, int, const int*, int,
                                 const float* const*, const float*, const ResidualWork<float>&,
                                 double*, double*, cudaStream_t);
template int residual_run<double>(const double*, int, const int64_t*, int, const int*, int,
                                  const double* const*, const double*,
                                  const ResidualWork<double>&, double*, double*, cudaStream_t);
template int residual_device<float>(const float*, int, const int64_t*, int, const int*, int,
                                    const float* const*, const float*, double*, Scratch&,
                                    cudaStream_t);
template int residual_device<double>(const double*, int, const int64_t*, int, const int*, int,
                                     const double* const*, const double*, double*, Scratch&,
                                     cudaStream_t);

}  // namespace nnc
