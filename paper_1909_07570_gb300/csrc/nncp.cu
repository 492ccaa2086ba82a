// nnCPD of Tucker cores (Alg. 1, step 2): multiplicative updates of
// B^(1), ..., B^(d) for 1/2 ||G - I x_n B^(n)||_F^2, one thread block per fit.
//
// A block keeps every B^(k) (m_k x r) and its Gram B^(k)T B^(k) (r x r) in
// shared memory and reads the core G through L1. A sweep, for n = 1..d:
//   V   = Hadamard product over k != n of Gram_k
//   Num = unfold_n(G) KR_{k!=n} B^(k)   (MTTKRP, factored loop over the modes)
//   B^(n) <- max(B^(n) * Num / max(B^(n) V, eps), 0);  Gram_n <- B^(n)T B^(n)
// The same kernel serves one fit (nncp_core_fit) and many uneven fits in one
// launch (nncp_core_fit_batched); no block waits on another.
#include <algorithm>
#include <string>

#include "kernels.cuh"
#include "nncp.cuh"
#include "small_batched.cuh"

namespace nnc {
namespace {

constexpr int kThreads = 256;

template <typename T, int D>
__device__ T mttkrp_entry(const T* __restrict__ G, const int* m, const int64_t* st,
                          T* const* Bs, int r, int n, int i, int q) {
  int o[D - 1];
  {
    int t = 0;
#pragma unroll
    for (int k = 0; k < D; ++k)
      if (k != n) o[t++] = k;
  }
  const T* g0 = G + (int64_t)i * st[n];
  T s = T(0);
  if constexpr (D == 3) {
    for (int j0 = 0; j0 < m[o[0]]; ++j0) {
      const T* g1 = g0 + j0 * st[o[0]];
      T inner = T(0);
      for (int j1 = 0; j1 < m[o[1]]; ++j1)
        inner = fma(g1[j1 * st[o[1]]], Bs[o[1]][j1 * r + q], inner);
      s = fma(Bs[o[0]][j0 * r + q], inner, s);
    }
  } else {
    for (int j0 = 0; j0 < m[o[0]]; ++j0) {
      const T* g1 = g0 + j0 * st[o[0]];
      T mid = T(0);
      for (int j1 = 0; j1 < m[o[1]]; ++j1) {
        const T* g2 = g1 + j1 * st[o[1]];
        T inner = T(0);
        for (int j2 = 0; j2 < m[o[2]]; ++j2)
          inner = fma(g2[j2 * st[o[2]]], Bs[o[2]][j2 * r + q], inner);
        mid = fma(Bs[o[1]][j1 * r + q], inner, mid);
      }
      s = fma(Bs[o[0]][j0 * r + q], mid, s);
    }
  }
  return s;
}

template <typename T, int D>
__device__ void fit_one(const nncp_job& job, int iters, T eps, unsigned char* smem, double* fpart,
                        double* rel_err_out, int* status_out) {
  const int r = job.r;
  int m[D];
  int64_t st[D];
#pragma unroll
  for (int k = 0; k < D; ++k) m[k] = job.m[k];
  st[D - 1] = 1;
#pragma unroll
  for (int k = D - 2; k >= 0; --k) st[k] = st[k + 1] * m[k + 1];
  int mmax = 0;
#pragma unroll
  for (int k = 0; k < D; ++k) mmax = m[k] > mmax ? m[k] : mmax;

  // Shared memory: B^(k) | Gram_k | V | Num
  T* p = reinterpret_cast<T*>(smem);
  T* Bs[D];
  T* Gram[D];
#pragma unroll
  for (int k = 0; k < D; ++k) {
    Bs[k] = p;
    p += m[k] * r;
  }
#pragma unroll
  for (int k = 0; k < D; ++k) {
    Gram[k] = p;
    p += r * r;
  }
  T* V = p;
  p += r * r;
  T* Num = p;

  const T* G = static_cast<const T*>(job.G);
  const int tid = threadIdx.x;

#pragma unroll
  for (int k = 0; k < D; ++k) {
    const T* src = static_cast<const T*>(job.B[k]);
    for (int e = tid; e < m[k] * r; e += blockDim.x) Bs[k][e] = src[e];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < D; ++k)
    for (int e = tid; e < r * r; e += blockDim.x) {
      const int a = e / r, b = e % r;
      T s = T(0);
      for (int i = 0; i < m[k]; ++i) s = fma(Bs[k][i * r + a], Bs[k][i * r + b], s);
      Gram[k][e] = s;
    }
  __syncthreads();

  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int n = 0; n < D; ++n) {
      for (int e = tid; e < r * r; e += blockDim.x) {
        T v = T(1);
#pragma unroll
        for (int k = 0; k < D; ++k)
          if (k != n) v *= Gram[k][e];
        V[e] = v;
      }
      for (int e = tid; e < m[n] * r; e += blockDim.x)
        Num[e] = mttkrp_entry<T, D>(G, m, st, Bs, r, n, e / r, e % r);
      __syncthreads();
      // New values go to Num first: every row of the old B^(n) is still read.
      for (int e = tid; e < m[n] * r; e += blockDim.x) {
        const int i = e / r, q = e % r;
        T den = T(0);
        for (int pp = 0; pp < r; ++pp) den = fma(Bs[n][i * r + pp], V[pp * r + q], den);
        const T v = Bs[n][e] * Num[e] / (den > eps ? den : eps);
        Num[e] = v > T(0) ? v : T(0);
      }
      __syncthreads();
      for (int e = tid; e < m[n] * r; e += blockDim.x) Bs[n][e] = Num[e];
      __syncthreads();
      for (int e = tid; e < r * r; e += blockDim.x) {
        const int a = e / r, b = e % r;
        T s = T(0);
        for (int i = 0; i < m[n]; ++i) s = fma(Bs[n][i * r + a], Bs[n][i * r + b], s);
        Gram[n][e] = s;
      }
      __syncthreads();
    }
  }

  bool finite = true;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    T* dst = static_cast<T*>(job.B[k]);
    for (int e = tid; e < m[k] * r; e += blockDim.x) {
      dst[e] = Bs[k][e];
      finite = finite && isfinite(Bs[k][e]);
    }
  }

  if (rel_err_out != nullptr || status_out != nullptr) {
    int64_t total = 1;
#pragma unroll
    for (int k = 0; k < D; ++k) total *= m[k];
    // FP64 sums in an order that does not depend on the block size.
    const double2 dg = fixed_sums2(total, [&](int64_t e) {
      int idx[D];
      int64_t rem = e;
#pragma unroll
      for (int k = D - 1; k >= 0; --k) {
        idx[k] = (int)(rem % m[k]);
        rem /= m[k];
      }
      T hat = T(0);
      for (int q = 0; q < r; ++q) {
        T prod = T(1);
#pragma unroll
        for (int k = 0; k < D; ++k) prod *= Bs[k][idx[k] * r + q];
        hat += prod;
      }
      const double g = (double)G[e];
      const double dd = g - (double)hat;
      return make_double2(dd * dd, g * g);
    }, fpart);
    if (tid == 0 && rel_err_out != nullptr)
      *rel_err_out = dg.y > 0.0 ? sqrt(dg.x / dg.y) : sqrt(dg.x);
    // The fit's status: a NaN or an overflow anywhere (in the core, or reached
    // during the sweeps) shows in the fitted factors or in the residual sums.
    if (status_out != nullptr) {
      const int ok = __syncthreads_and(finite ? 1 : 0);
      if (tid == 0)
        *status_out = (ok && isfinite(dg.x) && isfinite(dg.y)) ? NNC_OK : NNC_ERR_NONFINITE;
    }
  }
}

// ---- 3-way cores that fit in shared memory ---------------------------------------
//
// The same sweep in six intervals between block barriers, with the core itself in shared
// memory and two products of it per sweep instead of three:
//   1  T[i, j, :] = sum_k G[i, j, k] B3[k, :]        Gram3
//   2  B1 <- MU (Num1[i, q] = sum_j T[i, j, q] B2[j, q])
//   3  Num2[j, q] = sum_i T[i, j, q] B1[i, q]        Gram1
//   4  B2 <- MU
//   5  T'[i, k, :] = sum_j G[i, j, k] B2[j, :]       Gram2
//   6  B3 <- MU (Num3[k, q] = sum_i T'[i, k, q] B1[i, q])
// Every sum has fit_one's terms in fit_one's order, and so its bits (T' = G x_1 B1, ready an
// interval earlier, would sum mode 3 over i inside j; a few ill-conditioned fits among
// thousands amplify that rounding to 1e-3 of an entry).
// Rows of B and T are padded with zeros to RP entries and read in 16-byte pieces, a thread
// forming a whole row of T; rows of G have an odd pitch. A MU step writes the copy of
// the factor it does not read, and takes V as the product of two Grams in place. No sum
// depends on the block size. (fit_one reads G through L1 once per numerator entry and has a
// barrier after every step, where its warps spent 11 of the 19 cycles between two
// instructions; figures at nncp_kernel.)
constexpr size_t kFit3Bytes = kSmemBudget;
__host__ __device__ inline int fit3_rp(int r) { return r <= 4 ? 4 : (r <= 8 ? 8 : 16); }
__host__ __device__ inline size_t fit3_elems(const nncp_job& j) {
  const int rp = fit3_rp(j.r), m1 = j.m[0], m2 = j.m[1], m3 = j.m[2];
  const int msum = m1 + m2 + m3;
  const size_t t = (size_t)m1 * (m2 > m3 ? m2 : m3) * rp;
  return (size_t)2 * msum * rp + 3 * rp * rp + (size_t)m2 * rp + t + (size_t)m1 * m2 * (m3 | 1);
}
__host__ __device__ inline bool fit3_takes(const nncp_job& j, size_t elem) {
  return j.d == 3 && j.r <= 16 && fit3_elems(j) * elem <= kFit3Bytes;
}

template <typename T, int RP>
__device__ __forceinline__ void fit3(const nncp_job& job, int iters, T eps, unsigned char* smem,
                                     double* fpart, double* rel_err_out, int* status_out) {
  constexpr int VW = 16 / (int)sizeof(T);
  const int m1 = job.m[0], m2 = job.m[1], m3 = job.m[2], r = job.r, gp = m3 | 1;
  const int tid = threadIdx.x, nt = blockDim.x;
  T* B[3];
  T* Bn[3];
  B[0] = reinterpret_cast<T*>(smem);
  B[1] = B[0] + m1 * RP;
  B[2] = B[1] + m2 * RP;
  Bn[0] = B[2] + m3 * RP;
  Bn[1] = Bn[0] + m1 * RP;
  Bn[2] = Bn[1] + m2 * RP;
  T* Gr[3];
  Gr[0] = Bn[2] + m3 * RP;
  Gr[1] = Gr[0] + RP * RP;
  Gr[2] = Gr[1] + RP * RP;
  T* Num = Gr[2] + RP * RP;
  T* Tb = Num + m2 * RP;
  T* G = Tb + (size_t)m1 * max(m2, m3) * RP;
  const T* Gg = static_cast<const T*>(job.G);
  for (int e = tid; e < m1 * m2 * m3; e += nt) G[(e / m3) * gp + e % m3] = Gg[e];
#pragma unroll
  for (int n = 0; n < 3; ++n) {
    const T* src = static_cast<const T*>(job.B[n]);
    for (int e = tid; e < job.m[n] * RP; e += nt) {
      const int i = e / RP, q = e % RP;
      B[n][e] = q < r ? src[i * r + q] : T(0);
      Bn[n][e] = T(0);
    }
  }
  __syncthreads();
  auto gram = [&](const T* F, int m, T* S) {
    for (int e = tid; e < r * r; e += nt) {
      const int a = e / r, b = e - a * r;
      T s = T(0);
#pragma unroll 4
      for (int i = 0; i < m; ++i) s = fma(F[i * RP + a], F[i * RP + b], s);
      S[a * RP + b] = s;
    }
  };
  // acc[q] += v f[q] for a row f of RP entries.
  auto axpy = [&](T v, const T* f, T (&acc)[RP]) {
#pragma unroll
    for (int q = 0; q < RP; q += VW) {
      if constexpr (sizeof(T) == 4) {
        const float4 w = *reinterpret_cast<const float4*>(f + q);
        acc[q] = fma(v, w.x, acc[q]);
        acc[q + 1] = fma(v, w.y, acc[q + 1]);
        acc[q + 2] = fma(v, w.z, acc[q + 2]);
        acc[q + 3] = fma(v, w.w, acc[q + 3]);
      } else {
        const double2 w = *reinterpret_cast<const double2*>(f + q);
        acc[q] = fma(v, w.x, acc[q]);
        acc[q + 1] = fma(v, w.y, acc[q + 1]);
      }
    }
  };
  // Rows of T: out[row, :] = sum_{t < len} x[t xs] F[t, :], x = G + xo(row).
  auto products = [&](int rows, int len, int xs, auto xo, const T* F) {
    for (int row = tid; row < rows; row += nt) {
      T acc[RP];
#pragma unroll
      for (int q = 0; q < RP; ++q) acc[q] = T(0);
      const T* x = G + xo(row);
#pragma unroll 4
      for (int t = 0; t < len; ++t) axpy(x[t * xs], F + t * RP, acc);
#pragma unroll
      for (int q = 0; q < RP; q += VW) {
        if constexpr (sizeof(T) == 4)
          *reinterpret_cast<float4*>(Tb + row * RP + q) =
              make_float4(acc[q], acc[q + 1], acc[q + 2], acc[q + 3]);
        else
          *reinterpret_cast<double2*>(Tb + row * RP + q) = make_double2(acc[q], acc[q + 1]);
      }
    }
  };
  // sum_{t < len} T[to + t ts] F[t, q]
  auto numer = [&](const T* t0, int ts, const T* F, int len) {
    T s = T(0);
#pragma unroll 4
    for (int t = 0; t < len; ++t) s = fma(t0[t * ts], F[t * RP], s);
    return s;
  };
  auto mu = [&](int n, int i, int q, T num, const T* Ga, const T* Gb) {
    const T* row = B[n] + i * RP;
    T den = T(0);
#pragma unroll 4
    for (int p = 0; p < r; ++p) den = fma(row[p], Ga[p * RP + q] * Gb[p * RP + q], den);
    const T v = row[q] * num / (den > eps ? den : eps);
    Bn[n][i * RP + q] = v > T(0) ? v : T(0);
  };
  auto swap = [&](int n) {
    T* t = B[n];
    B[n] = Bn[n];
    Bn[n] = t;
  };
  gram(B[1], m2, Gr[1]);
  for (int it = 0; it < iters; ++it) {
    products(m1 * m2, m3, 1, [&](int row) { return row * gp; }, B[2]);
    gram(B[2], m3, Gr[2]);
    __syncthreads();
    for (int e = tid; e < m1 * r; e += nt) {
      const int i = e / r, q = e - i * r;
      mu(0, i, q, numer(Tb + i * m2 * RP + q, RP, B[1] + q, m2), Gr[1], Gr[2]);
    }
    swap(0);
    __syncthreads();
    gram(B[0], m1, Gr[0]);
    for (int e = tid; e < m2 * r; e += nt) {
      const int j = e / r, q = e - j * r;
      Num[j * RP + q] = numer(Tb + j * RP + q, m2 * RP, B[0] + q, m1);
    }
    __syncthreads();
    for (int e = tid; e < m2 * r; e += nt) {
      const int j = e / r, q = e - j * r;
      mu(1, j, q, Num[j * RP + q], Gr[0], Gr[2]);
    }
    swap(1);
    __syncthreads();
    gram(B[1], m2, Gr[1]);
    products(m1 * m3, m2, gp, [&](int row) { return (row / m3) * m2 * gp + row % m3; }, B[1]);
    __syncthreads();
    for (int e = tid; e < m3 * r; e += nt) {
      const int k = e / r, q = e - k * r;
      mu(2, k, q, numer(Tb + k * RP + q, m3 * RP, B[0] + q, m1), Gr[0], Gr[1]);
    }
    swap(2);
    __syncthreads();
  }
  __syncthreads();
  bool finite = true;
#pragma unroll
  for (int n = 0; n < 3; ++n) {
    T* dst = static_cast<T*>(job.B[n]);
    for (int e = tid; e < job.m[n] * r; e += nt) {
      const T v = B[n][(e / r) * RP + e % r];
      dst[e] = v;
      finite = finite && isfinite(v);
    }
  }
  if (rel_err_out != nullptr || status_out != nullptr) {
    // FP64 sums in an order that does not depend on the block size.
    const double2 dg = fixed_sums2((int64_t)m1 * m2 * m3, [&](int64_t e) {
      const int k = (int)(e % m3), ij = (int)(e / m3), j = ij % m2, i = ij / m2;
      T hat = T(0);
      for (int q = 0; q < r; ++q)
        hat += B[0][i * RP + q] * B[1][j * RP + q] * B[2][k * RP + q];
      const double g = (double)G[ij * gp + k], dd = g - (double)hat;
      return make_double2(dd * dd, g * g);
    }, fpart);
    if (tid == 0 && rel_err_out != nullptr)
      *rel_err_out = dg.y > 0.0 ? sqrt(dg.x / dg.y) : sqrt(dg.x);
    if (status_out != nullptr) {
      const int ok = __syncthreads_and(finite ? 1 : 0);
      if (tid == 0)
        *status_out = (ok && isfinite(dg.x) && isfinite(dg.y)) ? NNC_OK : NNC_ERR_NONFINITE;
    }
  }
}

// One block per job, each in its own form (a job gives the same bits alone and in any
// batch); RP: the largest row tile of the jobs that fit3 takes, 0 when there are none.
// 3584 fits of 4^3 to 16^3 cores at ranks 2..8, FP32, 200 sweeps: 12.4 ms with fit_one
// alone, 3.6 ms; one 5^3 core at r = 3, FP64, 200 sweeps: 2.0 -> 1.2 ms.
template <typename T, int RP>
__global__ void __launch_bounds__(kThreads)
nncp_kernel(const nncp_job* __restrict__ jobs, int iters, T eps, double* rel_errs,
            int* statuses) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double fpart[2 * kFixedLanes];  // of the fit's FP64 sums
  const nncp_job job = jobs[blockIdx.x];
  int* st = statuses ? statuses + blockIdx.x : nullptr;
  // A job the host skipped (its shared memory was not sized for it).
  if (!nncp_job_valid(job)) {
    if (st != nullptr && threadIdx.x == 0) *st = NNC_ERR_INVALID_ARG;
    return;
  }
  double* out = rel_errs ? rel_errs + blockIdx.x : nullptr;
  if constexpr (RP > 0) {
    if (fit3_takes(job, sizeof(T))) {
      if constexpr (RP > 8) {
        if (job.r > 8) return fit3<T, 16>(job, iters, eps, smem_raw, fpart, out, st);
      }
      if constexpr (RP > 4) {
        if (job.r > 4) return fit3<T, 8>(job, iters, eps, smem_raw, fpart, out, st);
      }
      return fit3<T, 4>(job, iters, eps, smem_raw, fpart, out, st);
    }
  }
  if (job.d == 3)
    fit_one<T, 3>(job, iters, eps, smem_raw, fpart, out, st);
  else
    fit_one<T, 4>(job, iters, eps, smem_raw, fpart, out, st);
}

}  // namespace

size_t nncp_smem_bytes(const nncp_job& j, size_t elem) {
  int mmax = 0, msum = 0;
  for (int k = 0; k < j.d; ++k) {
    msum += j.m[k];
    mmax = j.m[k] > mmax ? j.m[k] : mmax;
  }
  const size_t n = (size_t)msum * j.r + (size_t)(j.d + 1) * j.r * j.r + (size_t)mmax * j.r;
  return n * elem;
}

template <typename T>
int nncp_route(int n_jobs, const nncp_job* jobs, bool skip_invalid, NncpRoute* rt) {
  *rt = NncpRoute{};
  int64_t largest = 0;
  bool l2_ok = true;  // every valid job within the two-pass kernel's limits
  size_t smem1 = 0;  // shared memory of the one-pass kernel, each job in its form
  int rp = 0;
  size_t l2_elems = 0;
  for (int i = 0; i < n_jobs; ++i) {
    const nncp_job& j = jobs[i];
    if (!nncp_job_valid(j)) {
      if (!skip_invalid) {
        set_error_detail_text("batched nnCP: job " + std::to_string(i) +
                              " has a bad descriptor (d, m, r or a null pointer)");
        return NNC_ERR_INVALID_ARG;
      }
      ++rt->invalid;
      continue;
    }
    const size_t b = nncp_smem_bytes(j, sizeof(T));
    rt->smem = b > rt->smem ? b : rt->smem;
    if (fit3_takes(j, sizeof(T))) {
      smem1 = std::max(smem1, fit3_elems(j) * sizeof(T));
      rp = std::max(rp, fit3_rp(j.r));
    } else {
      smem1 = std::max(smem1, b);
    }
    int64_t e = 1;
    for (int k = 0; k < j.d; ++k) e *= j.m[k];
    largest = e > largest ? e : largest;
    if (j.d != 3 || j.r > 16) {
      l2_ok = false;
    } else {
      const size_t le = cpx_l2_elems(j);
      l2_elems = le > l2_elems ? le : l2_elems;
    }
  }
  l2_ok = l2_ok && l2_elems * sizeof(T) <= kSmemBudget;
  // The cluster form: every valid job 3-way with slabs within a CTA, and a
  // cluster per valid job on the GPU at once.
  bool cl_ok = true;
  int valid = 0, rmax = 1;
  for (int i = 0; i < n_jobs; ++i)
    if (nncp_job_valid(jobs[i])) rmax = std::max(rmax, (int)jobs[i].r);
  for (int i = 0; i < n_jobs; ++i) {
    const nncp_job& j = jobs[i];
    if (!nncp_job_valid(j)) continue;
    ++valid;
    if (j.d != 3 || cpx_cluster_elems(j, rmax, false) * sizeof(T) > kClusterSmem) cl_ok = false;
  }
  cl_ok = cl_ok && valid >= 1 && (int64_t)valid * cpx_cluster_ctas() <= device_sm_count();
  constexpr int64_t kTwoPassMinEntries = 16384;
  if (rt->smem > kSmemBudget) {
    if (!l2_ok) {
      set_error_detail_text("batched nnCP: a job's state exceeds one block of shared memory");
      return NNC_ERR_UNSUPPORTED;
    }
    rt->two_pass = true;
  } else {
    rt->two_pass = largest >= kTwoPassMinEntries && l2_ok;
  }
  rt->cluster = rt->two_pass && cl_ok;
  if (!rt->two_pass) {
    rt->rp = rp;
    rt->smem = smem1;
  }
  return NNC_OK;
}

template <typename T>
cudaError_t launch_nncp(const nncp_job* jobs_dev, int n_jobs, size_t smem, int rp, int iters,
                        double eps, double* rel_errs, int* statuses, cudaStream_t s,
                        int threads) {
  if (threads < 32 || threads > kThreads || threads % 32 != 0) return cudaErrorInvalidValue;
  const auto kern = rp == 0   ? nncp_kernel<T, 0>
                    : rp == 4 ? nncp_kernel<T, 4>
                    : rp == 8 ? nncp_kernel<T, 8>
                              : nncp_kernel<T, 16>;
  const cudaError_t e = raise_smem_limit((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<n_jobs, threads, smem, s>>>(jobs_dev, iters, (T)eps, rel_errs, statuses);
  note_launch(s);
  return cudaGetLastError();
}

TuneKey nncp_tune_key(const nncp_job* jobs, int n_jobs, size_t elem, int rp) {
  long long work = 1;
  for (int i = 0; i < n_jobs; ++i) {
    if (!nncp_job_valid(jobs[i])) continue;
    long long w = jobs[i].r;  // one sweep: every entry of the core once per mode and q
    for (int k = 0; k < jobs[i].d; ++k) w *= jobs[i].m[k];
    work = w > work ? w : work;
  }
  return TuneKey{rp ? kTuneNncp3 : kTuneNncp, (int)elem, size_class(work), size_class(n_jobs)};
}

template cudaError_t launch_nncp<float>(const nncp_job*, int, size_t, int, int, double, double*,
                                        int*, cudaStream_t, int);
template cudaError_t launch_nncp<double>(const nncp_job*, int, size_t, int, int, double, double*,
                                         int*, cudaStream_t, int);
template int nncp_route<float>(int, const nncp_job*, bool, NncpRoute*);
template int nncp_route<double>(int, const nncp_job*, bool, NncpRoute*);

}  // namespace nnc
