// nnCPD of a 3-way core by one thread-block cluster per fit (Alg. 1, step 2):
// the Gauss-Seidel sweep
//   T   = G x_3 A3^T              MT1[i, q] = sum_j T[i, j, q] A2[j, q]    A1 <- MU
//   T'  = G x_1 A1^T              MT2[j, q] = sum_k T'[j, k, q] A3[k, q]   A2 <- MU
//                                 MT3[k, q] = sum_j T'[j, k, q] A2[j, q]   A3 <- MU
// with A_n <- max(A_n * MT_n / max(A_n V_n, eps), 0), V_n the Hadamard product
// of the other factors' Grams, spread over kCl CTAs.
//
// CTA c of the cluster owns the rows of every factor in its ranges of i, j and k and keeps, in
// shared memory, the slab of the core with its i (for T), the slab with its j (for
// T'; read from L2 in place where it does not fit beside the rest), and full copies of every
// factor and Gram. T and T' on its slabs give MT1 and MT2 on its
// own rows and its share of MT3; new rows go to the other CTAs through distributed
// shared memory, into the copy of the factor that no CTA reads any more (two
// copies, swapped at the barrier), the shares of MT3 to the CTA that owns the row k, which
// adds them in CTA order: every CTA holds the same bits and results do not depend
// on timing. Three cluster barriers and three block barriers a sweep:
//   T, Gram3 | MT1, MU on A1, rows sent   || T', Gram1 | MT2, MU on A2, rows sent |
//   shares of MT3 sent || Gram2 | MT3, MU on A3, rows sent ||
// Every contraction is short and latency bounds it: eight lanes share an output of a
// MU step, one term in eight of the numerator and of the denominator each, and lane u
// sends the new entry to CTA u. In FP64 the FP64 units bound the products (a warp-wide FMA
// takes 16 cycles): no padded entry is formed and each Gram once, by symmetry.
// A sweep, FP32, against the form that took mode 2 from T (its MTTKRP summed over every
// CTA's slab and its MU step repeated in every CTA; two cluster barriers, twelve block barriers):
//   32^3, r = 16    10.7 -> 7.7 us          40^3, r = 10     19.4 -> 9.1 us
//   16 x 64 x 16    11.8 -> 6.8 us          64 x 4 x 64      10.5 -> 8.3 us (r = 13)
// and in FP64 32^3 at r = 16 50.8 -> 50.8, at r = 5 22.3 -> 20.3 us.
#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "kernels.cuh"
#include "nncp.cuh"

namespace nnc {
namespace cg = cooperative_groups;
namespace {

constexpr int kCl = 8;  // CTAs per fit (the portable cluster size)
constexpr int kClThreads = 512;

__host__ __device__ constexpr size_t al4(size_t x) { return (x + 3) & ~static_cast<size_t>(3); }

// Element offsets of one CTA's shared memory; factors, Grams and products have rows of rp.
struct ClLayout {
  int ni, nj, nk;  // rows of each factor a CTA owns
  int xpitch;      // row pitch of the i-slab
  size_t xi, xj, a[2][3], g[3], tb, in, total;
  __host__ __device__ ClLayout(const int* N, int rp, bool slab_j) {
    ni = (N[0] + kCl - 1) / kCl;
    nj = (N[1] + kCl - 1) / kCl;
    nk = (N[2] + kCl - 1) / kCl;
    size_t p = 0;
    xpitch = N[2] | 1;  // odd: the rows a warp reads fall on distinct banks
    xi = p;  p += al4((size_t)ni * N[1] * xpitch);  // [ii][j][k], rows xpitch apart
    xj = p;  p += slab_j ? al4((size_t)N[0] * nj * N[2]) : 0;  // [i][jj][k]
    for (int b = 0; b < 2; ++b)
      for (int n = 0; n < 3; ++n) { a[b][n] = p;  p += (size_t)N[n] * rp; }
    for (int n = 0; n < 3; ++n) { g[n] = p;  p += (size_t)rp * rp; }
    const size_t t3 = (size_t)ni * N[1] * rp, t1 = (size_t)nj * N[2] * rp;
    tb = p;  p += t3 > t1 ? t3 : t1;                // T [ii][j][q], then T' [jj][k][q]
    in = p;  p += (size_t)kCl * nk * rp;            // shares of MT3 for this CTA's k
    total = p;
  }
};

// P[row, q] = sum_{t < len} x[t xs] F[t, q] for row < rows, q < r, x = X + xo(row), F and P
// with rows of RP. FP32: a thread per 16-byte piece of a row; FP64: a thread per entry
// (the FP64 units bound it, so no entry of the padding is formed).
template <typename T, int RP, typename XO>
__device__ __forceinline__ void row_products(int rows, int len, int r, const T* X, XO xo, int xs,
                                             const T* F, T* P) {
  constexpr int VW = sizeof(T) == 4 ? 4 : 1;
  const int np = VW == 4 ? RP / 4 : r;
  for (int e = threadIdx.x; e < rows * np; e += kClThreads) {
    const int row = e / np, q = (e - row * np) * VW;
    const T* x = X + xo(row);
    if constexpr (VW == 4) {
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
      for (int t = 0; t < len; ++t) {
        const float v = x[t * xs];
        const float4 w = *reinterpret_cast<const float4*>(F + t * RP + q);
        s.x = fmaf(v, w.x, s.x);
        s.y = fmaf(v, w.y, s.y);
        s.z = fmaf(v, w.z, s.z);
        s.w = fmaf(v, w.w, s.w);
      }
      *reinterpret_cast<float4*>(P + row * RP + q) = s;
    } else {
      T s = T(0);
#pragma unroll 8
      for (int t = 0; t < len; ++t) s = fma(x[t * xs], F[t * RP + q], s);
      P[row * RP + q] = s;
    }
  }
}

// The entry (a, b), a <= b, of a Gram that a thread has a part in: four lanes an entry
// where the block has the threads (r <= 12: 78 entries), two for up to 136 entries.
template <int RP>
struct GramLane {
  int a = 0, b, u, nl;
  bool on;
  __device__ explicit GramLane(int r) {
    const int ne = r * (r + 1) / 2;
    nl = RP <= 12 || r <= 12 ? 4 : 2;  // by r alone: a batch's tile changes no bits
    const int e = (int)threadIdx.x / nl;
    u = (int)threadIdx.x % nl;
    on = e < ne;
    int k = e;
    while (a < r && k >= r - a) k -= r - a++;
    b = a + k;
  }
};

// S[a, b] = S[b, a] = sum_{i < n} A[i, a] A[i, b], the lanes' sums added.
template <typename T, int RP>
__device__ __forceinline__ void gram_lanes(const GramLane<RP>& g, const T* A, int n, T* S) {
  T s = T(0), s1 = T(0);  // two sums a lane: half the chain, and half its rounding
  if (g.on) {
    int i = g.u;
#pragma unroll 2
    for (; i + g.nl < n; i += 2 * g.nl) {
      s = fma(A[i * RP + g.a], A[i * RP + g.b], s);
      s1 = fma(A[(i + g.nl) * RP + g.a], A[(i + g.nl) * RP + g.b], s1);
    }
    if (i < n) s = fma(A[i * RP + g.a], A[i * RP + g.b], s);
    s += s1;
  }
  for (int o = g.nl / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (g.on && g.u == 0) S[g.a * RP + g.b] = S[g.b * RP + g.a] = s;
}

template <typename T, int RP>
__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(kClThreads)
    cpx_cluster_kernel(const nncp_job* __restrict__ jobs, int iters, T eps, bool slab_j,
                       double* rel_errs, int* statuses) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[2 * kFixedLanes];
  __shared__ double sums[2];
  cg::cluster_group cl = cg::this_cluster();
  const int c = (int)cl.block_rank();
  const int job = blockIdx.x / kCl;
  const nncp_job& jb = jobs[job];
  // A job the host skipped: every CTA of the cluster leaves before any
  // cluster barrier.
  if (!nncp_job_valid(jb) || jb.d != 3) {
    if (statuses != nullptr && c == 0 && threadIdx.x == 0) statuses[job] = NNC_ERR_INVALID_ARG;
    return;
  }
  const int N1 = jb.m[0], N2 = jb.m[1], N3 = jb.m[2], r = jb.r;
  const ClLayout L(jb.m, RP, slab_j);
  T* sm = reinterpret_cast<T*>(smem_raw);
  T* Xi = sm + L.xi;
  T* Xj = sm + L.xj;
  T* A[3] = {sm + L.a[0][0], sm + L.a[0][1], sm + L.a[0][2]};
  T* An[3] = {sm + L.a[1][0], sm + L.a[1][1], sm + L.a[1][2]};
  T* Gr[3] = {sm + L.g[0], sm + L.g[1], sm + L.g[2]};
  T* Tb = sm + L.tb;
  T* In = sm + L.in;  // [CTA][kk][q]
  const int i0 = min(c * L.ni, N1), ni = min(L.ni, N1 - i0);
  const int j0 = min(c * L.nj, N2), nj = min(L.nj, N2 - j0);
  const int k0 = min(c * L.nk, N3), nk = min(L.nk, N3 - k0);
  const T* X = static_cast<const T*>(jb.G);
  const int tid = threadIdx.x, nt = kClThreads;
  const GramLane<RP> gl(r);

  for (int e = tid; e < ni * N2 * N3; e += nt) {
    const int row = e / N3, k = e - row * N3;
    Xi[row * L.xpitch + k] = X[(int64_t)i0 * N2 * N3 + e];
  }
  if (slab_j)
    for (int e = tid; e < N1 * nj * N3; e += nt) {
      const int i = e / (nj * N3), jk = e - i * nj * N3;
      Xj[e] = X[((int64_t)i * N2 + j0) * N3 + jk];
    }
  for (int n = 0; n < 3; ++n) {
    const T* src = static_cast<const T*>(jb.B[n]);
    for (int e = tid; e < jb.m[n] * RP; e += nt) {
      const int i = e / RP, q = e % RP;
      A[n][e] = q < r ? src[i * r + q] : T(0);
      An[n][e] = T(0);
    }
  }
  __syncthreads();
  gram_lanes<T, RP>(gl, A[1], N2, Gr[1]);
  // No CTA sends before every CTA's copies are zeroed.
  cl.sync();

  // The MU step on rows r0 .. r0 + rows - 1 of factor n: num(i, q, u) is lane u's part of
  // the numerator of row r0 + i, Ga .* Gb = V_n. Eight lanes an entry; lane u sends
  // it to CTA u.
  const int u = tid & 7;
  auto mu_rows = [&](int n, int r0, int rows, const T* Ga, const T* Gb, auto num) {
    const T* f = A[n] + r0 * RP;
    for (int e0 = 0; e0 < rows * r; e0 += nt / 8) {
      const int e = e0 + tid / 8, i = e / r, q = e - i * r;
      const bool on = e < rows * r;
      T s = T(0), den = T(0);
      if (on) {
        s = num(i, q);
        for (int p = u; p < r; p += 8) den = fma(f[i * RP + p], Ga[p * RP + q] * Gb[p * RP + q], den);
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
      }
      if (on) {
        T v = f[i * RP + q] * s / (den > eps ? den : eps);
        v = v > T(0) ? v : T(0);
        T* const dst = An[n] + (r0 + i) * RP + q;
        if (u == c)
          *dst = v;
        else
          *cl.map_shared_rank(dst, u) = v;
      }
    }
  };
  auto swap = [&](int n) {
    T* t = A[n];
    A[n] = An[n];
    An[n] = t;
  };
  static_assert(kCl == 8, "lane u of an entry serves CTA u");

  for (int it = 0; it < iters; ++it) {
    // ---- T[ii, j, :] on this CTA's i; Gram3
    row_products<T, RP>(ni * N2, N3, r, Xi, [&](int row) { return row * L.xpitch; }, 1, A[2], Tb);
    gram_lanes<T, RP>(gl, A[2], N3, Gr[2]);
    __syncthreads();
    // ---- A1
    mu_rows(0, i0, ni, Gr[1], Gr[2], [&](int i, int q) {
      T s = T(0);
#pragma unroll 4
      for (int j = u; j < N2; j += 8) s = fma(Tb[(i * N2 + j) * RP + q], A[1][j * RP + q], s);
      return s;
    });
    cl.sync();
    swap(0);
    // ---- T'[jj, k, :] on this CTA's j; Gram1
    if (slab_j)
      row_products<T, RP>(nj * N3, N1, r, Xj, [&](int jk) { return jk; }, nj * N3, A[0], Tb);
    else
      row_products<T, RP>(nj * N3, N1, r, X + j0 * N3, [&](int jk) { return jk; }, N2 * N3, A[0],
                          Tb);
    gram_lanes<T, RP>(gl, A[0], N1, Gr[0]);
    __syncthreads();
    // ---- A2
    mu_rows(1, j0, nj, Gr[0], Gr[2], [&](int j, int q) {
      T s = T(0);
#pragma unroll 4
      for (int k = u; k < N3; k += 8) s = fma(Tb[(j * N3 + k) * RP + q], A[2][k * RP + q], s);
      return s;
    });
    __syncthreads();
    // ---- this CTA's share of MT3 to the owners of the rows k
    {
      const T* a2 = An[1] + j0 * RP;  // its new rows of A2
      for (int e = tid; e < N3 * r; e += nt) {
        const int k = e / r, q = e - k * r, o = k / L.nk;
        T s = T(0);
#pragma unroll 4
        for (int j = 0; j < nj; ++j) s = fma(Tb[(j * N3 + k) * RP + q], a2[j * RP + q], s);
        *cl.map_shared_rank(In + (c * L.nk + k - o * L.nk) * RP + q, o) = s;
      }
    }
    cl.sync();
    swap(1);
    // ---- Gram2; A3
    gram_lanes<T, RP>(gl, A[1], N2, Gr[1]);
    __syncthreads();
    mu_rows(2, k0, nk, Gr[0], Gr[1], [&](int k, int q) { return In[(u * L.nk + k) * RP + q]; });
    cl.sync();
    swap(2);
  }

  // ||G - I x_k A_k||^2 and ||G||^2 on this CTA's slab (FP64, in an order fixed
  // by the slab alone), then added over the cluster in CTA order.
  const double2 part = fixed_sums2((int64_t)ni * N2 * N3, [&](int64_t e) {
    const int k = (int)(e % N3), ij = (int)(e / N3), j = ij % N2, ii = ij / N2;
    T hat = T(0);
    for (int q = 0; q < r; ++q)
      hat = fma(A[0][(i0 + ii) * RP + q] * A[1][j * RP + q], A[2][k * RP + q], hat);
    const double g = (double)Xi[ij * L.xpitch + k], d = g - (double)hat;
    return make_double2(d * d, g * g);
  }, red);
  if (tid == 0) {
    sums[0] = part.x;
    sums[1] = part.y;
  }
  cl.sync();
  if (c == 0) {
    bool finite = true;
    for (int n = 0; n < 3; ++n) {
      T* dst = static_cast<T*>(jb.B[n]);
      for (int e = tid; e < jb.m[n] * r; e += nt) {
        const T v = A[n][(e / r) * RP + e % r];
        dst[e] = v;
        finite = finite && isfinite(v);
      }
    }
    const int ok = __syncthreads_and(finite ? 1 : 0);
    if (tid == 0) {
      double d2 = 0.0, x2 = 0.0;
      for (int s = 0; s < kCl; ++s) {
        const double* o = cl.map_shared_rank(sums, s);
        d2 += o[0];
        x2 += o[1];
      }
      if (rel_errs) rel_errs[job] = x2 > 0.0 ? sqrt(d2 / x2) : sqrt(d2);
      if (statuses)
        statuses[job] = (ok && isfinite(d2) && isfinite(x2)) ? NNC_OK : NNC_ERR_NONFINITE;
    }
  }
  // No CTA leaves while another may still read its shared memory.
  cl.sync();
}

}  // namespace

size_t cpx_cluster_elems(const nncp_job& j, int rmax, bool slab_j) {
  return ClLayout(j.m, (rmax + 3) / 4 * 4, slab_j).total;
}

int cpx_cluster_ctas() { return kCl; }

template <typename T>
int nncp_cluster_batched(int n_jobs, const nncp_job* jobs, int iters, double eps,
                         double* rel_errs, int* statuses, cudaStream_t s) {
  int rmax = 1;
  for (int i = 0; i < n_jobs; ++i) {
    if (!nncp_job_valid(jobs[i])) continue;  // the kernel reports it in its status
    rmax = jobs[i].r > rmax ? jobs[i].r : rmax;
    if (jobs[i].d != 3 || jobs[i].r > 16) {
      set_error_detail_text("cluster nnCP: a 4-way job or a rank above 16");
      return NNC_ERR_UNSUPPORTED;
    }
  }
  auto smem_of = [&](bool slab_j) {
    size_t elems = 0;
    for (int i = 0; i < n_jobs; ++i)
      if (nncp_job_valid(jobs[i])) elems = std::max(elems, cpx_cluster_elems(jobs[i], rmax, slab_j));
    return elems * sizeof(T);
  };
  const bool slab_j = smem_of(true) <= kClusterSmem;
  const size_t smem = smem_of(slab_j);
  if (smem > kClusterSmem) {
    set_error_detail_text("cluster nnCP: a job's slabs exceed one block of shared memory");
    return NNC_ERR_UNSUPPORTED;
  }
  Scratch sc(s);
  nncp_job* dev = nullptr;
  NNC_TRY(sc.get(&dev, (size_t)n_jobs));
  std::vector<nncp_job> host(jobs, jobs + n_jobs);  // staged before cudaMemcpyAsync returns
  NNC_CUDA_TRY(cudaMemcpyAsync(dev, host.data(), sizeof(nncp_job) * n_jobs,
                               cudaMemcpyHostToDevice, s));
  // rows of a multiple of four entries (16-byte reads), as few as the largest rank needs:
  // the slabs' limit in shared memory stays where rows of r put it, but for a few per cent
  const auto kern = rmax <= 4    ? cpx_cluster_kernel<T, 4>
                    : rmax <= 8  ? cpx_cluster_kernel<T, 8>
                    : rmax <= 12 ? cpx_cluster_kernel<T, 12>
                                 : cpx_cluster_kernel<T, 16>;
  NNC_CUDA_TRY(raise_smem_limit((const void*)kern, smem));
  kern<<<(unsigned)(n_jobs * kCl), kClThreads, smem, s>>>(dev, iters, (T)eps, slab_j, rel_errs,
                                                          statuses);
  note_launch(s);
  NNC_CUDA_TRY(cudaGetLastError());
  return NNC_OK;
}

template int nncp_cluster_batched<float>(int, const nncp_job*, int, double, double*, int*,
                                         cudaStream_t);
template int nncp_cluster_batched<double>(int, const nncp_job*, int, double, double*, int*,
                                          cudaStream_t);

}  // namespace nnc
