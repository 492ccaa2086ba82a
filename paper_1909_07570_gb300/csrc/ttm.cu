// SIMT mode products (n-mode multiplication, Appendix A) used by the FP32 and
// FP64 paths: the two passes over X of every sweep and all the small
// contractions around them.
//
// A tensor is viewed as (L, J, C) with J the contracted mode:
//   out[l, q, c] = sum_j Fm[j, q] * Y[l, j, c]
// The kernels by memory pattern:
//   * ttm_rows (C == 1): J is the contiguous axis (e.g. X x_3 F^(3)T). A block
//     stages tiles of Y's rows and the slice of Fm in a 3-deep cp.async ring;
//     each thread keeps TR rows x QP outputs in registers.
//   * ttm_cols_pipe (C > 1): J is strided (e.g. X x_1 F^(1)T). Each thread owns TC
//     flattened (l, c) columns and keeps QP outputs per column in registers; the
//     block's 256 TC columns are staged through a 3-deep cp.async ring of 16
//     rows j, so that two chunks are in flight while the third is consumed, and
//     Fm rows are broadcast from shared memory.
//   * ttm_cols_tc (float, C % 4 == 0, Q <= 32): the column product as a GEMM on
//     the tensor cores (TF32x3 on mma.sync, FP32-accurate), for the mode
//     products of the compressed tensors in the tensor-core paths.
// All accumulate in T and, when one pass would not fill the GPU, split J
// across blocks; partial sums are then added in split order (deterministic).
#include <type_traits>

#include "kernels.cuh"
#include "mma32.cuh"

namespace nnc {
namespace {

constexpr int kRowsThreads = 128;
// K-chunk of ttm_rows: 32 for float, 16 for double (static shared memory < 48 KB).
template <typename T>
__host__ __device__ constexpr int rows_bk() { return sizeof(T) == 4 ? 32 : 16; }
constexpr int kColsThreads = 256;
constexpr int kColsBJ = 32;

// Rows tile of BM = 128 TR rows x BK columns j in a 3-deep cp.async ring (single elements: a
// row of Y starts anywhere), with the chunk's rows of Fm; each thread keeps TR rows x QP
// outputs in registers, its terms in the order of k. What bounds it is the shared-memory
// reads, 1 + QP / 4 per TR rows and k; staged by plain loads between two barriers it waited
// on memory instead. 65317 x 255, Q = 12: 85.5 -> 32.7 us.
constexpr int kRowsStages = 3;
template <typename T, int QP, int TR>
constexpr size_t rows_smem_bytes() {
  constexpr size_t xs = (size_t)kRowsThreads * TR * (rows_bk<T>() + 1);
  return sizeof(T) * kRowsStages * (((xs + 3) & ~(size_t)3) + (size_t)rows_bk<T>() * QP);
}

template <typename T, int QP, int TR>
__global__ void __launch_bounds__(kRowsThreads)
ttm_rows_kernel(const T* __restrict__ Y, int64_t R, int K, int k_per_split,
                const T* __restrict__ Fm, int64_t fs_k, int64_t fs_q, int Q,
                T* __restrict__ out) {
  constexpr int BM = kRowsThreads * TR, BK = rows_bk<T>(), LD = BK + 1;
  constexpr int XS = (BM * LD + 3) & ~3;  // elements of one stage's Y tile
  constexpr int V = 16 / (int)sizeof(T);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* Xs = reinterpret_cast<T*>(smem_raw);
  T* Fs = Xs + kRowsStages * XS;

  const int tid = threadIdx.x;
  const int64_t r0 = (int64_t)blockIdx.x * BM;
  const int kbeg = blockIdx.y * k_per_split;
  const int kend = min(K, kbeg + k_per_split);
  const int nch = (kend - kbeg + BK - 1) / BK;
  const int rn = (int)min((int64_t)BM, R - r0);
  const T* y0 = Y + r0 * K;
  auto issue = [&](int c) {
    const int k0 = kbeg + c * BK, slot = c % kRowsStages;
    T* xs = Xs + slot * XS;
    const int kk = tid % BK, k = k0 + kk;
#pragma unroll 8
    for (int rr = tid / BK; rr < BM; rr += kRowsThreads / BK) {
      const bool ok = rr < rn && k < kend;
      cp_elem(xs + rr * LD + kk, ok ? y0 + (int64_t)rr * K + k : Y, ok);
    }
    T* fs = Fs + slot * BK * QP;
    for (int e = tid; e < BK * QP; e += kRowsThreads) {
      const int fk = e / QP, q = e % QP;
      const bool ok = q < Q && k0 + fk < kend;
      cp_elem(fs + e, ok ? Fm + ((k0 + fk) * fs_k + q * fs_q) : Fm, ok);
    }
  };

  T acc[TR][QP];
#pragma unroll
  for (int t = 0; t < TR; ++t)
#pragma unroll
    for (int q = 0; q < QP; ++q) acc[t][q] = T(0);

#pragma unroll
  for (int c = 0; c < kRowsStages - 1; ++c) {
    if (c < nch) issue(c);
    cp_commit();
  }
  for (int c = 0; c < nch; ++c) {
    if (c + kRowsStages - 1 < nch) issue(c + kRowsStages - 1);
    cp_commit();
    cp_wait<kRowsStages - 1>();
    __syncthreads();
    const T* xs = Xs + (c % kRowsStages) * XS + tid * LD;
    const T* fs = Fs + (c % kRowsStages) * BK * QP;
#pragma unroll 4
    for (int kk = 0; kk < BK; ++kk) {
      T x[TR];
#pragma unroll
      for (int t = 0; t < TR; ++t) x[t] = xs[t * kRowsThreads * LD + kk];
#pragma unroll
      for (int q = 0; q < QP; q += V) {
        T f[V];
        if constexpr (sizeof(T) == 4) {
          const float4 w = *reinterpret_cast<const float4*>(fs + kk * QP + q);
          f[0] = w.x; f[1] = w.y; f[2] = w.z; f[3] = w.w;
        } else {
          const double2 w = *reinterpret_cast<const double2*>(fs + kk * QP + q);
          f[0] = w.x; f[1] = w.y;
        }
#pragma unroll
        for (int u = 0; u < V; ++u)
#pragma unroll
          for (int t = 0; t < TR; ++t) acc[t][q + u] = fma(x[t], f[u], acc[t][q + u]);
      }
    }
    __syncthreads();
  }

  T* o = out + (int64_t)blockIdx.y * R * Q;
#pragma unroll
  for (int t = 0; t < TR; ++t) {
    const int64_t r = r0 + tid + t * kRowsThreads;
    if (r < R) {
#pragma unroll
      for (int q = 0; q < QP; ++q)
        if (q < Q) o[r * Q + q] = acc[t][q];
    }
  }
}

constexpr int kPipeBJ = 16;
constexpr int kPipeStages = 3;

template <typename T, int QP, int TC>
constexpr size_t pipe_smem_bytes() {
  return (size_t)kPipeStages * kPipeBJ * (kColsThreads * TC + QP) * sizeof(T);
}

// Flattened columns (l, c) col0 .. col0 + BC - 1 (BC = 256 TC, col0 =
// blockIdx.x BC), rows j of split blockIdx.y. Copies of CV entries: 16 bytes where
// C % CV == 0 keeps each in one row (l, j), else single entries (rows of Y that start
// anywhere: 301 x 55335, Q = 24, 66.6 us with loads straight into registers, whose
// latency nothing hid, 56.1 us through the ring, both beside the mode-2 branch). Rows
// and columns past the ends are staged as zeros (Fm rows too), so every chunk runs all
// kPipeBJ rows.
template <typename T, int QP, int TC, int CV>
__global__ void __launch_bounds__(kColsThreads, QP * TC * sizeof(T) < 256 ? 2 : 1)
ttm_cols_pipe_kernel(const T* __restrict__ Y, int64_t L, int J, int64_t C, int j_per_split, const T* __restrict__ Fm, int64_t fs_j, int64_t fs_q, int Q,
                     T* __restrict__ out) {
  constexpr int BC = kColsThreads * TC;
  constexpr int V = 16 / (int)sizeof(T);  // elements of a 16-byte read of Fm
  constexpr int CPR = BC / CV;            // copies per staged row
  static_assert(QP % V == 0, "QP must be a whole number of 16-byte vectors");
  using Vec = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* Ys = reinterpret_cast<T*>(smem_raw);      // [stage][kPipeBJ][BC]
  T* Fs = Ys + kPipeStages * kPipeBJ * BC;     // [stage][kPipeBJ][QP]
  const int tid = threadIdx.x;
  const int64_t ncols = L * C;
  const int64_t col0 = (int64_t)blockIdx.x * BC;
  const int jbeg = blockIdx.y * j_per_split;
  const int jend = min(J, jbeg + j_per_split);
  const int nchunks = (jend - jbeg + kPipeBJ - 1) / kPipeBJ;

  // This thread's copies: vector v of the rows jr, jr + RP, ... of a chunk.
  constexpr int RP = kColsThreads / CPR;
  static_assert(kColsThreads % CPR == 0 && kPipeBJ % RP == 0, "copy layout");
  const int v = tid % CPR, jr = tid / CPR;
  const int64_t vcol = col0 + (int64_t)v * CV;
  const bool cok = vcol < ncols;
  const int64_t vl = cok ? vcol / C : 0;
  const T* ysrc = Y + vl * (int64_t)J * C + (cok ? vcol - vl * C : 0);
  auto issue = [&](int chunk) {
    const int slot = chunk % kPipeStages;
    const int j0 = jbeg + chunk * kPipeBJ;
    T* ys = Ys + slot * kPipeBJ * BC + v * CV;
#pragma unroll
    for (int jj = jr; jj < kPipeBJ; jj += RP) {
      const int j = j0 + jj;
      const bool ok = cok && j < jend;
      const T* src = ok ? ysrc + (int64_t)j * C : Y;
      if constexpr (CV == 1) cp_elem(ys + jj * BC, src, ok);
      else cp_vec(ys + jj * BC, src, ok ? CV : 0);
    }
    // The Fm rows of the chunk go the same way (element copies), so that no
    // thread waits for them before the chunk it is about to consume.
    T* fs = Fs + slot * kPipeBJ * QP;
    for (int e = tid; e < kPipeBJ * QP; e += kColsThreads) {
      const int jj = e / QP, q = e % QP;
      const int j = j0 + jj;
      const bool ok = q < Q && j < jend;
      cp_elem(fs + e, ok ? Fm + (j * fs_j + q * fs_q) : Fm, ok);
    }
  };

  T acc[TC][QP];
#pragma unroll
  for (int t = 0; t < TC; ++t)
#pragma unroll
    for (int q = 0; q < QP; ++q) acc[t][q] = T(0);

#pragma unroll
  for (int p = 0; p < kPipeStages - 1; ++p) {
    if (p < nchunks) issue(p);
    cp_commit();
  }
  for (int it = 0; it < nchunks; ++it) {
    if (it + kPipeStages - 1 < nchunks) issue(it + kPipeStages - 1);
    cp_commit();
    cp_wait<kPipeStages - 1>();
    __syncthreads();
    const int slot = it % kPipeStages;
    const T* ys = Ys + slot * kPipeBJ * BC;
    const T* fs = Fs + slot * kPipeBJ * QP;
#pragma unroll 4
    for (int jj = 0; jj < kPipeBJ; ++jj) {
      T v[TC];
#pragma unroll
      for (int t = 0; t < TC; ++t) v[t] = ys[jj * BC + tid + t * kColsThreads];
      const Vec* fr = reinterpret_cast<const Vec*>(fs + jj * QP);
#pragma unroll
      for (int g = 0; g < QP / V; ++g) {
        const Vec f4 = fr[g];
        T f[V];
        if constexpr (sizeof(T) == 4) {
          f[0] = f4.x; f[1] = f4.y; f[2] = f4.z; f[3] = f4.w;
        } else {
          f[0] = f4.x; f[1] = f4.y;
        }
#pragma unroll
        for (int u = 0; u < V; ++u)
#pragma unroll
          for (int t = 0; t < TC; ++t) acc[t][g * V + u] = fma(f[u], v[t], acc[t][g * V + u]);
      }
    }
    __syncthreads();
  }

  T* o = out + (int64_t)blockIdx.y * L * Q * C;
#pragma unroll
  for (int t = 0; t < TC; ++t) {
    const int64_t col = col0 + tid + t * kColsThreads;
    if (col >= ncols) continue;
    const int64_t l = col / C;
    T* ot = o + l * Q * C + (col - l * C);
#pragma unroll
    for (int q = 0; q < QP; ++q)
      if (q < Q) ot[(int64_t)q * C] = acc[t][q];
  }
}

// Tensor-core column mode product (float, C % 4 == 0, Q <= 32): per block the
// GEMM D (kTcCols columns (l, c) x QP) = A (columns x rows j) B (rows j x QP),
// A the staged rows of Y (a column is an MMA row, j the MMA k), B the rows of
// Fm, on mma.sync m16n8k8 with TF32x3 operands (x = x_hi + x_lo, the three
// products lo*hi, hi*lo, hi*hi; the dropped lo*lo is below FP32 rounding) and
// FP32 accumulation. Each chunk of kTcBJ rows is summed in a fresh fragment
// and then added to the running sum with round-to-nearest, so the tensor
// core's truncating accumulation only ever acts on one chunk's sum. The rows
// are staged as in ttm_cols_pipe (a cp.async ring; rows and columns past the
// ends are zeros). Warp w owns columns 32 w .. 32 w + 31 (two M-tiles).
constexpr int kTcCols = 256;
constexpr int kTcBJ = 16;
constexpr int kTcStages = 4;
constexpr int kTcYS = kTcCols + 8;  // row stride: the A fragments hit 32 distinct banks

template <int QP>
__host__ __device__ constexpr int tc_fs() { return QP == 24 ? 24 : QP + 8; }
template <int QP>
constexpr size_t tc_smem_bytes() {
  return (size_t)kTcStages * kTcBJ * (kTcYS + tc_fs<QP>()) * sizeof(float);
}

__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  hi = mma32::tf32_rn(x);
  lo = mma32::tf32_rn(x - __uint_as_float(hi));
}

template <int QP>
__global__ void __launch_bounds__(kColsThreads, 2)
ttm_cols_tc_kernel(const float* __restrict__ Y, int64_t L, int J, int64_t C, int j_per_split,
                   const float* __restrict__ Fm, int64_t fs_j, int64_t fs_q, int Q,
                   float* __restrict__ out) {
  static_assert(kColsThreads == 256 && kTcCols == 256, "eight warps of 32 columns");
  constexpr int NT = QP / 8;
  constexpr int FS = tc_fs<QP>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* Ys = reinterpret_cast<float*>(smem_raw);  // [stage][kTcBJ][kTcYS]
  float* Fs = Ys + kTcStages * kTcBJ * kTcYS;       // [stage][kTcBJ][FS]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int64_t ncols = L * C;
  const int64_t col0 = (int64_t)blockIdx.x * kTcCols;
  const int jbeg = blockIdx.y * j_per_split;
  const int jend = min(J, jbeg + j_per_split);
  const int nchunks = (jend - jbeg + kTcBJ - 1) / kTcBJ;

  // This thread's copies: 16-byte vector v of rows jr, jr + 4, ... of a chunk
  // (a vector never crosses a row (l, j) because C % 4 == 0).
  const int v = tid & 63, jr = tid >> 6;
  const int64_t vcol = col0 + (int64_t)v * 4;
  const bool cok = vcol < ncols;
  const int64_t vl = cok ? vcol / C : 0;
  const float* ysrc = Y + vl * (int64_t)J * C + (cok ? vcol - vl * C : 0);
  auto issue = [&](int chunk) {
    const int slot = chunk % kTcStages;
    const int j0 = jbeg + chunk * kTcBJ;
    float* ys = Ys + slot * kTcBJ * kTcYS + v * 4;
#pragma unroll
    for (int jj = jr; jj < kTcBJ; jj += 4) {
      const int j = j0 + jj;
      const bool ok = cok && j < jend;
      cp_vec(ys + jj * kTcYS, ok ? ysrc + (int64_t)j * C : Y, ok ? 4 : 0);
    }
    float* fs = Fs + slot * kTcBJ * FS;
    for (int e = tid; e < kTcBJ * QP; e += kColsThreads) {
      const int jj = e / QP, q = e % QP;
      const int j = j0 + jj;
      const bool ok = q < Q && j < jend;
      cp_elem(fs + jj * FS + q, ok ? Fm + (j * fs_j + q * fs_q) : Fm, ok);
    }
  };

  float acc[2][NT][4], part[2][NT][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][n][e] = part[i][n][e] = 0.f;

#pragma unroll
  for (int p = 0; p < kTcStages - 1; ++p) {
    if (p < nchunks) issue(p);
    cp_commit();
  }
  for (int it = 0; it < nchunks; ++it) {
    if (it + kTcStages - 1 < nchunks) issue(it + kTcStages - 1);
    cp_commit();
    cp_wait<kTcStages - 1>();
    __syncthreads();
    const int slot = it % kTcStages;
    const float* ys = Ys + slot * kTcBJ * kTcYS + warp * 32 + g;
    const float* fs = Fs + slot * kTcBJ * FS + g;
#pragma unroll
    for (int ks = 0; ks < kTcBJ / 8; ++ks) {
      const float* y0 = ys + (ks * 8 + t) * kTcYS;
      const float* y1 = y0 + 4 * kTcYS;
      uint32_t ah[2][4], al[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        split_tf32(y0[16 * i], ah[i][0], al[i][0]);
        split_tf32(y0[16 * i + 8], ah[i][1], al[i][1]);
        split_tf32(y1[16 * i], ah[i][2], al[i][2]);
        split_tf32(y1[16 * i + 8], ah[i][3], al[i][3]);
      }
      const float* f0 = fs + (ks * 8 + t) * FS;
      const float* f1 = f0 + 4 * FS;
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        uint32_t bh0, bl0, bh1, bl1;
        split_tf32(f0[8 * n], bh0, bl0);
        split_tf32(f1[8 * n], bh1, bl1);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          mma32::mma_tf32(part[i][n], al[i], bh0, bh1);
          mma32::mma_tf32(part[i][n], ah[i], bl0, bl1);
          mma32::mma_tf32(part[i][n], ah[i], bh0, bh1);
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[i][n][e] += part[i][n][e];
          part[i][n][e] = 0.f;
        }
  }

  // D fragment: entry e of tile (i, n) is column 32 warp + 16 i + g + 8 (e / 2),
  // q = 8 n + 2 t + e % 2.
  float* o = out + (int64_t)blockIdx.y * L * Q * C;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t col = col0 + warp * 32 + 16 * i + g + 8 * h;
      if (col >= ncols) continue;
      const int64_t l = col / C;
      float* ot = o + l * Q * C + (col - l * C);
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int q = 8 * n + 2 * t + u;
          if (q < Q) ot[(int64_t)q * C] = acc[i][n][2 * h + u];
        }
    }
}

template <typename T>
__global__ void reduce_splits_kernel(const T* __restrict__ part, int splits, int64_t n,
                                     T* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    // Loads in groups of 8 (all in flight together), added in split order.
    T s = part[i];
    int p = 1;
    for (; p + 8 <= splits; p += 8) {
      T v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = part[(int64_t)(p + u) * n + i];
#pragma unroll
      for (int u = 0; u < 8; ++u) s += v[u];
    }
    for (; p < splits; ++p) s += part[(int64_t)p * n + i];
    out[i] = s;
  }
}

// The same sum where few outputs have many partials (the split-K products onto a
// factor's rows): a block takes 32 outputs, group g of 16 the partials p = g, g + 16,
// ... in order, and the groups are added in order. One thread per output would walk
// 288 partials one load group after another on six blocks: 15.1 -> 3.5 us (1536
// outputs).
constexpr int kRwCols = 32, kRwGroups = 16;
template <typename T>
__global__ void __launch_bounds__(kRwCols * kRwGroups)
reduce_splits_wide_kernel(const T* __restrict__ part, int splits, int64_t n,
                          T* __restrict__ out) {
  __shared__ T sums[kRwGroups][kRwCols];
  const int c = threadIdx.x % kRwCols, g = threadIdx.x / kRwCols;
  const int64_t i = (int64_t)blockIdx.x * kRwCols + c;
  T s = T(0);
  if (i < n) {
#pragma unroll 4
    for (int p = g; p < splits; p += kRwGroups) s += part[(int64_t)p * n + i];
  }
  sums[g][c] = s;
  __syncthreads();
  if (g == 0 && i < n) {
    for (int k = 1; k < kRwGroups; ++k) s += sums[k][c];
    out[i] = s;
  }
}

// The narrow form is the better one while its blocks fill the GPU or a thread has
// only a few load groups to walk.
template <typename T>
void reduce_splits(const T* part, int splits, int64_t n, T* out, cudaStream_t s) {
  const int64_t blocks = ceil_div(n, 256) < 4096 ? ceil_div(n, 256) : 4096;
  if (splits >= 2 * kRwGroups && blocks < device_sm_count())
    reduce_splits_wide_kernel<T><<<(unsigned)ceil_div(n, kRwCols), kRwCols * kRwGroups, 0, s>>>(
        part, splits, n, out);
  else
    reduce_splits_kernel<T><<<(unsigned)blocks, 256, 0, s>>>(part, splits, n, out);
  note_launch(s);
}

// Number of J-splits so that about two blocks per SM are in flight, bounded by
// the scratch capacity and by one 32-wide chunk of J per split.
int choose_splits(int64_t blocks, int J, int64_t out_elems, size_t split_cap, int chunk,
                  int* per_split) {
  const int64_t target = 2LL * device_sm_count();
  int splits = 1;
  if (blocks < target && J >= 2 * chunk && split_cap > 0) {
    int64_t want = ceil_div(target, blocks);
    int64_t by_j = J / chunk;
    int64_t by_cap = (int64_t)(split_cap / (size_t)out_elems);
    int64_t s = want;
    if (s > by_j) s = by_j;
    if (s > by_cap) s = by_cap;
    if (s > 1) splits = (int)s;
  }
  int per = (int)ceil_div(J, splits);
  per = (int)(ceil_div(per, chunk) * chunk);
  *per_split = per;
  return (int)ceil_div(J, per);
}

template <typename T, int QP>
cudaError_t ttm_dispatch(const T* Y, int64_t L, int J, int64_t C, const T* Fm, int64_t fs_j,
                         int64_t fs_q, int Q, T* out, T* split_buf, size_t split_cap,
                         cudaStream_t s) {
  const int64_t out_elems = L * Q * C;
  int per = J, splits = 1;
  if (C == 1) {
    // Two rows a thread (fewer reads of Fm) once the grid has four blocks per SM all the
    // same.
    constexpr bool two = sizeof(T) == 4 && QP <= 32;
    const bool use2 = two && ceil_div(L, 2 * kRowsThreads) >= 4LL * device_sm_count();
    const int64_t blocks = ceil_div(L, (use2 ? 2 : 1) * kRowsThreads);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    splits = choose_splits(blocks, J, out_elems, split_cap, rows_bk<T>(), &per);
    T* dst = splits > 1 ? split_buf : out;
    dim3 grid((unsigned)blocks, (unsigned)splits);
    auto run = [&](auto tr) -> cudaError_t {
      constexpr int TR = decltype(tr)::value;
      constexpr size_t smem = rows_smem_bytes<T, QP, TR>();
      const cudaError_t e0 = raise_smem_limit((const void*)ttm_rows_kernel<T, QP, TR>, smem);
      if (e0 != cudaSuccess) return e0;
      ttm_rows_kernel<T, QP, TR><<<grid, kRowsThreads, smem, s>>>(Y, L, J, per, Fm, fs_j, fs_q, Q,
                                                                  dst);
      return cudaSuccess;
    };
    const cudaError_t e0 = use2 ? run(std::integral_constant<int, two ? 2 : 1>{})
                                : run(std::integral_constant<int, 1>{});
    if (e0 != cudaSuccess) return e0;
    note_launch(s);
  } else {
    const int64_t ncols = L * C;
    constexpr int PV = 16 / (int)sizeof(T);
    const bool vec = C % PV == 0 && reinterpret_cast<uintptr_t>(Y) % 16 == 0;
    // Two columns per thread (16-byte copies only) when the grid still has two blocks per
    // SM.
    constexpr bool two = sizeof(T) == 4 && QP <= 32;
    const bool use2 = two && vec && ceil_div(ncols, 2 * kColsThreads) >= 2LL * device_sm_count();
    const int64_t blocks = ceil_div(ncols, (int64_t)(use2 ? 2 : 1) * kColsThreads);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    splits = choose_splits(blocks, J, out_elems, split_cap, kColsBJ, &per);
    T* dst = splits > 1 ? split_buf : out;
    dim3 grid((unsigned)blocks, (unsigned)splits);
    auto run = [&](auto tc, auto cv) -> cudaError_t {
      constexpr int TC = decltype(tc)::value, CV = decltype(cv)::value;
      constexpr size_t smem = pipe_smem_bytes<T, QP, TC>();
      const cudaError_t e0 = raise_smem_limit((const void*)ttm_cols_pipe_kernel<T, QP, TC, CV>, smem);
      if (e0 != cudaSuccess) return e0;
      ttm_cols_pipe_kernel<T, QP, TC, CV><<<grid, kColsThreads, smem, s>>>(Y, L, J, C, per, Fm, fs_j,
                                                                           fs_q, Q, dst);
      return cudaSuccess;
    };
    using One = std::integral_constant<int, 1>;
    using Vec16 = std::integral_constant<int, PV>;
    cudaError_t e0;
    if (use2) e0 = run(std::integral_constant<int, two ? 2 : 1>{}, Vec16{});
    else if (vec) e0 = run(One{}, Vec16{});
    else e0 = run(One{}, One{});
    if (e0 != cudaSuccess) return e0;
    note_launch(s);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || splits == 1) return e;
  reduce_splits<T>(split_buf, splits, out_elems, out, s);
  return cudaGetLastError();
}

template <int QP>
cudaError_t ttm_tc_dispatch(const float* Y, int64_t L, int J, int64_t C, const float* Fm,
                            int64_t fs_j, int64_t fs_q, int Q, float* out, float* split_buf,
                            size_t split_cap, cudaStream_t s) {
  const int64_t ncols = L * C, out_elems = L * Q * C;
  const int64_t blocks = ceil_div(ncols, kTcCols);
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  // Two or three blocks fit on an SM, so a grid of at least one block per SM
  // runs in one wave: J is split (with a second launch for the sums) only
  // below that (measured on the 4-way sweep's chains: 0.7 % faster per sweep).
  int per = J;
  const int splits = blocks >= device_sm_count()
                         ? 1
                         : choose_splits(blocks, J, out_elems, split_cap, kColsBJ, &per);
  float* dst = splits > 1 ? split_buf : out;
  constexpr size_t smem = tc_smem_bytes<QP>();
  const cudaError_t e0 = raise_smem_limit((const void*)ttm_cols_tc_kernel<QP>, smem);
  if (e0 != cudaSuccess) return e0;
  dim3 grid((unsigned)blocks, (unsigned)splits);
  ttm_cols_tc_kernel<QP><<<grid, kColsThreads, smem, s>>>(Y, L, J, C, per, Fm, fs_j, fs_q, Q, dst);
  note_launch(s);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || splits == 1) return e;
  reduce_splits<float>(split_buf, splits, out_elems, out, s);
  return cudaGetLastError();
}

}  // namespace

template <typename T>
cudaError_t launch_ttm(const T* Y, int64_t L, int J, int64_t C, const T* Fm, int64_t fs_j,
                       int64_t fs_q, int Q, T* out, T* split_buf, size_t split_cap,
                       cudaStream_t s) {
  if (L <= 0 || J <= 0 || C <= 0 || Q <= 0) return cudaErrorInvalidValue;
  if (Q <= 8) return ttm_dispatch<T, 8>(Y, L, J, C, Fm, fs_j, fs_q, Q, out, split_buf, split_cap, s);
  if (Q <= 12)
    return ttm_dispatch<T, 12>(Y, L, J, C, Fm, fs_j, fs_q, Q, out, split_buf, split_cap, s);
  if (Q <= 16) return ttm_dispatch<T, 16>(Y, L, J, C, Fm, fs_j, fs_q, Q, out, split_buf, split_cap, s);
  if (Q <= 24) return ttm_dispatch<T, 24>(Y, L, J, C, Fm, fs_j, fs_q, Q, out, split_buf, split_cap, s);
  if (Q <= 32) return ttm_dispatch<T, 32>(Y, L, J, C, Fm, fs_j, fs_q, Q, out, split_buf, split_cap, s);
  if (Q <= 64) return ttm_dispatch<T, 64>(Y, L, J, C, Fm, fs_j, fs_q, Q, out, split_buf, split_cap, s);
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_ttm_tc(const T* Y, int64_t L, int J, int64_t C, const T* Fm, int64_t fs_j,
                          int64_t fs_q, int Q, T* out, T* split_buf, size_t split_cap,
                          cudaStream_t s) {
  if constexpr (std::is_same<T, float>::value) {
    if (L > 0 && J > 0 && C > 1 && Q > 0 && Q <= 32 && C % 4 == 0 &&
        reinterpret_cast<uintptr_t>(Y) % 16 == 0) {
      if (Q <= 16)
        return ttm_tc_dispatch<16>(Y, L, J, C, Fm, fs_j, fs_q, Q, out, split_buf, split_cap, s);
      if (Q <= 24)
        return ttm_tc_dispatch<24>(Y, L, J, C, Fm, fs_j, fs_q, Q, out, split_buf, split_cap, s);
      return ttm_tc_dispatch<32>(Y, L, J, C, Fm, fs_j, fs_q, Q, out, split_buf, split_cap, s);
    }
  }
  return launch_ttm<T>(Y, L, J, C, Fm, fs_j, fs_q, Q, out, split_buf, split_cap, s);
}

template <typename T>
cudaError_t launch_reduce_splits(const T* part, int splits, int64_t n, T* out, cudaStream_t s) {
  reduce_splits<T>(part, splits, n, out, s);
  return cudaGetLastError();
}

template cudaError_t launch_reduce_splits<float>(const float*, int, int64_t, float*,
                                                 cudaStream_t);
template cudaError_t launch_reduce_splits<double>(const double*, int, int64_t, double*,
                                                  cudaStream_t);
template cudaError_t launch_ttm_tc<float>(const float*, int64_t, int, int64_t, const float*,
                                          int64_t, int64_t, int, float*, float*, size_t,
                                          cudaStream_t);
template cudaError_t launch_ttm_tc<double>(const double*, int64_t, int, int64_t, const double*,
                                           int64_t, int64_t, int, double*, double*, size_t,
                                           cudaStream_t);
template cudaError_t launch_ttm<float>(const float*, int64_t, int, int64_t, const float*, int64_t,
                                       int64_t, int, float*, float*, size_t, cudaStream_t);
template cudaError_t launch_ttm<double>(const double*, int64_t, int, int64_t, const double*,
                                        int64_t, int64_t, int, double*, double*, size_t,
                                        cudaStream_t);

}  // namespace nnc
