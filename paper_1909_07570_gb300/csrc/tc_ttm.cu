// Tensor-core (tcgen05) mode products: the two passes over X of an nnTD sweep
// (n-mode multiplication, Appendix A), in three number formats. The first two are
// described here, the FP16 pairs (F16x3, the FP32-accurate form of the fits) at
// f16_pass_kernel.
//
//   BF16    X is kept as a BF16 copy Xb with per-slice power-of-two scales s_i
//           (mode-1 slices), rows padded with zeros to Kp = roundup(N3, 64):
//             Xb[(i N2 + j) Kp + k] = bf16(X[i, j, k] / s_i)
//           Since s_i is a power of two, bf16(x / s_i) s_i == bf16(x): the
//           scales change no rounding. One BF16 MMA per K step, FP32 accumulate.
//   TF32x3  FP32-accurate: X is read as FP32 and every operand is split into
//           exact TF32 parts, x = x_hi + x_lo (x_hi: x rounded to TF32; x_lo:
//           x - x_hi rounded to TF32). Each K step issues two MMAs: x_hi
//           [f_hi; f_lo] (N = 2 NP, the two B parts stacked) and x_lo f_hi
//           (N = NP, into the f_lo half); the epilogue adds the two halves.
//           The dropped x_lo f_lo term and the rounding of the lo parts are
//           about 2^-22 of each product and of either sign.
//
// Pass 1, P3 = X x_3 F3^T: D[r, q] = sum_k A[r, k] B[q, k], r = (i, j), A K-major.
// Pass 2, P1 = X x_1 F1^T: D[c, a] = sum_i A[c, i] B[a, i], c = (j, k). BF16:
//   A read MN-major from Xb viewed as N1 x (N2 Kp). TF32x3: A read K-major
//   from Xt, a transposed copy of X made once per fit.
// B = F^T as operands [NP x K] (BF16: diag(s) folded into F1 for pass 2).
//
// Persistent CTAs, at most one per SM, each looping over 128-row tiles with
// warp roles:
//   warp 0        TMA producer: A tile and B slice of each K stage (a ring of as
//                 many stages as fit in shared memory, at most 8); the A tiles
//                 with an L2 evict-first hint (X is read once per pass)
//   warp 1        MMA issuer (one thread): tcgen05.mma into a double-buffered
//                 TMEM accumulator; tcgen05.commit frees stages and publishes
//                 finished accumulators
//   warps 2-5     epilogue: tcgen05.ld of the accumulator (warp w reads TMEM
//                 lanes 32 (w % 4) ..), scaled stores to global memory; with
//                 TcEpilogue::ysh also the tile's contraction with the
//                 matching factor rows (the nnTD sweep's mode-1 / mode-3 shares),
//                 by mma.sync on the tile staged in shared memory (mma32.cuh)
//   warps 6-9     TF32x3 only: split each staged A tile into x_hi (in place)
//                 and x_lo (into a 3-slot ring of its own)
// so a tile's epilogue overlaps the next tile's MMAs. The kernel is launched
// with programmatic stream serialization: the producer requests the first
// stages' A tiles (X, which no earlier kernel writes) before it waits for the
// preceding grid, and the B operands only after. Every mbarrier wait is
// bounded (about 2 s); on time-out the CTA flags an error, the other roles
// stop at their next wait, and TMEM is freed before the CTA exits.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <cstdio>
#include <mutex>
#include <type_traits>

#include "kernels.cuh"
#include "mma32.cuh"
#include "tc_ttm.cuh"

namespace nnc {
namespace tc {
namespace {

constexpr int kTileBytes = 128 * 128;  // one A stage: 128 rows x 128 bytes of K
constexpr int kThreadsTc = 320;        // 10 warps
constexpr long long kWaitCycles = 4000000000LL;  // about 2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait on phase `parity`. False when the limit ran out or another role
// of this CTA has already failed.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* fail,
                                          long long limit = kWaitCycles) {
  if (mbar_try_wait(bar, parity)) return true;  // the common case: no clock read
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (*fail) return false;
    if (clock64() - t0 > limit) {
      atomicExch(const_cast<int*>(fail), 1);
      return false;
    }
  }
  return true;
}

// An L2 policy that makes lines evicted first: the A tiles of a pass (X, its
// copies) are read once, so they should not push out the data the kernels
// after the pass read again (the pass result, the shares, factors and core).
__device__ __forceinline__ uint64_t l2_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void tma_load_2d_hint(void* dst, const CUtensorMap* tm, int x, int y,
                                                 uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, int x, int y,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor: 128-byte swizzle, descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr >> 4) & 0x3FFFu);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

// Instruction descriptor, FP32 accumulator, M = 128, N = n, B K-major.
// Operand format 1 = BF16 (kind::f16), 2 = TF32 (kind::tf32).
template <int KIND, bool kMN>
__device__ __forceinline__ uint32_t instr_desc(int n) {
  constexpr uint32_t fmt = KIND == kKindBf16 ? 1u : 2u;
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((kMN ? 1u : 0u) << 15) |
         (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(128 >> 4) << 24);
}

template <int KIND>
__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                    uint32_t idesc, uint32_t accumulate) {
  if constexpr (KIND == kKindBf16) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
        "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
        "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]),
        "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// x_hi: x rounded to TF32 (10 stored mantissa bits), to nearest with ties away
// from zero, by the integer rule of tf32_lo below. x - x_hi is then exact in
// FP32 and takes either sign, so on nonnegative data the dropped x_lo f_lo
// terms average out; with x_hi truncated every x_lo, and every dropped term,
// would be nonnegative and the products biased low. Finite |x| below
// (2 - 2^-11) 2^127.
__device__ __forceinline__ float tf32_hi(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}
// The remainder x - x_hi rounded to TF32, to nearest with ties away from zero:
// adding half of the dropped 13-bit field to the sign-magnitude bits and
// clearing the field rounds the magnitude (a carry moves into the exponent,
// as it should). Finite inputs only; this is the inner loop of the split, where
// integer operations run at full rate.
__device__ __forceinline__ float tf32_lo(float x, float hi) {
  return __uint_as_float((__float_as_uint(x - hi) + 0x1000u) & 0xFFFFE000u);
}

template <int KIND, int NP, bool FUSE = false>
struct TcLayout {
  static constexpr bool kTf32 = KIND == kKindTf32x3;
  // TF32x3: K stages rotate over kAcc accumulators that the epilogue adds in
  // FP32. The tensor core rounds its FP32 accumulation toward zero once per
  // MMA; shorter chains shrink that bias by kAcc.
  static constexpr int kAcc = kTf32 ? 128 / NP : 1;
  static_assert((kAcc & (kAcc - 1)) == 0, "accumulator index is taken by a mask");
  // TF32x3 accumulators are 2 NP columns wide: [0, NP) collects the main term
  // x_hi f_hi, [NP, 2 NP) the small terms x_hi f_lo (the same MMA of N = 2 NP
  // against the stacked [f_hi; f_lo] operand) and x_lo f_hi (an MMA of N = NP).
  static constexpr int kAccCols = kTf32 ? 2 * NP : NP;
  static constexpr int kTmemCols = 2 * kAcc * kAccCols;  // double-buffered
  static constexpr int kKStage = kTf32 ? 32 : 64;        // K elements per stage (128 bytes)
  static constexpr int kBBytes = NP * 128;               // one B slice
  // One ring stage: A | B (| B_lo right after B, so [B; B_lo] is one operand).
  static constexpr int kStageBytes = kTileBytes + kBBytes * (kTf32 ? 2 : 1);
  static constexpr int kOffB = kTileBytes;
  // TF32x3: x_lo tiles live in a short ring of their own; it only has to cover
  // the time from the split to the MMAs that read it.
  static constexpr int kLoSlots = kTf32 ? 3 : 0;
  static constexpr int kLoRing = kLoSlots > 0 ? kLoSlots : 1;  // index modulus
  static constexpr int kLoBytes = kLoSlots * kTileBytes;
  // Fused mode-1 contraction (pass X x_3 F3^T only): the tile's P3 rows and
  // the matching F2 rows, 128 x 32 FP32 each.
  static constexpr int kEpiBytes = FUSE ? 2 * 128 * 32 * 4 : 0;
  // As many stages as fit in the 227 KB of shared memory a CTA may use, less
  // the static barriers and the 1 KB alignment slack (at most 8).
  static constexpr int kStagesFit =
      (227 * 1024 - 512 - 1024 - kLoBytes - kEpiBytes) / kStageBytes;
  static constexpr int kStages = kStagesFit > 8 ? 8 : kStagesFit;
  static constexpr int kOffLo = kStages * kStageBytes;
  static constexpr int kOffEpi = kOffLo + kLoBytes;
  static constexpr int kSmem = 1024 + kOffEpi + kEpiBytes;
  static_assert(kTmemCols == 32 || kTmemCols == 64 || kTmemCols == 128 || kTmemCols == 256 ||
                kTmemCols == 512, "TMEM allocation must be a power of two >= 32 columns");
  static_assert(kStageBytes % 1024 == 0, "stages must keep 1024-byte swizzle atoms aligned");
  static_assert(!FUSE || NP == 32, "the fused contraction covers m3 <= 32");
};

// AND of `ok` over the 128 epilogue threads (named barrier 1).
__device__ __forceinline__ bool epi_all(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred q, p;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, 1, 128, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"(ok ? 1u : 0u)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// FUSE: row j of the factor (zero past yf_m) into row lr of Fs: rows of 8
// float4 chunks, chunk c stored at c ^ (row & 7), so that the row-per-thread
// stores and the chunk reads of the contraction avoid bank conflicts.
__device__ __forceinline__ void stage_factor_row(const TcEpilogue& ep, int64_t j, int lr,
                                                 float* Fs) {
  const float* f = ep.yf + j * ep.yf_m;
  float fr[32];
  if ((ep.yf_m & 3) == 0 && (reinterpret_cast<uintptr_t>(f) & 15) == 0) {
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float4 q = 4 * c < ep.yf_m ? *reinterpret_cast<const float4*>(f + 4 * c)
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
      fr[4 * c] = q.x; fr[4 * c + 1] = q.y; fr[4 * c + 2] = q.z; fr[4 * c + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int b = 0; b < 32; ++b) fr[b] = b < ep.yf_m ? f[b] : 0.f;
  }
#pragma unroll
  for (int c = 0; c < 8; ++c)
    *reinterpret_cast<float4*>(Fs + lr * 32 + ((c ^ (lr & 7)) << 2)) =
        make_float4(fr[4 * c], fr[4 * c + 1], fr[4 * c + 2], fr[4 * c + 3]);
}

// FUSE: contraction of the tile (one slab s, rows j0 .. j0 + 127) by the 128
// epilogue threads:
//   share[b, c] = sum_r F[j0 + r, b] P[(s, j0 + r), c]
// on the tensor cores (mma32.cuh: SPLIT = 1, TF32 operands beside the BF16
// rounding of X; 3, split TF32 in the FP32-accurate passes). The warp of quarter
// q takes rows 32 q .. 32 q + 31 with the whole 32 x 32 share (zero past m2,
// m3) in registers; the four partial shares are added in quarter order (`add`: onto what a
// round before wrote).
template <int SPLIT>
__device__ __forceinline__ void fused_share(const TcEpilogue& ep, int64_t tile, int lane,
                                            int quarter, float* Ps, const float* Fs,
                                            bool add = false) {
  const int et = threadIdx.x - 64;  // 0 .. 127
  const int o0 = mma32::frag_off(lane, 0), o1 = mma32::frag_off(lane, 1);
  float acc[2][4][4];
  mma32::zero(acc);
  epi_sync();  // Ps and Fs complete
#pragma unroll
  for (int ks = 4 * quarter; ks < 4 * quarter + 4; ++ks)
    mma32::step<SPLIT>(acc, Fs + ks * 256, Ps + ks * 256, o0, o1);
  epi_sync();  // Ps is reused for the partial shares
  float* red = Ps;  // 4 x 32 x 32
  mma32::store(red + quarter * 1024, acc, lane);
  epi_sync();
  const int m2 = ep.yf_m, m3 = ep.q, n = m2 * m3;
  float* yo = ep.ysh + tile * n;
  for (int e = et; e < n; e += 128) {
    const int bb = e / m3, cc = e % m3, o = mma32::tile_index(bb, cc);
    const float y = ((red[o] + red[o + 1024]) + red[o + 2048]) + red[o + 3072];
    float* z = yo + (ep.y_tr ? cc * m2 + bb : e);
    *z = add ? *z + y : y;
  }
  epi_sync();  // red and Fs are free for the next tile
}

template <int KIND, bool kMN, int NP, bool FUSE>
__global__ void __launch_bounds__(kThreadsTc, 1)
tc_pass_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmBlo, int nk, int64_t ntiles, TcEpilogue ep,
               int* err) {
  using L = TcLayout<KIND, NP, FUSE>;
  static_assert(!(L::kTf32 && kMN), "TF32x3 passes read A K-major");
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t full[L::kStages], empty[L::kStages], accfull[2], accempty[2];
  __shared__ uint64_t lofull[L::kLoRing], loempty[L::kLoRing];
  __shared__ uint32_t tmem_slot;
  __shared__ int fail;

  // 1024-byte aligned start, derived from smem_raw by pointer arithmetic so
  // that the compiler keeps every access through it in the shared space.
  unsigned char* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* vfail = &fail;
  // The successor kernel may be scheduled now; it waits for this grid itself.
  pdl_trigger();

  if (threadIdx.x == 0) {
    for (int s = 0; s < L::kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    if constexpr (L::kTf32) {
      for (int j = 0; j < L::kLoSlots; ++j) {
        mbar_init(&lofull[j], 4);
        mbar_init(&loempty[j], 1);
      }
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accfull[b], 1);
      mbar_init(&accempty[b], 4);
    }
    fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(L::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 0) {
    // ---- TMA producer ----------------------------------------------------------
    if (lane == 0) {
      // Stages this CTA runs: tiles blockIdx.x, blockIdx.x + gridDim.x, ...
      const int64_t my_tiles = (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
      const int64_t total = my_tiles * nk;
      const uint64_t stream_once = l2_evict_first();
      auto load_a = [&](int it_, unsigned char* st, uint64_t* bar) {
        const int64_t tile = blockIdx.x + static_cast<int64_t>(it_ / nk) * gridDim.x;
        const int m0 = static_cast<int>(tile * 128);
        const int k0 = (it_ % nk) * L::kKStage;
        if (!kMN) {
          tma_load_2d_hint(st, &tmA, k0, m0, bar, stream_once);
        } else {
          // 128 columns in 128-byte pieces: 2 (BF16) or 4 (TF32) boxes.
          constexpr int pieces = L::kTf32 ? 4 : 2;
          constexpr int piece_cols = 128 / pieces;
#pragma unroll
          for (int h = 0; h < pieces; ++h)
            tma_load_2d_hint(st + h * (kTileBytes / pieces), &tmA, m0 + h * piece_cols, k0, bar,
                             stream_once);
        }
      };
      auto load_b = [&](int it_, unsigned char* st, uint64_t* bar) {
        const int k0 = (it_ % nk) * L::kKStage;
        tma_load_2d(st + L::kOffB, &tmB, k0, 0, bar);
        if constexpr (L::kTf32) tma_load_2d(st + L::kOffB + L::kBBytes, &tmBlo, k0, 0, bar);
      };
      // X does not depend on earlier kernels: the first stages' A tiles are
      // requested before waiting for the predecessor grid, whose results (the
      // factor operands in B) are read only after the wait.
      const int pre = static_cast<int>(total < L::kStages ? total : L::kStages);
      for (int it = 0; it < pre; ++it) {
        mbar_expect_tx(&full[it], kTileBytes + L::kBBytes * (L::kTf32 ? 2 : 1));
        load_a(it, base + it * L::kStageBytes, &full[it]);
      }
      pdl_wait();
      for (int it = 0; it < pre; ++it) load_b(it, base + it * L::kStageBytes, &full[it]);
      int it = pre;
      bool ok = true;
      for (; it < total; ++it) {
        const int s = it % L::kStages;
        if (!mbar_wait(&empty[s], ((it / L::kStages) - 1) & 1, vfail)) {
          ok = false;
          break;
        }
        unsigned char* st = base + s * L::kStageBytes;
        mbar_expect_tx(&full[s], kTileBytes + L::kBBytes * (L::kTf32 ? 2 : 1));
        load_a(it, st, &full[s]);
        load_b(it, st, &full[s]);
      }
      if (!ok) {
        // Let the copies this CTA started land before it can exit (bounded).
        for (int back = 1; back <= L::kStages && it - back >= 0; ++back) {
          const int j = it - back;
          const long long t0 = clock64();
          while (!mbar_try_wait(&full[j % L::kStages], (j / L::kStages) & 1) &&
                 clock64() - t0 < kWaitCycles) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer --------------------------------------------------------------
    if (lane == 0) {
      const uint32_t idesc = instr_desc<KIND, kMN>(NP);
      const uint32_t idesc2 = instr_desc<KIND, kMN>(2 * NP);  // TF32x3: N = 2 NP
      int it = 0, tcount = 0;
      int rs = 0, rj = 0;         // stage and x_lo slot of `it`
      uint32_t rph = 0, jph = 0;  // their phase parities
      bool ok = true;
      for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x, ++tcount) {
        const int buf = tcount & 1;
        if (tcount >= 2 && !mbar_wait(&accempty[buf], ((tcount >> 1) - 1) & 1, vfail)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t acc0 = tmem + buf * L::kAcc * L::kAccCols;
        // One thread issues every MMA, so its own instruction count per stage
        // bounds the stage rate: ring positions advance by counters, and the
        // descriptors of a stage are formed once and stepped by constants (the
        // 14-bit address field of a shared-memory descriptor counts 16 bytes).
        for (int kc = 0; kc < nk; ++kc, ++it) {
          const uint32_t acc = acc0 + (kc & (L::kAcc - 1)) * L::kAccCols;
          if (!mbar_wait(&full[rs], rph, vfail) ||
              (L::kTf32 && !mbar_wait(&lofull[rj], jph, vfail))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t st = smem_u32(base + rs * L::kStageBytes);
          const uint64_t bdesc0 = smem_desc(st + L::kOffB, 16, 1024);
          uint64_t adesc0;
          if constexpr (kMN) {
            constexpr uint32_t lbo = L::kTf32 ? kTileBytes / 4 : kTileBytes / 2;
            adesc0 = smem_desc(st, lbo, 1024);
          } else {
            adesc0 = smem_desc(st, 16, 1024);
          }
          const uint64_t lodesc0 = smem_desc(smem_u32(base + L::kOffLo + rj * kTileBytes), 16, 1024);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            // K-major: +32 bytes per K step inside the swizzled 128-byte rows.
            // MN-major: +K-step rows of 128 bytes; column pieces LBO apart.
            constexpr uint32_t astep = kMN ? (L::kTf32 ? 1024 : 2048) : 32;
            const uint64_t adesc = adesc0 + (uint64_t)((kk * astep) >> 4);
            const uint64_t bdesc = bdesc0 + (uint64_t)((kk * 32) >> 4);
            const uint32_t accum = (kc >= L::kAcc || kk != 0) ? 1u : 0u;
            if constexpr (L::kTf32) {
              // x_hi [f_hi; f_lo] into columns [0, 2 NP), then x_lo f_hi into
              // [NP, 2 NP): the accumulator of the main term x_hi f_hi gets one
              // truncating add per K step, the small terms share the other.
              mma<KIND>(acc, adesc, bdesc, idesc2, accum);
              mma<KIND>(acc + NP, lodesc0 + (uint64_t)((kk * 32) >> 4), bdesc, idesc, 1u);
            } else {
              mma<KIND>(acc, adesc, bdesc, idesc, accum);
            }
          }
          mma_commit(&empty[rs]);
          if constexpr (L::kTf32) mma_commit(&loempty[rj]);
          if (++rs == L::kStages) {
            rs = 0;
            rph ^= 1u;
          }
          if (++rj == L::kLoRing) {
            rj = 0;
            jph ^= 1u;
          }
        }
        if (!ok) break;
        mma_commit(&accfull[buf]);
      }
    }
  } else if (warp < 6) {
    // ---- epilogue (warps 2-5) ------------------------------------------------
    const int quarter = warp & 3;  // TMEM lanes 32 quarter .. 32 quarter + 31
    const int lr = quarter * 32 + lane;  // tile row of this thread
    float* Ps = reinterpret_cast<float*>(base + L::kOffEpi);  // FUSE: 128 x 32 pass rows
    float* Fs = Ps + 128 * 32;                                // FUSE: 128 x 32 factor rows
    // FUSE: the factor may come from the preceding grid.
    if constexpr (FUSE) pdl_wait();
    int tcount = 0;
    int64_t fs_slice = -1;  // FUSE: the j range whose F2 rows Fs holds
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++tcount) {
      const int buf = tcount & 1;
      if constexpr (FUSE) {
        if (tile % ep.y_nh != fs_slice) {
          // F2 rows of this tile's j range (F2 is not written during the pass),
          // loaded when the range changes (never, when the grid is a multiple of
          // the tiles per slab); the previous tile ended with a barrier.
          fs_slice = tile % ep.y_nh;
          stage_factor_row(ep, fs_slice * 128 + lr, lr, Fs);
        }
      }
      const int64_t row = tile * 128 + lr;
      // Output row of the row-major layouts (-1: padding row, nothing stored)
      // and its scale, read before the wait so that the load is off the path.
      int64_t orow = -1;
      if (ep.p1_layout == 0) {
        if (row < ep.rows) orow = row;
      } else if (ep.p1_layout == 2) {
        const int64_t jj = row / ep.kp, k = row % ep.kp;
        if (jj < ep.n2 && k < ep.n3) orow = k * ep.n2 + jj;
      }
      const float sc = (orow >= 0 && ep.row_scale) ? ep.row_scale[orow / ep.rows_per_slice] : 1.f;
      const bool got = mbar_wait(&accfull[buf], (tcount >> 1) & 1, vfail);
      if constexpr (FUSE) {
        // All four warps take the same branch: the named barriers below need
        // every epilogue thread.
        if (!epi_all(got)) break;
      } else {
        // The warp-collective tcgen05.ld needs one decision for the whole warp.
        if (!__all_sync(0xffffffffu, got)) break;
      }
      tc_fence_after();
      const int nacc = nk < L::kAcc ? nk : L::kAcc;  // accumulators this tile wrote
      const uint32_t lanes = static_cast<uint32_t>(quarter * 32) << 16;
      const uint32_t accb = tmem + buf * L::kAcc * L::kAccCols + lanes;
#pragma unroll
      for (int c0 = 0; c0 < NP; c0 += 32) {
        uint32_t v[32];
        tmem_ld32(accb + c0, v);
        for (int q = 0; q < nacc; ++q) {
          if constexpr (L::kTf32) {
            uint32_t w[32];
            tmem_ld32(accb + q * L::kAccCols + NP + c0, w);  // x_hi f_lo
            if (q > 0) {
              uint32_t h[32];
              tmem_ld32(accb + q * L::kAccCols + c0, h);
#pragma unroll
              for (int t = 0; t < 32; ++t)
                w[t] = __float_as_uint(__uint_as_float(w[t]) + __uint_as_float(h[t]));
            }
#pragma unroll
            for (int t = 0; t < 32; ++t)
              v[t] = __float_as_uint(__uint_as_float(v[t]) + __uint_as_float(w[t]));
          } else if (q > 0) {
            uint32_t w[32];
            tmem_ld32(accb + q * L::kAccCols + c0, w);
#pragma unroll
            for (int t = 0; t < 32; ++t)
              v[t] = __float_as_uint(__uint_as_float(v[t]) + __uint_as_float(w[t]));
          }
        }
        if (ep.p1_layout != 1) {
          if (orow >= 0) {
            float* o = ep.out + orow * ep.q;
            if ((ep.q & 3) == 0) {
#pragma unroll
              for (int t = 0; t < 32; t += 4)
                if (c0 + t < ep.q)
                  *reinterpret_cast<float4*>(o + c0 + t) =
                      make_float4(__uint_as_float(v[t]) * sc, __uint_as_float(v[t + 1]) * sc,
                                  __uint_as_float(v[t + 2]) * sc, __uint_as_float(v[t + 3]) * sc);
            } else {
#pragma unroll
              for (int t = 0; t < 32; ++t)
                if (c0 + t < ep.q) o[c0 + t] = __uint_as_float(v[t]) * sc;
            }
          }
          if constexpr (FUSE) {
            // The stored P3 row (zero past m3) for the contraction below.
#pragma unroll
            for (int t = 0; t < 32; t += 4)
              *reinterpret_cast<float4*>(Ps + lr * 32 + (((t >> 2) ^ (lr & 7)) << 2)) =
                  make_float4(t < ep.q ? __uint_as_float(v[t]) * sc : 0.f,
                              t + 1 < ep.q ? __uint_as_float(v[t + 1]) * sc : 0.f,
                              t + 2 < ep.q ? __uint_as_float(v[t + 2]) * sc : 0.f,
                              t + 3 < ep.q ? __uint_as_float(v[t + 3]) * sc : 0.f);
          }
        } else {
          const int64_t jj = row / ep.kp, k = row % ep.kp;
          if (jj < ep.n2 && k < ep.n3) {
            float* o = ep.out + jj * ep.n3 + k;
#pragma unroll
            for (int t = 0; t < 32; ++t)
              if (c0 + t < ep.q) o[static_cast<int64_t>(c0 + t) * ep.slab] = __uint_as_float(v[t]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&accempty[buf]);
      if constexpr (FUSE) fused_share<L::kTf32 ? 3 : 1>(ep, tile, lane, quarter, Ps, Fs);
    }
  } else if constexpr (L::kTf32) {
    // ---- TF32 split of A (warps 6-9): A <- x_hi in place, x_lo to its ring ----
    const int ct = threadIdx.x - 192;  // 0 .. 127
    int it = 0;
    bool ok = true;
    for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
      for (int kc = 0; kc < nk; ++kc, ++it) {
        const int s = it % L::kStages, j = it % L::kLoRing;
        const bool got =
            mbar_wait(&full[s], (it / L::kStages) & 1, vfail) &&
            (it < L::kLoRing || mbar_wait(&loempty[j], ((it / L::kLoRing) - 1) & 1, vfail));
        if (!__all_sync(0xffffffffu, got)) {
          ok = false;
          break;
        }
        float4* a = reinterpret_cast<float4*>(base + s * L::kStageBytes);
        float4* alo = reinterpret_cast<float4*>(base + L::kOffLo + j * kTileBytes);
        // All loads of the stage are issued before the first store, so their
        // shared-memory latencies overlap instead of adding up.
        constexpr int kPer = kTileBytes / 16 / 128;
        float4 x[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) x[i] = a[ct + 128 * i];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          float4 h, l;
          h.x = tf32_hi(x[i].x); l.x = tf32_lo(x[i].x, h.x);
          h.y = tf32_hi(x[i].y); l.y = tf32_lo(x[i].y, h.y);
          h.z = tf32_hi(x[i].z); l.z = tf32_lo(x[i].z, h.z);
          h.w = tf32_hi(x[i].w); l.w = tf32_lo(x[i].w, h.w);
          a[ct + 128 * i] = h;
          alo[ct + 128 * i] = l;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&lofull[j]);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && fail) atomicExch(err, 1);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(L::kTmemCols)
                 : "memory");
  }
}

// ---- FP16 pair passes (kKindF16x3) ----------------------------------------------
//
// FP32-accurate passes on pairs of FP16 parts. X is kept as Xh + Xl, with
//   v = x / (s_i t_j u_k) = x_hi + 2^-11 x_lo,   x_hi = fp16(v), x_lo = fp16(2^11 (v - x_hi)),
// s, t, u powers of two that bring the largest entry of every slice of every mode
// close below 2^15. B is split the same way with u or s folded in and a power of two per
// column. x_hi [f_hi; f_lo] and x_lo f_hi are accumulated as in the TF32x3 pass, the last
// two in accumulators of their own that count 2^-11.
// Range: a pair holds 22 bits and a sign, as the TF32 pair does, from 2^-13 up (x_lo's
// factor takes it out of the subnormals: without it only from 2^-1), 28 powers of two
// below the largest entry; zeros are exact. The TF32 pair holds them at every magnitude. An X
// with a nonzero entry below 2^-18 is flagged by x_to_pair_kernel and runs with TF32x3 passes: down
// to there a pair loses a bit per power of two and is off by at most 2^-18 of the entry, no more
// than the truncating sums (over random tensors in blocks, with entries of X down to 2^-32 and rows
// of F down to 2^-66, the largest error of an entry of F from 64 bits after one to three
// sweeps is on average 0.85 times that of TF32x3 passes), and uniform 32-bit random numbers stay above
// it. Factor entries below the range (updates drive entries to zero) matter to an output
// that has no larger terms, as in a block of X of its own. What the products make of them is
// off by less than 2^-20 in the scales' units a term (the pair's 2^-36 of an entry of F times 2^15
// of X, the product of two low parts, which is not formed, and the tensor core's alignment of
// subnormal operands, whose products lose bits below 2^-23), so an output of 2^3 K or more over K
// terms is as exact as with 22 bits of every entry. A CTA that finds a smaller one goes
// over its tiles again, in rounds that take the entries of 28 powers of two each, scaled up into
// the range: the first overwrites the results, the others add to them, until no entry or no output
// is left below. A fit whose passes take such rounds often goes on with TF32x3 passes (PairGuard).
// Why pairs made once per fit instead of TF32 parts made in every pass: the
// TF32x3 stage moves each entry through shared memory five times (TMA in, read and
// two writes of the split, two reads by the MMAs, 8 bytes an entry in the last
// three) and no role of it bounds it alone, 137-151 us a pass at 512^3, m = 32. A pair
// is as large as the FP32 entry, comes in by TMA and goes out by the MMAs, at half the
// bytes. Both passes read the same copy: pass 1 K-major, pass 2 MN-major (no
// transposed copy). 512^3, m = 32: 137 -> 124 us (pass 1, with its shares) and
// 141 -> 97 us (pass 2) for 537 MB, 4.3 and 5.5 TB/s; 256^3, m = 20, where the pair (67 MB)
// stays in L2 from pass to pass: 27 -> 20-23 us in the sweep.
//
// Warps 0 and 1 as in tc_pass_kernel, warps 2-5 the epilogue. B stays in shared
// memory for the whole pass: warps 2-9 read the factor, find each column's
// largest entry, and write the split operand into the swizzled layout, while the first
// stages of X are in flight (no operand is formed by the updates, and a stage
// carries X alone).
constexpr int kF16Stage = 2 * kTileBytes;  // x_hi, x_lo: 128 rows x 64 K entries
constexpr int kF16MaxStages = 8;
constexpr int kF16MinStages = 3;
// Stages a set of accumulators sums before the epilogue adds them in FP32. The tensor
// core truncates as it accumulates, one-sided on nonnegative data and more with every
// product in an accumulator: at NP = 32 the four K steps of a stage go to four
// accumulators, 32 products each in a group of two stages. With one group a
// tile (64 products an accumulator at K = 256) the factors after 30 sweeps were
// 1.5 times as far from 64 bits as with the TF32x3 passes. Up to 128 K entries the
// TF32x3 pass puts 32 products in an accumulator too and the FP16 form is the less exact
// per product: there a group is one stage (128^3 x 64, 30 sweeps: F4 1.24e-6 from 64 bits
// with groups of two, 0.93e-6 with one, TF32x3 0.94e-6; 19.9 -> 20.4 ms). For longer K
// groups of two are closer than TF32x3 (512^3: 9e-7 against 1.3e-5) and 5 % faster.
__host__ __device__ constexpr int f16_group(int nk) { return nk <= 2 ? 1 : 2; }

struct F16Operand {
  const float* F;       // K x q row-major
  const float* kscale;  // u or s by K index
  int K, q;
};

template <int NP>
__host__ __device__ constexpr int f16_b_bytes(int nk) { return nk * 2 * NP * 128; }
// Stages that fit beside the operand and the epilogue's tiles.
template <int NP, bool FUSE>
__host__ __device__ inline int f16_stages(int nk) {
  const int room = 227 * 1024 - 1536 - 1024 - f16_b_bytes<NP>(nk) - (FUSE ? 2 * 128 * 32 * 4 : 0);
  const int n = room / kF16Stage;
  return n > kF16MaxStages ? kF16MaxStages : n;
}
template <int NP, bool FUSE>
__host__ __device__ inline int f16_smem(int nk) {
  return 1024 + f16_stages<NP, FUSE>(nk) * kF16Stage + f16_b_bytes<NP>(nk) +
         (FUSE ? 2 * 128 * 32 * 4 : 0);
}

__device__ __forceinline__ uint32_t f16_instr_desc(bool mn, int n) {
  // FP16 operands (format 0), FP32 accumulator, M = 128, B K-major.
  return (1u << 4) | ((mn ? 1u : 0u) << 15) | (static_cast<uint32_t>(n >> 3) << 17) |
         (static_cast<uint32_t>(128 >> 4) << 24);
}

// Exponent e with 2^14 <= v 2^-e < 2^15 for the bits of a positive float, within
// the range whose powers of two are normal floats; 0 for zero.
__device__ __forceinline__ int f16_exponent(unsigned bits) {
  const int e = (int)(bits >> 23) - 127 - 14;
  return bits == 0u ? 0 : (e < -126 ? -126 : e);
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// v = hi + lo / kF16LoScale; 22 bits for |v| in [kF16Least, 2^15).
constexpr float kF16LoScale = 2048.f;
constexpr float kF16Least = 0x1p-13f, kF16LeastX = 0x1p-18f;
__device__ __forceinline__ void split_f16(float v, __half& hi, __half& lo) {
  hi = __float2half_rn(v);
  lo = __float2half_rn((v - __half2float(hi)) * kF16LoScale);
}

// The pass's B operand in shared memory (256 threads: warps 2-9): for each 64-entry
// K chunk 2 NP rows of 128 bytes, rows [0, NP) f_hi and [NP, 2 NP) f_lo of
// F[k, q] kscale[k] / cscale[q], in the 128-byte swizzle. cs[q] gets cscale. *low gets 1 when
// a nonzero entry lies below the range. A column whose largest entry is so small that products
// with kscale may be subnormal is left to the rounds.
constexpr int kF16RoundBits = 28, kF16MaxRounds = 16;  // every product of two floats
constexpr int kF16LeaveExp = -112;
__device__ __forceinline__ unsigned char* f16_b_row(unsigned char* bs, int np, int o, int n) {
  return bs + (o >> 3) * (2 * np * 128) + n * 128 + (((o & 7) ^ (n & 7)) << 4);
}
template <int NP>
__device__ __forceinline__ void f16_operand(const F16Operand& fo, int nk, unsigned char* bs,
                                            float* cs, unsigned* cmax, int* low_out) {
  const int t = threadIdx.x - 64, lane = t & 31, w = t >> 5;
  constexpr int NC = NP / 32;  // columns per lane
  const int noct = nk * 8;     // octets of K entries
  auto in = [&](int k, int n) { return k < fo.K && n < fo.q; };
  for (int n = t; n < NP; n += 256) cmax[n] = 0u;
  asm volatile("bar.sync 2, 256;" ::: "memory");
  float mx[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) mx[c] = 0.f;
  for (int o = w; o < noct; o += 8) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = 8 * o + u, n = lane + 32 * c;
        v[u] = in(k, n) ? fo.F[(int64_t)k * fo.q + n] * fo.kscale[k] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) mx[c] = fmaxf(mx[c], fabsf(v[u]));
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) atomicMax(&cmax[lane + 32 * c], __float_as_uint(mx[c]));
  asm volatile("bar.sync 2, 256;" ::: "memory");
  float inv[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int e = f16_exponent(cmax[lane + 32 * c]);
    const bool leave = e < kF16LeaveExp;
    inv[c] = leave ? 0.f : pow2f(-e);
    if (w == 0) cs[lane + 32 * c] = pow2f(e);
  }
  bool low = false;
  for (int o = w; o < noct; o += 8) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int n = lane + 32 * c;
      float f[8], ks[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {  // sixteen loads in flight
        const int k = 8 * o + u;
        f[u] = in(k, n) ? fo.F[(int64_t)k * fo.q + n] : 0.f;
        ks[u] = in(k, n) ? fo.kscale[k] : 0.f;
      }
      union { __half h[8]; uint4 q; } hi, lo;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float y = f[u] * ks[u] * inv[c];
        low |= fabsf(y) < kF16Least && f[u] != 0.f;
        split_f16(y, hi.h[u], lo.h[u]);
      }
      unsigned char* row = f16_b_row(bs, NP, o, n);
      *reinterpret_cast<uint4*>(row) = hi.q;
      *reinterpret_cast<uint4*>(row + NP * 128) = lo.q;
    }
  }
  if (low) *low_out = 1;
}

// m 2^x: exact where the result is a normal float, else infinite or about as small as it is.
__device__ __forceinline__ float scaled(float m, int x) {
  for (; x > 127; x -= 127) m *= 0x1p127f;
  for (; x < -126; x += 126) m *= 0x1p-126f;
  return m * pow2f(x);
}

// The operand of round w > 0: the entries of the w-th 28 powers of two below the column's
// largest (and whatever is not below them, in round 1), scaled up into the first, zero for the
// others; *low_out as above.
__device__ __noinline__ void f16_operand_round(const F16Operand& fo, int np, int nk,
                                               unsigned char* bs, const unsigned* cmax, int round,
                                               int* low_out) {
  const int t = threadIdx.x - 64, lane = t & 31;
  bool low = false;
  for (int o = t >> 5; o < nk * 8; o += 8)
    for (int n = lane; n < np; n += 32) {
      const int up = kF16RoundBits * (round - 1) - f16_exponent(cmax[n]);
      float f[8], ks[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = 8 * o + u;
        const bool in = k < fo.K && n < fo.q;
        f[u] = in ? fo.F[(int64_t)k * fo.q + n] : 0.f;
        ks[u] = in ? fo.kscale[k] : 1.f;
      }
      union { __half h[8]; uint4 q; } hi, lo;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float y = scaled(f[u], (__float_as_int(ks[u]) >> 23) - 127 + up);
        const bool under = fabsf(y) < kF16Least;
        low |= under && f[u] != 0.f;
        split_f16(under || (round > 1 && !(fabsf(y) < 32768.f)) ? 0.f : y, hi.h[u], lo.h[u]);
      }
      unsigned char* row = f16_b_row(bs, np, o, n);
      *reinterpret_cast<uint4*>(row) = hi.q;
      *reinterpret_cast<uint4*>(row + np * 128) = lo.q;
    }
  if (low && round + 1 < kF16MaxRounds) *low_out = 1;
}

// AND of `ok` over warps 2-9 (named barrier 2).
__device__ __forceinline__ bool all_of_256(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred q, p;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, 2, 256, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"(ok ? 1u : 0u)
      : "memory");
  return r != 0;
}

template <bool kMN, int NP, bool FUSE>
__global__ void __launch_bounds__(kThreadsTc, 1)
f16_pass_kernel(const __grid_constant__ CUtensorMap tmHi, const __grid_constant__ CUtensorMap tmLo,
                F16Operand fo, int nk, int64_t ntiles, TcEpilogue ep, int* err) {
  static_assert(!FUSE || (NP == 32 && !kMN), "the fused contraction covers m3 <= 32 of pass 1");
  constexpr int kAcc = 128 / NP;      // accumulators the K stages rotate over
  constexpr int kAccCols = 2 * NP;    // [0, NP) x_hi f_hi, [NP, 2 NP) the small terms
  constexpr int kTmemCols = 2 * kAcc * kAccCols;
  static_assert(kTmemCols == 512, "all of the tensor memory");
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t full[kF16MaxStages], empty[kF16MaxStages], accfull[2], accempty[2], bready;
  __shared__ float cs[NP];
  __shared__ unsigned cmax[NP];
  // Of each round: an entry below the range (f16_operand), and another round to follow.
  __shared__ int low[kF16MaxRounds], again[kF16MaxRounds];
  __shared__ uint64_t decided;
  __shared__ uint32_t tmem_slot;
  __shared__ int fail;

  unsigned char* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int nst = f16_stages<NP, FUSE>(nk);
  unsigned char* bs = base + nst * kF16Stage;
  unsigned char* epi = bs + f16_b_bytes<NP>(nk);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* vfail = &fail;
  pdl_trigger();

  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accfull[b], 1);
      mbar_init(&accempty[b], 4);
    }
    mbar_init(&bready, 8);
    mbar_init(&decided, 1);
    for (int w = 0; w < kF16MaxRounds; ++w) low[w] = again[w] = 0;
    fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 0) {
    // ---- TMA producer ----------------------------------------------------------
    // The pair of X is complete before any pass is launched, so its tiles are
    // requested without waiting for the predecessor grid.
    if (lane == 0) {
      const int64_t my_tiles = (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
      const uint64_t once = l2_evict_first();
      auto load = [&](const CUtensorMap* tm, void* dst, int x, int y, uint64_t* bar) {
        if (ep.x_resident) tma_load_2d(dst, tm, x, y, bar);
        else tma_load_2d_hint(dst, tm, x, y, bar, once);
      };
      int64_t it = 0;
      int s = 0;
      uint32_t ph = 1;  // the first round's stages are free
      bool ok = true, more = true;
      for (int round = 0; ok && more; ++round) {
        // Whether another round may follow is known when this round's operand is; asked before
        // the round's last load, so that the next operand's phase cannot end meanwhile.
        int64_t ask = my_tiles * nk - 1;
        ask = ask < nst ? ask : nst;
        int64_t c = 0;
        for (int64_t q = 0; ok && q < my_tiles; ++q) {
          const int m0 = static_cast<int>((blockIdx.x + q * gridDim.x) * 128);
          for (int kc = 0; kc < nk; ++kc, ++it, ++c) {
            if (c == ask) {
              ok = mbar_wait(&bready, round & 1, vfail);
              more = ok && low[round] != 0;
            }
            if (!ok || (it >= nst && !mbar_wait(&empty[s], ph, vfail))) {
              ok = false;
              break;
            }
            unsigned char* st = base + s * kF16Stage;
            mbar_expect_tx(&full[s], kF16Stage);
            if (!kMN) {
              load(&tmHi, st, kc * 64, m0, &full[s]);
              load(&tmLo, st + kTileBytes, kc * 64, m0, &full[s]);
            } else {
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                load(&tmHi, st + h * (kTileBytes / 2), m0 + h * 64, kc * 64, &full[s]);
                load(&tmLo, st + kTileBytes + h * (kTileBytes / 2), m0 + h * 64, kc * 64,
                     &full[s]);
              }
            }
            if (++s == nst) {
              s = 0;
              ph ^= 1u;
            }
          }
        }
        if (ok && more) {
          ok = mbar_wait(&decided, round & 1, vfail);
          more = ok && again[round] != 0;
        }
      }
      if (!ok) {
        // Let the copies this CTA started land before it can exit (bounded).
        for (int back = 1; back <= nst && it - back >= 0; ++back) {
          const int64_t j = it - back;
          const long long t0 = clock64();
          while (!mbar_try_wait(&full[j % nst], (j / nst) & 1) && clock64() - t0 < kWaitCycles) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer ----------------------------------------------------------------
    if (lane == 0) {
      const uint32_t idesc = f16_instr_desc(kMN, NP);
      const uint32_t idesc2 = f16_instr_desc(kMN, 2 * NP);
      const uint64_t bdesc_base = smem_desc(smem_u32(bs), 16, 1024);
      int gcount = 0, rs = 0;  // groups of stages; the ring's stage
      const int group = f16_group(nk);
      uint32_t rph = 0;
      bool ok = true, more = true;
      for (int round = 0; ok && more; ++round) {
        ok = mbar_wait(&bready, round & 1, vfail);
        more = ok && low[round] != 0;
        for (int64_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
          for (int k0 = 0; ok && k0 < nk; k0 += group, ++gcount) {
            const int buf = gcount & 1, kend = min(nk, k0 + group);
            if (gcount >= 2 && !mbar_wait(&accempty[buf], ((gcount >> 1) - 1) & 1, vfail)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t acc0 = tmem + buf * kAcc * kAccCols;
            for (int kc = k0; kc < kend; ++kc) {
              if (!mbar_wait(&full[rs], rph, vfail)) {
                ok = false;
                break;
              }
              tc_fence_after();
              const uint32_t st = smem_u32(base + rs * kF16Stage);
              const uint64_t hidesc = smem_desc(st, kMN ? kTileBytes / 2 : 16, 1024);
              const uint64_t lodesc = smem_desc(st + kTileBytes, kMN ? kTileBytes / 2 : 16, 1024);
              const uint64_t bdesc0 = bdesc_base + (uint64_t)((kc * 2 * NP * 128) >> 4);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                constexpr uint32_t astep = kMN ? 2048 : 32;
                const uint64_t astep16 = (uint64_t)((kk * astep) >> 4);
                const uint64_t bdesc = bdesc0 + (uint64_t)((kk * 32) >> 4);
                const uint32_t acc = acc0 + (kk & (kAcc - 1)) * kAccCols;
                const uint32_t accum = (kc > k0 || kk >= kAcc) ? 1u : 0u;
                mma<kKindBf16>(acc, hidesc + astep16, bdesc, idesc2, accum);
                mma<kKindBf16>(acc + NP, lodesc + astep16, bdesc, idesc, 1u);
              }
              mma_commit(&empty[rs]);
              if (++rs == nst) {
                rs = 0;
                rph ^= 1u;
              }
            }
            if (ok) mma_commit(&accfull[buf]);
          }
        }
        if (ok && more) {
          ok = mbar_wait(&decided, round & 1, vfail);
          more = ok && again[round] != 0;
        }
      }
    }
  } else {
    // ---- the B operand (warps 2-9) -------------------------------------------------
    pdl_wait();
    int gcount = 0;
    // ---- epilogue of a round (warps 2-5); false: a wait gave up ------------------------
    bool starved = false;  // an output of the round's tiles is too small for what it lacks
    auto epilogue = [&](auto first, auto asked, int round) -> bool {
      constexpr bool kFirst = decltype(first)::value, kAsk = decltype(asked)::value;
      // The least output that needs none of what its round leaves out (see above): of the low
      // entries in round 0, of those of the ranges to come after it.
      const float enough = round == 0 ? 8.f * fo.K : 0x1p24f * fo.K;
      bool got = true;
      const int quarter = warp & 3;
      const int lr = quarter * 32 + lane;
      float* Ps = reinterpret_cast<float*>(epi);  // FUSE: 128 x 32 pass rows
      float* Fs = Ps + 128 * 32;                  // FUSE: 128 x 32 factor rows
      int64_t fs_slice = -1;
      const int group = f16_group(nk);
      for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        if constexpr (FUSE) {
          if (tile % ep.y_nh != fs_slice) {
            fs_slice = tile % ep.y_nh;
            stage_factor_row(ep, fs_slice * 128 + lr, lr, Fs);
          }
        }
        const int64_t row = tile * 128 + lr;
        // Row (a, b) = (row / kp, row % kp): (i, j) of pass 1, (j, k) of pass 2.
        const int64_t ra = row / ep.kp, rb = row % ep.kp;
        const bool live = ra < ep.ra_n && rb < ep.rb_n;
        int64_t orow = -1;
        if (live) orow = ep.p1_layout == 2 ? rb * ep.n2 + ra : row;
        const float rsc = live ? ep.ra_scale[ra] * ep.rb_scale[rb] : 1.f;
        // The tile's sums: every group's accumulators added in FP32.
        float sum[NP];
#pragma unroll
        for (int t = 0; t < NP; ++t) sum[t] = 0.f;
        for (int k0 = 0; k0 < nk; k0 += group, ++gcount) {
          const int buf = gcount & 1;
          got = mbar_wait(&accfull[buf], (gcount >> 1) & 1, vfail);
          if constexpr (FUSE) got = epi_all(got);
          else got = __all_sync(0xffffffffu, got);
          if (!got) break;
          tc_fence_after();
          const uint32_t accb =
              tmem + buf * kAcc * kAccCols + (static_cast<uint32_t>(quarter * 32) << 16);
#pragma unroll
          for (int c0 = 0; c0 < NP; c0 += 32) {
#pragma unroll
            for (int q = 0; q < kAcc; ++q) {
              uint32_t h[32], w[32];
              tmem_ld32(accb + q * kAccCols + c0, h);
              tmem_ld32(accb + q * kAccCols + NP + c0, w);
#pragma unroll
              for (int t = 0; t < 32; ++t)
                sum[c0 + t] += fmaf(__uint_as_float(w[t]), 1.f / kF16LoScale,
                                    __uint_as_float(h[t]));
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&accempty[buf]);
        }
        if (!got) break;
#pragma unroll
        for (int c0 = 0; c0 < NP; c0 += 32) {
          float* v = sum + c0;
          // Powers of two: the column's first (its result is the entry without the
          // row's scale), then the row's.
          const double down = kFirst ? 0.0 : ldexp((double)rsc, -kF16RoundBits * (round - 1));
          if constexpr (kFirst) {
            if (kAsk && live) {
              float least = INFINITY;
              if (c0 + 32 <= ep.q) {
#pragma unroll
                for (int t = 0; t < 32; ++t) least = fminf(least, fabsf(v[t]));
              } else {
#pragma unroll
                for (int t = 0; t < 32; ++t)
                  if (c0 + t < ep.q) least = fminf(least, fabsf(v[t]));
              }
              starved |= least < enough;
            }
#pragma unroll
            for (int t = 0; t < 32; ++t) v[t] = v[t] * cs[c0 + t] * rsc;
          } else {
#pragma unroll
            for (int t = 0; t < 32; ++t) v[t] = (float)((double)v[t] * cs[c0 + t] * down);
          }
          // A later round adds to what is there.
          auto add = [&](float* z, int t) {
            *z += v[t];
            starved |= kAsk && fabsf(*z) < (double)enough * cs[c0 + t] * down;
          };
          if (ep.p1_layout != 1) {
            if (orow >= 0) {
              float* o = ep.out + orow * ep.q;
              if constexpr (!kFirst) {
#pragma unroll
                for (int t = 0; t < 32; ++t)
                  if (c0 + t < ep.q) add(o + c0 + t, t);
              } else if ((ep.q & 3) == 0) {
#pragma unroll
                for (int t = 0; t < 32; t += 4)
                  if (c0 + t < ep.q)
                    *reinterpret_cast<float4*>(o + c0 + t) =
                        make_float4(v[t], v[t + 1],
                                    v[t + 2], v[t + 3]);
              } else {
#pragma unroll
                for (int t = 0; t < 32; ++t)
                  if (c0 + t < ep.q) o[c0 + t] = v[t];
              }
            }
            if constexpr (FUSE) {
#pragma unroll
              for (int t = 0; t < 32; t += 4)
                *reinterpret_cast<float4*>(Ps + lr * 32 + (((t >> 2) ^ (lr & 7)) << 2)) =
                    make_float4(t < ep.q ? v[t] : 0.f,
                                t + 1 < ep.q ? v[t + 1] : 0.f,
                                t + 2 < ep.q ? v[t + 2] : 0.f,
                                t + 3 < ep.q ? v[t + 3] : 0.f);
            }
          } else if (live) {
            float* o = ep.out + ra * ep.n3 + rb;
#pragma unroll
            for (int t = 0; t < 32; ++t)
              if (c0 + t < ep.q) {
                float* z = o + static_cast<int64_t>(c0 + t) * ep.slab;
                if constexpr (kFirst) *z = v[t];
                else add(z, t);
              }
          }
        }
        if constexpr (FUSE) fused_share<3>(ep, tile, lane, quarter, Ps, Fs, !kFirst);
      }
      return got;
    };
    // Whether another round follows (in all of warps 2-9 alike; the other roles are told). Every
    // MMA of the round is done: warps 2-5 have read its last accumulators.
    auto next_round = [&](bool got, int round) -> bool {
      if (low[round] == 0) return false;
      if (!all_of_256(got && *vfail == 0)) return false;  // the other roles stop at their waits
      const bool more = !all_of_256(!starved);
      if (threadIdx.x == 64) {
        again[round] = more ? 1 : 0;
        mbar_arrive(&decided);
      }
      starved = false;
      return more;
    };
    auto operand_done = [&]() {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&bready);
      asm volatile("bar.sync 2, 256;" ::: "memory");  // cs and low[round] complete
    };
    f16_operand<NP>(fo, nk, bs, cs, cmax, low);
    operand_done();
    bool got = true;
    const auto yes = std::true_type{};
    const auto no = std::false_type{};
    if (warp < 6) got = low[0] == 0 ? epilogue(yes, no, 0) : epilogue(yes, yes, 0);
    int round = 0;
    while (next_round(got, round)) {
      ++round;
      f16_operand_round(fo, NP, nk, bs, cmax, round, low + round);
      operand_done();
      if (warp < 6) got = round == 1 ? epilogue(yes, yes, 1) : epilogue(no, yes, round);
    }
    if (threadIdx.x == 64 && round > 0) atomicAdd(err + kFlagRounds, round);
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && fail) atomicExch(err, 1);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTmemCols)
                 : "memory");
  }
}

// ---- the FP16 pair of X ------------------------------------------------------------

// rmax[r] = bits of max_k |X[r, k]| over the rows of X (R x N3): LW lanes a row (the
// power of two at and above its 16-byte pieces, at most a warp), two rows in
// flight per lane group.
__global__ void __launch_bounds__(256)
row_max_kernel(const float* __restrict__ X, int64_t R, int N3, int lw, unsigned* __restrict__ rmax) {
  const int lane = threadIdx.x & (lw - 1);
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x / lw);
  const int64_t g0 = (int64_t)blockIdx.x * (blockDim.x / lw) + threadIdx.x / lw;
  const int nv = N3 >> 2;
  // Every group runs the same number of rounds: the shuffles take whole warps.
  const int64_t rounds = (R + 2 * groups - 1) / (2 * groups);
  for (int64_t q0 = 0; q0 < rounds; ++q0) {
    const int64_t r = g0 + q0 * 2 * groups;
    const bool one = r < R, two = r + groups < R;
    const float4* a = reinterpret_cast<const float4*>(X + (one ? r : 0) * N3);
    const float4* b = reinterpret_cast<const float4*>(X + (two ? r + groups : 0) * N3);
    float ma = 0.f, mb = 0.f;
#pragma unroll 4
    for (int v = lane; v < nv; v += lw) {
      const float4 p = a[v], q = b[v];
      ma = fmaxf(ma, fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fmaxf(fabsf(p.z), fabsf(p.w))));
      mb = fmaxf(mb, fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)), fmaxf(fabsf(q.z), fabsf(q.w))));
    }
    for (int o = lw >> 1; o > 0; o >>= 1) {
      ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
      mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    }
    if (lane == 0) {
      if (one) rmax[r] = __float_as_uint(ma);
      if (two) rmax[r + groups] = __float_as_uint(mb);
    }
  }
}

// s_i for mode-1 slice i: 2^e with 2^14 <= max 2^-e < 2^15, e >= kF16MinS so that
// s_i t_j u_k stays a normal float.
constexpr int kF16MinS = -96, kF16MinT = -15;
__global__ void __launch_bounds__(256)
slice_s_kernel(const unsigned* __restrict__ rmax, int64_t N2, float* __restrict__ s) {
  __shared__ unsigned m;
  if (threadIdx.x == 0) m = 0u;
  __syncthreads();
  unsigned v = 0u;
  for (int64_t j = threadIdx.x; j < N2; j += blockDim.x) {
    const unsigned x = rmax[(int64_t)blockIdx.x * N2 + j];
    v = x > v ? x : v;
  }
  atomicMax(&m, __reduce_max_sync(0xffffffffu, v));
  __syncthreads();
  if (threadIdx.x == 0) {
    const int e = f16_exponent(m);
    s[blockIdx.x] = pow2f(m == 0u ? 0 : (e < kF16MinS ? kF16MinS : e));
  }
}

// The power of two t in [2^kF16MinT, 1] that brings a slice whose largest scaled entry
// is max < 2^15 to 2^14 or more (1 for a slice of zeros).
__device__ __forceinline__ float slice_t(float mx) {
  if (!(mx > 0.f)) return 1.f;
  const int e = f16_exponent(__float_as_uint(mx));
  return pow2f(e > 0 ? 0 : (e < kF16MinT ? kF16MinT : e));
}

__global__ void __launch_bounds__(256)
slice_t_kernel(const unsigned* __restrict__ rmax, const float* __restrict__ s, int64_t N1,
               int64_t N2, float* __restrict__ t) {
  const int64_t j = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
  __shared__ float part[8][32];
  float m = 0.f;
  if (j < N2)
    for (int64_t i = threadIdx.x >> 5; i < N1; i += 8)
      m = fmaxf(m, __uint_as_float(rmax[i * N2 + j]) * (1.f / s[i]));
  part[threadIdx.x >> 5][threadIdx.x & 31] = m;
  __syncthreads();
  if (threadIdx.x < 32 && j < N2) {
    for (int w = 1; w < 8; ++w) m = fmaxf(m, part[w][threadIdx.x]);
    t[j] = slice_t(m);
  }
}

// umax[k] = bits of max over the rows (i, j) of |X| / (s_i t_j): a block takes
// 4 tx columns k (tx a power of two, at most 64, so that short rows use every
// thread too) and every gridDim.x-th group of 256 / tx rows.
__global__ void __launch_bounds__(256)
col_max_kernel(const float* __restrict__ X, int64_t R, int N2, int N3, int tx,
               const float* __restrict__ s, const float* __restrict__ t,
               unsigned* __restrict__ umax) {
  const int k = 4 * (blockIdx.y * tx + (threadIdx.x & (tx - 1)));
  const int ty = 256 / tx, sub = threadIdx.x / tx;
  float m[4] = {0.f, 0.f, 0.f, 0.f};
  if (k < N3) {
#pragma unroll 4
    for (int64_t r = (int64_t)blockIdx.x * ty + sub; r < R; r += (int64_t)ty * gridDim.x) {
      const unsigned i = (unsigned)r / (unsigned)N2;  // R <= 2^31
      const float inv = (1.f / s[i]) * (1.f / t[(unsigned)r - i * (unsigned)N2]);
      const float4 x = *reinterpret_cast<const float4*>(X + r * N3 + k);
      m[0] = fmaxf(m[0], fabsf(x.x) * inv);
      m[1] = fmaxf(m[1], fabsf(x.y) * inv);
      m[2] = fmaxf(m[2], fabsf(x.z) * inv);
      m[3] = fmaxf(m[3], fabsf(x.w) * inv);
    }
  }
  __shared__ float part[1024];  // [row group][4 tx]
#pragma unroll
  for (int c = 0; c < 4; ++c) part[threadIdx.x * 4 + c] = m[c];
  __syncthreads();
  const int col = blockIdx.y * 4 * tx + threadIdx.x;
  if (threadIdx.x < 4 * tx && col < N3) {
    float v = part[threadIdx.x];
    for (int q = 1; q < ty; ++q) v = fmaxf(v, part[q * 4 * tx + threadIdx.x]);
    if (v > 0.f) atomicMax(&umax[col], __float_as_uint(v));
  }
}

__global__ void slice_u_kernel(const unsigned* __restrict__ umax, int N3, int n3p,
                               float* __restrict__ u) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n3p) u[k] = k < N3 ? slice_t(__uint_as_float(umax[k])) : 1.f;
}

// Xh, Xl (rows of n3p entries, zero past N3) from X: eight entries a thread, tx threads
// (a power of two) a row, one division per row. *wide gets 1 when a nonzero entry lies below
// kF16LeastX.
__global__ void __launch_bounds__(256)
x_to_pair_kernel(const float* __restrict__ X, int64_t R, int N2, int N3, int n3p, int tx,
                 const float* __restrict__ s, const float* __restrict__ t,
                 const float* __restrict__ u, __half* __restrict__ Xh, __half* __restrict__ Xl,
                 int* __restrict__ wide) {
  const int oct = n3p >> 3, ty = 256 / tx;
  bool low = false;
  for (int64_t r = (int64_t)blockIdx.x * ty + threadIdx.x / tx; r < R;
       r += (int64_t)gridDim.x * ty) {
    const unsigned i = (unsigned)r / (unsigned)N2;  // R <= 2^31
    const float inv = (1.f / s[i]) * (1.f / t[(unsigned)r - i * (unsigned)N2]);
#pragma unroll 2
    for (int o = threadIdx.x & (tx - 1); o < oct; o += tx) {
      const int k = 8 * o;
      const float* x = X + r * N3 + k;
      float v[8];
      // N3 % 4 == 0: the first four entries exist, the last four all or none.
      const float4 a = *reinterpret_cast<const float4*>(x);
      const float4 b = k + 4 < N3 ? *reinterpret_cast<const float4*>(x + 4)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
      v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
      union { __half h[8]; uint4 q; } hi, lo;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float y = v[q] * inv * (1.f / u[k + q]);
        low |= v[q] != 0.f && fabsf(y) < kF16LeastX;
        split_f16(y, hi.h[q], lo.h[q]);
      }
      *reinterpret_cast<uint4*>(Xh + r * n3p + k) = hi.q;
      *reinterpret_cast<uint4*>(Xl + r * n3p + k) = lo.q;
    }
  }
  if (low) *wide = 1;
}

// ---- conversions -------------------------------------------------------------

// s_i = 2^e with max_{j,k} X[i, j, k] = f 2^e, f in [0.5, 1); 1 for an all-zero slice.
__global__ void slice_scale_kernel(const float* __restrict__ X, int64_t slab, float* scale,
                                   float* inv_scale) {
  __shared__ float red[32];
  float mx = 0.f;
  const float* x = X + static_cast<int64_t>(blockIdx.x) * slab;
  for (int64_t e = threadIdx.x; e < slab; e += blockDim.x) mx = fmaxf(mx, fabsf(x[e]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x < 32) {
    mx = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (threadIdx.x == 0) {
      int e = 0;
      if (mx > 0.f && isfinite(mx)) frexpf(mx, &e);
      scale[blockIdx.x] = ldexpf(1.f, e);
      inv_scale[blockIdx.x] = ldexpf(1.f, -e);
    }
  }
}

// The same scales from the rows' maxima.
__global__ void __launch_bounds__(256)
slice_scale_rows_kernel(const unsigned* __restrict__ rmax, int64_t N2, float* scale,
                        float* inv_scale) {
  __shared__ unsigned m;
  if (threadIdx.x == 0) m = 0u;
  __syncthreads();
  unsigned v = 0u;
  for (int64_t j = threadIdx.x; j < N2; j += blockDim.x) {
    const unsigned x = rmax[(int64_t)blockIdx.x * N2 + j];
    v = x > v ? x : v;
  }
  atomicMax(&m, __reduce_max_sync(0xffffffffu, v));
  __syncthreads();
  if (threadIdx.x == 0) {
    const float mx = __uint_as_float(m);
    int e = 0;
    if (mx > 0.f && isfinite(mx)) frexpf(mx, &e);
    scale[blockIdx.x] = ldexpf(1.f, e);
    inv_scale[blockIdx.x] = ldexpf(1.f, -e);
  }
}

// Xb (rows of kp entries, a multiple of 64, zero past n3) from X: eight entries a
// thread, tx threads (a power of two) a row. 512^3: 358 -> 128 us (one entry a thread,
// two divisions an entry).
template <bool VEC>
__global__ void __launch_bounds__(256)
x_to_bf16_kernel(const float* __restrict__ X, int64_t rows, int n3, int kp, int rows_per_slice,
                 int tx, const float* __restrict__ inv_scale, __nv_bfloat16* __restrict__ Xb) {
  const int oct = kp >> 3, ty = 256 / tx;
  for (int64_t r = (int64_t)blockIdx.x * ty + threadIdx.x / tx; r < rows;
       r += (int64_t)gridDim.x * ty) {
    const float inv = inv_scale[(unsigned)r / (unsigned)rows_per_slice];  // rows <= 2^31
#pragma unroll 2
    for (int o = threadIdx.x & (tx - 1); o < oct; o += tx) {
      const int k = 8 * o;
      const float* x = X + r * n3 + k;
      float v[8];
      if constexpr (VEC) {  // n3 % 4 == 0, rows on 16 bytes
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 a = k < n3 ? *reinterpret_cast<const float4*>(x) : z;
        const float4 b = k + 4 < n3 ? *reinterpret_cast<const float4*>(x + 4) : z;
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = k + q < n3 ? x[q] : 0.f;
      }
      union { __nv_bfloat16 h[8]; uint4 q; } out;
#pragma unroll
      for (int q = 0; q < 8; ++q) out.h[q] = __float2bfloat16_rn(v[q] * inv);
      *reinterpret_cast<uint4*>(Xb + r * kp + k) = out.q;
    }
  }
}

// B operands of a factor F (n x m): Bt[q, k] = F[k, q] * (scale ? scale[k] : 1)
// as BF16 (bt16), or as the TF32 pair (bhi, blo); zero outside q < m, k < n.
__global__ void factor_b_kernel(const float* __restrict__ F, int n, int m, int kpad, int np,
                                const float* __restrict__ scale, __nv_bfloat16* __restrict__ bt16,
                                float* __restrict__ bhi, float* __restrict__ blo) {
  const int64_t tot = static_cast<int64_t>(np) * kpad;
  for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < tot;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int q = static_cast<int>(e / kpad), k = static_cast<int>(e % kpad);
    float v = 0.f;
    if (q < m && k < n) v = F[static_cast<int64_t>(k) * m + q] * (scale ? scale[k] : 1.f);
    if (bt16) bt16[e] = __float2bfloat16_rn(v);
    if (bhi) {
      const float h = tf32_hi(v);
      bhi[e] = h;
      blo[e] = tf32_lo(v, h);
    }
  }
}

// Xt[c, i] = X[i, c] (X viewed N1 x C, Xt row length ldt >= N1, zero padded).
__global__ void transpose_kernel(const float* __restrict__ X, int64_t N1, int64_t C, int64_t ldt,
                                 float* __restrict__ Xt) {
  __shared__ float tile[32][33];
  const int64_t c0 = static_cast<int64_t>(blockIdx.x) * 32, i0 = static_cast<int64_t>(blockIdx.y) * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int64_t i = i0 + r, c = c0 + threadIdx.x;
    tile[r][threadIdx.x] = (i < N1 && c < C) ? X[i * C + c] : 0.f;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int64_t c = c0 + r, i = i0 + threadIdx.x;
    if (c < C && i < ldt) Xt[c * ldt + i] = tile[threadIdx.x][r];
  }
}

// Xt[(k N2 + j) ldt + i] = X[i, j, k] (Xt rows (k, j), row length ldt >= N1,
// zero padded); block (k tile, i tile) of 32 x 32, looping over j.
__global__ void transpose_kj_kernel(const float* __restrict__ X, int64_t N1, int64_t N2,
                                    int64_t N3, int64_t ldt, float* __restrict__ Xt) {
  __shared__ float tile[32][33];
  const int64_t k0 = static_cast<int64_t>(blockIdx.x) * 32, i0 = static_cast<int64_t>(blockIdx.y) * 32;
  for (int64_t j = blockIdx.z; j < N2; j += gridDim.z) {
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
      const int64_t i = i0 + r, k = k0 + threadIdx.x;
      tile[r][threadIdx.x] = (i < N1 && k < N3) ? X[(i * N2 + j) * N3 + k] : 0.f;
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
      const int64_t k = k0 + r, i = i0 + threadIdx.x;
      if (k < N3 && i < ldt) Xt[(k * N2 + j) * ldt + i] = tile[threadIdx.x][r];
    }
    __syncthreads();
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

int make_map(CUtensorMap* tm, CUtensorMapDataType dt, const void* base, uint64_t inner,
             uint64_t outer, uint64_t row_bytes, uint32_t box_inner, uint32_t box_outer) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (enc == nullptr) {
    set_error_detail_text("cuTensorMapEncodeTiled is not available from the driver");
    return NNC_ERR_CUDA;
  }
  const cuuint64_t dims[2] = {inner, outer};
  const cuuint64_t strides[1] = {row_bytes};
  const cuuint32_t box[2] = {box_inner, box_outer};
  const cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(tm, dt, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    char buf[160];
    snprintf(buf, sizeof(buf), "cuTensorMapEncodeTiled failed (%d): dims %llu x %llu, box %u x %u",
             static_cast<int>(r), (unsigned long long)inner, (unsigned long long)outer, box_inner,
             box_outer);
    set_error_detail_text(buf);
    return NNC_ERR_CUDA;
  }
  return NNC_OK;
}

// Fewest CTAs that keep the largest tile count per CTA of a grid over the
// SMs the pass may take: the time is the same, and the SMs left over run
// the small kernels of the sweep that the graph places beside the pass.
// With at least min_tiles tiles per SM the pass leaves `reserve` SMs to them. With y_nh
// tiles per slab (a fused pass) a grid that is a multiple of them gives every
// CTA tiles of one j range only, so it loads its factor rows once per pass.
int64_t pass_grid(int64_t tiles, int reserve, int64_t y_nh, int min_tiles) {
  const int sms = device_sm_count();
  const int avail = (tiles >= (int64_t)min_tiles * sms && reserve > 0 && reserve < sms / 2) ? sms - reserve : sms;
  const int64_t per = ceil_div(tiles, (int64_t)avail);
  int64_t grid = ceil_div(tiles, per);
  if (y_nh > 1) {
    const int64_t up = ceil_div(grid, y_nh) * y_nh;
    if (up <= avail) grid = up;
    else if (avail >= y_nh) grid = avail / y_nh * y_nh;
  }
  return grid;
}

template <int KIND, bool kMN, int NP, bool FUSE>
int launch_pass(const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& blo, int nk,
                int64_t tiles, const TcEpilogue& ep, int* err, int reserve, cudaStream_t s) {
  constexpr int smem = TcLayout<KIND, NP, FUSE>::kSmem;
  NNC_CUDA_TRY(raise_smem_limit((const void*)tc_pass_kernel<KIND, kMN, NP, FUSE>, smem));
  const int64_t grid = pass_grid(tiles, reserve, FUSE ? ep.y_nh : 1, /*min_tiles=*/8);
  NNC_CUDA_TRY(launch_pdl(tc_pass_kernel<KIND, kMN, NP, FUSE>, dim3(static_cast<unsigned>(grid)),
                          dim3(kThreadsTc), smem, s, a, b, blo, nk, tiles, ep, err));
  note_launch(s);
  return NNC_OK;
}

template <bool kMN, int NP, bool FUSE>
int launch_f16(const CUtensorMap& hi, const CUtensorMap& lo, const F16Operand& fo, int nk,
               int64_t tiles, const TcEpilogue& ep, int* err, int reserve, cudaStream_t s) {
  const int smem = f16_smem<NP, FUSE>(nk);
  NNC_CUDA_TRY(raise_smem_limit((const void*)f16_pass_kernel<kMN, NP, FUSE>, smem));
  const int64_t grid = pass_grid(tiles, reserve, FUSE ? ep.y_nh : 1, /*min_tiles=*/1);
  NNC_CUDA_TRY(launch_pdl(f16_pass_kernel<kMN, NP, FUSE>, dim3(static_cast<unsigned>(grid)),
                          dim3(kThreadsTc), smem, s, hi, lo, fo, nk, tiles, ep, err));
  note_launch(s);
  return NNC_OK;
}

template <int KIND, bool kMN>
int launch_np(int np, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& blo, int nk,
              int64_t tiles, const TcEpilogue& ep, int* err, int reserve, cudaStream_t s) {
  if constexpr (!kMN) {
    if (ep.ysh)
      return launch_pass<KIND, kMN, 32, true>(a, b, blo, nk, tiles, ep, err, reserve, s);
  }
  if (np == 32) return launch_pass<KIND, kMN, 32, false>(a, b, blo, nk, tiles, ep, err, reserve, s);
  return launch_pass<KIND, kMN, 64, false>(a, b, blo, nk, tiles, ep, err, reserve, s);
}

}  // namespace

// Threads (a power of two, at most 256) that share a row of n pieces.
static int row_threads(int n) {
  int t = 1;
  while (t < 256 && t < n) t *= 2;
  return t;
}

// rmax: the largest magnitude of every row (i, j) of X (rows on 16 bytes).
int TcPlan::row_maxima(const float* X, Scratch& sc, cudaStream_t s) {
  const int64_t rows = N1 * N2;
  NNC_TRY(sc.get(&rmax, static_cast<size_t>(rows)));
  int lw = 1;
  while (lw < 32 && lw < N3 / 4) lw *= 2;
  const int64_t rb = ceil_div(rows, 2 * (256 / lw)), most = 16LL * device_sm_count();
  row_max_kernel<<<(unsigned)(rb < most ? rb : most), 256, 0, s>>>(X, rows, (int)N3, lw, rmax);
  note_launch(s);
  NNC_CUDA_TRY(cudaGetLastError());
  return NNC_OK;
}

int TcPlan::init(int kind_, const float* X, int64_t N1_, int64_t N2_, int64_t N3_, int m1_,
                 int m3_, Scratch& sc, cudaStream_t s, bool p1_kj_, bool need_p1) {
  kind = kind_;
  p1_kj = p1_kj_;
  N1 = N1_;
  N2 = N2_;
  N3 = N3_;
  m1 = m1_;
  m3 = m3_;
  np1 = m1 <= 32 ? 32 : 64;
  np3 = m3 <= 32 ? 32 : 64;
  const int kstage = kind == kKindTf32x3 ? 32 : 64;
  // K of pass 1 is N3 (BF16: padded rows of Xb), K of pass 2 is N1.
  kp3 = kind == kKindBf16 ? static_cast<int>(ceil_div(N3, 64) * 64)
        : kind == kKindF16x3 ? static_cast<int>(ceil_div(N3, 8) * 8)
                             : static_cast<int>(N3);
  kb3 = static_cast<int>(ceil_div(N3, kstage) * kstage);
  kp1 = static_cast<int>(ceil_div(N1, kstage) * kstage);
  if (m1 > 64 || m3 > 64 || N1 * N2 > (1LL << 31) || N2 * kp3 > (1LL << 31)) {
    set_error_detail_text("tensor-core pass: shape outside the path (m <= 64)");
    return NNC_ERR_UNSUPPORTED;
  }
  if (kind == kKindF16x3) return init_f16(X, sc, s);
  if (kind == kKindTf32x3 && (N3 % 4) != 0) {
    set_error_detail_text("tensor-core TF32 pass: N3 must be a multiple of 4");
    return NNC_ERR_UNSUPPORTED;
  }
  const int64_t rows = N1 * N2;
  NNC_TRY(sc.get(&err, 1));
  NNC_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), s));
  NNC_TRY(sc.get(&scale, static_cast<size_t>(N1)));
  NNC_TRY(sc.get(&inv_scale, static_cast<size_t>(N1)));
  if (kind == kKindBf16) {
    NNC_TRY(sc.get(&Xb, static_cast<size_t>(rows * kp3)));
    NNC_TRY(sc.get(&Bt1, static_cast<size_t>(np1) * kp1));
    NNC_TRY(sc.get(&Bt3, static_cast<size_t>(np3) * kb3));
    NNC_CUDA_TRY(cudaMemsetAsync(Bt1, 0, sizeof(__nv_bfloat16) * np1 * kp1, s));
    NNC_CUDA_TRY(cudaMemsetAsync(Bt3, 0, sizeof(__nv_bfloat16) * np3 * kb3, s));
    const bool vec = N3 % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    if (vec) {
      NNC_TRY(row_maxima(X, sc, s));
      slice_scale_rows_kernel<<<static_cast<unsigned>(N1), 256, 0, s>>>(rmax, N2, scale,
                                                                        inv_scale);
    } else {
      slice_scale_kernel<<<static_cast<unsigned>(N1), 256, 0, s>>>(X, N2 * N3, scale, inv_scale);
    }
    note_launch(s);
    const int ox = row_threads(kp3 / 8);
    const int64_t xb = ceil_div(rows, 256 / ox), most = 32LL * device_sm_count();
    const unsigned blocks = static_cast<unsigned>(xb < most ? xb : most);
    if (vec)
      x_to_bf16_kernel<true><<<blocks, 256, 0, s>>>(X, rows, static_cast<int>(N3), kp3,
                                                    static_cast<int>(N2), ox, inv_scale, Xb);
    else
      x_to_bf16_kernel<false><<<blocks, 256, 0, s>>>(X, rows, static_cast<int>(N3), kp3,
                                                     static_cast<int>(N2), ox, inv_scale, Xb);
    note_launch(s);
    NNC_CUDA_TRY(cudaGetLastError());
    const CUtensorMapDataType bf = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    NNC_TRY(make_map(&mapA3, bf, Xb, kp3, rows, static_cast<uint64_t>(kp3) * 2, 64, 128));
    NNC_TRY(make_map(&mapB3, bf, Bt3, kb3, np3, static_cast<uint64_t>(kb3) * 2, 64, np3));
    NNC_TRY(make_map(&mapA1, bf, Xb, static_cast<uint64_t>(N2) * kp3, N1,
                     static_cast<uint64_t>(N2) * kp3 * 2, 64, 64));
    NNC_TRY(make_map(&mapB1, bf, Bt1, kp1, np1, static_cast<uint64_t>(kp1) * 2, 64, np1));
    mapB3lo = mapB3;
    mapB1lo = mapB1;
  } else {
    NNC_TRY(sc.get(&B1hi, static_cast<size_t>(np1) * kp1));
    NNC_TRY(sc.get(&B1lo, static_cast<size_t>(np1) * kp1));
    NNC_TRY(sc.get(&B3hi, static_cast<size_t>(np3) * kb3));
    NNC_TRY(sc.get(&B3lo, static_cast<size_t>(np3) * kb3));
    NNC_CUDA_TRY(cudaMemsetAsync(B1hi, 0, sizeof(float) * np1 * kp1, s));
    NNC_CUDA_TRY(cudaMemsetAsync(B1lo, 0, sizeof(float) * np1 * kp1, s));
    NNC_CUDA_TRY(cudaMemsetAsync(B3hi, 0, sizeof(float) * np3 * kb3, s));
    NNC_CUDA_TRY(cudaMemsetAsync(B3lo, 0, sizeof(float) * np3 * kb3, s));
    scale = nullptr;
    const CUtensorMapDataType f32 = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    NNC_TRY(make_map(&mapA3, f32, X, N3, rows, static_cast<uint64_t>(N3) * 4, 32, 128));
    NNC_TRY(make_map(&mapB3, f32, B3hi, kb3, np3, static_cast<uint64_t>(kb3) * 4, 32, np3));
    NNC_TRY(make_map(&mapB3lo, f32, B3lo, kb3, np3, static_cast<uint64_t>(kb3) * 4, 32, np3));
    if (!need_p1) return NNC_OK;
    // Pass 2 reads Xt = X viewed (N1 x N2 N3), transposed: K-major rows of N1p
    // in the order (j, k), or (k, j) for p1_kj.
    const int64_t C = N2 * N3, n1p = ceil_div(N1, 4) * 4;
    NNC_TRY(sc.get(&Xt, static_cast<size_t>(C * n1p)));
    if (p1_kj) {
      dim3 tgrid(static_cast<unsigned>(ceil_div(N3, 32)), static_cast<unsigned>(ceil_div(n1p, 32)),
                 static_cast<unsigned>(N2 < 65535 ? N2 : 65535));
      transpose_kj_kernel<<<tgrid, dim3(32, 8), 0, s>>>(X, N1, N2, N3, n1p, Xt);
    } else {
      dim3 tgrid(static_cast<unsigned>(ceil_div(C, 32)), static_cast<unsigned>(ceil_div(n1p, 32)));
      transpose_kernel<<<tgrid, dim3(32, 8), 0, s>>>(X, N1, C, n1p, Xt);
    }
    note_launch(s);
    NNC_CUDA_TRY(cudaGetLastError());
    NNC_TRY(make_map(&mapA1, f32, Xt, n1p, C, static_cast<uint64_t>(n1p) * 4, 32, 128));
    NNC_TRY(make_map(&mapB1, f32, B1hi, kp1, np1, static_cast<uint64_t>(kp1) * 4, 32, np1));
    NNC_TRY(make_map(&mapB1lo, f32, B1lo, kp1, np1, static_cast<uint64_t>(kp1) * 4, 32, np1));
  }
  return NNC_OK;
}

// The shapes the FP16 pair passes take: rows of X on 16 bytes, and both passes'
// operands (K x m, split, in shared memory for the whole pass) beside three
// stages at least: N3 up to 768 for m3 <= 32 (room for the fused contraction's tiles is
// kept), N1 up to 1024 for m1 <= 32, 512 each for m <= 64.
int TcPlan::init_f16(const float* X, Scratch& sc, cudaStream_t s) {
  const int64_t rows = N1 * N2;
  const int nk3 = kb3 / 64, nk1 = kp1 / 64;
  const int st3 = np3 == 32 ? f16_stages<32, true>(nk3) : f16_stages<64, false>(nk3);
  const int st1 = np1 == 32 ? f16_stages<32, false>(nk1) : f16_stages<64, false>(nk1);
  if (N3 % 4 != 0 || (reinterpret_cast<uintptr_t>(X) & 15) != 0 || st3 < kF16MinStages ||
      st1 < kF16MinStages || N2 > (1LL << 30)) {
    set_error_detail_text("FP16 pair pass: shape outside the path");
    return NNC_ERR_UNSUPPORTED;
  }
  unsigned* umax = nullptr;
  NNC_TRY(sc.get(&err, kFlags));
  NNC_TRY(sc.get(&scale, static_cast<size_t>(N1)));
  NNC_TRY(sc.get(&sc_t, static_cast<size_t>(N2)));
  NNC_TRY(sc.get(&sc_u, static_cast<size_t>(kp3)));
  NNC_TRY(sc.get(&umax, static_cast<size_t>(N3)));
  // One block, so that Xt fits where the pair was when the plan becomes TF32x3.
  const int64_t half = ceil_div(rows * kp3, 64) * 64;
  NNC_TRY(sc.get(&Xh, static_cast<size_t>(2 * half)));
  Xl = Xh + half;
  const int sms = device_sm_count();
  NNC_CUDA_TRY(cudaMemsetAsync(err, 0, kFlags * sizeof(int), s));
  if (rmax == nullptr) NNC_TRY(row_maxima(X, sc, s));
  slice_s_kernel<<<(unsigned)N1, 256, 0, s>>>(rmax, N2, scale);
  note_launch(s);
  slice_t_kernel<<<(unsigned)ceil_div(N2, 32), 256, 0, s>>>(rmax, scale, N1, N2, sc_t);
  note_launch(s);
  NNC_CUDA_TRY(cudaMemsetAsync(umax, 0, sizeof(unsigned) * N3, s));
  int tx = 1;
  while (tx < 64 && 4 * tx < N3) tx *= 2;
  const int64_t ky = ceil_div(N3, 4 * tx);
  const int64_t cb = ceil_div(rows, 4 * (256 / tx));
  const int64_t cx = ceil_div(8LL * sms, ky);
  col_max_kernel<<<dim3((unsigned)(cb < cx ? cb : cx), (unsigned)ky), 256, 0, s>>>(
      X, rows, (int)N2, (int)N3, tx, scale, sc_t, umax);
  note_launch(s);
  slice_u_kernel<<<(unsigned)ceil_div(kp3, 256), 256, 0, s>>>(umax, (int)N3, kp3, sc_u);
  note_launch(s);
  const int ox = row_threads(kp3 / 8);
  const int64_t xb = ceil_div(rows, 256 / ox);
  x_to_pair_kernel<<<(unsigned)(xb < 32LL * sms ? xb : 32LL * sms), 256, 0, s>>>(
      X, rows, (int)N2, (int)N3, kp3, ox, scale, sc_t, sc_u, Xh, Xl, err + kFlagWideX);
  note_launch(s);
  NNC_CUDA_TRY(cudaGetLastError());
  // A pass launched as a programmatic dependent reads the pair before it waits for its
  // predecessor, so that must not be the conversion: the error flag once more.
  NNC_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), s));
  // The pair stays in L2 (129 MB) from pass to pass with room for the pass results.
  x_resident = 4 * rows * kp3 <= 80LL << 20;
  const CUtensorMapDataType h = CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  const uint64_t ld = static_cast<uint64_t>(kp3) * 2, ldw = static_cast<uint64_t>(N2) * kp3 * 2;
  NNC_TRY(make_map(&mapA3, h, Xh, kp3, rows, ld, 64, 128));
  NNC_TRY(make_map(&mapL3, h, Xl, kp3, rows, ld, 64, 128));
  NNC_TRY(make_map(&mapA1, h, Xh, static_cast<uint64_t>(N2) * kp3, N1, ldw, 64, 64));
  NNC_TRY(make_map(&mapL1, h, Xl, static_cast<uint64_t>(N2) * kp3, N1, ldw, 64, 64));
  return NNC_OK;
}

int TcPlan::init_fp32(const float* X, int64_t N1_, int64_t N2_, int64_t N3_, int m1_, int m3_,
                      Scratch& sc, cudaStream_t s, bool p1_kj_) {
  const int st = init(kKindF16x3, X, N1_, N2_, N3_, m1_, m3_, sc, s, p1_kj_);
  if (st != NNC_ERR_UNSUPPORTED) return st;
  return init(kKindTf32x3, X, N1_, N2_, N3_, m1_, m3_, sc, s, p1_kj_);
}

int TcPlan::to_tf32(const float* X, Scratch& sc, cudaStream_t s) {
  sc.drop(Xh);
  Xh = Xl = nullptr;
  reserve_sms = 0;
  return init(kKindTf32x3, X, N1, N2, N3, m1, m3, sc, s, p1_kj);
}

int TcPlan::convert_b3(const float* F3, cudaStream_t s) const {
  if (kind == kKindF16x3) return NNC_OK;  // the pass forms its operand
  factor_b_kernel<<<64, 256, 0, s>>>(F3, static_cast<int>(N3), m3, kb3, np3, nullptr, Bt3, B3hi,
                                     B3lo);
  note_launch(s);
  NNC_CUDA_TRY(cudaGetLastError());
  return NNC_OK;
}

int TcPlan::convert_b1(const float* F1, cudaStream_t s) const {
  if (kind == kKindF16x3) return NNC_OK;
  factor_b_kernel<<<64, 256, 0, s>>>(F1, static_cast<int>(N1), m1, kp1, np1,
                                     kind == kKindBf16 ? scale : nullptr, Bt1, B1hi, B1lo);
  note_launch(s);
  NNC_CUDA_TRY(cudaGetLastError());
  return NNC_OK;
}

bool TcPlan::y1_fusable(int m2) const {
  // Tiles of pass 1 are single (i, j0 .. j0 + 127) row blocks when N2 % 128
  // == 0; the tile contraction runs on the tensor cores, which keeps it off
  // the BF16 pass's stage rate too.
  return np3 == 32 && m2 >= 1 && m2 <= 32 && N2 % 128 == 0;
}

bool TcPlan::y3_fusable(int m2) const {
  // Tiles of pass 2 are single (k, j0 .. j0 + 127) row blocks only when read
  // from the (k, j)-ordered Xt.
  return kind == kKindTf32x3 && p1_kj && np1 == 32 && m2 >= 1 && m2 <= 32 && N2 % 128 == 0;
}

int TcPlan::pass3(const float* F3, float* P3, cudaStream_t s, bool convert, const float* F2,
                  int m2, float* Y1) const {
  if (convert) NNC_TRY(convert_b3(F3, s));
  TcEpilogue ep{};
  ep.out = P3;
  ep.q = m3;
  ep.rows = N1 * N2;
  ep.rows_per_slice = N2;
  ep.row_scale = kind == kKindBf16 ? scale : nullptr;
  if (Y1) {
    if (!F2 || !y1_fusable(m2)) return NNC_ERR_UNSUPPORTED;
    ep.ysh = Y1;
    ep.yf = F2;
    ep.yf_m = m2;
    ep.y_nh = N2 / 128;
  }
  const int64_t tiles = ceil_div(N1 * N2, 128);
  if (kind == kKindF16x3) {
    ep.kp = N2;  // tile row (i, j)
    ep.ra_scale = scale;
    ep.ra_n = N1;
    ep.rb_scale = sc_t;
    ep.rb_n = N2;
    ep.x_resident = x_resident;
    const F16Operand fo{F3, sc_u, static_cast<int>(N3), m3};
    const int nkf = kb3 / 64, rsv = reserve_sms;
    if (ep.ysh) return launch_f16<false, 32, true>(mapA3, mapL3, fo, nkf, tiles, ep, err, rsv, s);
    if (np3 == 32) return launch_f16<false, 32, false>(mapA3, mapL3, fo, nkf, tiles, ep, err, rsv, s);
    return launch_f16<false, 64, false>(mapA3, mapL3, fo, nkf, tiles, ep, err, rsv, s);
  }
  const int stagek = kind == kKindBf16 ? 64 : 32;
  const int nk = static_cast<int>(ceil_div(N3, stagek));
  if (kind == kKindBf16)
    return launch_np<kKindBf16, false>(np3, mapA3, mapB3, mapB3lo, nk, tiles, ep, err,
                                       reserve_sms, s);
  return launch_np<kKindTf32x3, false>(np3, mapA3, mapB3, mapB3lo, nk, tiles, ep, err,
                                       reserve_sms, s);
}

int TcPlan::pass1(const float* F1, float* P1, cudaStream_t s, bool convert, const float* F2,
                  int m2, float* Y3) const {
  if (convert) NNC_TRY(convert_b1(F1, s));
  TcEpilogue ep{};
  ep.out = P1;
  ep.q = m1;
  ep.kp = kp3;
  ep.n2 = N2;
  ep.n3 = N3;
  ep.slab = N2 * N3;
  if (!p1_kj) {
    ep.p1_layout = 1;
  } else if (kind != kKindTf32x3) {
    ep.p1_layout = 2;  // MN-major tiles of Xb (Xh, Xl) have rows (j, k)
  } else {
    ep.p1_layout = 0;  // Xt already has rows (k, j)
    ep.rows = N2 * N3;
  }
  if (Y3) {
    if (!F2 || !y3_fusable(m2)) return NNC_ERR_UNSUPPORTED;
    ep.ysh = Y3;
    ep.yf = F2;
    ep.yf_m = m2;
    ep.y_tr = 1;  // Y3[k] is stored m1 x m2
    ep.y_nh = N2 / 128;
  }
  const int64_t tiles = ceil_div(N2 * kp3, 128);
  if (kind == kKindF16x3) {
    ep.ra_scale = sc_t;  // tile row (j, k)
    ep.ra_n = N2;
    ep.rb_scale = sc_u;
    ep.rb_n = N3;
    ep.x_resident = x_resident;
    const F16Operand fo{F1, scale, static_cast<int>(N1), m1};
    const int nkf = kp1 / 64, rsv = reserve_sms;
    if (np1 == 32) return launch_f16<true, 32, false>(mapA1, mapL1, fo, nkf, tiles, ep, err, rsv, s);
    return launch_f16<true, 64, false>(mapA1, mapL1, fo, nkf, tiles, ep, err, rsv, s);
  }
  const int stagek = kind == kKindBf16 ? 64 : 32;
  const int nk = static_cast<int>(ceil_div(N1, stagek));
  if (kind == kKindBf16)
    return launch_np<kKindBf16, true>(np1, mapA1, mapB1, mapB1lo, nk, tiles, ep, err,
                                      reserve_sms, s);
  return launch_np<kKindTf32x3, false>(np1, mapA1, mapB1, mapB1lo, nk, tiles, ep, err,
                                       reserve_sms, s);
}

// Self-test of the bounded waits: one CTA waits, with a limit of `cycles`, on
// the first phase of an mbarrier that expects one arrival and gets none (no
// copy or MMA is in flight). The wait must give up and flag the failure the
// way the pass kernel's roles do; status[0] = 1 then, 0 if the wait returned.
__global__ void wait_selftest_kernel(long long cycles, int* status) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int fail;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const bool got = mbar_wait(&bar, 0, &fail, cycles);
  __syncthreads();
  if (threadIdx.x == 0) status[0] = (got && !fail) ? 0 : 1;
}

int wait_selftest(long long cycles, cudaStream_t s) {
  if (cycles < 0) return NNC_ERR_INVALID_ARG;
  Scratch sc(s);
  int* d = nullptr;
  NNC_TRY(sc.get(&d, 1));
  NNC_CUDA_TRY(cudaMemsetAsync(d, 0, sizeof(int), s));
  wait_selftest_kernel<<<1, 32, 0, s>>>(cycles, d);
  note_launch(s);
  NNC_CUDA_TRY(cudaGetLastError());
  int h = 0;
  NNC_CUDA_TRY(cudaMemcpyAsync(&h, d, sizeof(int), cudaMemcpyDeviceToHost, s));
  NNC_CUDA_TRY(cudaStreamSynchronize(s));
  if (h != 0) {
    set_error_detail_text("self-test: the bounded wait gave up as it should");
    return NNC_ERR_TIMEOUT;
  }
  return NNC_OK;
}

namespace {
int timed_out(int flag) {
  if (flag == 0) return NNC_OK;
  set_error_detail_text("tensor-core mode product: a pipeline wait timed out");
  return NNC_ERR_TIMEOUT;
}
}  // namespace

// Page-locked words for the looks, one slot a fit: a copy to them and a wait for an event take no
// lock that other threads' launches wait for, as a copy to pageable memory does.
namespace {
constexpr int kSlots = 64;
std::mutex g_slot_mu;
int* g_slots = nullptr;  // kSlots x kFlags, allocated by the first fit that looks
bool g_slot_used[kSlots];
int* take_slot() {
  std::lock_guard<std::mutex> lk(g_slot_mu);
  if (g_slots == nullptr) {
    // (relaxed: the allocation must not break a capture of another thread)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    const cudaError_t e = cudaHostAlloc(reinterpret_cast<void**>(&g_slots),
                                        kSlots * kFlags * sizeof(int), cudaHostAllocPortable);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) {
      (void)cudaGetLastError();
      g_slots = nullptr;
      return nullptr;
    }
  }
  for (int k = 0; k < kSlots; ++k)
    if (!g_slot_used[k]) {
      g_slot_used[k] = true;
      return g_slots + k * kFlags;
    }
  return nullptr;
}
void give_slot(int* p) {
  std::lock_guard<std::mutex> lk(g_slot_mu);
  g_slot_used[(p - g_slots) / kFlags] = false;
}
}  // namespace

int PairGuard::start(const TcPlan* p, int first, cudaStream_t s) {
  plan = p;
  next = first;
  slot = take_slot();
  if (slot == nullptr) return NNC_OK;  // more fits at once than slots: this one does not look
  NNC_CUDA_TRY(cudaEventCreateWithFlags(&at, cudaEventDisableTiming));
  NNC_CUDA_TRY(cudaMemcpyAsync(slot, plan->err, kFlags * sizeof(int), cudaMemcpyDeviceToHost, s));
  NNC_CUDA_TRY(cudaEventRecord(at, s));
  pending = true;
  return NNC_OK;
}

int PairGuard::wide(cudaStream_t s, bool* w) {
  if (slot == nullptr) return plan->check(s, w);
  NNC_CUDA_TRY(cudaEventSynchronize(at));
  pending = false;
  *w = slot[kFlagWideX] != 0;
  return NNC_OK;
}

PairGuard::~PairGuard() {
  if (at) {
    // (a copy to the slot may be under way when a call ends early)
    if (pending) cudaEventSynchronize(at);
    cudaEventDestroy(at);
  }
  if (slot) give_slot(slot);
}

int PairGuard::step(cudaStream_t cs, int t) {
  if (slot == nullptr) return NNC_OK;
  if (!pending && t >= next) {
    NNC_CUDA_TRY(cudaMemcpyAsync(slot, plan->err, kFlags * sizeof(int), cudaMemcpyDeviceToHost, cs));
    NNC_CUDA_TRY(cudaEventRecord(at, cs));
    marked = t;
    pending = true;
  } else if (pending && t > marked) {
    NNC_CUDA_TRY(cudaEventSynchronize(at));
    pending = false;
    slow = 4LL * (slot[kFlagRounds] - rounds) > 2LL * (marked - looked);
    rounds = slot[kFlagRounds];
    looked = marked;
    next = t + (t > 80 ? t / 4 : 20);
    return timed_out(slot[0]);
  }
  return NNC_OK;
}

int TcPlan::check(cudaStream_t s, bool* wide) const {
  const bool pair = wide != nullptr && kind == kKindF16x3;
  int h[kFlags] = {};
  NNC_CUDA_TRY(cudaMemcpyAsync(h, err, (pair ? kFlags : 1) * sizeof(int), cudaMemcpyDeviceToHost, s));
  NNC_CUDA_TRY(cudaStreamSynchronize(s));
  if (wide) *wide = pair && h[kFlagWideX] != 0;
  return timed_out(h[0]);
}

}  // namespace tc
}  // namespace nnc
