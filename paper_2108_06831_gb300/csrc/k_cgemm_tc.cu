// Kernel (c), tensor-core forms: batched complex GEMM on tcgen05 with TMEM accumulators.
//
// A pairwise merge of two tensors is the product of Eq. 2.2, C[m][n] = sum_k A[m][k] B[n][k]
// once the legs are grouped (both operands with the contracted index contiguous).  The
// complex product is computed as one real GEMM: A (complex M x K, interleaved) is already
// the real M x 2K matrix [re im re im ...], and B is replaced by its 2x2 real embedding
// B2 (2N x 2K) with rows 2n = (Br, -Bi) and 2n+1 = (Bi, Br) per k, so that the real
// product A B2^T, read as interleaved pairs, is exactly Cr = ArBr - AiBi, Ci = ArBi + AiBr.
//
// FP32 accuracy on low-precision tensor cores comes from splitting the operands:
//   3XTF32:     x = hi + lo, hi = x rounded to TF32, lo = x - hi (exact);
//               C = hi*hi + hi*lo + lo*hi (kind::tf32, three MMAs per K slice);
//   SPLIT_BF16: x = x0 + x1 + x2 with x0 = bf16(x), x1 = bf16(x - x0), x2 = bf16(x - x0 - x1);
//               C = x0y0 + x0y1 + x1y0 + x0y2 + x1y1 + x2y0 (kind::f16 with bf16 operands).
// The embedding and split of B are written once per call into the workspace by a small prep
// kernel.  For 3XTF32 with at most two column tiles (HBM-bound merges) the A operand is
// split inside the GEMM: its FP32 tile arrives by TMA,
// and four converter warps overwrite it with hi and write lo beside it (same element size and
// swizzle, so the split is elementwise at equal offsets) before the MMAs read the stage; A
// then crosses HBM once, as FP32.  Otherwise A is split by a prep kernel too.  The GEMM
// streams the parts with TMA (128-byte swizzle) through a multi-stage mbarrier pipeline, a
// single thread issues tcgen05.mma into four 128 x BN FP32 accumulators in tensor memory,
// and the four converter/epilogue warps drain them with tcgen05.ld.  Inside the
// MMA an addend loses its low bits against a large accumulator, so, following Ootomo and
// Yokota's error-corrected TF32 GEMM, the correction products are summed apart from the
// leading one, and the leading product itself is spread over three accumulators (K tiles
// round robin); the epilogue adds the four in round-to-nearest FP32.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include "kernels.h"

namespace tnq {

cudaError_t launch_cgemm_fp32(long long batch, long long M, long long N, long long K, const float2 *A, const float2 *B,
                              float2 *C, void *ws, size_t ws_bytes, cudaStream_t s, const OutMap *om);
size_t cgemm_fp32_workspace(long long batch, long long M, long long N, long long K);

namespace {

constexpr int BM = 128;          // rows of A per CTA (MMA M)
constexpr int BN = 128;          // real columns of C per CTA (MMA N) = 64 complex columns
constexpr int KBYTES = 128;      // bytes of K per stage and operand row (one 128-byte swizzle span)
// warps 0-3: A split (3XTF32) and epilogue (warp w owns TMEM lanes 32w..32w+31);
// warp 4: TMA producer; warp 5: TMEM allocation and MMA issue
constexpr int kThreads = 192;
constexpr int kConvThreads = 128;
constexpr int kColBits = 6;  // log2 of the complex columns of a tile (BN / 2)
static_assert(BN / 2 == 1 << kColBits, "column table covers one tile");
constexpr int kMain = 3;                      // leading-product accumulators, used round robin by K tile
constexpr int kTmemCols = (kMain + 1) * BN;   // + one correction accumulator = all 512 columns
// tensor-memory columns of k_cgemm_tc's accumulators: the correction one between the first two leading
// ones, so that it is adjacent to either
constexpr int kCorrCol = BN;
__host__ __device__ constexpr int lead_col(int j) { return j == 0 ? 0 : (j + 1) * BN; }
constexpr unsigned long long kWaitNs = 2000000000ull;  // bound of every mbarrier wait
constexpr int kRasterRows = 8;  // row tiles per group of the tile order (k_cgemm_tc)

enum : int { PREC_TF32 = 1, PREC_BF16 = 2 };

template <int PREC>
struct Cfg;
template <>
struct Cfg<PREC_TF32> {
  static constexpr int kElem = 4, kParts = 2, kProducts = 3, kStages = 3, kMmaK = 8, kFmt = 2;
  __device__ static int pa(int p) { return p == 2 ? 1 : 0; }  // (hi,hi), (hi,lo), (lo,hi)
  __device__ static int pb(int p) { return p == 1 ? 1 : 0; }
};
template <>
struct Cfg<PREC_BF16> {
  static constexpr int kElem = 2, kParts = 3, kProducts = 6, kStages = 2, kMmaK = 16, kFmt = 1;
  // (0,0) (0,1) (1,0) (0,2) (1,1) (2,0)
  __device__ static int pa(int p) { return p == 2 ? 1 : p == 4 ? 1 : p == 5 ? 2 : 0; }
  __device__ static int pb(int p) { return p == 1 ? 1 : p == 3 ? 2 : p == 4 ? 1 : 0; }
};

constexpr int kTileA = BM * KBYTES;  // bytes of one A part per stage
constexpr int kTileB = BN * KBYTES;

__device__ __forceinline__ uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *b, int n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(b)), "r"(n));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t *b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(saddr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait (about two seconds of wall time): false, and the device status word set, if
// the phase never completed.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity, int *status) {
  if (mbar_try(b, parity)) return true;
  const unsigned long long t0 = now_ns();
  for (;;) {
    for (int i = 0; i < 256; ++i)
      if (mbar_try(b, parity)) return true;
    if (now_ns() - t0 > kWaitNs) break;
  }
  if (status) atomicCAS(status, 0, (int)TN_ERR_TIMEOUT);
  return false;
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::
          "r"(saddr(dst)),
      "l"(map), "r"(saddr(bar)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

// Shared-memory matrix descriptor (K-major operand, 128-byte swizzle, 8-row groups 1024 B apart).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);       // start address
  d |= (uint64_t)1 << 16;                        // leading byte offset (unused with this swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;              // stride byte offset: next 8-row group
  d |= (uint64_t)1 << 46;                        // descriptor version
  d |= (uint64_t)2 << 61;                        // 128-byte swizzle
  return d;
}

template <int PREC, int N>
__device__ __forceinline__ constexpr uint32_t instr_desc() {
  return (1u << 4)                                   // D: F32
         | ((uint32_t)Cfg<PREC>::kFmt << 7)          // A format
         | ((uint32_t)Cfg<PREC>::kFmt << 10)         // B format
         | ((uint32_t)(N >> 3) << 17)                // N
         | ((uint32_t)(BM >> 4) << 24);              // M
}

template <int PREC, int N = BN>
__device__ __forceinline__ void mma(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t acc) {
  constexpr uint32_t idesc = instr_desc<PREC, N>();
  if constexpr (PREC == PREC_TF32) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
  }
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar))
               : "memory");
}

// 32 consecutive fp32 columns of this warp's 32 TMEM lanes (one per thread); completes at
// the next tcgen05.wait::ld.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}

// Output index of natural flat index bits [lo, nbits) of f under the map.
__device__ __forceinline__ long long map_bits(const OutMap &om, long long f, int lo) {
  long long r = 0;
  for (int i = lo; i < om.nbits; ++i)
    if ((f >> i) & 1) r |= 1ll << om.pos[i];
  return r;
}

// One 32-column chunk (16 complex values, interleaved) of a row of C, either row-major
// (identity map) or at mapped positions: rowaddr = map of the row and column-tile bits,
// ctab[j] = map of the tile-local column bits (j < 64).
__device__ __forceinline__ void store_chunk(const OutMap &om, float *crow, float2 *C2, long long rowaddr,
                                            const long long *ctab, int c, const float (&v)[32]) {
  if (om.identity) {
    float4 *dst = reinterpret_cast<float4 *>(crow + c);
#pragma unroll
    for (int k = 0; k < 8; ++k) dst[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
  } else {
#pragma unroll
    for (int q = 0; q < 16; ++q) C2[rowaddr + ctab[c / 2 + q]] = make_float2(v[2 * q], v[2 * q + 1]);
  }
}

struct TmaMaps {
  CUtensorMap a[3];
  CUtensorMap b[3];
};

__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

__device__ __forceinline__ void mbar_arrive(uint64_t *b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(b)) : "memory");
}

// SPLIT_A (3XTF32 only): A arrives as FP32 and is split in shared memory by warps 0-3.
template <int PREC, bool SPLIT_A>
__global__ void __launch_bounds__(kThreads, 1) k_cgemm_tc(const __grid_constant__ TmaMaps maps, int k_tiles,
                                                          long long M, long long N2, float *__restrict__ C,
                                                          int *status, const __grid_constant__ OutMap om) {
  using CF = Cfg<PREC>;
  static_assert(!SPLIT_A || PREC == PREC_TF32, "on-chip split is the TF32 form");
  pdl_wait();  // before any memory access or TMEM allocation: the previous kernel has completed
  pdl_trigger();
  constexpr int S = CF::kStages;
  constexpr int stage_bytes = CF::kParts * (kTileA + kTileB);
  // bytes the TMA delivers per stage: A once as FP32 when it is split here, else its parts
  constexpr uint32_t tx_bytes = (SPLIT_A ? kTileA : CF::kParts * kTileA) + CF::kParts * kTileB;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // 1024-byte alignment of every tile (required by the 128-byte swizzle pattern)
  unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[S], conv[S], empty[S], done;
  __shared__ __align__(8) uint64_t drain;  // abort path: completion of the MMAs already issued
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  __shared__ int issued_parity[S];  // parity of the last TMA phase issued per stage, -1 if none
  __shared__ long long ctab[BN / 2];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // tile order: CTAs launch in linear order; consecutive CTAs walk kRasterRows row tiles before the
  // next column tile, so the CTAs resident at once read few A and B panels and the panels they share
  // stay in L2 (row-major order would re-read every B panel once per wave of CTAs)
  int n0, m0;
  {
    const int tn = (int)gridDim.x, tm = (int)gridDim.y;
    const int pid = (int)blockIdx.y * tn + (int)blockIdx.x;
    const int group = pid / (kRasterRows * tn);
    const int first = group * kRasterRows;
    const int rows = tm - first < kRasterRows ? tm - first : kRasterRows;
    const int in = pid - group * kRasterRows * tn;
    m0 = (first + in % rows) * BM;
    n0 = (in / rows) * BN;
  }
  const int bz = blockIdx.z;
  if (threadIdx.x < BN / 2) ctab[threadIdx.x] = om.identity ? 0 : map_bits(om, threadIdx.x, 0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&conv[s], kConvThreads);
      mbar_init(&empty[s], 1);
      issued_parity[s] = -1;
    }
    mbar_init(&done, 1);
    mbar_init(&drain, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 5) {  // the whole warp allocates the accumulators' columns of tensor memory
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_base)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_d = tmem_base;
  bool mma_issued = false;  // warp 5 lane 0: at least one MMA was issued

  if (warp == 4) {
    if (lane == 0) {  // TMA producer
      for (int kt = 0; kt < k_tiles; ++kt) {
        const int s = kt % S;
        if (kt >= S && !mbar_wait(&empty[s], ((kt / S) - 1) & 1, status)) {
          abort_flag = 1;
          break;
        }
        mbar_expect_tx(&full[s], tx_bytes);
        issued_parity[s] = (kt / S) & 1;
        unsigned char *st = smem + (size_t)s * stage_bytes;
        const int kc = kt * (KBYTES / CF::kElem);
        const int a_loads = SPLIT_A ? 1 : CF::kParts;
        for (int p = 0; p < a_loads; ++p) tma_load_3d(st + p * kTileA, &maps.a[p], &full[s], kc, m0, bz);
        for (int p = 0; p < CF::kParts; ++p) {
          const int at = kt % kMain == 1 && p < 2 ? 1 - p : p;  // see the MMA issuer
          tma_load_3d(st + CF::kParts * kTileA + at * kTileB, &maps.b[p], &full[s], kc, n0, bz);
        }
      }
    }
  } else if (warp == 5) {
    if (lane == 0) {  // MMA issuer
      bool ok = true;
      for (int kt = 0; kt < k_tiles; ++kt) {
        const int s = kt % S;
        if (!mbar_wait(SPLIT_A ? &conv[s] : &full[s], (kt / S) & 1, status)) {
          ok = false;
          abort_flag = 1;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t st = saddr(smem + (size_t)s * stage_bytes);
        // product 0 (the leading parts) of K tile kt accumulates in lead_col(j), j = kt mod kMain; the
        // correction products in kCorrCol.  Small terms never meet the large running sum inside the
        // MMA, and each leading accumulator sees a third of the K steps.  Products 0 and 1 share A's
        // leading part; for j = 0 and 1 their accumulators are adjacent, and B's first two parts lie in
        // the accumulators' order (leading, correction; for j = 1 correction, leading): one MMA of 2 BN
        // columns does both and reads A once.  The sums keep their order.
        constexpr int kSteps = KBYTES / (CF::kMmaK * CF::kElem);
        const int j = kt % kMain;
        const uint32_t b_at = st + CF::kParts * kTileA;
        const uint32_t b_lead = b_at + (j == 1 ? kTileB : 0), b_corr = b_at + (j == 1 ? 0 : kTileB);
#pragma unroll
        for (int kk = 0; kk < kSteps; ++kk) {
          const uint32_t off = kk * CF::kMmaK * CF::kElem;  // 32 bytes per MMA along K
          const bool acc_lead = kt >= kMain || kk > 0, acc_corr = kt > 0 || kk > 0;
          if (j < 2 && acc_lead == acc_corr) {
            mma<PREC, 2 * BN>(tmem_d + (uint32_t)(j * BN), smem_desc(st + off), smem_desc(b_at + off), acc_lead ? 1u : 0u);
          } else {
            mma<PREC>(tmem_d + (uint32_t)lead_col(j), smem_desc(st + off), smem_desc(b_lead + off), acc_lead ? 1u : 0u);
            mma<PREC>(tmem_d + kCorrCol, smem_desc(st + off), smem_desc(b_corr + off), acc_corr ? 1u : 0u);
          }
        }
#pragma unroll
        for (int p = 2; p < CF::kProducts; ++p) {
          const uint32_t a_base = st + CF::pa(p) * kTileA;
          const uint32_t b_base = CF::pb(p) == 0 ? b_lead : CF::pb(p) == 1 ? b_corr : b_at + CF::pb(p) * kTileB;
#pragma unroll
          for (int kk = 0; kk < kSteps; ++kk) {
            const uint32_t off = kk * CF::kMmaK * CF::kElem;
            mma<PREC>(tmem_d + kCorrCol, smem_desc(a_base + off), smem_desc(b_base + off), 1u);
          }
        }
        mma_issued = true;
        mma_commit(&empty[s]);  // frees the stage once these MMAs have read it
      }
      if (ok) mma_commit(&done);
    }
  } else if constexpr (SPLIT_A) {
    // A split: x -> hi = TF32(x) (in place), lo = x - hi (part 1 of the stage), then make the
    // generic-proxy writes visible to the tensor cores and report the stage converted
    for (int kt = 0; kt < k_tiles; ++kt) {
      const int s = kt % S;
      if (!mbar_wait(&full[s], (kt / S) & 1, status)) {
        abort_flag = 1;
        break;
      }
      float4 *hi = reinterpret_cast<float4 *>(smem + (size_t)s * stage_bytes);
      float4 *lo = reinterpret_cast<float4 *>(smem + (size_t)s * stage_bytes + kTileA);
#pragma unroll 4
      for (int c = threadIdx.x; c < kTileA / 16; c += kConvThreads) {
        const float4 v = hi[c];
        const float4 h = make_float4(tf32_rna(v.x), tf32_rna(v.y), tf32_rna(v.z), tf32_rna(v.w));
        lo[c] = make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w);
        hi[c] = h;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(&conv[s]);
    }
  }
  __syncwarp();

  // epilogue: warps 0-3 drain their 32 TMEM lanes (= 32 rows of the tile)
  bool have = !abort_flag && mbar_wait(&done, 0, status);
  have = __all_sync(0xFFFFFFFFu, have);  // tcgen05.ld is warp-collective: decide per warp
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (have && warp < 4) {
    const long long row = m0 + warp * 32 + lane;
    float *crow = C + ((long long)bz * M + row) * N2 + n0;
    long long rowaddr = 0;
    if (!om.identity) {
      int lgn = 0;
      while ((2ll << lgn) < N2) ++lgn;  // complex columns = 2^lgn
      rowaddr = map_bits(om, (((long long)bz * M + row) << lgn) | (long long)(n0 / 2), kColBits);
    }
    const int n_main = k_tiles < kMain ? k_tiles : kMain;  // accumulators that were written
    for (int c = 0; c < BN; c += 32) {
      const uint32_t taddr = tmem_d + ((uint32_t)(warp * 32) << 16) + (uint32_t)c;
      float v[32];
      {
        uint32_t e[32];
        tmem_ld32(taddr + kCorrCol, e);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(e[i]);
      }
      for (int j = 0; j < n_main; ++j) {  // corrections first, then the leading sums in order
        uint32_t r[32];
        tmem_ld32(taddr + lead_col(j), r);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] += __uint_as_float(r[i]);
      }
      store_chunk(om, crow, reinterpret_cast<float2 *>(C), rowaddr, ctab, c, v);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (abort_flag) {  // uniform: nothing writes the flag after the barrier above
    // let copies already in flight land (the last phase issued into each stage), and let the
    // MMAs already issued finish reading shared memory and writing TMEM, before the CTA
    // releases either
    if (threadIdx.x == 0)
      for (int s = 0; s < S; ++s)
        if (issued_parity[s] >= 0) mbar_wait(&full[s], (uint32_t)issued_parity[s], nullptr);
    if (warp == 5 && lane == 0 && mma_issued) {
      mma_commit(&drain);
      mbar_wait(&drain, 0, nullptr);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
  }
  if (warp == 5) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(kTmemCols));
  }
}

// Persistent form for short, HBM-bound merges (3XTF32 or SPLIT_BF16, A split on chip, at most
// kStreamMaxKTiles K tiles; a network merge has N = K = 64 and thousands of 128-row tiles):
// one CTA per SM walks the tiles (column tile fastest, then row tile, then batch), the TMA
// stage ring runs on across tile boundaries, and the accumulators are double-buffered in
// TMEM (leading + correction product per buffer, 2 x 2 x BN columns), so dedicated epilogue
// warps drain tile i while tile i+1 is loaded, split and multiplied.
// The first split_warps: A split; then one for TMA, one for TMEM allocation and MMA issue, and four for the
// epilogue (warp w owns TMEM lanes 32 (w mod 4)..+31).
// Warps of the A split: four for TF32; eight for BF16, whose split reads, converts and writes three times
// as much work per element (batch 64, 32768 x 64 x 64: 498 us with four, 462 with eight; TF32 399 and 403).
template <int PREC>
constexpr int split_warps() { return PREC == PREC_TF32 ? 4 : 8; }
template <int PREC>
constexpr int stream_threads() { return 32 * split_warps<PREC>() + 64 + 128; }  // + TMA, MMA and epilogue warps
constexpr int kStreamMaxKTiles = 8;  // a single leading accumulator per tile stays accurate

// How an epilogue warp writes back a chunk of 32 rows x 16 complex columns of C (built on the host by
// chunk_map).  The chunk's 9 local bits (4 column, 5 row) are enumerated by increasing stored position
// as the bits of u; lane and iteration give u = 64 it + 2 lane (+ 1).  The chunk is staged at
// row * 16 + (column ^ S(row)) with S linear over the row bits: s[k] is the staging contribution of u's
// bit k (combined by XOR), g[k] its stored offset (combined by addition), and S is chosen so that both
// the writes (lanes = rows) and the reads (lanes = bits 1-5 of u) of each half warp fall in distinct
// banks.  Loads of index tables and bank conflicts of a padded staging were 1500 of the 4100 shared-
// memory wavefronts of a tile, on a kernel bound by them.
enum { kStaged = 0, kDirectCols = 1, kDirectRows = 2 };
// (A parameter of every launch: 136 bytes; with all offsets in it, 228, a one-tile call took 10.65 us, 10.45 now.)
struct ChunkMap {
  long long g[9];
  long long chunk_g[2];  // stored offsets of the column bits above the chunk's
  int s[9];
  uint8_t row_swz[5];    // S of each row bit
  bool pairs;            // u and u + 1 are adjacent in memory
  // Written back from the registers instead, where a store of the warp covers runs of at least 128 bytes
  // so (64-byte runs filled by two stores for kDirectCols with column bit 2 below the row bits).
  // kDirectCols: column bits 0 and 1 are the lowest stored bits and row bits come next, a lane stores four
  // columns of its row, 32 bytes.  kDirectRows: row bits 0-3 are the lowest, a lane stores single columns.
  // Staging was 128 of the 900 KB that a tile moves through the shared-memory data pipe, which bounds this
  // kernel.  Batch 64, 32768 x 64 x 64 stored as the next merge reads it (column bits 0-2, the row bits, then
  // the others): 437 -> 386 us.  Row-major rows, 512 bytes apart, are staged: 399 us, 496 from registers.
  // Both take the row bits' offsets from g[1] .. g[5], where a staged chunk has its lanes', and the column
  // bits' from g[0], g[6], g[7] and g[8].
  uint8_t direct;
};
static_assert(sizeof(ChunkMap) == 136, "small as a kernel parameter");
// 32 bytes (a whole sector) in one store
__device__ __forceinline__ void store8(float2 *p, const float *v) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

// Split of one A stage from FP32 into three BF16 parts, in place: the FP32 tile is two 128-byte
// boxes (K elements 32j..32j+31 of every row, 16-byte chunks swizzled by row mod 8); part p is a
// 128 x 64 BF16 tile at p x 16 KB (chunk d = K elements 8d..8d+7, same swizzle).  Each of the
// converter threads first reads its output chunks' sources, then (after a named barrier: the
// parts overwrite the FP32 tile) writes x0 = bf16(x), x1 = bf16(x - x0), x2 = bf16(x - x0 - x1).
__device__ __forceinline__ void split_bf16_in_place(unsigned char *st) {
  constexpr int kSplitThreads = 32 * split_warps<PREC_BF16>(), kItems = 1024 / kSplitThreads;
  float v[kItems][8];
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int item = threadIdx.x + kSplitThreads * it, r = item >> 3, d = item & 7;
    const unsigned char *row = st + (d >> 2) * kTileA + r * 128;
    const int c0 = 2 * (d & 3);
    const float4 a = *reinterpret_cast<const float4 *>(row + ((c0 ^ (r & 7)) << 4));
    const float4 b = *reinterpret_cast<const float4 *>(row + (((c0 + 1) ^ (r & 7)) << 4));
    v[it][0] = a.x, v[it][1] = a.y, v[it][2] = a.z, v[it][3] = a.w;
    v[it][4] = b.x, v[it][5] = b.y, v[it][6] = b.z, v[it][7] = b.w;
  }
  asm volatile("bar.sync 1, %0;" ::"n"(kSplitThreads) : "memory");
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int item = threadIdx.x + kSplitThreads * it, r = item >> 3, d = item & 7;
    uint32_t w[3][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t h[3][2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float x = v[it][2 * q + e];
        const __nv_bfloat16 b0 = __float2bfloat16_rn(x);
        const float r1 = x - __bfloat162float(b0);
        const __nv_bfloat16 b1 = __float2bfloat16_rn(r1);
        const __nv_bfloat16 b2 = __float2bfloat16_rn(r1 - __bfloat162float(b1));
        h[0][e] = __bfloat16_as_ushort(b0);
        h[1][e] = __bfloat16_as_ushort(b1);
        h[2][e] = __bfloat16_as_ushort(b2);
      }
#pragma unroll
      for (int p = 0; p < 3; ++p) w[p][q] = h[p][0] | (h[p][1] << 16);
    }
#pragma unroll
    for (int p = 0; p < 3; ++p)
      *reinterpret_cast<uint4 *>(st + p * kTileA + r * 128 + ((d ^ (r & 7)) << 4)) =
          make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
  }
}

template <int PREC>
__global__ void __launch_bounds__(stream_threads<PREC>(), 1)
    k_cgemm_tc_stream(const __grid_constant__ TmaMaps maps, int k_tiles, int tiles_n, int tiles_m,
                      long long total_tiles, long long M, long long N2, float *__restrict__ C, int *status,
                      const __grid_constant__ OutMap om, const __grid_constant__ ChunkMap cm) {
  using CF = Cfg<PREC>;
  pdl_wait();  // before any memory access or TMEM allocation: the previous kernel has completed
  pdl_trigger();
  constexpr int S = CF::kStages, kSplitWarps = split_warps<PREC>(), kSplitThreads = 32 * kSplitWarps;
  constexpr int stage_bytes = CF::kParts * (kTileA + kTileB);
  // A arrives as FP32: one 128-byte box per row and K tile for TF32, two for BF16 (64 elements)
  constexpr int a_boxes = PREC == PREC_TF32 ? 1 : 2;
  constexpr uint32_t tx_bytes = a_boxes * kTileA + CF::kParts * kTileB;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[S], conv[S], empty[S], acc_full[2], acc_empty[2], drain;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  __shared__ int issued_parity[S];  // parity of the last TMA phase issued per stage, -1 if none
  __shared__ float2 stage_c[4][32 * 16];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&conv[s], kSplitThreads);
      mbar_init(&empty[s], 1);
      issued_parity[s] = -1;
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 128);
    }
    mbar_init(&drain, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kSplitWarps + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_base)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_d = tmem_base;
  bool mma_issued = false;  // MMA warp lane 0: at least one MMA was issued

  auto aborted = [&]() { return *reinterpret_cast<volatile int *>(&abort_flag) != 0; };
  auto decode = [&](long long t, int &nt, int &mt, int &bz) {
    nt = (int)(t % tiles_n);
    const long long r = t / tiles_n;
    mt = (int)(r % tiles_m);
    bz = (int)(r / tiles_m);
  };

  if (warp == kSplitWarps) {
    if (lane == 0) {  // TMA producer
      long long g = 0;
      for (long long t = blockIdx.x; t < total_tiles && !aborted(); t += gridDim.x) {
        int nt, mt, bz;
        decode(t, nt, mt, bz);
        for (int kt = 0; kt < k_tiles; ++kt, ++g) {
          const int s = (int)(g % S);
          if (g >= S && !mbar_wait(&empty[s], (uint32_t)(((g / S) - 1) & 1), status)) {
            abort_flag = 1;
            break;
          }
          mbar_expect_tx(&full[s], tx_bytes);
          issued_parity[s] = (int)((g / S) & 1);
          unsigned char *st = smem + (size_t)s * stage_bytes;
          const int kc = kt * (KBYTES / CF::kElem);  // K elements before this tile
          for (int j = 0; j < a_boxes; ++j) tma_load_3d(st + j * kTileA, &maps.a[0], &full[s], kc + 32 * j, mt * BM, bz);
          for (int p = 0; p < CF::kParts; ++p)
            tma_load_3d(st + CF::kParts * kTileA + p * kTileB, &maps.b[p], &full[s], kc, nt * BN, bz);
        }
      }
    }
  } else if (warp == kSplitWarps + 1) {
    if (lane == 0) {  // MMA issuer
      long long g = 0, li = 0;
      for (long long t = blockIdx.x; t < total_tiles && !aborted(); t += gridDim.x, ++li) {
        const int ab = (int)(li & 1);
        if (li >= 2 && !mbar_wait(&acc_empty[ab], (uint32_t)(((li / 2) - 1) & 1), status)) {
          abort_flag = 1;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t base = tmem_d + (uint32_t)(ab * 2 * BN);
        bool ok = true;
        for (int kt = 0; kt < k_tiles; ++kt, ++g) {
          const int s = (int)(g % S);
          if (!mbar_wait(&conv[s], (uint32_t)((g / S) & 1), status)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t st = saddr(smem + (size_t)s * stage_bytes);
          // products 0 and 1 share A's leading part, B's first two parts are adjacent in shared memory
          // and the leading and correction accumulators in tensor memory: one MMA of 2 BN columns per
          // K step does both, and reads A once.  The sums keep their order.
#pragma unroll
          for (int kk = 0; kk < KBYTES / (CF::kMmaK * CF::kElem); ++kk) {
            const uint32_t off = kk * CF::kMmaK * CF::kElem;
            mma<PREC, 2 * BN>(base, smem_desc(st + off), smem_desc(st + CF::kParts * kTileA + off),
                              kt > 0 || kk > 0 ? 1u : 0u);
          }
#pragma unroll
          for (int p = 2; p < CF::kProducts; ++p) {
            const uint32_t a_base = st + CF::pa(p) * kTileA;
            const uint32_t b_base = st + CF::kParts * kTileA + CF::pb(p) * kTileB;
#pragma unroll
            for (int kk = 0; kk < KBYTES / (CF::kMmaK * CF::kElem); ++kk) {
              const uint32_t off = kk * CF::kMmaK * CF::kElem;
              mma<PREC>(base + BN, smem_desc(a_base + off), smem_desc(b_base + off), 1u);
            }
          }
          mma_issued = true;
          mma_commit(&empty[s]);
        }
        if (!ok) {
          abort_flag = 1;
          break;
        }
        mma_commit(&acc_full[ab]);
      }
    }
  } else if (warp < kSplitWarps) {  // A split, as in k_cgemm_tc
    long long g = 0;
    for (long long t = blockIdx.x; t < total_tiles; t += gridDim.x) {
      bool ok = true;
      for (int kt = 0; kt < k_tiles; ++kt, ++g) {
        const int s = (int)(g % S);
        if (!mbar_wait(&full[s], (uint32_t)((g / S) & 1), status)) {
          ok = false;
          break;
        }
        if constexpr (PREC == PREC_TF32) {
          float4 *hi = reinterpret_cast<float4 *>(smem + (size_t)s * stage_bytes);
          float4 *lo = reinterpret_cast<float4 *>(smem + (size_t)s * stage_bytes + kTileA);
#pragma unroll 4
          for (int c = threadIdx.x; c < kTileA / 16; c += kSplitThreads) {
            const float4 v = hi[c];
            const float4 h = make_float4(tf32_rna(v.x), tf32_rna(v.y), tf32_rna(v.z), tf32_rna(v.w));
            lo[c] = make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w);
            hi[c] = h;
          }
        } else {
          split_bf16_in_place(smem + (size_t)s * stage_bytes);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(&conv[s]);
      }
      if (!ok) {
        abort_flag = 1;
        break;
      }
    }
  } else {  // epilogue warps
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    int lgn = 0;
    while ((2ll << lgn) < N2) ++lgn;  // complex columns = 2^lgn (with a permuted output)
    float2 *stg = stage_c[q];
    // this lane's part of the staging and stored offsets (u's bits 1-5)
    int wr = 0, rd = 0;
    long long go = 0;
    for (int k = 0; k < 5; ++k)
      if ((lane >> k) & 1) {
        wr ^= (16 << k) ^ cm.row_swz[k];
        rd ^= cm.s[k + 1];
        go += cm.g[k + 1];
      }
    long long li = 0;
    for (long long t = blockIdx.x; t < total_tiles; t += gridDim.x, ++li) {
      const int ab = (int)(li & 1);
      // the tile's stored offset, while its accumulators are still being summed (found per chunk and after the
      // wait, it was in the way of the tile's other work: 24-qubit blocks of 64 x 64 in split BF16 2375 us, so
      // 1824; 3xTF32 1629 and 1556)
      int nt, mt, bz;
      decode(t, nt, mt, bz);
      const long long row0 = (long long)bz * M + (long long)mt * BM + q * 32;  // the warp's first row
      float2 *Ct = reinterpret_cast<float2 *>(C) + go +
                   (om.identity ? row0 * (N2 / 2) + nt * (BN / 2)
                                : map_bits(om, (row0 << lgn) | ((long long)nt * (BN / 2)), 0));
      bool have = mbar_wait(&acc_full[ab], (uint32_t)((li / 2) & 1), status);
      have = __all_sync(0xFFFFFFFFu, have);
      if (!have) {
        abort_flag = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t base = tmem_d + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * 2 * BN);
      for (int c = 0; c < BN; c += 32) {
        uint32_t r[32], e[32];
        tmem_ld32(base + BN + c, e);  // corrections
        tmem_ld32(base + c, r);       // leading product
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        float2 *C2 = Ct + ((c & 32) ? cm.chunk_g[0] : 0) + ((c & 64) ? cm.chunk_g[1] : 0);
        if (cm.direct == kDirectRows) {
#pragma unroll
          for (int k = 0; k < 16; ++k)
            C2[((k & 1) ? cm.g[0] : 0) + ((k & 2) ? cm.g[6] : 0) + ((k & 4) ? cm.g[7] : 0) +
               ((k & 8) ? cm.g[8] : 0)] = make_float2(__uint_as_float(e[2 * k]) + __uint_as_float(r[2 * k]),
                                                          __uint_as_float(e[2 * k + 1]) + __uint_as_float(r[2 * k + 1]));
          continue;
        }
        if (cm.direct == kDirectCols) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(e[8 * k + i]) + __uint_as_float(r[8 * k + i]);
            store8(C2 + ((k & 1) ? cm.g[7] : 0) + ((k & 2) ? cm.g[8] : 0), v);
          }
          continue;
        }
#pragma unroll
        for (int k = 0; k < 16; ++k)
          stg[wr ^ k] = make_float2(__uint_as_float(e[2 * k]) + __uint_as_float(r[2 * k]),
                                    __uint_as_float(e[2 * k + 1]) + __uint_as_float(r[2 * k + 1]));
        __syncwarp();
#pragma unroll
        for (int it = 0; it < 8; ++it) {
          const int at = rd ^ ((it & 1) ? cm.s[6] : 0) ^ ((it & 2) ? cm.s[7] : 0) ^ ((it & 4) ? cm.s[8] : 0);
          float2 *dst = C2 + ((it & 1) ? cm.g[6] : 0) + ((it & 2) ? cm.g[7] : 0) + ((it & 4) ? cm.g[8] : 0);
          const float2 x0 = stg[at], x1 = stg[at ^ cm.s[0]];
          if (cm.pairs) {
            *reinterpret_cast<float4 *>(dst) = make_float4(x0.x, x0.y, x1.x, x1.y);
          } else {
            dst[0] = x0;
            dst[cm.g[0]] = x1;
          }
        }
        __syncwarp();
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      mbar_arrive(&acc_empty[ab]);
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (abort_flag) {  // uniform: nothing writes the flag after the barrier above
    // let copies already in flight land, and the MMAs already issued finish, before the CTA
    // releases its shared memory and tensor memory
    if (threadIdx.x == 0)
      for (int s = 0; s < S; ++s)
        if (issued_parity[s] >= 0) mbar_wait(&full[s], (uint32_t)issued_parity[s], nullptr);
    if (warp == kSplitWarps + 1 && lane == 0 && mma_issued) {
      mma_commit(&drain);
      mbar_wait(&drain, 0, nullptr);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
  }
  if (warp == kSplitWarps + 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(kTmemCols));
  }
}

// The chunk's write-back for columns lgn (log2, with a permuted output) or N complex columns (row-major).
void chunk_map(ChunkMap &cm, const OutMap &om, long long N, const void *C) {
  std::memset(&cm, 0, sizeof(cm));
  int lgn = 0, order[9];
  long long off[9];  // stored offset of local bit b: b < 4 column, else row
  while ((1ll << lgn) < N) ++lgn;
  for (int b = 0; b < 9; ++b) {
    order[b] = b;
    if (om.identity) off[b] = b < 4 ? 1ll << b : N << (b - 4);
    else off[b] = 1ll << (b < 4 ? om.pos[b] : om.pos[lgn + b - 4]);
  }
  for (int b = 4; b < kColBits; ++b) cm.chunk_g[b - 4] = 1ll << (om.identity ? b : om.pos[b]);
  std::sort(order, order + 9, [&](int x, int y) { return off[x] < off[y]; });
  // S: the row bits read by a half warp (bits 1-4 of u) take the column bits it does not read; the
  // other row bits among the first four, the lanes of a write, take what is left of the column bits
  bool col_read[4] = {false, false, false, false}, taken[4] = {false, false, false, false};
  bool row_read[5] = {false, false, false, false, false};
  for (int k = 1; k <= 4; ++k) (order[k] < 4 ? col_read[order[k]] : row_read[order[k] - 4]) = true;
  int next = 0;
  for (int r = 0; r < 5; ++r) {
    if (!row_read[r]) continue;
    while (col_read[next]) ++next;
    cm.row_swz[r] = (uint8_t)(1 << next);
    if (r < 4) taken[next] = true;
    ++next;
  }
  next = 0;
  for (int r = 0; r < 4; ++r) {
    if (row_read[r]) continue;
    while (taken[next]) ++next;
    cm.row_swz[r] = (uint8_t)(1 << next);
    taken[next] = true;
  }
  for (int k = 0; k < 9; ++k) {
    const int b = order[k];
    cm.s[k] = b < 4 ? 1 << b : (16 << (b - 4)) ^ cm.row_swz[b - 4];
    cm.g[k] = off[b];
  }
  cm.pairs = off[order[0]] == 1;
  if (off[0] == 1 && off[1] == 2 && order[3] >= 4 && (uintptr_t)C % 32 == 0) cm.direct = kDirectCols;
  if (off[4] == 1 && off[5] == 2 && off[6] == 4 && off[7] == 8) cm.direct = kDirectRows;
  if (cm.direct) {
    for (int k = 0; k < 5; ++k) cm.g[k + 1] = off[k + 4];
    cm.g[0] = off[0], cm.g[6] = off[1], cm.g[7] = off[2], cm.g[8] = off[3];
  }
}

// ------------------------------------------------------------------------------ prep kernels

// The parts of four consecutive elements, 16 (TF32) or 8 (BF16) bytes of each part per thread.
template <int PREC>
__device__ __forceinline__ void store_parts(float4 v, long long at, void *p0, void *p1, void *p2) {
  if constexpr (PREC == PREC_TF32) {
    const float4 h = make_float4(tf32_rna(v.x), tf32_rna(v.y), tf32_rna(v.z), tf32_rna(v.w));
    *reinterpret_cast<float4 *>(static_cast<float *>(p0) + at) = h;
    *reinterpret_cast<float4 *>(static_cast<float *>(p1) + at) = make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w);
  } else {
    const float x[4] = {v.x, v.y, v.z, v.w};
    uint32_t w[3][2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      uint32_t h[3][2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const __nv_bfloat16 b0 = __float2bfloat16_rn(x[2 * q + e]);
        const float r1 = x[2 * q + e] - __bfloat162float(b0);
        const __nv_bfloat16 b1 = __float2bfloat16_rn(r1);
        h[0][e] = __bfloat16_as_ushort(b0);
        h[1][e] = __bfloat16_as_ushort(b1);
        h[2][e] = __bfloat16_as_ushort(__float2bfloat16_rn(r1 - __bfloat162float(b1)));
      }
#pragma unroll
      for (int p = 0; p < 3; ++p) w[p][q] = h[p][0] | (h[p][1] << 16);
    }
    void *const part[3] = {p0, p1, p2};
#pragma unroll
    for (int p = 0; p < 3; ++p)
      *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(part[p]) + at) = make_uint2(w[p][0], w[p][1]);
  }
}

// A (n real values, a multiple of 4: operand rows are multiples of 16 bytes) -> parts.  HBM-bound: 4096 x
// 4096 complex into TF32 parts 98 us with one element per thread and store, 66 with four.
template <int PREC>
__global__ void k_split(const float *__restrict__ x, long long n, void *p0, void *p1, void *p2) {
  pdl_wait();
  pdl_trigger();
  for (long long i = 4 * ((long long)blockIdx.x * blockDim.x + threadIdx.x); i < n;
       i += 4 * (long long)gridDim.x * blockDim.x)
    store_parts<PREC>(*reinterpret_cast<const float4 *>(x + i), i, p0, p1, p2);
}

// B (complex [N][K], K even) -> 2x2 real embedding [2N][2K], then split: two values of k per thread.
template <int PREC>
__global__ void k_embed_split(const float2 *__restrict__ b, long long N, long long K, long long batch, void *p0,
                              void *p1, void *p2) {
  pdl_wait();
  pdl_trigger();
  const long long half = K / 2, total = batch * N * half;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long row = i / half, k = 2 * (i - row * half);  // row = bb N + n
    const float4 v = reinterpret_cast<const float4 *>(b)[i];
    const long long at = 4 * row * K + 2 * k;  // rows 2 row: (re, -im), and 2 row + 1: (im, re)
    store_parts<PREC>(make_float4(v.x, -v.y, v.z, -v.w), at, p0, p1, p2);
    store_parts<PREC>(make_float4(v.y, v.x, v.w, v.z), at + 2 * K, p0, p1, p2);
  }
}

// ------------------------------------------------------------------------------ host side

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static std::once_flag once;
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

bool make_map(CUtensorMap *m, const void *base, int elem, long long cols, long long rows, long long batch, int box_rows) {
  auto enc = encode_fn();
  if (!enc) return false;
  const CUtensorMapDataType dt = elem == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)cols * elem, (cuuint64_t)cols * rows * elem};
  cuuint32_t box[3] = {(cuuint32_t)(KBYTES / elem), (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return enc(m, dt, 3, const_cast<void *>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// K needs no multiple of the K tile: the TMA fills the part of a K tile beyond the operands
// with zeros (exact zero products); only the row stride must be a multiple of 16 bytes.
bool tc_shape_ok(int precision, long long M, long long N, long long K) {
  const long long elem = precision == TN_PREC_3XTF32 ? 4 : 2;
  return M % BM == 0 && (2 * N) % BN == 0 && (2 * K * elem) % 16 == 0 && M > 0 && N > 0 && K > 0 &&
         M * 2 * N < (1ll << 40);
}

int k_tiles_of(int precision, long long K) {
  const long long elem = precision == TN_PREC_3XTF32 ? 4 : 2;
  return (int)((2 * K * elem + KBYTES - 1) / KBYTES);
}

size_t part_bytes(int precision, long long rows, long long cols, long long batch) {
  return (size_t)rows * cols * batch * (precision == TN_PREC_3XTF32 ? 4 : 2);
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

// A is split on chip when few CTAs read each A tile (HBM-bound merges: the split copy would
// cost more traffic than the GEMM); with many column tiles the one-pass prep split is
// cheaper than converting every tile again in every CTA.
bool split_a_on_chip(int precision, long long N, long long K) {
  if ((2 * N) / BN > 2) return false;
  if (precision == TN_PREC_3XTF32) return true;
  // BF16 parts are made on chip by the streaming kernel only (short K)
  return precision == TN_PREC_SPLIT_BF16 && k_tiles_of(precision, K) <= kStreamMaxKTiles;
}

template <int PREC, bool SPLIT_A>
cudaError_t run_tc(long long batch, long long M, long long N, long long K, const float2 *A, const float2 *B, float2 *C,
                   void *ws, cudaStream_t s, const OutMap &om) {
  using CF = Cfg<PREC>;
  const int prec_abi = PREC == PREC_TF32 ? TN_PREC_3XTF32 : TN_PREC_SPLIT_BF16;
  const size_t pa = SPLIT_A ? 0 : align256(part_bytes(prec_abi, M, 2 * K, batch));
  const size_t pb = align256(part_bytes(prec_abi, 2 * N, 2 * K, batch));
  char *w = static_cast<char *>(ws);
  void *ap[3] = {w, w + pa, w + 2 * pa};
  char *wb = w + CF::kParts * pa;
  void *bp[3] = {wb, wb + pb, wb + 2 * pb};
  cudaError_t e = cudaSuccess;
  if (SPLIT_A) {
    ap[0] = const_cast<float2 *>(A);  // the GEMM reads A itself (FP32) and splits it on chip
  } else {
    const long long na = batch * M * 2 * K;
    e = launch_pdl(k_split<PREC>, dim3((unsigned)std::min<long long>((na / 4 + 255) / 256, 65535)), dim3(256), 0, s,
                   reinterpret_cast<const float *>(A), na, ap[0], ap[1], ap[2]);
    if (e != cudaSuccess) return e;
  }
  const long long nb = batch * N * K / 2;
  e = launch_pdl(k_embed_split<PREC>, dim3((unsigned)std::min<long long>((nb + 255) / 256, 65535)), dim3(256), 0, s,
                 B, N, K, batch, bp[0], bp[1], bp[2]);
  if (e != cudaSuccess) return e;
  TmaMaps maps;
  std::memset(&maps, 0, sizeof(maps));
  for (int p = 0; p < CF::kParts; ++p) {
    // A split on chip arrives as FP32 (4-byte elements) whatever the parts' type
    if ((!SPLIT_A || p == 0) && !make_map(&maps.a[p], ap[p], SPLIT_A ? 4 : CF::kElem, 2 * K, M, batch, BM))
      return cudaErrorInvalidValue;
    if (!make_map(&maps.b[p], bp[p], CF::kElem, 2 * K, 2 * N, batch, BN)) return cudaErrorInvalidValue;
  }
  const size_t smem = (size_t)CF::kStages * CF::kParts * (kTileA + kTileB) + 1024;
  const int k_tiles = k_tiles_of(prec_abi, K);
  if constexpr (SPLIT_A) {
    if (k_tiles <= kStreamMaxKTiles) {  // short merge: persistent CTAs with overlapped epilogue
      e = ensure_smem(reinterpret_cast<const void *>(k_cgemm_tc_stream<PREC>), smem);
      if (e != cudaSuccess) return e;
      const int tiles_n = (int)((2 * N) / BN), tiles_m = (int)(M / BM);
      const long long total = (long long)tiles_n * tiles_m * batch;
      const long long grid = std::min<long long>(total, num_sms());
      ChunkMap cm;
      chunk_map(cm, om, N, C);
      return launch_pdl(k_cgemm_tc_stream<PREC>, dim3((unsigned)grid), dim3(stream_threads<PREC>()), smem, s, maps, k_tiles,
                        tiles_n, tiles_m, total, M, 2 * N, reinterpret_cast<float *>(C),
                        static_cast<int *>(status_word_ptr()), om, cm);
    }
  }
  if constexpr (SPLIT_A && PREC == PREC_BF16) {
    return cudaErrorNotSupported;  // the on-chip BF16 split exists in the streaming form only
  } else {
    e = ensure_smem(reinterpret_cast<const void *>(k_cgemm_tc<PREC, SPLIT_A>), smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((2 * N) / BN), (unsigned)(M / BM), (unsigned)batch);
    return launch_pdl(k_cgemm_tc<PREC, SPLIT_A>, grid, dim3(kThreads), smem, s, maps, k_tiles, M, 2 * N,
                      reinterpret_cast<float *>(C), static_cast<int *>(status_word_ptr()), om);
  }
}

}  // namespace

size_t cgemm_workspace(int precision, long long batch, long long M, long long N, long long K) {
  if (precision == TN_PREC_FP32) return cgemm_fp32_workspace(batch, M, N, K);
  if (!tc_shape_ok(precision, M, N, K)) return 0;
  const int parts = precision == TN_PREC_3XTF32 ? 2 : 3;
  // A split on chip: only B's parts are stored
  if (split_a_on_chip(precision, N, K)) return parts * align256(part_bytes(precision, 2 * N, 2 * K, batch));
  return parts * (align256(part_bytes(precision, M, 2 * K, batch)) + align256(part_bytes(precision, 2 * N, 2 * K, batch)));
}

cudaError_t launch_cgemm(int precision, long long batch, long long M, long long N, long long K, const float2 *A,
                         const float2 *B, float2 *C, void *ws, size_t ws_bytes, cudaStream_t s, const OutMap *om) {
  if (precision == TN_PREC_FP32) return launch_cgemm_fp32(batch, M, N, K, A, B, C, ws, ws_bytes, s, om);
  const OutMap ident;
  const OutMap &m = om ? *om : ident;
  if (!tc_shape_ok(precision, M, N, K)) return cudaErrorNotSupported;
  if (batch > 65535 || M / BM > 65535) return cudaErrorNotSupported;
  if (ws_bytes < cgemm_workspace(precision, batch, M, N, K)) return cudaErrorInvalidValue;
  if (precision == TN_PREC_3XTF32)
    return split_a_on_chip(precision, N, K) ? run_tc<PREC_TF32, true>(batch, M, N, K, A, B, C, ws, s, m)
                                            : run_tc<PREC_TF32, false>(batch, M, N, K, A, B, C, ws, s, m);
  return split_a_on_chip(precision, N, K) ? run_tc<PREC_BF16, true>(batch, M, N, K, A, B, C, ws, s, m)
                                          : run_tc<PREC_BF16, false>(batch, M, N, K, A, B, C, ws, s, m);
}

}  // namespace tnq
