// Kernel (c), plain FP32 form: batched complex GEMM on the CUDA cores.
//
// A pairwise merge of two tensors, once their legs are grouped into row, contracted and
// column indices, is the matrix product of Eq. 2.2: C[m][n] = sum_k A[m][k] B[n][k]
// (both operands stored with the contracted index contiguous).  This kernel is the FP32
// reference the tensor-core forms are measured against, and the form used for merges too
// narrow for the tensor-core tiles.  One template covers the shapes a network contraction
// produces: a CTA of 128 threads computes a BM x BN tile in TM x TN complex blocks per thread,
// streaming 16-deep slices of K of both operands through shared memory, with FFMA accumulation.
#include <algorithm>
#include <cstring>
#include <vector>

#include "kernels.h"

namespace tnq {

namespace {

constexpr int kThreads = 128;  // of a tile's CTA

// An output map as runs: the natural index's bits lo[i] .. lo[i + 1] - 1 are stored from pos[i] up.  In bytes:
// it is a parameter of every launch, and the launches are what a network of small merges spends its time on
// (3 x 6 grid of depth 8, one bitstring, eager calls: 48.5 us with runs of three ints, 772 bytes in all, and 44.5).
struct MapRuns {
  uint8_t n, lo[64], pos[64];
};
static_assert(sizeof(MapRuns) == 129, "small as a kernel parameter");
MapRuns runs_of(const OutMap &om) {
  MapRuns m;
  int n = 0;
  if (om.identity) m.lo[n] = m.pos[n] = 0, ++n;
  for (int i = 0; !om.identity && i < om.nbits; ++i)
    if (i == 0 || om.pos[i] != om.pos[i - 1] + 1) m.lo[n] = (uint8_t)i, m.pos[n] = om.pos[i], ++n;
  m.n = (uint8_t)n;
  m.lo[n] = 63;  // a natural index has fewer bits
  return m;
}
__device__ __forceinline__ long long map_runs(const MapRuns &m, long long f) {
  long long r = 0;
  for (int i = 0; i < m.n; ++i) r += ((f >> m.lo[i]) & ((1ll << (m.lo[i + 1] - m.lo[i])) - 1)) << m.pos[i];
  return r;
}

// An output map with its permuted epilogue for one tile shape.  The tile's valid local bits are enumerated
// by increasing stored position as the bits of u: s[k] and g[k] are the staging and stored offsets of u's
// bit k.
constexpr int kTileBits = 12;
struct StagedMap {
  int identity;
  int lgn, L, pairs;
  int s[kTileBits];
  long long g[kTileBits];
  MapRuns runs;
};
void build_staged(StagedMap &sm, const OutMap &om, long long M, long long N, int BM, int BN);

// Output index of natural flat index bits [lo, nbits) of f under the map (0 for identity).
__device__ __forceinline__ long long map_bits(const OutMap &om, long long f, int lo) {
  long long r = 0;
  for (int i = lo; i < om.nbits; ++i)
    if ((f >> i) & 1) r |= 1ll << om.pos[i];
  return r;
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Permuted output: the tile staged in shared memory (smem, written by the caller, not yet synchronised)
// goes back in stored-index order, two elements of u a thread and step.  A thread's offsets are sums over
// the bits of its index, found once, and of the step; tables of them in shared memory took six loads for
// every two elements, and a loop over all bits of the map for the tile's own offset (f: its natural index)
// as many instructions as a tenth of an 8-column tile's.
template <int THREADS>
__device__ __forceinline__ void store_staged(const float2 *smem, float2 *__restrict__ C, long long f,
                                             const StagedMap &om) {
  constexpr int kLane = THREADS == 128 ? 7 : -1;
  static_assert(kLane > 0, "bits of the thread index");
  float2 *c = C + map_runs(om.runs, f);
  int at = 0;
#pragma unroll
  for (int k = 0; k < kLane; ++k)
    if ((threadIdx.x >> k) & 1) at += om.s[k + 1], c += om.g[k + 1];
  __syncthreads();
  if (om.L == 0) {
    if (threadIdx.x == 0) c[0] = smem[0];
    return;
  }
  if (threadIdx.x >> (om.L - 1)) return;  // a tile of fewer than two elements per thread
  const int steps = om.L > kLane + 1 ? 1 << (om.L - kLane - 1) : 1;
  for (int it = 0; it < steps; ++it) {
    int s = at;
    float2 *dst = c;
#pragma unroll
    for (int k = 0; k < kTileBits - kLane - 1; ++k)
      if ((it >> k) & 1) s += om.s[kLane + 1 + k], dst += om.g[kLane + 1 + k];
    const float2 x0 = smem[s], x1 = smem[s + om.s[0]];
    if (om.pairs) {  // adjacent in memory
      *reinterpret_cast<float4 *>(dst) = make_float4(x0.x, x0.y, x1.x, x1.y);
    } else {
      dst[0] = x0;
      dst[om.g[0]] = x1;
    }
  }
}

// Tiles: the columns fitted to N (8, 16, 32 or 64), the rows by short_tiles.  Bound: FMA issue, and for
// narrow N the loads of A beside it.  Before, 256 threads of 2 x 2 to 4 x 4 accumulators copied the slices
// 8 bytes at a time: the copies' address arithmetic and one shared-memory load for every four multiply-adds
// took more issue slots than the multiply-adds.  128 threads, 16-byte copies and 4 x 2 to 8 x 4 accumulators,
// four CTAs per SM or more: batch 64, 32768 x 8 x 64: 333 -> 253 us; x 16: 488 -> 364; x 32: 894 -> 612;
// 4096 x 64 x 64: 204 -> 156; 4096^3 11.9 -> 9.2 ms (59.6 TFLOP/s).  Slower at 4096^3: 128 x 64 tiles of
// 8 x 8 (9.6 ms; two CTAs per SM leave a worse last wave too: 2048^3 1394 against 1217 us), two steps of K
// per shared-memory load (9.3, spills), three slices in flight (9.8), and packed FP32x2 multiply-adds, with
// the operands duplicated in registers (39.5 against 57.9 TFLOP/s at 2432 x 2048 x 512) or laid out in pairs
// in shared memory (11.2 ms).
// Slices of 16 K are staged by cp.async, two in flight, in rows of 18 elements (16-byte aligned, a
// warp's reads conflict-free); VEC: 16-byte copies, for even K.  Four steps of K are unrolled.
constexpr int kSliceK = 16, kLd = kSliceK + 2, kStages = 2;
template <int BM, int BN>
constexpr size_t tile_smem() {
  constexpr int slices = kStages * (BM + BN) * kLd, tile = BM * (BN + 1);
  return sizeof(float2) * (slices > tile ? slices : tile);
}

// asynchronous copy of the first n of BYTES bytes, the rest zeros
template <int BYTES>
__device__ __forceinline__ void cp_async_z(void *dst, const void *src, int n) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(BYTES), "r"(n)
               : "memory");
}

template <bool VEC, bool SPLIT, int BM, int BN, int TM, int TN, int MINB>
__global__ void __launch_bounds__(kThreads, MINB) k_cgemm_fp32(long long M, long long N, long long K, long long k_len,
                                                            const float2 *__restrict__ A, const float2 *__restrict__ B,
                                                            float2 *__restrict__ C, float2 *__restrict__ P,
                                                            const __grid_constant__ StagedMap om) {
  static_assert((BM / TM) * (BN / TN) == kThreads, "one thread per TM x TN block");
  static_assert(BM * BN <= 1 << kTileBits, "StagedMap covers a tile");
  constexpr int NX = BN / TN, NY = BM / TM, kSlice = (BM + BN) * kLd;
  extern __shared__ __align__(16) float2 smem[];
  pdl_wait();
  pdl_trigger();
  // tiles of one batch element along x, n fastest (M may need more than 65535 row tiles)
  const long long tiles_n = (N + BN - 1) / BN;
  const long long b = blockIdx.z;
  const long long m0 = ((long long)blockIdx.x / tiles_n) * BM, n0 = ((long long)blockIdx.x % tiles_n) * BN;
  // SPLIT: this CTA sums k in [kb, ke) and stores its partial tile to P
  const long long kb = SPLIT ? (long long)blockIdx.y * k_len : 0, ke = SPLIT && kb + k_len < K ? kb + k_len : K;
  const float2 *Ab = A + (b * M + m0) * K, *Bb = B + (b * N + n0) * K;
  constexpr int kPer = VEC ? 2 : 1;        // elements per copy
  constexpr int kCols = kSliceK / kPer;    // copies per row
  constexpr int kStep = kThreads / kCols;  // rows copied at once
  const int lr = threadIdx.x / kCols, lc = (threadIdx.x % kCols) * kPer;
  const int rows_a = (int)(M - m0 < BM ? M - m0 : BM), rows_b = (int)(N - n0 < BN ? N - n0 : BN);
  // `most` rows of a slice of one operand: elements in range, zeros for the ragged edges
  auto load_rows = [&](float2 *dst, const float2 *src, const float2 *base, int rows, int most, bool in_k) {
#pragma unroll
    for (int r = lr; r < most; r += kStep) {
      const bool ok = in_k && r < rows;
      cp_async_z<8 * kPer>(dst + r * kLd + lc, ok ? src + r * K : base, ok ? 8 * kPer : 0);
    }
  };
  auto load_slice = [&](int sb, long long k0) {
    float2 *as = smem + sb * kSlice;
    load_rows(as, Ab + k0 + lc, A, rows_a, BM, k0 + lc < ke);
    load_rows(as + BM * kLd, Bb + k0 + lc, B, rows_b, BN, k0 + lc < ke);
  };
  const int tx = threadIdx.x % NX, ty = threadIdx.x / NX;
  float2 acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.f, 0.f);
  const int slices = (int)((ke - kb + kSliceK - 1) / kSliceK);
  if (slices > 0) load_slice(0, kb);
  cp_async_commit();
  for (int t = 0; t < slices; ++t) {
    cp_async_wait<kStages - 2>();
    __syncthreads();  // slice t has landed, and its successor's buffer (slice t - 1) is read out
    const long long k0 = kb + (long long)t * kSliceK;
    if (t + 1 < slices) load_slice((t + 1) % kStages, k0 + kSliceK);
    cp_async_commit();
    const float2 *as = smem + (t % kStages) * kSlice + ty * kLd;
    const float2 *bs = smem + (t % kStages) * kSlice + (BM + tx) * kLd;
    const int quads = ke - k0 >= kSliceK ? kSliceK / 4 : (int)(ke - k0 + 3) / 4;
#pragma unroll 1
    for (int q = 0; q < quads; ++q, as += 4, bs += 4)
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float2 bb[TN];
#pragma unroll
      for (int j = 0; j < TN; ++j) bb[j] = bs[NX * j * kLd + kk];
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float2 a = as[NY * i * kLd + kk];
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          acc[i][j].x = fmaf(a.x, bb[j].x, acc[i][j].x);
          acc[i][j].y = fmaf(a.x, bb[j].y, acc[i][j].y);
          acc[i][j].x = fmaf(-a.y, bb[j].y, acc[i][j].x);
          acc[i][j].y = fmaf(a.y, bb[j].x, acc[i][j].y);
        }
      }
    }
  }
  if (SPLIT || om.identity) {
    float2 *O = SPLIT ? P + ((long long)blockIdx.y * gridDim.z + b) * M * N : C + b * M * N;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const long long gm = m0 + ty + NY * i, gn = n0 + tx + NX * j;
        if (gm < M && gn < N) O[gm * N + gn] = acc[i][j];
      }
  } else {
    __syncthreads();  // the last slice is read out; nothing is in flight
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) smem[(ty + NY * i) * (BN + 1) + tx + NX * j] = acc[i][j];
    store_staged<kThreads>(smem, C, ((b * M + m0) << om.lgn) | n0, om);
  }
}

// Small merges (at most 2^18 complex multiply-adds, K <= 64; most merges of small circuits):
// one thread per output element reads its K-contiguous rows of A and B straight from global
// memory (cache-resident at this size) and stores through the output map, without tile
// staging.  The accumulation over k is the tiled kernel's (same order, same fused
// multiply-adds), so both give the same bits.
// The map goes bit by bit where there are few elements and so few bits (a run's shifts and loads take longer
// than two bits': 3 x 3 grid of depth 6, replayed from a graph, 13.0 us, 13.9 with runs), in runs where there are many.
__device__ __forceinline__ long long stored(const MapRuns &om, long long f) { return map_runs(om, f); }
__device__ __forceinline__ long long stored(const OutMap &om, long long f) { return om.identity ? f : map_bits(om, f, 0); }
template <class Map>
__global__ void __launch_bounds__(256) k_cgemm_small(long long M, long long N, long long K, long long total,
                                                     const float2 *__restrict__ A, const float2 *__restrict__ B,
                                                     float2 *__restrict__ C, const __grid_constant__ Map om) {
  pdl_wait();
  pdl_trigger();
  for (long long f = (long long)blockIdx.x * blockDim.x + threadIdx.x; f < total;
       f += (long long)gridDim.x * blockDim.x) {
    const long long n = f % N, bm = f / N;  // bm = b M + m
    const long long b = bm / M;
    const float2 *a = A + bm * K;
    const float2 *w = B + (b * N + n) * K;
    float2 acc = make_float2(0.f, 0.f);
    for (long long k = 0; k < K; ++k) {
      const float2 x = a[k], y = w[k];
      acc.x = fmaf(x.x, y.x, acc.x);
      acc.x = fmaf(-x.y, y.y, acc.x);
      acc.y = fmaf(x.x, y.y, acc.y);
      acc.y = fmaf(x.y, y.x, acc.y);
    }
    C[stored(om, f)] = acc;
  }
}
constexpr long long kSmallWork = 1ll << 18;
constexpr long long kFewElements = 1ll << 14;

// Sum of the split-K partials (in split order) of every output element, stored through the
// output map: C[map(f)] = sum_s P[s][f], f the natural index (b M + m) N + n.
__global__ void k_splitk_reduce(const float2 *__restrict__ P, int splits, long long total, float2 *__restrict__ C,
                                const __grid_constant__ OutMap om) {
  pdl_wait();
  pdl_trigger();
  for (long long f = (long long)blockIdx.x * blockDim.x + threadIdx.x; f < total;
       f += (long long)gridDim.x * blockDim.x) {
    float2 acc = P[f];
    for (int s = 1; s < splits; ++s) {
      const float2 v = P[(long long)s * total + f];
      acc.x += v.x;
      acc.y += v.y;
    }
    C[om.identity ? f : map_bits(om, f, 0)] = acc;
  }
}

// The same sum for few outputs: one block of 128 threads per output element strides over the
// splits, then a fixed tree (warp shuffles, then the four warp sums in order).
__global__ void k_splitk_reduce_few(const float2 *__restrict__ P, int splits, long long total, float2 *__restrict__ C,
                                    const __grid_constant__ OutMap om) {
  pdl_wait();
  pdl_trigger();
  const long long f = blockIdx.x;
  float2 acc = make_float2(0.f, 0.f);
  for (int s = threadIdx.x; s < splits; s += blockDim.x) {
    const float2 v = P[(long long)s * total + f];
    acc.x += v.x;
    acc.y += v.y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    acc.x += __shfl_down_sync(0xffffffffu, acc.x, o);
    acc.y += __shfl_down_sync(0xffffffffu, acc.y, o);
  }
  __shared__ float2 warp_sum[4];
  if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float2 r = warp_sum[0];
    for (int w = 1; w < 4; ++w) {
      r.x += warp_sum[w].x;
      r.y += warp_sum[w].y;
    }
    C[om.identity ? f : map_bits(om, f, 0)] = r;
  }
}

// The permuted epilogue for one tile shape (built on the host once per launch): the tile's valid local
// bits are vc column bits, then vr row bits.
void build_staged(StagedMap &sm, const OutMap &om, long long M, long long N, int BM, int BN) {
  int lgn = 0, lgm = 0, lbn = 0, lbm = 0;
  while ((1ll << lgn) < N) ++lgn;
  while ((1ll << lgm) < M) ++lgm;
  while ((1 << lbn) < BN) ++lbn;
  while ((1 << lbm) < BM) ++lbm;
  const int vc = std::min(lbn, lgn), vr = std::min(lbm, lgm);
  sm.lgn = lgn;
  sm.L = vc + vr;
  std::vector<int> order((size_t)sm.L);
  for (int k = 0; k < sm.L; ++k) order[(size_t)k] = k;
  auto spos = [&](int k) { return (int)(k < vc ? om.pos[k] : om.pos[lgn + k - vc]); };
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return spos(a) < spos(b); });
  for (int k = 0; k < sm.L; ++k) {
    const int b = order[(size_t)k];
    sm.s[k] = b < vc ? 1 << b : (BN + 1) << (b - vc);
    sm.g[k] = 1ll << spos(b);
  }
  sm.pairs = sm.L > 0 && sm.g[0] == 1;
  sm.runs = runs_of(om);
}

// Tile shape (BM x BN) by which an output of N columns is counted: the split of K and the planner's tile fill.
inline void tile_for(long long N, int *bm, int *bn) {
  *bn = N <= 8 ? 8 : N <= 16 ? 16 : N <= 32 ? 32 : 64;
  *bm = *bn == 64 ? 64 : 128;
}

// Split K: an output of few tiles with a long K (a merge that contracts most of two large
// operands into a small result) would leave most SMs idle and one CTA looping over K; K is
// then cut into ranges of at least 256 (a multiple of the K slice) so that about two CTAs
// per SM (152 SMs) run, each storing a partial tile, and k_splitk_reduce adds the partials.
constexpr long long kSplitTargetCtas = 2 * 152;
int split_k(long long batch, long long M, long long N, long long K, long long *k_len) {
  int bm = 0, bn = 0;
  tile_for(N, &bm, &bn);
  const long long tiles = batch * ((M + bm - 1) / bm) * ((N + bn - 1) / bn);
  *k_len = K;
  if (K < 512 || tiles >= kSplitTargetCtas) return 1;
  long long S = std::min<long long>((kSplitTargetCtas + tiles - 1) / tiles, K / 256);
  if (S <= 1) return 1;
  const int bk = K <= 8 ? 8 : 16;
  long long kl = (K + S - 1) / S;
  kl = (kl + bk - 1) / bk * bk;
  *k_len = kl;
  return (int)((K + kl - 1) / kl);
}

template <bool SPLIT, int BM, int BN, int TM, int TN, int MINB>
cudaError_t launch_tiles(long long batch, long long M, long long N, long long K, const float2 *A, const float2 *B,
                         float2 *C, float2 *P, const OutMap &om, cudaStream_t s) {
  const long long tiles = ((N + BN - 1) / BN) * ((M + BM - 1) / BM);
  if (tiles > 0x7fffffffll) return cudaErrorNotSupported;
  long long k_len = K;
  const int splits = SPLIT ? split_k(batch, M, N, K, &k_len) : 1;
  dim3 grid((unsigned)tiles, (unsigned)splits, (unsigned)batch);
  StagedMap sm;
  std::memset(&sm, 0, sizeof(sm));
  sm.identity = om.identity;
  if (!om.identity && !SPLIT) build_staged(sm, om, M, N, BM, BN);
  const bool vec = K % 2 == 0 && (((uintptr_t)A | (uintptr_t)B) & 15) == 0;
  auto *fn = vec ? k_cgemm_fp32<true, SPLIT, BM, BN, TM, TN, MINB>
                 : k_cgemm_fp32<false, SPLIT, BM, BN, TM, TN, MINB>;
  constexpr size_t bytes = tile_smem<BM, BN>();
  static_assert(bytes <= 48 * 1024, "no attribute is set");
  cudaError_t e = launch_pdl(fn, grid, dim3(kThreads), bytes, s, M, N, K, k_len, A, B, C, P, sm);
  if (e != cudaSuccess || !SPLIT) return e;
  const long long total = batch * M * N;
  if (total <= 4096)
    return launch_pdl(k_splitk_reduce_few, dim3((unsigned)total), dim3(128), 0, s, (const float2 *)P, splits, total, C,
                      om);
  return launch_pdl(k_splitk_reduce, dim3((unsigned)std::min<long long>((total + 255) / 256, 4096)), dim3(256), 0, s,
                    (const float2 *)P, splits, total, C, om);
}

// Whether 32-row tiles are faster than `rows`-row ones for `tiles` column tiles (of all batch elements):
// when the SM with the most rows has so many fewer of them that it makes up for their lower rate, `rate` of
// the larger tiles' (32768 rows, batch 64: 0.8 at 8 to 32 columns; 4096^3: 0.96, less where tiles are short).
// 2048 x 32 x 450: 53 and 20 us; 500^3: 58 and 38; 40 x 200 x 200 x 200: 92 and 76; the other way
// 1000 x 1000 x 300: 60 and 77; 32 x 2048 x 32 x 32: 14.7 and 15.7.
bool short_tiles(long long M, long long tiles, long long rows, double rate) {
  auto most = [&](long long bm) {
    const long long sms = num_sms();
    return (double)((tiles * ((M + bm - 1) / bm) + sms - 1) / sms * bm);
  };
  return most(32) < rate * most(rows);
}

}  // namespace

size_t cgemm_fp32_workspace(long long batch, long long M, long long N, long long K) {
  long long k_len = 0;
  const int splits = split_k(batch, M, N, K, &k_len);
  return splits > 1 ? (size_t)splits * (size_t)(batch * M * N) * sizeof(float2) : 0;
}

double cgemm_fp32_tile_fill(long long M, long long N) {
  int bm = 0, bn = 0;
  tile_for(N, &bm, &bn);
  const double rows = (double)M / (double)(((M + bm - 1) / bm) * bm);
  const double cols = (double)N / (double)(((N + bn - 1) / bn) * bn);
  return rows * cols;
}

cudaError_t launch_cgemm_fp32(long long batch, long long M, long long N, long long K, const float2 *A, const float2 *B,
                              float2 *C, void *ws, size_t ws_bytes, cudaStream_t s, const OutMap *om) {
  if (batch > 65535) return cudaErrorNotSupported;
  const size_t need = cgemm_fp32_workspace(batch, M, N, K);
  if (need > 0 && (ws == nullptr || ws_bytes < need)) return cudaErrorInvalidValue;
  float2 *P = need > 0 ? static_cast<float2 *>(ws) : nullptr;
  const OutMap ident;
  const OutMap &m = om ? *om : ident;
  const long long total = batch * M * N;
  // small merges, and tall narrow ones (at most four output columns, where the tiled kernel's
  // 8-column tiles would mostly compute padding) of any size: one thread per output element
  // (on the Fig. 3.1 amplitude sweep: up to 2 columns 12.1 ms per step, up to 4 12.0, up to 8
  // 13.1, none 22.4)
  if (K <= 64 && ((double)total * (double)K <= (double)kSmallWork || N <= 4)) {
    const long long blocks = std::min<long long>((total + 255) / 256, (long long)num_sms() * 16);
    if (total <= kFewElements)
      return launch_pdl(k_cgemm_small<OutMap>, dim3((unsigned)blocks), dim3(256), 0, s, M, N, K, total, A, B, C, m);
    return launch_pdl(k_cgemm_small<MapRuns>, dim3((unsigned)blocks), dim3(256), 0, s, M, N, K, total, A, B, C, runs_of(m));
  }
  if (P != nullptr) {  // few tiles: the short ones
    if (N <= 8) return launch_tiles<true, 32, 8, 2, 1, 8>(batch, M, N, K, A, B, C, P, m, s);
    if (N <= 16) return launch_tiles<true, 32, 16, 2, 2, 8>(batch, M, N, K, A, B, C, P, m, s);
    if (N <= 32) return launch_tiles<true, 32, 32, 4, 2, 8>(batch, M, N, K, A, B, C, P, m, s);
    return launch_tiles<true, 32, 64, 4, 4, 6>(batch, M, N, K, A, B, C, P, m, s);
  }
  if (N <= 8)
    return short_tiles(M, batch, 64, 0.8) ? launch_tiles<false, 32, 8, 2, 1, 8>(batch, M, N, K, A, B, C, P, m, s)
                                          : launch_tiles<false, 64, 8, 2, 2, 8>(batch, M, N, K, A, B, C, P, m, s);
  if (N <= 16)
    return short_tiles(M, batch, 128, 0.8) ? launch_tiles<false, 32, 16, 2, 2, 8>(batch, M, N, K, A, B, C, P, m, s)
                                           : launch_tiles<false, 128, 16, 4, 4, 4>(batch, M, N, K, A, B, C, P, m, s);
  if (N <= 32)
    return short_tiles(M, batch, 128, 0.8) ? launch_tiles<false, 32, 32, 4, 2, 8>(batch, M, N, K, A, B, C, P, m, s)
                                           : launch_tiles<false, 128, 32, 8, 4, 4>(batch, M, N, K, A, B, C, P, m, s);
  return short_tiles(M, batch * ((N + 63) / 64), 64, 0.92)
             ? launch_tiles<false, 32, 64, 4, 4, 6>(batch, M, N, K, A, B, C, P, m, s)
             : launch_tiles<false, 64, 64, 8, 4, 4>(batch, M, N, K, A, B, C, P, m, s);
}

}  // namespace tnq
