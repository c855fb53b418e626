// FP64 reductions over the contracted state: Pauli-sum expectation values and H psi.
//
// Closing the state's open legs against an operator (Sec. 2.2.3 closes them with a basis
// state; an observable closes them with <psi| P) is a reduction over all 2^N entries:
//   <psi|P|psi> = sum_x i^ny (-1)^popc(x & zm) conj(psi[x ^ xm]) psi[x]
// for P with X/Y factors on the bits xm and Z/Y factors on zm.  Terms are grouped into
// tile passes whose tiles contain every flip bit of their terms, so each pass reads the
// state once (coalesced, staged in shared memory) and evaluates all of its terms from
// the tile.  Precision, step by step: a term's contribution and the sum over terms at one
// amplitude are FP32 (coefficients rounded to FP32); a thread's sum over its amplitudes of one
// tile (tile / 256 of them, 16 for 12-qubit tiles) is FP32; the sums across tiles, warps and
// CTAs are FP64, and the per-CTA partials are summed in a fixed order (deterministic result).
// The FP32 steps add at most about (terms + tile/256) 2^-24 sum_k |c_k| <ps|ps> to the result
// (about 1e-5 absolute for the 39 unit terms of a 20-qubit Ising chain); FP64 takes over where
// the long sums and their cancellation are, over the 2^N / 16 per-thread partials.  Doing the
// per-amplitude work in FP64 would make the pass FP64-bound on GB300 (a few FP64 operations
// per SM and clock) instead of HBM-bound.
#include <algorithm>

#include "apply_common.cuh"
#include "kernels.h"

namespace tnq {

constexpr int kRedThreads = 256;
constexpr int kRedGroup = 8;  // rows (amplitudes tid + 256 j) a thread holds in registers at once, of up to 16
constexpr int kRedCtas = 4;    // resident CTAs per SM
constexpr int kRedMaxCTAs = 512;  // per pass and batch element

namespace {

// Shared memory of a tile: at least eight rows, so that a thread's rows beyond a small tile (never
// summed or stored) are still read from inside it.
__host__ __device__ constexpr size_t tile_bytes(int T) { return sizeof(float2) << (T < 11 ? 11 : T); }

struct TileCtx {
  int T, L, tile, lowmask;
  long long *run_off;
};

__device__ void setup_tile(const RedPass &rp, long long *run_off, TileCtx &c) {
  c.T = rp.T;
  c.L = c.T < kLowBits ? c.T : kLowBits;
  c.tile = 1 << c.T;
  c.lowmask = (1 << c.L) - 1;
  c.run_off = run_off;
  for (int r = threadIdx.x; r < (1 << (c.T - c.L)); r += blockDim.x) {
    long long off = 0;
    for (int j = 0; j < c.T - c.L; ++j)
      if ((r >> j) & 1) off |= 1ll << rp.tile_pos[c.L + j];
    run_off[r] = off;
  }
}

__device__ __forceinline__ unsigned long long tile_base(const RedPass &rp, long long t) {
  unsigned long long base = 0;
  for (int j = 0; j < rp.n_outer; ++j) base |= (unsigned long long)((t >> j) & 1) << rp.outer_pos[j];
  return base;
}

__device__ __forceinline__ void load_tile(float2 *sm, const float2 *st, unsigned long long base, const TileCtx &c) {
  for (int k = threadIdx.x; k < (c.tile >> 1); k += blockDim.x) {
    const int i = k << 1;
    const long long g = (long long)base + c.run_off[i >> c.L] + (i & c.lowmask);
    const float4 v = *reinterpret_cast<const float4 *>(st + g);
    sm[swz(i)] = make_float2(v.x, v.y);
    sm[swz(i + 1)] = make_float2(v.z, v.w);
  }
}

__device__ __forceinline__ double block_sum(double v, double *scratch) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) scratch[warp] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += scratch[w];
  __syncthreads();
  return s;
}

}  // namespace

// A term of a pass as the tile loop reads it: shared-memory copies with the tile-local Z mask (zl) and
// flips (xl), and per tile the coefficient with the sign of the tile's outer bits (cs).
struct alignas(16) TermSm {
  float cs;
  int zl;
  int xl_ny;  // xl | (ny mod 4) << 16
  float coef;
};
static_assert(sizeof(TermSm) == 16, "TermSm layout");

// A term's sign at amplitude i = tid + 256 J is the product of three parities: the tile's outer bits
// (in cs), the thread's bits (one popc per term and thread) and the row's, popc(J & m), m = zl >> 8.
// The rows of a term are one of a few unrolled forms, chosen by m (the same for all threads), with the
// row signs in the operands: a term costs a row one multiply-add (two rows per packed FP32x2
// instruction) and no integer work, and its other instructions are shared by 16 or 8 rows.  Every
// amplitude still sums its terms in term order and a thread its amplitudes in index order.
// Bound: instruction issue (63% of slots; ALU and FMA pipes about half busy), not HBM.  Measured
// before and after: 22-qubit Heisenberg energies of four states (85 terms, three passes) 794 and
// 330 us; 20-qubit Ising H psi of 64 states (39 terms, two passes) 2.64 and 1.3 ms.
using u64 = unsigned long long;
__device__ __forceinline__ u64 pk(float lo, float hi) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 up(u64 v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return make_float2(lo, hi);
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float flip_sign(float v, unsigned parity) {
  return __uint_as_float(__float_as_uint(v) ^ (parity << 31));
}
constexpr bool parity4(int v) { return ((v ^ (v >> 1) ^ (v >> 2) ^ (v >> 3)) & 1) != 0; }
// s[row pair] += (+-c, +-c) z[row pair], signs popc(j & M)
template <int M, int PAIRS>
__device__ __forceinline__ void rows_real(u64 (&s)[8], const u64 (&z)[PAIRS], float c, int first = 0) {
  const u64 p = pk(c, (M & 1) ? -c : c), n = pk(-c, (M & 1) ? c : -c);
#pragma unroll
  for (int q = 0; q < PAIRS; ++q) s[first + q] = fma2(parity4(2 * q & M) ? n : p, z[q], s[first + q]);
}
// s[row] += (+-p) w[row] on (re, im) pairs, w the eight rows in shared memory at byte address a0 ^ 8 swz(256 j)
template <int M, bool SWAP>
__device__ __forceinline__ void rows_pair(u64 (&s)[kRedGroup], const unsigned char *sm, int a0, float cx, float cy) {
  const u64 p = pk(cx, cy), n = pk(-cx, -cy);
#pragma unroll
  for (int j = 0; j < kRedGroup; ++j) {
    const float2 w = *reinterpret_cast<const float2 *>(sm + (a0 ^ (8 * swz(j << 8))));
    s[j] = fma2(parity4(j & M) ? n : p, SWAP ? pk(w.y, w.x) : pk(w.x, w.y), s[j]);
  }
}
template <int M>
__device__ __forceinline__ void rows_own(u64 (&s)[kRedGroup], const u64 (&v)[kRedGroup], float c) {
  const u64 p = pk(c, c), n = pk(-c, -c);
#pragma unroll
  for (int j = 0; j < kRedGroup; ++j) s[j] = fma2(parity4(j & M) ? n : p, v[j], s[j]);
}
#define TNQ_FORMS_8(m, call) \
  switch (m) {               \
    case 0: call(0); break;  \
    case 1: call(1); break;  \
    case 2: call(2); break;  \
    case 3: call(3); break;  \
    case 4: call(4); break;  \
    case 5: call(5); break;  \
    case 6: call(6); break;  \
    default: call(7); break; \
  }
#define TNQ_FORMS_16(m, call)  \
  switch (m) {                 \
    case 1: call(1); break;    \
    case 2: call(2); break;    \
    case 3: call(3); break;    \
    case 4: call(4); break;    \
    case 5: call(5); break;    \
    case 6: call(6); break;    \
    case 7: call(7); break;    \
    case 8: call(8); break;    \
    case 9: call(9); break;    \
    case 10: call(10); break;  \
    case 11: call(11); break;  \
    case 12: call(12); break;  \
    case 13: call(13); break;  \
    case 14: call(14); break;  \
    default: call(15); break;  \
  }

__device__ __forceinline__ int compress_bits(unsigned long long v, const RedPass &rp) {
  int r = 0;
  for (int j = 0; j < rp.T; ++j) r |= (int)((v >> rp.tile_pos[j]) & 1ull) << j;
  return r;
}

__global__ void __launch_bounds__(kRedThreads, kRedCtas) k_expect_pass(const RedPass *__restrict__ passes,
                                                                       int pass_idx, int n_passes,
                                                                       const DevTerm *__restrict__ terms,
                                                                       const float2 *__restrict__ state, int N,
                                                                       double *__restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ RedPass rp;
  __shared__ double scratch[kRedThreads / 32];
  for (int i = threadIdx.x; i < (int)(sizeof(RedPass) / 4); i += blockDim.x)
    reinterpret_cast<int *>(&rp)[i] = reinterpret_cast<const int *>(passes + pass_idx)[i];
  __syncthreads();
  TileCtx c;
  float2 *sm = reinterpret_cast<float2 *>(smem_raw);
  long long *run_off = reinterpret_cast<long long *>(smem_raw + tile_bytes(rp.T));
  const int n_runs = (1 << (rp.T - (rp.T < kLowBits ? rp.T : kLowBits)));
  const int nt = rp.term_end - rp.term_begin, nd = rp.n_diag;
  TermSm *rec = reinterpret_cast<TermSm *>(run_off + (n_runs < 2 ? 2 : n_runs));
  setup_tile(rp, run_off, c);
  for (int k = threadIdx.x; k < nt; k += blockDim.x) {
    const DevTerm &tm = terms[rp.term_begin + k];
    rec[k] = TermSm{0.f, compress_bits(tm.zm, rp), tm.xl | ((tm.ny & 3) << 16), (float)tm.coef};
  }
  __syncthreads();
  const int b = blockIdx.y, tid = threadIdx.x;
  const float2 *st = state + ((long long)b << N);
  const long long n_tiles = 1ll << rp.n_outer;
  const int nj = c.tile < kRedThreads ? 1 : c.tile / kRedThreads;
  const bool live = tid < c.tile;
  double acc = 0.0;
  for (long long t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    const unsigned long long base = tile_base(rp, t);
    for (int k = threadIdx.x; k < nt; k += blockDim.x)
      rec[k].cs = flip_sign(rec[k].coef, (unsigned)__popcll(base & terms[rp.term_begin + k].zm) & 1u);
    load_tile(sm, st, base, c);
    __syncthreads();
    float tacc = 0.f;
    if (live) {
      u64 sacc[8];  // the sums of rows 2 q, 2 q + 1
#pragma unroll
      for (int q = 0; q < 8; ++q) sacc[q] = 0ull;
      const int s0 = swz(tid);
      if (nd > 0) {  // terms without flips, all 16 rows at once
        u64 z[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          float2 a = make_float2(0.f, 0.f), e = a;
          if (2 * q < kRedGroup || nj > kRedGroup) {
            a = sm[s0 ^ swz((2 * q) << 8)];
            e = sm[s0 ^ swz((2 * q + 1) << 8)];
          }
          z[q] = pk(fmaf(a.x, a.x, a.y * a.y), fmaf(e.x, e.x, e.y * e.y));
        }
        for (int k = 0; k < nd; ++k) {
          const float2 r = *reinterpret_cast<const float2 *>(rec + k);  // (cs, zl)
          const int zl = __float_as_int(r.y);
          const float cs = flip_sign(r.x, (unsigned)__popc(tid & zl));
          if (zl < 256) {
            rows_real<0>(sacc, z, cs);
          } else {
#define TNQ_CALL(M) rows_real<M>(sacc, z, cs)
            TNQ_FORMS_16(zl >> 8, TNQ_CALL)
#undef TNQ_CALL
          }
        }
      }
#pragma unroll
      for (int g = 0; g < 2; ++g) {  // the others, eight rows at a time
        if (nd == nt || g * kRedGroup >= nj) continue;
        const int sg = s0 ^ swz((g * kRedGroup) << 8);
        float2 v[kRedGroup];
        u64 z[kRedGroup / 2];
#pragma unroll
        for (int j = 0; j < kRedGroup; ++j) v[j] = sm[sg ^ swz(j << 8)];
        int have = 0;  // what z holds: the flips, and bit 16 for the imaginary parts
        for (int k = nd; k < nt; ++k) {
          const TermSm tm = rec[k];
          const int zl = tm.zl, ny = tm.xl_ny >> 16, want = tm.xl_ny & 0x1FFFF;
          if (want != have) {  // one part of conj(w) v of the partners w, kept for the next terms of these flips
            have = want;
            const int sx = sg ^ swz(want & 0xFFFF);
            const bool im = (ny & 1) != 0;
#pragma unroll
            for (int q = 0; q < kRedGroup / 2; ++q) {
              const float2 w0 = sm[sx ^ swz((2 * q) << 8)], w1 = sm[sx ^ swz((2 * q + 1) << 8)];
              const float2 v0 = v[2 * q], v1 = v[2 * q + 1];
              z[q] = im ? pk(fmaf(w0.x, v0.y, -w0.y * v0.x), fmaf(w1.x, v1.y, -w1.y * v1.x))
                        : pk(fmaf(w0.x, v0.x, w0.y * v0.y), fmaf(w1.x, v1.x, w1.y * v1.y));
            }
          }
          // Re(i^ny z): z.x, -z.y, -z.x, z.y
          const unsigned p = (unsigned)__popc(tid & zl) ^ (unsigned)((ny + 1) >> 1) ^ (unsigned)(g ? zl >> 11 : 0);
          const float cs = flip_sign(tm.cs, p);
          if ((zl & 0x700) == 0) {
            rows_real<0>(sacc, z, cs, g * (kRedGroup / 2));
          } else {
#define TNQ_CALL(M) rows_real<M>(sacc, z, cs, g * (kRedGroup / 2))
            TNQ_FORMS_8((zl >> 8) & 7, TNQ_CALL)
#undef TNQ_CALL
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float2 a = up(sacc[q]);
        if (2 * q < nj) tacc += a.x;
        if (2 * q + 1 < nj) tacc += a.y;
      }
    }
    acc += (double)tacc;
    __syncthreads();
  }
  const double tot = block_sum(acc, scratch);
  if (threadIdx.x == 0) part[((long long)b * n_passes + pass_idx) * kRedMaxCTAs + blockIdx.x] = tot;
}

// out[b] = sum over passes and CTAs of the partials (fixed order).
__global__ void k_expect_final(const double *__restrict__ part, int n_passes, int gx, double *__restrict__ out) {
  __shared__ double scratch[kRedThreads / 32];
  const int b = blockIdx.x;
  double v = 0.0;
  for (int k = threadIdx.x; k < n_passes * gx; k += blockDim.x) {
    const int p = k / gx, x = k % gx;
    v += part[((long long)b * n_passes + p) * kRedMaxCTAs + x];
  }
  const double tot = block_sum(v, scratch);
  if (threadIdx.x == 0) out[b] = tot;
}

// lam (+)= (sum of the pass's terms) psi, lam[x] = sum_t c_t i^ny (-1)^popc((x^xm)&zm) psi[x^xm].
// With dot != NULL (the last pass) the CTA also sums Re conj(psi[x]) lam[x] over its amplitudes:
// <psi|H|psi> from the finished lam, in the precision steps of k_expect_pass (the product and a
// thread's sum over its amplitudes of one tile FP32, the rest FP64), into dot[b][blockIdx.x].
__global__ void __launch_bounds__(kRedThreads, kRedCtas) k_hamiltonian_pass(const RedPass *__restrict__ passes,
                                                                            int pass_idx,
                                                                            const DevTerm *__restrict__ terms,
                                                                            const float2 *__restrict__ psi,
                                                                            float2 *__restrict__ lam, int N,
                                                                            int accumulate, double *__restrict__ dot) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ RedPass rp;
  __shared__ double scratch[kRedThreads / 32];
  for (int i = threadIdx.x; i < (int)(sizeof(RedPass) / 4); i += blockDim.x)
    reinterpret_cast<int *>(&rp)[i] = reinterpret_cast<const int *>(passes + pass_idx)[i];
  __syncthreads();
  TileCtx c;
  float2 *sm = reinterpret_cast<float2 *>(smem_raw);
  long long *run_off = reinterpret_cast<long long *>(smem_raw + tile_bytes(rp.T));
  const int n_runs = (1 << (rp.T - (rp.T < kLowBits ? rp.T : kLowBits)));
  const int nt = rp.term_end - rp.term_begin, nd = rp.n_diag;
  TermSm *rec = reinterpret_cast<TermSm *>(run_off + (n_runs < 2 ? 2 : n_runs));
  setup_tile(rp, run_off, c);
  for (int k = threadIdx.x; k < nt; k += blockDim.x) {
    const DevTerm &tm = terms[rp.term_begin + k];
    rec[k] = TermSm{0.f, compress_bits(tm.zm, rp), tm.xl | ((tm.ny & 3) << 16), (float)tm.coef};
  }
  __syncthreads();
  const int b = blockIdx.y, tid = threadIdx.x;
  const float2 *st = psi + ((long long)b << N);
  float2 *lt = lam + ((long long)b << N);
  const long long n_tiles = 1ll << rp.n_outer;
  const int nj = c.tile < kRedThreads ? 1 : c.tile / kRedThreads;
  const bool live = tid < c.tile;
  double acc = 0.0;
  for (long long t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    const unsigned long long base = tile_base(rp, t);
    // parity of the Z mask on the outer bits; x ^ xm has the same outer bits as x
    for (int k = threadIdx.x; k < nt; k += blockDim.x)
      rec[k].cs = flip_sign(rec[k].coef, (unsigned)__popcll(base & terms[rp.term_begin + k].zm) & 1u);
    load_tile(sm, st, base, c);
    __syncthreads();
    float tacc = 0.f;
    for (int j0 = 0; j0 < nj && live; j0 += kRedGroup) {
      const int s0 = swz(tid + (j0 << 8));
      u64 v[kRedGroup], sacc[kRedGroup];
#pragma unroll
      for (int j = 0; j < kRedGroup; ++j) {
        const int i = tid + ((j0 + j) << 8);
        const float2 a = sm[s0 ^ swz(j << 8)];
        v[j] = pk(a.x, a.y);
        sacc[j] = 0ull;
        if (accumulate && j0 + j < nj) {
          const float2 o = lt[base + (unsigned long long)c.run_off[i >> c.L] + (unsigned long long)(i & c.lowmask)];
          sacc[j] = pk(o.x, o.y);
        }
      }
      for (int k = 0; k < nd; ++k) {  // terms without flips scale the thread's own amplitudes
        const float2 r = *reinterpret_cast<const float2 *>(rec + k);  // (cs, zl)
        const int zl = __float_as_int(r.y);
        const float cs = flip_sign(r.x, (unsigned)__popc(tid & zl) ^ (j0 ? (unsigned)zl >> 11 : 0u));
        if ((zl & 0x700) == 0) {
          rows_own<0>(sacc, v, cs);
        } else {
#define TNQ_CALL(M) rows_own<M>(sacc, v, cs)
          TNQ_FORMS_8((zl >> 8) & 7, TNQ_CALL)
#undef TNQ_CALL
        }
      }
      for (int k = nd; k < nt; ++k) {
        const TermSm tm = rec[k];
        const int zl = tm.zl, xl = tm.xl_ny & 0xFFFF, ny = tm.xl_ny >> 16;
        const int a0 = 8 * (s0 ^ swz(xl));
        // sign of the index read, i ^ x; i^ny = (-1)^(ny / 2) i^(ny mod 2)
        const unsigned p = (unsigned)__popc((tid ^ xl) & zl) ^ (unsigned)(ny >> 1) ^ (j0 ? (unsigned)zl >> 11 : 0u);
        const float cs = flip_sign(tm.cs, p);
        if ((zl & 0x700) == 0 && (ny & 1) == 0) {
          rows_pair<0, false>(sacc, smem_raw, a0, cs, cs);
        } else if (ny & 1) {  // i c w = (-c w.y, c w.x)
#define TNQ_CALL(M) rows_pair<M, true>(sacc, smem_raw, a0, -cs, cs)
          TNQ_FORMS_8((zl >> 8) & 7, TNQ_CALL)
#undef TNQ_CALL
        } else {
#define TNQ_CALL(M) rows_pair<M, false>(sacc, smem_raw, a0, cs, cs)
          TNQ_FORMS_8((zl >> 8) & 7, TNQ_CALL)
#undef TNQ_CALL
        }
      }
#pragma unroll
      for (int j = 0; j < kRedGroup; ++j) {
        if (j0 + j >= nj) break;
        const int i = tid + ((j0 + j) << 8);
        const float2 o = up(sacc[j]);
        lt[base + (unsigned long long)c.run_off[i >> c.L] + (unsigned long long)(i & c.lowmask)] = o;
        if (dot) {
          const float2 a = up(v[j]);
          tacc = fmaf(a.x, o.x, fmaf(a.y, o.y, tacc));
        }
      }
    }
    acc += (double)tacc;
    __syncthreads();
  }
  if (dot) {
    const double tot = block_sum(acc, scratch);
    if (threadIdx.x == 0) dot[(long long)b * kRedMaxCTAs + blockIdx.x] = tot;
  }
}

namespace {
size_t red_smem(const RedPass &rp) {
  const int T = rp.T;
  const int L = T < kLowBits ? T : kLowBits;
  const size_t runs = ((size_t)1 << (T - L)) < 2 ? 2 : ((size_t)1 << (T - L));
  const size_t nt = (size_t)(rp.term_end - rp.term_begin);
  return tile_bytes(T) + runs * sizeof(long long) + nt * sizeof(TermSm);
}
// CTAs per batch element of one pass: kRedCtas per SM or what its shared memory allows, spread over the batch
int red_grid_x(const tn_observable *o, int pass, int batch) {
  const RedPass &rp = o->passes[pass];
  const long long per_sm =
      std::max<long long>(1, std::min<long long>(kRedCtas, (227 * 1024) / (long long)(red_smem(rp) + 2048)));
  return (int)std::min<long long>(kRedMaxCTAs, grid_per_row(1ll << rp.n_outer, batch, (int)per_sm));
}
}  // namespace

size_t observable_partials(const tn_observable *o, int batch) {
  return (size_t)batch * o->passes.size() * kRedMaxCTAs;
}

cudaError_t launch_expectation(const tn_observable *o, int batch, const float2 *state, double *part, double *out,
                               cudaStream_t s) {
  const int np = (int)o->passes.size();
  if (np == 0) return cudaMemsetAsync(out, 0, sizeof(double) * batch, s);
  // one grid for all passes (their tiles have one size): every partial the final sum reads is written
  int gx = kRedMaxCTAs;
  for (int p = 0; p < np; ++p) {
    cudaError_t e = ensure_smem((const void *)k_expect_pass, red_smem(o->passes[p]));
    if (e != cudaSuccess) return e;
    gx = std::min(gx, red_grid_x(o, p, batch));
  }
  for (int p = 0; p < np; ++p) {
    dim3 grid((unsigned)gx, (unsigned)batch);
    k_expect_pass<<<grid, kRedThreads, red_smem(o->passes[p]), s>>>(o->d_passes, p, np, o->d_terms, state, o->n,
                                                                     part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  k_expect_final<<<batch, kRedThreads, 0, s>>>(part, np, gx, out);
  return cudaGetLastError();
}

cudaError_t launch_apply_hamiltonian(const tn_observable *o, int batch, const float2 *psi, float2 *lam,
                                     cudaStream_t s, double *part, double *out) {
  const int np = (int)o->passes.size();
  if (np == 0) {
    cudaError_t e = cudaMemsetAsync(lam, 0, (sizeof(float2) << o->n) * batch, s);
    if (e == cudaSuccess && out) e = cudaMemsetAsync(out, 0, sizeof(double) * batch, s);
    return e;
  }
  int gx_last = 1;
  for (int p = 0; p < np; ++p) {
    const size_t smem = red_smem(o->passes[p]);
    cudaError_t e = ensure_smem((const void *)k_hamiltonian_pass, smem);
    if (e != cudaSuccess) return e;
    const int gx = red_grid_x(o, p, batch);
    double *dot = (out && p == np - 1) ? part : nullptr;
    dim3 grid((unsigned)gx, (unsigned)batch);
    k_hamiltonian_pass<<<grid, kRedThreads, smem, s>>>(o->d_passes, p, o->d_terms, psi, lam, o->n, p > 0 ? 1 : 0,
                                                       dot);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    gx_last = gx;
  }
  if (out) {  // every CTA of the last pass wrote its partial: no clearing needed
    k_expect_final<<<batch, kRedThreads, 0, s>>>(part, 1, gx_last, out);
    return cudaGetLastError();
  }
  return cudaSuccess;
}

}  // namespace tnq
