// Fixed-point emulation of the paper's datapath (Sec. 3: complex arithmetic in 32-bit fixed
// point with 28 bits behind the binary point, Q4.28).
//
// The state is int32 pairs (re, im) with value q / 2^28.  Every gate is quantised once,
// Uq = round(U 2^28), and applied once: each output component is the exact sum of the
// integer products (64-bit; for unitary gates on states of norm <= 1 every sum stays below
// 2^60) rounded back to Q4.28, round half up ((acc + 2^27) >> 28, an arithmetic shift), and
// saturated to the int32 range.  Integer sums are exact in any order, so the result is
// bit-for-bit reproducible.
//
// Rounding after every gate does not commute, so gates act on every amplitude strictly in
// circuit order.  What can be shared is the trip to memory: consecutive gates whose mixed
// qubits lie in one set of tile bits form a pass (q428_build), which holds a tile of 2^T
// amplitudes in shared memory and applies its gates in order; inside a pass consecutive gates
// whose mixed qubits are among four bits form a phase, in which a thread holds 16 amplitudes in
// registers.  Diagonal gates and a CNOT's control mix nothing and read any bit, of the register
// index, the thread or the tile.
//
// Bound: the widening 32-bit multiplier (the heavy half of the FMA pipe: 21.7 multiply-adds of 32 x 32 bits
// onto 64 per SM and clock, 6.82e12 a second, measured with 16 independent chains per thread) and the latency in
// front of it.  A U3 takes 11 products per amplitude pair (Gauss); a pass's memory traffic (16 bytes per
// amplitude) is shared by about 14 gates and hides behind the arithmetic of the SM's other CTAs.  24-qubit
// brickwork of depth 20 (480 U3, 230 CZ in 50 passes, 4.4e10 products: 6.5 ms at that rate): 11.2 ms, 58% of the
// rate; 34.4 ms with one launch per gate (711 launches, each at 82% of the copy bandwidth).
// Warps count for more than registers: 2, 3 and 4 CTAs of 256 threads per SM (128, 80 and 64 registers) measured
// 18.9, 13.0 and 11.3 ms; 2^11-amplitude tiles 13.4 ms (more passes), 8 amplitudes a thread 13.6 (more phases).
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <vector>

#include "apply_common.cuh"
#include "kernels.h"
#include "tnq_internal.h"

namespace tnq {

namespace {

constexpr int kQTile = 12;       // qubits per tile: 2^12 int32 pairs = 32 KB, 256 threads of 16 amplitudes
constexpr int kQCtas = 4, kQHeavyCtas = 2;  // resident CTAs per SM
constexpr int kQReg = 4;         // register bits of a phase
constexpr int kQMinQubits = 4;   // narrower states (fewer than 16 amplitudes) take one launch per gate
constexpr int kQMaxOps = 128;    // ops of one pass staged in shared memory
constexpr int kQMaxMat = 2048;   // int32 matrix entries of one pass staged in shared memory

// Forms of an op; the quantised matrix decides (zeros contribute nothing and ones map exactly:
// (2^28 v + 2^27) >> 28 = v).
enum QType : uint8_t {
  Q_ANY1 = 0,   // 2x2 on register bit a, any int32 entries (8)
  Q_G1 = 1,     // the same with entries below 2^29 (12: see gauss_entries)
  Q_V1 = 2,     // 2x2 with a real first entry (a U3), entries below 2^29 (12)
  Q_REAL1 = 3,  // real 2x2 (8)
  Q_RX1 = 4,    // real diagonal, imaginary off-diagonal (8)
  Q_X1 = 5,     // exchange of register bit b where bit a (any source; kind 255 = always) is 1
  Q_NEG = 6,    // sign flip where bits a and b (any source) are both 1
  Q_DIAG = 7,   // diagonal on bits a, b (any source): entry 2 bit(a) + bit(b), 8 entries; ones skipped
  Q_G2 = 8,     // general 4x4 on register bits a (high), b (low): 32 entries
  Q_SWAP = 9,   // exchange of register bits a and b
};
constexpr uint8_t kAlways = 255;

struct alignas(16) QOp {
  uint8_t type, a_kind, a_pos, b_kind, b_pos;
  uint8_t ones;  // Q_DIAG: bit v set when entry v is exactly one
  uint8_t pad[2];
  int32_t mat;   // first entry in the pass's table
  int32_t pad2;
};
static_assert(sizeof(QOp) == 16, "QOp layout");

struct alignas(16) QPhase {
  int32_t op_begin, op_end;
  uint8_t reg_pos[4];
  uint8_t thr_pos[8];
  uint8_t pad[12];
};
static_assert(sizeof(QPhase) == 32, "QPhase layout");
constexpr int kQMaxPhases = 64;  // phases of one pass staged in shared memory
// a gate mixes at most two bits, so every phase of a pass but the last holds at least two gates
static_assert(kQReg == 4 && kQMaxPhases >= kQMaxOps / 2, "the ops of a pass bound its phases");

struct alignas(16) QPass {
  int32_t T, n_outer, init;  // init: the first pass, whose tile is synthesised
  int32_t phase_begin, phase_end, op_begin, op_end, mat_begin, mat_end;
  uint8_t tile_pos[16], outer_pos[40];
  int32_t heavy;  // the pass holds a dense 4x4 (its kernel takes more registers)
};

struct Q428U2 {
  int32_t u[8];  // 2x2, row-major, (re, im) interleaved
};
struct Q428U4 {
  int32_t u[32];  // 4x4
};

__device__ __forceinline__ int32_t q_clamp(long long r) {
  return (int32_t)(r > INT_MAX ? (long long)INT_MAX : (r < INT_MIN ? (long long)INT_MIN : r));
}
__device__ __forceinline__ int32_t q_round(long long acc) { return q_clamp((acc + (1ll << 27)) >> 28); }

// (a + ib) (c + id) accumulated into (re, im), exactly
__device__ __forceinline__ void cmac(long long &re, long long &im, int32_t ur, int32_t ui, int2 v) {
  re += (long long)ur * v.x - (long long)ui * v.y;
  im += (long long)ur * v.y + (long long)ui * v.x;
}

// Insert a zero bit at position p of j.
__device__ __forceinline__ long long insert0(long long j, int p) {
  return ((j >> p) << (p + 1)) | (j & ((1ll << p) - 1));
}

__global__ void k_q428_g1(int2 *__restrict__ st, long long pairs, int p, const __grid_constant__ Q428U2 g) {
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < pairs; j += (long long)gridDim.x * blockDim.x) {
    const long long i0 = insert0(j, p), i1 = i0 | (1ll << p);
    const int2 a = st[i0], b = st[i1];
    long long r0 = 0, m0 = 0, r1 = 0, m1 = 0;
    cmac(r0, m0, g.u[0], g.u[1], a);
    cmac(r0, m0, g.u[2], g.u[3], b);
    cmac(r1, m1, g.u[4], g.u[5], a);
    cmac(r1, m1, g.u[6], g.u[7], b);
    st[i0] = make_int2(q_round(r0), q_round(m0));
    st[i1] = make_int2(q_round(r1), q_round(m1));
  }
}

// pa: bit of the first qubit (high bit of the 4x4 index), pb: the second's
__global__ void k_q428_g2(int2 *__restrict__ st, long long quads, int pa, int pb, const __grid_constant__ Q428U4 g) {
  const int lo = pa < pb ? pa : pb, hi = pa < pb ? pb : pa;
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < quads; j += (long long)gridDim.x * blockDim.x) {
    const long long i00 = insert0(insert0(j, lo), hi);
    long long idx[4];
    idx[0] = i00;
    idx[1] = i00 | (1ll << pb);
    idx[2] = i00 | (1ll << pa);
    idx[3] = i00 | (1ll << pa) | (1ll << pb);
    int2 v[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = st[idx[m]];
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      long long re = 0, im = 0;
#pragma unroll
      for (int m = 0; m < 4; ++m) cmac(re, im, g.u[2 * (4 * l + m)], g.u[2 * (4 * l + m) + 1], v[m]);
      st[idx[l]] = make_int2(q_round(re), q_round(im));
    }
  }
}

__global__ void k_q428_basis(int2 *__restrict__ st, long long n_amps, unsigned long long init) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n_amps; i += (long long)gridDim.x * blockDim.x)
    st[i] = make_int2(i == (long long)init ? (1 << 28) : 0, 0);
}

// ------------------------------------------------------------------------------ tile kernel

constexpr long long kHalf = 1ll << 27;  // accumulators start at the rounding half

__device__ __forceinline__ long long wide(int32_t a, int32_t b, long long c) { return (long long)a * b + c; }

// (acc >> 28) without its saturation: bits 28..59.  `out` collects whether any result leaves
// [-2^29, 2^29): acc / 2^32 lies in [-2^25, 2^25) exactly when the high word plus 2^25, unsigned,
// is below 2^26.
__device__ __forceinline__ int32_t q_low(long long acc, unsigned &out) {
  const unsigned hi = (unsigned)((unsigned long long)acc >> 32);
  out |= hi + (1u << 25);
  return (int32_t)__funnelshift_r((unsigned)acc, hi, 28);
}
__device__ __forceinline__ bool q_big(unsigned out) { return (out & ~((1u << 26) - 1u)) != 0u; }

// four accumulators -> two amplitudes.  A result outside [-2^29, 2^29) clears `small` (and is
// saturated); as long as a thread's amplitudes are small, the sum of two parts fits 32 bits.
__device__ __forceinline__ void q_pair(long long r0, long long m0, long long r1, long long m1, int2 &x, int2 &y,
                                       bool &small) {
  unsigned o = 0;
  x.x = q_low(r0, o);
  x.y = q_low(m0, o);
  y.x = q_low(r1, o);
  y.y = q_low(m1, o);
  if (q_big(o)) {
    x = make_int2(q_clamp(r0 >> 28), q_clamp(m0 >> 28));
    y = make_int2(q_clamp(r1 >> 28), q_clamp(m1 >> 28));
    small = false;
  }
}

// A 2x2 on register bit R.  Q_G1 and Q_V1 take complex products of small amplitudes with three
// multiplications (Gauss): with s = y.re + y.im,
//   Re(u y) = ur s - (ur + ui) y.im,  Im(u y) = ur s + (ui - ur) y.re,
// and the products ur s of a row are shared by its two sums; 12 (11 for a real first entry) widening
// multiply-adds a pair instead of 16 (14).  Entries: per matrix entry ur, -(ur + ui), ui - ur.
// The integer identity is exact, so the sums are the same.
template <int R, int FORM>
__device__ __forceinline__ void q_g1(int2 (&a)[16], const int32_t *__restrict__ u, bool &small) {
  int e[12];
#pragma unroll
  for (int k = 0; k < (FORM == Q_G1 || FORM == Q_V1 ? 3 : 2); ++k) {
    const int4 v = *reinterpret_cast<const int4 *>(u + 4 * k);
    e[4 * k] = v.x, e[4 * k + 1] = v.y, e[4 * k + 2] = v.z, e[4 * k + 3] = v.w;
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << R)) continue;
    const int2 x = a[j], y = a[j | (1 << R)];
    long long r0 = kHalf, m0 = kHalf, r1 = kHalf, m1 = kHalf;
    if (FORM == Q_ANY1) {
      cmac(r0, m0, e[0], e[1], x);
      cmac(r0, m0, e[2], e[3], y);
      cmac(r1, m1, e[4], e[5], x);
      cmac(r1, m1, e[6], e[7], y);
    } else if (FORM == Q_G1 || FORM == Q_V1) {
      const int sx = x.x + x.y, sy = y.x + y.y;
      const long long t1 = wide(e[9], sy, wide(e[6], sx, kHalf));
      r1 = wide(e[10], y.y, wide(e[7], x.y, t1));
      m1 = wide(e[11], y.x, wide(e[8], x.x, t1));
      if (FORM == Q_V1) {
        const long long t0 = wide(e[3], sy, kHalf);
        r0 = wide(e[4], y.y, wide(e[0], x.x, t0));
        m0 = wide(e[5], y.x, wide(e[0], x.y, t0));
      } else {
        const long long t0 = wide(e[3], sy, wide(e[0], sx, kHalf));
        r0 = wide(e[4], y.y, wide(e[1], x.y, t0));
        m0 = wide(e[5], y.x, wide(e[2], x.x, t0));
      }
    } else if (FORM == Q_REAL1) {
      r0 = wide(e[2], y.x, wide(e[0], x.x, r0));
      m0 = wide(e[2], y.y, wide(e[0], x.y, m0));
      r1 = wide(e[6], y.x, wide(e[4], x.x, r1));
      m1 = wide(e[6], y.y, wide(e[4], x.y, m1));
    } else {  // Q_RX1: entries (u00, 0), (-, u01), (-, u10), (u11, 0); chosen only without INT_MIN
      r0 = wide(-e[3], y.y, wide(e[0], x.x, r0));
      m0 = wide(e[3], y.x, wide(e[0], x.y, m0));
      r1 = wide(e[6], y.x, wide(-e[5], x.y, r1));
      m1 = wide(e[6], y.y, wide(e[5], x.x, m1));
    }
    q_pair(r0, m0, r1, m1, a[j], a[j | (1 << R)], small);
  }
}
template <int FORM>
__device__ __forceinline__ void q_g1_at(int2 (&a)[16], int r, const int32_t *u, bool &small) {
  switch (r) {
    case 0: q_g1<0, FORM>(a, u, small); break;
    case 1: q_g1<1, FORM>(a, u, small); break;
    case 2: q_g1<2, FORM>(a, u, small); break;
    default: q_g1<3, FORM>(a, u, small); break;
  }
}

// The same 2x2 for amplitudes of any size: the entries are recovered from the Gauss layout
// (u11's and the others' (ur, ui) = (e0, e0 + e2)).
__device__ __noinline__ int4 q_g1_slow(int2 x, int2 y, const int32_t *u) {
  long long r0 = kHalf, m0 = kHalf, r1 = kHalf, m1 = kHalf;
  cmac(r0, m0, u[0], u[0] + u[2], x);
  cmac(r0, m0, u[3], u[3] + u[5], y);
  cmac(r1, m1, u[6], u[6] + u[8], x);
  cmac(r1, m1, u[9], u[9] + u[11], y);
  return make_int4(q_clamp(r0 >> 28), q_clamp(m0 >> 28), q_clamp(r1 >> 28), q_clamp(m1 >> 28));
}
template <int R>
__device__ __forceinline__ void q_g1_slow_r(int2 (&a)[16], const int32_t *u) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << R)) continue;
    const int4 v = q_g1_slow(a[j], a[j | (1 << R)], u);
    a[j] = make_int2(v.x, v.y);
    a[j | (1 << R)] = make_int2(v.z, v.w);
  }
}
__device__ __forceinline__ void q_g1_slow_at(int2 (&a)[16], int r, const int32_t *u) {
  switch (r) {
    case 0: q_g1_slow_r<0>(a, u); break;
    case 1: q_g1_slow_r<1>(a, u); break;
    case 2: q_g1_slow_r<2>(a, u); break;
    default: q_g1_slow_r<3>(a, u); break;
  }
}

// exchange along register bit R of the pairs whose lower member j has bit j of pred set
template <int R>
__device__ __forceinline__ void q_x1(int2 (&a)[16], uint32_t pred) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & (1 << R)) continue;
    const bool p = (pred >> j) & 1u;
    const int2 x = a[j], y = a[j | (1 << R)];
    a[j] = make_int2(p ? y.x : x.x, p ? y.y : x.y);
    a[j | (1 << R)] = make_int2(p ? x.x : y.x, p ? x.y : y.y);
  }
}

__device__ __forceinline__ int32_t q_neg(int32_t v) { return -max(v, -INT_MAX); }  // -INT_MIN saturates

// The sign flips collected in neg.  Flips of small amplitudes are exact, so a run of them (a layer of
// CZ) is applied at once; others saturate one by one.
__device__ __forceinline__ void q_flush(int2 (&a)[16], uint32_t &neg) {
#pragma unroll
  for (int j = 0; j < 16; ++j)
    if ((neg >> j) & 1u) a[j] = make_int2(q_neg(a[j].x), q_neg(a[j].y));
  neg = 0u;
}

template <int RA, int RB>
__device__ __forceinline__ void q_g2(int2 (&a)[16], const int32_t *__restrict__ u) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j & ((1 << RA) | (1 << RB))) continue;
    const int id[4] = {j, j | (1 << RB), j | (1 << RA), j | (1 << RA) | (1 << RB)};
    const int2 v[4] = {a[id[0]], a[id[1]], a[id[2]], a[id[3]]};
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      long long re = kHalf, im = kHalf;
#pragma unroll
      for (int m = 0; m < 4; ++m) cmac(re, im, u[2 * (4 * l + m)], u[2 * (4 * l + m) + 1], v[m]);
      a[id[l]] = make_int2(q_clamp(re >> 28), q_clamp(im >> 28));
    }
  }
}
template <int RA, int RB>
__device__ __forceinline__ void q_swap(int2 (&a)[16]) {
#pragma unroll
  for (int j = 0; j < 16; ++j)
    if ((j & (1 << RA)) && !(j & (1 << RB))) {
      const int j2 = (j & ~(1 << RA)) | (1 << RB);
      const int2 t = a[j];
      a[j] = a[j2];
      a[j2] = t;
    }
}
template <int RA, int RB>
__device__ __forceinline__ void q_two(int2 (&a)[16], bool swap, const int32_t *u) {
  if (swap) q_swap<RA, RB>(a);
  else q_g2<RA, RB>(a, u);
}

// small: every amplitude of the thread lies in [-2^29, 2^29] (kept by the exchanges and the sign)
template <bool HEAVY>
__device__ __forceinline__ void q_apply(int2 (&a)[16], const QOp &op, const BitCtx &c, const int32_t *mats,
                                        bool &small, uint32_t &neg) {
  const int32_t *u = mats + op.mat;
  if (op.type == Q_NEG) {
    neg ^= src_mask(c, op.a_kind, op.a_pos) & src_mask(c, op.b_kind, op.b_pos);
    if (!small) q_flush(a, neg);
    return;
  }
  if (neg) q_flush(a, neg);
  switch (op.type) {
    case Q_G1:
      if (small) q_g1_at<Q_G1>(a, op.a_pos, u, small);
      else q_g1_slow_at(a, op.a_pos, u);
      break;
    case Q_V1:
      if (small) q_g1_at<Q_V1>(a, op.a_pos, u, small);
      else q_g1_slow_at(a, op.a_pos, u);
      break;
    case Q_REAL1: q_g1_at<Q_REAL1>(a, op.a_pos, u, small); break;
    case Q_RX1: q_g1_at<Q_RX1>(a, op.a_pos, u, small); break;
    case Q_ANY1:
      if constexpr (HEAVY) q_g1_at<Q_ANY1>(a, op.a_pos, u, small);
      break;
    case Q_X1: {
      const uint32_t pred = op.a_kind == kAlways ? c.full : src_mask(c, op.a_kind, op.a_pos);
      switch (op.b_pos) {
        case 0: q_x1<0>(a, pred); break;
        case 1: q_x1<1>(a, pred); break;
        case 2: q_x1<2>(a, pred); break;
        default: q_x1<3>(a, pred); break;
      }
      break;
    }
    case Q_DIAG: {
      const uint32_t ma = src_mask(c, op.a_kind, op.a_pos), mb = src_mask(c, op.b_kind, op.b_pos);
#pragma unroll 1
      for (int v = 0; v < 4; ++v) {
        const uint32_t m = ((v & 2) ? ma : ~ma) & ((v & 1) ? mb : ~mb) & c.full;
        if (((op.ones >> v) & 1) || m == 0u) continue;
        const int32_t dr = u[2 * v], di = u[2 * v + 1];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          long long re = kHalf, im = kHalf;
          cmac(re, im, dr, di, a[j]);
          unsigned o = 0;
          int2 r = make_int2(q_low(re, o), q_low(im, o));
          const bool big = q_big(o), take = (m >> j) & 1u;
          if (big) r = make_int2(q_clamp(re >> 28), q_clamp(im >> 28));
          if (take) a[j] = r;
          if (big && take) small = false;
        }
      }
      break;
    }
    default: {  // Q_G2, Q_SWAP
      const bool sw = op.type == Q_SWAP;
      if (!HEAVY) break;
      if (!sw) small = false;
      switch (op.a_pos * 4 + op.b_pos) {
        case 1: q_two<0, 1>(a, sw, u); break;
        case 2: q_two<0, 2>(a, sw, u); break;
        case 3: q_two<0, 3>(a, sw, u); break;
        case 4: q_two<1, 0>(a, sw, u); break;
        case 6: q_two<1, 2>(a, sw, u); break;
        case 7: q_two<1, 3>(a, sw, u); break;
        case 8: q_two<2, 0>(a, sw, u); break;
        case 9: q_two<2, 1>(a, sw, u); break;
        case 11: q_two<2, 3>(a, sw, u); break;
        case 12: q_two<3, 0>(a, sw, u); break;
        case 13: q_two<3, 1>(a, sw, u); break;
        case 14: q_two<3, 2>(a, sw, u); break;
      }
      break;
    }
  }
}

// One pass.  256 threads of 16 amplitudes at the full tile size (fewer for states narrower than a
// tile); the ops and entries of the pass are staged in shared memory once per CTA.  Dense 4x4s and
// 2x2s of large entries (HEAVY) have a kernel of their own, so that their registers do not cost the
// others a CTA.
template <bool HEAVY>
__global__ void __launch_bounds__(1 << (kQTile - kQReg), HEAVY ? kQHeavyCtas : kQCtas)
    k_q428_pass(const __grid_constant__ QPass pd, const QPhase *__restrict__ phases,
                const QOp *__restrict__ ops, const int32_t *__restrict__ mats, int2 *__restrict__ st,
                unsigned long long init) {
  __shared__ __align__(16) int2 sm[1 << kQTile];
  __shared__ __align__(16) QOp s_ops[kQMaxOps];
  __shared__ __align__(16) int32_t s_mat[kQMaxMat];
  __shared__ __align__(16) QPhase s_ph[kQMaxPhases];
  __shared__ long long run_off[1 << (kQTile - kLowBits)];
  const int T = pd.T, tile = 1 << T, runs = 1 << (T - kLowBits);
  for (int r = threadIdx.x; r < runs; r += blockDim.x) {
    long long off = 0;
    for (int j = 0; j < T - kLowBits; ++j)
      if ((r >> j) & 1) off |= 1ll << pd.tile_pos[kLowBits + j];
    run_off[r] = off;
  }
  const int n_ops = pd.op_end - pd.op_begin, n_mat = pd.mat_end - pd.mat_begin;
  for (int i = threadIdx.x; i < n_ops; i += blockDim.x) s_ops[i] = ops[pd.op_begin + i];
  for (int i = threadIdx.x; i < n_mat; i += blockDim.x) s_mat[i] = mats[pd.mat_begin + i];
  for (int i = threadIdx.x; i < pd.phase_end - pd.phase_begin; i += blockDim.x) s_ph[i] = phases[pd.phase_begin + i];
  unsigned long long outer_mask = 0;
  for (int j = 0; j < pd.n_outer; ++j) outer_mask |= 1ull << pd.outer_pos[j];
  const long long n_tiles = 1ll << pd.n_outer;
  constexpr int kLowMask = (1 << kLowBits) - 1;
  __syncthreads();
  // the tables above belong to the plan; the state is the previous pass's
  pdl_wait();
  pdl_trigger();
  for (long long t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    unsigned long long base = 0;
    for (int j = 0; j < pd.n_outer; ++j) base |= (unsigned long long)((t >> j) & 1) << pd.outer_pos[j];
    int2 *g = st + base;
    if (pd.init) {
      // the basis state is zero outside one tile, and zeros stay zero through every gate
      const bool here = (init & outer_mask) == base;
      if (!here) {
        for (int i = threadIdx.x; i < tile; i += blockDim.x) g[run_off[i >> kLowBits] + (i & kLowMask)] = make_int2(0, 0);
        continue;
      }
      int li = 0;
      for (int j = 0; j < T; ++j) li |= (int)((init >> pd.tile_pos[j]) & 1ull) << j;
      for (int i = threadIdx.x; i < tile; i += blockDim.x) sm[swz(i)] = make_int2(i == li ? (1 << 28) : 0, 0);
    } else {
#pragma unroll 8
      for (int i = threadIdx.x; i < tile; i += blockDim.x) sm[swz(i)] = g[run_off[i >> kLowBits] + (i & kLowMask)];
    }
    __syncthreads();
    for (int p = 0; p < pd.phase_end - pd.phase_begin; ++p) {
      const QPhase &ph = s_ph[p];
      BitCtx ctx;
      ctx.tb = deposit(threadIdx.x, ph.thr_pos, T - kQReg);
      ctx.base = base;
      ctx.full = 0xFFFFu;
      const int pb = swz(ctx.tb);
      int d[4];
#pragma unroll
      for (int r = 0; r < kQReg; ++r) d[r] = swz(1 << ph.reg_pos[r]);
      auto at = [&](int j) {
        return pb ^ ((j & 1) ? d[0] : 0) ^ ((j & 2) ? d[1] : 0) ^ ((j & 4) ? d[2] : 0) ^ ((j & 8) ? d[3] : 0);
      };
      int2 a[16];
      unsigned o = 0;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        a[j] = sm[at(j)];
        o |= (unsigned)(a[j].x + (1 << 29)) | (unsigned)(a[j].y + (1 << 29));
      }
      bool small = (o >> 30) == 0u;
      uint32_t neg = 0u;
      const int o_end = ph.op_end - pd.op_begin;
#pragma unroll 1
      for (int k = ph.op_begin - pd.op_begin; k < o_end; ++k) q_apply<HEAVY>(a, s_ops[k], ctx, s_mat, small, neg);
      if (neg) q_flush(a, neg);
      // the addresses are formed again here rather than held in registers through the ops
#pragma unroll
      for (int r = 0; r < kQReg; ++r) asm volatile("" : "+r"(d[r]));
#pragma unroll
      for (int j = 0; j < 16; ++j) sm[at(j)] = a[j];
      __syncthreads();
    }
#pragma unroll 8
    for (int i = threadIdx.x; i < tile; i += blockDim.x) g[run_off[i >> kLowBits] + (i & kLowMask)] = sm[swz(i)];
    __syncthreads();
  }
}

unsigned grid_for(long long items) {
  return (unsigned)std::max<long long>(1, std::min<long long>((items + 255) / 256, 152ll * 16));
}

bool is_one(const int32_t *e) { return e[0] == (1 << 28) && e[1] == 0; }
bool is_zero(const int32_t *e) { return e[0] == 0 && e[1] == 0; }

// The op of one quantised gate: its form, and which of its qubits (0 first, 1 second) it mixes.
// Bits are filled in by the planner.
struct QForm {
  int type;
  bool mix_a, mix_b, heavy;
  uint8_t ones;
  int n_mat;
  int32_t mat[32];
};
QForm form_of(const Q428Gate &g) {
  QForm f{};
  const int dim = g.nq == 1 ? 2 : 4;
  auto e = [&](int i, int j) { return g.u + 2 * (dim * i + j); };
  bool diag = true, min = false;
  for (int i = 0; i < dim; ++i)
    for (int j = 0; j < dim; ++j) diag = diag && (i == j || is_zero(e(i, j)));
  for (int i = 0; i < 2 * dim * dim; ++i) min = min || g.u[i] == INT_MIN;
  if (diag) {
    // entry 2 bit(a) + bit(b); a one-qubit gate has a = b (entries 0 and 3)
    f.type = Q_DIAG;
    f.n_mat = 8;
    for (int v = 0; v < 4; ++v) {
      const int32_t *d = dim == 4 ? e(v, v) : e(v >> 1, v >> 1);
      f.mat[2 * v] = d[0];
      f.mat[2 * v + 1] = d[1];
      if (is_one(d)) f.ones |= (uint8_t)(1 << v);
    }
    const int32_t *last = f.mat + 6;
    if (last[0] == -(1 << 28) && last[1] == 0 && (dim == 4 ? f.ones == 7 : is_one(f.mat))) {
      f.type = Q_NEG;
      f.n_mat = 0;
    }
    return f;
  }
  if (dim == 2) {
    f.mix_a = true;
    if (is_zero(e(0, 0)) && is_zero(e(1, 1)) && is_one(e(0, 1)) && is_one(e(1, 0))) {
      f.type = Q_X1;
      return f;
    }
    const int32_t *u = g.u;
    bool fits = true;  // the sums of the Gauss layout (and of small amplitudes) stay within 32 bits
    for (int i = 0; i < 8; ++i) fits = fits && u[i] > -(1 << 29) && u[i] < (1 << 29);
    if (min) f.type = Q_ANY1;
    else if (u[1] == 0 && u[3] == 0 && u[5] == 0 && u[7] == 0) f.type = Q_REAL1;
    else if (u[1] == 0 && u[7] == 0 && u[2] == 0 && u[4] == 0) f.type = Q_RX1;
    else if (!fits) f.type = Q_ANY1;
    else f.type = u[1] == 0 ? Q_V1 : Q_G1;
    f.heavy = f.type == Q_ANY1;
    if (f.type == Q_G1 || f.type == Q_V1) {
      for (int k = 0; k < 4; ++k) {
        const int32_t ur = u[2 * k], ui = u[2 * k + 1];
        f.mat[f.n_mat++] = ur;
        f.mat[f.n_mat++] = -(ur + ui);
        f.mat[f.n_mat++] = ui - ur;
      }
    } else {
      std::copy(u, u + 8, f.mat);
      f.n_mat = 8;
    }
    return f;
  }
  auto perm_is = [&](const int *to) {  // column j has a single one, in row to[j]
    for (int i = 0; i < 4; ++i)
      for (int j = 0; j < 4; ++j)
        if (!(i == to[j] ? is_one(e(i, j)) : is_zero(e(i, j)))) return false;
    return true;
  };
  const int cnot[4] = {0, 1, 3, 2}, swap[4] = {0, 2, 1, 3};
  if (perm_is(cnot)) {
    f.type = Q_X1;
    f.mix_b = true;
    return f;
  }
  f.mix_a = f.mix_b = f.heavy = true;
  f.type = perm_is(swap) ? Q_SWAP : Q_G2;
  if (f.type == Q_G2) {
    std::copy(g.u, g.u + 32, f.mat);
    f.n_mat = 32;
  }
  return f;
}

}  // namespace

// Passes and phases of a fixed-point plan, on the host and (NULL when host-only) on the device.
struct Q428Plan {
  std::vector<Q428Gate> gates;
  std::vector<QPass> passes;
  std::vector<QPhase> phases;
  std::vector<QOp> ops;
  std::vector<int32_t> mats;
  unsigned char *d_tables = nullptr;  // phases, ops and mats back to back (each a multiple of 16 bytes)
  size_t ops_at() const { return sizeof(QPhase) * phases.size(); }
  size_t mats_at() const { return ops_at() + sizeof(QOp) * ops.size(); }
};

int32_t q428_quantize(double x) {
  const double r = std::floor(x * 268435456.0 + 0.5);  // x 2^28, round half up (exact for |x| < 2^24)
  return (int32_t)std::max(std::min(r, (double)INT_MAX), (double)INT_MIN);
}

Q428Plan *q428_build(const tn_circuit &c) {
  Q428Plan *p = new Q428Plan();
  p->gates.reserve(c.gates.size());
  for (const TnGate &g : c.gates) {
    double m[32];
    const int dim = gate_matrix(g.kind, FORM_U, g.angle, g.mat, m);
    Q428Gate q;
    q.nq = dim == 2 ? 1 : 2;
    q.pos[0] = c.n - 1 - g.q[0];
    q.pos[1] = q.nq == 2 ? c.n - 1 - g.q[1] : -1;
    for (int i = 0; i < 2 * dim * dim; ++i) q.u[i] = q428_quantize(m[i]);
    p->gates.push_back(q);
  }
  const int n = c.n, G = (int)p->gates.size();
  if (n < kQMinQubits || G == 0) return p;
  const int T = std::min(n, kQTile);
  std::vector<QForm> forms((size_t)G);
  size_t entries = 0;
  for (int k = 0; k < G; ++k) entries += (size_t)(forms[(size_t)k] = form_of(p->gates[(size_t)k])).n_mat;
  p->ops.reserve((size_t)G);
  p->mats.reserve(entries);
  auto mixed = [&](int k) {  // state bits gate k mixes
    uint64_t b = 0;
    if (forms[(size_t)k].mix_a) b |= 1ull << p->gates[(size_t)k].pos[0];
    if (forms[(size_t)k].mix_b) b |= 1ull << p->gates[(size_t)k].pos[1];
    return b;
  };
  const uint64_t low = (1ull << kLowBits) - 1;
  // records keep 16-byte aligned entries (8, 12 or 32 of them)
  for (int k0 = 0; k0 < G;) {
    // the longest run of gates whose mixed bits fit the tile (beside the low bits, which keep runs of
    // 128 bytes) and whose records fit the staging
    uint64_t S = low;
    int k1 = k0, n_mat = 0;
    for (; k1 < G && k1 - k0 < kQMaxOps; ++k1) {
      const uint64_t U = S | mixed(k1);
      const int nm = forms[(size_t)k1].n_mat;
      if (__builtin_popcountll(U) > T || n_mat + nm > kQMaxMat) break;
      S = U;
      n_mat += nm;
    }
    for (int b = 0; b < n && __builtin_popcountll(S) < T; ++b) S |= 1ull << b;
    QPass pd;
    std::memset(&pd, 0, sizeof(pd));
    pd.T = T;
    pd.init = k0 == 0 ? 1 : 0;
    int tile_of[64], tl = 0, ol = 0;
    for (int b = 0; b < 64; ++b) tile_of[b] = -1;
    for (int b = 0; b < n; ++b) {
      if ((S >> b) & 1) {
        tile_of[b] = tl;
        pd.tile_pos[tl++] = (uint8_t)b;
      } else {
        pd.outer_pos[ol++] = (uint8_t)b;
      }
    }
    pd.n_outer = ol;
    pd.phase_begin = (int)p->phases.size();
    pd.op_begin = (int)p->ops.size();
    pd.mat_begin = (int)p->mats.size();
    while (k0 < k1) {
      uint64_t R = 0;
      int k2 = k0;
      for (; k2 < k1; ++k2) {
        const uint64_t U = R | mixed(k2);
        if (__builtin_popcountll(U) > kQReg) break;
        R = U;
      }
      for (int b = n - 1; b >= 0 && __builtin_popcountll(R) < kQReg; --b)  // fill from the high tile bits
        if ((S >> b) & 1) R |= 1ull << b;
      QPhase ph;
      std::memset(&ph, 0, sizeof(ph));
      int reg_of[64], r = 0;
      for (int b = 0; b < 64; ++b) reg_of[b] = -1;
      for (int b = 0; b < n; ++b)
        if ((R >> b) & 1) {
          ph.reg_pos[r] = (uint8_t)tile_of[b];
          reg_of[b] = r++;
        }
      // thread bits: the first five (lanes) cover the residues mod 4 where they can, so a warp's
      // shared-memory accesses fall in distinct banks under the tile's swizzle
      int rest[kQTile], n_rest = 0, t = 0;
      bool used[kQTile] = {};
      for (int b = 0; b < n; ++b)
        if (((S >> b) & 1) && !((R >> b) & 1)) rest[n_rest++] = tile_of[b];
      for (int res = 0; res < 4; ++res)
        for (int i = 0; i < n_rest; ++i)
          if (!used[i] && (rest[i] & 3) == res) {
            ph.thr_pos[t++] = (uint8_t)rest[i];
            used[i] = true;
            break;
          }
      for (int i = 0; i < n_rest; ++i)
        if (!used[i]) ph.thr_pos[t++] = (uint8_t)rest[i];
      auto source = [&](int bit, uint8_t &kind, uint8_t &pos) {
        if (reg_of[bit] >= 0) kind = SRC_REG, pos = (uint8_t)reg_of[bit];
        else if (tile_of[bit] >= 0) kind = SRC_TILE, pos = (uint8_t)tile_of[bit];
        else kind = SRC_GLOB, pos = (uint8_t)bit;
      };
      ph.op_begin = (int)p->ops.size();
      for (; k0 < k2; ++k0) {
        const Q428Gate &g = p->gates[(size_t)k0];
        const QForm &f = forms[(size_t)k0];
        QOp op;
        std::memset(&op, 0, sizeof(op));
        op.type = (uint8_t)f.type;
        op.ones = f.ones;
        source(g.pos[0], op.a_kind, op.a_pos);
        source(g.nq == 2 ? g.pos[1] : g.pos[0], op.b_kind, op.b_pos);
        if (f.type == Q_X1 && g.nq == 1) op.a_kind = kAlways;
        pd.heavy |= f.heavy ? 1 : 0;
        op.mat = (int)p->mats.size() - pd.mat_begin;
        p->mats.insert(p->mats.end(), f.mat, f.mat + f.n_mat);
        p->ops.push_back(op);
      }
      ph.op_end = (int)p->ops.size();
      p->phases.push_back(ph);
    }
    pd.phase_end = (int)p->phases.size();
    pd.op_end = (int)p->ops.size();
    pd.mat_end = (int)p->mats.size();
    p->passes.push_back(pd);
  }
  return p;
}

cudaError_t q428_upload(Q428Plan *p) {
  if (p->passes.empty()) return cudaSuccess;
  // One allocation and one copy (9-qubit QFT beside other plans: made in 102 us and freed in 5, 110 and 11 with
  // three of each, 79 on the host alone; the first allocation of a process takes 90 more).
  std::vector<unsigned char> t(p->mats_at() + sizeof(int32_t) * p->mats.size());
  std::memcpy(t.data(), p->phases.data(), p->ops_at());
  std::memcpy(t.data() + p->ops_at(), p->ops.data(), sizeof(QOp) * p->ops.size());
  if (!p->mats.empty()) std::memcpy(t.data() + p->mats_at(), p->mats.data(), sizeof(int32_t) * p->mats.size());
  cudaError_t e = cudaMalloc((void **)&p->d_tables, t.size());
  if (e == cudaSuccess) e = cudaMemcpy(p->d_tables, t.data(), t.size(), cudaMemcpyHostToDevice);
  return e == cudaSuccess ? tables_ready() : e;
}

void q428_free(Q428Plan *p) {
  if (!p) return;
  // a plan made for the host alone has no tables, and even cudaFree(NULL) would start the runtime
  if (p->d_tables) cudaFree(p->d_tables);
  delete p;
}

int q428_gates(const Q428Plan *p) { return (int)p->gates.size(); }
int q428_launches(const Q428Plan *p) {
  return p->passes.empty() ? 1 + (int)p->gates.size() : (int)p->passes.size();
}

cudaError_t launch_q428(const Q428Plan *p, int n, unsigned long long init, int32_t *state, cudaStream_t s) {
  int2 *st = reinterpret_cast<int2 *>(state);
  const long long amps = 1ll << n;
  if (!p->passes.empty()) {
    const int T = p->passes.front().T, threads = 1 << (T - kQReg);
    cudaError_t e = cudaSuccess;
    for (size_t i = 0; e == cudaSuccess && i < p->passes.size(); ++i) {
      const bool heavy = p->passes[i].heavy != 0;
      const long long grid = std::min<long long>(1ll << (n - T), (long long)num_sms() * (heavy ? kQHeavyCtas : kQCtas));
      e = launch_pdl(heavy ? k_q428_pass<true> : k_q428_pass<false>, dim3((unsigned)grid), dim3((unsigned)threads), 0, s, p->passes[i],
                     reinterpret_cast<const QPhase *>(p->d_tables), reinterpret_cast<const QOp *>(p->d_tables + p->ops_at()),
                     reinterpret_cast<const int32_t *>(p->d_tables + p->mats_at()), st, init);
    }
    return e;
  }
  k_q428_basis<<<grid_for(amps), 256, 0, s>>>(st, amps, init);
  cudaError_t e = cudaGetLastError();
  for (size_t k = 0; e == cudaSuccess && k < p->gates.size(); ++k) {
    const Q428Gate &q = p->gates[k];
    if (q.nq == 1) {
      Q428U2 g;
      std::copy(q.u, q.u + 8, g.u);
      k_q428_g1<<<grid_for(amps / 2), 256, 0, s>>>(st, amps / 2, q.pos[0], g);
    } else {
      Q428U4 g;
      std::copy(q.u, q.u + 32, g.u);
      k_q428_g2<<<grid_for(amps / 4), 256, 0, s>>>(st, amps / 4, q.pos[0], q.pos[1], g);
    }
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace tnq
