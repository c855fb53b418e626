// Small kernels of libtnq: per-call gate-matrix tables, amplitude gather, gradient
// scaling, device status word.
#include <algorithm>
#include <vector>

#include "apply_common.cuh"
#include "kernels.h"

namespace tnq {

// Gate tensors are built once per call from the parameters (angles in FP64, entries stored as
// complex64).  The slot array lists the fused blocks (KIND_F2) first.  Few fused blocks (small
// batches): each block and batch element takes one warp -- lanes evaluate the members' sines and
// cosines one angle each, lane m embeds member m's matrix as a 4x4, then lanes 0..15 form the product
// one entry each, member by member.  Many (kFusedPerThread or more): one thread each, members applied
// in turn to a 4x4 held by the thread (all lanes busy).  Either way the product is stored in the packed
// layout (SHAPE_M4X).  Every other slot and batch element takes one thread, or four (one per angle)
// where there are few.
// Bound: FP64, two operations per SM and clock, so a warp's instruction takes 16 clocks of its SM and a
// sincos about a microsecond with nothing beside it.  Hence one warp per CTA: the warps spread over the
// SMs instead of queueing on one FP64 unit.  Whole calls with four warps per CTA and one thread per
// slot or member, and now: 10-qubit brickwork of depth 8, 16 sets 14.4 and 12.4 us; 16 qubits, depth 10,
// one set 37 and 33 us; 22 qubits 159 and 155 us.
constexpr long long kFusedPerThread = 1024;  // fused blocks x batch from which each takes one thread
// Other slots x batch up to which each takes four threads: whole calls with one thread per slot and with four,
// 10 qubits, replayed from a graph: U3 slots 2560 12.2 and 11.2 us, 5120 12.2 and 11.5, 10240 12.4 and 13.6;
// slots of one angle 1920 10.1 either way, 3840 9.8 and 10.7.
constexpr long long kSpreadSlots = 4096;

// One regular slot (one gate's matrix) for one batch element; prow: its parameters (may be NULL).
__device__ void materialize_one(const MatSlot &s, const double *prow, float2 *table) {
  double ang[3] = {s.angle[0], s.angle[1], s.angle[2]};
  for (int a = 0; a < 3; ++a)
    for (int q = 0; q < 2; ++q)
      if (s.pidx[a][q] >= 0) ang[a] += prow[s.pidx[a][q]];
  double tmp[32], x[3] = {0.0, 0.0, 0.0}, sn[3], cs[3];
  float ent[32];
  const int nx = gate_trig(s.kind, ang, x);
  for (int a = 0; a < nx; ++a) sincos2(x[a], &sn[a], &cs[a]);
  const int n = slot_entries(s, sn, cs, tmp, ent);
  float2 *dst = table + s.offset;
  for (int i = 0; i < n; ++i) dst[i] = make_float2(ent[2 * i], ent[2 * i + 1]);
}

// One regular slot by four consecutive lanes: lane a evaluates angle a's sine and cosine, lane 0 composes.
__device__ void materialize_spread(const MatSlot &s, const double *prow, float2 *table, int lane, bool live) {
  double x[3] = {0.0, 0.0, 0.0}, sn = 0.0, cs = 0.0;
  const int a = lane & 3;
  if (live) {
    double ang[3] = {s.angle[0], s.angle[1], s.angle[2]};
    for (int k = 0; k < 3; ++k)
      for (int q = 0; q < 2; ++q)
        if (s.pidx[k][q] >= 0) ang[k] += prow[s.pidx[k][q]];
    if (a < gate_trig(s.kind, ang, x)) sincos2(a == 0 ? x[0] : a == 1 ? x[1] : x[2], &sn, &cs);
  }
  double sv[3], cv[3];
  for (int k = 0; k < 3; ++k) {
    sv[k] = __shfl_sync(0xFFFFFFFFu, sn, (lane & ~3) + k);
    cv[k] = __shfl_sync(0xFFFFFFFFu, cs, (lane & ~3) + k);
  }
  if (!live || a != 0) return;
  double tmp[32];
  float ent[32];
  const int n = slot_entries(s, sv, cv, tmp, ent);
  float2 *dst = table + s.offset;
  for (int i = 0; i < n; ++i) dst[i] = make_float2(ent[2 * i], ent[2 * i + 1]);
}

__global__ void __launch_bounds__(32) k_materialize(const MatSlot *__restrict__ slots, int n_slots,
                                                               int n_fused_slots,
                                                               const FusedMember *__restrict__ fused,
                                                               const double *__restrict__ params, int n_params,
                                                               int batch, long long mstride, float2 *__restrict__ out,
                                                               int fused_per_thread, int spread) {
  __shared__ double emb[kMaxFusedMembers][32];
  __shared__ double acc[2][32];
  __shared__ double trig[kMaxFusedMembers][3][2];  // sine, cosine
  __shared__ int shape[kMaxFusedMembers];  // which entries of a row of emb can be nonzero: 0 all, 1 diagonal, 2 on a, 3 on b
  const int lane = threadIdx.x;
  const long long gw = blockIdx.x;
  if (fused_per_thread) {
    // many fused blocks (large batches): one thread each, every lane busy in FP64
    const long long n_ft = (long long)n_fused_slots * batch;
    const long long n_fwt = (n_ft + 31) / 32;                    // warps of the fused blocks
    if (gw < n_fwt) {
      const long long t = gw * 32 + lane;
      if (t >= n_ft) return;
      const int b = (int)(t / n_fused_slots);
      const MatSlot &s = slots[t % n_fused_slots];
      const double *prow = params ? params + (long long)b * n_params : nullptr;
      double M[32];
      for (int i = 0; i < 32; ++i) M[i] = (i & 1) == 0 && ((i >> 1) % 5) == 0 ? 1.0 : 0.0;
      for (int m = 0; m < s.fuse_count; ++m) fused_apply_member(fused[s.fuse_begin + m], prow, M);
      float2 *dst = out + (long long)b * mstride + s.offset;
      for (int k = 0; k < 16; ++k) {
        const float re = (float)M[2 * k], im = (float)M[2 * k + 1];
        dst[2 * k] = make_float2(re, re);
        dst[2 * k + 1] = make_float2(-im, im);
      }
      return;
    }
    const int n_reg = n_slots - n_fused_slots;
    const long long t = (gw - n_fwt) * 32 + lane;
    if (t >= (long long)n_reg * batch) return;
    const int b = (int)(t / n_reg);
    materialize_one(slots[n_fused_slots + t % n_reg], params ? params + (long long)b * n_params : nullptr,
                    out + (long long)b * mstride);
    return;
  }
  const long long n_fw = (long long)n_fused_slots * batch;      // warps of the fused blocks
  if (gw < n_fw) {
    const int b = (int)(gw / n_fused_slots);
    const MatSlot &s = slots[gw % n_fused_slots];
    float2 *dst = out + (long long)b * mstride + s.offset;
    const double *prow = params ? params + (long long)b * n_params : nullptr;
    const int cnt = s.fuse_count;
    for (int it = lane; it < 3 * cnt; it += 32) {
      const int m = it / 3, a = it - 3 * m;
      const FusedMember &f = fused[s.fuse_begin + m];
      double ang[3] = {f.angle[0], f.angle[1], f.angle[2]}, x[3] = {0.0, 0.0, 0.0};
      for (int k = 0; k < 3; ++k)
        for (int q = 0; q < 2; ++q)
          if (f.pidx[k][q] >= 0 && prow) ang[k] += prow[f.pidx[k][q]];
      if (a < gate_trig(f.kind, ang, x)) sincos2(a == 0 ? x[0] : a == 1 ? x[1] : x[2], &trig[m][a][0], &trig[m][a][1]);
    }
    acc[0][lane] = (lane & 1) == 0 && ((lane >> 1) % 5) == 0 ? 1.0 : 0.0;  // identity
    __syncwarp();
    if (lane < cnt) {
      double sn[3], cs[3];
      for (int a = 0; a < 3; ++a) sn[a] = trig[lane][a][0], cs[a] = trig[lane][a][1];
      const FusedMember &f = fused[s.fuse_begin + lane];
      fused_embed(f, sn, cs, emb[lane]);
      shape[lane] = gate_nqubits(f.kind) == 1 ? (f.role == ROLE_A ? 2 : 3) : f.kind == TN_GATE_CZ || f.kind == TN_GATE_CP ? 1 : 0;
    }
    __syncwarp();
    int cur = 0;
    for (int m = 0; m < cnt; ++m) {  // acc <- emb[m] * acc
      if (lane < 16) {
        const int i = lane >> 2, j = lane & 3;
        double re = 0.0, im = 0.0;
        const int sh = shape[m], terms = sh == 0 ? 4 : sh == 1 ? 1 : 2;
        for (int k = 0; k < terms; ++k) {  // the others are zero
          const int q = sh == 0 ? k : sh == 1 ? i : sh == 2 ? 2 * k + (i & 1) : (i & 2) + k;
          const double xr = emb[m][2 * (4 * i + q)], xi = emb[m][2 * (4 * i + q) + 1];
          const double yr = acc[cur][2 * (4 * q + j)], yi = acc[cur][2 * (4 * q + j) + 1];
          re += xr * yr - xi * yi;
          im += xr * yi + xi * yr;
        }
        acc[cur ^ 1][2 * lane] = re;
        acc[cur ^ 1][2 * lane + 1] = im;
      }
      __syncwarp();
      cur ^= 1;
    }
    if (lane < 16) {  // packed entry (re, re, -im, im)
      const float re = (float)acc[cur][2 * lane], im = (float)acc[cur][2 * lane + 1];
      dst[2 * lane] = make_float2(re, re);
      dst[2 * lane + 1] = make_float2(-im, im);
    }
    return;
  }
  const int n_reg = n_slots - n_fused_slots;
  if (n_reg == 0) return;
  if (spread) {
    const long long t = (gw - n_fw) * 8 + (lane >> 2);
    const bool live = t < (long long)n_reg * batch;
    const int b = live ? (int)(t / n_reg) : 0;
    materialize_spread(slots[n_fused_slots + (live ? t % n_reg : 0)], params ? params + (long long)b * n_params : nullptr,
                       out + (long long)b * mstride, lane, live);
    return;
  }
  const long long t = (gw - n_fw) * 32 + lane;
  if (t >= (long long)n_reg * batch) return;
  const int b = (int)(t / n_reg);
  materialize_one(slots[n_fused_slots + t % n_reg], params ? params + (long long)b * n_params : nullptr,
                  out + (long long)b * mstride);
}

cudaError_t launch_materialize(const MatSlot *d_slots, int n_slots, int n_fused_slots, const FusedMember *d_fused,
                               const double *params, int n_params, int batch, long long mstride, float2 *out,
                               cudaStream_t s) {
  const long long nf = (long long)n_fused_slots * batch, nr = (long long)(n_slots - n_fused_slots) * batch;
  const int per_thread = nf >= kFusedPerThread ? 1 : 0, spread = !per_thread && nr <= kSpreadSlots ? 1 : 0;
  const long long warps = (per_thread ? (nf + 31) / 32 : nf) + (spread ? (nr + 7) / 8 : (nr + 31) / 32);
  if (warps == 0) return cudaSuccess;
  k_materialize<<<(unsigned)warps, 32, 0, s>>>(d_slots, n_slots, n_fused_slots, d_fused, params, n_params, batch, mstride,
                                               out, per_thread, spread);
  return cudaGetLastError();
}

// Slot order the materialisation kernel expects: the fused blocks first.
int order_slots_fused_first(std::vector<MatSlot> &slots) {
  std::stable_partition(slots.begin(), slots.end(), [](const MatSlot &m) { return m.kind == KIND_F2; });
  int n = 0;
  for (const MatSlot &m : slots) n += m.kind == KIND_F2 ? 1 : 0;
  return n;
}

// Closing the output legs with <x| (Sec. 2.2.3) on a contracted state is a gather.
__global__ void k_gather(const float2 *__restrict__ state, int N, int batch, const uint64_t *__restrict__ xs,
                         long long nx, float2 *__restrict__ amps) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nx * batch) return;
  const long long b = i / nx, k = i % nx;
  amps[i] = state[((long long)b << N) + (long long)xs[k]];
}

cudaError_t launch_gather(const float2 *state, int N, int batch, const uint64_t *xs, long long nx, float2 *amps,
                          cudaStream_t s) {
  const long long total = nx * batch;
  if (total == 0) return cudaSuccess;
  k_gather<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(state, N, batch, xs, nx, amps);
  return cudaGetLastError();
}

__global__ void k_scale_grad(double *grad, const double *gout, int batch, int P) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)batch * P) return;
  grad[i] *= gout[i / P];
}

cudaError_t launch_scale_grad(double *grad, const double *gout, int batch, int P, cudaStream_t s) {
  if (gout == nullptr || (long long)batch * P == 0) return cudaSuccess;
  const long long total = (long long)batch * P;
  k_scale_grad<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(grad, gout, batch, P);
  return cudaGetLastError();
}

cudaError_t launch_zero(void *p, size_t bytes, cudaStream_t s) {
  if (bytes == 0) return cudaSuccess;
  return cudaMemsetAsync(p, 0, bytes, s);
}

cudaError_t tables_ready() { return cudaStreamSynchronize(cudaStreamLegacy); }

// ---------------------------------------------------------------------------------------
// Device status word: kernels with bounded waits or finiteness checks record the first
// failure here (atomicCAS from 0); tn_sync_status reads and clears it.
// ---------------------------------------------------------------------------------------
__device__ int g_tn_status = 0;

void *status_word_ptr() {
  void *p = nullptr;
  if (cudaGetSymbolAddress(&p, g_tn_status) != cudaSuccess) return nullptr;
  return p;
}

cudaError_t read_and_clear_status(int *value, cudaStream_t s) {
  cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  int v = 0;
  e = cudaMemcpyFromSymbol(&v, g_tn_status, sizeof(int));
  if (e != cudaSuccess) return e;
  if (v != 0) {
    const int zero = 0;
    e = cudaMemcpyToSymbol(g_tn_status, &zero, sizeof(int));
    if (e == cudaSuccess) e = tables_ready();
    if (e != cudaSuccess) return e;
  }
  *value = v;
  return cudaSuccess;
}

}  // namespace tnq
