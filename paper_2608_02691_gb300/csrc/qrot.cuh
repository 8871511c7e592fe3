// Query rotation of one (sequence, KV head), shared by its own kernel, the
// fused decode-step prologue (decode.cu) and the one-launch decode of small
// batches (decode_tc.cu).
#pragma once

#include "decode_common.cuh"

namespace optr {

// One CTA per (sequence, KV head), 512 threads = 4 slices x 128 channels:
// slice s sums q[i] R[i][j] over i in [32s, 32s+32) for the 4 query heads of
// the group, the slices are added in shared memory.
constexpr int kQrotThreads = 512;

struct QrotSmem {
  float qsm[4][kD];
  float part[4][4][kD];  // [slice][head][channel]
  float qrs[4][kD];
  float hmax[4][4];
  int warp_tot[2][kQrotThreads / 32];
  long long koff_part[kQrotThreads / 32][kGroups];
};

// This thread's slice of R_k[h]: rows [32 sl, 32 sl + 32) of column j, thread
// (sl, j) = (tid / 128, tid % 128); library-owned, so it may be loaded before
// pdl_wait().
__device__ __forceinline__ void load_rotation_slice(const float* __restrict__ R_k, int h,
                                                    float (&rv)[32]) {
  const int sl = threadIdx.x >> 7, j = threadIdx.x & 127;
  const float* R = R_k + (size_t)h * kD * kD + (size_t)(32 * sl) * kD + j;
#pragma unroll
  for (int i = 0; i < 32; ++i) rv[i] = __ldg(R + i * kD);  // all in flight
}

// The 4 query rows at q rotated by the loaded slices: q' (qf [4][128], may be
// null), its group sums (qs [4][4]), the tensor-core fragments (frag [32][16]),
// their code-offset sums (koff [4][4][2]) and inverse prescales (invs [4]), in
// global or shared memory.  512 threads.
__device__ __forceinline__ void rotate_query(
    QrotSmem& sm, const __nv_bfloat16* __restrict__ q, const float (&rv)[32], float qscale,
    float* qf, float* qs, uint32_t* frag, float* koff, float* invs) {
  float (&qsm)[4][kD] = sm.qsm;
  float (&part)[4][4][kD] = sm.part;
  float (&qrs)[4][kD] = sm.qrs;
  float (&hmax)[4][4] = sm.hmax;
  long long (&koff_part)[kQrotThreads / 32][kGroups] = sm.koff_part;
  const int tid = threadIdx.x;
  const int sl = tid >> 7, j = tid & 127;
  const int warp = tid >> 5, lane = tid & 31;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  // Global stores wait until the end: a __syncthreads() after a store waits
  // for it to complete, which made each phase an L2 round trip.
  {
    const int r = tid >> 7;  // 512 threads load the 4 x 128 query values
    qsm[r][j] = __bfloat162float(q[r * kD + j]);
  }
  __syncthreads();
#pragma unroll
  for (int i4 = 0; i4 < 8; ++i4)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 qv = *reinterpret_cast<const float4*>(&qsm[r][32 * sl + 4 * i4]);
      acc[r] = fmaf(qv.x, rv[4 * i4 + 0], acc[r]);
      acc[r] = fmaf(qv.y, rv[4 * i4 + 1], acc[r]);
      acc[r] = fmaf(qv.z, rv[4 * i4 + 2], acc[r]);
      acc[r] = fmaf(qv.w, rv[4 * i4 + 3], acc[r]);
    }
#pragma unroll
  for (int r = 0; r < 4; ++r) part[sl][r][j] = acc[r];
  __syncthreads();
  // thread (r, j): the 4 slices of head r, channel j (512 threads)
  const int qr = tid >> 7;
  const float qx = (part[0][qr][j] + part[1][qr][j] + part[2][qr][j] + part[3][qr][j]) * qscale;
  float qsum = qx;
  {
    const int r = qr;
    const float x = qx;
    qrs[r][j] = x;
    float s = x, a = fabsf(x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, o);
      a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
    }
    qsum = s;
    if (lane == 0) hmax[r][j >> 5] = a;
  }
  __syncthreads();
  // Tensor-core B fragments (see decode_tc.cu): per head a power-of-two
  // prescale 2^e brings max |q'| * 2^e into [2^13, 2^14), so that the fp16
  // hi/lo split stays in the normal range for all but tiny elements.  The
  // key codes enter the MMA as 1024 + code * 2^pos (pos = kCodePos[G&1][r]),
  // so the fragment of channel 32G + 4w + r also carries 2^-pos, and koff
  // holds the offset sum 1024 * sum over the group of the fragment values,
  // per (query head, group, hi/lo column), which the MMA starts from
  // (negated) so that the accumulator sums code * q' exactly as before.
  {
    const int ridx = tid;  // 512 fragment registers, one per thread
    const int L = ridx >> 4, reg = ridx & 15;
    const int G = reg >> 2, kk = (reg >> 1) & 1, which = reg & 1;
    const int g = L >> 2, c = L & 3;
    const int head = g >> 1, part_hl = g & 1;
    const float mx = fmaxf(fmaxf(hmax[head][0], hmax[head][1]),
                           fmaxf(hmax[head][2], hmax[head][3]));
    const int e = max(-100, min(100, mx > 0.f ? 13 - ilogbf(mx) : 0));
    const int r = 2 * kk + which;
    const int ch = 32 * G + 8 * c + r;   // low half; +4 high
    const float sc = ldexpf(1.f, e - code_pos(G, r));
    const float x0 = qrs[head][ch] * sc, x1 = qrs[head][ch + 4] * sc;
    const __half h0 = __float2half_rn(x0), h1 = __float2half_rn(x1);
    __half v0 = h0, v1 = h1;
    if (part_hl) {
      v0 = __float2half_rn(x0 - __half2float(h0));
      v1 = __float2half_rn(x1 - __half2float(h1));
    }
    const uint32_t fragv =
        (uint32_t)__half_as_ushort(v0) | ((uint32_t)__half_as_ushort(v1) << 16);
    // offset sum over the 32 channels of group G for column g: reduce over
    // (kk, which) = lane bits 0-1, c bit 0 = lane bit 4, c bit 1 = warp bit 0.
    // Exact, in fixed point: an fp16 value times 2^24 is an integer below
    // 2^40, so 64 of them sum exactly in int64; one rounding to float, then
    // 1024 * 2^-24 = 2^-14 (exact) gives the correctly rounded koff.
    long long t = __float2ll_rn(__half2float(v0) * 16777216.0f) +
                  __float2ll_rn(__half2float(v1) * 16777216.0f);
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    t += __shfl_xor_sync(0xffffffffu, t, 2);
    t += __shfl_xor_sync(0xffffffffu, t, 16);
    if ((lane & 15) % 4 == 0) koff_part[warp][G] = t;
    __syncthreads();
    if (tid < 32) {  // tid = (g, G): koff[head][G][hl] for column g
      const int gg = tid >> 2, GG = tid & 3;
      const long long tot = koff_part[2 * gg][GG] + koff_part[2 * gg + 1][GG];
      koff[(gg >> 1) * 8 + GG * 2 + (gg & 1)] =
          __ll2float_rn(tot) * 0x1p-14f;
    }
    if (ridx < 4) {
      const float m2 = fmaxf(fmaxf(hmax[ridx][0], hmax[ridx][1]),
                             fmaxf(hmax[ridx][2], hmax[ridx][3]));
      const int e2 = max(-100, min(100, m2 > 0.f ? 13 - ilogbf(m2) : 0));
      invs[ridx] = ldexpf(1.f, -e2);
    }
    frag[ridx] = fragv;
  }
  if (qf != nullptr) qf[qr * kD + j] = qx;
  if (lane == 0) qs[qr * kGroups + (j >> 5)] = qsum;
}

}  // namespace optr
