// Pieces shared by the packed direct-form sweeps (lamp_direct.cu, lamp_direct_small.cu): the
// inner points' records in shared memory and the arithmetic of one pair of entries.
#pragma once

#include <cmath>
#include <cstdint>

#include "lamp_common.cuh"

namespace lamp {

enum DirectSweep : int { M_ROWSUM = 0, M_COLSUM = 1 };

constexpr int kDTile = kDirectTile;  // inner points per shared-memory tile
constexpr int kDPairs = kDTile / 2;  // pairs per tile
constexpr int kDFold = 32;           // pairs between float-float folds of the packed sums

template <int D>
struct DirectCfg {
  static constexpr int R = D <= 4 ? 4 : 2;  // outer points per thread
  static constexpr int DP = (D + 1) & ~1;   // coordinates per pair record, even
  static constexpr int REC = DP * 2 + 8;    // floats per pair record: coords [DP][2], offsets/weights A, B
};

__device__ __forceinline__ void cp_async4(void* dst, const void* src, bool valid) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// stage inner tile `it` (points it*128 ..) into the record buffer `rec`
template <int D>
__device__ __forceinline__ void direct_stage(float* rec, const float* __restrict__ P_in, int64_t n_in,
                                             const float4* __restrict__ pairs, int64_t it, int tid, int nthreads) {
  using C = DirectCfg<D>;
  const int64_t i0 = it * kDTile;
  for (int idx = tid; idx < kDTile * D; idx += nthreads) {
    const int b = idx / D, k = idx - (idx / D) * D;
    const bool ok = i0 + b < n_in;
    const float* src = ok ? P_in + (i0 + b) * D + k : P_in;
    cp_async4(rec + (b >> 1) * C::REC + k * 2 + (b & 1), src, ok);
  }
  // offsets / weights: pairs [2(i0/2 + p)] (stream A) and [2(i0/2 + p) + 1] (stream B);
  // the pair arrays are padded to 128 entries, so a whole tile is always in bounds
  for (int idx = tid; idx < kDPairs * 2; idx += nthreads) {
    const int p = idx >> 1, s = idx & 1;
    cp_async16(rec + p * C::REC + C::DP * 2 + 4 * s, pairs + (i0 >> 1) * 2 + idx);
  }
}

// |x_k - y_k| for a pair of entries: clear both sign bits
__device__ __forceinline__ uint64_t f2abs(uint64_t v) {
  uint64_t r;
  asm("and.b64 %0, %1, 0x7FFFFFFF7FFFFFFF;" : "=l"(r) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t f2max(uint64_t a, uint64_t b) {
  const float2 x = upk(a), y = upk(b);
  return pk(fmaxf(x.x, y.x), fmaxf(x.y, y.y));
}

// one pair of inner points, as read from its record
template <int D>
struct DirectPair {
  uint64_t y2[DirectCfg<D>::DP];
  uint64_t oA2, wA2, dC2, wB2;  // stream A: -offset, weight; stream B: dB (columns), weight
  __device__ __forceinline__ void load(const float* rp) {
    constexpr int DP = DirectCfg<D>::DP;
#pragma unroll
    for (int kk = 0; kk < DP; kk += 2) {
      const float4 t = *reinterpret_cast<const float4*>(rp + 2 * kk);
      y2[kk] = pk(t.x, t.y);
      y2[kk + 1] = pk(t.z, t.w);
    }
    const float4 dA = *reinterpret_cast<const float4*>(rp + 2 * DP);
    const float4 dB = *reinterpret_cast<const float4*>(rp + 2 * DP + 4);
    oA2 = pk(dA.x, dA.y);
    wA2 = pk(dA.z, dA.w);
    dC2 = pk(dB.x, dB.y);
    wB2 = pk(dB.z, dB.w);
  }
};

// sums per outer point
template <int MODE, int EV>
constexpr int kDirectSums = MODE == M_ROWSUM && EV ? 1 : 2;

// the two entries (outer point, pair) added to the packed sums acc: {A, B}, or in an evaluation
// pass (EV) stream A alone, {A} (rows) or {A, cost-weighted A} (columns).  MODE = M_ROWSUM or
// M_COLSUM; CK = the ground cost (Consts::cost_op): 0 |x - y|^2, 1 l1, 2 l-inf.  own, ownD:
// -offset of the outer point, and a column's dB = BqA - BcolB
template <int MODE, int D, int EV, int CK, int NACC>
__device__ __forceinline__ void direct_pair(const uint64_t (&x2)[D], uint64_t own, uint64_t ownD,
                                            const DirectPair<D>& t, uint64_t ahA2, uint64_t alA2, uint64_t da2,
                                            uint64_t (&acc)[NACC]) {
  uint64_t z2;
  if constexpr (CK == 0) {
    uint64_t df = f2sub(x2[0], t.y2[0]);
    z2 = f2mul(df, df);
#pragma unroll
    for (int kk = 1; kk < D; ++kk) {
      df = f2sub(x2[kk], t.y2[kk]);
      z2 = f2fma(df, df, z2);
    }
  } else {
    z2 = f2abs(f2sub(x2[0], t.y2[0]));
#pragma unroll
    for (int kk = 1; kk < D; ++kk) {
      const uint64_t ad = f2abs(f2sub(x2[kk], t.y2[kk]));
      z2 = CK == 1 ? f2add(z2, ad) : f2max(z2, ad);
    }
  }
  const uint64_t vA = f2fma(alA2, z2, f2fma(ahA2, z2, f2add(own, t.oA2)));
  const float2 vAf = upk(vA);
  const uint64_t eA = pk(ex2(vAf.x), ex2(vAf.y));
  if constexpr (EV && MODE == M_COLSUM) {
    const uint64_t pA = f2mul(eA, t.wA2);
    acc[0] = f2add(acc[0], pA);
    acc[1] = f2fma(z2, pA, acc[1]);
  } else {
    acc[0] = f2fma(eA, t.wA2, acc[0]);
  }
  if constexpr (!EV) {
    const float2 vBf = upk(f2fma(da2, z2, f2add(vA, MODE == M_ROWSUM ? t.dC2 : ownD)));
    const uint64_t eB = pk(ex2(vBf.x), ex2(vBf.y));
    // row sums of stream B carry no weight (it is inside dB_j); column sums weight by q^B_i
    if constexpr (MODE == M_ROWSUM) acc[1] = f2add(acc[1], eB);
    else acc[1] = f2fma(eB, t.wB2, acc[1]);
  }
}

}  // namespace lamp
