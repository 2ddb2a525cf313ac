// Low-dimensional point clouds (d <= 8, float32, packed f32x2): the sweeps over all n m entries
// that are not the iteration's two sums.
//
//   k_direct_wsum  sum_b 2^{v_ab} weight_b value_b of stream A over the inner points: the
//                  envelope gradient (values = the points' coordinates), the transport map
//                  (value columns), and the plain row sum next to it; or, without the exponential,
//                  Round's C delta_c of an l1 or l-inf cost
//   k_direct_max   row maxima: the K pass, the prime pass and the eta = 0 dual bound's second
//                  pass (launch_dual)
//
// Layout as in the iteration's sweeps (lamp_direct.cu): a thread owns R outer points, the inner
// points stream through shared memory in tiles of 128 (cp.async, double-buffered) and every
// thread reads the same pair of them, so that one f32x2 instruction serves two entries and
// nothing is reduced across threads.  Bound by the FMA pipe: 2 d + 4 + 3 NV lane operations (2 NV of
// them the folds of the values' sums) and one ex2 per entry (weighted sums), 2 d + 1 (maxima).  A
// block of 8 x 8 entries per thread with float64 accumulators per tile took 2.78 ms for n = 65536,
// m = 16384, d = 3, three columns (the float64 additions, at 1/64 of the float32 rate, bound it),
// after an evaluation pass of 1.06 ms; the whole call, with the row sums in the same pass and no
// evaluation: 3.93 -> 0.65 ms (0.57 ms with folds every 32 pairs, whose sums of 64 float32 terms were
// up to 8 u off, u = 2^-24, where 8 terms are within 4.5 u).
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "lamp_common.cuh"

namespace lamp {

namespace wsum {

constexpr int kThreads = 256;
constexpr int kTile = kDirectTile;   // inner points per tile
constexpr int kPairs = kTile / 2;
constexpr int kFold = 32;            // pairs between float-float folds of the packed sums of weights
constexpr int kFoldValues = 4;       // ... of the weighted values: 8 float32 terms

__device__ __forceinline__ void cp4(void* dst, const void* src, bool valid) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp16(void* dst, const void* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// unscaled costs of a pair of entries (Consts::cost_op: |x - y|^2, l1, l-inf), coordinates in order
template <int D>
__device__ __forceinline__ uint64_t pair_cost(const uint64_t* x2, const uint64_t* y2, int op) {
  const uint64_t abs2 = 0x7FFFFFFF7FFFFFFFull;
  uint64_t df = f2sub(x2[0], y2[0]);
  uint64_t z2;
  if (op == 0) {
    z2 = f2mul(df, df);
#pragma unroll
    for (int kk = 1; kk < D; ++kk) {
      df = f2sub(x2[kk], y2[kk]);
      z2 = f2fma(df, df, z2);
    }
  } else {
    z2 = df & abs2;
#pragma unroll
    for (int kk = 1; kk < D; ++kk) {
      const uint64_t ad = f2sub(x2[kk], y2[kk]) & abs2;
      if (op == 1) {
        z2 = f2add(z2, ad);
      } else {
        const float2 a = upk(z2), b = upk(ad);
        z2 = pk(fmaxf(a.x, b.x), fmaxf(a.y, b.y));
      }
    }
  }
  return z2;
}

struct Args {
  const float* P_out;
  const float* P_in;
  int64_t n_out, n_in;
  // of both state buffers (the current one is the device's dev->cur):
  const float* own[2];     // outer offsets of stream A, `own_stride` floats apart
  int own_stride;
  const float4* pairs[2];  // inner packed-pair data (entry 2p: {-off, -off, w, w}), padded to whole tiles
  const float* values;   // nv values per inner point, row-major
  int nv;
  double* part;          // weighted sums: [split][n_out][nv + SUM]
  float* pmax;           // maxima: [split][2][n_out]
  int tiles_per_split;
};

// coordinates of tile `it` as pairs [coordinate][2] at stride `rec` floats; pad: points past the
// end read as zeros (0) or as the last point (1)
template <int D>
__device__ __forceinline__ void stage_points(float* buf, int rec, const Args& a, int64_t it, int pad, int tid) {
  const int64_t i0 = it * kTile;
  for (int idx = tid; idx < kTile * D; idx += kThreads) {
    const int b = idx / D, kk = idx - (idx / D) * D;
    const bool in = i0 + b < a.n_in;
    const int64_t g = in ? i0 + b : a.n_in - 1;
    cp4(buf + (b >> 1) * rec + kk * 2 + (b & 1), a.P_in + g * D + kk, in || pad);
  }
}

// NV value columns (COORDS: the inner points' coordinates), SUM: also the sum of the weights alone
// (BILIN: the weights times the unscaled cost, without the exponential)
template <int D, int NV, bool COORDS, bool SUM>
struct SumCfg {
  static constexpr int NA = NV + (SUM ? 1 : 0);           // sums per outer point
  static constexpr int R = D <= 4 && NA <= 4 ? 4 : 2;     // outer points per thread
  static constexpr int DP = (D + 1) & ~1;
  static constexpr int VP = COORDS ? 0 : (NV + 1) & ~1;
  static constexpr int REC = 2 * DP + 4 + 2 * VP;         // floats per pair: coordinates, {-off, w}, values
};

template <int D, int NV, bool COORDS, bool SUM, bool BILIN = false>
__global__ void __launch_bounds__(kThreads, 2)
k_direct_wsum(const Args a, const DevState* __restrict__ dev, const Consts k) {
  using C = SumCfg<D, NV, COORDS, SUM>;
  constexpr int R = C::R, REC = C::REC, NA = C::NA;
  __shared__ __align__(16) float srec[2][kPairs * REC];
  const int tid = threadIdx.x;
  const int cur = dev->cur;
  const float4* __restrict__ pairs = cur ? a.pairs[1] : a.pairs[0];
  const float* __restrict__ owns = cur ? a.own[1] : a.own[0];
  const int64_t o0 = (int64_t)blockIdx.x * (kThreads * R);
  const int64_t ntiles = (a.n_in + kTile - 1) / kTile;
  const int64_t it0 = (int64_t)blockIdx.y * a.tiles_per_split;
  const int64_t it1 = it0 + a.tiles_per_split < ntiles ? it0 + a.tiles_per_split : ntiles;
  const auto stage = [&](int buf, int64_t it) {
    stage_points<D>(srec[buf], REC, a, it, 0, tid);
    for (int p = tid; p < kPairs; p += kThreads)
      cp16(srec[buf] + p * REC + 2 * C::DP, pairs + (it * kPairs + p) * 2);
    if (!COORDS) {
      for (int idx = tid; idx < kTile * NV; idx += kThreads) {
        const int b = idx / (NV > 0 ? NV : 1), q = idx - b * NV;
        const bool ok = q < a.nv && it * kTile + b < a.n_in;
        cp4(srec[buf] + (b >> 1) * REC + 2 * C::DP + 4 + q * 2 + (b & 1),
            ok ? a.values + (it * kTile + b) * a.nv + q : a.values, ok);
      }
    }
  };
  if (it0 < it1) stage(0, it0);
  cp_commit();
  // the padding slots of odd counts are read by the 16-byte loads, never used
  for (int p = tid; p < 2 * kPairs; p += kThreads) {
    float* r = srec[p / kPairs] + (p % kPairs) * REC;
    if (C::DP > D) r[2 * D] = r[2 * D + 1] = 0.f;
    if (C::VP > NV) r[2 * C::DP + 4 + 2 * NV] = r[2 * C::DP + 4 + 2 * NV + 1] = 0.f;
  }
  const SweepF sp = sweep_floats_of(dev, k);
  const uint64_t ah2 = pk(sp.ahA, sp.ahA), al2 = pk(sp.alA, sp.alA);
  const int op = COORDS ? 0 : k.cost_op;
  uint64_t x2[R][D], own[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    int64_t go = o0 + tid + (int64_t)kThreads * r;
    if (go >= a.n_out) go = a.n_out - 1;
#pragma unroll
    for (int kk = 0; kk < D; ++kk) {
      const float v = a.P_out[go * D + kk];
      x2[r][kk] = pk(v, v);
    }
    const float o = -owns[go * a.own_stride];
    own[r] = pk(o, o);
  }
  float hi[R][NA], lo[R][NA];
  uint64_t acc[R][NA];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      hi[r][q] = lo[r][q] = 0.f;
      acc[r][q] = 0ull;
    }
  // the sums [q0, q1) into their float-float pairs
  const auto fold = [&](int q0, int q1) {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int q = 0; q < NA; ++q) {
        if (q < q0 || q >= q1) continue;
        const float2 s = upk(acc[r][q]);
        ff_add(hi[r][q], lo[r][q], s.x + s.y);
        acc[r][q] = 0ull;
      }
  };
  // Weighted values go into the float-float pairs after 8 float32 terms: the gradient and the map
  // take differences of such sums, so their partial sums carry no more rounding than those of
  // kernels that add 8 terms and go on in float64, and the pairs have 48 bits.  The sums of the
  // weights alone (row sums) keep the groups of the iteration's sweeps.
  // Round's C delta_c (BILIN): 32 terms.
  constexpr int kGroup = BILIN ? kFold / 2 : kFold, kStep = NV > 0 ? kFoldValues : kGroup;
  for (int64_t it = it0; it < it1; ++it) {
    const int buf = (int)((it - it0) & 1);
    if (it + 1 < it1) stage(buf ^ 1, it + 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
#pragma unroll 1
    for (int p0 = 0; p0 < kPairs; p0 += kGroup) {
#pragma unroll 1
      for (int p1 = p0; p1 < p0 + kGroup; p1 += kStep) {
#pragma unroll 4
        for (int p = p1; p < p1 + kStep; ++p) {
          const float* rp = srec[buf] + p * REC;
          uint64_t y2[C::DP], v2[C::VP + 1];
#pragma unroll
          for (int kk = 0; kk < C::DP; kk += 2) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(rp + 2 * kk);
            y2[kk] = t.x;
            y2[kk + 1] = t.y;
          }
          const ulonglong2 dA = *reinterpret_cast<const ulonglong2*>(rp + 2 * C::DP);
#pragma unroll
          for (int q = 0; q < C::VP; q += 2) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(rp + 2 * C::DP + 4 + 2 * q);
            v2[q] = t.x;
            v2[q + 1] = t.y;
          }
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const uint64_t z2 = pair_cost<D>(x2[r], y2, op);
            const uint64_t e2 = BILIN ? z2 : exp2_pair(ah2, al2, z2, f2add(own[r], dA.x));
            if (NV == 0) {
              acc[r][0] = f2fma(e2, dA.y, acc[r][0]);
            } else {
              const uint64_t p2 = f2mul(e2, dA.y);
#pragma unroll
              for (int q = 0; q < NV; ++q) acc[r][q] = f2fma(p2, COORDS ? y2[q] : v2[q], acc[r][q]);
              if (SUM) acc[r][NA - 1] = f2add(acc[r][NA - 1], p2);
            }
          }
        }
        fold(0, NV);
      }
      fold(NV, NA);
    }
    __syncthreads();  // every thread is done with srec[buf] before it is refilled
  }
  cp_wait<0>();
  const int na = a.nv + (SUM ? 1 : 0);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t go = o0 + tid + (int64_t)kThreads * r;
    if (go >= a.n_out) continue;
    double* out = a.part + ((int64_t)blockIdx.y * a.n_out + go) * na;
#pragma unroll
    for (int q = 0; q < NV; ++q)
      if (q < a.nv) out[q] = (double)hi[r][q] + (double)lo[r][q];
    if (SUM) out[a.nv] = (double)hi[r][NA - 1] + (double)lo[r][NA - 1];
  }
}

// MODE: kDirectMax: max_b a z - off (no outer offset); kDirectMax2: max_b a z - (own + off) - Br,
// Br in the pairs' weight fields; kDirectKmax: max z and max -z
template <int D, int MODE>
__global__ void __launch_bounds__(kThreads, 2)
k_direct_max(const Args a, const DevState* __restrict__ dev, const Consts k) {
  constexpr int R = 4, DP = (D + 1) & ~1, REC = 2 * DP + 4;
  __shared__ __align__(16) float srec[2][kPairs * REC];
  const int tid = threadIdx.x;
  const int cur = dev->cur;
  const float4* __restrict__ pairs = cur ? a.pairs[1] : a.pairs[0];
  const float* __restrict__ owns = cur ? a.own[1] : a.own[0];
  const int64_t o0 = (int64_t)blockIdx.x * (kThreads * R);
  const int64_t ntiles = (a.n_in + kTile - 1) / kTile;
  const int64_t it0 = (int64_t)blockIdx.y * a.tiles_per_split;
  const int64_t it1 = it0 + a.tiles_per_split < ntiles ? it0 + a.tiles_per_split : ntiles;
  const auto stage = [&](int buf, int64_t it) {
    stage_points<D>(srec[buf], REC, a, it, MODE == kDirectKmax, tid);
    if (MODE != kDirectKmax)
      for (int p = tid; p < kPairs; p += kThreads) cp16(srec[buf] + p * REC + 2 * DP, pairs + (it * kPairs + p) * 2);
  };
  if (it0 < it1) stage(0, it0);
  cp_commit();
  if (DP > D)
    for (int p = tid; p < 2 * kPairs; p += kThreads) {
      float* r = srec[p / kPairs] + (p % kPairs) * REC;
      r[2 * D] = r[2 * D + 1] = 0.f;
    }
  const SweepF sp = sweep_floats_of(dev, k);
  const uint64_t ah2 = pk(sp.ahA, sp.ahA), al2 = pk(sp.alA, sp.alA);
  uint64_t x2[R][D], own[R];
  float mx[R], mn[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    int64_t go = o0 + tid + (int64_t)kThreads * r;
    if (go >= a.n_out) go = a.n_out - 1;
#pragma unroll
    for (int kk = 0; kk < D; ++kk) {
      const float v = a.P_out[go * D + kk];
      x2[r][kk] = pk(v, v);
    }
    const float o = MODE == kDirectMax2 ? -owns[go * a.own_stride] : 0.f;
    own[r] = pk(o, o);
    mx[r] = mn[r] = -INFINITY;
  }
  for (int64_t it = it0; it < it1; ++it) {
    const int buf = (int)((it - it0) & 1);
    if (it + 1 < it1) stage(buf ^ 1, it + 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
#pragma unroll 4
    for (int p = 0; p < kPairs; ++p) {
      const float* rp = srec[buf] + p * REC;
      uint64_t y2[DP];
#pragma unroll
      for (int kk = 0; kk < DP; kk += 2) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(rp + 2 * kk);
        y2[kk] = t.x;
        y2[kk + 1] = t.y;
      }
      const ulonglong2 dA = MODE == kDirectKmax ? ulonglong2{0ull, 0ull}
                                                : *reinterpret_cast<const ulonglong2*>(rp + 2 * DP);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        uint64_t u = pair_cost<D>(x2[r], y2, k.cost_op);
        if (MODE == kDirectMax) u = f2fma(ah2, u, dA.x);
        if (MODE == kDirectMax2) u = f2sub(f2fma(al2, u, f2fma(ah2, u, f2add(own[r], dA.x))), dA.y);
        const float2 f = upk(u);
        mx[r] = fmaxf(mx[r], fmaxf(f.x, f.y));
        if (MODE == kDirectKmax) mn[r] = fmaxf(mn[r], fmaxf(-f.x, -f.y));
      }
    }
    __syncthreads();
  }
  cp_wait<0>();
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t go = o0 + tid + (int64_t)kThreads * r;
    if (go >= a.n_out) continue;
    // stream B's maxima are not used under the shared row shift
    a.pmax[((int64_t)blockIdx.y * 2 + 0) * a.n_out + go] = mx[r];
    a.pmax[((int64_t)blockIdx.y * 2 + 1) * a.n_out + go] = MODE == kDirectKmax ? mn[r] : mx[r];
  }
}

// the weights of stream A in pair data become the float32 values of v (padding entries keep theirs, 0)
__global__ void __launch_bounds__(256)
k_weight_pairs(const double* __restrict__ v, int64_t np, float4* __restrict__ pairs) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < np) reinterpret_cast<float*>(pairs + (e >> 1) * 2)[2 + (e & 1)] = (float)v[e];
}

// rowterm_i = s dr_i sum_s part[s][i]
__global__ void __launch_bounds__(256)
k_bilinear_fin(const double* __restrict__ part, int splits, int64_t np, const double* __restrict__ dr, double s,
               double* __restrict__ rowterm) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  double acc = 0.0;
#pragma unroll 8
  for (int u = 0; u < splits; ++u) acc += part[(int64_t)u * np + i];
  rowterm[i] = s * acc * dr[i];
}

// out_i = 2 s (mass_i p_i - weight_i sum_s part[s][i]), one thread per coordinate
__global__ void __launch_bounds__(256)
k_wgrad_fin(const double* __restrict__ part, int splits, int64_t np, int d, const float* __restrict__ P,
            const double* __restrict__ mass, const float4* __restrict__ wsrc, double s, float* __restrict__ out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= np * d) return;
  const int64_t i = e / d;
  double acc = 0.0;
#pragma unroll 8
  for (int u = 0; u < splits; ++u) acc += part[(int64_t)u * np * d + e];
  out[e] = (float)(2.0 * s * (mass[i] * (double)P[e] - (double)wsrc[i].y * acc));
}

// transport map, rows: out_i = sum_s acc / sum_s S, and log Z_i as the row finalize forms it; rows
// whose sum leaves the representable range set LAMP_E_NUMERIC as there
__global__ void __launch_bounds__(128)
k_wmap_rows_fin(const double* __restrict__ part, int splits, int64_t n, int nv, const Work w,
                float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) w.dev->t_logz = w.dev->t;
  if (i >= n) return;
  const int cur = w.dev->cur;
  const int na = nv + 1;
  double S = 0.0;
#pragma unroll 8
  for (int s = 0; s < splits; ++s) S += part[((int64_t)s * n + i) * na + nv];
  if (!(S > 1.0 / 1.0e36 && S < 1.0e36)) {
    atomicExch(&w.dev->status, 5 /* LAMP_E_NUMERIC */);
    S = S > 0.0 ? S : 1.0;
  }
  w.logZ[i] = kLn2 * ((double)w.rowshift[cur][i].x + log2(S));  // direct form: no |x_i|^2 term
  const double inv = 1.0 / S;
  for (int q = 0; q < nv; ++q) {
    double acc = 0.0;
#pragma unroll 8
    for (int s = 0; s < splits; ++s) acc += part[((int64_t)s * n + i) * na + q];
    out[i * nv + q] = (float)(acc * inv);
  }
}

// transport map, columns, first step: log Z_i and the inner pair data {-Rq_i, 1 / S_i} of the rows
// (entries past n: {-2^100, 0})
__global__ void __launch_bounds__(128)
k_wmap_weights(const double* __restrict__ part, int splits, int64_t n, int64_t n_pad, const Work w,
               float4* __restrict__ pairs) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) w.dev->t_logz = w.dev->t;
  if (i >= n_pad) return;
  const int cur = w.dev->cur;
  float* f = reinterpret_cast<float*>(pairs + (i >> 1) * 2);
  const int h = (int)(i & 1);
  if (i >= n) {
    f[h] = -0x1p100f;
    f[2 + h] = 0.f;
    return;
  }
  double S = 0.0;
#pragma unroll 8
  for (int s = 0; s < splits; ++s) S += part[(int64_t)s * n + i];
  if (!(S > 1.0 / 1.0e36 && S < 1.0e36)) {
    atomicExch(&w.dev->status, 5 /* LAMP_E_NUMERIC */);
    S = S > 0.0 ? S : 1.0;
  }
  const float rq = w.rowshift[cur][i].x;
  w.logZ[i] = kLn2 * ((double)rq + log2(S));
  f[h] = -rq;
  f[2 + h] = (float)(1.0 / S);
}

// transport map, columns: out_j = w_j sum_s acc
__global__ void __launch_bounds__(256)
k_wmap_cols_fin(const double* __restrict__ part, int splits, int64_t m, int nv, const Work w,
                float* __restrict__ out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m * nv) return;
  double acc = 0.0;
#pragma unroll 8
  for (int s = 0; s < splits; ++s) acc += part[(int64_t)s * m * nv + e];
  out[e] = (float)((double)w.colq[w.dev->cur][e / nv].y * acc);
}

inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

template <int D, int NV, bool COORDS, bool SUM>
cudaError_t go_sum(Args a, int splits, const Work& w, const Consts& k, cudaStream_t st) {
  a.tiles_per_split = (int)cdiv(cdiv(a.n_in, kTile), splits);
  const dim3 grid((unsigned)cdiv(a.n_out, (int64_t)kThreads * SumCfg<D, NV, COORDS, SUM>::R), (unsigned)splits);
  k_direct_wsum<D, NV, COORDS, SUM><<<grid, kThreads, 0, st>>>(a, w.dev, k);
  return cudaGetLastError();
}

// nv = 0: the sum of the weights alone
template <int D, bool SUM>
cudaError_t go_values(const Args& a, int splits, const Work& w, const Consts& k, cudaStream_t st) {
  switch (a.nv) {
    case 1: return go_sum<D, 1, false, SUM>(a, splits, w, k, st);
    case 2: return go_sum<D, 2, false, SUM>(a, splits, w, k, st);
    case 3: return go_sum<D, 3, false, SUM>(a, splits, w, k, st);
    case 4: return go_sum<D, 4, false, SUM>(a, splits, w, k, st);
    default: return go_sum<D, 8, false, SUM>(a, splits, w, k, st);
  }
}

template <int D, int MODE>
cudaError_t go_max(Args a, int splits, const Work& w, const Consts& k, cudaStream_t st) {
  a.tiles_per_split = (int)cdiv(cdiv(a.n_in, kTile), splits);
  k_direct_max<D, MODE><<<dim3((unsigned)cdiv(a.n_out, kThreads * 4), (unsigned)splits), kThreads, 0, st>>>(a, w.dev, k);
  return cudaGetLastError();
}

// f(std::integral_constant<int, d>) for 1 <= d <= 8
template <class F>
cudaError_t by_dim(int d, F&& f) {
  switch (d) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 5: return f(std::integral_constant<int, 5>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 7: return f(std::integral_constant<int, 7>{});
    case 8: return f(std::integral_constant<int, 8>{});
    default: return cudaErrorNotSupported;
  }
}

Args side(const Inputs& in, const Consts& k, const Work& w, bool rows) {
  Args a{};
  a.P_out = rows ? in.x : in.y;
  a.P_in = rows ? in.y : in.x;
  a.n_out = rows ? k.n : k.m;
  a.n_in = rows ? k.m : k.n;
  a.own_stride = rows ? 2 : 4;
  for (int b = 0; b < 2; ++b) {
    a.own[b] = rows ? reinterpret_cast<const float*>(w.rowshift[b]) : reinterpret_cast<const float*>(w.colq[b]);
    a.pairs[b] = rows ? w.colq2[b] : w.g2row2;
  }
  return a;
}

}  // namespace wsum

// outer points per CTA for `sums` sums per point, and inner points per tile
int wsum_outer(int d, int sums) { return wsum::kThreads * (d <= 4 && sums <= 4 ? 4 : 2); }
int wsum_inner() { return wsum::kTile; }

cudaError_t direct_grad(bool rows, const Inputs& in, const Work& w, const Consts& k, int cur, int splits, double* part,
                        float* out, cudaStream_t st) {
  wsum::Args a = wsum::side(in, k, w, rows);
  a.nv = k.d;
  a.part = part;
  cudaError_t e = wsum::by_dim(k.d, [&](auto dd) {
    constexpr int D = decltype(dd)::value;
    return wsum::go_sum<D, D, true, false>(a, splits, w, k, st);
  });
  if (e != cudaSuccess) return e;
  wsum::k_wgrad_fin<<<(unsigned)wsum::cdiv(a.n_out * k.d, 256), 256, 0, st>>>(
      part, splits, a.n_out, k.d, a.P_out, rows ? in.r : w.colA, rows ? w.g2row : w.colq[cur], k.s, out);
  return cudaGetLastError();
}

cudaError_t direct_map(int side, const Inputs& in, const Work& w, const Consts& k, const float* V, int nv,
                       int splits_rows, int splits_cols, double* part, float4* pairs, float* out, cudaStream_t st) {
  wsum::Args a = wsum::side(in, k, w, true);
  a.part = part;
  a.values = V;
  a.nv = side == 0 ? nv : 0;
  cudaError_t e = wsum::by_dim(k.d, [&](auto dd) {
    constexpr int D = decltype(dd)::value;
    if (side == 0) return wsum::go_values<D, true>(a, splits_rows, w, k, st);
    return wsum::go_sum<D, 0, false, true>(a, splits_rows, w, k, st);
  });
  if (e != cudaSuccess) return e;
  if (side == 0) {
    wsum::k_wmap_rows_fin<<<(unsigned)wsum::cdiv(k.n, 128), 128, 0, st>>>(part, splits_rows, k.n, nv, w, out);
    return cudaGetLastError();
  }
  const int64_t n_pad = wsum::cdiv(k.n, wsum::kTile) * wsum::kTile;
  wsum::k_wmap_weights<<<(unsigned)wsum::cdiv(n_pad, 128), 128, 0, st>>>(part, splits_rows, k.n, n_pad, w, pairs);
  a = wsum::side(in, k, w, false);
  a.pairs[0] = a.pairs[1] = pairs;
  a.part = part;
  a.values = V;
  a.nv = nv;
  e = wsum::by_dim(k.d, [&](auto dd) { return wsum::go_values<decltype(dd)::value, false>(a, splits_cols, w, k, st); });
  if (e != cudaSuccess) return e;
  wsum::k_wmap_cols_fin<<<(unsigned)wsum::cdiv(k.m * nv, 256), 256, 0, st>>>(part, splits_cols, k.m, nv, w, out);
  return cudaGetLastError();
}

cudaError_t direct_bilinear(const Inputs& in, const Work& w, const Consts& k, int splits, const double* dr,
                            const double* dc, float4* pairs, double* part, double* rowterm, cudaStream_t st) {
  wsum::k_weight_pairs<<<(unsigned)wsum::cdiv(k.m, 256), 256, 0, st>>>(dc, k.m, pairs);
  wsum::Args a = wsum::side(in, k, w, true);
  a.pairs[0] = a.pairs[1] = pairs;
  a.part = part;
  a.tiles_per_split = (int)wsum::cdiv(wsum::cdiv(k.m, wsum::kTile), splits);
  cudaError_t e = wsum::by_dim(k.d, [&](auto dd) {
    constexpr int D = decltype(dd)::value;
    const dim3 grid((unsigned)wsum::cdiv(k.n, (int64_t)wsum::kThreads * wsum::SumCfg<D, 0, false, true>::R),
                    (unsigned)splits);
    wsum::k_direct_wsum<D, 0, false, true, true><<<grid, wsum::kThreads, 0, st>>>(a, w.dev, k);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  wsum::k_bilinear_fin<<<(unsigned)wsum::cdiv(k.n, 256), 256, 0, st>>>(part, splits, k.n, dr, k.s, rowterm);
  return cudaGetLastError();
}

cudaError_t direct_max(int mode, const Inputs& in, const Work& w, const Consts& k, int splits, cudaStream_t st) {
  wsum::Args a = wsum::side(in, k, w, true);
  a.pmax = w.rowmax;
  return wsum::by_dim(k.d, [&](auto dd) {
    constexpr int D = decltype(dd)::value;
    if (mode == kDirectMax) return wsum::go_max<D, kDirectMax>(a, splits, w, k, st);
    if (mode == kDirectMax2) return wsum::go_max<D, kDirectMax2>(a, splits, w, k, st);
    return wsum::go_max<D, kDirectKmax>(a, splits, w, k, st);
  });
}

}  // namespace lamp
