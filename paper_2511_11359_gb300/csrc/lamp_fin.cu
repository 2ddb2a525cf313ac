// Finalize kernels of an iteration: the O(n) and O(m) float64 work between the sweeps.
//
//   RF (k_row_fin)  S_i of both streams -> the row weights q_i = r_i / S_i and the next row
//                   shifts; evaluation passes also write log Z_i and <r, log Z>
//   CF (k_col_fin)  both column marginals -> the dual step of Alg. 2 (thetabar, nu, thetahat,
//                   tclip), the residual ||col - c||_1, the next sweep's column data; its last
//                   block reduces the block partials and applies or rejects the update
//
// What bounds them: this part issues one float64 instruction per scheduler every 64 cycles
// (measured: a dependent chain and independent chains alike take 64 cycles per warp
// instruction, a division 565, log2 2215, tanh 977), so a kernel's time is the number of
// float64 instructions of the longest warp, plus the latency of its loads and of the last
// block's tail.  Hence: the two streams of a point are worked by two warps on different
// schedulers, what only an evaluation pass reports is computed there alone, the mirror step's
// gain is kept per column, divisions start from a float32 reciprocal, the row shift's log2
// comes from a table, and the parameters of the next iteration are prepared by a block of RF
// instead of by CF's last thread.  RF + CF together, against one thread per point doing all of
// it in blocks of 128: 22.9 -> 12.8 us at 4096 points (16 splits), 37.5 -> 24.4 us at 2^15 (19
// splits).
#include <cmath>

#include "lamp_common.cuh"

namespace lamp {

namespace {

constexpr int kPts = kFinPoints;      // points of a block
constexpr int kThreads = 2 * kPts;    // four warps, one per scheduler: two per stream
constexpr int kWarps = kPts / 32;     // warps per stream

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// a / b, b within float32's normal range: a float32 reciprocal, one Newton step (2^-46), and
// the quotient corrected by its exact remainder: 5 float64 operations instead of the 9 of a
// division.  The error before the last rounding is ~2^-93 of the quotient, so the result is
// the correctly rounded one except where the quotient lies that close to a rounding boundary.
__device__ __forceinline__ double div_seeded(double a, double b) {
  float yf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"((float)b));
  const double y0 = (double)yf;
  const double y = fma(y0, fma(-b, y0, 1.0), y0);
  const double q = a * y;
  return fma(fma(-q, b, a), y, q);
}

// nearest multiple of the power of two g, ties to even: adding and subtracting 1.5 2^52 g
// rounds |x| < 2^51 g there (two operations; the explicit roundings keep x's product unfused)
__device__ __forceinline__ double quantize_add(double x, double g) {
  const double M = g * 6755399441055744.0;
  return __dadd_rn(__dadd_rn(x, M), -M);
}

// log2 by table lookup (P. T. P. Tang, "Table-driven implementation of the logarithm function in
// IEEE floating-point arithmetic", ACM TOMS 16(4), 1990): x = 2^e m, inv_i ~ 1/m from the top 7
// bits of m, log2 x = e - log2 inv_i + log2(1 + r), r = m inv_i - 1, |r| <= 2^-8, and the Taylor
// series of log2(1 + r) to r^7 (remainder below 2^-66).  For normal x > 0; 10 float64
// operations instead of the 34 of log2, whose result differs in the last bit.  Used for the row
// shifts, which are rounded to the offset grid.
struct LogEntry {
  double inv, t;  // a float32 number near 1/m, and -log2 of it
};
__device__ const LogEntry kLogTab[128] = {
    {0x1.fe01fe0000000p-1, 0x1.709c4848ff3ddp-8}, {0x1.fa11ca0000000p-1, 0x1.13632eb186117p-6},
    {0x1.f6310a0000000p-1, 0x1.c93660ce8fe6bp-6}, {0x1.f25f640000000p-1, 0x1.3ed30f682c99bp-5},
    {0x1.ee9c800000000p-1, 0x1.985bf0a9f1682p-5}, {0x1.eae8080000000p-1, 0x1.f1389043d4afep-5},
    {0x1.e741aa0000000p-1, 0x1.24b5bc1e1dbfcp-4}, {0x1.e3a9180000000p-1, 0x1.507b7eafe13b6p-4},
    {0x1.e01e020000000p-1, 0x1.7beee7e3206a7p-4}, {0x1.dca01e0000000p-1, 0x1.a7111b55df32fp-4},
    {0x1.d92f220000000p-1, 0x1.d1e350a4f6b57p-4}, {0x1.d5cac80000000p-1, 0x1.fc66a14d0527ep-4},
    {0x1.d272ca0000000p-1, 0x1.134e1cdc84c46p-3}, {0x1.cf26e60000000p-1, 0x1.284293339b4a1p-3},
    {0x1.cbe6da0000000p-1, 0x1.3d1142d675bdep-3}, {0x1.c8b2660000000p-1, 0x1.51bab70047027p-3},
    {0x1.c5894e0000000p-1, 0x1.663f699674dfdp-3}, {0x1.c26b540000000p-1, 0x1.7a9fe9b172390p-3},
    {0x1.bf583e0000000p-1, 0x1.8edcb48259c41p-3}, {0x1.bc4fd60000000p-1, 0x1.a2f6347eaa238p-3},
    {0x1.b951e20000000p-1, 0x1.b6ecf61ac13c6p-3}, {0x1.b65e2e0000000p-1, 0x1.cac1655b653e1p-3},
    {0x1.b374840000000p-1, 0x1.de7402d451bb0p-3}, {0x1.b094b40000000p-1, 0x1.f2052d8777449p-3},
    {0x1.adbe880000000p-1, 0x1.02baba0dbb1edp-2}, {0x1.aaf1d20000000p-1, 0x1.0c629ab11b4d6p-2},
    {0x1.a82e660000000p-1, 0x1.15fa643277d88p-2}, {0x1.a574100000000p-1, 0x1.1f82610d07e69p-2},
    {0x1.a2c2a80000000p-1, 0x1.28fab511c6b50p-2}, {0x1.a01a020000000p-1, 0x1.326394e238a67p-2},
    {0x1.9d79f20000000p-1, 0x1.3bbd381f99a2dp-2}, {0x1.9ae24e0000000p-1, 0x1.4507d24038eb2p-2},
    {0x1.9852f00000000p-1, 0x1.4e438b1f6332ep-2}, {0x1.95cbb00000000p-1, 0x1.57709467b5eb3p-2},
    {0x1.934c680000000p-1, 0x1.608f1b2b7f437p-2}, {0x1.90d4f20000000p-1, 0x1.699f4f0f94941p-2},
    {0x1.8e65280000000p-1, 0x1.72a16250a7782p-2}, {0x1.8bfce80000000p-1, 0x1.7b957adc2ff3bp-2},
    {0x1.899c100000000p-1, 0x1.847bc0e55cd91p-2}, {0x1.87427c0000000p-1, 0x1.8d54667727585p-2},
    {0x1.84f00c0000000p-1, 0x1.961f90e87e59dp-2}, {0x1.82a4a00000000p-1, 0x1.9edd67b6077b9p-2},
    {0x1.8060180000000p-1, 0x1.a78e14869136bp-2}, {0x1.7e22560000000p-1, 0x1.b031bb7403122p-2},
    {0x1.7beb3a0000000p-1, 0x1.b8c88a63afc52p-2}, {0x1.79baa60000000p-1, 0x1.c152a99f3049ep-2},
    {0x1.7790820000000p-1, 0x1.c9d02be2a14a1p-2}, {0x1.756cac0000000p-1, 0x1.d2414cffb4308p-2},
    {0x1.734f0c0000000p-1, 0x1.daa6236f1986fp-2}, {0x1.7137860000000p-1, 0x1.e2fed737fa71bp-2},
    {0x1.6f26020000000p-1, 0x1.eb4b82363c72ap-2}, {0x1.6d1a620000000p-1, 0x1.f38c582110ab4p-2},
    {0x1.6b14900000000p-1, 0x1.fbc16e44a4df2p-2}, {0x1.6914740000000p-1, 0x1.01f571c44164cp-1},
    {0x1.6719f40000000p-1, 0x1.0604705635b21p-1}, {0x1.6524f80000000p-1, 0x1.0a0dc3fcadb74p-1},
    {0x1.63356c0000000p-1, 0x1.0e11765cb301cp-1}, {0x1.614b360000000p-1, 0x1.120f9e4bfe307p-1},
    {0x1.5f66440000000p-1, 0x1.160842bb2ef14p-1}, {0x1.5d867c0000000p-1, 0x1.19fb7c13ec9cbp-1},
    {0x1.5babcc0000000p-1, 0x1.1de952af508efp-1}, {0x1.59d6200000000p-1, 0x1.21d1d3bf9937ap-1},
    {0x1.5805600000000p-1, 0x1.25b515b99e5f1p-1}, {0x1.56397c0000000p-1, 0x1.29931ea921c92p-1},
    {0x1.54725e0000000p-1, 0x1.2d6c021eb8ab1p-1}, {0x1.52aff60000000p-1, 0x1.313fc75ba6defp-1},
    {0x1.50f22e0000000p-1, 0x1.350e834af3119p-1}, {0x1.4f38f60000000p-1, 0x1.38d83e67f2e8fp-1},
    {0x1.4d843c0000000p-1, 0x1.3c9d0620a5a43p-1}, {0x1.4bd3ee0000000p-1, 0x1.405ce87fe228fp-1},
    {0x1.4a27fa0000000p-1, 0x1.4417f42e5e494p-1}, {0x1.4880520000000p-1, 0x1.47ce2f7524d79p-1},
    {0x1.46dce40000000p-1, 0x1.4b7faa190522ep-1}, {0x1.453d9e0000000p-1, 0x1.4f2c747f9c4c5p-1},
    {0x1.43a2740000000p-1, 0x1.52d491fe838e1p-1}, {0x1.420b520000000p-1, 0x1.567818a22275dp-1},
    {0x1.40782e0000000p-1, 0x1.5a170824dcce0p-1}, {0x1.3ee8f40000000p-1, 0x1.5db177b29e834p-1},
    {0x1.3d5d9a0000000p-1, 0x1.614767ed4efe4p-1}, {0x1.3bd60e0000000p-1, 0x1.64d8ec764d04ep-1},
    {0x1.3a52440000000p-1, 0x1.68660b7c324e1p-1}, {0x1.38d22e0000000p-1, 0x1.6beed048f5fafp-1},
    {0x1.3755be0000000p-1, 0x1.6f7346a0cafd6p-1}, {0x1.35dce60000000p-1, 0x1.72f37ac2df0e6p-1},
    {0x1.34679a0000000p-1, 0x1.766f749fcab59p-1}, {0x1.32f5ce0000000p-1, 0x1.79e73c8d7c803p-1},
    {0x1.3187760000000p-1, 0x1.7d5adb47eadaap-1}, {0x1.301c820000000p-1, 0x1.80ca63a8f68e1p-1},
    {0x1.2eb4ea0000000p-1, 0x1.8435d59a8b483p-1}, {0x1.2d50a00000000p-1, 0x1.879d3ff5de45dp-1},
    {0x1.2bef980000000p-1, 0x1.8b00ad26f6a09p-1}, {0x1.2a91ca0000000p-1, 0x1.8e601e1dc1494p-1},
    {0x1.2937260000000p-1, 0x1.91bba7e7b4821p-1}, {0x1.27dfa40000000p-1, 0x1.95134c31fee02p-1},
    {0x1.268b380000000p-1, 0x1.986716eeae7a4p-1}, {0x1.2539d80000000p-1, 0x1.9bb70f71a7b25p-1},
    {0x1.23eb7a0000000p-1, 0x1.9f033d63e21a3p-1}, {0x1.22a0120000000p-1, 0x1.a24badd94221ap-1},
    {0x1.2157980000000p-1, 0x1.a590641cbbf9fp-1}, {0x1.2012020000000p-1, 0x1.a8d168d9b1253p-1},
    {0x1.1ecf440000000p-1, 0x1.ac0eca394c359p-1}, {0x1.1d8f560000000p-1, 0x1.af488c7aab24dp-1},
    {0x1.1c52300000000p-1, 0x1.b27eb41dfa14fp-1}, {0x1.1b17c60000000p-1, 0x1.b5b15054cb48fp-1},
    {0x1.19e0120000000p-1, 0x1.b8e06107ba768p-1}, {0x1.18ab080000000p-1, 0x1.bc0bf6152db08p-1},
    {0x1.1778a20000000p-1, 0x1.bf340ff0d9a55p-1}, {0x1.1648d60000000p-1, 0x1.c258b9d8b8af5p-1},
    {0x1.151b9a0000000p-1, 0x1.c579ff6598542p-1}, {0x1.13f0e80000000p-1, 0x1.c897e1d664aeep-1},
    {0x1.12c8b80000000p-1, 0x1.cbb267f7d978ap-1}, {0x1.11a3020000000p-1, 0x1.cec998dba8709p-1},
    {0x1.107fbc0000000p-1, 0x1.d1dd8144bc735p-1}, {0x1.0f5ee00000000p-1, 0x1.d4ee236f8798ep-1},
    {0x1.0e40660000000p-1, 0x1.d7fb873eebbc6p-1}, {0x1.0d24460000000p-1, 0x1.db05b4dc43651p-1},
    {0x1.0c0a780000000p-1, 0x1.de0cb4b7bd86fp-1}, {0x1.0af2f80000000p-1, 0x1.e110847743666p-1},
    {0x1.09ddba0000000p-1, 0x1.e4113814174b4p-1}, {0x1.08cabc0000000p-1, 0x1.e70ec8182b847p-1},
    {0x1.07b9f20000000p-1, 0x1.ea0949129567bp-1}, {0x1.06ab5a0000000p-1, 0x1.ed00b3ea0c777p-1},
    {0x1.059eea0000000p-1, 0x1.eff5181f2fdcbp-1}, {0x1.04949c0000000p-1, 0x1.f2e67a3c24e4cp-1},
    {0x1.038c6c0000000p-1, 0x1.f5d4d94c4f007p-1}, {0x1.0286500000000p-1, 0x1.f8c0459b53d2dp-1},
    {0x1.0182440000000p-1, 0x1.fba8be9ffab02p-1}, {0x1.0080400000000p-1, 0x1.fe8e4f721237ap-1},
};

__device__ __forceinline__ double log2_table(double x, const LogEntry* __restrict__ tab) {
  const int hi = __double2hiint(x);
  const LogEntry en = tab[(hi >> 13) & 127];
  const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(x));
  // the exponent as a double: 2^52 + (e + 1023) has it in its low bits
  const double e = __hiloint2double(0x43300000, (hi >> 20) & 0x7ff) - (4503599627370496.0 + 1023.0);
  const double r = fma(m, en.inv, -1.0);
  double p = 0.20609929155555663;   // 1 / (7 ln 2)
  p = fma(p, r, -0.24044917348149390);
  p = fma(p, r, 0.28853900817779268);
  p = fma(p, r, -0.36067376022224085);
  p = fma(p, r, 0.48089834696298783);
  p = fma(p, r, -0.72134752044448170);
  p = fma(p, r, 1.4426950408889634);  // 1 / ln 2
  return fma(p, r, en.t + e);
}

// 1e-36 < v < 1e36, as the bits of positive doubles order them (false for NaN, zero, negative)
__device__ __forceinline__ bool in_range(double v) {
  const long long b = __double_as_longlong(v);
  return b > __double_as_longlong(1.0 / 1.0e36) && b < __double_as_longlong(1.0e36);
}

// one field of a packed-pair entry (layout: store_pair_entry)
__device__ __forceinline__ void store_pair_field(float4* __restrict__ a, int64_t e, int field, float v) {
  reinterpret_cast<float*>(a + (e >> 1) * 2)[2 * field + (int)(e & 1)] = v;
}

// RF: row finalize of iteration t.  The warps of stream A give q^A; those of stream B q^B and the row shifts of iteration t + 1, where stream A has
// kappa_{t+1} (stream B here) and stream B is extrapolated linearly in t.  Block `rowblocks`
// prepares make_sweep_params of kappa_{t+2} for CF.  Evaluation passes have stream A alone, and
// the second warps form log Z.
template <bool EVAL>
__global__ void __launch_bounds__(kThreads)
k_row_fin(const Work w, int splits, const double* __restrict__ r, int rowblocks, const Consts k) {
  DevState* __restrict__ dev = w.dev;
  if (dev->done) return;
  if (!EVAL && (int)blockIdx.x == rowblocks) {
    if (threadIdx.x == 0) {
      SweepParams sp, spn;
      iteration_params_of(dev, k, sp, spn);
      dev->spq = make_sweep_params(spn.kapB, k);
    }
    return;
  }
  __shared__ LogEntry stab[128];
  __shared__ double sx[kPts];  // log2 Z of stream A, for the warps of stream B
  __shared__ double sred[kWarps];
  const int role = threadIdx.x >= kPts ? 1 : 0;  // warp-uniform
  const int p = threadIdx.x - role * kPts;
  const int64_t i = (int64_t)blockIdx.x * kPts + p;
  if (threadIdx.x < 128) stab[threadIdx.x] = kLogTab[threadIdx.x];
  const int cur = dev->cur;
  const bool valid = i < k.n;
  double S = 0.0, ri = 0.0, snx = 0.0;
  float2 rq = make_float2(0.f, 0.f);
  SweepParams sp, spn;
  iteration_params_of(dev, k, sp, spn);
  if (valid) {
    rq = w.rowshift[cur][i];
    ri = r[i];
    if (k.zdot && (EVAL || !k.shared_shift)) snx = k.s * w.nx[i];
    // the partials' loads are independent and in flight together; the sums keep the split order
    // (evaluation passes sweep stream A alone: one sum per split, read by both warps)
    constexpr int na = EVAL ? 1 : 2;
    const double* __restrict__ part = w.rowpart + (int64_t)(EVAL ? 0 : role) * k.n + i;
#pragma unroll 8
    for (int s = 0; s < splits; ++s) S += part[(int64_t)s * na * k.n];
    if (!in_range(S)) {
      atomicExch(&dev->status, 5 /* LAMP_E_NUMERIC */);
      S = 1.0;
    }
  }
  __syncthreads();
  double contrib = 0.0, ls = 0.0;
  if (valid) {
    // float64 log2 and divisions: with float32 ones (log2f carries an absolute error of
    // ~2^-22 near 1) the potentials of 100-iteration trajectories drifted from the oracle's
    // by ~1e-6 instead of ~1e-8, and log Z, which amplifies nu by 2 K kappa, by ~1e-4
    if (role == 0) {
      // the row weight q = r / S, a float32 factor of the column sweep
      const float q = (float)div_seeded(ri, S);
      reinterpret_cast<float2*>(w.g2row + i)[0] = make_float2(rq.x, q);
      if (w.g2row2) {
        store_pair_field(w.g2row2, i, 0, -rq.x);
        store_pair_field(w.g2row2, i, 1, q);
      }
      if (!EVAL && !k.shared_shift) {
        sx[p] = (double)rq.x - sp.lamA * snx + log2_table(S, stab);
      }
    } else if (EVAL) {
      const double lz = kLn2 * ((double)rq.x - sp.lamA * snx + log2(S));  // log Z of X^t
      w.logZ[i] = lz;
      contrib = ri * lz;
    } else {
      const float q = (float)div_seeded(ri, S);
      reinterpret_cast<float2*>(w.g2row + i)[1] = make_float2(rq.y, q);
      if (w.g2row2) {
        store_pair_field(w.g2row2, i, 2, k.shared_shift ? 0.f : -rq.y);
        store_pair_field(w.g2row2, i, 3, q);
      }
      ls = log2_table(S, stab);
    }
  }
  if (EVAL) {
    if (role == 1) {
      contrib = warp_sum_d(contrib);
      if ((threadIdx.x & 31) == 0) sred[p >> 5] = contrib;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double v = 0.0;
      for (int q = 0; q < kWarps; ++q) v += sred[q];
      w.rowred[blockIdx.x] = v;
    }
    return;
  }
  if (!k.shared_shift) __syncthreads();
  if (role == 1 && valid) {
    const float qA = (float)quantize_add((double)rq.y + ls, spn.g);
    float qB = qA;
    if (!k.shared_shift) {
      const double L2B = (double)rq.y - sp.lamB * snx + ls;  // log2 Z of Xbar^{t+1}
      qB = (float)quantize_add(spn.lamB * snx + 2.0 * L2B - sx[p], spn.g);
    }
    w.rowshift[cur ^ 1][i] = make_float2(qA, qB);
  }
}

// CF: column finalize of iteration t, dual step of Alg. 2, and the decision.  The warps of
// stream A take col(X^t): residual, nu^{t+1} and its column data; those of stream B take
// col(Xbar^{t+1}): theta^{t+1}, and nubar^{t+2} with its column data, from the nu^{t+1} that
// stream A's warps hand over.  Evaluation passes update nothing: the first warps take col(X^t)
// and <col, nu>, the second ones the cost.
template <bool EVAL>
__global__ void __launch_bounds__(kThreads)
k_col_fin(const Work w, int splits, const double* __restrict__ cvec, int rowblocks, const Consts k) {
  DevState* __restrict__ dev = w.dev;
  if (dev->done) return;
  const int cur = dev->cur;
  __shared__ double snu[kPts], sq[kPts];
  __shared__ double sred[4][kThreads / 32];
  __shared__ bool amLast;
  const int role = threadIdx.x >= kPts ? 1 : 0;  // warp-uniform
  const int p = threadIdx.x - role * kPts;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t j = (int64_t)blockIdx.x * kPts + p;
  const bool valid = j < k.m;
  double res = 0.0, cost = 0.0, cnu = 0.0, zsum = 0.0;
  double nun = 0.0, thn = 0.0, sny = 0.0;
  SweepParams sp, spn;
  iteration_params_of(dev, k, sp, spn);
  if (valid) {
    // partials of split s: [s][2][m], the streams' sums; evaluation passes: stream A's sums and
    // the cost-weighted ones, which the second warps take
    constexpr int na = 2;
    const float4 cq = w.colq[cur][j];
    const double cj = cvec[j];
    const double nuj = w.nu[cur][j], thj = EVAL ? 0.0 : w.theta[cur][j];
    const double gj = EVAL ? 0.0 : w.gj[j];
    const double* __restrict__ part = w.colpart + (int64_t)role * k.m + j;
    if (k.zdot) sny = k.s * w.ny[j];
    double a = 0.0;
    // the partials' loads are independent and in flight together; the sums keep the split order
#pragma unroll 8
    for (int s = 0; s < splits; ++s) a += part[(int64_t)s * na * k.m];
    if (EVAL && role) zsum = (double)cq.y * a;
    if (role == 0) {
      const double A = (double)cq.y * a;  // col(X^t)_j
      w.colA[j] = A;
      res = fabs(A - cj);
      if (EVAL) {
        cnu = A * nuj;
        snu[p] = A;
      } else {
        // the dual mirror steps (Eq. def:closed_form_opt) tanh(g (col - c) + atanh theta), in
        // float64 through the addition theorem tanh(u + atanh theta) = (tanh u + theta) /
        // (1 + theta tanh u): one tanh per stream and no atanh (|theta^t| <= tanh(beta/2) < 1,
        // so the denominator is at least 1 - tanh(beta/2))
        const double tA = tanh(gj * (A - cj));
        const double thbar = div_seeded(tA + thj, fma(tA, thj, 1.0));  // M_{tau2}(theta^t; p^{eta_t}(nu^t))
        nun = nuj + sp.wB * (thbar - nuj);                             // nu^{t+1}
        snu[p] = nun;
        w.nu[cur ^ 1][j] = nun;
      }
    } else if (!EVAL) {
      // col(Xbar^{t+1})_j; under the shared row shift the column weight of stream B is
      // already inside the sweep's exponents
      const double B = k.shared_shift ? a : (double)cq.w * a;
      const double tB = tanh(gj * (B - cj));
      const double thhat = div_seeded(tB + thj, fma(tB, thj, 1.0));  // M_{tau2}(theta^t; p^{eta_{t+1}}(nubar^{t+1}))
      thn = fmin(fmax(thhat, -k.clipb), k.clipb);                    // tclip
      w.theta[cur ^ 1][j] = thn;
    }
  }
  float qBf = 0.f, wBf = 0.f;
  double bB = 0.0;
  if (!EVAL) {
    __syncthreads();
    // column data of iteration t + 1: Bcol of each stream rounded to the grid, the factor
    // 2^{-remainder}, and stream B's term dB = BqA - BcolB (column_data of the header)
    if (valid && role == 0) {
      const double bA = spn.lamA * (sny + 2.0 * k.K * nun);
      const double qA = quantize_add(bA, spn.g);
      sq[p] = qA;
      const float qf = (float)qA, wf = exp2f((float)(qA - bA));
      reinterpret_cast<float2*>(w.colq[cur ^ 1] + j)[0] = make_float2(qf, wf);
      if (w.colq2[cur ^ 1]) {
        store_pair_field(w.colq2[cur ^ 1], j, 0, -qf);
        store_pair_field(w.colq2[cur ^ 1], j, 1, wf);
      }
    } else if (valid) {
      const double nu1 = snu[p];
      const double nbn = nu1 + spn.wB * (thn - nu1);  // nubar^{t+2}
      bB = spn.lamB * (sny + 2.0 * k.K * nbn);
      const double qB = quantize_add(bB, spn.g);
      qBf = (float)qB;
      wBf = exp2f((float)(qB - bB));
      reinterpret_cast<float2*>(w.colq[cur ^ 1] + j)[1] = make_float2(qBf, wBf);
    }
  }
  if (EVAL) {
    __syncthreads();
    if (role == 1 && valid) {
      // dot form: + sum_i r_i s|x_i|^2, added once below
      cost = k.zdot ? k.s * w.ny[j] * snu[p] - 2.0 * k.s * zsum : k.s * zsum;
      if (w.colz) w.colz[j] = cost;
    }
  }
  if (role == 0) {
    res = warp_sum_d(res);
    if (EVAL) cnu = warp_sum_d(cnu);
    if (lane == 0) {
      sred[0][wid] = res;
      if (EVAL) sred[2][wid] = cnu;
    }
  } else if (EVAL) {
    cost = warp_sum_d(cost);
    if (lane == 0) sred[1][wid - kWarps] = cost;
  }
  __syncthreads();
  // block partials: {res, cost, <col, nu>} per block in evaluation passes, else res alone
  constexpr int nf = EVAL ? 3 : 1;
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < nf; ++q) {
      double v = 0.0;
      for (int u = 0; u < kWarps; ++u) v += sred[q][u];
      w.colred[(int64_t)nf * blockIdx.x + q] = v;
    }
    __threadfence();
    const unsigned int tk = atomicAdd(&dev->ticket, 1u);
    amLast = (tk == gridDim.x - 1);
  }
  if (!EVAL && valid && role == 1 && w.colq2[cur ^ 1]) {
    store_pair_field(w.colq2[cur ^ 1], j, 2, (float)(sq[p] - bB));
    store_pair_field(w.colq2[cur ^ 1], j, 3, wBf);
  }
  __syncthreads();
  if (!amLast) return;
  // last block: reduce all partials in a fixed order (thread t takes blocks t, t + threads, ..,
  // then a fixed tree over the threads) and decide
  __threadfence();
  double R = 0.0, Cx = 0.0, Cn = 0.0, RL = 0.0;
  for (unsigned int b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
    R += ((volatile double*)w.colred)[(int64_t)nf * b + 0];
    if (EVAL) {
      Cx += ((volatile double*)w.colred)[(int64_t)nf * b + 1];
      Cn += ((volatile double*)w.colred)[(int64_t)nf * b + 2];
    }
  }
  if (EVAL)
    for (int b = threadIdx.x; b < rowblocks; b += blockDim.x) RL += ((volatile const double*)w.rowred)[b];
  R = warp_sum_d(R);
  if (EVAL) {
    Cx = warp_sum_d(Cx);
    Cn = warp_sum_d(Cn);
    RL = warp_sum_d(RL);
  }
  if (lane == 0) { sred[0][wid] = R; sred[1][wid] = Cx; sred[2][wid] = Cn; sred[3][wid] = RL; }
  __syncthreads();
  if (threadIdx.x == 0) {
    R = Cx = Cn = RL = 0.0;
    for (int q = 0; q < kThreads / 32; ++q) {
      R += sred[0][q];
      if (EVAL) {
        Cx += sred[1][q];
        Cn += sred[2][q];
        RL += sred[3][q];
      }
    }
    dev->ticket = 0u;
    dev->res = R;
    // what only evaluation passes compute
    dev->costA = EVAL ? Cx + k.rnx : NAN;
    dev->colnu = EVAL ? Cn : NAN;
    dev->rlogZ = EVAL ? RL : NAN;
    if (EVAL) {
      dev->t_eval = dev->t;
      dev->kappa_eval = dev->kappa;
    }
    if (dev->status != 0 || !isfinite(R)) {
      if (dev->status == 0) dev->status = 5;
      dev->done = 1;
    } else if (EVAL) {
      dev->done = 1;
    } else if ((dev->t >= 1 && R <= dev->tol &&
                (k.eta == 0.0 || k.infeas_only || 1.0 - dev->kappa * k.eta <= dev->tol)) ||
               dev->t >= dev->tmax) {
      dev->done = 1;
    } else {
      dev->t = dev->t + 1;
      dev->kappa = sp.kapB;
      dev->cur ^= 1;
      // the next iteration's parameters, once per iteration instead of once per thread
      // (make_sweep_params of kappa_{t+2} comes from RF)
      dev->spc = spn;
      dev->spn = dev->spq;
      dev->swf = sweep_floats(spn);
      dev->swf_kap = spn.kapA;
    }
    __threadfence();
  }
}

// the gain of the mirror step 2 tau2 K / c^alpha_j, c^alpha = c + alpha/m (Section 3.1)
__global__ void k_mirror_gain(const double* __restrict__ c, double* __restrict__ gj, const Consts k) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < k.m) gj[j] = 2.0 * k.tau2 * k.K / (c[j] + k.alpha_m);
}

inline unsigned blocks_of(int64_t len, int pts) { return (unsigned)((len + pts - 1) / pts); }

}  // namespace

cudaError_t launch_mirror_gain(const Inputs& in, const Consts& k, const Work& w, cudaStream_t st) {
  k_mirror_gain<<<blocks_of(k.m, 256), 256, 0, st>>>(in.c, w.gj, k);
  return cudaGetLastError();
}

cudaError_t launch_row_fin(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int eval,
                           cudaStream_t st) {
  const unsigned nb = blocks_of(k.n, kPts);
  if (eval) return launch_kernel(k_row_fin<true>, nb, kThreads, 0, st, w, g.rows_split, in.r, (int)nb, k);
  return launch_kernel(k_row_fin<false>, nb + 1, kThreads, 0, st, w, g.rows_split, in.r, (int)nb, k);
}

cudaError_t launch_col_fin(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int eval,
                           cudaStream_t st) {
  return launch_kernel(eval ? k_col_fin<true> : k_col_fin<false>, blocks_of(k.m, kPts), kThreads, 0, st, w, g.cols_split,
                    in.c, (int)blocks_of(k.n, kPts), k);
}

}  // namespace lamp
