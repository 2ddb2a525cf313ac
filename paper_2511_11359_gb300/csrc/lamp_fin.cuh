// Float64 pieces of the finalize step, shared by the finalize kernels (lamp_fin.cu) and the
// whole-iteration kernel of small problems (lamp_cluster.cu).
#pragma once

#include <cmath>

#include "lamp_common.cuh"

namespace lamp {

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
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
static __device__ const LogEntry kLogTab[128] = {
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

template <int G>
__device__ __forceinline__ void add_group(double& a, const double* __restrict__ p, int64_t stride) {
  double v[G];
#pragma unroll
  for (int u = 0; u < G; ++u) v[u] = p[u * stride];
#pragma unroll
  for (int u = 0; u < G; ++u) a += v[u];
}

// 0 + p[0] + p[stride] + ... in split order.  The adds are one dependent chain of float64 (64 cycles
// each) and the loads of a group of 8 take as long as its adds, so the next group is loaded while
// one is added: column finalize of 3001 x 2777 (41 splits) 18.4 -> 14.3 us between events, 50
// iterations there 2.25 -> 2.08 ms, on 4096 x 4096 2.15 -> 2.11.  No guarded adds: one that is
// predicated off takes its 64 cycles too.
__device__ __forceinline__ double split_sum(const double* __restrict__ p, int64_t stride, int splits) {
  double a = 0.0;
  int s = 0;
  if (splits >= 8) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = p[u * stride];
    for (s = 8; s + 8 <= splits; s += 8) {
      double x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = p[(s + u) * stride];
#pragma unroll
      for (int u = 0; u < 8; ++u) a += v[u];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = x[u];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) a += v[u];
  }
  if (splits & 4) {
    add_group<4>(a, p + s * stride, stride);
    s += 4;
  }
  if (splits & 2) {
    add_group<2>(a, p + s * stride, stride);
    s += 2;
  }
  if (splits & 1) a += p[s * stride];
  return a;
}

// one field of a packed-pair entry (layout: store_pair_entry)
__device__ __forceinline__ void store_pair_field(float4* __restrict__ a, int64_t e, int field, float v) {
  reinterpret_cast<float*>(a + (e >> 1) * 2)[2 * field + (int)(e & 1)] = v;
}

}  // namespace lamp
