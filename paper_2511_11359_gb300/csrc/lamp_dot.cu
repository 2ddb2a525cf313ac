// Float32 dot-form sweeps (|x - y|^2 and cosine with d > 8, LAMP_PREC_FP32): z = x.y on the FMA
// pipe, the row sweep G1, the column sweep G2, the row-max passes and the envelope gradient.
//
// What bounds them: 2 d of the ~2 d + 16 float operations of an entry are the contraction, so
// the FMA pipe (128 lanes per clock and SM), and next to it shared memory, which hands the warps
// 128 bytes per clock: a thread that computes an 8 x 8 block reads 64 bytes for 64 FMA, and both
// are saturated at the same time.  So here a thread owns 8 outer x 16 inner points (96 bytes for
// 128 FMA), accumulates pairs of inner points with f32x2 (half the issue slots), and reads
// points that a transposed copy (one row per coordinate) lets it stage with 16-byte asynchronous
// copies, one stage ahead of the arithmetic.  One CTA of 256 threads per SM (the 8 x 16 block
// takes 128 of its 255 registers), persistent over (outer tile, inner split) items, so that an
// item's first stage is copied while the previous item finishes.  n = m = 8192, d = 64: 0.230 ms
// per sweep (8 x 8 blocks staged through registers: 0.32 ms); the FMAs alone are 0.107 ms at the
// pipe's rate, and f32x2 FMAs with three distinct register operands and their shared-memory
// loads, alone, ran at 72 % of it.  Scalar FMAs: 0.27 ms.
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "lamp_common.cuh"

namespace lamp {

namespace dot {

constexpr int kOut = 128;     // outer points of an item
constexpr int kIn = 128;      // inner points of a tile: the unit of the splits and of the float32 sums
constexpr int kStage = 256;   // inner points of a stage (two tiles)
constexpr int kThreads = 256;
constexpr int kGradFold = 8;  // float32 terms of the gradient's and the map's sums between folds

// kRowEval, kColEval: evaluation passes (stream A alone; columns also weighted by the cost)
enum Mode : int { kRowSum = 0, kColSum = 1, kRowEval = 2, kColEval = 3, kMax = 4, kMax2 = 5, kKmax = 6 };

__device__ __forceinline__ void cp16(void* dst, const void* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp8(void* dst, const void* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// the operands of one launch: transposed copies (d rows of ld floats, zero-padded to whole
// stages), the outer points' offsets and the inner points' data of both state buffers
struct Args {
  const float* out_t;
  const float* in_t;
  int64_t ld_out, ld_in;
  int64_t n_out, n_in;
  int d;
  int splits, tiles_per_split, ntiles, out_tiles;
  const float2* off2[2];  // row sweeps and row-max passes: row shifts
  const float4* off4[2];  // column sweeps: column data
  const float4* dat[2];   // inner data {offset A, weight A, offset B, weight B}, padded with {inf, 0, inf, 0}
  double* part;
  float* pmax;
};

struct Item {
  int64_t o;     // outer tile
  int split;
  int it0, it1;  // inner tiles
  int steps;     // stages (0: an empty split)
};

__device__ __forceinline__ Item item_of(int64_t idx, const Args& a) {
  Item t;
  t.split = (int)(idx / a.out_tiles);
  t.o = idx - (int64_t)t.split * a.out_tiles;
  t.it0 = t.split * a.tiles_per_split;
  t.it1 = t.it0 + a.tiles_per_split < a.ntiles ? t.it0 + a.tiles_per_split : a.ntiles;
  t.steps = t.it1 > t.it0 ? (t.it1 - t.it0 + 1) / 2 : 0;
  return t;
}

// shared memory: outer points and offsets of two items, inner points and data of two stages
__host__ __device__ constexpr size_t smem_floats(int d) {
  return 2 * ((size_t)d * kOut + 4 * kOut) + 2 * ((size_t)d * kStage + 4 * kStage);
}

template <int MODE>
__device__ __forceinline__ void load_outer(float* so, float4* soff, const Args& a, const Item& t, int cur, int tid) {
  const float* src = a.out_t + t.o * kOut;
  for (int c = tid; c < a.d * (kOut / 4); c += kThreads) {
    const int kk = c / (kOut / 4), q = c % (kOut / 4);
    cp16(so + kk * kOut + 4 * q, src + (int64_t)kk * a.ld_out + 4 * q);
  }
  if (MODE != kMax && tid < kOut) {
    int64_t go = t.o * kOut + tid;
    if (go >= a.n_out) go = a.n_out - 1;
    if (MODE == kColSum || MODE == kColEval)
      cp16(soff + tid, (cur ? a.off4[1] : a.off4[0]) + go);
    else
      cp8(soff + tid, (cur ? a.off2[1] : a.off2[0]) + go);
  }
}

__device__ __forceinline__ void load_stage(float* si, float4* sd, const Args& a, const Item& t, int step, int cur,
                                           int tid) {
  const int64_t p0 = (int64_t)(t.it0 + 2 * step) * kIn;
  const int np = t.it0 + 2 * step + 1 < t.it1 ? kStage : kIn;
  const float* src = a.in_t + p0;
  for (int c = tid; c < a.d * (kStage / 4); c += kThreads) {
    const int kk = c / (kStage / 4), q = c % (kStage / 4);
    if (4 * q < np) cp16(si + kk * kStage + 4 * q, src + (int64_t)kk * a.ld_in + 4 * q);
  }
  if (tid < np) cp16(sd + tid, (cur ? a.dat[1] : a.dat[0]) + p0 + tid);
}

template <int MODE>
struct Acc {
  static constexpr bool kSums = MODE <= kColEval;
  static constexpr int N = MODE == kRowEval ? 1 : 2;
  float hi[8][N], lo[8][N];  // kSums: float-float sums; else hi = the running maxima
  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int q = 0; q < N; ++q) {
        hi[r][q] = kSums ? 0.f : -INFINITY;
        lo[r][q] = 0.f;
      }
  }
};

// NU tiles of a stage: the contraction in coordinate order, then the exponents and sums of one
// tile after the other.  Thread (tx, ty): outer points 4 ty + {0..3}, 64 + 4 ty + {0..3}, inner
// points 4 tx + {0..3}, 64 + 4 tx + {0..3} of each tile; a tile's eight terms are added in that
// order from zero and folded into the float-float pair.
template <int MODE, int NU>
__device__ __forceinline__ void tile_sums(const float* __restrict__ so, const float4* __restrict__ soff,
                                          const float* __restrict__ si, const float4* __restrict__ sd, int d, int tx,
                                          int ty, const SweepF& sp, int64_t left, Acc<MODE>& acc) {
  uint64_t z2[8][4 * NU];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int p = 0; p < 4 * NU; ++p) z2[r][p] = 0ull;
  // fragments of two coordinates: the loads of the next one are in flight during the current FMAs
  float4 fa[2][2];
  ulonglong2 fb[2][2 * NU];
  auto ld = [&](int kk, int q) {
    fa[q][0] = *reinterpret_cast<const float4*>(so + kk * kOut + ty * 4);
    fa[q][1] = *reinterpret_cast<const float4*>(so + kk * kOut + 64 + ty * 4);
#pragma unroll
    for (int h = 0; h < 2 * NU; ++h) fb[q][h] = *reinterpret_cast<const ulonglong2*>(si + kk * kStage + h * 64 + tx * 4);
  };
  auto mm = [&](int q) {
    const float av[8] = {fa[q][0].x, fa[q][0].y, fa[q][0].z, fa[q][0].w, fa[q][1].x, fa[q][1].y, fa[q][1].z, fa[q][1].w};
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const uint64_t aa = pk(av[r], av[r]);
#pragma unroll
      for (int h = 0; h < 2 * NU; ++h) {
        z2[r][2 * h] = f2fma(aa, fb[q][h].x, z2[r][2 * h]);
        z2[r][2 * h + 1] = f2fma(aa, fb[q][h].y, z2[r][2 * h + 1]);
      }
    }
  };
  ld(0, 0);
  int kk = 0;
  for (; kk + 2 <= d; kk += 2) {
    ld(kk + 1, 1);
    mm(0);
    ld(kk + 2 < d ? kk + 2 : kk, 0);
    mm(1);
  }
  if (kk < d) mm(0);
  const uint64_t ahA2 = pk(sp.ahA, sp.ahA), alA2 = pk(sp.alA, sp.alA);
  const uint64_t ahB2 = pk(sp.ahB, sp.ahB), alB2 = pk(sp.alB, sp.alB);
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    float4 dat[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) dat[b] = sd[u * kIn + ((b < 4) ? (tx * 4 + b) : (64 + tx * 4 + b - 4))];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int ro = (r < 4) ? (ty * 4 + r) : (64 + ty * 4 + r - 4);
      float oA = 0.f, oB = 0.f;
      if (MODE == kColSum || MODE == kColEval) {
        const float4 o = soff[ro];
        oA = o.x;
        oB = o.z;
      } else if (MODE != kMax) {
        const float2 o = *reinterpret_cast<const float2*>(soff + ro);
        oA = o.x;
        oB = o.y;
      }
      if constexpr (Acc<MODE>::kSums) {
        const uint64_t oA2 = pk(-oA, -oA), oB2 = pk(-oB, -oB);
        float sA = 0.f, sB = 0.f;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const uint64_t z = z2[r][4 * u + p];
          const float4 d0 = dat[2 * p], d1 = dat[2 * p + 1];
          const float2 eA = upk(exp2_pair(ahA2, alA2, z, f2sub(oA2, pk(d0.x, d1.x))));
          if (MODE == kRowSum || MODE == kRowEval) {
            sA = __fmaf_rn(eA.y, d1.y, __fmaf_rn(eA.x, d0.y, sA));
          } else {
            const float p0 = __fmul_rn(eA.x, d0.y), p1 = __fmul_rn(eA.y, d1.y);
            sA = __fadd_rn(__fadd_rn(sA, p0), p1);
            if (MODE == kColEval) {
              const float2 zf = upk(z);
              sB = __fmaf_rn(zf.y, p1, __fmaf_rn(zf.x, p0, sB));
            }
          }
          if (MODE == kRowSum || MODE == kColSum) {
            const float2 eB = upk(exp2_pair(ahB2, alB2, z, f2sub(oB2, pk(d0.z, d1.z))));
            sB = __fmaf_rn(eB.y, d1.w, __fmaf_rn(eB.x, d0.w, sB));
          }
        }
        ff_add(acc.hi[r][0], acc.lo[r][0], sA);
        if (Acc<MODE>::N > 1) ff_add(acc.hi[r][Acc<MODE>::N - 1], acc.lo[r][Acc<MODE>::N - 1], sB);
      } else {
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const float2 zf = upk(z2[r][4 * u + p]);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float zz = h ? zf.y : zf.x;
            const float4 dd = dat[2 * p + h];
            if (MODE == kMax) {
              acc.hi[r][0] = fmaxf(acc.hi[r][0], __fmaf_rn(sp.ahA, zz, -dd.x));
              acc.hi[r][1] = fmaxf(acc.hi[r][1], __fmaf_rn(sp.ahB, zz, -dd.z));
            } else if (MODE == kMax2) {
              // u = a z - (Rq + Bq) - Br (the eta = 0 dual bound's second pass, see launch_dual)
              const float v = __fmaf_rn(sp.alA, zz, __fmaf_rn(sp.ahA, zz, -(oA + dd.x))) - dd.y;
              acc.hi[r][0] = fmaxf(acc.hi[r][0], v);
            } else {
              // |x|^2 + |y|^2 - 2 x.y and its negative; oA = |x|^2, dd.x = |y|^2
              const int b = 2 * p + h;
              const bool pad = u * kIn + ((b < 4) ? (tx * 4 + b) : (64 + tx * 4 + b - 4)) >= left;
              const float D = __fmaf_rn(-2.0f, zz, oA + dd.x);
              acc.hi[r][0] = fmaxf(acc.hi[r][0], pad ? -INFINITY : D);
              acc.hi[r][1] = fmaxf(acc.hi[r][1], pad ? -INFINITY : -D);
            }
          }
        }
      }
    }
  }
}

// sums over the 16 lanes of a half-warp of 16 values per lane, as the butterfly xor 8, 4, 2, 1
// adds them; each level halves the values a lane carries (the two operands of an addition
// commute, so the sums are those of the full butterfly), 15 additions instead of 64; value q
// ends in lane tx = q.
__device__ __forceinline__ double halfwarp_sum16(double (&v)[16], int tx) {
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const int o = 8 >> l;
    const bool up = (tx & o) != 0;
    const int half = 8 >> l;
#pragma unroll
    for (int q = 0; q < half; ++q) {
      const double keep = up ? v[half + q] : v[q];
      const double give = up ? v[q] : v[half + q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  return v[0];
}

template <int MODE>
__device__ __forceinline__ void write_item(const Args& a, const Item& t, Acc<MODE>& acc, int tx, int ty) {
  constexpr int NACC = Acc<MODE>::N;
  if constexpr (Acc<MODE>::kSums) {
    // value 8 q + r: sum q of outer point r (evaluation row sums have q = 0 alone)
    double v[16];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int q = 0; q < 2; ++q) v[8 * q + r] = q < NACC ? (double)acc.hi[r][q % NACC] + (double)acc.lo[r][q % NACC] : 0.0;
    const double s = halfwarp_sum16(v, tx);
    const int r = tx & 7, q = tx >> 3;
    const int64_t go = t.o * kOut + ((r < 4) ? (ty * 4 + r) : (64 + ty * 4 + r - 4));
    if (go < a.n_out && q < NACC) a.part[((int64_t)t.split * NACC + q) * a.n_out + go] = s;
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int64_t go = t.o * kOut + ((r < 4) ? (ty * 4 + r) : (64 + ty * 4 + r - 4));
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float m = acc.hi[r][q];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (tx == 0 && go < a.n_out) a.pmax[((int64_t)t.split * 2 + q) * a.n_out + go] = m;
      }
    }
  }
}

template <int MODE>
__global__ void __launch_bounds__(kThreads, 1)
k_dot_sweep(const Args a, const DevState* __restrict__ dev, const Consts k) {
  if (Acc<MODE>::kSums && dev->done) return;
  extern __shared__ __align__(16) float smem[];
  // outer points, inner points, outer offsets, inner data, two buffers each
  const int outf = a.d * kOut, inf = a.d * kStage;
  float* so = smem;
  float* si = smem + 2 * outf;
  float4* soff = reinterpret_cast<float4*>(si + 2 * inf);
  float4* sd = soff + 2 * kOut;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int cur = dev->cur;
  const SweepF sp = sweep_floats_of(dev, k);
  const int64_t items = (int64_t)a.out_tiles * a.splits;

  Acc<MODE> acc;
  // the stage that is copied next: (item ni, step ns), into stage buffer nb and, for a first
  // step, outer buffer no
  int64_t ni = blockIdx.x;
  int nb = 0, no = 0;
  Item nt{};
  for (; ni < items; ni += gridDim.x) {
    nt = item_of(ni, a);
    if (nt.steps) break;  // (an empty split has no stage)
  }
  if (ni < items) {
    load_outer<MODE>(so, soff, a, nt, cur, tid);
    load_stage(si, sd, a, nt, 0, cur, tid);
  }
  cp_commit();
  int cb = 0, co = 0;  // the buffers of the stage that is computed
  for (int64_t i = blockIdx.x; i < items; i += gridDim.x) {
    const Item t = item_of(i, a);
    acc.reset();
    for (int s = 0; s < t.steps; ++s) {
      cp_wait<0>();
      __syncthreads();  // the stage has landed, and every warp is done with the other buffers
      // copy what comes next: this item's next stage, or the next item's first
      nb = cb ^ 1;
      no = co;
      if (s + 1 < t.steps) {
        load_stage(si + nb * inf, sd + nb * kStage, a, t, s + 1, cur, tid);
      } else {
        no = co ^ 1;
        for (ni = i + gridDim.x; ni < items; ni += gridDim.x) {
          nt = item_of(ni, a);
          if (nt.steps) break;
        }
        if (ni < items) {
          load_outer<MODE>(so + no * outf, soff + no * kOut, a, nt, cur, tid);
          load_stage(si + nb * inf, sd + nb * kStage, a, nt, 0, cur, tid);
        }
      }
      cp_commit();
      const int64_t left = a.n_in - (int64_t)(t.it0 + 2 * s) * kIn;
      if (t.it0 + 2 * s + 1 < t.it1)
        tile_sums<MODE, 2>(so + co * outf, soff + co * kOut, si + cb * inf, sd + cb * kStage, a.d, tx, ty, sp, left,
                           acc);
      else
        tile_sums<MODE, 1>(so + co * outf, soff + co * kOut, si + cb * inf, sd + cb * kStage, a.d, tx, ty, sp, left,
                           acc);
      cb = nb;
      if (s + 1 == t.steps) co = no;
    }
    write_item<MODE>(a, t, acc, tx, ty);
  }
  cp_wait<0>();
}

// transposed copy: out[q][i] = P[i][q], zero beyond np (32 x 32 tiles through shared memory)
__global__ void __launch_bounds__(256)
k_transpose_points(const float* __restrict__ P, int64_t np, int d, float* __restrict__ out, int64_t ld) {
  __shared__ float t[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32;
  const int q0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int64_t i = i0 + r;
    const int q = q0 + threadIdx.x;
    t[r][threadIdx.x] = (i < np && q < d) ? P[i * d + q] : 0.f;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int q = q0 + r;
    if (q < d && i0 + threadIdx.x < ld) out[(int64_t)q * ld + i0 + threadIdx.x] = t[threadIdx.x][r];
  }
}

// ------------------------------------------------------------------------------------------
// Envelope gradient (and transport map), one side: O_a = sum_b P_ab p_b over the inner points'
// coordinates (or value columns) p_b, P_ab = 2^{v_ab} weight_b with stream A's exponent (X never
// stored).  Two contractions per tile of 128 x 128
// entries: z = x.y as in the sweeps (8 x 8 block per thread), P to shared memory, then O += P p
// with all coordinates at once: 0.61 ms a side at n = m = 8192, d = 64 (a pass per 8 coordinates
// computed every exponent and every product x.y d / 8 times, 8 x 0.67 ms a side).  In the second
// contraction the halves of the CTA take 64 inner points each and thread (og, cg) the outer
// points 4 og + {0..3}, 64 + 4 og + {0..3} and the CQ coordinates from CQ cg: 8 float32 terms
// per output, then a fold into a float-float pair (a fold per 64 terms: 0.49 ms a side, but chains
// of 64 additions were up to 12 u off, u = 2^-24, and the gradient is a difference of such sums; 8
// terms are within 4.5 u); the halves meet in float64.  P is stored
// with its 16-byte chunks permuted by the row (chunk ^ (row / 4) % 8), which keeps both the
// stores (one row per lane) and the loads (one row per warp) free of bank conflicts.

struct GradArgs {
  const float* out_t;   // transposed outer points (ld_out)
  const float* in_t;    // transposed inner points (ld_in)
  const float* in_v;    // dv values of each inner point, row-major (the gradient: the points)
  int64_t ld_out, ld_in, n_out, n_in;
  int d, dv;
  int tiles_per_split, ntiles;
  const float4* off;    // outer data: {offset A, ...}
  const float4* dat;    // inner data: {offset A, weight A, ...}, n_in entries
  double* part;         // [splits][n_out][dv]
};

template <int CQ>
constexpr size_t grad_smem_floats(int d) {
  return 2 * (size_t)d * kOut + (size_t)kIn * 8 * CQ + (size_t)kIn * kOut + 4 * kIn + kOut;
}

template <int CQ>
__device__ __forceinline__ void load_rows(float* sy, const GradArgs& a, int64_t tile, int tid) {
  // rows of 8 CQ floats, zero beyond dv and beyond the points
  for (int c = tid; c < kIn * 8 * CQ; c += kThreads) {
    const int j = c / (8 * CQ), q = c % (8 * CQ);
    const int64_t gj = tile * kIn + j;
    const bool ok = gj < a.n_in && q < a.dv;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(sy + c);
    const float* src = ok ? a.in_v + gj * a.dv + q : a.in_v;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(ok ? 4 : 0) : "memory");
  }
}

__device__ __forceinline__ void load_tile_t(float* st, const float* src_t, int64_t ld, int64_t tile, int d, int tid) {
  for (int c = tid; c < d * (kIn / 4); c += kThreads) {
    const int kk = c / (kIn / 4), q = c % (kIn / 4);
    cp16(st + kk * kIn + 4 * q, src_t + (int64_t)kk * ld + tile * kIn + 4 * q);
  }
}

__device__ __forceinline__ void load_dat(float4* sd, const GradArgs& a, int64_t tile, int tid) {
  if (tid >= kIn) return;
  const int64_t gj = tile * kIn + tid;
  if (gj < a.n_in)
    cp16(sd + tid, a.dat + gj);
  else
    sd[tid] = make_float4(INFINITY, 0.f, INFINITY, 0.f);  // contributes 2^-inf times 0
}

// NV = 8 CQ values at most
template <int CQ>
__global__ void __launch_bounds__(kThreads, 1)
k_dot_grad(const GradArgs a, const DevState* __restrict__ dev, const Consts k) {
  extern __shared__ __align__(16) float smem[];
  float* so = smem;                          // [d][128] outer points
  float* si = so + a.d * kOut;               // [d][128] inner points of a tile
  float* sy = si + a.d * kIn;                // [128][8 CQ] the same, row-major
  float* sP = sy + kIn * 8 * CQ;             // [128 inner][128 outer], chunks permuted
  float4* sd = reinterpret_cast<float4*>(sP + kIn * kOut);
  float* soff = reinterpret_cast<float*>(sd + kIn);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int half = tid >> 7, og = tid & 15, cg = (tid >> 4) & 7;
  const int64_t o0 = (int64_t)blockIdx.x * kOut;
  const int it0 = (int)blockIdx.y * a.tiles_per_split;
  const int it1 = it0 + a.tiles_per_split < a.ntiles ? it0 + a.tiles_per_split : a.ntiles;
  const SweepF sp = sweep_floats_of(dev, k);
  const uint64_t ahA2 = pk(sp.ahA, sp.ahA), alA2 = pk(sp.alA, sp.alA);

  // sums of this thread's 8 outer points x CQ coordinates, as pairs of outer points
  uint64_t hi[4][CQ], lo[4][CQ];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < CQ; ++q) hi[r][q] = lo[r][q] = 0ull;

  load_tile_t(so, a.out_t, a.ld_out, blockIdx.x, a.d, tid);
  if (tid < kOut) soff[tid] = a.off[o0 + tid < a.n_out ? o0 + tid : a.n_out - 1].x;
  if (it0 < it1) {
    load_tile_t(si, a.in_t, a.ld_in, it0, a.d, tid);
    load_dat(sd, a, it0, tid);
  }
  cp_commit();
  for (int it = it0; it < it1; ++it) {
    load_rows<CQ>(sy, a, it, tid);  // used after the first contraction
    cp_commit();
    cp_wait<1>();
    __syncthreads();  // the tile's transposed points and data have landed
    {
      uint64_t z2[8][4];
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int p = 0; p < 4; ++p) z2[r][p] = 0ull;
#pragma unroll 2
      for (int kk = 0; kk < a.d; ++kk) {
        const float4 a0 = *reinterpret_cast<const float4*>(so + kk * kOut + ty * 4);
        const float4 a1 = *reinterpret_cast<const float4*>(so + kk * kOut + 64 + ty * 4);
        const ulonglong2 t0 = *reinterpret_cast<const ulonglong2*>(si + kk * kIn + tx * 4);
        const ulonglong2 t1 = *reinterpret_cast<const ulonglong2*>(si + kk * kIn + 64 + tx * 4);
        const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const uint64_t aa = pk(av[r], av[r]);
          z2[r][0] = f2fma(aa, t0.x, z2[r][0]);
          z2[r][1] = f2fma(aa, t0.y, z2[r][1]);
          z2[r][2] = f2fma(aa, t1.x, z2[r][2]);
          z2[r][3] = f2fma(aa, t1.y, z2[r][3]);
        }
      }
      float oA[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) oA[r] = soff[(r < 4) ? (ty * 4 + r) : (64 + ty * 4 + r - 4)];
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const int j0 = (p < 2 ? 0 : 64) + tx * 4 + 2 * (p & 1);  // the pair's inner points j0, j0 + 1
        const float4 d0 = sd[j0], d1 = sd[j0 + 1];
        float e0[8], e1[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const float2 e =
              upk(f2mul(exp2_pair(ahA2, alA2, z2[r][p], f2sub(pk(-oA[r], -oA[r]), pk(d0.x, d1.x))), pk(d0.y, d1.y)));
          e0[r] = e.x;
          e1[r] = e.y;
        }
        const int sw = (j0 >> 2) & 7;  // j0 and j0 + 1 share it
        float4* r0 = reinterpret_cast<float4*>(sP + j0 * kOut);
        float4* r1 = r0 + kOut / 4;
        r0[ty ^ sw] = make_float4(e0[0], e0[1], e0[2], e0[3]);
        r0[(16 + ty) ^ sw] = make_float4(e0[4], e0[5], e0[6], e0[7]);
        r1[ty ^ sw] = make_float4(e1[0], e1[1], e1[2], e1[3]);
        r1[(16 + ty) ^ sw] = make_float4(e1[4], e1[5], e1[6], e1[7]);
      }
    }
    cp_wait<0>();
    __syncthreads();  // P and the row-major points are in place; the transposed tile is free
    if (it + 1 < it1) {
      load_tile_t(si, a.in_t, a.ld_in, it + 1, a.d, tid);
      load_dat(sd, a, it + 1, tid);
    }
    cp_commit();
#pragma unroll 1
    for (int j0 = 64 * half; j0 < 64 * half + 64; j0 += kGradFold) {
      uint64_t acc[4][CQ];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < CQ; ++q) acc[r][q] = 0ull;
#pragma unroll 2
      for (int j = j0; j < j0 + kGradFold; ++j) {
        const int sw = (j >> 2) & 7;
        const ulonglong2* pr = reinterpret_cast<const ulonglong2*>(sP + j * kOut);
        const ulonglong2 p0 = pr[og ^ sw], p1 = pr[(16 + og) ^ sw];
        float y[CQ];
#pragma unroll
        for (int q = 0; q < CQ; q += 2) {
          const float2 t = *reinterpret_cast<const float2*>(sy + j * 8 * CQ + cg * CQ + q);
          y[q] = t.x;
          y[q + 1] = t.y;
        }
#pragma unroll
        for (int q = 0; q < CQ; ++q) {
          const uint64_t yy = pk(y[q], y[q]);
          acc[0][q] = f2fma(p0.x, yy, acc[0][q]);
          acc[1][q] = f2fma(p0.y, yy, acc[1][q]);
          acc[2][q] = f2fma(p1.x, yy, acc[2][q]);
          acc[3][q] = f2fma(p1.y, yy, acc[3][q]);
        }
      }
      // TwoSum per lane (two_sum of the header), errors into the low parts
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < CQ; ++q) {
          const uint64_t s = f2add(hi[r][q], acc[r][q]);
          const uint64_t bb = f2sub(s, hi[r][q]);
          const uint64_t e = f2add(f2sub(hi[r][q], f2sub(s, bb)), f2sub(acc[r][q], bb));
          hi[r][q] = s;
          lo[r][q] = f2add(lo[r][q], e);
        }
    }
    __syncthreads();  // P and the row-major points may be overwritten
  }
  cp_wait<0>();
  __syncthreads();
  // the two halves: the second one's sums through shared memory (the P buffer holds 128 x 64
  // doubles = 64 KB: [q][outer])
  double* sx = reinterpret_cast<double*>(sP);
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    if (half == 1 - w) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < CQ; ++q) {
          const float2 h = upk(hi[r][q]), l = upk(lo[r][q]);
          const int oc = (r < 2 ? 0 : 64) + og * 4 + 2 * (r & 1);
          const int qq = cg * CQ + q;
          double* c = sx + (int64_t)qq * kOut + oc;
          if (w == 0) {
            c[0] = (double)h.x + (double)l.x;
            c[1] = (double)h.y + (double)l.y;
          } else if (qq < a.dv) {
            const double v0 = c[0] + ((double)h.x + (double)l.x), v1 = c[1] + ((double)h.y + (double)l.y);
            double* p = a.part + ((int64_t)blockIdx.y * a.n_out + o0 + oc) * a.dv + qq;
            if (o0 + oc < a.n_out) p[0] = v0;
            if (o0 + oc + 1 < a.n_out) p[a.dv] = v1;
          }
        }
    }
    __syncthreads();
  }
}

// out_i = 2 s (mass_i p_i - weight_i sum_s part[s][i]), one thread per coordinate
__global__ void __launch_bounds__(256)
k_dot_grad_fin(const double* __restrict__ part, int splits, int64_t np, int d, const float* __restrict__ P,
               const double* __restrict__ mass, const float4* __restrict__ wsrc, double s, float* __restrict__ out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= np * d) return;
  const int64_t i = e / d;
  double acc = 0.0;
#pragma unroll 4
  for (int u = 0; u < splits; ++u) acc += part[(int64_t)u * np * d + e];
  out[e] = (float)(2.0 * s * (mass[i] * (double)P[e] - (double)wsrc[i].y * acc));
}

}  // namespace dot

int64_t dot_pad(int64_t np) { return (np + dot::kStage - 1) / dot::kStage * dot::kStage; }

cudaError_t dot_transpose(const float* P, int64_t np, int d, float* out, cudaStream_t st) {
  const int64_t ld = dot_pad(np);
  dim3 grid((unsigned)(ld / 32), (unsigned)((d + 31) / 32));
  dot::k_transpose_points<<<grid, dim3(32, 8), 0, st>>>(P, np, d, out, ld);
  return cudaGetLastError();
}

namespace {

template <int MODE>
cudaError_t launch_mode(const dot::Args& a, const Work& w, const Consts& k, int sms, cudaStream_t st) {
  const int64_t items = (int64_t)a.out_tiles * a.splits;
  const unsigned grid = (unsigned)(items < sms ? items : sms);
  return launch_kernel(dot::k_dot_sweep<MODE>, grid, dot::kThreads, dot::smem_floats(a.d) * sizeof(float), st, a, w.dev, k);
}

template <class K>
cudaError_t set_smem(K kern, size_t floats) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(floats * sizeof(float)));
}

}  // namespace

// the shared-memory limits of these kernels on the current device
cudaError_t dot_prepare() {
  const size_t sweep = dot::smem_floats(64);
  for (const auto kern : {dot::k_dot_sweep<dot::kRowSum>, dot::k_dot_sweep<dot::kColSum>, dot::k_dot_sweep<dot::kRowEval>,
                          dot::k_dot_sweep<dot::kColEval>, dot::k_dot_sweep<dot::kMax>, dot::k_dot_sweep<dot::kMax2>,
                          dot::k_dot_sweep<dot::kKmax>}) {
    const cudaError_t e = set_smem(kern, sweep);
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = set_smem(dot::k_dot_grad<2>, dot::grad_smem_floats<2>(64));
  if (e == cudaSuccess) e = set_smem(dot::k_dot_grad<4>, dot::grad_smem_floats<4>(64));
  if (e == cudaSuccess) e = set_smem(dot::k_dot_grad<6>, dot::grad_smem_floats<6>(64));
  if (e == cudaSuccess) e = set_smem(dot::k_dot_grad<8>, dot::grad_smem_floats<8>(64));
  return e;
}

int dot_tile() { return dot::kOut; }

// one side's sums of P times dv value columns per inner point, of the `count` outer points from
// `first` (a multiple of 128) on: part[splits][count][dv].  off / dat: outer and inner data (n_out and
// n_in entries)
cudaError_t dot_weighted(bool rows, const Work& w, const Consts& k, int64_t first, int64_t count, const float* values,
                         int dv, const float4* off, const float4* dat, int splits, double* part, cudaStream_t st) {
  dot::GradArgs a{};
  a.out_t = (rows ? w.xt : w.yt) + first;
  a.in_t = rows ? w.yt : w.xt;
  a.in_v = values;
  a.n_out = count;
  a.n_in = rows ? k.m : k.n;
  a.ld_out = dot_pad(rows ? k.n : k.m);
  a.ld_in = dot_pad(a.n_in);
  a.d = k.d;
  a.dv = dv;
  a.ntiles = (int)((a.n_in + dot::kIn - 1) / dot::kIn);
  a.tiles_per_split = (a.ntiles + splits - 1) / splits;
  a.off = off + first;
  a.dat = dat;
  a.part = part;
  const dim3 grid((unsigned)((a.n_out + dot::kOut - 1) / dot::kOut), (unsigned)splits);
  const auto go = [&](auto cq) {
    constexpr int CQ = decltype(cq)::value;
    dot::k_dot_grad<CQ><<<grid, dot::kThreads, dot::grad_smem_floats<CQ>(k.d) * sizeof(float), st>>>(a, w.dev, k);
  };
  switch ((dv + 15) / 16) {  // pairs of value columns per thread
    case 1: go(std::integral_constant<int, 2>{}); break;
    case 2: go(std::integral_constant<int, 4>{}); break;
    case 3: go(std::integral_constant<int, 6>{}); break;
    default: go(std::integral_constant<int, 8>{}); break;
  }
  return cudaGetLastError();
}

// the gradient of the `count` outer points from `first` on
cudaError_t dot_grad(bool rows, const Inputs& in, const Work& w, const Consts& k, int cur, int64_t first, int64_t count,
                     int splits, double* part, float* out, cudaStream_t st) {
  // rows: weights w_j of the column data, outer offsets RqA; columns: weights q_i, offsets BqA
  const float4* off = rows ? w.g2row : w.colq[cur];
  const float4* dat = rows ? w.colq[cur] : w.g2row;
  cudaError_t e = dot_weighted(rows, w, k, first, count, rows ? in.y : in.x, k.d, off, dat, splits, part, st);
  if (e != cudaSuccess) return e;
  dot::k_dot_grad_fin<<<(unsigned)((count * k.d + 255) / 256), 256, 0, st>>>(
      part, splits, count, k.d, (rows ? in.x : in.y) + first * k.d, (rows ? in.r : w.colA) + first, off + first, k.s,
      out + first * k.d);
  return cudaGetLastError();
}

cudaError_t dot_launch(int mode, const Work& w, const Consts& k, const Geometry& g, cudaStream_t st) {
  const bool cols = mode == kDotColSum || mode == kDotColEval;
  dot::Args a{};
  a.out_t = cols ? w.yt : w.xt;
  a.in_t = cols ? w.xt : w.yt;
  a.n_out = cols ? k.m : k.n;
  a.n_in = cols ? k.n : k.m;
  a.ld_out = dot_pad(a.n_out);
  a.ld_in = dot_pad(a.n_in);
  a.d = k.d;
  a.splits = cols ? g.cols_split : g.rows_split;
  a.ntiles = (int)((a.n_in + dot::kIn - 1) / dot::kIn);
  a.tiles_per_split = (a.ntiles + a.splits - 1) / a.splits;
  a.out_tiles = (int)((a.n_out + dot::kOut - 1) / dot::kOut);
  for (int b = 0; b < 2; ++b) {
    a.off2[b] = w.rowshift[b];
    a.off4[b] = w.colq[b];
    a.dat[b] = cols ? w.g2row : w.colq[b];
  }
  a.part = cols ? w.colpart : w.rowpart;
  a.pmax = w.rowmax;
  switch (mode) {
    case kDotRowSum: return launch_mode<dot::kRowSum>(a, w, k, g.sms, st);
    case kDotColSum: return launch_mode<dot::kColSum>(a, w, k, g.sms, st);
    case kDotRowEval: return launch_mode<dot::kRowEval>(a, w, k, g.sms, st);
    case kDotColEval: return launch_mode<dot::kColEval>(a, w, k, g.sms, st);
    case kDotMax: return launch_mode<dot::kMax>(a, w, k, g.sms, st);
    case kDotMax2: return launch_mode<dot::kMax2>(a, w, k, g.sms, st);
    default: return launch_mode<dot::kKmax>(a, w, k, g.sms, st);
  }
}

}  // namespace lamp
