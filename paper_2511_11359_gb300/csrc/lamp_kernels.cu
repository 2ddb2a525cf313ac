// CUDA kernels of the LAMP hot path (arXiv 2511.11359, Alg. 2 and Section 4).
//
// One iteration = four launches:
//   G1  row sweep     S^A_i, S^B_i = sum_j 2^{v_ij} w_j          (row LSE, Section 4.1)
//   RF  row finalize  log Z_i, weights q_i = r_i / S_i, next row shifts
//   G2  column sweep  col_j = w_j sum_i 2^{v_ij} q_i for both streams, and
//                     sum_i z_ij X_ij for <C, X^t>                 (column sum, Section 4.1)
//   CF  column finalize: the O(m) float64 dual step of Alg. 2 (thetabar, nu, thetahat,
//                     tclip), residual ||col - c||_1, the next sweep's column data; its
//                     last block reduces the block partials and applies or rejects the update.
// RF and CF are in lamp_fin.cu.  Only the column sweeps of evaluation passes accumulate <C, X^t>.
// See lamp_common.cuh for the compensated exponent.
#include <cfloat>
#include <cmath>

#include "lamp_common.cuh"

namespace lamp {

// ------------------------------------------------------------------------------------------
// small helpers

__device__ __forceinline__ float warp_max_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ float warp_min_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// ------------------------------------------------------------------------------------------
// sweeps over point clouds (LAMP_COST_SQEUCLID, float32 CUDA-core x.y)

// stage a tile of 128 points (rows base.., np valid) x d coordinates into s[kk * 128 + p]:
// thread (p = idx % 128, coordinate quad) reads up to 4 consecutive coordinates of one
// point (one 16-byte load when d % 4 == 0 and the points are 16-byte aligned, which a caller's
// need not be) and consecutive threads write consecutive p, so the transposed shared stores are
// free of bank conflicts
__device__ __forceinline__ void stage_points(float* __restrict__ s, const float* __restrict__ P, int64_t base,
                                             int64_t np, int d, int tid, int nthreads) {
  const int dq = (d + 3) >> 2;
  const bool vec = (d & 3) == 0 && (reinterpret_cast<uintptr_t>(P) & 15) == 0;
  for (int idx = tid; idx < 128 * dq; idx += nthreads) {
    const int p = idx & 127, kq = (idx >> 7) << 2;
    const int64_t g = base + p;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (g < np) {
      if (vec) {
        const float4 t = *reinterpret_cast<const float4*>(P + g * d + kq);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (kq + q < d) v[q] = P[g * d + kq + q];
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (kq + q < d) s[(kq + q) * 128 + p] = v[q];
  }
}
//
// A CTA of 256 threads owns 128 "outer" points and loops over tiles of 128
// "inner" points; each thread computes an 8x8 block of z = x.y (outer rows
// {4ty..4ty+3, 64+4ty..}, inner columns {4tx..4tx+3, 64+4tx..}), in a fixed
// k order so that the row sweep and the column sweep produce bit-identical z.
// Row sweep: outer = rows (x), inner = columns (y).  Column sweep: the reverse.

constexpr int kPT = 128;
constexpr int kThreads = 256;

// M_MAX2: row maxima of u_ij = v_ij - Br_j with the row shifts applied and the column
// remainders Br_j (floats, in the column data's second field) subtracted: the refinement
// pass of the eta = 0 dual bound (see launch_dual), accurate to a few ulps of the grid
enum SweepMode : int { M_ROWSUM = 0, M_COLSUM = 1, M_MAX = 2, M_KMAX = 3, M_GRAD = 4, M_MAX2 = 5 };

// buffers of a sweep, indexed by the state-buffer parity dev->cur
struct SweepIO {
  const float2* off2[2];
  const float4* off4[2];
  const float4* indat[2];
};

// M_ROWSUM, M_COLSUM: DG = 1 is an evaluation pass (stream A alone, column sums also weighted by
// the cost).
// M_GRAD accumulates sum_b 2^{v_ab} weight_b V_b[0:DG], V = Vin (n_in x DG, row-major): the
// transport map of costs that the packed kernels do not serve (l1, l-inf with d > 8)
template <int MODE, int DG>
__global__ void __launch_bounds__(kThreads, MODE == M_GRAD ? 1 : 2)
k_pts_sweep(const float* __restrict__ P_out, const float* __restrict__ P_in, int64_t n_out, int64_t n_in, int d,
            const SweepIO io, double* __restrict__ part, float* __restrict__ pmax, int tiles_per_split,
            const DevState* __restrict__ dev, const Consts k, const float* __restrict__ Vin) {
  if ((MODE == M_ROWSUM || MODE == M_COLSUM) && dev->done) return;
  const int cur = dev->cur;
  const float2* __restrict__ off2 = cur ? io.off2[1] : io.off2[0];
  const float4* __restrict__ off4 = cur ? io.off4[1] : io.off4[0];
  const float4* __restrict__ in_data = cur ? io.indat[1] : io.indat[0];
  extern __shared__ __align__(16) float smem[];
  float* sOut = smem;                          // [d][128]
  float* sIn = smem + d * kPT;                 // [d][128]
  float4* sDat = reinterpret_cast<float4*>(smem + 2 * d * kPT);  // [128]
  float* sV = smem + 2 * d * kPT + 4 * kPT;                        // [DG][128] (M_GRAD with Vin)

  const int tid = threadIdx.x;
  const int tx = tid & 15;
  const int ty = tid >> 4;
  const int64_t o0 = (int64_t)blockIdx.x * kPT;
  const int split = blockIdx.y;
  const int64_t ntiles_in = (n_in + kPT - 1) / kPT;
  const int64_t it0 = (int64_t)split * tiles_per_split;
  int64_t it1 = it0 + tiles_per_split;
  if (it1 > ntiles_in) it1 = ntiles_in;

  const SweepF sp = sweep_floats_of(dev, k);

  stage_points(sOut, P_out, o0, n_out, d, tid, kThreads);

  // outer offsets of this thread's 8 outer points
  float oA[8], oB[8];
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    int64_t go = o0 + ((a < 4) ? (ty * 4 + a) : (64 + ty * 4 + a - 4));
    if (go >= n_out) go = n_out - 1;
    if (MODE == M_COLSUM) {
      float4 q = off4[go];
      oA[a] = q.x;
      oB[a] = q.z;
    } else if (MODE == M_GRAD) {
      float4 q = off4[go];  // row gradient: g2row {RqA, ..}; column gradient: colq {BqA, ..}
      oA[a] = q.x;
      oB[a] = 0.f;
    } else if (MODE == M_MAX) {
      oA[a] = 0.f;
      oB[a] = 0.f;
    } else if (MODE == M_MAX2) {
      oA[a] = off2[go].x;
      oB[a] = 0.f;
    } else {
      float2 q = off2[go];
      oA[a] = q.x;
      oB[a] = q.y;
    }
  }

  const float ahA = sp.ahA, alA = sp.alA, ahB = sp.ahB, alB = sp.alB;

  constexpr bool EV = MODE <= M_COLSUM && DG > 0;  // evaluation pass: stream A alone
  constexpr bool WC = MODE == M_COLSUM && EV;      // ... and the cost-weighted sums
  constexpr int NACC = EV && !WC ? 1 : 2;
  float hi[8][NACC], lo[8][NACC];
  float mx[8][2];
  double gacc[8][DG > 0 ? DG : 1];
#pragma unroll
  for (int a = 0; a < 8; ++a) {
#pragma unroll
    for (int q = 0; q < NACC; ++q) { hi[a][q] = 0.f; lo[a][q] = 0.f; }
    mx[a][0] = -INFINITY;
    mx[a][1] = -INFINITY;
#pragma unroll
    for (int q = 0; q < (DG > 0 ? DG : 1); ++q) gacc[a][q] = 0.0;
  }

  for (int64_t it = it0; it < it1; ++it) {
    const int64_t i0 = it * kPT;
    __syncthreads();
    stage_points(sIn, P_in, i0, n_in, d, tid, kThreads);
    if (MODE == M_GRAD) {
      for (int idx = tid; idx < DG * kPT; idx += kThreads) {
        int p = idx / (DG > 0 ? DG : 1), q = idx - p * (DG > 0 ? DG : 1);
        int64_t gi = i0 + p;
        sV[q * kPT + p] = gi < n_in ? Vin[gi * DG + q] : 0.0f;
      }
    }
    if (tid < kPT) {
      int64_t gi = i0 + tid;
      float4 v;
      if (gi < n_in) {
        v = in_data[gi];
      } else {
        v = make_float4(INFINITY, 0.f, INFINITY, 0.f);
        if (MODE == M_KMAX) v.x = -INFINITY;
      }
      sDat[tid] = v;
    }
    __syncthreads();

    float z[8][8];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 8; ++b) z[a][b] = 0.f;

#pragma unroll 2
    for (int kk = 0; kk < d; ++kk) {
      float4 a0 = *reinterpret_cast<const float4*>(&sOut[kk * kPT + ty * 4]);
      float4 a1 = *reinterpret_cast<const float4*>(&sOut[kk * kPT + 64 + ty * 4]);
      float4 b0 = *reinterpret_cast<const float4*>(&sIn[kk * kPT + tx * 4]);
      float4 b1 = *reinterpret_cast<const float4*>(&sIn[kk * kPT + 64 + tx * 4]);
      float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
      {
        // the ground cost of the direct form (Consts::cost_op; uniform branch)
        if (k.cost_op == 0) {
#pragma unroll
          for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) {
              const float df = av[a] - bv[b];
              z[a][b] = __fmaf_rn(df, df, z[a][b]);
            }
        } else if (k.cost_op == 1) {
#pragma unroll
          for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) z[a][b] += fabsf(av[a] - bv[b]);
        } else {
#pragma unroll
          for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) z[a][b] = fmaxf(z[a][b], fabsf(av[a] - bv[b]));
        }
      }
    }

    float4 dat[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) dat[b] = sDat[(b < 4) ? (tx * 4 + b) : (64 + tx * 4 + b - 4)];

    if (MODE == M_ROWSUM || MODE == M_COLSUM) {
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        float sA = 0.f, sB = 0.f;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          const float zz = z[a][b];
          const float eA = ex2(__fmaf_rn(alA, zz, __fmaf_rn(ahA, zz, -(oA[a] + dat[b].x))));
          if (MODE == M_ROWSUM) {
            sA = __fmaf_rn(eA, dat[b].y, sA);
          } else {
            const float pA = __fmul_rn(eA, dat[b].y);
            sA = __fadd_rn(sA, pA);
            if (WC) sB = __fmaf_rn(zz, pA, sB);
          }
          if (!EV) {
            const float eB = ex2(__fmaf_rn(alB, zz, __fmaf_rn(ahB, zz, -(oB[a] + dat[b].z))));
            sB = __fmaf_rn(eB, dat[b].w, sB);
          }
        }
        ff_add(hi[a][0], lo[a][0], sA);
        if (NACC > 1) ff_add(hi[a][NACC - 1], lo[a][NACC - 1], sB);
      }
    } else if (MODE == M_MAX) {
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          mx[a][0] = fmaxf(mx[a][0], __fmaf_rn(ahA, z[a][b], -dat[b].x));
          mx[a][1] = fmaxf(mx[a][1], __fmaf_rn(ahB, z[a][b], -dat[b].z));
        }
    } else if (MODE == M_MAX2) {
      // u = a z - (Rq + Bq) - Br: the offsets' sum is exact on the grid, a z exact in the fma,
      // and |u| is a few grid steps near the row maximum (Rq comes from the M_MAX pass)
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          const float zz = z[a][b];
          const float u = __fmaf_rn(alA, zz, __fmaf_rn(ahA, zz, -(oA[a] + dat[b].x))) - dat[b].y;
          mx[a][0] = fmaxf(mx[a][0], u);
        }
    } else if (MODE == M_KMAX) {
      // the unscaled cost
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          const bool pad = (dat[b].x == -INFINITY);
          const float dd = z[a][b];
          mx[a][0] = fmaxf(mx[a][0], pad ? -INFINITY : dd);
          mx[a][1] = fmaxf(mx[a][1], pad ? -INFINITY : -dd);
        }
    } else if (MODE == M_GRAD) {
      // sum over inner b of 2^{v_ab} * weight_b * P_in[b][:], stream A only
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        float g[DG > 0 ? DG : 1];
#pragma unroll
        for (int q = 0; q < DG; ++q) g[q] = 0.f;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          const float zz = z[a][b];
          const float vA = __fmaf_rn(alA, zz, __fmaf_rn(ahA, zz, -(oA[a] + dat[b].x)));
          const float pA = ex2(vA) * dat[b].y;
          const int ib = (b < 4) ? (tx * 4 + b) : (64 + tx * 4 + b - 4);
#pragma unroll
          for (int q = 0; q < DG; ++q) g[q] = __fmaf_rn(pA, sV[q * kPT + ib], g[q]);
        }
#pragma unroll
        for (int q = 0; q < DG; ++q) gacc[a][q] += (double)g[q];
      }
    }
  }

  // reduce over the 16 threads (tx) that share each outer point: lanes of one half-warp
  if (MODE == M_ROWSUM || MODE == M_COLSUM) {
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      int64_t go = o0 + ((a < 4) ? (ty * 4 + a) : (64 + ty * 4 + a - 4));
#pragma unroll
      for (int q = 0; q < NACC; ++q) {
        double v = (double)hi[a][q] + (double)lo[a][q];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (tx == 0 && go < n_out) part[((int64_t)split * NACC + q) * n_out + go] = v;
      }
    }
  } else if (MODE == M_MAX || MODE == M_KMAX || MODE == M_MAX2) {
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      int64_t go = o0 + ((a < 4) ? (ty * 4 + a) : (64 + ty * 4 + a - 4));
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float v = mx[a][q];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (tx == 0 && go < n_out) pmax[((int64_t)split * 2 + q) * n_out + go] = v;
      }
    }
  } else if (MODE == M_GRAD) {
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      int64_t go = o0 + ((a < 4) ? (ty * 4 + a) : (64 + ty * 4 + a - 4));
#pragma unroll
      for (int q = 0; q < DG; ++q) {
        double v = gacc[a][q];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (tx == 0 && go < n_out) part[((int64_t)split * n_out + go) * DG + q] = v;
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// sweeps over a stored dense cost (LAMP_COST_DENSE), streamed from HBM with coalesced loads

// Row sweep: a CTA of 256 threads owns kDR rows and steps over chunks of 1024 columns (thread t
// takes columns t + 256 q); column sweep: a CTA of 128 threads owns 256 columns (two per thread)
// and walks a split's rows in groups of 16.  These serve stored costs whose rows are not a
// multiple of 16 bytes apart (lamp_dense.cu streams the others).  Bound by the latency of the
// loads at the sizes that fit the L2 and by HBM above: the row sweep loads the next chunk's entries
// while the current one is evaluated, the column sweep the 32 entries of a thread's group at once, and
// the grid is fine enough to fill the SMs.  3001 x 2777: 19.9 -> 12.3 us (rows; 8 rows per CTA, no
// load ahead, a butterfly of five steps per sum), 20.4 -> 13.9 us (columns; 1024 columns per CTA).
constexpr int kDR = 4;          // rows per CTA in the row sweep
constexpr int kDSplitRows = 8;  // rows per tile in the choice of its splits
constexpr int kDChunk = 1024;   // columns per CTA step (4 per thread, stride 256)

// MODE = M_ROWSUM, M_MAX or M_MAX2; EV = 1: row sums of an evaluation pass (stream A alone)
template <int MODE, int EV = 0>
__global__ void __launch_bounds__(kThreads, 3)
k_dense_rows(const float* __restrict__ C, int64_t ldc, int64_t n, int64_t m, const Work w,
             int chunks_per_split, const Consts k) {
  const DevState* __restrict__ dev = w.dev;
  const int4 ctl = read_control(dev);
  if (MODE == M_ROWSUM && ctl.y) return;  // done
  const int cur = ctl.x;
  const float2* __restrict__ rowshift = w.rowshift[cur];
  const float4* __restrict__ colq = w.colq[cur];
  constexpr int NV = 2 * kDR;  // values per thread: both streams of kDR rows
  __shared__ double sred[kThreads / 32][NV];
  const int tid = threadIdx.x;
  const int64_t r0 = (int64_t)blockIdx.x * kDR;
  const int split = blockIdx.y;
  const int64_t nchunks = (m + kDChunk - 1) / kDChunk;
  const int64_t c0 = (int64_t)split * chunks_per_split;
  int64_t c1 = c0 + chunks_per_split;
  if (c1 > nchunks) c1 = nchunks;
  const SweepF sp = sweep_floats_of(dev, k);
  const uint64_t ahA2 = pk(sp.ahA, sp.ahA), alA2 = pk(sp.alA, sp.alA);
  const uint64_t ahB2 = pk(sp.ahB, sp.ahB), alB2 = pk(sp.alB, sp.alB);

  float oA[kDR], oB[kDR];
  const float* crow[kDR];
#pragma unroll
  for (int a = 0; a < kDR; ++a) {
    int64_t gr = r0 + a;
    if (gr >= n) gr = n - 1;
    float2 q = MODE == M_MAX ? make_float2(0.f, 0.f) : rowshift[gr];
    oA[a] = -q.x;
    oB[a] = -q.y;
    crow[a] = C + gr * ldc;
  }
  // sums: float-float values [2 a + stream]; maxima: hi alone
  float hi[NV], lo[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    hi[q] = MODE == M_ROWSUM ? 0.f : -INFINITY;
    lo[q] = 0.f;
  }
  const auto load = [&](int64_t ch, float (&cv)[kDR][4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t j = ch * kDChunk + tid + q * kThreads;
#pragma unroll
      for (int a = 0; a < kDR; ++a) cv[a][q] = j < m ? __ldg(crow[a] + j) : 0.f;
    }
  };
  float nx[kDR][4];
  if (c0 < c1) load(c0, nx);
  for (int64_t ch = c0; ch < c1; ++ch) {
    float cv[kDR][4];
#pragma unroll
    for (int a = 0; a < kDR; ++a)
#pragma unroll
      for (int q = 0; q < 4; ++q) cv[a][q] = nx[a][q];
    float4 cd[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t j = ch * kDChunk + tid + q * kThreads;
      cd[q] = j < m ? colq[j] : make_float4(INFINITY, 0.f, INFINITY, 0.f);
    }
    if (ch + 1 < c1) load(ch + 1, nx);
#pragma unroll
    for (int a = 0; a < kDR; ++a) {
      float sA = 0.f, sB = 0.f;
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const float4 d0 = cd[2 * p], d1 = cd[2 * p + 1];
        const uint64_t z2 = pk(cv[a][2 * p], cv[a][2 * p + 1]);
        if (MODE == M_ROWSUM) {
          const float2 eA = upk(exp2_pair(ahA2, alA2, z2, f2sub(pk(oA[a], oA[a]), pk(d0.x, d1.x))));
          sA = __fmaf_rn(eA.y, d1.y, __fmaf_rn(eA.x, d0.y, sA));
          if (!EV) {
            const float2 eB = upk(exp2_pair(ahB2, alB2, z2, f2sub(pk(oB[a], oB[a]), pk(d0.z, d1.z))));
            sB = __fmaf_rn(eB.y, d1.w, __fmaf_rn(eB.x, d0.w, sB));
          }
        } else if (MODE == M_MAX2) {
          // refinement pass of the eta = 0 dual bound (see k_pts_sweep, M_MAX2)
          const float2 u = upk(f2sub(f2fma(alA2, z2, f2fma(ahA2, z2, f2sub(pk(oA[a], oA[a]), pk(d0.x, d1.x)))),
                                     pk(d0.y, d1.y)));
          hi[2 * a] = fmaxf(hi[2 * a], fmaxf(u.x, u.y));
        } else {
          const float2 uA = upk(f2fma(ahA2, z2, pk(-d0.x, -d1.x))), uB = upk(f2fma(ahB2, z2, pk(-d0.z, -d1.z)));
          hi[2 * a] = fmaxf(hi[2 * a], fmaxf(uA.x, uA.y));
          hi[2 * a + 1] = fmaxf(hi[2 * a + 1], fmaxf(uB.x, uB.y));
        }
      }
      if (MODE == M_ROWSUM) {
        ff_add(hi[2 * a], lo[2 * a], sA);
        ff_add(hi[2 * a + 1], lo[2 * a + 1], sB);
      }
    }
  }

  const int lane = tid & 31, wid = tid >> 5;
  if (MODE == M_ROWSUM) {
    warp_sums_ff<NV>(hi, lo, lane);
    if ((lane & (32 / NV - 1)) == 0) sred[wid][lane / (32 / NV)] = (double)hi[0] + (double)lo[0];
    __syncthreads();
    if (tid < NV) {
      double v = 0.0;
      for (int u = 0; u < kThreads / 32; ++u) v += sred[u][tid];
      const int a = tid >> 1, s = tid & 1;
      if (r0 + a < n && s < 2 - EV) w.rowpart[((int64_t)split * (2 - EV) + s) * n + r0 + a] = v;
    }
  } else {
    __shared__ float fred[kThreads / 32][NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      const float v = warp_max_f(hi[q]);
      if (lane == 0) fred[wid][q] = v;
    }
    __syncthreads();
    if (tid < NV) {
      float v = -INFINITY;
      for (int u = 0; u < kThreads / 32; ++u) v = fmaxf(v, fred[u][tid]);
      const int a = tid >> 1, s = tid & 1;
      if (r0 + a < n) w.rowmax[((int64_t)split * 2 + s) * n + r0 + a] = v;
    }
  }
}

constexpr int kDColRows = 16;      // rows per group: the unit of the column sums
constexpr int kDColThreads = 128;  // two columns per thread
constexpr int kDCols = 2 * kDColThreads;

template <int WC>  // 1: an evaluation pass: stream A's sums and the cost-weighted ones
__global__ void __launch_bounds__(kDColThreads, 6)
k_dense_cols(const float* __restrict__ C, int64_t ldc, int64_t n, int64_t m, const Work w, int64_t rows_per_split,
             const Consts k) {
  const DevState* __restrict__ dev = w.dev;
  const int4 ctl = read_control(dev);
  if (ctl.y) return;  // done
  const float4* __restrict__ g2row = w.g2row;
  const float4* __restrict__ colq = w.colq[ctl.x];
  double* __restrict__ part = w.colpart;
  const int tid = threadIdx.x;
  const int split = blockIdx.y;
  const int64_t i0 = (int64_t)split * rows_per_split;
  int64_t i1 = i0 + rows_per_split;
  if (i1 > n) i1 = n;
  const SweepF sp = sweep_floats_of(dev, k);
  const uint64_t ahA2 = pk(sp.ahA, sp.ahA), alA2 = pk(sp.alA, sp.alA);
  const uint64_t ahB2 = pk(sp.ahB, sp.ahB), alB2 = pk(sp.alB, sp.alB);

  int64_t jj[2];
  bool ok[2];
  float oA[2], oB[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    jj[q] = (int64_t)blockIdx.x * kDCols + tid + q * kDColThreads;
    ok[q] = jj[q] < m;
    const float4 cd = ok[q] ? colq[jj[q]] : make_float4(0.f, 0.f, 0.f, 0.f);
    oA[q] = -cd.x;
    oB[q] = -cd.z;
  }
  const uint64_t oA2 = pk(oA[0], oA[1]), oB2 = pk(oB[0], oB[1]);
  float hiA[2], loA[2], hiB[2], loB[2], hiC[2], loC[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) hiA[q] = loA[q] = hiB[q] = loB[q] = hiC[q] = loC[q] = 0.f;

  // the entries of a group; rows past the split's end read its last row and are not added
  const auto load = [&](int64_t ib, float (&cv)[kDColRows][2]) {
#pragma unroll
    for (int a = 0; a < kDColRows; ++a) {
      const int64_t gi = ib + a < i1 ? ib + a : i1 - 1;
#pragma unroll
      for (int q = 0; q < 2; ++q) cv[a][q] = ok[q] ? __ldg(C + gi * ldc + jj[q]) : 0.f;
    }
  };
  for (int64_t ib = i0; ib < i1; ib += kDColRows) {
    float cv[kDColRows][2];
    load(ib, cv);
    float sA[2] = {0.f, 0.f}, sB[2] = {0.f, 0.f}, sC[2] = {0.f, 0.f};
#pragma unroll
    for (int a = 0; a < kDColRows; ++a) {
      if (ib + a >= i1) break;
      const float4 rd = __ldg(g2row + ib + a);
      const uint64_t z2 = pk(cv[a][0], cv[a][1]);
      const float2 eA = upk(exp2_pair(ahA2, alA2, z2, f2sub(oA2, pk(rd.x, rd.x))));
      const float pA[2] = {__fmul_rn(eA.x, rd.y), __fmul_rn(eA.y, rd.y)};
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        sA[q] = __fadd_rn(sA[q], pA[q]);
        if (WC) sC[q] = __fmaf_rn(cv[a][q], pA[q], sC[q]);
      }
      if (!WC) {
        const float2 eB = upk(exp2_pair(ahB2, alB2, z2, f2sub(oB2, pk(rd.z, rd.z))));
        sB[0] = __fmaf_rn(eB.x, rd.w, sB[0]);
        sB[1] = __fmaf_rn(eB.y, rd.w, sB[1]);
      }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      ff_add(hiA[q], loA[q], sA[q]);
      if (WC) ff_add(hiC[q], loC[q], sC[q]);
      else ff_add(hiB[q], loB[q], sB[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    if (!ok[q]) continue;
    part[((int64_t)split * 2 + 0) * m + jj[q]] = (double)hiA[q] + (double)loA[q];
    part[((int64_t)split * 2 + 1) * m + jj[q]] = WC ? (double)hiC[q] + (double)loC[q] : (double)hiB[q] + (double)loB[q];
  }
}

// dense cost: max, min and finiteness of C (the K pass, Section 2: K = ||C||_inf)
__global__ void k_dense_stats(const float* __restrict__ C, int64_t ldc, int64_t n, int64_t m, double* out) {
  __shared__ float smx[kThreads / 32], smn[kThreads / 32];
  __shared__ int sbad[kThreads / 32];
  float mx = -INFINITY, mn = INFINITY;
  int bad = 0;
  const int64_t total = n * m;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = e / m, j = e - i * m;
    float v = C[i * ldc + j];
    if (!isfinite(v)) bad = 1;
    mx = fmaxf(mx, v);
    mn = fminf(mn, v);
  }
  mx = warp_max_f(mx);
  mn = warp_min_f(mn);
  bad = __any_sync(0xffffffffu, bad);
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) { smx[wid] = mx; smn[wid] = mn; sbad[wid] = bad; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kThreads / 32; ++w) { mx = fmaxf(mx, smx[w]); mn = fminf(mn, smn[w]); bad |= sbad[w]; }
    mx = fmaxf(mx, smx[0]); mn = fminf(mn, smn[0]); bad |= sbad[0];
    out[3 * blockIdx.x + 0] = mx;
    out[3 * blockIdx.x + 1] = mn;
    out[3 * blockIdx.x + 2] = bad;
  }
}

// ------------------------------------------------------------------------------------------
// O(n + m) kernels

__global__ void k_norms(const float* __restrict__ P, int64_t np, int d, double* __restrict__ nrm,
                        float2* __restrict__ f2, float4* __restrict__ f4) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  double s = 0.0;
  float sf = 0.f;
  for (int k = 0; k < d; ++k) {
    float v = P[i * d + k];
    s += (double)v * (double)v;
    sf = __fmaf_rn(v, v, sf);
  }
  nrm[i] = s;
  if (f2) f2[i] = make_float2(sf, 0.f);
  if (f4) f4[i] = make_float4(sf, 0.f, 0.f, 0.f);
}

// cosine cost: out_i = P_i / (sqrt 2 |P_i|) (float64 norm); rows with a zero or non-finite
// norm are counted in *bad and written as zeros
__global__ void k_unit_rows(const float* __restrict__ P, int64_t np, int d, float* __restrict__ out,
                            unsigned int* __restrict__ bad) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  double s = 0.0;
  for (int q = 0; q < d; ++q) s += (double)P[i * d + q] * (double)P[i * d + q];
  double sc = 0.0;
  if (s > 0.0 && isfinite(s)) sc = 1.0 / sqrt(2.0 * s);
  else atomicAdd(bad, 1u);
  for (int q = 0; q < d; ++q) out[i * d + q] = (float)((double)P[i * d + q] * sc);
}

// what lamp_create reads back of its inputs, in one pass: per block kStatFields doubles
//   0 sum r   1 min r   2 r not finite   3 -sum r log r   4 sum r |x|^2   5 max |x|^2
//   6 sum c   7 min c   8 c not finite   9 max |y|^2   10 max of rowmax[.][0]   11 max of rowmax[.][1]
// (nx, ny null: no norms; rows = 0: no K pass)
__global__ void __launch_bounds__(kThreads)
k_create_stats(const double* __restrict__ r, int64_t n, const double* __restrict__ c, int64_t m,
               const double* __restrict__ nx, const double* __restrict__ ny, const float* __restrict__ rowmax,
               int64_t rows, int splits, double* __restrict__ out) {
  double v[kStatFields];
#pragma unroll
  for (int q = 0; q < kStatFields; ++q) v[q] = 0.0;
  v[1] = v[7] = INFINITY;
  float mx = -INFINITY, mn = -INFINITY;
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = i0; i < n; i += step) {
    const double x = r[i];
    if (!isfinite(x)) v[2] = 1.0;
    v[0] += x;
    v[1] = fmin(v[1], x);
    v[3] -= x * log(x);
    if (nx) {
      v[4] += x * nx[i];
      v[5] = fmax(v[5], nx[i]);
    }
  }
  for (int64_t j = i0; j < m; j += step) {
    const double x = c[j];
    if (!isfinite(x)) v[8] = 1.0;
    v[6] += x;
    v[7] = fmin(v[7], x);
    if (ny) v[9] = fmax(v[9], ny[j]);
  }
  for (int s = 0; s < splits; ++s)
    for (int64_t i = i0; i < rows; i += step) {
      mx = fmaxf(mx, rowmax[((int64_t)s * 2 + 0) * rows + i]);
      mn = fmaxf(mn, rowmax[((int64_t)s * 2 + 1) * rows + i]);
    }
  v[10] = mx;
  v[11] = mn;
  __shared__ double sh[kThreads / 32][kStatFields];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // sums in the fields 0, 3, 4, 6; minima in 1, 7; maxima in the others
#pragma unroll
  for (int q = 0; q < kStatFields; ++q) {
    const bool add = q == 0 || q == 3 || q == 4 || q == 6, low = q == 1 || q == 7;
    double x = v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double y = __shfl_xor_sync(0xffffffffu, x, o);
      x = add ? x + y : low ? fmin(x, y) : fmax(x, y);
    }
    if (lane == 0) sh[wid][q] = x;
  }
  __syncthreads();
  if (threadIdx.x < kStatFields) {
    const int q = threadIdx.x;
    const bool add = q == 0 || q == 3 || q == 4 || q == 6, low = q == 1 || q == 7;
    double x = sh[0][q];
    for (int u = 1; u < kThreads / 32; ++u) x = add ? x + sh[u][q] : low ? fmin(x, sh[u][q]) : fmax(x, sh[u][q]);
    out[kStatFields * blockIdx.x + q] = x;
  }
}

// set the column data of the current state buffer from its (nu, theta) and dev->kappa
__global__ void k_init_cols(const Work w, const Consts k, int zero) {
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= k.m) return;
  const DevState* __restrict__ dev = w.dev;
  const int cur = dev->cur;
  const double* __restrict__ ny = w.ny;
  double* __restrict__ nu = w.nu[cur];
  double* __restrict__ theta = w.theta[cur];
  float4* __restrict__ colq = w.colq[cur];
  if (zero) { nu[j] = 0.0; theta[j] = 0.0; }
  SweepParams sp = make_sweep_params(sweep_kappa(dev->kappa, k), k);
  double wt = k.tau1 / sp.kapB;  // tau1 eta_{t+1}
  double nb = nu[j] + wt * (theta[j] - nu[j]);
  double sny = k.zdot ? k.s * ny[j] : 0.0;
  float dB;
  const float4 cd = column_data(nu[j], nb, sny, sp, k, &dB);
  colq[j] = cd;
  if (w.colq2[cur]) store_pair_entry(w.colq2[cur], j, cd.x, cd.y, dB, cd.w);
}

// row shifts from the prime pass' row maxima: Rq = round_g(max_j (a z_ij - Bq_j))
__global__ void k_prime_fin(const Work w, int splits, const Consts k) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= k.n) return;
  const DevState* __restrict__ dev = w.dev;
  const float* __restrict__ pmax = w.rowmax;
  float2* __restrict__ rowshift = w.rowshift[dev->cur];
  SweepParams sp = make_sweep_params(sweep_kappa(dev->kappa, k), k);
  float mA = -INFINITY, mB = -INFINITY;
  for (int s = 0; s < splits; ++s) {
    mA = fmaxf(mA, pmax[((int64_t)s * 2 + 0) * k.n + i]);
    mB = fmaxf(mB, pmax[((int64_t)s * 2 + 1) * k.n + i]);
  }
  double qA = isfinite(mA) ? quantize((double)mA, sp.g) : 0.0;
  double qB = isfinite(mB) ? quantize((double)mB, sp.g) : 0.0;
  if (k.shared_shift) qB = qA;
  rowshift[i] = make_float2((float)qA, (float)qB);
}

// ------------------------------------------------------------------------------------------
// launch glue

static inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

static size_t pts_smem(int d, int dv = 0) {
  return (size_t)(2 * d * kPT + dv * kPT) * sizeof(float) + kPT * sizeof(float4);
}

static SweepIO io_same(const float2* o2, const float4* o4, const float4* in) {
  SweepIO io;
  io.off2[0] = io.off2[1] = o2;
  io.off4[0] = io.off4[1] = o4;
  io.indat[0] = io.indat[1] = in;
  return io;
}

template <int MODE, int DG>
static cudaError_t launch_pts(const float* Pout, const float* Pin, int64_t nout, int64_t nin, int d, const SweepIO& io,
                              double* part, float* pmax, int splits, const DevState* dev, const Consts& k,
                              cudaStream_t st, const float* V = nullptr) {
  auto kern = k_pts_sweep<MODE, DG>;
  size_t sm = pts_smem(d, V ? DG : 0);
  int64_t tin = cdiv(nin, kPT);
  int tps = (int)cdiv(tin, splits);
  dim3 grid((unsigned)cdiv(nout, kPT), (unsigned)splits);
  return launch_kernel(kern, grid, kThreads, sm, st, Pout, Pin, nout, nin, d, io, part, pmax, tps, dev, k, V);
}

// the packed direct-form sweeps serve |x - y|^2 with d <= 8 in float32
bool uses_direct_sweeps(const Consts& k, int prec) {
  return k.kind == COST_SQEUCLID && !k.zdot && prec != 1 /* LAMP_PREC_BF16_TC */ && k.d >= 1 && k.d <= 8;
}

cudaError_t launch_unit_rows(const float* P, int64_t np, int d, float* out, unsigned int* bad, cudaStream_t st) {
  k_unit_rows<<<(unsigned)cdiv(np, 256), 256, 0, st>>>(P, np, d, out, bad);
  return cudaGetLastError();
}

cudaError_t launch_norms(const Inputs& in, const Consts& k, const Work& w, cudaStream_t st) {
  if (k.kind != COST_SQEUCLID) return cudaSuccess;
  // float32 norms go into buffers that are unused before the first iteration
  k_norms<<<(unsigned)cdiv(k.n, 256), 256, 0, st>>>(in.x, k.n, k.d, w.nx, w.rowshift[1], nullptr);
  k_norms<<<(unsigned)cdiv(k.m, 256), 256, 0, st>>>(in.y, k.m, k.d, w.ny, nullptr, w.colq[1]);
  return cudaGetLastError();
}

// the K pass's column data in the packed-pair layout: -offA = |y_j|^2 (the float norms that
// k_norms left in f4[j].x)
__global__ void k_norm_pairs(const float4* __restrict__ f4, float4* __restrict__ pairs, int64_t m) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < m) store_pair_entry(pairs, j, -f4[j].x, 0.f, 0.f, 0.f);
}

cudaError_t launch_kmax(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int prec,
                        cudaStream_t st) {
  if (k.kind == COST_DENSE) {
    k_dense_stats<<<4 * g.sms, kThreads, 0, st>>>(in.C, in.ldc, k.n, k.m, w.scratch);
    return cudaGetLastError();
  }
  if (prec == 1 /* LAMP_PREC_BF16_TC */ && g.map_x && w.colq2[1]) {
    // on the tensor cores, with the products of the bf16 points the iteration uses: the
    // row data (rowshift[1].x) hold |x_i|^2, the pair data |y_j|^2
    k_norm_pairs<<<(unsigned)cdiv(k.m, 256), 256, 0, st>>>(w.colq[1], w.colq2[1], k.m);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    Work w2 = w;
    w2.rowshift[0] = w2.rowshift[1] = w.rowshift[1];
    w2.colq2[0] = w2.colq2[1] = w.colq2[1];
    return tc_launch_rowmax(3, g, w2, k, g.rows_split, st);
  }
  if (w.xt) {
    Work w2 = w;
    w2.rowshift[0] = w2.rowshift[1] = w.rowshift[1];
    w2.colq[0] = w2.colq[1] = w.colq[1];
    return dot_launch(kDotKmax, w2, k, g, st);
  }
  if (k.shared_shift) return direct_max(kDirectKmax, in, w, k, g.rows_split, st);
  // l1 and l-inf with d > 8: rowmax[split][0][n] = max_j D_ij, rowmax[split][1][n] = max_j -D_ij, D the
  // unscaled cost
  return launch_pts<M_KMAX, 0>(in.x, in.y, k.n, k.m, k.d, io_same(w.rowshift[1], nullptr, w.colq[1]), nullptr,
                               w.rowmax, g.rows_split, w.dev, k, st);
}

cudaError_t launch_create_stats(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, bool kpass,
                                cudaStream_t st) {
  const bool pts = k.kind == COST_SQEUCLID;
  k_create_stats<<<kStatBlocks, kThreads, 0, st>>>(in.r, k.n, in.c, k.m, pts ? w.nx : nullptr, pts ? w.ny : nullptr,
                                                   w.rowmax, kpass && pts ? k.n : 0, g.rows_split, w.stats);
  return cudaGetLastError();
}

cudaError_t launch_init_state(const Inputs& in, const Consts& k, const Work& w, int zero, cudaStream_t st) {
  k_init_cols<<<(unsigned)cdiv(k.m, 256), 256, 0, st>>>(w, k, zero);
  return cudaGetLastError();
}

static cudaError_t launch_row_sweep(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int mode,
                                    int eval, cudaStream_t st) {
  if (k.kind == COST_DENSE && g.map_c)
    return mode == M_ROWSUM ? dense_launch_sweep(true, eval, g, w, k, g.rows_split, st)
                            : dense_launch_rowmax(mode == M_MAX2 ? 2 : 1, g, w, k, g.rows_split, st);
  if (k.kind == COST_DENSE) {
    int64_t nch = cdiv(k.m, kDChunk);
    int cps = (int)cdiv(nch, g.rows_split);
    dim3 grid((unsigned)cdiv(k.n, kDR), (unsigned)g.rows_split);
    const auto kern = mode == M_ROWSUM ? (eval ? k_dense_rows<M_ROWSUM, 1> : k_dense_rows<M_ROWSUM>) : mode == M_MAX2 ? k_dense_rows<M_MAX2> : k_dense_rows<M_MAX>;
    return launch_kernel(kern, grid, kThreads, 0, st, in.C, in.ldc, k.n, k.m, w, cps, k);
  }
  if (mode == M_ROWSUM && k.shared_shift) return launch_direct_sweep(true, eval, in, k, w, g, st);
  if (k.shared_shift) return direct_max(mode == M_MAX2 ? kDirectMax2 : kDirectMax, in, w, k, g.rows_split, st);
  if (k.zdot)
    return dot_launch(mode == M_ROWSUM ? (eval ? kDotRowEval : kDotRowSum) : mode == M_MAX2 ? kDotMax2 : kDotMax, w, k, g, st);
  SweepIO io;
  for (int b = 0; b < 2; ++b) {
    io.off2[b] = w.rowshift[b];
    io.off4[b] = nullptr;
    io.indat[b] = w.colq[b];
  }
  if (mode == M_ROWSUM && eval)
    return launch_pts<M_ROWSUM, 1>(in.x, in.y, k.n, k.m, k.d, io, w.rowpart, nullptr, g.rows_split, w.dev, k, st);
  if (mode == M_ROWSUM)
    return launch_pts<M_ROWSUM, 0>(in.x, in.y, k.n, k.m, k.d, io, w.rowpart, nullptr, g.rows_split, w.dev, k, st);
  if (mode == M_MAX2)
    return launch_pts<M_MAX2, 0>(in.x, in.y, k.n, k.m, k.d, io, nullptr, w.rowmax, g.rows_split, w.dev, k, st);
  return launch_pts<M_MAX, 0>(in.x, in.y, k.n, k.m, k.d, io, nullptr, w.rowmax, g.rows_split, w.dev, k, st);
}

static cudaError_t launch_col_sweep(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int eval,
                                    cudaStream_t st) {
  if (k.kind == COST_DENSE && g.map_c) return dense_launch_sweep(false, eval, g, w, k, g.cols_split, st);
  if (k.kind == COST_DENSE) {
    int64_t rps = cdiv(k.n, g.cols_split);
    rps = cdiv(rps, kDColRows) * kDColRows;
    dim3 grid((unsigned)cdiv(k.m, kDCols), (unsigned)g.cols_split);
    return launch_kernel(eval ? k_dense_cols<1> : k_dense_cols<0>, grid, kDColThreads, 0, st, in.C, in.ldc, k.n, k.m, w, rps, k);
  }
  if (k.shared_shift) return launch_direct_sweep(false, eval, in, k, w, g, st);
  if (k.zdot) return dot_launch(eval ? kDotColEval : kDotColSum, w, k, g, st);
  SweepIO io;
  for (int b = 0; b < 2; ++b) {
    io.off2[b] = nullptr;
    io.off4[b] = w.colq[b];
    io.indat[b] = w.g2row;
  }
  if (eval)
    return launch_pts<M_COLSUM, 1>(in.y, in.x, k.m, k.n, k.d, io, w.colpart, nullptr, g.cols_split, w.dev, k, st);
  return launch_pts<M_COLSUM, 0>(in.y, in.x, k.m, k.n, k.d, io, w.colpart, nullptr, g.cols_split, w.dev, k, st);
}

cudaError_t launch_prime(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int prec,
                         cudaStream_t st) {
  // the tensor-core context takes its row maxima from the tensor-core sweep (the cost its
  // iteration uses)
  cudaError_t e = prec == 1 /* LAMP_PREC_BF16_TC */ && g.map_x ? tc_launch_rowmax(1, g, w, k, g.rows_split, st)
                                                                : launch_row_sweep(in, k, w, g, M_MAX, 0, st);
  if (e != cudaSuccess) return e;
  k_prime_fin<<<(unsigned)cdiv(k.n, 256), 256, 0, st>>>(w, g.rows_split, k);
  return cudaGetLastError();
}

cudaError_t launch_rowmax_refined(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int prec,
                                  cudaStream_t st) {
  if (prec == 1 /* LAMP_PREC_BF16_TC */ && g.map_x) return tc_launch_rowmax(2, g, w, k, g.rows_split, st);
  return launch_row_sweep(in, k, w, g, M_MAX2, 0, st);
}

cudaError_t launch_iteration_part(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int prec,
                                  int part, int eval, cudaStream_t st) {
  const bool tcpath = prec == 1 /* LAMP_PREC_BF16_TC */;
  switch (part) {
    case 0:
      if (tcpath) return tc_launch_sweep(true, eval, g, w, k, g.rows_split, st);
      return launch_row_sweep(in, k, w, g, M_ROWSUM, eval, st);
    case 1:
      return launch_row_fin(in, k, w, g, eval, st);
    case 2:
      if (tcpath) return tc_launch_sweep(false, eval, g, w, k, g.cols_split, st);
      return launch_col_sweep(in, k, w, g, eval, st);
    default:
      return launch_col_fin(in, k, w, g, eval, st);
  }
}

cudaError_t launch_iteration(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int prec,
                             int eval, cudaStream_t st) {
  for (int part = 0; part < 4; ++part) {
    cudaError_t e = launch_iteration_part(in, k, w, g, prec, part, eval, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int launches_per_iteration(const Consts& k, int prec) { return 4; }

template <int MODE, int DG>
static cudaError_t set_attr() {
  const int sm = (int)pts_smem(64, DG);
  return cudaFuncSetAttribute(k_pts_sweep<MODE, DG>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
}

// Raise the dynamic shared-memory limits of the sweeps that serve this problem, before any capture.
// The limits belong to the current device (and end with cudaDeviceReset), so every context sets those
// of its own kernels: a flag per process left the second device's launches without them.  The packed
// sweeps (d <= 8) and the stored-cost ones of this file need none.
cudaError_t prepare_kernels(const Consts& k, int prec) {
  if (k.kind != COST_SQEUCLID || prec == 1 /* LAMP_PREC_BF16_TC */ || uses_direct_sweeps(k, prec)) return cudaSuccess;
  if (k.zdot) return dot_prepare();
  for (const auto set : {set_attr<M_ROWSUM, 0>, set_attr<M_ROWSUM, 1>, set_attr<M_COLSUM, 0>, set_attr<M_COLSUM, 1>,
                         set_attr<M_MAX, 0>, set_attr<M_MAX2, 0>, set_attr<M_KMAX, 0>, set_attr<M_GRAD, 1>,
                         set_attr<M_GRAD, 2>, set_attr<M_GRAD, 3>, set_attr<M_GRAD, 4>, set_attr<M_GRAD, 5>,
                         set_attr<M_GRAD, 6>, set_attr<M_GRAD, 7>, set_attr<M_GRAD, 8>}) {
    const cudaError_t e = set();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int sweep_blocks_per_sm(const Consts& k, int prec, int which) {
  int nb = 0;
  if (k.kind == COST_DENSE) {
    // the splits decide how the float32 partial sums are grouped: they stay those of the tiles
    // below at two (rows) and three (columns) CTAs per SM, whatever the kernels' grids
    nb = which == 0 ? 2 : 3;
  } else if (uses_direct_sweeps(k, prec)) {
    nb = direct_blocks_per_sm();
  } else {
    // the splits of the dot form are those of two CTAs per SM too: they decide how the float32
    // partial sums are grouped, and its persistent sweep takes any number of them
    if (k.zdot) return 2;
    auto kern = which == 0 ? k_pts_sweep<M_ROWSUM, 0> : k_pts_sweep<M_COLSUM, 1>;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kThreads, pts_smem(k.d));
  }
  return nb > 0 ? nb : 1;
}

// fixed / streamed points per CTA of each sweep (the split choice of lamp_create uses them)
int tile_outer(const Consts& k, int prec) {
  if (prec == 1 /* LAMP_PREC_BF16_TC */) return tc_tile_fixed();
  return k.kind == COST_DENSE ? kDSplitRows : uses_direct_sweeps(k, prec) ? direct_outer(k.d) : kPT;
}
int tile_inner(const Consts& k, int prec) {
  if (prec == 1) return tc_tile_stream();
  return k.kind == COST_DENSE ? kDChunk : uses_direct_sweeps(k, prec) ? kDirectTile : kPT;
}
int tile_outer_cols(const Consts& k, int prec) {
  if (prec == 1) return tc_tile_fixed();
  return k.kind == COST_DENSE ? kDChunk : uses_direct_sweeps(k, prec) ? direct_outer(k.d) : kPT;
}
int tile_inner_cols(const Consts& k, int prec) {
  if (prec == 1) return tc_tile_stream();
  return k.kind == COST_DENSE ? kDColRows : uses_direct_sweeps(k, prec) ? kDirectTile : kPT;
}

// ------------------------------------------------------------------------------------------
// transport-map application (App. E, colour transfer): out = p V (side 0, V: m x k) or
// out = p^T U (side 1, U: n x k) for the current X^t = diag(r) p, 1 <= k <= 8

// out[i][q] = scale_i sum_s part[(s np + i) k + q], scale_i = src[i].y (/ div[i])
__global__ void k_map_fin(const double* __restrict__ part, int splits, int64_t np, int dk,
                          const float4* __restrict__ src, const double* __restrict__ div, float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  double sc = (double)src[i].y;
  if (div) sc /= div[i];
  for (int q = 0; q < dk; ++q) {
    double acc = 0.0;
    for (int s = 0; s < splits; ++s) acc += part[((int64_t)s * np + i) * dk + q];
    out[i * dk + q] = (float)(sc * acc);
  }
}

// inner weights of side 1: 1 / S_i = q_i / r_i, in the g2row layout
__global__ void k_map_rowweights(const float4* __restrict__ g2row, const double* __restrict__ r, int64_t n,
                                 float4* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float4 g = g2row[i];
  out[i] = make_float4(g.x, (float)((double)g.y / r[i]), g.z, g.w);
}

// stored cost, side 0: one warp per row, sum_j 2^{v_ij} w_j V_j, times q_i / r_i
template <int DK>
__global__ void __launch_bounds__(kThreads)
k_dense_map_rows(const float* __restrict__ C, int64_t ldc, int64_t n, int64_t m, const float4* __restrict__ colq,
                 const float4* __restrict__ g2row, const double* __restrict__ r, const float* __restrict__ V,
                 float* __restrict__ out, const DevState* __restrict__ dev, const Consts k) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
  if (i >= n) return;  // warp-uniform
  const SweepParams sp = make_sweep_params(sweep_kappa(dev->kappa, k), k);
  const float4 gr = g2row[i];
  const float* crow = C + i * ldc;
  double acc[DK];
#pragma unroll
  for (int q = 0; q < DK; ++q) acc[q] = 0.0;
  for (int64_t j0 = 0; j0 < m; j0 += 32 * 64) {
    float a[DK];
#pragma unroll
    for (int q = 0; q < DK; ++q) a[q] = 0.f;
    const int64_t j1 = j0 + 32 * 64 < m ? j0 + 32 * 64 : m;
    for (int64_t j = j0 + lane; j < j1; j += 32) {
      const float4 cd = colq[j];
      const float z = crow[j];
      const float v = __fmaf_rn(sp.alA, z, __fmaf_rn(sp.ahA, z, -(gr.x + cd.x)));
      const float e = ex2(v) * cd.y;
#pragma unroll
      for (int q = 0; q < DK; ++q) a[q] = __fmaf_rn(e, V[j * DK + q], a[q]);
    }
#pragma unroll
    for (int q = 0; q < DK; ++q) acc[q] += (double)a[q];
  }
  const double sc = (double)gr.y / r[i];
#pragma unroll
  for (int q = 0; q < DK; ++q) {
    double v = acc[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) out[i * DK + q] = (float)(sc * v);
  }
}

// stored cost, side 1: one thread per column, sum_i 2^{v_ij} U_i / S_i, times w_j
template <int DK>
__global__ void __launch_bounds__(kThreads)
k_dense_map_cols(const float* __restrict__ C, int64_t ldc, int64_t n, int64_t m, const float4* __restrict__ colq,
                 const float4* __restrict__ g2row, const double* __restrict__ r, const float* __restrict__ U,
                 float* __restrict__ out, const DevState* __restrict__ dev, const Consts k) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= m) return;
  const SweepParams sp = make_sweep_params(sweep_kappa(dev->kappa, k), k);
  const float4 cd = colq[j];
  double acc[DK];
#pragma unroll
  for (int q = 0; q < DK; ++q) acc[q] = 0.0;
  for (int64_t i0 = 0; i0 < n; i0 += 64) {
    float a[DK];
#pragma unroll
    for (int q = 0; q < DK; ++q) a[q] = 0.f;
    const int64_t i1 = i0 + 64 < n ? i0 + 64 : n;
    for (int64_t i = i0; i < i1; ++i) {
      const float4 gr = g2row[i];
      const float z = C[i * ldc + j];
      const float v = __fmaf_rn(sp.alA, z, __fmaf_rn(sp.ahA, z, -(gr.x + cd.x)));
      const float e = ex2(v) * (float)((double)gr.y / r[i]);
#pragma unroll
      for (int q = 0; q < DK; ++q) a[q] = __fmaf_rn(e, U[i * DK + q], a[q]);
    }
#pragma unroll
    for (int q = 0; q < DK; ++q) acc[q] += (double)a[q];
  }
#pragma unroll
  for (int q = 0; q < DK; ++q) out[j * DK + q] = (float)((double)cd.y * acc[q]);
}

template <int DK>
static cudaError_t launch_map_k(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int cur,
                                const float* V, float* out, int side, int splits, double* part, cudaStream_t st) {
  if (k.kind == COST_DENSE) {
    if (side == 0)
      k_dense_map_rows<DK><<<(unsigned)cdiv(k.n, kThreads / 32), kThreads, 0, st>>>(
          in.C, in.ldc, k.n, k.m, w.colq[cur], w.g2row, in.r, V, out, w.dev, k);
    else
      k_dense_map_cols<DK><<<(unsigned)cdiv(k.m, kThreads), kThreads, 0, st>>>(
          in.C, in.ldc, k.n, k.m, w.colq[cur], w.g2row, in.r, V, out, w.dev, k);
    return cudaGetLastError();
  }
  if (k.zdot) {
    const float4* inner = w.colq[cur];
    if (side == 1) {
      float4* rw = reinterpret_cast<float4*>(w.rowpart);
      k_map_rowweights<<<(unsigned)cdiv(k.n, 256), 256, 0, st>>>(w.g2row, in.r, k.n, rw);
      inner = rw;
    }
    const float4* outer = side == 0 ? w.g2row : w.colq[cur];
    const int64_t np = side == 0 ? k.n : k.m;
    cudaError_t e = dot_weighted(side == 0, w, k, 0, np, V, DK, outer, inner, splits, part, st);
    if (e != cudaSuccess) return e;
    k_map_fin<<<(unsigned)cdiv(np, 256), 256, 0, st>>>(part, splits, np, DK, outer, side == 0 ? in.r : nullptr, out);
    return cudaGetLastError();
  }
  if (side == 0) {
    // outer = rows (x), inner = columns (y): weights w_j of colq, outer offsets RqA of g2row
    SweepIO io;
    for (int b = 0; b < 2; ++b) { io.off2[b] = nullptr; io.off4[b] = w.g2row; io.indat[b] = w.colq[b]; }
    cudaError_t e = launch_pts<M_GRAD, DK>(in.x, in.y, k.n, k.m, k.d, io, w.rowpart, nullptr, g.rows_split, w.dev,
                                           k, st, V);
    if (e != cudaSuccess) return e;
    k_map_fin<<<(unsigned)cdiv(k.n, 256), 256, 0, st>>>(w.rowpart, g.rows_split, k.n, DK, w.g2row, in.r, out);
    return cudaGetLastError();
  }
  // outer = columns (y), inner = rows (x) with weights 1 / S_i (in rowpart, free here)
  float4* rw = reinterpret_cast<float4*>(w.rowpart);
  k_map_rowweights<<<(unsigned)cdiv(k.n, 256), 256, 0, st>>>(w.g2row, in.r, k.n, rw);
  SweepIO io;
  for (int b = 0; b < 2; ++b) { io.off2[b] = nullptr; io.off4[b] = w.colq[b]; io.indat[b] = rw; }
  cudaError_t e = launch_pts<M_GRAD, DK>(in.y, in.x, k.m, k.n, k.d, io, w.colpart, nullptr, g.cols_split, w.dev, k,
                                         st, V);
  if (e != cudaSuccess) return e;
  k_map_fin<<<(unsigned)cdiv(k.m, 256), 256, 0, st>>>(w.colpart, g.cols_split, k.m, DK, w.colq[cur], nullptr, out);
  return cudaGetLastError();
}

cudaError_t launch_map(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int cur, const float* V,
                       int dk, float* out, int side, int splits, double* part, cudaStream_t st) {
  switch (dk) {
    case 1: return launch_map_k<1>(in, k, w, g, cur, V, out, side, splits, part, st);
    case 2: return launch_map_k<2>(in, k, w, g, cur, V, out, side, splits, part, st);
    case 3: return launch_map_k<3>(in, k, w, g, cur, V, out, side, splits, part, st);
    case 4: return launch_map_k<4>(in, k, w, g, cur, V, out, side, splits, part, st);
    case 5: return launch_map_k<5>(in, k, w, g, cur, V, out, side, splits, part, st);
    case 6: return launch_map_k<6>(in, k, w, g, cur, V, out, side, splits, part, st);
    case 7: return launch_map_k<7>(in, k, w, g, cur, V, out, side, splits, part, st);
    case 8: return launch_map_k<8>(in, k, w, g, cur, V, out, side, splits, part, st);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace lamp
