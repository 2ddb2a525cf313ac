// Packed f32x2 direct-form sweeps of the LAMP hot path (arXiv 2511.11359, Alg. 2,
// Section 4.1) for on-the-fly costs of low-dimensional point clouds (d <= 8): the row
// sweep G1 and the column sweep G2 of both streams, for the ground costs |x - y|^2,
// |x - y|_1 and |x - y|_inf (App. E.2 compares LAMP under all three).  See lamp_common.cuh for the
// compensated exponent and the shared row shift.
#include <cmath>
#include <cstdint>

#include "lamp_direct.cuh"

namespace lamp {

namespace {

constexpr int kThreads = 256;

inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// ------------------------------------------------------------------------------------------
// direct-form sweeps over point clouds with d <= 8 (LAMP_COST_SQEUCLID, float32, packed f32x2)
//
// Each thread owns kR(D) outer points o0 + tid + 256 r for the CTA's lifetime and
// keeps their coordinates and exponent offsets in registers as duplicated pairs
// (x, x).  The CTA streams the inner points through shared memory in tiles of 128
// (64 pairs, double-buffered with cp.async) and all threads read the same inner
// pair at the same time (broadcast loads), so one f32x2 instruction serves the two
// entries (outer, 2p) and (outer, 2p + 1).  Per pair of entries: d subtractions
// and d multiply-adds for z = |x - y|^2; stream A one add, two fma (compensated
// exponent), two ex2 and one fma (weighted sum); stream B, through the shared row
// shift (see lamp_common.cuh), one add, one fma, two ex2 and one add (row sums) or
// fma (column sums).  Evaluation
// passes also accumulate sum_i z_ij X_ij in the column sweep (two more).
// z = sum_k (x_k - y_k)^2 is accumulated in the same k order in both sweeps, and
// (y - x)^2 == (x - y)^2 in IEEE arithmetic, so the row and the column sweep see
// bit-identical exponents.  The inner data are the packed-pair arrays (see Work).

// MODE = M_ROWSUM or M_COLSUM; EV = 1: an evaluation pass (stream A alone, see direct_pair), else 0;
// CK = the ground cost (Consts::cost_op): 0 |x - y|^2, 1 l1, 2 l-inf
template <int MODE, int D, int EV, int CK>
__global__ void __launch_bounds__(kThreads, 2)
k_pts_direct(const float* __restrict__ P_out, const float* __restrict__ P_in, int64_t n_out, int64_t n_in,
             const Work w, double* __restrict__ part, int tiles_per_split, const Consts k) {
  using C = DirectCfg<D>;
  constexpr int R = C::R, DP = C::DP, REC = C::REC;
  constexpr int NACC = kDirectSums<MODE, EV>;
  const DevState* __restrict__ dev = w.dev;
  const int4 ctl = read_control(dev);
  if (ctl.y) return;  // done
  const int cur = ctl.x;
  // row sweep: inner = columns (colq2 of the current state); column sweep: inner = rows (g2row2)
  const float4* __restrict__ pairs = MODE == M_ROWSUM ? w.colq2[cur] : w.g2row2;
  __shared__ __align__(16) float srec[2][kDPairs * REC];

  const int tid = threadIdx.x;
  const int64_t o0 = (int64_t)blockIdx.x * kThreads * R;
  const int split = blockIdx.y;
  const int64_t ntiles = (n_in + kDTile - 1) / kDTile;
  const int64_t it0 = (int64_t)split * tiles_per_split;
  const int64_t it1 = it0 + tiles_per_split < ntiles ? it0 + tiles_per_split : ntiles;

  if (it0 < it1) direct_stage<D>(srec[0], P_in, n_in, pairs, it0, tid, kThreads);
  cp_async_commit();
  if (DP > D) {  // the padding coordinate of odd d is read by the 16-byte loads, never used
    for (int p = tid; p < 2 * kDPairs; p += kThreads) {
      srec[p / kDPairs][(p % kDPairs) * REC + 2 * D] = 0.f;
      srec[p / kDPairs][(p % kDPairs) * REC + 2 * D + 1] = 0.f;
    }
  }

  const SweepF sp = sweep_floats_of(dev, k);
  const uint64_t ahA2 = pk(sp.ahA, sp.ahA), alA2 = pk(sp.alA, sp.alA);
  const float dal = sp.dal;  // a^B - a^A
  const uint64_t da2 = pk(dal, dal);

  // own offsets: -RqA_i (row sweep), or -BqA_j and dB_j = BqA_j - BqB_j (column sweep)
  uint64_t x2[R][D], ownA[R], ownD[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    int64_t go = o0 + tid + (int64_t)kThreads * r;
    if (go >= n_out) go = n_out - 1;
#pragma unroll
    for (int kk = 0; kk < D; ++kk) {
      const float v = P_out[go * D + kk];
      x2[r][kk] = pk(v, v);
    }
    float qa, db = 0.f;
    if (MODE == M_ROWSUM) {
      qa = w.rowshift[cur][go].x;
    } else {
      qa = w.colq[cur][go].x;
      db = pair_dB(w.colq2[cur], go);  // the same float the row sweep reads for this column
    }
    ownA[r] = pk(-qa, -qa);
    ownD[r] = pk(db, db);
  }

  float hi[R][NACC], lo[R][NACC];
  uint64_t acc[R][NACC];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int q = 0; q < NACC; ++q) {
      hi[r][q] = 0.f;
      lo[r][q] = 0.f;
      acc[r][q] = 0ull;  // (+0, +0)
    }

  for (int64_t it = it0; it < it1; ++it) {
    const int buf = (int)((it - it0) & 1);
    if (it + 1 < it1) direct_stage<D>(srec[buf ^ 1], P_in, n_in, pairs, it + 1, tid, kThreads);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    const float* rec = srec[buf];
#pragma unroll 1
    for (int p0 = 0; p0 < kDPairs; p0 += kDFold) {
      // unrolled, because the FMA pipe waited on the record loads: by 8, or by 4 where 8 made the
      // kernel spill (d <= 2) or lengthened it (d = 5).  2^17 points, rows / columns, ms, unrolled by
      // 2, 4, 8: d = 1 5.64 / 6.07, 5.46 / 5.68, 5.51 / 5.73; d = 3 7.58 / 7.88, 7.36 / 7.58, 7.31 /
      // 7.50; d = 5 9.39 / 10.14, 9.32 / 9.54, 9.44 / 9.67; d = 8 12.01 / 12.37, 11.83 / 11.99,
      // 11.81 / 12.12; l1 and l-inf alike
      constexpr int U = D <= 2 || D == 5 ? 4 : 8;
#pragma unroll U
      for (int p = p0; p < p0 + kDFold; ++p) {
        DirectPair<D> t;
        t.load(rec + p * REC);
#pragma unroll
        for (int r = 0; r < R; ++r)
          direct_pair<MODE, D, EV, CK>(x2[r], ownA[r], ownD[r], t, ahA2, alA2, da2, acc[r]);
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int q = 0; q < NACC; ++q) {
          const float2 s = upk(acc[r][q]);
          ff_add(hi[r][q], lo[r][q], s.x + s.y);
          acc[r][q] = 0ull;
        }
    }
    __syncthreads();  // every thread is done with srec[buf] before it is refilled
  }
  cp_async_wait<0>();

#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t go = o0 + tid + (int64_t)kThreads * r;
    if (go >= n_out) continue;
#pragma unroll
    for (int q = 0; q < NACC; ++q) part[((int64_t)split * NACC + q) * n_out + go] = (double)hi[r][q] + (double)lo[r][q];
  }
}

template <int MODE, int D, int EV, int CK>
static cudaError_t launch_direct_d(const float* Pout, const float* Pin, int64_t nout, int64_t nin, const Work& w,
                                   double* part, int splits, const Consts& k, cudaStream_t st) {
  int64_t tin = cdiv(nin, kDTile);
  int tps = (int)cdiv(tin, splits);
  dim3 grid((unsigned)cdiv(nout, kThreads * DirectCfg<D>::R), (unsigned)splits);
  return launch_kernel(k_pts_direct<MODE, D, EV, CK>, grid, kThreads, 0, st, Pout, Pin, nout, nin, w, part, tps, k);
}

template <int MODE, int EV, int CK>
static cudaError_t launch_direct_ck(const float* Pout, const float* Pin, int64_t nout, int64_t nin, const Work& w,
                                    double* part, int splits, const Consts& k, cudaStream_t st) {
  switch (k.d) {
    case 1: return launch_direct_d<MODE, 1, EV, CK>(Pout, Pin, nout, nin, w, part, splits, k, st);
    case 2: return launch_direct_d<MODE, 2, EV, CK>(Pout, Pin, nout, nin, w, part, splits, k, st);
    case 3: return launch_direct_d<MODE, 3, EV, CK>(Pout, Pin, nout, nin, w, part, splits, k, st);
    case 4: return launch_direct_d<MODE, 4, EV, CK>(Pout, Pin, nout, nin, w, part, splits, k, st);
    case 5: return launch_direct_d<MODE, 5, EV, CK>(Pout, Pin, nout, nin, w, part, splits, k, st);
    case 6: return launch_direct_d<MODE, 6, EV, CK>(Pout, Pin, nout, nin, w, part, splits, k, st);
    case 7: return launch_direct_d<MODE, 7, EV, CK>(Pout, Pin, nout, nin, w, part, splits, k, st);
    case 8: return launch_direct_d<MODE, 8, EV, CK>(Pout, Pin, nout, nin, w, part, splits, k, st);
    default: return cudaErrorNotSupported;
  }
}

template <int MODE, int EV>
static cudaError_t launch_direct(const float* Pout, const float* Pin, int64_t nout, int64_t nin, const Work& w,
                                 double* part, int splits, const Consts& k, cudaStream_t st) {
  switch (k.cost_op) {
    case 0: return launch_direct_ck<MODE, EV, 0>(Pout, Pin, nout, nin, w, part, splits, k, st);
    case 1: return launch_direct_ck<MODE, EV, 1>(Pout, Pin, nout, nin, w, part, splits, k, st);
    case 2: return launch_direct_ck<MODE, EV, 2>(Pout, Pin, nout, nin, w, part, splits, k, st);
    default: return cudaErrorNotSupported;
  }
}


}  // namespace

int direct_outer(int d) { return kThreads * (d <= 4 ? DirectCfg<4>::R : DirectCfg<8>::R); }

int direct_blocks_per_sm() {
  // two CTAs per SM (__launch_bounds__ of every instantiation); a constant, because the splits that
  // follow from it decide how the float32 partial sums are grouped
  return 2;
}

cudaError_t launch_direct_sweep(bool rows, int eval, const Inputs& in, const Consts& k, const Work& w,
                                const Geometry& g, cudaStream_t st) {
  if (direct_small_serves(rows ? k.n : k.m, rows ? k.m : k.n, k.d, rows ? g.rows_split : g.cols_split, g.sms))
    return launch_direct_small(rows, eval, in, k, w, g, st);
  if (rows && eval) return launch_direct<M_ROWSUM, 1>(in.x, in.y, k.n, k.m, w, w.rowpart, g.rows_split, k, st);
  if (rows) return launch_direct<M_ROWSUM, 0>(in.x, in.y, k.n, k.m, w, w.rowpart, g.rows_split, k, st);
  if (eval) return launch_direct<M_COLSUM, 1>(in.y, in.x, k.m, k.n, w, w.colpart, g.cols_split, k, st);
  return launch_direct<M_COLSUM, 0>(in.y, in.x, k.m, k.n, w, w.colpart, g.cols_split, k, st);
}

}  // namespace lamp
