// Packed direct-form sweeps for grids that would leave SMs idle: the arithmetic of
// lamp_direct.cu, spread over more warps.
//
// lamp_direct.cu gives a CTA 1024 (d <= 4) or 512 outer points and a whole inner split, so that
// a problem of a few thousand points is a few dozen CTAs of 8 warps (n = m = 8192, d = 3: 128
// CTAs for 152 SMs; n = m = 256: 2).  Here a warp owns 32 R outer points, and the groups of 64
// inner points of a split, whose float32 sums the other kernel folds one after the other, are
// dealt to the CTA's four warps; the group sums meet in shared memory and are folded there in
// the same order, so the results are the same to the bit.  The whole split's records are staged
// at once (at most kMaxTiles tiles), one exposed copy per CTA.
// n = m = 8192, d = 3: 41 -> 37 us per sweep; n = m = 256, d = 2: 9.5 -> 3.7 us.
#include <cmath>
#include <cstdint>

#include "lamp_direct.cuh"

namespace lamp {

namespace {

constexpr int kMaxTiles = 8;  // tiles of a split: 16 groups

inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

template <int MODE, int D, int EV, int CK, int R>
__global__ void __launch_bounds__(128, R == 1 ? 5 : 4)
k_direct_small(const float* __restrict__ P_out, const float* __restrict__ P_in, int64_t n_out, int64_t n_in,
               const Work w, double* __restrict__ part, int tiles_per_split, const Consts k) {
  using C = DirectCfg<D>;
  constexpr int REC = C::REC;
  constexpr int NACC = kDirectSums<MODE, EV>;
  constexpr int kPts = 32 * R;
  const DevState* __restrict__ dev = w.dev;
  const int4 ctl = read_control(dev);
  if (ctl.y) return;  // done
  const int cur = ctl.x;
  const float4* __restrict__ pairs = MODE == M_ROWSUM ? w.colq2[cur] : w.g2row2;
  extern __shared__ __align__(16) float smem[];
  float* rec = smem;                                                   // [tiles][64 pairs][REC]
  float* gs = smem + (size_t)tiles_per_split * kDPairs * REC;          // [groups][NACC][kPts]
  const int tid = threadIdx.x, nthreads = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = nthreads >> 5;
  const int64_t o0 = (int64_t)blockIdx.x * kPts;
  const int split = blockIdx.y;
  const int64_t ntiles = (n_in + kDTile - 1) / kDTile;
  const int64_t it0 = (int64_t)split * tiles_per_split;
  const int64_t it1 = it0 + tiles_per_split < ntiles ? it0 + tiles_per_split : ntiles;
  const int tiles = it1 > it0 ? (int)(it1 - it0) : 0;  // 0: an empty split writes zeros
  for (int t = 0; t < tiles; ++t) direct_stage<D>(rec + t * kDPairs * REC, P_in, n_in, pairs, it0 + t, tid, nthreads);
  cp_async_commit();
  if (C::DP > D)  // the padding coordinate of odd d is read by the 16-byte loads, never used
    for (int p = tid; p < tiles * kDPairs; p += nthreads) rec[p * REC + 2 * D] = rec[p * REC + 2 * D + 1] = 0.f;

  const SweepF sp = sweep_floats_of(dev, k);
  const uint64_t ahA2 = pk(sp.ahA, sp.ahA), alA2 = pk(sp.alA, sp.alA), da2 = pk(sp.dal, sp.dal);
  uint64_t x2[R][D], ownA[R], ownD[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    int64_t go = o0 + lane + 32 * r;
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
      db = pair_dB(w.colq2[cur], go);
    }
    ownA[r] = pk(-qa, -qa);
    ownD[r] = pk(db, db);
  }
  cp_async_wait<0>();
  __syncthreads();

  const int groups = tiles * (kDPairs / kDFold);
  for (int g = warp; g < groups; g += nwarps) {
    uint64_t acc[R][NACC];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int q = 0; q < NACC; ++q) acc[r][q] = 0ull;
    const float* rp = rec + (size_t)g * kDFold * REC;
    // 40.5 -> 38.5 us at 8192 points against an unroll of 2
#pragma unroll 4
    for (int p = 0; p < kDFold; ++p) {
      DirectPair<D> t;
      t.load(rp + p * REC);
#pragma unroll
      for (int r = 0; r < R; ++r)
        direct_pair<MODE, D, EV, CK>(x2[r], ownA[r], ownD[r], t, ahA2, alA2, da2, acc[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int q = 0; q < NACC; ++q) {
        const float2 s = upk(acc[r][q]);
        gs[(g * NACC + q) * kPts + 32 * r + lane] = s.x + s.y;
      }
  }
  __syncthreads();
  for (int e = tid; e < kPts * NACC; e += nthreads) {
    const int q = e / kPts, p = e - q * kPts;
    float hi = 0.f, lo = 0.f;
    for (int g = 0; g < groups; ++g) ff_add(hi, lo, gs[(g * NACC + q) * kPts + p]);
    if (o0 + p < n_out) part[((int64_t)split * NACC + q) * n_out + o0 + p] = (double)hi + (double)lo;
  }
}

struct Launch {
  const float* Pout;
  const float* Pin;
  int64_t nout, nin;
  double* part;
  int splits, tps;
  bool wide;  // R = 4 (d <= 4) or 2 outer points per lane, else 1
};

template <int MODE, int D, int EV, int CK, int R>
cudaError_t go(const Launch& l, const Work& w, const Consts& k, cudaStream_t st) {
  constexpr int NACC = kDirectSums<MODE, EV>;
  const int groups = l.tps * (kDPairs / kDFold);
  const unsigned threads = 32u * (unsigned)(groups < 4 ? groups : 4);
  const size_t smem = ((size_t)l.tps * kDPairs * DirectCfg<D>::REC + (size_t)groups * NACC * 32 * R) * sizeof(float);
  static_assert(((size_t)kMaxTiles * kDPairs * DirectCfg<8>::REC + (size_t)2 * kMaxTiles * 2 * 128) * 4 <= 100 * 1024, "");
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_direct_small<MODE, D, EV, CK, R>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    if (e != cudaSuccess) return e;
  }
  return launch_kernel(k_direct_small<MODE, D, EV, CK, R>, dim3((unsigned)cdiv(l.nout, 32 * R), (unsigned)l.splits), threads,
                    smem, st, l.Pout, l.Pin, l.nout, l.nin, w, l.part, l.tps, k);
}

template <int MODE, int D, int EV>
cudaError_t go_cost(const Launch& l, const Work& w, const Consts& k, cudaStream_t st) {
  constexpr int RW = DirectCfg<D>::R;
  switch (k.cost_op) {
    case 0: return l.wide ? go<MODE, D, EV, 0, RW>(l, w, k, st) : go<MODE, D, EV, 0, 1>(l, w, k, st);
    case 1: return l.wide ? go<MODE, D, EV, 1, RW>(l, w, k, st) : go<MODE, D, EV, 1, 1>(l, w, k, st);
    case 2: return l.wide ? go<MODE, D, EV, 2, RW>(l, w, k, st) : go<MODE, D, EV, 2, 1>(l, w, k, st);
    default: return cudaErrorNotSupported;
  }
}

template <int MODE, int EV>
cudaError_t go_dim(const Launch& l, const Work& w, const Consts& k, cudaStream_t st) {
  switch (k.d) {
    case 1: return go_cost<MODE, 1, EV>(l, w, k, st);
    case 2: return go_cost<MODE, 2, EV>(l, w, k, st);
    case 3: return go_cost<MODE, 3, EV>(l, w, k, st);
    case 4: return go_cost<MODE, 4, EV>(l, w, k, st);
    case 5: return go_cost<MODE, 5, EV>(l, w, k, st);
    case 6: return go_cost<MODE, 6, EV>(l, w, k, st);
    case 7: return go_cost<MODE, 7, EV>(l, w, k, st);
    case 8: return go_cost<MODE, 8, EV>(l, w, k, st);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace

bool direct_small_serves(int64_t nout, int64_t nin, int d, int splits, int sms) {
  // the other kernel's grid is less than one wave of two CTAs per SM, and a split's records and
  // group sums fit shared memory
  const int tps = (int)cdiv(cdiv(nin, kDTile), splits);
  return cdiv(nout, direct_outer(d)) * splits < 2 * (int64_t)sms && tps <= kMaxTiles;
}

cudaError_t launch_direct_small(bool rows, int eval, const Inputs& in, const Consts& k, const Work& w,
                                const Geometry& g, cudaStream_t st) {
  Launch l{};
  l.Pout = rows ? in.x : in.y;
  l.Pin = rows ? in.y : in.x;
  l.nout = rows ? k.n : k.m;
  l.nin = rows ? k.m : k.n;
  l.part = rows ? w.rowpart : w.colpart;
  l.splits = rows ? g.rows_split : g.cols_split;
  l.tps = (int)cdiv(cdiv(l.nin, kDTile), l.splits);
  // several outer points per lane share each record load (a 16-byte broadcast load fills the
  // same 512 bytes of registers as any other): the wide form once it gives two CTAs per SM
  l.wide = cdiv(l.nout, 32 * (k.d <= 4 ? 4 : 2)) * l.splits >= 2 * (int64_t)g.sms;
  if (rows && eval) return go_dim<M_ROWSUM, 1>(l, w, k, st);
  if (rows) return go_dim<M_ROWSUM, 0>(l, w, k, st);
  if (eval) return go_dim<M_COLSUM, 1>(l, w, k, st);
  return go_dim<M_COLSUM, 0>(l, w, k, st);
}

}  // namespace lamp
