// Whole iterations of small low-dimensional problems (up to about 900 x 900 points, d <= 8, packed
// direct form) in one launch: a cluster of 16 CTAs keeps the state on chip and runs `passes` iterations of
// Alg. 2.
//
// What bounds a small problem is the chain of an iteration, not its entries (256 x 256: 0.02 us
// of exponentials): four launches, each with its own ramp, its loads of what the previous one
// stored, and in the last one a block that waits for all others.  Here CTA c owns n / 16 rows and
// m / 16 columns; every CTA holds the records of all points (coordinates, offsets, weights) in
// shared memory.  An iteration is
//   row sums of the own rows over all columns, their finalize, the rows' new records to all CTAs;
//   cluster barrier;
//   column sums of the own columns over all rows, the dual step, the columns' new records and the
//   residual's partial to all CTAs;
//   cluster barrier; every CTA adds the 16 partials and takes the same decision.
// The arithmetic is that of the four kernels (lamp_direct.cuh, lamp_fin.cuh): a thread evaluates
// one row (column) over a group of 64 points, the group sums are folded per split and the splits
// added in the same order, so the states are the same to the bit.  The residual is not: it is added
// per 1 / 16 of the columns here and per 64 columns there, so its last bits differ, and a tolerance
// that lies between the two values stops one iteration apart.
// n = m = 256, d = 2: 16.9 (graphs of the four kernels) -> 7.7 us per iteration: 2.1 us of sums, 3.9
// of finalize chains, 1.7 of exchanges.
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "lamp_direct.cuh"
#include "lamp_fin.cuh"

namespace lamp {

namespace {

constexpr int kCtas = 16;
constexpr int kThreads = 512;
constexpr int kMaxOwn = 64;                    // rows or columns of a CTA
constexpr int kMaxPoints = kCtas * kMaxOwn;
constexpr int kGroup = 2 * kDFold;             // points of a group (one float32 partial sum)

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address of this CTA's shared location p in CTA `cta` of the cluster
__device__ __forceinline__ uint32_t peer(const void* p, uint32_t cta) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(cta));
  return a;
}
__device__ __forceinline__ void peer_store4(uint32_t a, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ void peer_store_d(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void fin_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

struct Shape {
  int own_rows, own_cols;      // per CTA, even
  int groups_rows, groups_cols;  // groups of 64 points of all rows / columns
  int tps_rows, tps_cols;      // tiles (two groups) per split of the row / column sweep
};

// floats of the shared-memory layout (records, group sums; the small arrays are static)
template <int D>
constexpr size_t smem_floats(const Shape& s) {
  const size_t rec = (size_t)(s.groups_rows + s.groups_cols) * kDFold * DirectCfg<D>::REC;
  const size_t gr = (size_t)s.groups_cols * 2 * s.own_rows, gc = (size_t)s.groups_rows * 2 * s.own_cols;
  return rec + (gr > gc ? gr : gc);
}

constexpr int kMaxSmem = 128 * 1024;  // more than the largest shape takes
static_assert((2 * (kMaxPoints / kGroup) * kDFold * DirectCfg<8>::REC + (kMaxPoints / kGroup) * 2 * kMaxOwn) * 4 <= kMaxSmem,
              "shared memory of the largest shape");

// the group sums of `own` outer points (coordinates xs[own][D], offsets, dB) over all groups of
// the inner records: gs[(group * 2 + stream) * own + point]
template <int MODE, int D, int CK>
__device__ __forceinline__ void group_sums(const float* __restrict__ rec, int groups, const float* __restrict__ xs,
                                           const float* __restrict__ off, const float* __restrict__ dB, int own,
                                           const SweepF& sp, float* __restrict__ gs) {
  constexpr int REC = DirectCfg<D>::REC;
  const uint64_t ahA2 = pk(sp.ahA, sp.ahA), alA2 = pk(sp.alA, sp.alA), da2 = pk(sp.dal, sp.dal);
  for (int e = threadIdx.x; e < own * groups; e += kThreads) {
    const int g = e / own, p = e - g * own;
    uint64_t x2[D];
#pragma unroll
    for (int kk = 0; kk < D; ++kk) x2[kk] = pk(xs[p * D + kk], xs[p * D + kk]);
    const uint64_t o2 = pk(off[p], off[p]), d2 = MODE == M_COLSUM ? pk(dB[p], dB[p]) : 0ull;
    uint64_t acc[2] = {0ull, 0ull};
    const float* rp = rec + (size_t)g * kDFold * REC;
#pragma unroll 4
    for (int q = 0; q < kDFold; ++q) {
      DirectPair<D> t;
      t.load(rp + q * REC);
      direct_pair<MODE, D, 0, CK>(x2, o2, d2, t, ahA2, alA2, da2, acc);
    }
    const float2 a = upk(acc[0]), b = upk(acc[1]);
    gs[(2 * g) * own + p] = a.x + a.y;
    gs[(2 * g + 1) * own + p] = b.x + b.y;
  }
}

// one point's sum of one stream: the groups of a split folded as a float-float pair, the splits
// added in float64
__device__ __forceinline__ double fold_sums(const float* __restrict__ gs, int groups, int tps, int own, int stream,
                                            int p) {
  double S = 0.0;
  for (int g0 = 0; g0 < groups; g0 += 2 * tps) {
    float hi = 0.f, lo = 0.f;
    const int g1 = g0 + 2 * tps < groups ? g0 + 2 * tps : groups;
    for (int g = g0; g < g1; ++g) ff_add(hi, lo, gs[(2 * g + stream) * own + p]);
    S += (double)hi + (double)lo;
  }
  return S;
}

// records of all points: coordinates, and the pair data {-off, w}, {dB, w} of `pairs`
template <int D>
__device__ void load_records(float* __restrict__ rec, int groups, const float* __restrict__ P, int64_t np,
                             const float4* __restrict__ pairs) {
  constexpr int REC = DirectCfg<D>::REC, DP = DirectCfg<D>::DP;
  for (int e = threadIdx.x; e < groups * kGroup; e += kThreads) {
    float* r = rec + (e >> 1) * REC;
    for (int kk = 0; kk < DP; ++kk) r[2 * kk + (e & 1)] = e < np && kk < D ? P[(int64_t)e * D + kk] : 0.f;
  }
  for (int e = threadIdx.x; e < groups * kGroup; e += kThreads)
    *reinterpret_cast<float4*>(rec + (e >> 1) * REC + 2 * DP + 4 * (e & 1)) = pairs[e];
}

// the own points' staged pair data to the records of every CTA
template <int D>
__device__ __forceinline__ void push_records(float* rec, const float4* stage, int first, int own) {
  constexpr int REC = DirectCfg<D>::REC, DP = DirectCfg<D>::DP;
  for (int e = threadIdx.x; e < own * kCtas; e += kThreads) {
    const int cta = e / own, q = e - cta * own;  // q: pair q / 2, half q % 2
    peer_store4(peer(rec + (size_t)((first + q) >> 1) * REC + 2 * DP + 4 * (q & 1), (uint32_t)cta), stage[q]);
  }
}

template <int D, int CK>
__global__ void __launch_bounds__(kThreads, 1)
k_cluster_iterate(const Inputs in, const Work w, const Shape s, int64_t passes, const Consts k) {
  DevState* __restrict__ dev = w.dev;
  if (dev->done) return;  // uniform over the cluster: nothing writes it before the last barrier
  extern __shared__ __align__(16) float smem[];
  constexpr int REC = DirectCfg<D>::REC;
  float* crec = smem;                                                 // columns' records
  float* rrec = crec + (size_t)s.groups_cols * kDFold * REC;          // rows' records
  float* gs = rrec + (size_t)s.groups_rows * kDFold * REC;            // group sums
  __shared__ float xs[kMaxOwn * D], ys[kMaxOwn * D];                  // own points
  __shared__ float roff[kMaxOwn], coff[kMaxOwn], cw[kMaxOwn], cdB[kMaxOwn];  // -RqA; -BqA, wA, dB
  __shared__ float4 rstage[kMaxOwn], cstage[kMaxOwn];                 // pair data of the own rows, columns
  // residual partials of all CTAs, by parity of the iteration; the sign bit: a row sum out of range
  __shared__ double res[2][kCtas];
  __shared__ double snu[kMaxOwn], sq[kMaxOwn], srp[kMaxOwn];
  __shared__ LogEntry stab[128];
  __shared__ SweepParams sp[3];                                       // of kappa_t, kappa_{t+1}, kappa_{t+2}
  __shared__ SweepF sf;                                               // the sweeps' constants at kappa_t
  __shared__ int bad, verdict;                                        // 0 go on, 1 stop, 5 LAMP_E_NUMERIC

  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const uint32_t rank = cluster_rank();
  const int r0 = (int)rank * s.own_rows, c0 = (int)rank * s.own_cols;
  const int cur0 = dev->cur;
  const int status0 = dev->status;  // of an earlier call: the first decision is then to stop, as in k_col_fin
  const double tol = dev->tol;
  const long long tmax = dev->tmax;
  long long t = dev->t;
  double kap = dev->kappa;
  // the finalize steps are chains of float64 instructions, one every 64 cycles per scheduler: the
  // first eight warps share them out, warp w role w % 4 (its scheduler) of the points 32 (w / 4) + lane
  const int role = wid & 3, p = lane + 32 * (wid >> 2);
  const bool fin = wid < 8;
  const bool rok = fin && p < s.own_rows && r0 + p < k.n, cok = fin && p < s.own_cols && c0 + p < k.m;

  load_records<D>(crec, s.groups_cols, in.y, k.m, w.colq2[cur0]);
  load_records<D>(rrec, s.groups_rows, in.x, k.n, w.g2row2);
  if (tid < 128) stab[tid] = kLogTab[tid];
  if (tid == 0) {
    bad = 0;
    sp[0] = make_sweep_params(kap, k);
    sp[1] = make_sweep_params(sp[0].kapB, k);
    sf = sweep_floats(sp[0]);
  }
  for (int e = tid; e < kMaxOwn * D; e += kThreads) {
    const int q = e / D, kk = e - q * D;
    xs[e] = q < s.own_rows && r0 + q < k.n ? in.x[(int64_t)(r0 + q) * D + kk] : 0.f;
    ys[e] = q < s.own_cols && c0 + q < k.m ? in.y[(int64_t)(c0 + q) * D + kk] : 0.f;
  }
  for (int q = tid; q < kMaxOwn; q += kThreads) {
    roff[q] = q < s.own_rows && r0 + q < k.n ? -w.rowshift[cur0][r0 + q].x : 0.f;
    const bool ok = q < s.own_cols && c0 + q < k.m;
    const float4 cq = ok ? w.colq[cur0][c0 + q] : make_float4(0.f, 0.f, 0.f, 0.f);
    coff[q] = -cq.x;
    cw[q] = cq.y;
    cdB[q] = ok ? pair_dB(w.colq2[cur0], c0 + q) : 0.f;
  }
  // padding halves of the own points' pair data stay {-2^100, 0}
  for (int q = tid; q < kMaxOwn; q += kThreads) srp[q] = 0.0;
  for (int q = tid; q < kMaxOwn; q += kThreads)
    rstage[q] = cstage[q] = make_float4(-0x1p100f, -0x1p100f, 0.f, 0.f);
  // fields 0, 2, 4, 6: -off, wA, dB, wB
  float* fr = reinterpret_cast<float*>(rstage) + (p >> 1) * 8 + (p & 1);
  float* fc = reinterpret_cast<float*>(cstage) + (p >> 1) * 8 + (p & 1);
  const double ri = rok ? in.r[r0 + p] : 0.0;
  double nuj = 0.0, thj = 0.0, cj = 0.0, gj = 0.0, bB = 0.0;  // bB: BcolB of the own column (stream B's threads)
  if (cok) {
    nuj = w.nu[cur0][c0 + p];
    thj = w.theta[cur0][c0 + p];
    cj = in.c[c0 + p];
    gj = w.gj[c0 + p];
  }
  int applied = 0, done = 0;
  double R = 0.0;
  cluster_sync();  // every CTA has started and set up: its shared memory may be written

  for (int64_t it = 0; it < passes && !done; ++it) {
    const int par = (int)(it & 1);
    // ---- row sums and row finalize (k_row_fin) ----
    group_sums<M_ROWSUM, D, CK>(crec, s.groups_cols, xs, roff, nullptr, s.own_rows, sf, gs);
    __syncthreads();
    // roles: 0 q^A, 1 q^B, 2 the row shift of iteration t + 1
    float rnext = 0.f;
    if (rok && role < 3) {
      double S = fold_sums(gs, s.groups_cols, s.tps_rows, s.own_rows, role ? 1 : 0, p);
      if (!in_range(S)) {
        bad = 1;
        S = 1.0;
      }
      if (role == 2) {
        rnext = -(float)quantize_add((double)(-roff[p]) + log2_table(S, stab), sp[1].g);
      } else {
        const float q = (float)(ri / S);
        if (role == 0) {
          fr[0] = roff[p];
          fr[2] = q;
        } else {
          fr[4] = 0.f;
          fr[6] = q;
        }
      }
    }
    __syncthreads();
    push_records<D>(rrec, rstage, r0, s.own_rows);
    cluster_sync();
    // ---- column sums and dual step (k_col_fin) ----
    group_sums<M_COLSUM, D, CK>(rrec, s.groups_rows, ys, coff, cdB, s.own_cols, sf, gs);
    __syncthreads();
    // roles: 0 stream A (residual, nu^{t+1}, its column data), 1 stream B (theta^{t+1}, nubar^{t+2},
    // its column data), 2 the residual's sum, 3 the parameters of iteration t + 2
    double nun = 0.0, thn = 0.0, bBn = 0.0;
    if (fin) {
      if (cok && role < 2) {
        const double a = fold_sums(gs, s.groups_rows, s.tps_cols, s.own_cols, role, p);
        if (role == 0) {
          const double A = __dmul_rn((double)cw[p], a);  // rounded, as the column sum that k_col_fin stores
          srp[p] = fabs(A - cj);
          const double tA = tanh(gj * (A - cj));
          const double thbar = (tA + thj) / fma(tA, thj, 1.0);
          nun = nuj + sp[0].wB * (thbar - nuj);
          snu[p] = nun;
        } else {
          const double tB = tanh(gj * (a - cj));
          const double thhat = (tB + thj) / fma(tB, thj, 1.0);
          thn = fmin(fmax(thhat, -k.clipb), k.clipb);
        }
      } else if (tid == 3 * 32) {
        sp[2] = make_sweep_params(sp[1].kapB, k);
      }
      fin_bar();
      // column data of the state X^{t+1} would have
      if (cok && role == 0) {
        const double bA = sp[1].lamA * (2.0 * k.K * nun);
        const double qA = quantize_add(bA, sp[1].g);
        sq[p] = qA;
        fc[0] = -(float)qA;
        fc[2] = exp2f((float)(qA - bA));
      } else if (cok && role == 1) {
        nun = snu[p];
        bBn = sp[1].lamB * (2.0 * k.K * (nun + sp[1].wB * (thn - nun)));
        fc[6] = exp2f((float)(quantize_add(bBn, sp[1].g) - bBn));
      } else if (wid == 2) {
        const double rp = warp_sum_d(srp[lane] + srp[lane + 32]);
        if (lane < kCtas) peer_store_d(peer(&res[par][rank], (uint32_t)lane), bad ? -rp : rp);
      }
      fin_bar();
      if (cok && role == 1) fc[4] = (float)(sq[p] - bBn);
    }
    __syncthreads();
    push_records<D>(crec, cstage, c0, s.own_cols);
    cluster_sync();
    // ---- the decision, the same in every CTA: one warp's work, float64 is slow on this part ----
    if (wid == 0) {
      const double part = res[par][lane & (kCtas - 1)];
      const bool range = __any_sync(0xffffffffu, signbit(part));
      double v = fabs(part);
#pragma unroll
      for (int o = kCtas / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      R = v;
      if (lane == 0) {
        const bool rule = t >= 1 && v <= tol && (k.eta == 0.0 || k.infeas_only || 1.0 - kap * k.eta <= tol);
        verdict = range || !isfinite(v) ? 5 : status0 != 0 || rule || t >= tmax ? 1 : 0;
      }
    }
    __syncthreads();
    done = verdict != 0;
    if (!done) {
      ++t;
      ++applied;
      if (tid == 0) kap = sp[0].kapB;
      if (cok) {
        // both streams' threads keep (nu, theta) of their column
        if (role == 0) {
          coff[p] = fc[0];
          cw[p] = fc[2];
          cdB[p] = fc[4];
        } else if (role == 1) {
          sq[p] = thn;
          bB = bBn;
        }
      }
      if (rok && role == 2) roff[p] = rnext;
    }
    __syncthreads();
    if (!done) {
      if (cok) {
        nuj = snu[p];
        thj = sq[p];
      }
      if (tid == 0) {
        sp[0] = sp[1];
        sp[1] = sp[2];
        sf = sweep_floats(sp[0]);
      }
    }
    __syncthreads();
  }

  // ---- the state back to memory, in the buffers its parity names ----
  const int cur = cur0 ^ (applied & 1);
  if (applied > 0) {
    if (rok && role == 0) w.rowshift[cur][r0 + p] = make_float2(-roff[p], -roff[p]);
    if (cok && role == 0) {
      w.nu[cur][c0 + p] = nuj;
      w.theta[cur][c0 + p] = thj;
    } else if (cok && role == 1) {
      const int64_t j = c0 + p;
      const double qB = quantize_add(bB, sp[0].g);
      const float wB = exp2f((float)(qB - bB));
      w.colq[cur][j] = make_float4(-coff[p], cw[p], (float)qB, wB);
      store_pair_entry(w.colq2[cur], j, -coff[p], cw[p], cdB[p], wB);
    }
  }
  if (rank == 0 && tid == 0) {
    dev->t = t;
    dev->kappa = kap;
    dev->cur = cur;
    dev->res = R;
    dev->costA = dev->colnu = dev->rlogZ = NAN;  // what only evaluation passes compute
    if (done && verdict == 5 && dev->status == 0) dev->status = 5;
    if (done) dev->done = 1;
    dev->spc = sp[0];
    dev->spn = sp[1];
    dev->swf = sweep_floats(sp[0]);
    dev->swf_kap = sp[0].kapA;
  }
}

int even_share(int64_t np) { return (int)(((np + kCtas - 1) / kCtas + 1) / 2 * 2); }

Shape shape_of(const Consts& k, const Geometry& g) {
  const auto tps = [](int64_t np, int splits) {
    const int64_t tiles = (np + kDTile - 1) / kDTile;
    return (int)((tiles + splits - 1) / splits);
  };
  Shape s;
  s.own_rows = even_share(k.n);
  s.own_cols = even_share(k.m);
  s.groups_rows = (int)((k.n + kGroup - 1) / kGroup);
  s.groups_cols = (int)((k.m + kGroup - 1) / kGroup);
  s.tps_rows = tps(k.m, g.rows_split);  // the row sweep's splits are of the columns
  s.tps_cols = tps(k.n, g.cols_split);
  return s;
}

// f(std::integral_constant<int, d>, std::integral_constant<int, cost op>)
template <class F>
cudaError_t by_kind(const Consts& k, F&& f) {
  const auto cost = [&](auto d) {
    switch (k.cost_op) {
      case 0: return f(d, std::integral_constant<int, 0>{});
      case 1: return f(d, std::integral_constant<int, 1>{});
      default: return f(d, std::integral_constant<int, 2>{});
    }
  };
  switch (k.d) {
    case 1: return cost(std::integral_constant<int, 1>{});
    case 2: return cost(std::integral_constant<int, 2>{});
    case 3: return cost(std::integral_constant<int, 3>{});
    case 4: return cost(std::integral_constant<int, 4>{});
    case 5: return cost(std::integral_constant<int, 5>{});
    case 6: return cost(std::integral_constant<int, 6>{});
    case 7: return cost(std::integral_constant<int, 7>{});
    case 8: return cost(std::integral_constant<int, 8>{});
    default: return cudaErrorNotSupported;
  }
}

template <int D>
cudaLaunchConfig_t config(const Shape& s, cudaLaunchAttribute& at, cudaStream_t st) {
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = kCtas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(kCtas);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem_floats<D>(s) * sizeof(float);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cfg;
}

}  // namespace

bool cluster_serves(const Consts& k, const Geometry& g) {
  if (!k.shared_shift || k.zdot || k.kind != COST_SQEUCLID || k.d < 1 || k.d > 8) return false;
  if (k.n > kMaxPoints || k.m > kMaxPoints) return false;
  // 16 SMs against 152: above this many FMA-pipe operations a sweep takes longer here than the four
  // kernels' ramps (us per iteration here | there: d = 3, 700 points 14.8 | 20.1, 850 18.5 | 20.2,
  // 1000 21.1 | 18.5; d = 8, 700 18.0 | 20.8, 1000 27.0 | 20.5)
  if ((double)k.n * (double)k.m * (2 * k.d + 7) > 1.1e7) return false;
  const Shape s = shape_of(k, g);
  const cudaError_t e = by_kind(k, [&](auto dd, auto ck) {
    constexpr int D = decltype(dd)::value, CK = decltype(ck)::value;
    const auto kern = k_cluster_iterate<D, CK>;
    cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (r != cudaSuccess) return r;
    // a cluster of 16 needs that many free SMs in one GPC
    cudaLaunchAttribute at{};
    cudaLaunchConfig_t cfg = config<D>(s, at, nullptr);
    int clusters = 0;
    r = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
    return r == cudaSuccess && clusters < 1 ? cudaErrorNotSupported : r;
  });
  if (e != cudaSuccess) (void)cudaGetLastError();  // not served: the four kernels run instead
  return e == cudaSuccess;
}

cudaError_t launch_cluster(const Inputs& in, const Consts& k, const Work& w, const Geometry& g, int64_t passes,
                           cudaStream_t st) {
  const Shape s = shape_of(k, g);
  return by_kind(k, [&](auto dd, auto ck) {
    constexpr int D = decltype(dd)::value, CK = decltype(ck)::value;
    cudaLaunchAttribute at{};
    cudaLaunchConfig_t cfg = config<D>(s, at, st);
    return cudaLaunchKernelEx(&cfg, k_cluster_iterate<D, CK>, in, w, s, passes, k);
  });
}

}  // namespace lamp
