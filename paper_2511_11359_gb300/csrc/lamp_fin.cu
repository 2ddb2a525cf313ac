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
// gain is kept per column, the row shift's log2 comes from a table, and the parameters of the
// next iteration are prepared by a block of RF instead of by CF's last thread.  RF + CF together,
// against one thread per point doing all of it in blocks of 128: 22.9 -> 12.0 us at 4096 points
// (16 splits), 37.5 -> 23.1 us at 2^15 (19 splits).  Divisions stay the correctly rounded ones: a
// quotient from a float32 seed and one Newton step takes 4 operations less, 0.1 to 0.2 us an
// iteration, but rounds the other way next to a tie.
#include <cmath>

#include "lamp_fin.cuh"

namespace lamp {

namespace {

constexpr int kPts = kFinPoints;      // points of a block
constexpr int kThreads = 2 * kPts;    // four warps, one per scheduler: two per stream
constexpr int kWarps = kPts / 32;     // warps per stream

// RF: row finalize of iteration t.  The warps of stream A give q^A; those of stream B q^B and the row shifts of iteration t + 1, where stream A has
// kappa_{t+1} (stream B here) and stream B is extrapolated linearly in t.  Block `rowblocks`
// prepares make_sweep_params of kappa_{t+2} for CF.  Evaluation passes have stream A alone, and
// the second warps form log Z.
template <bool EVAL>
__global__ void __launch_bounds__(kThreads)
k_row_fin(const Work w, int splits, const double* __restrict__ r, int rowblocks, const Consts k) {
  DevState* __restrict__ dev = w.dev;
  const int4 ctl = read_control(dev);
  if (ctl.y) return;  // done
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
  const int cur = ctl.x;
  const bool valid = i < k.n;
  double S = 0.0, ri = 0.0, snx = 0.0;
  float2 rq = make_float2(0.f, 0.f);
  SweepParams sp, spn;
  iteration_params_of(dev, k, sp, spn);
  if (valid) {
    rq = w.rowshift[cur][i];
    ri = r[i];
    if (k.zdot && (EVAL || !k.shared_shift)) snx = k.s * w.nx[i];
    // evaluation passes sweep stream A alone: one sum per split, read by both warps
    constexpr int na = EVAL ? 1 : 2;
    const double* __restrict__ part = w.rowpart + (int64_t)(EVAL ? 0 : role) * k.n + i;
    S = split_sum(part, (int64_t)na * k.n, splits);
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
      const float q = (float)(ri / S);
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
      const float q = (float)(ri / S);
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
  const int4 ctl = read_control(dev);
  if (ctl.y) return;  // done
  const int cur = ctl.x;
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
  // what the deciding thread needs, loaded with everything else instead of behind the last barrier
  const long long t = dev->t, tmax = dev->tmax;
  const double kappa = dev->kappa, tol = dev->tol;
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
    double a = split_sum(part, (int64_t)na * k.m, splits);
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
        const double thbar = (tA + thj) / fma(tA, thj, 1.0);  // M_{tau2}(theta^t; p^{eta_t}(nu^t))
        nun = nuj + sp.wB * (thbar - nuj);                             // nu^{t+1}
        snu[p] = nun;
        w.nu[cur ^ 1][j] = nun;
      }
    } else if (!EVAL) {
      // col(Xbar^{t+1})_j; under the shared row shift the column weight of stream B is
      // already inside the sweep's exponents
      const double B = k.shared_shift ? a : (double)cq.w * a;
      const double tB = tanh(gj * (B - cj));
      const double thhat = (tB + thj) / fma(tB, thj, 1.0);  // M_{tau2}(theta^t; p^{eta_{t+1}}(nubar^{t+1}))
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
      dev->t_eval = t;
      dev->kappa_eval = kappa;
    }
    if (ctl.z != 0 || !isfinite(R)) {  // status: RF has completed, and CF does not set it before this point
      if (ctl.z == 0) dev->status = 5;
      dev->done = 1;
    } else if (EVAL) {
      dev->done = 1;
    } else if ((t >= 1 && R <= tol && (k.eta == 0.0 || k.infeas_only || 1.0 - kappa * k.eta <= tol)) || t >= tmax) {
      dev->done = 1;
    } else {
      dev->t = t + 1;
      dev->kappa = sp.kapB;
      dev->cur = cur ^ 1;
      // the next iteration's parameters, once per iteration instead of once per thread
      // (make_sweep_params of kappa_{t+2} comes from RF)
      dev->spc = spn;
      dev->spn = dev->spq;
      dev->swf = sweep_floats(spn);
      dev->swf_kap = spn.kapA;
    }
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
