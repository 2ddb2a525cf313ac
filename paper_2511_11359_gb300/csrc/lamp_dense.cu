// Stored-cost sweeps fed by TMA: the row sweep G1 and the column sweep G2 of Alg. 2 over a
// dense float32 cost C (n x m, row-major, leading dimension ldc), one pass per sweep with
// both streams A (kappa_t, nu^t) and B (kappa_{t+1}, nubar^{t+1}) (Section 4.1).
//
// One producer warp streams 32-row x 256-column tiles of C (2-D tensor copies, 32 KB)
// together with the per-point data of the tile (G1: the 256 columns' {BqA, wA, BqB, wB};
// G2: the 32 rows' packed pairs, plain bulk copies) through a 3-stage shared-memory
// ring; eight consumer warps evaluate the compensated exponents of both streams, two entries at
// a time (f32x2: issue slots bound a sweep whose C is in the L2; 4096 x 4096: 15.5 -> 13.7 us
// rows, 15.1 -> 14.5 us columns; 16384 x 16384: 178 / 193 -> 166 / 165 us, 96 % of the measured
// copy rate), and their ex2 in float32 and accumulate:
//   G1: warp w owns rows 4w .. 4w + 3 of the CTA's 32-row block, lane l the columns
//       l + 32 q (q < 8) of each tile; per-row float-float sums, one warp reduction at the
//       end, partials per column split;
//   G2: warp w owns the 32 columns 32 w .. 32 w + 31 of the CTA's 256-column block (one
//       per lane) and walks the 32 rows of each tile; partials per row split.
// The exponent of entry (i, j) is formed from the same operands in the same order in both
// sweeps, so G2 sums exactly the entries that G1 normalised.  Every wait is bounded
// (lamp_async.cuh).
#include <cuda.h>

#include <cmath>
#include <cstdint>

#include "lamp_async.cuh"
#include "lamp_common.cuh"

namespace lamp {

namespace dense {

constexpr int kTR = 32;                                  // rows of a tile
constexpr int kTC = 256;                                 // columns of a tile (TMA box inner extent)
constexpr int kStages = 3;
constexpr int kTileBytes = kTR * kTC * 4;                // 32 KiB
constexpr int kAuxMax = kTC;                             // float4 per-point data per stage (G1: 256)
constexpr int kConsumerWarps = 8;
constexpr int kConsumers = kConsumerWarps * 32;
constexpr int kProducerWarp = kConsumerWarps;
constexpr int kThreads = kConsumers + 32;
static_assert(kConsumerWarps * 4 == kTR && kConsumerWarps * 32 == kTC, "warp / tile layout");

struct __align__(8) Bars {
  uint64_t full[kStages];
  uint64_t empty[kStages];
  int err;
};

// tiles, per-point data, barriers, and slack to align the dynamic buffer to 128 bytes
constexpr size_t kSmemBytes = (size_t)kStages * kTileBytes + (size_t)kStages * kAuxMax * sizeof(float4) + 128 + 128;

// WC = 1: an evaluation pass (stream A alone; the column sums also weighted by the cost)
// MX (row sweeps): 0 sums; 1 row maxima of both streams' exponents without row shift (the prime
// pass); 2 of stream A's with the row shifts and the column remainders subtracted (launch_dual)
template <bool ROWS, int WC, int MX = 0>
__global__ void __launch_bounds__(kThreads, 2)
k_dense_tma(const __grid_constant__ CUtensorMap map_c, const Work w, int64_t n, int64_t m, int tiles_per_split,
            const Consts k) {
  DevState* __restrict__ dev = w.dev;
  const int4 ctl = read_control(dev);
  if (MX == 0 && ctl.y) return;  // done
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  float* sC = reinterpret_cast<float*>(smem);                                    // kStages x kTR x kTC
  float4* sAux = reinterpret_cast<float4*>(smem + (size_t)kStages * kTileBytes);  // kStages x kAuxMax
  Bars* B = reinterpret_cast<Bars*>(smem + (size_t)kStages * kTileBytes + (size_t)kStages * kAuxMax * 16);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int cur = ctl.x;
  const int64_t ntiles_all = ROWS ? (m + kTC - 1) / kTC : (n + kTR - 1) / kTR;
  const int64_t it0 = (int64_t)blockIdx.y * tiles_per_split;
  int64_t it1 = it0 + tiles_per_split;
  if (it1 > ntiles_all) it1 = ntiles_all;
  const int ntiles = it1 > it0 ? (int)(it1 - it0) : 0;
  constexpr int kAux = ROWS ? kTC : kTR;  // per-point data entries per tile

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      async::mbar_init(&B->full[s], 1);
      async::mbar_init(&B->empty[s], kConsumers);
    }
    B->err = 0;
    async::mbar_init_fence();
  }
  __syncthreads();

  if (warp == kProducerWarp) {
    if (lane == 0) {
      const float4* __restrict__ aux_src = ROWS ? w.colq[cur] : w.g2row2;
      int issued = 0;
      for (int i = 0; i < ntiles; ++i) {
        const int s = i % kStages;
        if (i >= kStages && !async::mbar_wait(&B->empty[s], ((i / kStages) & 1) ^ 1, &B->err, dev)) break;
        const int64_t t = it0 + i;
        async::mbar_expect_tx(&B->full[s], kTileBytes + kAux * (uint32_t)sizeof(float4));
        if (ROWS) {
          async::tma_load_2d(sC + (size_t)s * kTR * kTC, &map_c, &B->full[s], (int)(t * kTC), (int)(blockIdx.x * kTR));
        } else {
          async::tma_load_2d(sC + (size_t)s * kTR * kTC, &map_c, &B->full[s], (int)(blockIdx.x * kTC), (int)(t * kTR));
        }
        // the per-point arrays are padded (columns to whole 256-column tiles, rows to
        // whole 128-row units) with entries whose offsets are +inf and weights 0, so the
        // entries past the end of C (read as 0 by the tensor copy) contribute 0
        async::bulk_load(sAux + (size_t)s * kAuxMax, aux_src + t * kAux, kAux * (uint32_t)sizeof(float4), &B->full[s]);
        issued = i + 1;
      }
      if (*(volatile int*)&B->err) {
        // error: let this thread's copies in flight land before the CTA exits
        for (int i = issued - kStages < 0 ? 0 : issued - kStages; i < issued; ++i)
          async::mbar_drain(&B->full[i % kStages], (i / kStages) & 1);
      }
    }
  } else {
    const SweepF sp = sweep_floats_of(dev, k);
    const uint64_t ahA2 = pk(sp.ahA, sp.ahA), alA2 = pk(sp.alA, sp.alA);
    const uint64_t ahB2 = pk(sp.ahB, sp.ahB), alB2 = pk(sp.alB, sp.alB);
    if (ROWS) {
      // ---------------- G1: rows 4 warp .. 4 warp + 3 of this row block ----------------
      const int64_t g0 = (int64_t)blockIdx.x * kTR + 4 * warp;
      uint64_t oA2[4], oB2[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float2 q = MX == 1 ? make_float2(0.f, 0.f) : w.rowshift[cur][g0 + a < n ? g0 + a : n - 1];
        oA2[a] = pk(-q.x, -q.x);
        oB2[a] = pk(-q.y, -q.y);
      }
      float hi[8], lo[8];  // float-float sums [2 row + stream], or the maxima in hi
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        hi[q] = MX ? -INFINITY : 0.f;
        lo[q] = 0.f;
      }
      bool ok = true;
      for (int i = 0; i < ntiles; ++i) {
        const int s = i % kStages;
        ok = async::mbar_wait(&B->full[s], (i / kStages) & 1, &B->err, dev);
        if (!__all_sync(0xffffffffu, ok)) {
          ok = false;
          break;
        }
        const float* tC = sC + (size_t)s * kTR * kTC + (size_t)(4 * warp) * kTC;
        const float4* tA = sAux + (size_t)s * kAuxMax;
        float sA[4] = {0.f, 0.f, 0.f, 0.f}, sB[4] = {0.f, 0.f, 0.f, 0.f};
        // two columns at a time; a row's terms are added column by column
#pragma unroll
        for (int q = 0; q < kTC / 64; ++q) {
          const int c0 = lane + 64 * q, c1 = c0 + 32;
          const float4 d0 = tA[c0], d1 = tA[c1];
          const uint64_t xA2 = pk(d0.x, d1.x), xB2 = pk(d0.z, d1.z);
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const uint64_t z2 = pk(tC[a * kTC + c0], tC[a * kTC + c1]);
            if constexpr (MX == 1) {
              const float2 uA = upk(f2fma(ahA2, z2, f2sub(0ull, xA2))), uB = upk(f2fma(ahB2, z2, f2sub(0ull, xB2)));
              hi[2 * a] = fmaxf(hi[2 * a], fmaxf(uA.x, uA.y));
              hi[2 * a + 1] = fmaxf(hi[2 * a + 1], fmaxf(uB.x, uB.y));
              continue;
            }
            if constexpr (MX == 2) {
              const float2 u =
                  upk(f2sub(f2fma(alA2, z2, f2fma(ahA2, z2, f2sub(oA2[a], xA2))), pk(d0.y, d1.y)));
              hi[2 * a] = fmaxf(hi[2 * a], fmaxf(u.x, u.y));
              continue;
            }
            const float2 eA = upk(exp2_pair(ahA2, alA2, z2, f2sub(oA2[a], xA2)));
            sA[a] = __fmaf_rn(eA.y, d1.y, __fmaf_rn(eA.x, d0.y, sA[a]));
            if (!WC) {
              const float2 eB = upk(exp2_pair(ahB2, alB2, z2, f2sub(oB2[a], xB2)));
              sB[a] = __fmaf_rn(eB.y, d1.w, __fmaf_rn(eB.x, d0.w, sB[a]));
            }
          }
        }
#pragma unroll
        for (int a = 0; a < 4 && !MX; ++a) {
          ff_add(hi[2 * a], lo[2 * a], sA[a]);
          ff_add(hi[2 * a + 1], lo[2 * a + 1], sB[a]);
        }
        // the tile was read through the generic proxy; the next tensor copy into it is an
        // async-proxy write
        async::fence_proxy_async_smem();
        async::mbar_arrive(&B->empty[s]);
      }
      // warp-uniform: the reduction below needs every lane
      if (__all_sync(0xffffffffu, ok && !*(volatile int*)&B->err)) {
        if constexpr (MX != 0) {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            float v = hi[q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
            const int64_t gi = g0 + (q >> 1);
            if (lane == 0 && gi < n) w.rowmax[((int64_t)blockIdx.y * 2 + (q & 1)) * n + gi] = v;
          }
        } else {
          warp_sums_ff<8>(hi, lo, lane);  // value lane / 4: row (lane / 8), stream (lane / 4) % 2
          const int64_t gi = g0 + (lane >> 3);
          const int q = (lane >> 2) & 1;
          if ((lane & 3) == 0 && gi < n && q < 2 - WC)
            w.rowpart[((int64_t)blockIdx.y * (2 - WC) + q) * n + gi] = (double)hi[0] + (double)lo[0];
        }
      }
    } else {
      // ---------------- G2: column 32 warp + lane of this column block ----------------
      const int64_t gj = (int64_t)blockIdx.x * kTC + 32 * warp + lane;
      const int64_t mp = (m + 127) / 128 * 128;  // the column data are padded to mp
      const float4 cq = w.colq[cur][gj < mp ? gj : mp - 1];
      const uint64_t oA2 = pk(-cq.x, -cq.x), oB2 = pk(-cq.z, -cq.z);
      float hA = 0.f, lA = 0.f, hB = 0.f, lB = 0.f, hC = 0.f, lC = 0.f;
      bool ok = true;
      for (int i = 0; i < ntiles; ++i) {
        const int s = i % kStages;
        ok = async::mbar_wait(&B->full[s], (i / kStages) & 1, &B->err, dev);
        if (!__all_sync(0xffffffffu, ok)) {
          ok = false;
          break;
        }
        const float* tC = sC + (size_t)s * kTR * kTC + 32 * warp + lane;
        // packed rows: {-RqA pair, qA pair}, {-RqB pair, qB pair}
        const ulonglong2* tR = reinterpret_cast<const ulonglong2*>(sAux + (size_t)s * kAuxMax);
        float sA = 0.f, sB = 0.f, sCx = 0.f;
#pragma unroll 4
        for (int a = 0; a < kTR; a += 2) {
          const ulonglong2 rA = tR[a], rB = tR[a + 1];
          const uint64_t z2 = pk(tC[a * kTC], tC[(a + 1) * kTC]);
          const float2 pA = upk(f2mul(exp2_pair(ahA2, alA2, z2, f2add(oA2, rA.x)), rA.y));
          sA = __fadd_rn(__fadd_rn(sA, pA.x), pA.y);
          if (WC) {
            const float2 zf = upk(z2);
            sCx = __fmaf_rn(zf.y, pA.y, __fmaf_rn(zf.x, pA.x, sCx));
          }
          if (!WC) {
            const float2 eB = upk(exp2_pair(ahB2, alB2, z2, f2add(oB2, rB.x))), wB = upk(rB.y);
            sB = __fmaf_rn(eB.y, wB.y, __fmaf_rn(eB.x, wB.x, sB));
          }
        }
        ff_add(hA, lA, sA);
        if (WC) ff_add(hC, lC, sCx);
        else ff_add(hB, lB, sB);
        async::fence_proxy_async_smem();
        async::mbar_arrive(&B->empty[s]);
      }
      if (ok && !*(volatile int*)&B->err && gj < m) {
        w.colpart[((int64_t)blockIdx.y * 2 + 0) * m + gj] = (double)hA + (double)lA;
        w.colpart[((int64_t)blockIdx.y * 2 + 1) * m + gj] = WC ? (double)hC + (double)lC : (double)hB + (double)lB;
      }
    }
  }
  __syncthreads();
}

}  // namespace dense

// encode the float32 tensor map of a stored cost (n x m, leading dimension ldc floats):
// boxes of 32 rows x 256 columns; needs a 16-byte aligned base and ldc a multiple of 4
cudaError_t dense_make_map(void* map_out, const float* C, int64_t n, int64_t m, int64_t ldc) {
  if (reinterpret_cast<uintptr_t>(C) % 16 != 0 || ldc % 4 != 0 || ldc < m) return cudaErrorInvalidValue;
  typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                               const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                               CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static EncodeFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !p) return cudaErrorNotSupported;
    fn = reinterpret_cast<EncodeFn>(p);
  }
  cuuint64_t dims[2] = {(cuuint64_t)m, (cuuint64_t)n};
  cuuint64_t strides[1] = {(cuuint64_t)ldc * 4};
  cuuint32_t box[2] = {(cuuint32_t)dense::kTC, (cuuint32_t)dense::kTR};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(reinterpret_cast<CUtensorMap*>(map_out), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(C),
                  dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t dense_prepare() {
  cudaError_t e = cudaSuccess;
  for (const void* f : {(const void*)dense::k_dense_tma<true, 0>, (const void*)dense::k_dense_tma<true, 1>,
                        (const void*)dense::k_dense_tma<true, 0, 1>, (const void*)dense::k_dense_tma<true, 0, 2>,
                        (const void*)dense::k_dense_tma<false, 0>,
                        (const void*)dense::k_dense_tma<false, 1>}) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dense::kSmemBytes);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  }
  return e;
}

int dense_tile_rows() { return dense::kTR; }
int dense_tile_cols() { return dense::kTC; }

int dense_blocks_per_sm() {
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, dense::k_dense_tma<false, 1>, dense::kThreads, dense::kSmemBytes);
  return nb > 0 ? nb : 1;
}

cudaError_t dense_launch_sweep(bool rows, int eval, const Geometry& g, const Work& w, const Consts& k, int splits,
                               cudaStream_t st) {
  const int64_t nblk = rows ? (k.n + dense::kTR - 1) / dense::kTR : (k.m + dense::kTC - 1) / dense::kTC;
  const int64_t ntiles = rows ? (k.m + dense::kTC - 1) / dense::kTC : (k.n + dense::kTR - 1) / dense::kTR;
  const int tps = (int)((ntiles + splits - 1) / splits);
  dim3 grid((unsigned)nblk, (unsigned)splits);
  const CUtensorMap& map = *reinterpret_cast<const CUtensorMap*>(g.map_c);
  const auto kern = rows ? (eval ? dense::k_dense_tma<true, 1> : dense::k_dense_tma<true, 0>) : eval ? dense::k_dense_tma<false, 1> : dense::k_dense_tma<false, 0>;
  return launch_kernel(kern, grid, dense::kThreads, dense::kSmemBytes, st, map, w, k.n, k.m, tps, k);
}

// Row maxima per split into w.rowmax: mode 1 the prime pass, 2 the refined pass of the dual bound.
// Bound by HBM as the sweeps are; a kernel of plain loads took 237 us at 16384 x 16384.
cudaError_t dense_launch_rowmax(int mode, const Geometry& g, const Work& w, const Consts& k, int splits,
                                cudaStream_t st) {
  const int64_t ntiles = (k.m + dense::kTC - 1) / dense::kTC;
  const int tps = (int)((ntiles + splits - 1) / splits);
  const dim3 grid((unsigned)((k.n + dense::kTR - 1) / dense::kTR), (unsigned)splits);
  return launch_kernel(mode == 1 ? dense::k_dense_tma<true, 0, 1> : dense::k_dense_tma<true, 0, 2>, grid, dense::kThreads,
                       dense::kSmemBytes, st, *reinterpret_cast<const CUtensorMap*>(g.map_c), w, k.n, k.m, tps, k);
}

}  // namespace lamp
