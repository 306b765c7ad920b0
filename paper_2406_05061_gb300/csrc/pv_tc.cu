// Second half of the map step on integer-grid operands (Alg. 2 / Alg. 3): with
// P_ij = 2^{t_ij - L_i + 14} and its row sums left by a kModeProb sweep (sweep_tc.cu),
//   T_i = sum_j P_ij y_j / sum_j P_ij,   x_i <- x_i + alpha (T_i - x_i),
// as a product over the column index on tcgen05: half-precision P (hi, lo) against the
// y operand's parts, read as an MN-major matrix.
//
// tcgen05 accumulates with truncation, so a sum over thousands of columns would drift
// toward zero by one part in 2^24 per K step. Each unit of 64 columns therefore starts a
// fresh pair of TMEM accumulators (P hi . y hi in one, the small products in the other),
// and the two epilogue warpgroups add the finished unit to float32 registers, rounding to
// nearest, while the products of the next unit run into the other pair.
//
// One CTA = (128-row block, up to 128 coordinates, a share of the units); the CTAs that
// share a block form a cluster of up to 8 and reduce their sums through distributed shared
// memory in rank order (deterministic, no partials in global memory). P is stored as the
// shared-memory image of the operand tile, so a unit's P is one 32 KB bulk copy.
// Warps: 0 producer, 1 TMEM owner and MMA issuer, 2-9 two warpgroups, each half of the
// coordinates. Every mbarrier wait is bounded as in the sweeps; a CTA that gives up still
// reaches the cluster barriers and leaves NaN rows and the fault flag.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "progot_internal.h"
#include "tc_common.cuh"

namespace progot {
namespace tc {

constexpr int PV_NTHREADS = 320;
constexpr int PV_UNIT = 64;                   // columns j per unit
constexpr uint32_t PV_P_BYTES = 2 * 128 * 64 * 2;  // P hi and lo of a unit: 32 KB
constexpr uint32_t PV_Y_BYTES = 64 * 64 * 2;       // one part of 64 coordinates of a unit: 8 KB
constexpr int PV_MAXST = 4;

struct PvShared {
  uint64_t full[PV_MAXST], empty[PV_MAXST];
  uint64_t acc_full[2], acc_empty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int32_t abort_flag;
};

struct PvParams {
  const float* X;
  float* out;
  const float* rsum;
  const unsigned char* prob;
  const GridWords* words;
  const float* mu;
  int32_t* fault;
  int64_t rows;
  int32_t d, units, chunks, splits, stages;
  float alpha, inv_sc;
};

// 64-coordinate column groups of a unit's K-major y tiles, read as one MN-major matrix:
// 8-row groups 1024 bytes apart, the next 64 coordinates one tile on.
__device__ __forceinline__ uint64_t pv_desc_mn(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(PV_Y_BYTES >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ float ld_peer(uint32_t saddr, uint32_t rank) {
  uint32_t a;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(saddr), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

// NB: blocks of 64 coordinates per CTA (1 or 2).
template <int NB>
__global__ void __launch_bounds__(PV_NTHREADS, 1)
    pv_tc(const __grid_constant__ CUtensorMap mapY0, const __grid_constant__ CUtensorMap mapY1,
          const __grid_constant__ CUtensorMap mapY2, const PvParams pp) {
  constexpr int N = 64 * NB, NH = N / 2;  // coordinates of the CTA and of one warpgroup
  if (__ldg(&pp.words->bad) != 0) {  // no P was written
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return;
  }
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ PvShared sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = pp.stages;
  constexpr uint32_t st_bytes = PV_P_BYTES + kGridParts * NB * PV_Y_BYTES;
  const int rank = blockIdx.x % pp.splits, tile = blockIdx.x / pp.splits;
  const int chunk = tile % pp.chunks, rb = tile / pp.chunks;
  const int u0 = (int)((int64_t)rank * pp.units / pp.splits), u1 = (int)((int64_t)(rank + 1) * pp.units / pp.splits);
  const int nu = u1 - u0;
  volatile int32_t* abort_flag = &sh.abort_flag;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sh.acc_full[b], 1);
      mbar_init(&sh.acc_empty[b], 8);
    }
    mbar_init(&sh.drain, 1);
    sh.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_base)),
                 "r"(4 * N)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = sh.tmem_base;
  // programmatic launch: the set-up above overlaps the sweep that writes P
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");

  float o[NH];
  if (warp == 0) {
    // ------------------------------------------------------------ producer
    bool ok = true;
    int u = 0, s_cur = 0;  // ring position and fill parity kept without division
    uint32_t s_par = 0;
    for (; u < nu; ++u) {
      const int s = s_cur;
      ok = warp_wait(&sh.empty[s], s_par ^ 1u, abort_flag);
      if (!ok) break;
      if (++s_cur == S) {
        s_cur = 0;
        s_par ^= 1u;
      }
      unsigned char* st = smem + s * st_bytes;
      if (elect_one()) {
        mbar_arrive_expect_tx(&sh.full[s], st_bytes);
        bulk_load(st, pp.prob + ((int64_t)rb * pp.units + u0 + u) * PV_P_BYTES, PV_P_BYTES, &sh.full[s]);
        for (int q = 0; q < kGridParts; ++q) {
          const CUtensorMap* mY = q == 0 ? &mapY0 : q == 1 ? &mapY1 : &mapY2;
          // coordinates past the operand's width are filled with zeros
          for (int b = 0; b < NB; ++b)
            tma_load_2d(st + PV_P_BYTES + (q * NB + b) * PV_Y_BYTES, mY, &sh.full[s], chunk * N + b * 64,
                        (u0 + u) * PV_UNIT);
        }
      }
      __syncwarp();
    }
    if (!ok)  // drain this CTA's own copies still in flight
      for (int v = max(0, u - S); v < u; ++v) warp_wait(&sh.full[v % S], (uint32_t)((v / S) & 1), abort_flag, true);
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    constexpr uint32_t kId = make_idesc_f16(BM, N) | (1u << 16);  // A K-major, B MN-major
    bool ok = true;
    int s_cur = 0;
    uint32_t s_par = 0;
    for (int u = 0; u < nu && ok; ++u) {
      const int s = s_cur, b = u & 1;
      ok = warp_wait(&sh.acc_empty[b], (uint32_t)(((u >> 1) & 1) ^ 1), abort_flag) &&
           warp_wait(&sh.full[s], s_par, abort_flag);
      if (!ok) break;
      if (++s_cur == S) {
        s_cur = 0;
        s_par ^= 1u;
      }
      tc_fence_after();
      const uint32_t st = smem_u32(smem + s * st_bytes);
      const uint64_t ph = desc_sw128(st), pl = desc_sw128(st + PV_P_BYTES / 2);
      const uint64_t y0 = pv_desc_mn(st + PV_P_BYTES), y1 = pv_desc_mn(st + PV_P_BYTES + NB * PV_Y_BYTES),
                     y2 = pv_desc_mn(st + PV_P_BYTES + 2 * NB * PV_Y_BYTES);
      const uint32_t d1 = tmem_base + (uint32_t)(b * 2 * N), d2 = d1 + N;
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < PV_UNIT / 16; ++kk) {
          // +32 bytes per K = 16 step in P's 128-byte rows; +16 rows (2048 bytes) of the y tiles
          const uint64_t adv = (uint64_t)(kk * 2), bdv = (uint64_t)(kk * 128);
          const uint32_t more = kk > 0 ? 1u : 0u;
          umma_id(d1, ph + adv, y0 + bdv, kId, more);
          umma_id(d2, ph + adv, y1 + bdv, kId, more);
          umma_id(d2, pl + adv, y0 + bdv, kId, 1u);
          umma_id(d2, pl + adv, y1 + bdv, kId, 1u);
          umma_id(d2, ph + adv, y2 + bdv, kId, 1u);
        }
        umma_commit(&sh.empty[s]);
        umma_commit(&sh.acc_full[b]);
      }
      __syncwarp();
    }
    if (elect_one()) umma_commit(&sh.drain);
    __syncwarp();
    warp_wait(&sh.drain, 0, abort_flag, true);
  } else {
    // ------------------------------------------------------------ float32 sums of the units
    const int wg = (warp - 2) >> 2, quarter = warp & 3;
#pragma unroll
    for (int e = 0; e < NH; ++e) o[e] = 0.f;
    bool ok = true;
    for (int u = 0; u < nu && ok; ++u) {
      const int b = u & 1;
      ok = warp_wait(&sh.acc_full[b], (uint32_t)((u >> 1) & 1), abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t t1 = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * 2 * N + wg * NH);
#pragma unroll
      for (int cc = 0; cc < NH / 32; ++cc) {
        float v[32], w[32];
        PROGOT_TMEM_LD32(t1 + cc * 32, v);
        PROGOT_TMEM_LD32(t1 + N + cc * 32, w);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 32; ++e) o[cc * 32 + e] += v[e] + w[e];
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.acc_empty[b]);
    }
    if (!ok) {
#pragma unroll
      for (int e = 0; e < NH; ++e) o[e] = NAN;
    }
  }
  // every role of this CTA is done with the stages: they hold the sums now (row pitch N + 1
  // words: conflict-free in both directions)
  __syncthreads();
  float* osum = reinterpret_cast<float*>(smem);
  if (warp >= 2) {
    const int wg = (warp - 2) >> 2, row = (warp & 3) * 32 + lane;
#pragma unroll
    for (int e = 0; e < NH; ++e) osum[row * (N + 1) + wg * NH + e] = o[e];
  }
  if (pp.splits > 1)
    cluster_sync_all();
  else
    __syncthreads();
  // ---- rows of this rank: sums over the ranks in order, then x + alpha (T - x)
  {
    const int r0 = rank * BM / pp.splits, r1 = (rank + 1) * BM / pp.splits;
    const int64_t left = pp.rows - (int64_t)rb * BM;
    const int rend = left < r1 ? (int)left : r1;
    const float scale = pp.inv_sc * __ldg(&pp.words->inv_ey);
    const uint32_t base = smem_u32(osum);
    for (int q = r0 * N + threadIdx.x; q < rend * N; q += PV_NTHREADS) {
      const int r = q / N, k = q % N, kk = chunk * N + k;
      if (kk >= pp.d) continue;
      float sum = 0.f;
      if (pp.splits > 1) {
        for (int t = 0; t < pp.splits; ++t) sum += ld_peer(base + (uint32_t)(r * (N + 1) + k) * 4u, (uint32_t)t);
      } else {
        sum = osum[r * (N + 1) + k];
      }
      const int64_t i = (int64_t)rb * BM + r;
      const float x = pp.X[i * pp.d + kk];
      const float T = fmaf(sum / __ldg(pp.rsum + i), scale, __ldg(pp.mu + kk));
      pp.out[i * pp.d + kk] = fmaf(pp.alpha, T - x, x);
    }
  }
  // no CTA leaves while a peer reads its sums
  if (pp.splits > 1) cluster_sync_all();
  tc_fence_before();
  __syncthreads();
  if (sh.abort_flag != 0 && threadIdx.x == 0 && pp.fault) atomicExch(pp.fault, 1);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(4 * N) : "memory");
  }
}

}  // namespace tc

int64_t pv_prob_bytes_per_block(int64_t m) { return (m + 127) / 128 * 2 * (int64_t)tc::PV_P_BYTES; }

template <int NB>
static cudaError_t pv_attributes(size_t smem) {
  static thread_local size_t attr_bytes = 0;
  if (smem <= attr_bytes) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(tc::pv_tc<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) attr_bytes = smem;
  return e;
}

static void pv_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, int grid, int splits, size_t smem,
                      cudaStream_t stream) {
  *cfg = {};
  cfg->gridDim = dim3(grid);
  cfg->blockDim = dim3(tc::PV_NTHREADS);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = splits;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 2;
}

// Clusters of `splits` CTAs that run at once: fewer than the SMs allow, since a cluster stays inside
// one GPC (15 of eight and 36 of four on a GB300).
template <int NB>
static int pv_clusters(int splits, size_t smem, int sms) {
  static thread_local int cached[9] = {};
  if (cached[splits] == 0) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    pv_config(&cfg, attr, splits * sms, splits, smem, nullptr);
    cfg.numAttrs = 1;
    int c = 0;
    if (cudaOccupancyMaxActiveClusters(&c, tc::pv_tc<NB>, &cfg) != cudaSuccess || c < 1) {
      (void)cudaGetLastError();
      c = std::max(1, sms / splits);
    }
    cached[splits] = c;
  }
  return cached[splits];
}

template <int NB>
static cudaError_t launch_pv(tc::PvParams pp, int64_t tiles, size_t smem, const void* const* maps, int sms,
                             cudaStream_t stream) {
  cudaError_t e = pv_attributes<NB>(smem);
  if (e != cudaSuccess) return e;
  // CTAs per tile: the share that finishes first in waves of the clusters that run at once, a CTA
  // costing about three units besides its own (2368 x 753, d = 17: 45.4 us a map step with waves of
  // SMs, which took eight CTAs for each of the 19 row blocks and so a second wave, 40.4 so)
  double best = 0.0;
  pp.splits = 1;
  for (int s = 1; s <= 8 && s <= pp.units; s *= 2) {
    const int c = pv_clusters<NB>(s, smem, sms);
    const double cost = (double)((tiles + c - 1) / c) * ((double)((pp.units + s - 1) / s) + 3.0);
    if (s == 1 || cost < best) {
      best = cost;
      pp.splits = s;
    }
  }
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  pv_config(&cfg, attr, (int)(tiles * pp.splits), pp.splits, smem, stream);
  auto at = [](const void* p) -> const CUtensorMap& { return *reinterpret_cast<const CUtensorMap*>(p); };
  return cudaLaunchKernelEx(&cfg, tc::pv_tc<NB>, at(maps[0]), at(maps[1]), at(maps[2]), pp);
}

cudaError_t launch_pv_tc(const PvLaunch& p, int sms, cudaStream_t stream) {
  tc::PvParams pp;
  pp.X = p.X;
  pp.out = p.out;
  pp.rsum = p.rsum;
  pp.prob = (const unsigned char*)p.prob;
  pp.words = p.words;
  pp.mu = p.mu;
  pp.fault = p.fault;
  pp.rows = p.rows;
  pp.d = p.d;
  pp.alpha = p.alpha;
  pp.inv_sc = p.inv_sc;
  const int nb = p.d > 64 ? 2 : 1;
  pp.units = (int)((p.m + 127) / 128 * 2);
  pp.chunks = (p.d + 64 * nb - 1) / (64 * nb);
  const int64_t tiles = (p.rows + 127) / 128 * pp.chunks;
  const uint32_t st_bytes = tc::PV_P_BYTES + (uint32_t)kGridParts * nb * tc::PV_Y_BYTES;
  pp.stages = std::min<int>(tc::PV_MAXST, (int)((225 * 1024) / st_bytes));
  const size_t smem = std::max<size_t>((size_t)pp.stages * st_bytes, (size_t)128 * (64 * nb + 1) * 4) + 1024;
  const cudaError_t e = nb == 2 ? launch_pv<2>(pp, tiles, smem, p.mapY, sms, stream)
                                : launch_pv<1>(pp, tiles, smem, p.mapY, sms, stream);
  count_launch();
  return e;
}

}  // namespace progot
