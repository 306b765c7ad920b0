// Operands of the tensor-core kernels: the centre mu of both clouds, then for every row of
// both clouds the split of sqrt(c) (x - mu), its squared norm and its bias row, and the
// work-split tables of a persistent loop that follows. Two launches for the bf16 operands,
// three for the integer grid's (whose exponents need the largest norm first); at the sizes
// of a request these launches, not their bytes, are the cost, so everything that can share
// one does. Sums that were float64 (GB300's float64 pipe runs at two per clock and SM) are
// pairs of floats carried without loss.
#include <cuda_bf16.h>

#include <algorithm>

#include "grid_split.cuh"
#include "progot_internal.h"
#include "tc_common.cuh"

namespace progot {

// s + e <- s + e + v without loss to ~2^-45 of s
__device__ __forceinline__ void acc2(float& s, float& e, float v) {
  const float t = s + v, bb = t - s;
  e += (s - (t - bb)) + (v - bb);
  s = t;
}

constexpr int kCenterWarps = 8;
constexpr int kCenterCols = 256;  // coordinates per block: 32 lanes x 8

// Coordinates the last block of the centre handles at a time: a power of two, 4 to 256.
__host__ __device__ inline int center_cols(int d) {
  int c = 4;
  while (c < d && c < 32 * kCenterWarps) c *= 2;
  return c;
}

// Column sums of both clouds (blockIdx.y), coordinates [256 blockIdx.z, ...): warp w of
// block b sums rows b W + w, + gridDim.x W, ..., four rows in flight; the block adds its
// warps in order, the cluster of CL blocks its blocks (one slice of the coordinates each,
// through distributed shared memory), and the last block of the grid the clusters, all in a
// fixed order, and writes mu. (Without clusters the last block read 152 blocks' sums: 16 us
// of the 48 at 16384 + 32768 rows, d = 256.)
template <int CL>
__global__ void __launch_bounds__(32 * kCenterWarps)
    center_kernel(const float* __restrict__ X, int64_t n, const float* __restrict__ Y, int64_t m, int32_t d,
                  double* __restrict__ partial, unsigned* __restrict__ ticket, float* __restrict__ mu,
                  GridWords* __restrict__ words) {
  __shared__ double acc[kCenterWarps][kCenterCols];
  __shared__ double tot[kCenterCols];
  __shared__ int s_last;
  const float* Z = blockIdx.y ? Y : X;
  const int64_t rows = blockIdx.y ? m : n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k0 = blockIdx.z * kCenterCols, kw = min(kCenterCols, d - k0);
  const int64_t step = (int64_t)gridDim.x * kCenterWarps;
  for (int j0 = 0; j0 < (kw + 31) / 32; j0 += 4) {
    // four groups of 32 coordinates and four rows: sixteen loads in flight a lane
    float s[4] = {0.f, 0.f, 0.f, 0.f}, e[4] = {0.f, 0.f, 0.f, 0.f};
    const float* z = Z + k0 + j0 * 32 + lane;
    for (int64_t row = (int64_t)blockIdx.x * kCenterWarps + warp; row < rows; row += 4 * step) {
      float v[4][4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          v[q][j] = (row + q * step < rows && (j0 + j) * 32 + lane < kw) ? __ldg(z + (row + q * step) * d + 32 * j) : 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc2(s[j], e[j], v[q][j]);
    }
    // an infinite sum leaves a NaN in e: the mean is then not finite either way
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if ((j0 + j) * 32 < kCenterCols) acc[warp][(j0 + j) * 32 + lane] = (double)s[j] + (double)e[j];
  }
  __syncthreads();
  const int parts = gridDim.x / CL;
  double* out = partial + ((int64_t)blockIdx.y * parts + blockIdx.x / CL) * d + k0;
  for (int k = threadIdx.x; k < kw; k += blockDim.x) {
    double t = 0.0;
    for (int w = 0; w < kCenterWarps; ++w) t += acc[w][k];
    if (CL == 1)
      out[k] = t;
    else
      tot[k] = t;
  }
  if constexpr (CL > 1) {
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
    const int rank = blockIdx.x % CL, w = (kw + CL - 1) / CL;
    const int k = rank * w + (int)threadIdx.x;
    if ((int)threadIdx.x < w && k < kw) {
      double v[CL], t = 0.0;
#pragma unroll
      for (int q = 0; q < CL; ++q) {
        uint32_t a;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(tc::smem_u32(&tot[k])), "r"(q));
        asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[q]) : "r"(a) : "memory");
      }
#pragma unroll
      for (int q = 0; q < CL; ++q) t += v[q];
      out[k] = t;
    }
    // no block leaves while a peer reads its sums
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned total = gridDim.x * gridDim.y * gridDim.z;
    s_last = atomicInc(ticket, total - 1) == total - 1;  // back to zero after the last block
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  if (words != nullptr && threadIdx.x < 2) {  // for grid_norms_kernel
    words->norm2_max[threadIdx.x] = 0.f;
    words->nonzero[threadIdx.x] = 0u;
    words->exp_sum[threadIdx.x] = words->raw_sum[threadIdx.x] = 0;
  }
  // 256 coordinates at a time; where there are fewer, several threads share a coordinate's
  // blocks (slices added in order)
  const int cols = center_cols(d), slices = 32 * kCenterWarps / cols;
  const int col = threadIdx.x % cols, sl = threadIdx.x / cols;
  double* red = &acc[0][0];  // [2][slices][cols]
  for (int kc = 0; kc < d; kc += cols) {
    const int k = kc + col;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      double sum = 0.0;
      if (k < d) {
        const double* src = partial + (int64_t)c * parts * d + k;
        const int b1 = (sl + 1) * parts / slices;
        for (int b = sl * parts / slices; b < b1; b += 8) {
          double v[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = b + q < b1 ? __ldcg(src + (int64_t)(b + q) * d) : 0.0;
#pragma unroll
          for (int q = 0; q < 8; ++q) sum += v[q];
        }
      }
      red[(c * slices + sl) * cols + col] = sum;
    }
    __syncthreads();
    if (sl == 0 && k < d) {
      double sx = 0.0, sy = 0.0;
      for (int q = 0; q < slices; ++q) {
        sx += red[q * cols + col];
        sy += red[(slices + q) * cols + col];
      }
      mu[k] = (float)(0.5 * (sx / (double)n + sy / (double)m));
    }
    __syncthreads();
  }
}

// Tables and initial words of a persistent loop (loop_tc.cu): CTA c's segments, a row
// block's contributors (offset, count): row block r of the remainder starts at slot
// first contributor + r, which leaves a gap of at most one slot between row blocks; in an
// aligned split CTA c's only segment has slot c.
__device__ void loop_setup(const LoopSetup& ls, int64_t tid, int64_t nthreads) {
  for (int sd = 0; sd < 2; ++sd) {
    const LoopSetupSide& S = ls.side[sd];
    const tc::Split sp = tc::make_split(S.R, S.T, ls.G);
    for (int64_t c = tid; c < ls.G; c += nthreads) {
      if (ls.aligned) {
        const tc::Seg sg = tc::aligned_segment(S.R, S.T, ls.G, (int)c);
        S.nseg[c] = 1;
        reinterpret_cast<int4*>(S.segs)[c] = make_int4(sg.r, sg.t0, sg.t1, 0);
        S.cslot[c] = (int)c;
        continue;
      }
      const int ns = tc::num_segments(sp, (int)c);
      S.nseg[c] = ns;
      int4* segs = reinterpret_cast<int4*>(S.segs) + c * ls.maxseg;
      for (int k = 0; k < ns; ++k) {
        const tc::Seg sg = tc::segment(sp, (int)c, k);
        segs[k] = make_int4(sg.r, sg.t0, sg.t1, 0);
      }
    }
    for (int64_t r = tid; r < S.R; r += nthreads) {
      if (ls.aligned) {
        const int c0 = tc::aligned_begin(S.R, ls.G, (int)r);
        S.crow[r] = make_int2(c0, tc::aligned_begin(S.R, ls.G, (int)r + 1) - c0);
      } else {
        int c0, c1;
        tc::contributors(sp, (int)r, &c0, &c1);
        const int off = r < (int64_t)sp.nb * sp.G ? (int)r : (int)r + c0;
        S.crow[r] = make_int2(off, c1 - c0 + 1);
        for (int cc = c0; cc <= c1; ++cc) S.cslot[off + cc - c0] = cc * ls.maxseg + tc::seg_of(sp, (int)r, cc);
      }
      S.flag[r] = S.flag_init;
      S.cnt[r] = 0ull;
    }
    if (tid == 0) *S.done = 0ull;
  }
  if (tid < 2) {
    SolverState st;
    st.it = 0;
    st.done = 0;
    st.status = kRunning;
    st.fcur = 0;
    st.best_it = 0;
    st.pad_[0] = st.pad_[1] = st.pad_[2] = 0;
    st.err = 0.0;
    st.best_err = INFINITY;
    ls.state[tid] = st;
  }
}

// |x_i - mu|^2 of one row by one warp: exact differences and squares as float pairs. raw (or
// NULL): |x_i|^2, rounded.
__device__ __forceinline__ float row_norm(const float* __restrict__ v, const float* __restrict__ mu, int d, int lane,
                                          float* raw = nullptr) {
  float s = 0.f, e = 0.f, r = 0.f;
  for (int k = lane; k < d; k += 32) {
    const float x = __ldg(v + k), c = __ldg(mu + k);
    const float u = x - c;
    const float bb = u - x;
    const float ue = (x - (u - bb)) - (c + bb);
    const float p = u * u;
    acc2(s, e, p);
    e += fmaf(u, u, -p) + 2.f * u * ue;
    if (raw) r = fmaf(x, x, r);
  }
  if (raw) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
    *raw = r;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float so = __shfl_xor_sync(0xffffffffu, s, off), eo = __shfl_xor_sync(0xffffffffu, e, off);
    acc2(s, e, so);
    e += eo;
  }
  return isfinite(s) ? s + e : s;
}

// Centred squared norms of both clouds; of each the largest, through an integer maximum of the
// (non-negative) floats' bits, NaN above all, and the sums of exponents of GridWords.
__global__ void grid_norms_kernel(OperandPrep op) {
  __shared__ int red[2], cnt[2], exps[2], raws[2];
  if (threadIdx.x < 2) red[threadIdx.x] = cnt[threadIdx.x] = exps[threadIdx.x] = raws[threadIdx.x] = 0;
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int best[2] = {0, 0}, nz[2] = {0, 0}, ex[2] = {0, 0}, rex[2] = {0, 0};
  float raw;
  for (int64_t row = (int64_t)blockIdx.x * 8 + warp; row < op.n + op.m; row += (int64_t)gridDim.x * 8) {
    const int side = row < op.n ? 0 : 1;
    const int64_t i = side ? row - op.n : row;
    const float nv = row_norm((side ? op.y : op.x) + i * (int64_t)op.d, op.mu, op.d, lane, &raw);
    if (lane == 0) (side ? op.ync : op.xnc)[i] = nv;
    best[side] = max(best[side], __float_as_int(nv));
    if (nv > 0.f && isfinite(nv)) {
      nz[side] += 1;
      ex[side] += ilogbf(nv);
      rex[side] += ilogbf(raw > 0.f && isfinite(raw) ? raw : nv);
    }
  }
  if (lane == 0) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (best[q] > 0) atomicMax(&red[q], best[q]);
      if (nz[q] > 0) {
        atomicAdd(&cnt[q], nz[q]);
        atomicAdd(&exps[q], ex[q]);
        atomicAdd(&raws[q], rex[q]);
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    const int q = threadIdx.x;
    if (red[q] > 0) atomicMax(reinterpret_cast<int*>(op.words->norm2_max) + q, red[q]);
    if (cnt[q] > 0) {
      atomicAdd(&op.words->nonzero[q], (unsigned)cnt[q]);
      atomicAdd(reinterpret_cast<unsigned long long*>(op.words->exp_sum) + q, (unsigned long long)(long long)exps[q]);
      atomicAdd(reinterpret_cast<unsigned long long*>(op.words->raw_sum) + q, (unsigned long long)(long long)raws[q]);
    }
  }
}

// One warp per row (and per padding row of the bias buffers): parts, norm and bias row.
// GRID: 0 bf16; 1 the integer grid, whose norms exist already; 2 the integer grid on clouds
// that moved inside the hull of those whose largest norms op.words holds (a map step's), which
// bound theirs. Blocks past the rows set a loop up.
template <int GRID>
__global__ void operands_kernel(OperandPrep op, LoopSetup ls, int row_blocks) {
  // launched while the map step before it drains; what follows reads its results
  if constexpr (GRID == 2) asm volatile("griddepcontrol.wait;" ::: "memory");
  if ((int)blockIdx.x >= row_blocks) {
    loop_setup(ls, (int64_t)(blockIdx.x - row_blocks) * blockDim.x + threadIdx.x,
               (int64_t)(gridDim.x - row_blocks) * blockDim.x);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t row = (int64_t)blockIdx.x * 8 + warp;
  const int64_t npad = (op.n + 255) / 256 * 256, mpad = (op.m + 255) / 256 * 256;
  if (row >= npad + mpad) return;
  const int side = row < npad ? 0 : 1;
  const int64_t i = side ? row - npad : row, rows = side ? op.m : op.n;
  GridScale gs;
  float pe = 1.f;
  if constexpr (GRID) {
    gs = grid_scale(*op.words, op.sc, GRID == 2);
    pe = ldexpf(1.f, side ? gs.ey : gs.ex);
    if (row == 0 && lane == 0) {
      op.words->s2 = gs.s2;
      op.words->inv = gs.inv;
      op.words->inv_ey = ldexpf(1.f, -gs.ey);
      const GridReach gr = grid_reach(*op.words, op.d, GRID == 2);
      op.words->cross = gr.x1 > kGridCross;
      if (op.words->bad == 0 && grid_out_of_range(*op.words, gs, gr, op.min_exp)) op.words->bad = op.step;
    }
  }
  float nv = 0.f;
  if (i < rows) {
    const float* v = (side ? op.y : op.x) + i * (int64_t)op.d;
    void* const* parts = side ? op.yp : op.xp;
    uint32_t* h_out = reinterpret_cast<uint32_t*>(parts[0]) + i * (op.dp / 2);
    uint32_t* l_out = parts[1] ? reinterpret_cast<uint32_t*>(parts[1]) + i * (op.dp / 2) : nullptr;
    uint32_t* r_out = parts[2] ? reinterpret_cast<uint32_t*>(parts[2]) + i * (op.dp / 2) : nullptr;
    if constexpr (GRID == 2) nv = row_norm(v, op.mu, op.d, lane);
    float s = 0.f, se = 0.f;
    for (int k2 = lane; k2 < op.dp / 2; k2 += 32) {
      uint32_t h = 0u, l = 0u, r = 0u;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int k = 2 * k2 + e;
        const float x = k < op.d ? __ldg(v + k) : 0.f, c = k < op.d ? __ldg(op.mu + k) : 0.f;
        const float u = x - c;
        if constexpr (GRID) {
          // v = (x - mu) sqrt(c) 2^e as an unevaluated sum of two floats
          const float bb = u - x;
          const float ue = (x - (u - bb)) - (c + bb);
          const float vh = u * op.sc;
          const float ve = fmaf(u, op.sc, -vh) + fmaf(ue, op.sc, u * op.sc_lo);
          const float a = vh * pe, b = ve * pe;
          const float hv = rintf(a);
          const __half lh = __float2half_rn((a - hv) + b);
          const float rv = ((a - hv) - __half2float(lh)) + b;
          h |= (uint32_t)__half_as_ushort(__float2half_rn(hv)) << (16 * e);
          l |= (uint32_t)__half_as_ushort(lh) << (16 * e);
          r |= (uint32_t)__half_as_ushort(__float2half_rn(rv)) << (16 * e);
        } else {
          const float p = u * u;
          acc2(s, se, p);
          se += fmaf(u, u, -p);
          const float vh = u * op.sc;
          const __nv_bfloat16 hb = __float2bfloat16_rn(vh);
          h |= (uint32_t)__bfloat16_as_ushort(hb) << (16 * e);
          l |= (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(vh - __bfloat162float(hb))) << (16 * e);
        }
      }
      h_out[k2] = h;
      if (l_out) l_out[k2] = l;
      if (r_out) r_out[k2] = r;
    }
    if constexpr (GRID == 1) {
      nv = (side ? op.ync : op.xnc)[i];
    } else if constexpr (GRID == 2) {
      if (lane == 0) (side ? op.ync : op.xnc)[i] = nv;
    } else {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const float so = __shfl_xor_sync(0xffffffffu, s, off), eo = __shfl_xor_sync(0xffffffffu, se, off);
        acc2(s, se, so);
        se += eo;
      }
      nv = isfinite(s) ? s + se : s;
      if (lane == 0) (side ? op.ync : op.xnc)[i] = nv;
    }
  }
  const float* pot = side ? op.g : op.f;
  if (pot != nullptr && lane < 2) {
    __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>((side ? op.yb : op.xb)[lane]);
    if (dst != nullptr) {
      if constexpr (GRID)
        write_bias_row_grid(dst + i * 16,
                            i < rows ? grid_beta(pot[i], nv, op.bscale, op.bscale_lo) : make_float2(-INFINITY, 0.f),
                            gs.s2);
      else
        tc::write_bias_row(dst + i * 16, i < rows ? (pot[i] - nv) * op.bscale : -INFINITY);
    }
  }
}

cudaError_t launch_center(const float* X, int64_t n, const float* Y, int64_t m, int32_t d, double* partial,
                          unsigned* ticket, float* mu, GridWords* words, cudaStream_t s) {
  // at least four rows a warp (one load round); clusters of eight where the last block
  // would otherwise add more than two rounds of block sums a thread
  const int64_t rows = std::max<int64_t>(n, m);
  int parts = (int)std::max<int64_t>(1, std::min<int64_t>(reduce_parts() / 2, rows / (4 * kCenterWarps)));
  const int z = (d + kCenterCols - 1) / kCenterCols;
  if (parts * center_cols(d) <= 16 * 32 * kCenterWarps) {
    center_kernel<1><<<dim3(parts, 2, z), 32 * kCenterWarps, 0, s>>>(X, n, Y, m, d, partial, ticket, mu, words);
    count_launch();
    return cudaGetLastError();
  }
  parts = parts / 8 * 8;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(parts, 2, z);
  cfg.blockDim = dim3(32 * kCenterWarps);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 8;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, center_kernel<8>, X, n, Y, m, d, partial, ticket, mu, words);
  count_launch();
  return e;
}

cudaError_t launch_operands(const OperandPrep& op, OperandKind kind, const LoopSetup* loop, cudaStream_t s) {
  if (kind == OperandKind::kGrid) {
    const int64_t blocks = std::min<int64_t>((op.n + op.m + 7) / 8, 152 * 16);
    grid_norms_kernel<<<(unsigned)blocks, 256, 0, s>>>(op);
    count_launch();
  }
  const int64_t rows = (op.n + 255) / 256 * 256 + (op.m + 255) / 256 * 256;
  const int row_blocks = (int)(rows / 8);
  LoopSetup ls = {};
  int extra = 0;
  if (loop != nullptr) {
    ls = *loop;
    extra = (int)std::min<int64_t>(8, (std::max(ls.side[0].R, ls.side[1].R) + 255) / 256 + 1);
  }
  if (kind == OperandKind::kGrid)
    operands_kernel<1><<<(unsigned)(row_blocks + extra), 256, 0, s>>>(op, ls, row_blocks);
  else if (kind == OperandKind::kGridHull) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(row_blocks + extra));
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, operands_kernel<2>, op, ls, row_blocks);
    if (e != cudaSuccess) return e;
  } else
    operands_kernel<0><<<(unsigned)(row_blocks + extra), 256, 0, s>>>(op, ls, row_blocks);
  count_launch();
  return cudaGetLastError();
}

// The end of a persistent loop: row log-sum-exps for the map step from the potential its
// last f-update wrote, L_i = (eps log w_i + |a_i|^2 - f_i) / (eps ln2) in float64 (w = NULL:
// log w_i = log_w_uniform), and the current f into its place when it is in the other buffer.
__global__ void loop_finish_kernel(const float* f_new, const float* __restrict__ an, const float* __restrict__ w,
                                   double log_w_uniform, double eps, double inv, int64_t n, float* __restrict__ L,
                                   const float* f_cur, float* f_out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float fn = f_new[i];
  if (f_out != nullptr) f_out[i] = f_cur[i];  // f_out may be f_new: read above
  const double logw = w ? log((double)w[i]) : log_w_uniform;
  L[i] = (float)((eps * logw + (double)an[i] - (double)fn) * inv);
}

cudaError_t launch_loop_finish(const float* f_new, const float* an, const float* w, double log_w_uniform, double eps,
                               int64_t n, float* L, const float* f_cur, float* f_out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  loop_finish_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(f_new, an, w, log_w_uniform, eps,
                                                                 1.0 / (eps * kLn2), n, L, f_cur, f_out);
  count_launch();
  return cudaGetLastError();
}

// Warm start of Alg. 2: g_k = c g_{k-1}, f <- c f (g_prev = NULL: both start at zero).
__global__ void warm_start_kernel(float* g, const float* __restrict__ g_prev, int64_t m, float* f, int64_t n, float c) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) g[i] = g_prev ? g_prev[i] * c : 0.f;
  if (i < n) f[i] = g_prev ? f[i] * c : 0.f;
}

cudaError_t launch_warm_start(float* g, const float* g_prev, int64_t m, float* f, int64_t n, float c, cudaStream_t s) {
  const int64_t k = std::max(n, m);
  if (k <= 0) return cudaSuccess;
  warm_start_kernel<<<(unsigned)((k + 255) / 256), 256, 0, s>>>(g, g_prev, m, f, n, c);
  count_launch();
  return cudaGetLastError();
}

}  // namespace progot
