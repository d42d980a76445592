// Redundancy analysis (the pairwise key / value similarity the paper plots as heat maps and
// summarises per head, Sec. 1 and Sec. 3.1): block-mean cosine similarity map of the rows of one
// tensor.  The mean of cos(x_i, x_j) over a cell (i in block I, j in block J) is
// u_I . u_J / (n_I n_J) with u_I the sum of the unit rows of block I, the same identity that turns
// the mean of the whole matrix into Eq. 4.  So a map needs one streaming pass over the rows, which
// leaves the block sums (k_block_sums, here), and the Gram matrix of the block sums on the tensor
// cores (k_gram, similarity_tc.cu): never more than T x T x d multiply-adds for T x T cells, T = L
// only where a cell is one pair of rows.
#include <cooperative_groups.h>

#include <cuda_fp16.h>
#include <math.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace mixkv {
namespace {

constexpr int kSumWarps = 8;
constexpr int kSumThreads = kSumWarps * 32;
constexpr int kSumStep = 16;        // rows a warp holds in registers at a time (4 KB of loads in flight)
constexpr int kSumSteps = 2;        // steps of a warp, at least
constexpr int kSumRows = kSumStep * kSumSteps;
constexpr int kSumMaxCluster = 8;

// Three layouts of the work of k_block_sums, by the rows per block.
enum { kRowsOne = 0,    // block == 1: every row leaves as its own "sum"
       kRowsFew = 1,    // block <= 16: a warp takes whole blocks
       kRowsMany = 2 }; // longer blocks: the warps of a CTA (or of a cluster) share one

__host__ __device__ constexpr int sum_mode(int block) {
  return block == 1 ? kRowsOne : block <= kSumStep ? kRowsFew : kRowsMany;
}
// Blocks one CTA (or cluster) takes.
__host__ __device__ inline int blocks_per_cta(int block) {
  if (block <= kSumStep) return kSumWarps * kSumSteps * (kSumStep / block);
  const int sub = (block + kSumRows - 1) / kSumRows;
  return sub < kSumWarps ? kSumWarps / sub : 1;
}

// x (scaled) as two fp16, value and remainder: 11 bits each and the remainder's sign, 23 of fp32's 24.  A quarter of the values
// lose their last bit, up to 2^-23 of the value.
__device__ __forceinline__ void split_pair(const float (&x)[8], uint4& hi, uint4& lo) {
  __half2 h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    h[e] = __floats2half2_rn(x[2 * e], x[2 * e + 1]);
    const float2 b = __half22float2(h[e]);
    l[e] = __floats2half2_rn(x[2 * e] - b.x, x[2 * e + 1] - b.y);
  }
  hi = *reinterpret_cast<const uint4*>(h);
  lo = *reinterpret_cast<const uint4*>(l);
}
// A unit row as two bf16, 16 bits for what comes from 8.
__device__ __forceinline__ void split_row(const float (&x)[8], uint4& hi, uint4& lo) {
  __nv_bfloat162 h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    h[e] = __floats2bfloat162_rn(x[2 * e], x[2 * e + 1]);
    const float2 b = __bfloat1622float2(h[e]);
    l[e] = __floats2bfloat162_rn(x[2 * e] - b.x, x[2 * e + 1] - b.y);
  }
  hi = *reinterpret_cast<const uint4*>(h);
  lo = *reinterpret_cast<const uint4*>(l);
}
// The power of two that the sums are scaled by: a component of a block's sum is at most its rows, which go to 2^15, half of
// fp16's range, so that the remainder of everything down to 2^-17 of that has its bits.
inline float sum_scale(const int block) {
  int bits = 0;
  while (bits < 31 && (1LL << bits) < block) ++bits;
  return ldexpf(1.f, 15 - bits);
}

// grid (slices * cluster, H).  Sums of the unit rows of every block, times `scale`, written as two fp16 parts
// ([2][H][T][d]; a row that stands for itself as two bf16, unscaled: as fp16 4 heads of 5000 single rows took 3 % longer), the
// number of non-zero rows of every block, and per slice (what one CTA or cluster read) the sum of
// its unit rows and its non-zero rows, from which the head mean comes.
//
// HBM bound: every row is read once, 16 lanes of 16 bytes to a row, the 16 rows of a warp's step asked for
// before the first is used (4 KB per warp, 32 warps per SM: with 32 rows per step and 16 warps the last of two
// waves was half empty).  The squared norms of a step are reduced by folding (8 exchanges per lane instead of 32
// for 8 butterflies), bf16 pairs are widened in place and multiplied as packed fp32.
// B: the rows per block where they are a power of two up to 16 (the places where a block ends are then known
// to the compiler; 14 us with a test after every row, 131072 rows in blocks of 16), else 0.
template <int MODE, int B>
__global__ void __launch_bounds__(kSumThreads, MODE == kRowsMany ? 4 : 3)
k_block_sums(const __nv_bfloat16* __restrict__ X, const int L, const int block_arg, const int T, const float scale,
             uint16_t* __restrict__ parts, int* __restrict__ nz, float* __restrict__ us,
             int* __restrict__ nzs) {
  const int block = B ? B : block_arg;
  __shared__ __align__(16) float part[kSumWarps][kHeadDim];
  __shared__ int cnt[kSumWarps];
  __shared__ float csum[kHeadDim];
  __shared__ int ccnt;
  cg::cluster_group cluster = cg::this_cluster();
  const int S = MODE == kRowsMany ? (int)cluster.num_blocks() : 1;
  const int rank = MODE == kRowsMany ? (int)cluster.block_rank() : 0;
  const int slice = blockIdx.x / S, h = blockIdx.y, H = gridDim.y, nslices = gridDim.x / S;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, half = lane >> 4, c = lane & 15;
  const int bpc = blocks_per_cta(block);
  const size_t part_stride = (size_t)H * T * kHeadDim;
  const __nv_bfloat16* base = X + (size_t)h * L * kHeadDim + 8 * c;
  uint16_t* prow = parts + (size_t)h * T * kHeadDim + 8 * c;
  pdl_launch_dependents();
  pdl_wait();

  f32x2 tot[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) tot[e] = pack2(0.f, 0.f);
  int tot_nz = 0;

  // The warp's rows: whole blocks (few rows per block), or a share of one block.
  int r0, end, step;           // first row of a step, end of the warp's range, rows between its steps
  int again = 0, blk = 0;      // rows skipped after every second step (a cluster's turns); block of the step
  if (MODE != kRowsMany) {
    const int per_step = kSumStep / block;
    blk = slice * bpc + warp * kSumSteps * per_step;
    r0 = blk * block;
    step = per_step * block;
    end = min(L, r0 + kSumSteps * step);
  } else {
    const int sub = (block + kSumRows - 1) / kSumRows;   // shares of kSumRows rows in a block
    const int share = sub < kSumWarps ? sub : kSumWarps; // warps of a CTA on one block
    const int slot = warp / share;
    blk = slice * bpc + slot;
    r0 = blk * block + (rank * share + warp - slot * share) * kSumRows;
    end = slot < bpc ? min(L, (blk + 1) * block) : 0;
    step = kSumStep;
    again = (S * share - 1) * kSumRows;
  }
#pragma unroll 1
  for (int turn = 0; r0 < end; ++turn, r0 += step + ((turn & 1) ? 0 : again)) {
    const int stop = MODE == kRowsMany ? end : min(end, r0 + step);
    uint4 v[8];
    float p[8];
    const uint4* rp = reinterpret_cast<const uint4*>(base + (size_t)(r0 + half) * kHeadDim);
    const int left = stop - r0 - half;
#pragma unroll
    for (int i = 0; i < 8; ++i) {   // one address, constant offsets
      v[i] = make_uint4(0, 0, 0, 0);
      if (2 * i < left) v[i] = __ldg(rp + 2 * i * (kHeadDim / 8));
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
      f32x2 sq = pack2(0.f, 0.f);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        // (byte permutes here, bf16x2_wide below: widened by the same instructions in both sweeps, all values
        // would be kept in between, which does not fit the registers)
        const f32x2 f = pack2(__uint_as_float(__byte_perm(w[e], 0u, 0x1044)),
                              __uint_as_float(__byte_perm(w[e], 0u, 0x3244)));
        sq = fma2(f, f, sq);
      }
      float s0, s1;
      unpack2(sq, s0, s1);
      p[i] = s0 + s1;
    }
    // folding: lanes 2 i, 2 i + 1 of a half are left with the squared norm of row 2 i + half
#pragma unroll
    for (int o = 8; o >= 2; o >>= 1) {
      const bool up = (c & o) != 0;
#pragma unroll
      for (int k = 0; k < o / 2; ++k) {
        const float send = up ? p[k] : p[k + o / 2], keep = up ? p[k + o / 2] : p[k];
        p[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    p[0] += __shfl_xor_sync(0xffffffffu, p[0], 1);
    const float inv = p[0] > 0.f ? rsqrtf(p[0]) : 0.f;
    // bit r of `alive`: row r of the step is not zero (row r = 2 i + half stands with lane 16 half + 2 i)
    const float of_row = __shfl_sync(0xffffffffu, inv, ((lane & 1) << 4) | (lane & 14));
    const unsigned alive = __ballot_sync(0xffffffffu, of_row > 0.f) & 0xffffu;
    tot_nz += __popc(alive);
    f32x2 acc[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[e] = pack2(0.f, 0.f);
    // sum of the two halves' accumulators -> the parts of block `blk` (rows a .. b-1 of the step)
    auto flush = [&](const int a, const int b) {
      float s[8];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        unpack2(acc[e], s[2 * e], s[2 * e + 1]);
        s[2 * e] += __shfl_xor_sync(0xffffffffu, s[2 * e], 16);
        s[2 * e + 1] += __shfl_xor_sync(0xffffffffu, s[2 * e + 1], 16);
        tot[e] = add2(tot[e], pack2(s[2 * e], s[2 * e + 1]));
      }
      if (blk < T) {
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] *= scale;
        uint4 hi, lo;
        split_pair(s, hi, lo);   // half 0 writes the values, half 1 the remainders
        *reinterpret_cast<uint4*>(prow + (size_t)half * part_stride + (size_t)blk * kHeadDim) = half ? lo : hi;
        if (lane == 0) nz[(size_t)h * T + blk] = __popc(alive & ((1u << b) - (1u << a)));
      }
      ++blk;
    };
    int next = block, a0 = 0;   // kRowsFew: row of the step at which the current block ends / starts
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if constexpr (B > 1) next = 2 * i / B * B + B, a0 = next - B;
      const float w = __shfl_sync(0xffffffffu, inv, (lane & 16) | (2 * i));
      const f32x2 w2 = pack2(w, w);
      const uint32_t q[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
      f32x2 f[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) f[e] = bf16x2_wide(q[e]);
      if (MODE == kRowsOne) {
        const int r = r0 + 2 * i + half;
        float x[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          tot[e] = fma2(f[e], w2, tot[e]);
          float x0, x1;
          unpack2(f[e], x0, x1);
          x[2 * e] = x0 * w, x[2 * e + 1] = x1 * w;
        }
        if (r < stop) {
          uint4 hi, lo;
          split_row(x, hi, lo);
          *reinterpret_cast<uint4*>(prow + (size_t)r * kHeadDim) = hi;
          *reinterpret_cast<uint4*>(prow + part_stride + (size_t)r * kHeadDim) = lo;
          if (c == 0) nz[(size_t)h * T + r] = w > 0.f ? 1 : 0;
        }
      } else if (MODE == kRowsFew) {
        if (B < 2 && next == 2 * i + 1) {   // the block ends between the two rows of this pair
          const f32x2 mine = half == 0 ? w2 : pack2(0.f, 0.f), rest = half == 0 ? pack2(0.f, 0.f) : w2;
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[e] = fma2(f[e], mine, acc[e]);
          flush(a0, next);
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[e] = fma2(f[e], rest, pack2(0.f, 0.f));
          a0 = next;
          next += block;
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[e] = fma2(f[e], w2, acc[e]);
        }
        if (next == 2 * i + 2) {
          flush(a0, next);
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[e] = pack2(0.f, 0.f);
          a0 = next;
          next += block;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) tot[e] = fma2(f[e], w2, tot[e]);
      }
    }
  }
  // per-warp sums of unit rows (kRowsFew: the two halves already hold the same totals)
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float s0, s1;
    unpack2(tot[e], s0, s1);
    if (MODE != kRowsFew) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, 16);
      s1 += __shfl_xor_sync(0xffffffffu, s1, 16);
    }
    if (half == 0) *reinterpret_cast<float2*>(&part[warp][8 * c + 2 * e]) = make_float2(s0, s1);
  }
  if (lane == 0) cnt[warp] = tot_nz;
  __syncthreads();
  if (MODE == kRowsMany) {
    const int sub = (block + kSumRows - 1) / kSumRows;
    const int share = sub < kSumWarps ? sub : kSumWarps;
    if (S > 1) {   // one block per cluster: every CTA's sum, then rank 0 adds them in rank order
      if (tid < kHeadDim) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kSumWarps; ++w) s += part[w][tid];
        csum[tid] = s;
      }
      if (tid == 0) {
        int n = 0;
        for (int w = 0; w < kSumWarps; ++w) n += cnt[w];
        ccnt = n;
      }
      cluster.sync();
      if (rank == 0) {
        if (tid < kHeadDim) {
          float s = 0.f;
          for (int r = 0; r < S; ++r) s += *cluster.map_shared_rank(&csum[tid], r);
          part[0][tid] = s;
#pragma unroll
          for (int w = 1; w < kSumWarps; ++w) part[w][tid] = 0.f;
        }
        if (tid == 0) {
          int n = 0;
          for (int r = 0; r < S; ++r) n += *cluster.map_shared_rank(&ccnt, r);
          cnt[0] = n;
          for (int w = 1; w < kSumWarps; ++w) cnt[w] = 0;
        }
      }
      cluster.sync();   // the peers' shared memory stays alive until rank 0 has read it
      if (rank != 0) return;
    }
    // block sums: one warp per block of the CTA, lane -> four dimensions
    if (warp < bpc && slice * bpc + warp < T) {
      const int I = slice * bpc + warp;
      float s[4] = {0.f, 0.f, 0.f, 0.f};
      int n = 0;
      for (int w = warp * share; w < (warp + 1) * share; ++w) {
#pragma unroll
        for (int e = 0; e < 4; ++e) s[e] += part[w][4 * lane + e];
        n += cnt[w];
      }
      __half2 o[2][2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float x = s[2 * e] * scale, y = s[2 * e + 1] * scale;
        o[0][e] = __floats2half2_rn(x, y);
        const float2 b = __half22float2(o[0][e]);
        o[1][e] = __floats2half2_rn(x - b.x, y - b.y);
      }
#pragma unroll
      for (int k = 0; k < 2; ++k)
        *reinterpret_cast<uint2*>(parts + k * part_stride + ((size_t)h * T + I) * kHeadDim + 4 * lane) =
            *reinterpret_cast<const uint2*>(o[k]);
      if (lane == 0) nz[(size_t)h * T + I] = n;
    }
  }
  if (tid < kHeadDim) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kSumWarps; ++w) s += part[w][tid];
    us[((size_t)h * nslices + slice) * kHeadDim + tid] = s;
  }
  if (tid == 0) {
    int n = 0;
#pragma unroll
    for (int w = 0; w < kSumWarps; ++w) n += cnt[w];
    nzs[(size_t)h * nslices + slice] = n;
  }
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// What a call of this shape needs between its two kernels.
struct SimPlan {
  int T, slices;
  size_t parts_bytes, nz_bytes, us_bytes, nzs_bytes;
  SimPlan(int heads, int L, int block) {
    T = (int)(((long long)L + block - 1) / block);
    const int bpc = blocks_per_cta(block);
    slices = (T + bpc - 1) / bpc;
    parts_bytes = align256((size_t)2 * heads * T * kHeadDim * 2);
    nz_bytes = align256((size_t)heads * T * 4);
    us_bytes = align256((size_t)heads * slices * kHeadDim * 4);
    nzs_bytes = align256((size_t)heads * slices * 4);
  }
  size_t bytes() const { return parts_bytes + nz_bytes + us_bytes + nzs_bytes; }
};

}  // namespace
}  // namespace mixkv

using namespace mixkv;

extern "C" {

int mixkv_similarity_workspace_size(int32_t heads, int32_t L, int32_t block, size_t* bytes) {
  if (!bytes || heads < 1 || L < 1 || block < 1) return MIXKV_ERR_INVALID_ARG;
  *bytes = SimPlan(heads, L, block).bytes();
  return MIXKV_OK;
}

int mixkv_similarity_map(const void* X, int32_t heads, int32_t L, int32_t head_dim, int32_t block,
                         void* workspace, size_t workspace_bytes, float* cells, float* mean_opt,
                         void* stream) {
  if (!X || !workspace || !cells || heads < 1 || L < 1 || block < 1) return MIXKV_ERR_INVALID_ARG;
  if (head_dim != kHeadDim) return MIXKV_ERR_UNSUPPORTED;
  if ((reinterpret_cast<uintptr_t>(X) & 15u) || (reinterpret_cast<uintptr_t>(workspace) & 15u))
    return MIXKV_ERR_INVALID_ARG;
  if (block > L) block = L;   // one block either way
  const SimPlan pl(heads, L, block);
  size_t need = 0;
  mixkv_similarity_workspace_size(heads, L, block, &need);
  if (workspace_bytes < need) return MIXKV_ERR_WORKSPACE_TOO_SMALL;
  if (pl.T > 65535 || heads > 65535) return MIXKV_ERR_UNSUPPORTED;   // grid limits
  {
    const int rc = device_check(nullptr);
    if (rc != MIXKV_OK) return rc;
  }
  cudaStream_t s = (cudaStream_t)stream;
  unsigned char* wsb = reinterpret_cast<unsigned char*>(workspace);
  uint16_t* parts = reinterpret_cast<uint16_t*>(wsb);
  const float scale = block == 1 ? 1.f : sum_scale(block);
  wsb += pl.parts_bytes;
  int* nz = reinterpret_cast<int*>(wsb);
  wsb += pl.nz_bytes;
  float* us = reinterpret_cast<float*>(wsb);
  wsb += pl.us_bytes;
  int* nzs = reinterpret_cast<int*>(wsb);
  // Long blocks of which there are too few to fill the GPU: a cluster of CTAs per block, as long as
  // every warp keeps a full share of 32 rows.
  int S = 1;
  while (S < kSumMaxCluster && (long long)heads * pl.slices * S < device_sm_count() &&
         (long long)2 * S * kSumWarps * kSumRows <= block)
    S *= 2;
  const dim3 grid((unsigned)(pl.slices * S), (unsigned)heads);
  const __nv_bfloat16* x = reinterpret_cast<const __nv_bfloat16*>(X);
  cudaError_t e;
  auto sums = [&](auto kernel) {
    return launch_pdl(kernel, grid, dim3(kSumThreads), 0, s, S, x, L, block, pl.T, scale, parts, nz, us, nzs);
  };
  if (sum_mode(block) == kRowsMany) e = sums(k_block_sums<kRowsMany, 0>);
  else switch (block) {
    case 1: e = sums(k_block_sums<kRowsOne, 1>); break;
    case 2: e = sums(k_block_sums<kRowsFew, 2>); break;
    case 4: e = sums(k_block_sums<kRowsFew, 4>); break;
    case 8: e = sums(k_block_sums<kRowsFew, 8>); break;
    case 16: e = sums(k_block_sums<kRowsFew, 16>); break;
    default: e = sums(k_block_sums<kRowsFew, 0>); break;
  }
  if (e != cudaSuccess) return MIXKV_ERR_CUDA;
  GramArgs g;
  g.parts = parts, g.inv_scale2 = 1.0f / (scale * scale), g.nz = nz, g.us = us, g.nzs = nzs, g.slices = pl.slices;
  g.heads = heads, g.L = L, g.block = block, g.T = pl.T, g.cells = cells, g.mean = mean_opt;
  return launch_gram(g, s) == cudaSuccess ? MIXKV_OK : MIXKV_ERR_CUDA;
}

}  // extern "C"
