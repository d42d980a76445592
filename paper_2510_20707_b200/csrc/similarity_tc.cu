// Second kernel of the redundancy analysis: the Gram matrix of the block sums on the tensor cores,
// cell (I, J) = u_I . u_J / pairs (similarity.cu leaves the scaled sums u as two fp16 parts, single rows as two bf16).
//
// u = hi + lo but for up to 2^-23 of a component, and u.u = hi.lo + lo.hi + hi.hi but for lo.lo, up to 2^-22 of a term and
// mostly 2^-24.  Both lie below what the accumulation in fp32 leaves, so the small products go first, while the sum is small:
// against 64 bits the cells of 32768 video keys in blocks of 16 are 3.5e-7 off (2-norm); with three bf16 parts, which hold all
// of fp32's bits, and six products in the order in which they came 1.34e-6.  Blocks of 2 to 4096 and text, random, sparse and
// cancelling rows: 1.8e-8 to 1.8e-6, never above what the three parts left.  (They moved half as many bytes again: 4 heads of
// 32768 rows in blocks of 16 30.5 us a call, now 25.4; of 20000 in blocks of 4 124, now 104.)
// Persistent CTAs walk a contiguous run of tiles (head, I, J): 128 blocks I on M, NT blocks J on N,
// only tiles that touch or lie right of the diagonal.  The parts of I stay in shared memory while
// J runs (2 x 32 KB), the parts of J go through a ring of four half parts, and two accumulator stages
// let the epilogue of a tile overlap the MMA of the next.
//
// What bounds it: the output, T x T x 4 bytes per head, once T is large: a tile and its mirror image leave
// as stores of 128 consecutive bytes of a row.
//
// NT = 128 where there are tiles enough for every SM, NT = 32 below that: a small map is one chain
// of load, MMA and store per CTA, and a quarter of the columns shortens all three.
#include <cuda.h>

#include "tc_common.cuh"

namespace mixkv {
namespace {

constexpr int kGThreads = 12 * 32;   // TMA, MMA, 2 head-mean, 8 epilogue warps
constexpr int kGEpiWarp0 = 4, kGEpiWarps = 8;
constexpr int kPartBytes = 128 * 256;   // one part of 128 blocks: two 64-column halves of 16 KB
constexpr int kParts = 2;
// Halves (64 columns) of one part of the blocks on N: one tile's worth.  Twice as many gain nothing, and with 64 KB less the
// next call's first kernel finds room beside this one (4 heads of 32768 rows in blocks of 16 26.8 us a call, now 25.4).
constexpr int kGStages = 4;

struct GBars {
  uint64_t afull, afree;
  uint64_t bfull[kGStages], bempty[kGStages];
  uint64_t tfull[2], tempty[2];
  uint64_t mmas;   // the issuer's last ones
  uint32_t tmem_base;
  int abort;
};

// Column tiles of tile row I: J starts at the diagonal (I * 128).
template <int NT>
__host__ __device__ __forceinline__ int row_tiles(const int T, const int I) {
  return (T - I * 128 + NT - 1) / NT;
}

// The tiles of one CTA, of `total` in (head, I, c) order; column tile c covers blocks I * 128 + c * NT ...  DEALT: runs of
// `run` tiles, dealt out in turn, else one contiguous share (see gram_run).
template <int NT, bool DEALT>
struct GramWalk {
  int id, hi, T, nT, h, I, c, nc, run, left;
  bool fresh;   // first tile of this CTA in its (head, I): the parts of I have to be loaded
  __device__ GramWalk(const int T_, const int per_head, const int total, const int run_)
      : T(T_), nT((T_ + 127) / 128), run(run_), left(run_) {
    id = DEALT ? (int)blockIdx.x * run : (int)((long long)total * blockIdx.x / gridDim.x);
    hi = DEALT ? total : (int)((long long)total * (blockIdx.x + 1) / gridDim.x);
    h = id / per_head;
    c = id - h * per_head;
    I = 0;
    nc = row_tiles<NT>(T, 0);
    while (c >= nc) row();
    fresh = true;
  }
  __device__ __forceinline__ void row() {   // c lies behind the end of row I
    c -= nc;
    fresh = true;
    if (++I == nT) {
      I = 0;
      ++h;
    }
    nc = row_tiles<NT>(T, I);
  }
  __device__ __forceinline__ bool valid() const { return id < hi; }
  // after this tile the parts of I are loaded again, if there is another tile
  __device__ __forceinline__ bool row_last() const { return id + 1 == hi || c + 1 == nc || (DEALT && left == 1); }
  __device__ __forceinline__ void next() {
    fresh = false;
    if (DEALT) {
      int ahead = 1;
      if (--left == 0) {
        ahead += ((int)gridDim.x - 1) * run;
        left = run;
        fresh = true;
      }
      id += ahead;
      c += ahead;
      while (c >= nc) row();
    } else {
      ++id;
      if (++c == nc) row();
    }
  }
};

// Mean over all ordered pairs i != j of a head (Eq. 4), by two warps that have nothing else to do: either takes
// every other slice, a lane four dimensions, and all loads of a round are in flight together: what a short call
// waits for is their round trips, not their bytes (4 heads of 32768 tokens, blocks of 256: 14.4 -> 13.4 us a call).
__device__ void head_mean(const float* __restrict__ us, const int* __restrict__ nzs, const int slices,
                          const int h, const int L, const int t, float4* half_sum, int* half_nz,
                          float* __restrict__ mean) {
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  int z = 0;
  const int w = t >> 5, lane = t & 31;
  const float4* row = reinterpret_cast<const float4*>(us + (size_t)h * slices * kHeadDim) + lane;
  constexpr int kDepth = 16;
  for (int k0 = w; k0 < slices; k0 += 2 * kDepth) {
    float4 v[kDepth];
#pragma unroll
    for (int k = 0; k < kDepth; ++k)
      v[k] = k0 + 2 * k < slices ? __ldcg(row + (size_t)(k0 + 2 * k) * (kHeadDim / 4))
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < kDepth; ++k) s.x += v[k].x, s.y += v[k].y, s.z += v[k].z, s.w += v[k].w;
  }
  for (int k = t; k < slices; k += 64) z += __ldcg(nzs + (size_t)h * slices + k);
  z = __reduce_add_sync(0xffffffffu, z);
  if (w == 1) {
    half_sum[lane] = s;
    if (lane == 0) *half_nz = z;
  }
  named_bar_sync(1, 64);
  if (w == 0) {
    const float4 o = half_sum[lane];
    s.x += o.x, s.y += o.y, s.z += o.z, s.w += o.w;
    double nn = (double)((s.x * s.x + s.y * s.y) + (s.z * s.z + s.w * s.w));
#pragma unroll
    for (int x = 16; x > 0; x >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, x);
    const double Ld = (double)L;
    if (lane == 0) mean[h] = L > 1 ? (float)((nn - (double)(z + *half_nz)) / (Ld * (Ld - 1.0))) : 0.f;
  }
  named_bar_sync(1, 64);
}

template <int NT, bool DEALT>
__global__ void __launch_bounds__(kGThreads, 1)
k_gram(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
       const int* __restrict__ nz, const float* __restrict__ us, const int* __restrict__ nzs,
       const int slices, const int H, const int L, const int block, const int T, const int per_head, const int run,
       const float inv_scale2, const uint32_t idesc, float* __restrict__ cells, float* __restrict__ mean) {
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* base =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
  constexpr int kBHalf = NT * 128;                      // half a part of the NT blocks on N
  unsigned char* sA = base;                             // both parts
  unsigned char* sB = sA + kParts * kPartBytes;              // kGStages x half a part
  float* sT = reinterpret_cast<float*>(sB + kGStages * kBHalf);   // [8 warps][32 x 32]
  GBars* bars = reinterpret_cast<GBars*>(sT + kGEpiWarps * 1024);
  __shared__ float4 half_sum[32];   // head means
  __shared__ int half_nz;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const GramWalk<NT, DEALT> walk(T, per_head, H * per_head, run);   // (divisions: ahead of the wait)
  volatile int* abort = &bars->abort;

  pdl_launch_dependents();
  if (tid == 0) {
    mbar_init(&bars->afull, 1);
    mbar_init(&bars->afree, 1);
    for (int s = 0; s < kGStages; ++s) {
      mbar_init(&bars->bfull[s], 1);
      mbar_init(&bars->bempty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars->tfull[s], 1);
      mbar_init(&bars->tempty[s], NT == 128 ? kGEpiWarps : 4);
    }
    mbar_init(&bars->mmas, 1);
    bars->abort = 0;
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc(&bars->tmem_base, 256);
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  pdl_wait();

  if (warp == 0) {
    // -------------------------------------------------------------------- TMA producer
    if (lane == 0) {
      int s = 0, ph = 1, rown = 0, it = 0;
      bool ok = true;
      for (GramWalk<NT, DEALT> w = walk; w.valid() && ok; w.next()) {
        if (w.fresh) {
          if (rown > 0 && !mbar_wait(&bars->afree, (rown - 1) & 1, abort)) break;
          mbar_expect_tx(&bars->afull, kParts * kPartBytes);
          for (int p = 0; p < kParts; ++p) {
            tma_load_3d(sA + p * kPartBytes, &tmA, 0, w.I * 128, p * H + w.h, &bars->afull);
            tma_load_3d(sA + p * kPartBytes + 16384, &tmA, 64, w.I * 128, p * H + w.h, &bars->afull);
          }
          ++rown;
        }
        for (int x = 0; x < 2 * kParts && ok; ++x) {   // both halves of the remainders, then of the values
          if (!mbar_wait(&bars->bempty[s], ph, abort)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&bars->bfull[s], kBHalf);
          tma_load_3d(sB + s * kBHalf, &tmB, (x & 1) * 64, w.I * 128 + w.c * NT, (x < 2 ? H : 0) + w.h, &bars->bfull[s]);
          if (++s == kGStages) s = 0, ph ^= 1;
          ++it;
        }
      }
      drain_ring(bars->bfull, kGStages, it);
      drain_ring(&bars->afull, 1, rown);
    }
  } else if (warp == 1) {
    // -------------------------------------------------------------------- MMA issuer
    {
      const uint32_t on = elect_one();
      const uint32_t a0 = umma_desc_lo(smem_u32(sA)), b0 = umma_desc_lo(smem_u32(sB));
      int s = 0, ph = 0, rown = 0, tile = 0;
      bool ok = true;
      for (GramWalk<NT, DEALT> w = walk; w.valid() && ok; w.next()) {
        if (w.fresh) {
          if (!mbar_wait(&bars->afull, rown & 1, abort)) break;
          ++rown;
        }
        const int ts = tile & 1, tph = (tile >> 1) & 1;
        if (!mbar_wait(&bars->tempty[ts], tph ^ 1, abort)) break;
        // part pa of I, half `half` of the contraction, times the half part of J in stage sb
        auto product = [&](const int pa, const int half, const int sb, const bool first) {
          const uint32_t oa = a0 + (uint32_t)(pa * (kPartBytes >> 4) + half * (16384 >> 4));
          const uint32_t ob = b0 + (uint32_t)sb * (kBHalf >> 4);
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            if (first && ks == 0) umma_f16_lo<0>(tmem + ts * 128, oa + ks * 2, ob + ks * 2, idesc, on);
            else umma_f16_lo<1>(tmem + ts * 128, oa + ks * 2, ob + ks * 2, idesc, on);
          }
        };
        int values0 = 0;   // stage of the values' first half
#pragma unroll
        for (int x = 0; x < 2 * kParts; ++x) {
          if (!mbar_wait(&bars->bfull[s], ph, abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          if (x < 2) {
            product(0, x, s, x == 0);   // hi.lo
            umma_commit(&bars->bempty[s], on);
          } else {
            product(1, x & 1, s, false);   // lo.hi
            if (x == 2) {
              values0 = s;
            } else {   // hi.hi
              product(0, 0, values0, false);
              umma_commit(&bars->bempty[values0], on);
              product(0, 1, s, false);
              umma_commit(&bars->bempty[s], on);
            }
          }
          if (++s == kGStages) s = 0, ph ^= 1;
        }
        umma_commit(&bars->tfull[ts], on);
        if (w.row_last()) umma_commit(&bars->afree, on);
        ++tile;
      }
      umma_commit(&bars->mmas, on);
      drain_ring(&bars->mmas, 1, 1);
    }
  } else if (warp < kGEpiWarp0) {
    // -------------------------------------------------------------------- head means
    if (mean)
      for (int h = blockIdx.x; h < H; h += gridDim.x)
        head_mean(us, nzs, slices, h, L, tid - 64, half_sum, &half_nz, mean);
  } else if (NT == 128 || warp < kGEpiWarp0 + 4) {
    // -------------------------------------------------------------------- epilogue
    // warp % 4 = TMEM lane quarter (32 blocks I of the tile), (warp - 4) / 4 = 64-column half.
    const int quarter = warp & 3, ch = (warp - kGEpiWarp0) >> 2;
    constexpr int kChunks = NT == 128 ? 2 : 1;
    float* st = sT + (warp - kGEpiWarp0) * 1024;
    const float inv_b = 1.0f / (float)block, last_n = (float)(L - (T - 1) * block);
    const bool rows16 = (T & 3) == 0 && (reinterpret_cast<uintptr_t>(cells) & 15) == 0;
    int tile = 0;
    for (GramWalk<NT, DEALT> w = walk; w.valid(); w.next()) {
      const int i0 = w.I * 128 + quarter * 32, i = i0 + lane;   // this thread's block I
      const bool last_i = i == T - 1;
      const float inv_i = last_i ? 1.0f / last_n : inv_b;
      const bool on_diag = w.c * NT < 128;    // inside the diagonal 128 x 128 tile: no mirrored store
      float* out = cells + (size_t)w.h * T * T;
      const int ts = tile & 1, tph = (tile >> 1) & 1;
      // A wait that runs out has no status word to go to: this tile's cells, and those of the CTA's tiles behind it (their
      // waits fail at once then), come out as NaN instead of whatever the map's memory held.
      const float inv_j = mbar_wait(&bars->tfull[ts], tph, abort) ? inv_b : __int_as_float(0x7fffffff);
      tc_fence_after();
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + ts * 128 + ch * 64;
#pragma unroll 1
      for (int k = 0; k < kChunks; ++k) {
        const int j0 = w.I * 128 + w.c * NT + ch * 64 + k * 32;   // first block J of the chunk
        uint32_t v[32];
        tmem_ld32(taddr + k * 32, v);
        tmem_ld_wait();
        tmem_ld_fence(v);
        if (k + 1 == kChunks) {   // the accumulator stage is read: the MMA may fill it again
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars->tempty[ts]);
        }
        if (j0 >= T || i0 >= T) continue;
        const float sc = inv_i * inv_j * inv_scale2;
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) * sc);
        if (j0 + 31 >= T - 1 || j0 == i0) {   // the last block, or cells of the diagonal
          const bool diag = j0 == i0;
          const float n = last_i ? last_n : (float)block, pairs = n * (n - 1.0f);
          // the pairs of a row with itself are left out: cosine 1 each
          const float own = pairs > 0.f ? 1.0f / pairs : 0.f;
          const float z = diag && i < T ? (float)nz[(size_t)w.h * T + i] : 0.f;
          const float fix = (float)block / last_n;   // columns of the last block
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            float x = __uint_as_float(v[j]);
            if (j0 + j == T - 1) x *= fix;
            if (diag && j == lane) x = (x * n * n - z) * own;
            v[j] = __float_as_uint(x);
          }
        }
        // The mirrored tile leaves straight from the registers, where 32 lanes hold 128 consecutive bytes of a row of
        // the map (turned in shared memory first, into 16-byte stores of four rows per instruction, 4 heads of 32768 rows
        // in blocks of 16 took 32.2 us a call, now 31.4).  The tile itself goes through a swizzled 32 x 32 tile in shared
        // memory (cell (i, j) of the chunk at word 4 ((j / 4) ^ (i & 7)) + j % 4 of row i) and leaves as 16-byte
        // stores, four rows of 128 bytes per instruction; where the rows of the map are not 16-byte aligned (a
        // caller's map need only be aligned to 4 bytes), or the chunk is cut by its edge, as 4-byte stores, one row
        // per instruction.
        const bool vec = rows16 && i0 + 32 <= T && j0 + 32 <= T;
        const int sub = lane >> 3, quad = lane & 7;   // row of a group of four, four columns of it
        if (!on_diag) {   // mirrored tile: rows J
          if (i < T) {
            float* p = out + (size_t)j0 * T + i;
            if (j0 + 32 <= T) {
#pragma unroll
              for (int j = 0; j < 32; ++j) p[(size_t)j * T] = __uint_as_float(v[j]);
            } else {
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (j0 + j < T) p[(size_t)j * T] = __uint_as_float(v[j]);
            }
          }
        }
        // the tile itself: rows I
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 32; j += 4)
          *reinterpret_cast<float4*>(st + lane * 32 + 4 * ((j >> 2) ^ (lane & 7))) =
              make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]), __uint_as_float(v[j + 2]),
                          __uint_as_float(v[j + 3]));
        __syncwarp();
        if (vec) {
          float* p = out + (size_t)(i0 + sub) * T + j0 + 4 * quad;
#pragma unroll
          for (int r = 0; r < 32; r += 4)
            *reinterpret_cast<float4*>(p + (size_t)r * T) =
                *reinterpret_cast<const float4*>(st + (r + sub) * 32 + 4 * (quad ^ ((r + sub) & 7)));
        } else if (j0 + lane < T) {
          float* p = out + (size_t)i0 * T + j0 + lane;
#pragma unroll
          for (int r = 0; r < 32; ++r)
            if (i0 + r < T) p[(size_t)r * T] = st[r * 32 + 4 * ((lane >> 2) ^ (r & 7)) + (lane & 3)];
        }
      }
      ++tile;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 256);
}

// Bytes of L2 on the current device.
long long device_l2_bytes() {
  static std::atomic<int> cached[kMaxDevices];
  const int dev = device_slot();
  int n = dev < 0 ? 0 : cached[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if (dev < 0 || !answered(cudaDeviceGetAttribute(&n, cudaDevAttrL2CacheSize, dev)) || n < 1) return 132644864;
    cached[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

// How the tiles are shared out: 0 contiguous (a CTA keeps its parts of I from tile to tile), else runs of so many in turn,
// so that all CTAs together write whole rows of the map at a time.  That counts where the map goes to HBM: it leaves L2
// in about the order in which it was written.  Contiguous / in runs, us, B200 (L2 of 133 MB), maps in turn on four inputs:
//   Rows that do not start on 32-byte sectors (T not a multiple of 8, or a map that does not): neighbouring tiles share
//   sectors, and a sector that leaves half written is read again.  Runs of one from half of L2 on: 8 heads x 1451 cells a side
//   (67 MB) in blocks of 1, 4, 16 43.5 / 38.8, 41.1 / 36.4, 41.4 / 41.0, 4 x 2101 (71 MB) 43.9 / 37.8, 41.9 / 35.4, 42.2 / 37.4,
//   4 x 2801 (126 MB) 66.5 / 54.3, 64.5 / 53.6, 64.6 / 54.3; below it 4 x 2001 (64 MB) 38.7 / 34.2, 36.4 / 31.6, 37.1 / 33.7,
//   4 x 1801 (52 MB) 34.8 / 34.1, 32.4 / 31.6, 32.7 / 33.1, 4 x 1501 (36 MB) 28.2 / 28.8, 25.8 / 26.5, 24.5 / 26.8.  (One map
//   written over and over stays in L2 and is better off contiguous up to 58 MB: 4 x 1901 32.2 / 34.0, 4 x 2001 35.5 / 34.2.)
//   Whole sectors: only the largest maps gain (pages of HBM filled in one go), from 9/4 of L2 on: single rows in runs of
//   one (4 x 4400, 310 MB, 86.4 / 83.7, x 5000 113 / 105), sums in runs of two (4 x 4400 89.0 / 84.3, x 5000 117 / 107,
//   x 5600 136 / 125; 4 x 4000, 256 MB, 73.9 / 72.3).
int gram_run(const int heads, const int T, const bool single_rows, const bool whole_sectors, const long long l2) {
  const long long bytes = 4LL * heads * T * T;
  if (!whole_sectors) return 2 * bytes > l2 ? 1 : 0;
  return 4 * bytes > 9 * l2 ? (single_rows ? 1 : 2) : 0;
}

template <int NT, bool DEALT>
cudaError_t launch_gram_t(const GramArgs& g, const long long per_head, const int run, cudaStream_t s) {
  static std::atomic<bool> done[kMaxDevices];
  const size_t smem = 1024 + (size_t)kParts * kPartBytes + (size_t)kGStages * NT * 128 +
                      (size_t)kGEpiWarps * 4096 + sizeof(GBars);
  const cudaError_t e = ensure_smem(k_gram<NT, DEALT>, smem, done);
  if (e != cudaSuccess) return e;
  const long long total = per_head * g.heads;
  if (total > 0x7fffffffLL) return cudaErrorInvalidValue;
  CUtensorMap tmA, tmB;
  const unsigned long long dims[3] = {(unsigned long long)kHeadDim, (unsigned long long)g.T,
                                      (unsigned long long)kParts * g.heads};
  const unsigned long long strides[2] = {(unsigned long long)kHeadDim * 2,
                                         (unsigned long long)g.T * kHeadDim * 2};
  const unsigned boxA[3] = {64, 128, 1}, boxB[3] = {64, (unsigned)NT, 1};
  if (!encode_map_16bit(&tmA, g.parts, 3, dims, strides, boxA) ||
      !encode_map_16bit(&tmB, g.parts, 3, dims, strides, boxB))
    return cudaErrorInvalidValue;
  const int grid = (int)(total < device_sm_count() ? total : device_sm_count());
  return launch_pdl(k_gram<NT, DEALT>, dim3((unsigned)grid), dim3(kGThreads), smem, s, 1, tmA, tmB, g.nz, g.us,
                    g.nzs, g.slices, g.heads, g.L, g.block, g.T, (int)per_head,
                    run, g.inv_scale2, g.block == 1 ? umma_idesc_bf16(128, NT) : umma_idesc_f16(128, NT), g.cells, g.mean);
}

template <int NT>
long long tiles_per_head(const int T) {
  long long n = 0;
  for (int I = 0; I < (T + 127) / 128; ++I) n += row_tiles<NT>(T, I);
  return n;
}

}  // namespace

cudaError_t launch_gram(const GramArgs& g, cudaStream_t s) {
  const long long wide = tiles_per_head<128>(g.T);
  const bool narrow = wide * g.heads < device_sm_count();
  const long long per_head = narrow ? tiles_per_head<32>(g.T) : wide;
  const bool whole_sectors = g.T % 8 == 0 && (reinterpret_cast<uintptr_t>(g.cells) & 31) == 0;
  const int run = narrow ? 0 : gram_run(g.heads, g.T, g.block == 1, whole_sectors, device_l2_bytes());
  return narrow ? launch_gram_t<32, false>(g, per_head, 0, s)
         : run  ? launch_gram_t<128, true>(g, per_head, run, s)
                : launch_gram_t<128, false>(g, per_head, 0, s);
}

}  // namespace mixkv

extern "C" int mixkv_internal_gram_run(int32_t heads, int32_t cells, int32_t parts, int32_t whole_sectors, int64_t l2_bytes) {
  return mixkv::gram_run(heads, cells, parts == 2, whole_sectors != 0, l2_bytes);
}
