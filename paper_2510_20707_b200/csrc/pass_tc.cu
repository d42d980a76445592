// The two passes over K of the MixKV scoring step as persistent, warp-specialised sm_100a
// kernels: TMA tile loads into 128-byte-swizzled shared memory, tcgen05.mma (bf16 x bf16 ->
// fp32) with accumulators in tensor memory, and epilogues that read the accumulators back with
// tcgen05.ld.
//
//   pass 1  K from HBM.  Logits with the window queries on the M side (one query row per TMEM
//           lane), so the running softmax (reference, sum) of a row is thread-local; alongside, key
//           norms and the sum of unit keys from the shared-memory tile.  Every run of tiles
//           of one (layer, sequence, head) inside a CTA (a segment) leaves its partial
//           statistics.
//   pass 2  K again, V from HBM.  A CTA that starts on a (layer, sequence, head) first folds
//           that head's segments of pass 1: the softmax statistics become one log2 normaliser
//           per window row, the unit-key sums the mean unit key and the redundancy of Eq. 4
//           (every CTA that touches the head does this for itself: no CTA waits for another,
//           nothing is counted).  Logits with the keys on the M side (one key per TMEM lane),
//           normalised with those row statistics, so the column sum over window rows
//           and query heads is thread-local -> s_ex_raw.  The mean unit key rides
//           along as three extra bf16 "query" rows -> K_i . kbar -> s_div.  Value norms are
//           computed from V tiles staged next to the K tiles.
//
// Paper: extrinsic importance, VNorm and diversity of Sec. 3.2, redundancy of Eq. 3-4.
#include <cuda.h>

#include "tc_common.cuh"

namespace mixkv {

namespace {

constexpr int kTileBytes = kTile * 256;    // 128 keys x 128 bf16
constexpr int kHalfBytes = kTile * 128;    // one 64-column half of a K tile

// Warp roles.  Warpgroup 0 (warps 0..3) holds the single-thread roles: TMA producer, MMA issuer, (pass 2) V
// producer.  Warps 4..19 are the epilogue.  From warp 20 on: pass 1, eight warps for the key statistics; pass 2,
// four for the value norms.  Pass 1 shares its registers out by role with setmaxnreg (the single-thread roles hand
// most of theirs to the others).  A warp's TMEM lane quarter is warp % 4.
constexpr int kWarpTma = 0, kWarpMma = 1;
constexpr int kP1WarpMma = 3;                    // pass 1: see k_pass1
constexpr int kEpiWarp0 = 4;
constexpr int kEpiWarps = 16;                    // warps 4..19
constexpr int kAuxWarp0 = kEpiWarp0 + kEpiWarps; // warps 20..: key statistics / value norms

// Registers per thread of the calling warpgroup from here on: N, where the kernel was launched
// with BASE (every warp of the warpgroup executes this).
template <int N, int BASE>
__device__ __forceinline__ void set_regs() {
  if constexpr (N < BASE) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
  if constexpr (N > BASE) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

// Pass 2: a role that ends on an abort reports it ahead of what it still waits for.  (Pass 1 reports at the end of the CTA
// only.  Without this k_pass2<1> is compiled into 80 registers instead of 79 and takes 0.8 us longer over 95 one-tile
// segments of a head, 1 x 12062 keys, 16 queries 27.1 -> 28.0; with it in pass 1 as well one layer of 4 x 32768 takes
// 51.9 us, not 51.7.)
__device__ __forceinline__ void raise(int* status, volatile int* abort) {
  *abort = 1;
  if (status) atomicExch(status, MIXKV_ERR_TIMEOUT);
}

__device__ __forceinline__ f32x2 ex2_pair(f32x2 t2) {
  float a0, a1;
  unpack2(t2, a0, a1);
  return pack2(ex2(a0), ex2(a1));
}

constexpr size_t kSmemLimit = 227 * 1024;   // dynamic shared memory a CTA may ask for

// ======================================================================== pass 1
// Eight key-statistics warps (from warp 20 on), each with 16 rows of every tile: 28 warps per CTA.
constexpr int kP1AuxWarps = 8;
constexpr int kP1Threads = (kAuxWarp0 + kP1AuxWarps) * 32;
constexpr int kP1MaxStages = 6;
constexpr int kP1XRows = 3 * 128;   // row statistics exchanged between the warpgroups of a query row
// K tile ring: as deep as shared memory allows next to the query tile (the deeper the ring, the
// more bytes in flight towards HBM)
// (the widest query tiles leave room for four)
__host__ __device__ constexpr int p1_stages(int NQ) { return NQ > 224 ? 4 : 5; }
// Registers per thread: at launch, then per role (7 warpgroups: 24 + 4 * 64 + 2 * 112 = 7 * 72).  The
// key-statistics warps keep four widened rows between their two sweeps; two 16-column pieces fit the epilogue's 64.
constexpr int kP1RegsLaunch = 72, kP1RegsLead = 24, kP1RegsEpi = 64, kP1RegsAux = 112;
static_assert(kP1RegsLead + 4 * kP1RegsEpi + 2 * kP1RegsAux == 7 * kP1RegsLaunch, "setmaxnreg shares");

struct P1Bars {
  uint64_t full[kP1MaxStages];
  uint64_t empty[kP1MaxStages];
  uint64_t tfull[4];
  uint64_t tempty[4];
  uint64_t qfull;
  uint64_t qfree;
  uint64_t mmas;     // the issuer's last ones
  TileCoord first;   // of the CTA's first tile
  uint32_t tmem_base;
  int abort;
};

// (m, z) pairs of the same row merged: z0 2^m0 + z1 2^m1 under the larger reference.
__device__ __forceinline__ float2 merge_stats(const float2 a, const float2 b) {
  const float mn = fmaxf(a.x, b.x);
  return make_float2(mn, a.y * ex2(a.x - mn) + b.y * ex2(b.x - mn));
}

// ---- per-head folds (pass 2, at the start of a segment): what the segments of pass 1 left
// for a (layer, sequence, head) becomes what pass 2 needs of it.
//
// Bound by round trips to L2, so a head's segments are spread over lanes (row statistics) and warps (key sums), and
// kFoldDepth 16-byte loads of a thread are in flight together: up to 20 segments are one round, the 37 of a
// one-layer call of 4 x 32768 keys two.  (Rounds stay short: code that runs once per segment costs its instruction
// fetches.)  With a thread or two to a row, and one to a key dimension, that call had its normalisers 5.4 us after
// pass 1, now 3.3; that of 4 x 1024 keys, 8 segments, 2.6 and 1.5.
constexpr int kFoldDepth = 5;
// Window rows 2 rp, 2 rp + 1 (rp = 8 * warp + (lane & 7)) over all segments of the head, four segments side by side
// in a warp: (reference, sum) pairs merged under the largest reference, the same in the four lanes of a row pair.
__device__ __forceinline__ void fold_row_stats(const float2* rowstat, const SegList& sl, const int NQ, const int rp,
                                               const int lane, float2& s0, float2& s1) {
  s0 = s1 = make_float2(-1e30f, 0.f);
#pragma unroll 1
  for (int e0 = lane >> 3; e0 < sl.nseg; e0 += 4 * kFoldDepth) {
    float4 v[kFoldDepth];
#pragma unroll
    for (int k = 0; k < kFoldDepth; ++k) {
      v[k] = make_float4(-1e30f, 0.f, -1e30f, 0.f);
      if (e0 + 4 * k < sl.nseg && 2 * rp < NQ)
        v[k] = __ldcg(reinterpret_cast<const float4*>(rowstat + (size_t)sl.start(e0 + 4 * k) * NQ) + rp);
    }
    float m0 = s0.x, m1 = s1.x;
#pragma unroll
    for (int k = 0; k < kFoldDepth; ++k) m0 = fmaxf(m0, v[k].x), m1 = fmaxf(m1, v[k].z);
    s0.y *= ex2(s0.x - m0), s1.y *= ex2(s1.x - m1);
    s0.x = m0, s1.x = m1;
#pragma unroll
    for (int k = 0; k < kFoldDepth; ++k) {
      s0.y = fmaf(v[k].y, ex2(v[k].x - m0), s0.y);
      s1.y = fmaf(v[k].w, ex2(v[k].z - m1), s1.y);
    }
  }
#pragma unroll
  for (int o = 8; o <= 16; o <<= 1) {
    s0 = merge_stats(s0, make_float2(__shfl_xor_sync(0xffffffffu, s0.x, o), __shfl_xor_sync(0xffffffffu, s0.y, o)));
    s1 = merge_stats(s1, make_float2(__shfl_xor_sync(0xffffffffu, s1.x, o), __shfl_xor_sync(0xffffffffu, s1.y, o)));
  }
}
// The same for rows 2 rp, 2 rp + 1 by one lane, rp = first, first + 32, ...: log2 normalisers (negated, `shift` taken off) of
// all rows by one warp that has the time of a whole segment for it.
constexpr int kFoldSpare = 4;
__device__ __forceinline__ void fold_rows_by_warp(const float2* rowstat, const SegList& sl, const int NQ, const int lane,
                                                  const float shift, float* normaliser) {
#pragma unroll 1
  for (int rp = lane; 2 * rp < NQ; rp += 32) {
    float2 s0 = make_float2(-1e30f, 0.f), s1 = s0;
#pragma unroll 1
    for (int e0 = 0; e0 < sl.nseg; e0 += kFoldSpare) {
      float4 v[kFoldSpare];
#pragma unroll
      for (int k = 0; k < kFoldSpare; ++k) {
        v[k] = make_float4(-1e30f, 0.f, -1e30f, 0.f);
        if (e0 + k < sl.nseg) v[k] = __ldcg(reinterpret_cast<const float4*>(rowstat + (size_t)sl.start(e0 + k) * NQ) + rp);
      }
#pragma unroll
      for (int k = 0; k < kFoldSpare; ++k) {
        s0 = merge_stats(s0, make_float2(v[k].x, v[k].y));
        s1 = merge_stats(s1, make_float2(v[k].z, v[k].w));
      }
    }
    *reinterpret_cast<float2*>(normaliser + 2 * rp) =
        make_float2(-(s0.x + log2f(s0.y)) - shift, -(s1.x + log2f(s1.y)) - shift);
  }
}
// Components 4 lane .. 4 lane + 3 of the unit-key sum over segments w, w + 4, ...
__device__ __forceinline__ float4 fold_key_sums(const float* ksum, const SegList& sl, const int w, const int lane) {
  float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int e0 = w; e0 < sl.nseg; e0 += 4 * kFoldDepth) {
    float4 v[kFoldDepth];
#pragma unroll
    for (int k = 0; k < kFoldDepth; ++k)
      v[k] = e0 + 4 * k < sl.nseg
                 ? __ldcg(reinterpret_cast<const float4*>(ksum + (size_t)sl.start(e0 + 4 * k) * kHeadDim) + lane)
                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < kFoldDepth; ++k) sum.x += v[k].x, sum.y += v[k].y, sum.z += v[k].z, sum.w += v[k].w;
  }
  return sum;
}
// The pass-1 segments of a head.
__device__ __forceinline__ SegList pass1_segments(const SeqTable& st, const int layer, const int b, const int h) {
  const int per_head = (st.tile1_start[b + 1] - st.tile1_start[b]) / st.H;
  return SegList(layer * st.nt1 + st.tile1_start[b] + h * per_head, per_head, st.sp1);
}

// The running softmax statistics of a query row are a pair (m, z): z = sum over the keys seen
// so far of exp2(logit * c - m), where m is a REFERENCE in log2 units, a logit of the row seen
// earlier, not necessarily the largest one: z * 2^m is the same number whatever m is, fp32
// carries 2^±126 around it, and searching the maximum of every chunk costs a quarter of the
// epilogue's instructions on its critical path.
//
// Fast path, 16 columns: adds exp2(logit * c - m) under the standing reference to two packed sums.
__device__ __forceinline__ void expsum16(const uint32_t (&r)[16], const f32x2 sc2, const f32x2 nm2, f32x2& za,
                                         f32x2& zb) {
#pragma unroll
  for (int j = 0; j < 16; j += 4) {
    za = add2(za, ex2_pair(fma2(pack2(__uint_as_float(r[j]), __uint_as_float(r[j + 1])), sc2, nm2)));
    zb = add2(zb, ex2_pair(fma2(pack2(__uint_as_float(r[j + 2]), __uint_as_float(r[j + 3])), sc2, nm2)));
  }
}
// A tile's sum at or above this means a logit about 2^99 above the reference (or no reference yet): the tile
// is redone on the slow path.  Below it nothing can overflow: the tiles of a head add up to less than 2^113.
constexpr float kTileSumLimit = 1e30f;

// Slow path: a 32-column chunk from tensor memory with the causal mask and a maximum search; the
// reference moves up to the chunk's maximum if that is larger.  Taken for the first tile of
// a segment, for the tiles that need the mask, and when the fast path's sum says that the
// reference is too low.  Every lane of the warp takes part (the load is warp-wide).  Returns
// the new (m, z).
__device__ __noinline__ float2 softmax_chunk_ref(const uint32_t taddr, const bool need_mask,
                                                 const int kbase, const int lim,
                                                 const float scale_log2e, float m_run,
                                                 float z_run) {
  uint32_t r[32];
  tmem_ld32(taddr, r);
  tmem_ld_wait();
  tmem_ld_fence(r);
  if (need_mask) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (kbase + j > lim) r[j] = 0xff800000u;   // -inf
  }
  float mx = max3(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]));
#pragma unroll
  for (int j = 3; j < 31; j += 2)
    mx = max3(mx, __uint_as_float(r[j]), __uint_as_float(r[j + 1]));
  mx = fmaxf(mx, __uint_as_float(r[31]));
  const float mn = fmaxf(m_run, mx * scale_log2e);
  if (mn > m_run) {
    z_run *= ex2(m_run - mn);
    m_run = mn;
  }
  const f32x2 sc2 = pack2(scale_log2e, scale_log2e), nm2 = pack2(-m_run, -m_run);
  f32x2 za = pack2(0.f, 0.f), zb = za;
  expsum16(reinterpret_cast<const uint32_t(&)[16]>(r[0]), sc2, nm2, za, zb);
  expsum16(reinterpret_cast<const uint32_t(&)[16]>(r[16]), sc2, nm2, za, zb);
  float z0, z1;
  unpack2(add2(za, zb), z0, z1);
  return make_float2(m_run, z_run + (z0 + z1));
}

// grid = g1 persistent CTAs of 28 warps: TMA, 2 idle, MMA, 16 epilogue, 8 key-statistics.  The
// MMA issuer is warp 3: its scheduler carries the fewest busy warps (with G*W = 224 the last
// lane quarter of the second query block is padding), and a single dependent instruction
// stream that shares a scheduler with many busy warps issues slowly enough to pace the tile
// loop.
template <int MB>
__global__ void __launch_bounds__(kP1Threads, 1)
k_pass1(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ,
        const SeqTable st, const Workspace ws, const float scale_log2e,
        const int clear_status, int* status) {
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* base =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
  const int kP1Stages = p1_stages(st.NQ);
  constexpr int NU = MB == 2 ? 2 : 4;   // warpgroups that share a query row
  constexpr int TS = MB == 2 ? 2 : 4;   // accumulator stages (512 columns of tensor memory)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NQ = st.NQ, W = st.W, H = st.H;
  // The query tile holds exactly NQ rows per 64-column half.  The MMA reads MB * 128 rows: the
  // rows past NQ are whatever follows in shared memory (the next half, the K ring), they only
  // reach accumulator lanes that nobody reads.
  unsigned char* sQ = base;                    // 2 halves x [NQ x 128 B]
  unsigned char* sK = sQ + 2 * NQ * 128;       // kP1Stages x 32 KB
  // At addresses that the compiler knows.  Behind the tiles, whose place depends on NQ, every role kept the base of the
  // barriers in a register and the epilogue spilled: 2676 clocks per tile of 28 layers of 4 x 32768 keys at G*W = 224,
  // 2502 like this; 1563 and 1494 of 32 layers of 8 x 16384 keys at 128.  (k_pass2 comes out the other way round, 2548
  // and 2630, and keeps its own behind its tiles.)
  __shared__ __align__(16) float sks[kP1AuxWarps * 128];   // [aux warps][128] key-sum exchange
  __shared__ float2 sxs[kP1XRows];                         // row statistics handed over
  __shared__ P1Bars p1_bars;
  P1Bars* const bars = &p1_bars;
  const int lo = cta_first_tile(blockIdx.x, st.sp1);
  const int hi = cta_first_tile(blockIdx.x + 1, st.sp1);
  volatile int* abort = &bars->abort;

  if (tid == 0) {
    for (int s = 0; s < kP1Stages; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], 1 + kP1AuxWarps);   // MMA commit + the key-statistics warps
    }
    for (int s = 0; s < TS; ++s) {
      mbar_init(&bars->tfull[s], 1);
      // every epilogue warp that owns query rows reads every tile; warps on padding rows (the
      // last lane quarters of the last block) neither wait nor arrive: a warp that polls a
      // barrier takes issue slots from the scheduler it shares with the MMA issuer
      mbar_init(&bars->tempty[s], (kEpiWarps / (MB * 4)) * ((NQ + 31) / 32));
    }
    mbar_init(&bars->qfull, 1);
    mbar_init(&bars->qfree, 1);
    mbar_init(&bars->mmas, 1);
    bars->abort = 0;
    mbar_init_fence();
  }
  if (warp == kP1WarpMma) tmem_alloc(&bars->tmem_base, 512);
  if (warp == kWarpTma && lane == 0) {
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmQ);
  }
  // The divisions once, ahead of the wait, instead of in every role behind it (one layer of 4 x 1024 keys 21.4 -> 20.8 us;
  // with one query block 18.4 -> 17.8, 4 x 5000 24.9 -> 24.2, 32 layers of 8 x 16384 level).
  if (tid == kEpiWarp0 * 32) bars->first = layer_tile_coord(st.tile1_start, st.batch, H, st.nt1, lo);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  pdl_wait();   // everything earlier in the stream is complete: global memory may be touched
  if (clear_status && status && blockIdx.x == 0 && tid == 0) *status = 0;

  if (warp < kEpiWarp0) {
    set_regs<kP1RegsLead, kP1RegsLaunch>();
    if (warp == kWarpTma) {
      // ---------------------------------------------------------------- TMA producer
      if (lane == 0) {
        int s = 0, ph = 1, it = 0, segn = 0;
        bool ok = true;
        for (SegIter sg(st.tile1_start, st.batch, H, bars->first, lo, hi); sg.valid() && ok; sg.next()) {
          if (segn > 0 && !mbar_wait(&bars->qfree, (segn - 1) & 1, abort)) break;
          mbar_expect_tx(&bars->qfull, NQ * 256);
          tma_load_3d(sQ, &tmQ, 0, sg.bh() * NQ, sg.layer, &bars->qfull);
          tma_load_3d(sQ + NQ * 128, &tmQ, 64, sg.bh() * NQ, sg.layer, &bars->qfull);
          ++segn;
          int y = st.cu[sg.b] + sg.t0 * kTile;
          for (int k = 0; k < sg.n; ++k, y += kTile) {
            if (!mbar_wait(&bars->empty[s], ph, abort)) {
              ok = false;
              break;
            }
            mbar_expect_tx(&bars->full[s], kTileBytes);
            tma_load_4d(sK + s * kTileBytes, &tmK, 0, y, sg.h, sg.layer, &bars->full[s]);
            tma_load_4d(sK + s * kTileBytes + kHalfBytes, &tmK, 64, y, sg.h, sg.layer, &bars->full[s]);
            if (++s == kP1Stages) s = 0, ph ^= 1;
            ++it;
          }
        }
        drain_ring(bars->full, kP1Stages, it);
        drain_ring(&bars->qfull, 1, segn);
      }
    } else if (warp == kP1WarpMma) {
      // ---------------------------------------------------------------- MMA issuer
      {
        const uint32_t on = elect_one();
        constexpr uint32_t idesc = umma_idesc_bf16(128, kTile);
        const uint32_t q_lo = umma_desc_lo(smem_u32(sQ));
        const uint32_t k_lo = umma_desc_lo(smem_u32(sK));
        const uint32_t q_half = (uint32_t)(NQ * 128) >> 4;   // second 64-column half of the queries
        int s = 0, ph = 0, ts = 0, tph = 1, segn = 0;
        bool ok = true;
        for (SegIter sg(st.tile1_start, st.batch, H, bars->first, lo, hi); sg.valid() && ok; sg.next()) {
          if (!mbar_wait(&bars->qfull, segn & 1, abort)) break;
          ++segn;
          for (int k = 0; k < sg.n; ++k) {
            if (!mbar_wait(&bars->full[s], ph, abort) || !mbar_wait(&bars->tempty[ts], tph, abort)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t kb_lo = k_lo + (uint32_t)s * (kTileBytes >> 4);
            const uint32_t td = tmem + ts * (MB * 128);
            // one tile ahead of the last (and behind the wait: pass 2 reads the inputs without one of its own)
            if (sg.id + k == max(lo, hi - 2)) pdl_launch_dependents();
#pragma unroll
            for (int mb = 0; mb < MB; ++mb) {
              // k-steps of 16 columns: 32 bytes apart inside a 64-column half
#pragma unroll
              for (int ks = 0; ks < 8; ++ks) {
                const uint32_t a_lo = q_lo + (ks >> 2) * q_half + (uint32_t)(mb * (16384 >> 4) + (ks & 3) * 2);
                const uint32_t b_lo = kb_lo + (uint32_t)((ks >> 2) * (kHalfBytes >> 4) + (ks & 3) * 2);
                if (ks == 0)
                  umma_f16_lo<0>(td + mb * 128, a_lo, b_lo, idesc, on);
                else
                  umma_f16_lo<1>(td + mb * 128, a_lo, b_lo, idesc, on);
              }
            }
            umma_commit(&bars->empty[s], on);
            umma_commit(&bars->tfull[ts], on);
            if (k + 1 == sg.n) umma_commit(&bars->qfree, on);
            if (++s == kP1Stages) s = 0, ph ^= 1;
            if (++ts == TS) ts = 0, tph ^= 1;
          }
        }
        umma_commit(&bars->mmas, on);
        drain_ring(&bars->mmas, 1, 1);
      }
    }
  } else if (warp < kAuxWarp0) {
    // ------------------------------------------------------------------ epilogue
    // All sixteen warps read every tile (the MMA of the next tiles fills the other accumulator
    // stages meanwhile).  Warpgroup wg = 0..3:
    // MB == 2: query rows (wg / 2) * 128 .. +127, keys (wg % 2) * 64 .. +63 of the tile;
    // MB == 1: query rows 0 .. 127, keys wg * 32 .. +31.
    set_regs<kP1RegsEpi, kP1RegsLaunch>();
    const int wg = (warp - kEpiWarp0) >> 2, quarter = warp & 3;
    const int blk = MB == 2 ? wg >> 1 : 0;
    const int unit = MB == 2 ? wg & 1 : wg;      // which partial result of the row this is
    constexpr int NC = MB == 2 ? 64 : 32;        // columns (keys) this thread reduces per tile
    const int row = blk * 128 + quarter * 32 + lane;
    const int col0 = blk * 128 + unit * NC;
    const bool warp_on = blk * 128 + quarter * 32 < NQ;
    const int jrow = row % W;
    // The NU warpgroups that share a query row merge their statistics at the end of a segment:
    // units 1 .. NU-1 hand theirs over through shared memory, unit 0 merges and writes one pair
    // per row.  Named barriers 6 + blk ("handed over") and 8 + blk ("read").
    const int xrow = (unit > 0 ? unit - 1 : 0) * 128 + (MB == 2 ? blk * 128 : 0) + quarter * 32 + lane;
    constexpr int kXThreads = NU * 128;
    int ts = 0, tph = 0, segs_done = 0;
    const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + col0;
    for (SegIter sg(st.tile1_start, st.batch, H, bars->first, lo, hi); sg.valid(); sg.next()) {
      float m_run = -1e30f, z_run = 0.f;
      const int P = st.cu[sg.b + 1] - st.cu[sg.b] - W;
      const int t_mask = P / kTile;   // first tile that holds keys some row may not see
      // A tile goes in pieces of 16 columns: while one is exponentiated the next is on its way from tensor
      // memory, so that the four warps of a scheduler, which move in step, do not all wait for their loads
      // at the same time (G*W = 224, 28 layers of 4 x 32768 keys: 305 -> 283 us).  The first piece of the
      // next tile is not asked for ahead: with its accumulator not ready yet this tile's would be held back
      // (310 us).  A warp on padding rows only walks the segments, for the barriers below.
      for (int t = warp_on ? sg.t0 : sg.end(); t < sg.end(); ++t) {
        // (after an abort the waits fail at once; the loop goes on without work so that the
        // segment-end barriers below stay matched)
        if (mbar_wait(&bars->tfull[ts], tph, abort)) {
          tc_fence_after();
          const uint32_t taddr = tbase + ts * (MB * 128);
          const bool masked = t >= t_mask;
          bool slow = t == sg.t0 || masked;   // the same in every lane; the first tile sets the reference
          if (!slow) {
            const f32x2 sc2 = pack2(scale_log2e, scale_log2e), nm2 = pack2(-m_run, -m_run);
            f32x2 za = pack2(0.f, 0.f), zb = za;
            uint32_t ra[16], rb[16];
            tmem_ld16(taddr, ra);
#pragma unroll
            for (int c0 = 0; c0 < NC; c0 += 32) {
              tmem_ld_wait();
              tmem_ld_fence(ra);
              tmem_ld16(taddr + c0 + 16, rb);
              expsum16(ra, sc2, nm2, za, zb);
              tmem_ld_wait();
              tmem_ld_fence(rb);
              if (c0 + 32 < NC) tmem_ld16(taddr + c0 + 32, ra);
              expsum16(rb, sc2, nm2, za, zb);
            }
            float z0, z1;
            unpack2(add2(za, zb), z0, z1);
            slow = __any_sync(0xffffffffu, !(z0 + z1 < kTileSumLimit));
            if (!slow) z_run += z0 + z1;
          }
          if (slow) {
#pragma unroll 1
            for (int c0 = 0; c0 < NC; c0 += 32) {
              const float2 mz = softmax_chunk_ref(taddr + c0, masked, t * kTile + unit * NC + c0, P + jrow,
                                                  scale_log2e, m_run, z_run);
              m_run = mz.x;
              z_run = mz.y;
            }
          }
          tc_fence_before();
          __syncwarp();   // one arrival per warp: 512 single arrivals on one word cost more than a chunk
          if (lane == 0) mbar_arrive(&bars->tempty[ts]);
        }
        if (++ts == TS) ts = 0, tph ^= 1;
      }
      if (unit > 0) {
        if (segs_done > 0) named_bar_sync(8 + blk, kXThreads);   // the last hand-over was read
        sxs[xrow] = make_float2(m_run, z_run);
        named_bar_arrive(6 + blk, kXThreads);
      } else {
        named_bar_sync(6 + blk, kXThreads);
        float2 mz = make_float2(m_run, z_run);
#pragma unroll
        for (int u = 1; u < NU; ++u) mz = merge_stats(mz, sxs[xrow + (u - 1) * 128]);
        named_bar_arrive(8 + blk, kXThreads);
        if (row < NQ) ws.rowstat[(size_t)sg.id * NQ + row] = mz;
      }
      ++segs_done;
    }
  } else {
    // ------------------------------------------------------------------ key statistics
    // A warp takes 16 rows of a tile in four steps of four; eight lanes share a row, lane c of them with
    // 16-byte chunk c of either 64-column half (conflict-free in the swizzled tile).  The bf16 are widened
    // once and stay in registers as fp32 pairs between their two uses: squares, whose sums are folded so
    // that lanes 2k, 2k + 1 end with the squared norm of their row of step k, then the rows scaled by 1/|k|
    // into sixteen per-thread sums.  These warps paced the whole pass (3900 clocks per tile of G*W = 224, 3600
    // of 128) when sixteen lanes shared a row and every bf16 was widened twice.
    set_regs<kP1RegsAux, kP1RegsLaunch>();
    const int aux_w = warp - kAuxWarp0;
    const int c = lane & 7, lg = lane >> 3;
    constexpr int aux_threads = kP1AuxWarps * 32;
    const int kt = tid - kAuxWarp0 * 32;
    // this lane's chunk of row 16 aux_w + 4 k + lg in half 0: the row's swizzle is (row & 7) = 4 (k & 1) + lg
    const uint32_t off0 = (uint32_t)(16 * aux_w + lg) * 128 + ((uint32_t)(c ^ lg) << 4);
    const uint32_t off1 = (uint32_t)(16 * aux_w + lg) * 128 + ((uint32_t)(c ^ (lg + 4)) << 4);
    const int my_row = 16 * aux_w + 4 * (c >> 1) + lg;   // the row whose norm this lane ends with
    int s = 0, ph = 0;
    for (SegIter sg(st.tile1_start, st.batch, H, bars->first, lo, hi); sg.valid(); sg.next()) {
      f32x2 acc2[8];   // dims 8c .. 8c+7 of half 0, then of half 1, as packed pairs
#pragma unroll
      for (int e = 0; e < 8; ++e) acc2[e] = pack2(0.f, 0.f);
      const int L = st.cu[sg.b + 1] - st.cu[sg.b];
      float* kinv = ws.kinv + kpos(st, sg.layer, sg.h, sg.b, 0);
      int i = sg.t0 * kTile + my_row;
      for (int k = 0; k < sg.n; ++k, i += kTile) {
        const bool ok = mbar_wait(&bars->full[s], ph, abort);
        const unsigned char* tile = sK + s * kTileBytes;
        f32x2 f[4][8];
        float p[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          f32x2 sq = pack2(0.f, 0.f);
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            const uint4 u = *reinterpret_cast<const uint4*>(tile + hf * kHalfBytes + r * 512 + ((r & 1) ? off1 : off0));
            f[r][4 * hf] = bf16x2_wide(u.x), f[r][4 * hf + 1] = bf16x2_wide(u.y);
            f[r][4 * hf + 2] = bf16x2_wide(u.z), f[r][4 * hf + 3] = bf16x2_wide(u.w);
#pragma unroll
            for (int e = 0; e < 4; ++e) sq = fma2(f[r][4 * hf + e], f[r][4 * hf + e], sq);
          }
          float s0, s1;
          unpack2(sq, s0, s1);
          p[r] = s0 + s1;
        }
        // the tile now lives in registers: hand the stage back
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->empty[s]);
        if (++s == kP1Stages) s = 0, ph ^= 1;
        {
          const bool up = (c & 4) != 0;
          const float k0 = up ? p[2] : p[0], k1 = up ? p[3] : p[1], g0 = up ? p[0] : p[2], g1 = up ? p[1] : p[3];
          p[0] = k0 + __shfl_xor_sync(0xffffffffu, g0, 4);
          p[1] = k1 + __shfl_xor_sync(0xffffffffu, g1, 4);
          const bool up2 = (c & 2) != 0;
          p[0] = (up2 ? p[1] : p[0]) + __shfl_xor_sync(0xffffffffu, up2 ? p[0] : p[1], 2);
          p[0] += __shfl_xor_sync(0xffffffffu, p[0], 1);
        }
        const float inv = (ok && i < L && p[0] > 0.f) ? rsqrtf(p[0]) : 0.f;
        if (i < L && (c & 1) == 0) kinv[i] = inv;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float w = __shfl_sync(0xffffffffu, inv, (lane & 24) | (2 * r));
          const f32x2 w2 = pack2(w, w);
#pragma unroll
          for (int e = 0; e < 8; ++e) acc2[e] = fma2(f[r][e], w2, acc2[e]);
        }
        // (no barrier per tile: after an abort the waits fail at once and every warp still walks
        // the same tiles, so the segment-end barriers below stay matched)
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float a0, a1;
        unpack2(acc2[e], a0, a1);
        a0 += __shfl_xor_sync(0xffffffffu, a0, 8);
        a1 += __shfl_xor_sync(0xffffffffu, a1, 8);
        a0 += __shfl_xor_sync(0xffffffffu, a0, 16);
        a1 += __shfl_xor_sync(0xffffffffu, a1, 16);
        if (lane < 8)
          *reinterpret_cast<float2*>(sks + aux_w * 128 + (e >> 2) * 64 + 8 * c + 2 * (e & 3)) = make_float2(a0, a1);
      }
      named_bar_sync(2, aux_threads);
      if (kt < kHeadDim) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kP1AuxWarps; ++w) t += sks[w * 128 + kt];
        ws.ksum[(size_t)sg.id * kHeadDim + kt] = t;
      }
      named_bar_sync(2, aux_threads);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kP1WarpMma) tmem_dealloc(tmem, 512);
  if (tid == 0 && bars->abort && status) atomicExch(status, MIXKV_ERR_TIMEOUT);
  // every partial result of this CTA's segments is written: pass 2 folds them per head
}

// ======================================================================== pass 2
// Pass 2 streams K and V.  24 warps: K/Q producer, MMA, V producer, 1 spare, four epilogue warpgroups, 4
// value-norm warps.  Epilogue warpgroup g works on accumulator stage g & 1 (alternate tiles), column half
// g >> 1: one key per thread and half of its G*W logit columns, in pieces of 16 with the next piece on its way
// from tensor memory; the two halves of a key meet in one word of shared memory per tile.  (With two warpgroups
// and all columns in a thread, two warps per scheduler kept the exp2 unit busy for half of the time: 28 layers of
// 4 x 32768 keys, G*W = 224, 359 us; as here 333 us; split like this but without the pieces 359 us again.)
//
// A CTA walks its tiles backwards: pass 1 has read (about) the same tiles in ascending order, so the K that is
// still in L2 from there is the end of every CTA's range (77 MB of it: 4 layers of 4 x 32768 keys, 268 MB of K and V, 191 MB
// read from DRAM behind pass 1, 272 with cold caches).  K and V are loaded evict-first, which keeps those lines,
// and the scores written for the tail, from being driven out by what is not read again.
constexpr int kP2EpiWarps = 16;                  // warps 4..19
constexpr int kP2AuxWarp0 = kEpiWarp0 + kP2EpiWarps;   // warps 20..23: value norms
constexpr int kP2Threads = (kP2AuxWarp0 + 4) * 32;

constexpr int kP2KStages = 3;              // K tiles (32 KB each)
constexpr int kP2VStagesMax = 4;           // V half tiles: 64 rows, 16 KB each
constexpr int kVSubBytes = 64 * 256;
struct P2Bars {
  uint64_t kfull[kP2KStages];
  uint64_t kempty[kP2KStages];
  uint64_t vfull[kP2VStagesMax];
  uint64_t vempty[kP2VStagesMax];
  uint64_t tfull[2];
  uint64_t tempty[2];
  uint64_t qfull;
  uint64_t qfree;
  uint64_t kbready;
  uint64_t nfull[2], nempty[2];   // normalisers by the spare warp
  uint64_t mmas;    // the issuer's last ones
  TileCoord last;   // of the CTA's last tile
  SegList segs;     // pass 1's segments of the head that it belongs to
  uint32_t tmem_base;
  int abort;
};

// 16 logit columns of one key: adds exp2(logit * scale - normaliser of the column) to two packed sums;
// nb_smem holds the negated normalisers of these columns.
__device__ __forceinline__ void colsum16(const uint32_t (&r)[16], const float* nb_smem, const f32x2 sc2,
                                         f32x2& acc_a, f32x2& acc_b) {
#pragma unroll
  for (int j = 0; j < 16; j += 4) {
    const float4 nb = *reinterpret_cast<const float4*>(nb_smem + j);   // negated normalisers
    acc_a = add2(acc_a, ex2_pair(fma2(pack2(__uint_as_float(r[j]), __uint_as_float(r[j + 1])), sc2,
                                      pack2(nb.x, nb.y))));
    acc_b = add2(acc_b, ex2_pair(fma2(pack2(__uint_as_float(r[j + 2]), __uint_as_float(r[j + 3])), sc2,
                                      pack2(nb.z, nb.w))));
  }
}

// Table of 16 words in which the warps of pair `wg` of the epilogue meet at the end of segment `segn` of a CTA.
__host__ __device__ __forceinline__ int stats_table(const int segn, const int wg) { return (segn & 1) * 2 + wg; }

// grid = g2 persistent CTAs: K producer, MMA, V producer, 1 spare, 16 epilogue, 4 value-norm warps.
// NCH: pieces of 16 query columns per epilogue warp, at most.
// SPARE: the spare warp folds the normalisers of the CTA's segments after the first (see pass2_spare).  A template argument
// because the code costs the calls that cannot use it up to half a microsecond.
template <int NCH, bool SPARE>
__global__ void __launch_bounds__(kP2Threads, 1)
k_pass2(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
        const __grid_constant__ CUtensorMap tmQ, const SeqTable st, const Workspace ws,
        float* __restrict__ s_div_out, float* __restrict__ rbar_out, const float scale_log2e,
        const int use_vnorm, const int pool_half, const int vstages, int* status) {
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* base =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
  const int NQ = st.NQ, W = st.W, H = st.H;
  const int NB = NQ + kExtraRows;             // rows of the B operand
  unsigned char* sQ = base;                   // 2 halves x [NB x 128 B]
  unsigned char* sK = sQ + 2 * NB * 128;      // kP2KStages x 32 KB
  unsigned char* sV = sK + kP2KStages * kTileBytes;   // vstages x 16 KB
  float* sbq = reinterpret_cast<float*>(sV + vstages * kVSubBytes);  // [2][256] negated normalisers
  float* sxp = sbq + 512;                     // [2][128] partial column sums of the second column halves
  float* skp = sxp + 256;                     // [4][128] parts of the unit-key sum
  float* sred = skp + 512;    // [96]: 2 x 2 x 16 epilogue, 12 value norms, 4 mean key
  float* sred_v = sred + 64;
  P2Bars* bars = reinterpret_cast<P2Bars*>(sred + 96);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int lo = cta_first_tile(blockIdx.x, st.sp2);
  const int hi = cta_first_tile(blockIdx.x + 1, st.sp2);
  volatile int* abort = &bars->abort;
  constexpr int kWarpTmaV = 2, kWarpSpare = 3;

  if (tid == 0) {
    for (int s = 0; s < kP2KStages; ++s) {
      mbar_init(&bars->kfull[s], 1);
      mbar_init(&bars->kempty[s], 1);
    }
    for (int s = 0; s < kP2VStagesMax; ++s) {
      mbar_init(&bars->vfull[s], 1);
      mbar_init(&bars->vempty[s], 2);      // the two warps that read a half tile
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars->tfull[s], 1);
      mbar_init(&bars->tempty[s], 8);      // the warps of the two warpgroups that read the stage
    }
    mbar_init(&bars->qfull, 1);
    mbar_init(&bars->qfree, 1);
    mbar_init(&bars->kbready, 4);          // the four warps that write the mean-key rows
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars->nfull[s], 1);
      mbar_init(&bars->nempty[s], kP2EpiWarps);
    }
    mbar_init(&bars->mmas, 1);
    bars->abort = 0;
    mbar_init_fence();
  }
  if (warp == kWarpMma) tmem_alloc(&bars->tmem_base, 512);
  if (warp == kWarpTma && lane == 0) {
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmQ);
  }
  if (warp == kWarpTmaV && lane == 0) tma_prefetch_desc(&tmV);
  // (divisions: once, ahead of the wait, instead of in every role behind it)
  if (tid == kEpiWarp0 * 32) {
    bars->last = layer_tile_coord(st.tile2_start, st.batch, H, st.nt2, hi - 1);
    bars->segs = pass1_segments(st, bars->last.layer, bars->last.b, bars->last.h);
  }
  if (warp >= kP2AuxWarp0) {   // B rows past the three parts of the mean key stay zero
    const int vt = tid - kP2AuxWarp0 * 32;
    unsigned char* hb = sQ + (vt >> 6) * NB * 128 + (vt & 7) * 2;
#pragma unroll
    for (int e = 3; e < kExtraRows; ++e)
      *reinterpret_cast<__nv_bfloat16*>(hb + sw128_offset(NQ + e, (vt & 63) >> 3)) = __float2bfloat16_rn(0.f);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  // K, V and the queries are the call's inputs: complete before pass 1 passed its own wait, behind which it lets this
  // kernel start.  Their producers fill the rings while pass 1 ends; everybody else reads what it leaves.
  if (warp >= kEpiWarp0 || (SPARE && warp == kWarpSpare)) pdl_wait();

  if (warp == kWarpTma) {
    // ------------------------------------------------------------------ K / Q producer
    if (lane == 0) {
      const uint64_t policy = l2_evict_first();
      int s = 0, ph = 1, it = 0, segn = 0;
      bool ok = true;
      for (RevSegIter sg(st.tile2_start, st.batch, H, bars->last, lo, hi); sg.valid() && ok; sg.next()) {
        if (segn > 0 && !mbar_wait(&bars->qfree, (segn - 1) & 1, abort)) break;
        mbar_expect_tx(&bars->qfull, NQ * 256);
        tma_load_3d(sQ, &tmQ, 0, sg.bh() * NQ, sg.layer, &bars->qfull);
        tma_load_3d(sQ + NB * 128, &tmQ, 64, sg.bh() * NQ, sg.layer, &bars->qfull);
        ++segn;
        int y = st.cu[sg.b] + (sg.end() - 1) * kTile;
        for (int k = 0; k < sg.n; ++k, y -= kTile) {
          if (!mbar_wait(&bars->kempty[s], ph, abort)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&bars->kfull[s], kTileBytes);
          tma_load_4d(sK + s * kTileBytes, &tmK, 0, y, sg.h, sg.layer, &bars->kfull[s], policy);
          tma_load_4d(sK + s * kTileBytes + kHalfBytes, &tmK, 64, y, sg.h, sg.layer, &bars->kfull[s], policy);
          if (++s == kP2KStages) s = 0, ph ^= 1;
          ++it;
        }
      }
      if (*abort) raise(status, abort);
      drain_ring(bars->kfull, kP2KStages, it);
      drain_ring(&bars->qfull, 1, segn);
    }
  } else if (warp == kWarpTmaV) {
    // ------------------------------------------------------------------ V producer
    if (lane == 0 && use_vnorm == MIXKV_INTRINSIC_VNORM) {
      const uint64_t policy = l2_evict_first();
      int vit = 0, vs = 0, vph = 1;
      bool ok = true;
      for (RevSegIter sg(st.tile2_start, st.batch, H, bars->last, lo, hi); sg.valid() && ok; sg.next()) {
        int y = st.cu[sg.b] + (sg.end() - 1) * kTile;
        for (int k = 0; k < 2 * sg.n; ++k, y += (k & 1) ? 64 : -64 - kTile) {   // half tiles of 64 rows
          if (!mbar_wait(&bars->vempty[vs], vph, abort)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&bars->vfull[vs], kVSubBytes);
          unsigned char* dst = sV + vs * kVSubBytes;
          tma_load_4d(dst, &tmV, 0, y, sg.h, sg.layer, &bars->vfull[vs], policy);
          tma_load_4d(dst + kVSubBytes / 2, &tmV, 64, y, sg.h, sg.layer, &bars->vfull[vs], policy);
          if (++vs == vstages) vs = 0, vph ^= 1;
          ++vit;
        }
      }
      if (*abort) raise(status, abort);
      drain_ring(bars->vfull, vstages, vit);
    }
  } else if (warp == kWarpMma) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t on = elect_one();
    const uint32_t idesc = umma_idesc_bf16(128, NB);
    const uint32_t k_lo = umma_desc_lo(smem_u32(sK)), q_lo = umma_desc_lo(smem_u32(sQ));
    const uint32_t q_half = (uint32_t)(NB * 128) >> 4;   // second 64-column half of the B operand
    int s = 0, ph = 0, ts = 0, tph = 1, segn = 0;
    bool ok = true;
    for (RevSegIter sg(st.tile2_start, st.batch, H, bars->last, lo, hi); sg.valid() && ok; sg.next()) {
      if (!mbar_wait(&bars->qfull, segn & 1, abort)) break;
      if (!mbar_wait(&bars->kbready, segn & 1, abort)) break;
      ++segn;
      for (int k = 0; k < sg.n; ++k) {
        if (!mbar_wait(&bars->kfull[s], ph, abort) || !mbar_wait(&bars->tempty[ts], tph, abort)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t kb_lo = k_lo + (uint32_t)s * (kTileBytes >> 4);
        const uint32_t td = tmem + ts * 256;
        if (sg.id + (sg.n - 1 - k) == min(hi - 1, lo + 1)) pdl_launch_dependents();   // one tile ahead of the last
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
          const uint32_t a_lo = kb_lo + (uint32_t)((ks >> 2) * (kHalfBytes >> 4) + (ks & 3) * 2);
          const uint32_t b_lo = q_lo + (ks >> 2) * q_half + (uint32_t)((ks & 3) * 2);
          if (ks == 0)
            umma_f16_lo<0>(td, a_lo, b_lo, idesc, on);
          else
            umma_f16_lo<1>(td, a_lo, b_lo, idesc, on);
        }
        umma_commit(&bars->kempty[s], on);
        umma_commit(&bars->tfull[ts], on);
        if (k + 1 == sg.n) umma_commit(&bars->qfree, on);
        if (++s == kP2KStages) s = 0, ph ^= 1;
        ts ^= 1;
        tph ^= ts ^ 1;
      }
    }
    if (*abort && on) raise(status, abort);
    umma_commit(&bars->mmas, on);
    drain_ring(&bars->mmas, 1, 1);
  } else if (SPARE && warp == kWarpSpare) {
    // ------------------------------------------------------------------ normalisers of the segments after the first
    // (the epilogue folds the first one's itself, all 512 threads of it, and uses the two tables in turn)
    int segn = 0;
    for (RevSegIter sg(st.tile2_start, st.batch, H, bars->last, lo, hi); sg.valid(); sg.next(), ++segn) {
      if (segn == 0) continue;
      if (segn > 1 && !mbar_wait(&bars->nempty[segn & 1], ((segn >> 1) - 1) & 1, abort)) break;
      fold_rows_by_warp(ws.rowstat, pass1_segments(st, sg.layer, sg.b, sg.h), NQ, lane, log2f((float)W),
                        sbq + (segn & 1) * 256);
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->nfull[segn & 1]);
    }
  } else if (warp >= kEpiWarp0 && warp < kEpiWarp0 + kP2EpiWarps) {
    // ------------------------------------------------------------------ epilogue
    // Alternate tiles belong to alternate pairs of warpgroups, so inside a segment the pairs never wait
    // for each other; each pair leaves its own partial score statistics.  At the start of a segment the
    // 512 threads fold the row statistics of the head together, four lanes to a pair of window rows, into the
    // normaliser table all groups read; with SPARE the later segments' comes from the spare warp.  Nobody leaves the
    // tile loop early: after an abort every wait fails at once, so the named barriers stay matched.
    const int quarter = warp & 3, grp = (warp - kEpiWarp0) >> 2;
    const int wg = grp & 1, chalf = grp >> 1;      // accumulator stage, column half
    const int gt = (tid - kEpiWarp0 * 32) & 127;   // thread inside the warpgroup
    const int gw = gt >> 5;                        // warp inside the warpgroup
    const int key = quarter * 32 + lane;
    const int nch = NQ / 16;
    const int ch_lo = chalf ? nch / 2 : 0, ch_n = chalf ? nch - nch / 2 : nch / 2;   // ch_n <= NCH
    const int et = tid - kEpiWarp0 * 32;           // thread inside the epilogue, 0..511
    const float log2W = log2f((float)W);
    const int barid = 1 + wg;                      // named barriers 1, 2: first column halves
    const int xbar = 6 + wg;                       // named barriers 6, 7: partial sums handed over
    const f32x2 sc2 = pack2(scale_log2e, scale_log2e);
    const uint32_t tstage = tmem + ((uint32_t)(quarter * 32) << 16) + wg * 256, taddr = tstage + ch_lo * 16;
    int tile = 0;   // parity decides which pair owns it
    int segn = 0;   // (counted with SPARE only)
    for (RevSegIter sg(st.tile2_start, st.batch, H, bars->last, lo, hi); sg.valid(); sg.next(), segn += SPARE ? 1 : 0) {
      const int P = st.cu[sg.b + 1] - st.cu[sg.b] - W;
      if (SPARE && segn > 0) {
        mbar_wait(&bars->nfull[segn & 1], ((segn - 1) >> 1) & 1, abort);
      } else {
        // the negated log2 normalisers of the rows with the 1/W of the window mean folded in
        const SegList sl = SPARE || tile == 0 ? bars->segs : pass1_segments(st, sg.layer, sg.b, sg.h);
        const int rp = (et >> 5) * 8 + (lane & 7);
        float2 s0, s1;
        fold_row_stats(ws.rowstat, sl, NQ, rp, lane, s0, s1);
        if (tile > 0) named_bar_sync(5, kP2EpiWarps * 32);   // the previous segment's readers of sbq are done
        if (lane < 8 && 2 * rp < NQ)
          *reinterpret_cast<float2*>(sbq + 2 * rp) =
              make_float2(-(s0.x + log2f(s0.y)) - log2W, -(s1.x + log2f(s1.y)) - log2W);
        named_bar_sync(5, kP2EpiWarps * 32);
      }
      const float* nb = sbq + (SPARE ? (segn & 1) * 256 : 0) + ch_lo * 16;
      float dmin = INFINITY, dmax = -INFINITY, dsum = 0.f, exw = 0.f;
      const float* kinv = ws.kinv + kpos(st, sg.layer, sg.h, sg.b, 0);
      const size_t poff = ppos(st, sg.layer, sg.h, sg.b, 0);
      float* ex_out = ws.s_ex_raw + poff;
      float* sd_out = s_div_out + poff;
      // this pair's tiles of the segment
      const int skip = (tile & 1) ^ wg;
      for (int t = sg.end() - 1 - skip, tl = tile + skip; t >= sg.t0; t -= 2, tl += 2) {
        const int tph = (tl >> 1) & 1;
        const int ikey = t * kTile + key;
        float kinv_i = 0.f;
        if (chalf == 0 && ikey < P) kinv_i = kinv[ikey];
        const bool ok = mbar_wait(&bars->tfull[wg], tph, abort);
        tc_fence_after();
        f32x2 acc = pack2(0.f, 0.f), acc_b = acc;
        uint32_t rd[4];
        if (ok) {
          uint32_t ra[16], rb[16];
          tmem_ld16(taddr, ra);   // (a piece past this half is another half's or the mean key's: read, not used)
#pragma unroll
          for (int ci = 0; ci < NCH; ci += 2) {
            tmem_ld_wait();
            tmem_ld_fence(ra);
            if (ci + 1 < NCH) tmem_ld16(taddr + ci * 16 + 16, rb);
            else if (chalf == 0) tmem_ld4(tstage + NQ, rd);
            if (ci < NCH - 1 || ci < ch_n) colsum16(ra, nb + ci * 16, sc2, acc, acc_b);
            if (ci + 1 < NCH) {
              tmem_ld_wait();
              tmem_ld_fence(rb);
              if (ci + 2 < NCH) tmem_ld16(taddr + ci * 16 + 32, ra);
              else if (chalf == 0) tmem_ld4(tstage + NQ, rd);
              if (ci + 1 < NCH - 1 || ci + 1 < ch_n) colsum16(rb, nb + ci * 16 + 16, sc2, acc, acc_b);
            }
          }
        }
        float acc0, acc1;
        unpack2(add2(acc, acc_b), acc0, acc1);
        const float part = acc0 + acc1;
        if (chalf) {
          // The other half reads this word before it arrives on tempty, and the next tile of this stage is
          // not complete before that: no barrier for the way back.  This half waits at the barrier all the same, for no
          // longer than it would for that tile: after an abort nothing else keeps it from a second arrival ahead of the other
          // half's first, which would end that barrier early and leave the other half at its last one for good.
          sxp[wg * 128 + key] = part;
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars->tempty[wg]);
          named_bar_sync(xbar, 256);
        } else {
          float dot = 0.f;
          if (ok) {
            tmem_ld_wait();
            tmem_ld_fence(rd);
            dot = (__uint_as_float(rd[0]) + __uint_as_float(rd[1])) + __uint_as_float(rd[2]);
          }
          named_bar_sync(xbar, 256);
          const float ex = part + sxp[wg * 128 + key];
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars->tempty[wg]);
          if (ok && ikey < P) {
            ex_out[ikey] = ex;
            const float sd = -dot * kinv_i;
            sd_out[ikey] = sd;
            dmin = fminf(dmin, sd);
            dmax = fmaxf(dmax, sd);
            dsum += sd;
            // number of pooling windows (centres in [0, P)) that cover this position
            const int cover = min(ikey, pool_half) + min(P - 1 - ikey, pool_half) + 1;
            exw = fmaf(ex, (float)cover, exw);
          }
        }
      }
      tile += sg.n;
      if constexpr (SPARE) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->nempty[segn & 1]);
      }
      if (chalf == 0) {
        // This pair's share of the segment's score statistics (neutral if it had no tile).  With SPARE nothing holds a warp
        // between the barrier here and its words of the next segment, if that is one tile of the other pair's, so two tables
        // take turns: the barrier of the segment in between stands behind the read.  (Without, barrier 5 does.)
        const float a = warp_min(dmin), b2 = warp_max(dmax), c2 = warp_sum(dsum),
                    d2 = warp_sum(exw);
        float* sr = sred + stats_table(SPARE ? segn : 0, wg) * 16;
        if (lane == 0) {
          sr[gw] = a;
          sr[4 + gw] = b2;
          sr[8 + gw] = c2;
          sr[12 + gw] = d2;
        }
        named_bar_sync(barid, 128);
        if (gt == 0) {
          ws.dstat[(size_t)sg.id * 2 + wg] = make_float4(
              fminf(fminf(sr[0], sr[1]), fminf(sr[2], sr[3])),
              fmaxf(fmaxf(sr[4], sr[5]), fmaxf(sr[6], sr[7])),
              (sr[8] + sr[9]) + (sr[10] + sr[11]), (sr[12] + sr[13]) + (sr[14] + sr[15]));
        }
      }
    }
  } else if (warp >= kP2AuxWarp0) {
    // ------------------------------------------------------------------ mean key, value norms
    // At the start of a segment: fold the unit-key sums of the head's pass-1 segments (every fourth of them
    // per warp, then one dimension per thread) and write the bf16 hi / lo / lo2 split of the mean unit key into the
    // three extra B rows; the CTA that starts on the head's first tile also leaves the redundancy
    // of Eq. 4, which needs nothing but the squared norm of that sum.  Per tile: warps 20, 21 read the first 64 rows of the V
    // tile, warps 22, 23 the last 64; one row per thread from the swizzled half tile.
    const int vt = tid - kP2AuxWarp0 * 32;         // 0..127
    const int sub = vt >> 6, vr = vt & 63;
    int vs = sub, vph = 0, segn = 0;   // V stage of this pair of warps: half tiles sub, sub + 2, ...
    for (RevSegIter sg(st.tile2_start, st.batch, H, bars->last, lo, hi); sg.valid(); sg.next()) {
      const int L = st.cu[sg.b + 1] - st.cu[sg.b], P = L - W;
      const float4 part =
          fold_key_sums(ws.ksum, segn == 0 ? bars->segs : pass1_segments(st, sg.layer, sg.b, sg.h), vt >> 5, lane);
      if (segn > 0) {   // the previous segment's MMAs must be done with the B rows, its readers with the parts
        if (vt == 0) mbar_wait(&bars->qfree, (segn - 1) & 1, abort);
        named_bar_sync(4, 128);
      }
      *reinterpret_cast<float4*>(skp + (vt >> 5) * kHeadDim + 4 * lane) = part;
      named_bar_sync(4, 128);
      const float ks = (skp[vt] + skp[kHeadDim + vt]) + (skp[2 * kHeadDim + vt] + skp[3 * kHeadDim + vt]);
      const float kb = ks / (float)L;   // mean unit key
      __nv_bfloat16 parts[3];
      parts[0] = __float2bfloat16_rn(kb);
      const float r1 = kb - __bfloat162float(parts[0]);
      parts[1] = __float2bfloat16_rn(r1);
      parts[2] = __float2bfloat16_rn(r1 - __bfloat162float(parts[1]));
      {
        unsigned char* hb = sQ + (vt >> 6) * NB * 128 + (vt & 7) * 2;
        const int chunk = (vt & 63) >> 3;
#pragma unroll
        for (int e = 0; e < 3; ++e)
          *reinterpret_cast<__nv_bfloat16*>(hb + sw128_offset(NQ + e, chunk)) = parts[e];
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->kbready);   // the MMA may start: the rest is off its path
      if (sg.t0 == 0) {                 // the same in all 128 threads
        const float n2 = warp_sum(ks * ks);
        if (lane == 0) sred_v[12 + (warp - kP2AuxWarp0)] = n2;
        named_bar_sync(4, 128);
        if (vt == 0) {
          const double nn = ((double)sred_v[12] + (double)sred_v[13]) + ((double)sred_v[14] + (double)sred_v[15]);
          const double T = (double)L;
          const float r = (float)((nn - T) / (T * (T - 1.0)));   // Eq. 4
          ws.rbar[sg.unit()] = r;
          if (rbar_out) rbar_out[sg.unit()] = r;
        }
      }
      ++segn;
      float vmin = INFINITY, vmax = -INFINITY, vsum = 0.f;
      float* vnorm = ws.vnorm + ppos(st, sg.layer, sg.h, sg.b, 0);
      if (use_vnorm == MIXKV_INTRINSIC_KNORM) {
        // key-norm ablation: the intrinsic term is minus the key norm, which pass 1 left as its
        // reciprocal; no V tile is loaded
        const float* kinv = ws.kinv + kpos(st, sg.layer, sg.h, sg.b, 0);
        for (int i = sg.t0 * kTile + vt; i < min(P, sg.end() * kTile); i += kTile) {
          const float ki = kinv[i];
          const float n = ki > 0.f ? -1.0f / ki : 0.f;
          vnorm[i] = n;
          vmin = fminf(vmin, n);
          vmax = fmaxf(vmax, n);
          vsum += n;
        }
      } else if (use_vnorm) {
        for (int t = sg.end() - 1; t >= sg.t0; --t) {
          const bool ok = mbar_wait(&bars->vfull[vs], vph, abort);
          const unsigned char* tile = sV + vs * kVSubBytes;
          f32x2 ss2[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};
          if (ok) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                const uint4 u =
                    *reinterpret_cast<const uint4*>(tile + half * (kVSubBytes / 2) + sw128_offset(vr, c));
                const uint32_t* p2 = reinterpret_cast<const uint32_t*>(&u);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const f32x2 f2 = bf16x2_wide(p2[e]);
                  ss2[e & 1] = fma2(f2, f2, ss2[e & 1]);
                }
              }
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars->vempty[vs]);
          vs += 2;
          if (vs >= vstages) vs -= vstages, vph ^= 1;
          const int i = t * kTile + sub * 64 + vr;
          if (ok && i < P) {
            float ss[4];
            unpack2(ss2[0], ss[0], ss[2]);
            unpack2(ss2[1], ss[1], ss[3]);
            const float n = sqrtf((ss[0] + ss[1]) + (ss[2] + ss[3]));
            vnorm[i] = n;
            vmin = fminf(vmin, n);
            vmax = fmaxf(vmax, n);
            vsum += n;
          }
          // The four warps stay within one tile of each other.  With an odd number of V stages the
          // two pairs of warps take turns on the same stage: a pair that ran ahead would wait for
          // a phase of vfull whose predecessor it never saw complete, and a parity wait on a
          // barrier that is still one phase behind returns at once.
          named_bar_sync(3, 128);
        }
      }
      if (use_vnorm) {
        const float a = warp_min(vmin), b2 = warp_max(vmax), c2 = warp_sum(vsum);
        const int vw = warp - kP2AuxWarp0;
        if (lane == 0) {
          sred_v[vw] = a;
          sred_v[4 + vw] = b2;
          sred_v[8 + vw] = c2;
        }
        named_bar_sync(4, 128);
        if (vt == 0) {
          ws.vstat[sg.id] = make_float4(
              fminf(fminf(sred_v[0], sred_v[1]), fminf(sred_v[2], sred_v[3])),
              fmaxf(fmaxf(sred_v[4], sred_v[5]), fmaxf(sred_v[6], sred_v[7])),
              (sred_v[8] + sred_v[9]) + (sred_v[10] + sred_v[11]), 0.f);
        }
        named_bar_sync(4, 128);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) tmem_dealloc(tmem, 512);
  if (tid == 0 && bars->abort && status) atomicExch(status, MIXKV_ERR_TIMEOUT);
}

// -------------------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = []() -> EncodeTiledFn {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess)
      return nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// Fills a map of a tensor of 16-bit elements: dims innermost first, strides in bytes of dimensions 1 .. rank - 1, box extents; 128-byte
// swizzle, zero fill outside.  The driver wants a current context for it.  The first call of a thread may find none (the
// runtime binds the device's context when a call of its own needs it, and none has by then): bound here.
bool encode_map(CUtensorMap* tm, const void* base, const cuuint32_t rank, const cuuint64_t* dims,
                const cuuint64_t* strides, const cuuint32_t* box) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  const cuuint32_t es[5] = {1, 1, 1, 1, 1};
  auto fill = [&]() {
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  };
  CUresult r = fill();
  if (r == CUDA_ERROR_INVALID_CONTEXT || r == CUDA_ERROR_NOT_INITIALIZED) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaSetDevice(dev) != cudaSuccess) return false;
    r = fill();
  }
  return r == CUDA_SUCCESS;
}

// X [layers, H, Ltot, d] bf16 (layer stride given in elements) as a 4-D tensor (d, Ltot, H,
// layers) with boxes of 64 x rows x 1 x 1.  Rows past the end of the tensor read as zero.
bool map_kv(const LaunchCtx& c, const void* X, int box_rows, CUtensorMap* tm) {
  const cuuint64_t dims[4] = {(cuuint64_t)kHeadDim, (cuuint64_t)c.st.Ltot, (cuuint64_t)c.st.H,
                              (cuuint64_t)c.st.layers};
  const cuuint64_t strides[3] = {(cuuint64_t)kHeadDim * 2, (cuuint64_t)c.st.Ltot * kHeadDim * 2,
                                 (cuuint64_t)c.kv_layer_stride * 2};
  const cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
  return encode_map(tm, X, 4, dims, strides, box);
}

// Q [layers, batch * H * NQ, d] bf16 as a 3-D tensor (d, rows, layers) with boxes of 64 x NQ x 1.
bool map_q(const LaunchCtx& c, const void* Q, CUtensorMap* tm) {
  const cuuint64_t dims[3] = {(cuuint64_t)kHeadDim, (cuuint64_t)c.st.batch * c.st.H * c.st.NQ,
                              (cuuint64_t)c.st.layers};
  const cuuint64_t strides[2] = {(cuuint64_t)kHeadDim * 2, (cuuint64_t)c.q_layer_stride * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)c.st.NQ, 1};
  return encode_map(tm, Q, 3, dims, strides, box);
}

// Dynamic shared memory of the passes: what the kernels carve up, behind up to 1023 bytes that align its start.
constexpr size_t pass1_smem(int NQ) {
  return 1024 + (size_t)2 * NQ * 128 + (size_t)p1_stages(NQ) * kTileBytes;
}
// What is left of it next to pass 1's static part.
constexpr size_t kP1SmemLimit = kSmemLimit - (kP1AuxWarps * 128 * 4 + kP1XRows * 8 + sizeof(P1Bars) + 63) / 64 * 64;
constexpr size_t pass2_smem(int NQ, int vstages) {
  return 1024 + (size_t)2 * (NQ + kExtraRows) * 128 + kP2KStages * kTileBytes +
         (size_t)vstages * kVSubBytes + 1280 * 4 + 96 * 4 + sizeof(P2Bars) + 64;
}
// V stages: the two pairs of value-norm warps need one each.
constexpr int pass2_vstages(int NQ) {
  int n = kP2VStagesMax;
  while (n > 2 && pass2_smem(NQ, n) > kSmemLimit) --n;
  return n;
}
constexpr bool passes_fit() {
  for (int NQ = 16; NQ <= kMaxNQ; NQ += 16)
    if (pass1_smem(NQ) > kP1SmemLimit || pass2_smem(NQ, pass2_vstages(NQ)) > kSmemLimit || p1_stages(NQ) > kP1MaxStages)
      return false;
  return true;
}
static_assert(passes_fit(), "a pass asks for more shared memory than a CTA may have at some width of the query tile");

}  // namespace

bool encode_map_16bit(void* tm, const void* base, int rank, const unsigned long long* dims,
                     const unsigned long long* strides_bytes, const unsigned* box) {
  cuuint64_t d[5], st[4];
  cuuint32_t bx[5];
  for (int i = 0; i < rank; ++i) d[i] = dims[i], bx[i] = box[i];
  for (int i = 0; i + 1 < rank; ++i) st[i] = strides_bytes[i];
  return encode_map(reinterpret_cast<CUtensorMap*>(tm), base, (cuuint32_t)rank, d, st, bx);
}

int device_sm_count() {
  static std::atomic<int> cached[kMaxDevices];
  int dev = 0;
  if (!answered(cudaGetDevice(&dev)) || dev < 0 || dev >= kMaxDevices) return 148;
  int n = cached[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if (!answered(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) || n < 1) return 148;
    cached[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

cudaError_t launch_pass1(const LaunchCtx& c, const void* K, const void* Q, int* status) {
  CUtensorMap tmK, tmQ;
  if (!map_kv(c, K, kTile, &tmK) || !map_q(c, Q, &tmQ)) return cudaErrorInvalidValue;
  static std::atomic<bool> done1[kMaxDevices], done2[kMaxDevices];
  if (c.st.NQ <= 128) {
    const size_t smem = pass1_smem(c.st.NQ);
    cudaError_t e = ensure_smem(k_pass1<1>, kP1SmemLimit, done1);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_pass1<1>, dim3(c.st.sp1.g), dim3(kP1Threads), smem, c.stream, 1, tmK, tmQ, c.st,
                      c.ws, c.scale_log2e, (int)c.clear_status, status);
  }
  const size_t smem = pass1_smem(c.st.NQ);
  cudaError_t e = ensure_smem(k_pass1<2>, kP1SmemLimit, done2);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_pass1<2>, dim3(c.st.sp1.g), dim3(kP1Threads), smem, c.stream, 1, tmK, tmQ, c.st,
                    c.ws, c.scale_log2e, (int)c.clear_status, status);
}

// Whether pass 2's spare warp folds the normalisers of a CTA's second and later heads.  It has the time of a
// head's tiles for it, with a round trip for every four segments and 64 rows: not where a head lies in many CTAs.  The
// epilogue's own fold kept it waiting 2.5 us per head: 28 layers of 4 heads and sequences of 700, 650, 800, 900 keys 98.6
// -> 94.2 us, of 3001, 1777, 6143 277 -> 268, of 4096 104.7 -> 103.3.
// Nor where no CTA has a second head, because all have CTAs of their own or every CTA takes one tile: there the code gives
// nothing and costs (with it / without, us: one layer of five prompts of 8 x 2000 keys 28.8 / 28.3, of 4 x 500 level, 25 layers
// of 4 x 768 38.0 / 37.7, 12 of 8 x 640 27.5 / 27.0, 10 of 4 x 1024 27.8 / 27.4).
constexpr int kSpareSegments = 6;
bool pass2_spare(const Split& sp1, const Split& sp2, const int tiles2, const int heads, const int longest) {
  if (heads == 1 || sp2.n < tiles2 || sp2.g == tiles2) return false;
  return longest / sp1.q + 2 <= kSpareSegments;
}

namespace {
bool pass2_spare(const LaunchCtx& c) {
  const SeqTable& st = c.st;
  return pass2_spare(st.sp1, st.sp2, st.layers * st.nt2, st.layers * st.batch * st.H, (c.max_seq_len + kTile - 1) / kTile);
}
struct P2Maps {
  CUtensorMap K, V, Q;
};
template <int NCH, bool SPARE>
cudaError_t launch_pass2_s(const LaunchCtx& c, const P2Maps& m, float* s_div_out, float* rbar_out, int vstages,
                           int* status) {
  static std::atomic<bool> done[kMaxDevices];
  cudaError_t e = ensure_smem(k_pass2<NCH, SPARE>, kSmemLimit, done);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_pass2<NCH, SPARE>, dim3(c.st.sp2.g), dim3(kP2Threads), pass2_smem(c.st.NQ, vstages), c.stream, 1, m.K, m.V,
                    m.Q, c.st, c.ws, s_div_out, rbar_out, c.scale_log2e, c.p.use_vnorm, c.p.pool_kernel >> 1,
                    vstages, status);
}
template <int NCH>
cudaError_t launch_pass2_t(const LaunchCtx& c, const P2Maps& m, float* s_div_out, float* rbar_out, int vstages,
                           int* status) {
  return pass2_spare(c) ? launch_pass2_s<NCH, true>(c, m, s_div_out, rbar_out, vstages, status)
                        : launch_pass2_s<NCH, false>(c, m, s_div_out, rbar_out, vstages, status);
}
}  // namespace

cudaError_t launch_pass2(const LaunchCtx& c, const void* K, const void* V, const void* Q,
                         float* s_div_out, float* rbar_out, int* status) {
  CUtensorMap tmK, tmV, tmQ;
  const void* Vsrc = c.p.use_vnorm == MIXKV_INTRINSIC_VNORM ? V : K;   // the V map is never used without VNorm
  if (!map_kv(c, K, kTile, &tmK) || !map_kv(c, Vsrc, 64, &tmV) || !map_q(c, Q, &tmQ))
    return cudaErrorInvalidValue;
  const int vstages = pass2_vstages(c.st.NQ);
  const P2Maps m{tmK, tmV, tmQ};
  switch ((c.st.NQ / 16 + 1) / 2) {   // pieces of 16 columns per epilogue warp
    case 1: return launch_pass2_t<1>(c, m, s_div_out, rbar_out, vstages, status);
    case 2: return launch_pass2_t<2>(c, m, s_div_out, rbar_out, vstages, status);
    case 3: return launch_pass2_t<3>(c, m, s_div_out, rbar_out, vstages, status);
    case 4: return launch_pass2_t<4>(c, m, s_div_out, rbar_out, vstages, status);
    case 5: return launch_pass2_t<5>(c, m, s_div_out, rbar_out, vstages, status);
    case 6: return launch_pass2_t<6>(c, m, s_div_out, rbar_out, vstages, status);
    case 7: return launch_pass2_t<7>(c, m, s_div_out, rbar_out, vstages, status);
    default: return launch_pass2_t<8>(c, m, s_div_out, rbar_out, vstages, status);
  }
}

}  // namespace mixkv

extern "C" int mixkv_internal_stats_table(int32_t segment, int32_t pair) { return mixkv::stats_table(segment, pair); }
