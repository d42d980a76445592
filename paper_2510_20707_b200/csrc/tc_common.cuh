// Blackwell (sm_100a) building blocks used by the two K passes: mbarriers with bounded
// waits, TMA tile loads, tcgen05 (UMMA) descriptors / issue / commit, TMEM allocation and
// loads.  Every wait is bounded in wall-clock time: when it expires the waiting thread raises
// the CTA-wide abort flag and the kernel drains and returns with an error status instead of
// hanging.
#pragma once

#include <cuda.h>
#include <stdint.h>

#include "common.cuh"

namespace mixkv {

constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s per wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

// Waits for the barrier phase `parity`.  Returns false (after raising *abort) when the time
// limit passes or another thread of the CTA has already aborted.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort) {
  if (mbar_try(bar, parity)) return true;
  unsigned long long t0 = 0;   // the clock is first read after a few hundred tries: most waits end before
  for (uint32_t it = 1;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 255u) == 0) {
      if (*abort) return false;
      const unsigned long long now = global_ns();
      if (t0 == 0) t0 = now;
      if (now - t0 > kWaitLimitNs) {
        *abort = 1;
        return false;
      }
    }
  }
}

// TMA tile loads (no multicast); coordinates innermost first.
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tm, int x, int y, int z,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], "
      "[%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(tm), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* tm, int x, int y, int z,
                                            int w, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], "
      "[%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
      "l"(tm), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
      : "memory");
}
// The same with an L2 eviction policy.
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* tm, int x, int y, int z,
                                            int w, uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
      "[%1, {%2, %3, %4, %5}], [%6], %7;" ::"r"(smem_u32(dst)),
      "l"(tm), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ uint64_t l2_evict_first() {
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  return policy;
}
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* tm) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(tm) : "memory");
}

// Shared-memory matrix descriptors are for K-major bf16 operands stored as rows of 128 bytes with the
// 128-byte swizzle (what a TMA box of 64 bf16 x rows writes): 8-row groups 1024 bytes apart (stride byte
// offset), leading byte offset unused, version 1 (bit 46), SWIZZLE_128B (2 in bits 61 ..).

// Instruction descriptor: D f32, A and B bf16, both K-major, M x N tile.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// The same with A and B fp16.
__host__ __device__ constexpr uint32_t umma_idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// A descriptor as two 32-bit halves: the high half is a constant, the low half is
// ((address >> 4) & 0x3fff) | 1 << 16, so stepping an operand by n bytes (n a multiple of 16,
// inside shared memory) is an integer add of n >> 4 to the low half.
//
// Issuing: ONE thread issues an MMA, but the whole warp walks the tile loop and `on` (elect_one, nonzero
// in one lane) predicates the instruction itself.  The operands of the instruction live in uniform
// registers; under a branch of a single lane they are moved there one by one, and behind seven busy warps of
// its scheduler that serial stream took 165 clocks per 128 x 128 x 16 step (64 of tensor time): it, not the
// tensor cores or the epilogue, paced pass 1.  With converged control flow the compiler computes them in
// the uniform registers in the first place.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t on;
  asm volatile(
      "{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(on));
  return on;
}
constexpr uint32_t kUmmaDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t umma_desc_lo(uint32_t saddr) {
  return ((saddr >> 4) & 0x3FFFu) | (1u << 16);
}
template <int ACC>
__device__ __forceinline__ void umma_f16_lo(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo,
                                             uint32_t idesc, uint32_t on) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, %5, 0;\n\tsetp.ne.b32 q, %6, 0;\n\t"
      "mov.b64 da, {%1, %3};\n\t"
      "mov.b64 db, {%2, %3};\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}" ::"r"(tmem_d),
      "r"(a_lo), "r"(b_lo), "r"(kUmmaDescHi), "r"(idesc), "n"(ACC), "r"(on)
      : "memory");
}
// Arrives on the barrier once every MMA issued so far by the elected thread has completed.
__device__ __forceinline__ void umma_commit(uint64_t* bar, uint32_t on) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(
          smem_u32(bar)),
      "r"(on)
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(slot)),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols)
               : "memory");
}
// 32 lanes x 16 consecutive 32-bit columns: thread l of the warp gets lane (base lane + l).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// The registers written by tcgen05.ld are only valid after tcgen05.wait::ld.  This empty
// statement makes every later use of r depend on a point after the wait (volatile asm
// statements keep their order), so the compiler cannot hoist arithmetic above it.
__device__ __forceinline__ void tmem_ld_fence(uint32_t (&r)[16]) {
  asm volatile(""
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                 "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]),
                 "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_ld_fence(uint32_t (&r)[32]) {
  asm volatile(""
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                 "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]),
                 "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
  asm volatile(""
               : "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]),
                 "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_ld_fence(uint32_t (&r)[4]) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]) : : "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void named_bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Arrives at a named barrier without waiting (the other side calls named_bar_sync with the
// same thread count); shared-memory writes before it are visible to the threads that sync.
__device__ __forceinline__ void named_bar_arrive(int id, int threads) {
  __threadfence_block();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Byte offset of element (row r, 16-byte chunk c in 0..7) inside a [rows x 128 B] half tile
// written with the 128-byte swizzle (tile base 1024-byte aligned).
__device__ __forceinline__ uint32_t sw128_offset(int r, int c) {
  return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4));
}

// ---- persistent tile schedule shared by every role of a CTA ----------------------------
// Tiles are 128 consecutive keys of one (sequence, head), numbered in (b, h, t) order.
struct TileCoord {
  int b, h, t, layer, per_head;   // per_head: tiles of each head of sequence b
};

__device__ __forceinline__ TileCoord tile_coord(const int* tile_start, int batch, int H,
                                                int id) {
  const int b = find_seq(tile_start, batch, id);
  const int per_head = (tile_start[b + 1] - tile_start[b]) / H;
  const int rem = id - tile_start[b];
  TileCoord c;
  c.b = b;
  c.h = rem / per_head;
  c.t = rem - c.h * per_head;
  c.layer = 0;
  c.per_head = per_head;
  return c;
}
// The same for a tile id that runs over all layers, nt tiles each.
__device__ __forceinline__ TileCoord layer_tile_coord(const int* tile_start, int batch, int H, int nt, int id) {
  const int layer = id / nt;
  TileCoord c = tile_coord(tile_start, batch, H, id - layer * nt);
  c.layer = layer;
  return c;
}
// Walks the tiles [lo, hi) of one CTA segment by segment: a segment is a run of tiles t0 .. t0 + n - 1 of
// one (layer, sequence, head), so that a role's loop over the tiles of a segment carries nothing but the
// tile index.  Tile ids run over all layers: id = layer * nt + (tile of the layer).
struct SegIter {
  int id, hi, layer, b, h, t0, n, per_head, H, batch;
  const int* tile_start;
  // first: of tile lo
  __device__ SegIter(const int* tile_start_, int batch_, int H_, const TileCoord& first, int lo, int hi_)
      : id(lo), hi(hi_), layer(first.layer), b(first.b), h(first.h), t0(first.t), per_head(first.per_head), H(H_),
        batch(batch_), tile_start(tile_start_) {
    n = min(per_head - t0, hi - id);
  }
  __device__ __forceinline__ bool valid() const { return id < hi; }
  // (sequence, head) of the segment inside its layer, and over all layers
  __device__ __forceinline__ int bh() const { return b * H + h; }
  __device__ __forceinline__ int unit() const { return (layer * batch + b) * H + h; }
  __device__ __forceinline__ int end() const { return t0 + n; }
  __device__ __forceinline__ void next() {
    id += n;
    t0 = 0;
    if (++h == H) {
      h = 0;
      if (++b == batch) {
        b = 0;
        ++layer;
      }
      per_head = (tile_start[b + 1] - tile_start[b]) / H;
    }
    n = min(per_head, hi - id);
  }
};

// The same tiles from the last to the first: segments in descending order, tiles end() - 1 down to t0 inside
// them.  id is the first (lowest) tile of the segment, as in SegIter.
struct RevSegIter {
  int id, lo, left, layer, b, h, t0, n, H, batch;
  const int* tile_start;
  // last: of tile hi - 1
  __device__ RevSegIter(const int* tile_start_, int batch_, int H_, const TileCoord& last, int lo_, int hi)
      : lo(lo_), left(hi), layer(last.layer), b(last.b), h(last.h), H(H_), batch(batch_), tile_start(tile_start_) {
    set(last.t + 1);
  }
  __device__ __forceinline__ void set(int end) {   // the segment ends before tile `end` of its head
    n = min(end, left - lo);
    t0 = end - n;
    id = left - n;
  }
  __device__ __forceinline__ bool valid() const { return left > lo; }
  __device__ __forceinline__ int bh() const { return b * H + h; }
  __device__ __forceinline__ int unit() const { return (layer * batch + b) * H + h; }
  __device__ __forceinline__ int end() const { return t0 + n; }
  __device__ __forceinline__ void next() {
    left -= n;
    if (--h < 0) {
      h = H - 1;
      if (--b < 0) {
        b = batch - 1;
        --layer;
      }
    }
    set((tile_start[b + 1] - tile_start[b]) / H);
  }
};

// Segments of one (b, h) whose tiles [T0, T0 + per_head) lie in one run of a split: segment e starts at T0 for e = 0 and
// at the first tile of CTA c0 + e otherwise (c0 = CTA that owns T0).
struct SegList {
  int T0, base, k0, q, r, nseg;   // base: first tile of the run, k0: c0 inside it
  SegList() = default;
  __device__ SegList(int T0_, int per_head, const Split& sp) : T0(T0_), q(sp.q), r(sp.r) {
    const int run = T0_ / sp.n, c0 = tile_owner(T0_, sp);
    base = run * sp.n;
    k0 = c0 - run * sp.p;
    nseg = tile_owner(T0_ + per_head - 1, sp) - c0 + 1;
  }
  __device__ __forceinline__ int start(int e) const {
    const int k = k0 + e;
    return e == 0 ? T0 : base + k * q + (k < r ? k : r);
  }
};

// Lets what a role has started arrive before the CTA, its shared and its tensor memory go away: `it` loads were issued into
// a ring of `stages` barriers.  A role does this at its end, whatever ended it: when it ends early because its tiles fit the
// ring, a wait of another role may still run out, and nobody would wait for what is under way.  Else the consumers wait
// for the same things anyway.
__device__ __forceinline__ void drain_ring(uint64_t* full, int stages, int it) {
  for (int k = max(0, it - stages); k < it; ++k) {
    const unsigned long long t0 = global_ns();
    while (!mbar_try(&full[k % stages], (k / stages) & 1) && global_ns() - t0 < kWaitLimitNs) {
    }
  }
}

}  // namespace mixkv
