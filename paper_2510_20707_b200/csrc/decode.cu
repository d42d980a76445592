// The step after compression: one new query token per sequence attends over the compact cache
// (paper Sec. 3.1, Eq. 1: generation continues on the compressed K, V).  All layers of a model go
// in one launch.  With one query token and G query heads per KV head the two contractions have
// 7 .. 16 rows on one side: too few for the 64- or 128-row tcgen05 tiles (nine tenths of such a
// tile would be padding), too many multiply-adds for the fp32 pipe at HBM speed (2 * 2 * G * 128
// per 512-byte row pair), so they run as warp-level mma.sync m16n8k16 (bf16 x bf16 -> fp32):
//
//   * a warp takes 16 cache rows per step, copied asynchronously into a ring of one to four (K, V) slot pairs of its
//     own (rows on a 272-byte pitch); a slot is asked for again as soon as its rows are used.  logits:
//     D[head, row] = q[head, :] . K[row, :], A = q (held in registers for the whole kernel), B = K rows.  The
//     contraction index may be permuted freely as long as A and B agree, so a lane takes 64
//     CONTIGUOUS bytes of its row (four 16-byte loads, in an order that keeps the shared-memory banks
//     apart) and deals them out over the eight k-steps.
//   * softmax weights with a running (reference, sum) per head in log2 units; the weights leave
//     as TWO bf16 (value and remainder), so the value sum is fp32-grade.
//   * values: D[head, dim] += P[head, row] . V[row, dim].  B wants two rows of one dim per
//     register: a lane loads 32 contiguous bytes of four rows and byte-permutes pairs of rows
//     together; which output column a lane's dim lands in is again a free permutation.
//
// What bounds it: a step is a serial chain of about 1000 clocks in one warp (two dependent contractions with a
// softmax between them) behind a DRAM round trip, so the rate is set by the warps per SM and by how far ahead
// each of them asks.  With the operands of two steps in registers (255 of them) eight warps fit an SM: 896
// ragged heads of 512 rows on average 69.7 us (3.4 TB/s).  Sixteen warps with one slot pair each: 59.6 us; twelve
// with two: 52.4 us (4.6 TB/s), and the short chains of few warps gain too (one head of 8192 rows 18.6 -> 15.3 us).
// (Eight persistent warps that run through the unit boundaries, the next unit taken from the hardware's launch
// control: 82 us.)
//
// The rows of a (layer, sequence, KV head) unit are dealt out in steps of 16 over the warps of a
// thread-block cluster (1 to 8 CTAs of four warps; as many as fit the GPU in one wave).  Warps
// merge through shared memory, the CTAs of a cluster through distributed shared memory, every CTA taking a
// slice of the outputs.  Every row is read once.
#include <cooperative_groups.h>

#include "internal_api.h"
#include "tc_common.cuh"

namespace cg = cooperative_groups;

namespace mixkv {
namespace {

constexpr int kDecWarps = 4;
constexpr int kDecThreads = kDecWarps * 32;
constexpr int kDecMaxG = 16;
constexpr int kDecStep = 16;     // cache rows per warp step

constexpr int kDecPitch = 272;                      // bytes between the rows of a slot
constexpr int kDecSlot = kDecStep * kDecPitch;      // one K or V slot
// Steps a warp has on their way or in work: two with three CTAs on an SM, three with two, four when a CTA has an
// SM for itself (decode_shape).
constexpr int kDecDepth = 2, kDecDepthPair = 3, kDecDepthAlone = 4;
constexpr int kDecDepthEven = 1;   // one (in the room of three) with two CTAs and long heads of one length

// Dynamic shared memory for GP = 8 or 16 head slots: per warp its ring and then, the steps being over, its value
// sums [GP][132] in the same place; the CTA's sums xo [GP][128] behind those of warp 0, in what was its ring (with
// room of their own sixteen head slots left two CTAs on an SM where the split counts on three: 32 layers x 4
// sequences of 603 rows and 12 heads 25.3 us); wm / wz [warps][16], xm / xz [16], allm / allz [8][16] every
// rank's (reference, sum) during the cluster merge.
constexpr int kDecHeadPitch = kHeadDim + 4;   // floats between the heads of a warp's value sums
__host__ __device__ constexpr size_t dec_warp_bytes(int depth) {
  return 2 * (size_t)(depth == kDecDepthEven ? kDecDepthPair : depth) * kDecSlot;
}
static_assert(16 * (kDecHeadPitch + kHeadDim) * 4 <= dec_warp_bytes(kDecDepth), "sums of a warp and of the CTA fit a ring");
constexpr size_t dec_smem(int depth) {
  return kDecWarps * dec_warp_bytes(depth) + (2 * kDecWarps + 2 + 2 * 8) * kDecMaxG * 4;
}
// Slot of dimension `dim` inside a head of a warp's value sums: one pad word per 32 dimensions
// and a head pitch of 132 put the 32 lanes of a fragment store (8 heads x 4 dimensions 32 apart)
// into 32 different banks.
__device__ __forceinline__ int dec_slot(int dim) { return dim + (dim >> 5); }

// D (16 x 8, fp32) += A (16 x 16, bf16, row) * B (16 x 8, bf16, col).  Lane l = 4 g + t holds
//   A: a0 (row g, k 2t..2t+1)  a1 (row g+8, same k)  a2 (row g, k 2t+8..2t+9)  a3 (row g+8, ..)
//   B: b0 (k 2t..2t+1, col g)  b1 (k 2t+8..2t+9, col g)
//   D: d0 d1 (row g, cols 2t, 2t+1)  d2 d3 (row g+8, same cols)
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t b0,
                                         const uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// The same with rows 8 .. 15 of A (and of D) zero: two accumulator registers.
__device__ __forceinline__ void mma_bf16_low(float (&d)[2], const uint32_t a0, const uint32_t a2,
                                             const uint32_t b0, const uint32_t b1) {
  asm volatile(
      "{\n\t.reg .f32 u, v;\n\t"
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, u, v}, {%2, %3, %4, %3}, "
      "{%5, %6}, {%0, %1, %7, %7};\n\t}"
      : "+f"(d[0]), "+f"(d[1])
      : "r"(a0), "r"(0u), "r"(a2), "r"(b0), "r"(b1), "f"(0.f));
}
// bf16 pair (x in the low half) of two floats, and what rounding left over.
__device__ __forceinline__ uint32_t pack_bf16(const float x, const float y) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ void split_bf16(const float x, const float y, uint32_t& hi, uint32_t& lo) {
  hi = pack_bf16(x, y);
  lo = pack_bf16(x - __uint_as_float(hi << 16), y - __uint_as_float(hi & 0xffff0000u));
}
__device__ __forceinline__ uint32_t word_of(const uint4& v, const int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}
__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// Sixteen rows of X into a slot: chunk c (16 bytes) of row r at r * 272 + 16 c.  Rows past the end repeat
// the last row; their weights are zero.
__device__ __forceinline__ void copy_rows(unsigned char* slot, const __nv_bfloat16* X, const int rb, const int n,
                                          const int lane) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = 2 * i + (lane >> 4), c = lane & 15;
    const int row = min(rb + r, n - 1);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(slot + r * kDecPitch + 16 * c)),
                 "l"(X + (size_t)row * kHeadDim + 8 * c)
                 : "memory");
  }
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// All copies of this lane but the newest groups (everything asked for after the tile needed now) have landed;
// with every lane of the warp past this, all rows of that tile.
template <int DEPTH>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(2 * DEPTH - 1) : "memory");
  __syncwarp();
}

// What a warp holds of a unit: query fragments, value sums, running softmax.  Register pair i of lane (g, t)
// covers dimensions 32 t + 8 c .. + 7, c = (i + 2 (t / 2)) % 4, of heads g and g + 8 (two k-steps: the first two
// of four dimensions as a0 / a1, the last two as a2 / a3).  Value sums: tile dt, registers 0 1 = head g,
// dimensions 16 (2t) + dt and 16 (2t + 1) + (dt ^ 8); registers 2 3 = head g + 8.
template <bool WIDE>
struct DecState {
  static constexpr int R = WIDE ? 4 : 2;
  uint32_t qa[8][R];
  float acc[16][R];
  float m0, m1, z0, z1;

  __device__ __forceinline__ void start(const __nv_bfloat16* q, const int G, const int g, const int t) {
    const uint4* q0 = reinterpret_cast<const uint4*>(q + (size_t)g * kHeadDim + 32 * t);
    const uint4* q1 = reinterpret_cast<const uint4*>(q + (size_t)(g + 8) * kHeadDim + 32 * t);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = (i + 2 * (t >> 1)) & 3;
      uint4 u0 = make_uint4(0, 0, 0, 0), u1 = u0;
      if (g < G) u0 = __ldg(q0 + c);
      if (WIDE && g + 8 < G) u1 = __ldg(q1 + c);
      if constexpr (WIDE) {
        qa[2 * i][0] = u0.x, qa[2 * i][2] = u0.y, qa[2 * i + 1][0] = u0.z, qa[2 * i + 1][2] = u0.w;
        qa[2 * i][1] = u1.x, qa[2 * i][3] = u1.y, qa[2 * i + 1][1] = u1.z, qa[2 * i + 1][3] = u1.w;
      } else {
        qa[2 * i][0] = u0.x, qa[2 * i][1] = u0.y, qa[2 * i + 1][0] = u0.z, qa[2 * i + 1][1] = u0.w;
      }
    }
#pragma unroll
    for (int dt = 0; dt < 16; ++dt)
#pragma unroll
      for (int c = 0; c < R; ++c) acc[dt][c] = 0.f;
    m0 = m1 = -INFINITY, z0 = z1 = 0.f;
  }

  // logits of a step: s[j] registers 0 1 = head g, rows 8 j + 2t, + 1; 2 3 = head g + 8
  __device__ __forceinline__ void logits(const unsigned char* slot, const int g, const int t, float (&s)[2][R]) const {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const unsigned char* row = slot + (8 * j + g) * kDecPitch + 64 * t;
#pragma unroll
      for (int c = 0; c < R; ++c) s[j][c] = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint4 k = *reinterpret_cast<const uint4*>(row + 16 * ((i + 2 * (t >> 1)) & 3));
        if constexpr (WIDE) {
          mma_bf16(s[j], qa[2 * i], k.x, k.y);
          mma_bf16(s[j], qa[2 * i + 1], k.z, k.w);
        } else {
          mma_bf16_low(s[j], qa[2 * i][0], qa[2 * i][1], k.x, k.y);
          mma_bf16_low(s[j], qa[2 * i + 1][0], qa[2 * i + 1][1], k.z, k.w);
        }
      }
    }
  }

  // softmax weights of one head (registers c0, c0 + 1 of s) under its running reference, log2 units; `left`: rows
  // of the unit from this step on
  template <int C0>
  __device__ __forceinline__ void weights(float (&s)[2][R], float& m, float& z, const int left,
                                          const float scale_log2e, const int t) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int c = 0; c < 2; ++c)
        s[j][C0 + c] = 8 * j + 2 * t + c < left ? s[j][C0 + c] * scale_log2e : -INFINITY;
    const float mx = quad_max(fmaxf(fmaxf(s[0][C0], s[0][C0 + 1]), fmaxf(s[1][C0], s[1][C0 + 1])));
    const float mn = fmaxf(m, mx), f = exp2f(m - mn);   // mx is finite: the step has a row
    if (f != 1.f) {
      z *= f;
#pragma unroll
      for (int dt = 0; dt < 16; ++dt) acc[dt][C0] *= f, acc[dt][C0 + 1] *= f;
    }
    m = mn;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      s[j][C0] = exp2f(s[j][C0] - mn);
      s[j][C0 + 1] = exp2f(s[j][C0 + 1] - mn);
      z += s[j][C0] + s[j][C0 + 1];
    }
  }

  // values: the weights as bf16 value + bf16 remainder (A fragments over the 16 rows of the step) times V;
  // tile dt takes dimension 16 g + (dt ^ 8 (g & 1)) of this lane's four rows
  __device__ __forceinline__ void values(const unsigned char* slot, const int g, const int t, const float (&p)[2][R]) {
    uint32_t ahi[4] = {0, 0, 0, 0}, alo[4] = {0, 0, 0, 0};
    split_bf16(p[0][0], p[0][1], ahi[0], alo[0]);
    split_bf16(p[1][0], p[1][1], ahi[2], alo[2]);
    if constexpr (WIDE) {
      split_bf16(p[0][2], p[0][3], ahi[1], alo[1]);
      split_bf16(p[1][2], p[1][3], ahi[3], alo[3]);
    }
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      uint4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        v[u] = *reinterpret_cast<const uint4*>(slot + (2 * t + (u & 1) + 8 * (u >> 1)) * kDecPitch + 32 * g +
                                               16 * (half ^ (g & 1)));
#pragma unroll
      for (int d = 0; d < 8; ++d) {
        const int dt = 8 * half + d;
        const uint32_t sel = (d & 1) ? 0x7632u : 0x5410u;
        const uint32_t b0 = __byte_perm(word_of(v[0], d >> 1), word_of(v[1], d >> 1), sel);
        const uint32_t b1 = __byte_perm(word_of(v[2], d >> 1), word_of(v[3], d >> 1), sel);
        if constexpr (WIDE) {
          mma_bf16(acc[dt], ahi, b0, b1);
          mma_bf16(acc[dt], alo, b0, b1);
        } else {
          mma_bf16_low(acc[dt], ahi[0], ahi[2], b0, b1);
          mma_bf16_low(acc[dt], alo[0], alo[2], b0, b1);
        }
      }
    }
  }
};

// A warp's value sums and (reference, sum) pairs into shared memory.
template <bool WIDE>
__device__ __forceinline__ void store_partial(const DecState<WIDE>& st, float* wacc, float* wm, float* wz,
                                              const int g, const int t) {
  const float z0 = quad_sum(st.z0), z1 = quad_sum(st.z1);
  float* w0 = wacc + (size_t)g * kDecHeadPitch;
#pragma unroll
  for (int dt = 0; dt < 16; ++dt) {
    w0[dec_slot(16 * (2 * t) + dt)] = st.acc[dt][0];
    w0[dec_slot(16 * (2 * t + 1) + (dt ^ 8))] = st.acc[dt][1];
    if constexpr (WIDE) {
      w0[8 * kDecHeadPitch + dec_slot(16 * (2 * t) + dt)] = st.acc[dt][2];
      w0[8 * kDecHeadPitch + dec_slot(16 * (2 * t + 1) + (dt ^ 8))] = st.acc[dt][3];
    }
  }
  if (t == 0) {
    wm[g] = st.m0, wz[g] = z0;
    wm[g + 8] = WIDE ? st.m1 : -INFINITY, wz[g + 8] = WIDE ? z1 : 0.f;
  }
}

// grid: n_layers * batch * H * S, clusters of S.  WIDE: more than eight query heads per KV head
// (head slots 8..15 of the tiles carry data).
constexpr int kDecPerSm = 3;   // CTAs per SM (12 warps, 208 KB of slots)
template <bool WIDE, int DEPTH>
__global__ void __launch_bounds__(kDecThreads, kDecPerSm)
k_decode_attention(const __nv_bfloat16* __restrict__ Kc, const __nv_bfloat16* __restrict__ Vc,
                   const int* __restrict__ row_offsets, const long long rows_cap,
                   const __nv_bfloat16* __restrict__ q, const int BH, const int H, const int G,
                   const float scale_log2e, const int max_rows, float* __restrict__ out) {
  constexpr int GP = WIDE ? 16 : 8;
  extern __shared__ __align__(16) float dsm[];
  constexpr int kWarpFloats = (int)(dec_warp_bytes(DEPTH) / 4);
  float* wacc = dsm;                                   // [warps]: slots, then [GP][kDecHeadPitch]
  float* xo = wacc + GP * kDecHeadPitch;               // [GP][128], behind the sums of warp 0
  float* wm = wacc + kDecWarps * kWarpFloats;          // [warps][16]
  float* wz = wm + kDecWarps * kDecMaxG;               // [warps][16]
  float* xm = wz + kDecWarps * kDecMaxG;               // [16]
  float* xz = xm + kDecMaxG;                           // [16]
  float* allm = xz + kDecMaxG;                         // [8][16]
  float* allz = allm + 8 * kDecMaxG;                   // [8][16]
  cg::cluster_group cluster = cg::this_cluster();
  const int S = (int)cluster.num_blocks(), crank = (int)cluster.block_rank();
  const int unit = blockIdx.x / S, layer = unit / BH, bh = unit % BH, b = bh / H, h = bh % H;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  const size_t qoff = (((size_t)layer * (BH / H) + b) * H + h) * (size_t)G * kHeadDim;
  pdl_launch_dependents();
  pdl_wait();
  const int* ro = row_offsets + (size_t)layer * (BH + 1);
  const int r0 = ro[bh], n = min(ro[bh + 1] - r0, max_rows);
  const __nv_bfloat16* Kb = Kc + ((size_t)layer * rows_cap + r0) * kHeadDim;
  const __nv_bfloat16* Vb = Vc + ((size_t)layer * rows_cap + r0) * kHeadDim;
  DecState<WIDE> st;
  const int nsteps = (n + kDecStep - 1) / kDecStep;
  float* mine = wacc + warp * kWarpFloats;
  {
    unsigned char* ring = reinterpret_cast<unsigned char*>(mine);   // [depth] x (K slot, V slot)
    const int stride = S * kDecWarps;
    int step = crank * kDecWarps + warp;
#pragma unroll
    for (int d = 0; d < DEPTH; ++d) {
      const int ahead = step + d * stride;
      if (ahead < nsteps) copy_rows(ring + 2 * d * kDecSlot, Kb, ahead * kDecStep, n, lane);
      copy_commit();
      if (ahead < nsteps) copy_rows(ring + (2 * d + 1) * kDecSlot, Vb, ahead * kDecStep, n, lane);
      copy_commit();
    }
    st.start(q + qoff, G, g, t);
    for (int d = 0; step < nsteps; step += stride, d = d + 1 == DEPTH ? 0 : d + 1) {
      unsigned char* sK = ring + 2 * d * kDecSlot;
      unsigned char* sV = sK + kDecSlot;
      const int ahead = step + DEPTH * stride;
      const int left = n - step * kDecStep;
      float p[2][DecState<WIDE>::R];
      copy_wait<DEPTH>();     // K of this step
      st.logits(sK, g, t, p);
      __syncwarp();    // every lane has read the slot
      if (ahead < nsteps) copy_rows(sK, Kb, ahead * kDecStep, n, lane);
      copy_commit();
      st.template weights<0>(p, st.m0, st.z0, left, scale_log2e, t);
      if constexpr (WIDE) st.template weights<2>(p, st.m1, st.z1, left, scale_log2e, t);
      copy_wait<DEPTH>();     // V of this step
      st.values(sV, g, t, p);
      __syncwarp();
      if (ahead < nsteps) copy_rows(sV, Vb, ahead * kDecStep, n, lane);
      copy_commit();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
  }

  // ---- the warps of the CTA merge through shared memory
  store_partial(st, mine, wm + warp * kDecMaxG, wz + warp * kDecMaxG, g, t);
  __syncthreads();
  for (int e = tid; e < GP * kHeadDim; e += kDecThreads) {
    const int head = e / kHeadDim, dim = e % kHeadDim;
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) M = fmaxf(M, wm[w * kDecMaxG + head]);
    float num = 0.f, den = 0.f;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) {
      const float mw = wm[w * kDecMaxG + head];
      const float sc = mw == -INFINITY ? 0.f : exp2f(mw - M);
      num = fmaf(wacc[w * kWarpFloats + head * kDecHeadPitch + dec_slot(dim)], sc, num);
      den = fmaf(wz[w * kDecMaxG + head], sc, den);
    }
    xo[e] = num;
    if (dim == 0) xm[head] = M, xz[head] = den;
  }

  // ---- the CTAs of the cluster merge through distributed shared memory: every CTA copies all
  // ranks' (reference, sum) pairs, then takes a slice of the G * 128 outputs
  cluster.sync();
  for (int e = tid; e < S * G; e += kDecThreads) {
    const int r = e / G, head = e % G;
    allm[r * kDecMaxG + head] = *cluster.map_shared_rank(&xm[head], r);
    allz[r * kDecMaxG + head] = *cluster.map_shared_rank(&xz[head], r);
  }
  __syncthreads();
  const int per = (G * kHeadDim + S - 1) / S;
  for (int e = crank * per + tid; e < min((crank + 1) * per, G * kHeadDim); e += kDecThreads) {
    const int head = e / kHeadDim;
    float M = -INFINITY;
    for (int r = 0; r < S; ++r) M = fmaxf(M, allm[r * kDecMaxG + head]);
    float num = 0.f, den = 0.f;
    if (M != -INFINITY) {
      for (int r = 0; r < S; ++r) {
        const float mr = allm[r * kDecMaxG + head];
        const float sc = mr == -INFINITY ? 0.f : exp2f(mr - M);
        num = fmaf(*cluster.map_shared_rank(&xo[e], r), sc, num);
        den = fmaf(allz[r * kDecMaxG + head], sc, den);
      }
    }
    out[qoff + e] = den > 0.f ? num / den : 0.f;
  }
  cluster.sync();   // a CTA's shared memory stays alive until its peers have read it
}

using DecKernel = void (*)(const __nv_bfloat16*, const __nv_bfloat16*, const int*, long long, const __nv_bfloat16*, int,
                           int, int, float, int, float*);
DecKernel dec_kernel(const bool wide, const int depth) {
  switch (depth) {
    case kDecDepthAlone: return wide ? k_decode_attention<true, kDecDepthAlone> : k_decode_attention<false, kDecDepthAlone>;
    case kDecDepthEven: return wide ? k_decode_attention<true, kDecDepthEven> : k_decode_attention<false, kDecDepthEven>;
    case kDecDepthPair: return wide ? k_decode_attention<true, kDecDepthPair> : k_decode_attention<false, kDecDepthPair>;
    default: return wide ? k_decode_attention<true, kDecDepth> : k_decode_attention<false, kDecDepth>;
  }
}

// CTAs per unit and depth of their rings.  shared(n) and alone(n): clusters of n CTAs that are resident at once with
// three CTAs to an SM and with one; even: the cache has room for max_rows rows of every head.  They may be of one length
// then; the caches of a layer schedule and of budgets per head have that room too and are not, and the host cannot tell.
struct DecodeShape {
  int S, depth;
};
template <typename Shared, typename Alone>
DecodeShape decode_shape(const long long units, const int max_rows, const bool even, const int sms,
                         const Shared& shared, const Alone& alone) {
  // CTAs per unit: as many as still fit the GPU in one wave while every warp keeps a step (one head of 512
  // rows on 8 CTAs 5.8 us, on 4 6.4; 112 heads of 512 rows on 3 CTAs each 11.5 us, on 2 12.8)
  const long long slots = (long long)kDecPerSm * sms;
  const long long steps = ((long long)max_rows + kDecStep - 1) / kDecStep;
  // One cluster more than are resident at once costs a second wave (48 clusters of eight were, 56 of seven, 71 of
  // six, 82 of five; units of 1500 rows: 48 on eight CTAs 12.0 us, 49 17.3, on seven 13; 70 on six 15.3, 72 20.7, on
  // five 16.2).
  long long most = slots / units < kMaxCluster ? slots / units : kMaxCluster;
  while (most > 1 && units > shared((int)most)) --most;
  if (most > steps / kDecWarps) most = steps / kDecWarps;
  int S = most < 1 ? 1 : (int)most;
  // One wave and a bit of a second: halves even that out where a warp then still has eight steps (560 ragged heads
  // of 2500 rows on average 152 -> 130 us, with five steps per warp or a nearly empty second wave nothing)
  if (units * 10 >= slots * 11 && units * 2 <= slots * 3 && steps >= 2 * kDecWarps * 8) S = 2;
  // Eight units and more: as long as all clusters are resident with an SM to each CTA, that and the deeper ring.  Where
  // there is room for three, the CTAs of a cluster end up sharing SMs while others idle (13 units of 3500 rows 15.9 ->
  // 10.3 us, 20 of them 16.2 -> 13.7, 30 of 1000 9.3 -> 8.5; fewer than eight units gain nothing).
  // Fewer than eight CTAs only where the heads can be of one length: else the longest head decides, and it wants eight
  // (28 ragged heads of 2500 rows on average 21.7 us on four CTAs, 17.7 on eight).
  // One cluster of eight too many: only one group of SMs has to share, and eight CTAs stay ahead of six as long as a
  // warp has few steps (16 units where 15 fit, six CTAs against eight: 512 rows 6.4 / 6.2 us, 512 of wide heads 11.7 /
  // 11.2, 3500 12.9 / 12.9, 8000 20.1 / 21.2; 17 units of 1500 rows 8.9 / 10.3).
  const int eight = units >= 8 ? alone(kMaxCluster) : 0;
  if (units >= 8 && !(units == eight + 1 && S == kMaxCluster && steps < 8 * kMaxCluster * kDecWarps)) {
    int x = kMaxCluster;
    while (x >= (even ? 4 : kMaxCluster) && units > alone(x)) --x;
    if (x >= (even ? 4 : kMaxCluster) && steps >= kDecWarps * x) return {x, kDecDepthAlone};
  }
  // A CTA per unit and no more than two per SM: those two, with the ring of three (with room for a third some SMs
  // get three and others one: 280 units of 5000 rows 142.6 -> 124.4 us, 256 of 300 13.6 -> 12.9, of 512 ragged
  // 41 -> 31).  Long heads of one length leave DRAM no gap then, and the SMs that get their rows first run ahead with
  // their rings while the others decide the call (SMs 81 % active, with a step in registers 89): one slot pair in
  // flight per warp keeps them level (296 units of 5000 rows 129.9 -> 120.1 us, with operands in registers 118.4; 256 of
  // 3400 80.8 -> 74.9, registers 79.5; 296 of 1000 30.7 -> 29.5).  Heads of several lengths in a cache of that very size
  // lose by it what an SM with one head, or with one that ends early, could have had in flight.  One pair against three, from
  // 1300 to 8000 rows, in a layer schedule of taper 0.3 / 0.5 / 0.8, per-head shares of 1/4 to 1, and equal heads: 224 units
  // -1 to +6 % / +2 to +6 / -1 to +11 / +2 to +8, equal -3 to -7; 240 to 256 units -2 to +1 / 0 to +5 / -1 to +8 / +3 to
  // +5, equal -4 to -8; 280 and 296 -4 to +4 / -2 to +4 / +1 to +6 / -1 to +4, equal -6 to -10; 152 units nothing either way.
  // So from 1.6 units per SM on, where equal heads gain what the others lose at worst, and not for short ones.
  const bool pair = S == 1 && units > sms && units <= 2LL * sms;
  return {S, !pair ? kDecDepth : even && steps >= 80 && units * 5 >= sms * 8LL ? kDecDepthEven : kDecDepthPair};
}

}  // namespace
}  // namespace mixkv

using namespace mixkv;

extern "C" void mixkv_internal_decode_shape(int64_t units, int32_t max_rows, int32_t even, int32_t sms,
                                            const int32_t* shared, const int32_t* alone, int32_t* ctas,
                                            int32_t* depth) {
  const DecodeShape s = decode_shape(units, max_rows, even != 0, sms, [&](const int n) { return shared[n]; },
                                     [&](const int n) { return alone[n]; });
  *ctas = s.S, *depth = s.depth;
}

extern "C" int mixkv_decode_attention(const void* K_cache, const void* V_cache,
                                      const int32_t* out_row_offsets, int64_t rows_cap,
                                      const void* q, int32_t n_layers, int32_t batch,
                                      int32_t kv_heads, int32_t gqa_ratio, int32_t head_dim,
                                      float softmax_scale, int32_t max_rows, float* out,
                                      void* stream) {
  if (!K_cache || !V_cache || !out_row_offsets || !q || !out) return MIXKV_ERR_INVALID_ARG;
  if (n_layers < 1 || batch < 1 || kv_heads < 1 || gqa_ratio < 1 || rows_cap < 0 || max_rows < 1 ||
      !(softmax_scale >= 0.f))
    return MIXKV_ERR_INVALID_ARG;
  if (head_dim != kHeadDim || gqa_ratio > kDecMaxG) return MIXKV_ERR_UNSUPPORTED;
  if ((reinterpret_cast<uintptr_t>(K_cache) & 15u) || (reinterpret_cast<uintptr_t>(V_cache) & 15u) ||
      (reinterpret_cast<uintptr_t>(q) & 15u))
    return MIXKV_ERR_INVALID_ARG;
  {
    const int rc = device_check(nullptr);
    if (rc != MIXKV_OK) return rc;
  }
  const long long units = (long long)n_layers * batch * kv_heads;
  if (units * 8 > 0x7fffffffLL) return MIXKV_ERR_UNSUPPORTED;
  const bool wide = gqa_ratio > 8;
  static std::atomic<bool> done[10][kMaxDevices];
  static ClusterFit fit[10];   // (by variant, as `done`)
  const int dev = device_slot();
  auto variant = [&](const int depth) { return 2 * depth + wide; };
  auto resident = [&](const int depth) {
    return [&, depth](const int size) {
      const DecKernel k = dec_kernel(wide, depth);
      if (!answered(ensure_smem(k, dec_smem(depth), done[variant(depth)], dev))) return 0;
      return fit[variant(depth)].ask(k, kDecThreads, dec_smem(depth), size, dev);
    };
  };
  const DecodeShape shape = decode_shape(units, max_rows, rows_cap >= (long long)max_rows * batch * kv_heads,
                                         device_sm_count(), resident(kDecDepth), resident(kDecDepthAlone));
  const int S = shape.S, depth = shape.depth;
  const size_t smem = dec_smem(depth);
  const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)kHeadDim);
  const __nv_bfloat16 *K = reinterpret_cast<const __nv_bfloat16*>(K_cache),
                      *V = reinterpret_cast<const __nv_bfloat16*>(V_cache),
                      *qq = reinterpret_cast<const __nv_bfloat16*>(q);
  const DecKernel kernel = dec_kernel(wide, depth);
  cudaError_t e = ensure_smem(kernel, smem, done[variant(depth)], dev);
  if (e != cudaSuccess) return MIXKV_ERR_CUDA;
  e = launch_pdl(kernel, dim3((unsigned)(units * S)), dim3(kDecThreads), smem, (cudaStream_t)stream, S, K, V,
                 out_row_offsets, (long long)rows_cap, qq, batch * kv_heads, kv_heads, gqa_ratio, scale * kLog2e,
                 max_rows, out);
  return e == cudaSuccess ? MIXKV_OK : MIXKV_ERR_CUDA;
}
