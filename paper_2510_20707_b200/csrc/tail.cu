// Everything after the two K passes: the per-head scalars, pooling, the head-wise mix (Eq. 2,
// Eq. 5), budgets, per-head top-B selection and the gather (Algorithm 1, step 2 and the TopB
// line).  The fixed-budget layer call runs all of it in ONE kernel, k_tail: one CTA or a cluster of
// them per (sequence, head) mixes the scores of its slice, finds the selection threshold (binned counts,
// combined through distributed shared memory), compacts the kept positions in ascending order and
// copies the kept K / V rows.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "internal_api.h"
#include "tc_common.cuh"

namespace cg = cooperative_groups;

namespace mixkv {

namespace {

// ------------------------------------------------------------------- per-head scalars
// Everything Eq. 2 / Eq. 5 need besides the per-position values, folded from the per-segment
// partials pass 2 left behind.  Computed by one warp; the five results go to sc[0..4]:
//   s_in_scaled  = (|V_i| - sc[0]) * sc[1]
//   s_div_scaled = (s_div_i - sc[2]) * sc[3]
//   sc[4]        = redundancy used by the mix
//
// In the tail it stands between the loads of the first positions and their mix, so what it reads is asked for ahead of
// them (load_head_parts: two segments per lane).
struct HeadParts {
  float4 d[2], e[2], v[2];
  float rbar;
};
__device__ __forceinline__ void load_head_parts(HeadParts& hp, const Workspace& ws, const SegList& sl, const int use_vnorm,
                                                const int e0) {
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int e = e0 + 32 * k;
    hp.d[k] = hp.e[k] = hp.v[k] = make_float4(INFINITY, -INFINITY, 0.f, 0.f);
    if (e < sl.nseg) {
      const int start = sl.start(e);
      hp.d[k] = ws.dstat[(size_t)start * 2];
      hp.e[k] = ws.dstat[(size_t)start * 2 + 1];
      if (use_vnorm) hp.v[k] = ws.vstat[start];
    }
  }
}
__device__ __forceinline__ void first_head_parts(HeadParts& hp, const Workspace& ws, const SegList& sl, const int unit,
                                                 const int use_vnorm, const float* __restrict__ rbar_in, const int lane) {
  load_head_parts(hp, ws, sl, use_vnorm, lane);
  hp.rbar = rbar_in ? rbar_in[unit] : ws.rbar[unit];
}
__device__ void head_scalars(HeadParts& hp, const SeqTable& st, const Workspace& ws, const SegList& sl, const int layer,
                             const int b, const int h, const int pool_k, const int pool_mode, const int use_vnorm,
                             const float eps, const int lane, float* sc) {
  const int P = st.cu[b + 1] - st.cu[b] - st.W;
  float dmin = INFINITY, dmax = -INFINITY, dsum = 0.f, exw = 0.f;
  float vmin = INFINITY, vmax = -INFINITY, vsum = 0.f;
  for (int e0 = lane;;) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      dmin = fminf(dmin, fminf(hp.d[k].x, hp.e[k].x));
      dmax = fmaxf(dmax, fmaxf(hp.d[k].y, hp.e[k].y));
      dsum += hp.d[k].z + hp.e[k].z;
      exw += hp.d[k].w + hp.e[k].w;
      vmin = fminf(vmin, hp.v[k].x);
      vmax = fmaxf(vmax, hp.v[k].y);
      vsum += hp.v[k].z;
    }
    e0 += 64;
    if (e0 - lane >= sl.nseg) break;
    load_head_parts(hp, ws, sl, use_vnorm, e0);
  }
  float ex;
  if (pool_mode == MIXKV_POOL_AVG) {
    // sum of the zero-padded average-pooled score = sum of raw[m] * (windows covering m) / k
    ex = warp_sum(exw) / (float)pool_k;
  } else {
    float e = 0.f;
    for (int c = st.pchunk_start[b] + lane; c < st.pchunk_start[b + 1]; c += 32)
      e += ws.exsum[((size_t)layer * st.H + h) * st.pchunks_total + c];
    ex = warp_sum(e);
  }
  dmin = warp_min(dmin);
  dmax = warp_max(dmax);
  dsum = warp_sum(dsum);
  vmin = warp_min(vmin);
  vmax = warp_max(vmax);
  vsum = warp_sum(vsum);
  if (lane == 0) {
    const float invP = 1.0f / (float)P;
    const float mean_ex = ex * invP;
    float v0 = 0.f, cin = 0.f, mean_imp = mean_ex;
    if (use_vnorm) {
      const float vinv = 1.0f / (vmax - vmin + eps);
      const float mean_in = (vsum * invP - vmin) * vinv;
      const float a_in = mean_ex / (mean_in + eps);
      v0 = vmin;
      cin = vinv * a_in;
      mean_imp = mean_ex + mean_in * a_in;
    }
    const float dinv = 1.0f / (dmax - dmin + eps);
    const float mean_dn = (dsum * invP - dmin) * dinv;
    const float a_div = mean_imp / (mean_dn + eps);
    sc[0] = v0;
    sc[1] = cin;
    sc[2] = dmin;
    sc[3] = dinv * a_div;
    sc[4] = hp.rbar;
  }
}

// Pooled attention score at one position from a staged window w[0..k) (centre at w[k/2]);
// positions outside the candidates were staged as 0 (average) or -inf (max).
__device__ __forceinline__ float pool_window(const float* w, const int k, const int mode,
                                             const float invk) {
  if (mode == MIXKV_POOL_AVG) {
    float v = 0.f;
    for (int u = 0; u < k; ++u) v += w[u];
    return v * invk;
  }
  float v = -INFINITY;
  for (int u = 0; u < k; ++u) v = fmaxf(v, w[u]);
  return v;
}

// Eq. 5 with VNorm (Eq. 2); v0 .. r: the head scalars.  Rounding written out, so that every kernel that
// mixes gives the same bits.
__device__ __forceinline__ float mix_headwise(const float ex, const float vn, const float dv, const float v0,
                                              const float vs, const float d0, const float ds, const float r) {
  const float imp = __fmaf_rn(vn - v0, vs, ex);
  const float dsc = __fmul_rn(dv - d0, ds);
  return __fmaf_rn(1.0f - r, imp, __fmul_rn(r, dsc));
}

// The other modes, out of line: in the kernels that pool and mix, code that a call does not run only lengthens the way
// to the code that it does (one layer of 4 x 1024 keys 22.5 -> 21.9 us).
__device__ __noinline__ float mix_one(const float ex, const float vn, const float dv,
                                         const float* sc, const int use_vnorm,
                                         const int mix_mode) {
  if (use_vnorm && mix_mode == MIXKV_MIX_HEADWISE)
    return mix_headwise(ex, vn, dv, sc[0], sc[1], sc[2], sc[3], sc[4]);
  const float imp = use_vnorm ? __fmaf_rn(vn - sc[0], sc[1], ex) : ex;
  const float dsc = __fmul_rn(dv - sc[2], sc[3]);
  const float r = sc[4];
  switch (mix_mode) {
    case MIXKV_MIX_HEADWISE: return __fmaf_rn(1.0f - r, imp, __fmul_rn(r, dsc));   // Eq. 5
    case MIXKV_MIX_IMPORTANCE_ONLY: return imp;
    case MIXKV_MIX_DIVERSITY_ONLY: return dv;
    default: return __fadd_rn(imp, dsc);
  }
}

// The pass-2 segments of a head.
__device__ __forceinline__ SegList pass2_segments(const SeqTable& st, const int layer, const int b, const int h) {
  const int per_head = (st.tile2_start[b + 1] - st.tile2_start[b]) / st.H;
  return SegList(layer * st.nt2 + st.tile2_start[b] + h * per_head, per_head, st.sp2);
}

struct MixParams {
  int pool_k, pool_mode, use_vnorm, mix_mode;
  float eps;
};

__device__ __noinline__ float pool_wide(const float* w, const int k, const int mode, const float invk) {
  return pool_window(w, k, mode, invk);
}

// Pooled scores of four consecutive positions from staged windows (16-byte aligned; a window of up to nine raw
// scores around each of the four is three 16-byte loads), additions in the order of pool_window.
__device__ __forceinline__ void pool4(const float* w0, const int k, const bool avg, const int mode, const float invk,
                                      float (&ex)[4]) {
  if (k <= 9) {
    float w[12];
#pragma unroll
    for (int u = 0; u < 3; ++u) *reinterpret_cast<float4*>(w + 4 * u) = *reinterpret_cast<const float4*>(w0 + 4 * u);
#pragma unroll
    for (int e = 0; e < 4; ++e) ex[e] = avg ? 0.f : -INFINITY;
#pragma unroll
    for (int u = 0; u < 9; ++u) {
      if (u < k) {
#pragma unroll
        for (int e = 0; e < 4; ++e) ex[e] = avg ? ex[e] + w[e + u] : fmaxf(ex[e], w[e + u]);
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) ex[e] = avg ? ex[e] * invk : ex[e];
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) ex[e] = pool_wide(w0 + e, k, mode, invk);
  }
}
__device__ __forceinline__ void mix4(const float (&ex)[4], const float4 v4, const float4 d4, const float* sc,
                                     const int use_vnorm, const int mix_mode, float (&m)[4]) {
  const float vv[4] = {v4.x, v4.y, v4.z, v4.w}, dd[4] = {d4.x, d4.y, d4.z, d4.w};
  if (mix_mode == MIXKV_MIX_HEADWISE && use_vnorm) {   // (scalars in registers)
    const float r = sc[4], a0 = sc[0], a1 = sc[1], d0 = sc[2], d1 = sc[3];
#pragma unroll
    for (int e = 0; e < 4; ++e) m[e] = mix_headwise(ex[e], vv[e], dd[e], a0, a1, d0, d1, r);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) m[e] = mix_one(ex[e], vv[e], dd[e], sc, use_vnorm, mix_mode);
  }
}

// --------------------------------------------------------------------------- poolsum
// Max pooling only: per-chunk sums of the pooled score (its mean enters Eq. 2).  A short chain with as many threads as a CTA
// has (256 threads, eight positions each: scores and selection of three sequences 53.1 us a call, now 52.1).
__global__ void __launch_bounds__(1024)
k_poolsum(const SeqTable st, const Workspace ws, const int k) {
  __shared__ float tile[kPChunk + 64];
  __shared__ float sred[32];
  pdl_launch_dependents();
  pdl_wait();
  const int pcx = blockIdx.x, h = blockIdx.y, layer = blockIdx.z;
  const int b = find_seq(st.pchunk_start, st.batch, pcx);
  const int P = st.cu[b + 1] - st.cu[b] - st.W;
  const int p0 = (pcx - st.pchunk_start[b]) * kPChunk;
  const int p1 = min(p0 + kPChunk, P);
  const size_t poff = ppos(st, layer, h, b, 0);
  const int half = k >> 1;
  for (int t = threadIdx.x; t < (p1 - p0) + 2 * half; t += 1024) {
    const int i = p0 - half + t;
    tile[t] = (i >= 0 && i < P) ? ws.s_ex_raw[poff + i] : -INFINITY;
  }
  __syncthreads();
  float sum = 0.f;
  for (int t = threadIdx.x; t < p1 - p0; t += 1024) sum += pool_window(tile + t, k, MIXKV_POOL_MAX, 0.f);
  sum = warp_sum(sum);
  if ((threadIdx.x & 31) == 0) sred[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x < 32) sum = warp_sum(sred[threadIdx.x]);
  if (threadIdx.x == 0) {
    const float s = sum;
    ws.exsum[((size_t)layer * st.H + h) * st.pchunks_total + pcx] = s;
  }
}

// --------------------------------------------------------------------------- mixpool
// Pooling and the mix over a grid of position chunks (the scores entry point, adaptive budgets).  A chunk is read
// with consecutive threads on consecutive positions, all loads in flight at once, staged in shared memory and
// mixed four consecutive positions per thread, as in k_tail.
//
// CH: positions per CTA.  A chunk is a chain (scalars, loads, stage, stores) that shorter ones shorten: where chunks of 2048
// leave SMs without one, 512 (scores and selection of three sequences, 80 chunks, 54.9 -> 53.9 us a call).
template <int CH>
__global__ void __launch_bounds__(256, 4)
k_mixpool(const SeqTable st, const Workspace ws, const float* __restrict__ s_div,
          const float* __restrict__ rbar_in, float* __restrict__ s_ex_out,
          float* __restrict__ s_comp, const MixParams mp) {
  __shared__ __align__(16) float tile[CH + 64], svn[CH], sdv[CH];
  __shared__ float sc[8];
  pdl_launch_dependents();
  constexpr int kSplit = kPChunk / CH;
  const int pcx = blockIdx.x / kSplit, h = blockIdx.y, layer = blockIdx.z, tid = threadIdx.x;
  const int b = find_seq(st.pchunk_start, st.batch, pcx);
  const int P = st.cu[b + 1] - st.cu[b] - st.W;
  const int p0 = (pcx - st.pchunk_start[b]) * kPChunk + (int)blockIdx.x % kSplit * CH;
  const int n = min(CH, P - p0);   // (may be none of the last chunk)
  const size_t poff = ppos(st, layer, h, b, 0);
  const int half = mp.pool_k >> 1;
  const bool avg = mp.pool_mode == MIXKV_POOL_AVG;
  const float pad = avg ? 0.f : -INFINITY;
  const SegList sl = pass2_segments(st, layer, b, h);   // (divisions: ahead of the wait)
  pdl_wait();
  // rounds of 256 positions (+ the pooling halo in one more)
  constexpr int kRounds = CH / 256;
  const int nstage = n + 2 * half;
  float raw[kRounds + 1], vn[kRounds], dv[kRounds];
#pragma unroll
  for (int e = 0; e <= kRounds; ++e) {
    const int t = e * 256 + tid, i = p0 - half + t;
    raw[e] = (t < nstage && i >= 0 && i < P) ? ws.s_ex_raw[poff + i] : pad;
  }
#pragma unroll
  for (int e = 0; e < kRounds; ++e) {
    const int t = e * 256 + tid;
    vn[e] = (mp.use_vnorm && t < n) ? ws.vnorm[poff + p0 + t] : 0.f;
    dv[e] = t < n ? s_div[poff + p0 + t] : 0.f;
  }
  if (tid < 32) {
    HeadParts hp;
    first_head_parts(hp, ws, sl, (layer * st.batch + b) * st.H + h, mp.use_vnorm, rbar_in, tid);
    head_scalars(hp, st, ws, sl, layer, b, h, mp.pool_k, mp.pool_mode, mp.use_vnorm, mp.eps, tid, sc);
  }
#pragma unroll
  for (int e = 0; e <= kRounds; ++e) {
    const int t = e * 256 + tid;
    if (t < nstage) tile[t] = raw[e];
  }
#pragma unroll
  for (int e = 0; e < kRounds; ++e) svn[e * 256 + tid] = vn[e], sdv[e * 256 + tid] = dv[e];
  __syncthreads();
  const float invk = 1.0f / (float)mp.pool_k;
  // the pooled scores take the place of the value norms, the mixed ones that of the diversity scores
#pragma unroll
  for (int g = 0; g < (CH + 1023) / 1024; ++g) {
    const int q = g * 1024 + 4 * tid;
    if (q >= n) break;
    float ex[4], m[4];
    pool4(tile + q, mp.pool_k, avg, mp.pool_mode, invk, ex);
    const float4 v4 = *reinterpret_cast<const float4*>(svn + q), d4 = *reinterpret_cast<const float4*>(sdv + q);
    mix4(ex, v4, d4, sc, mp.use_vnorm, mp.mix_mode, m);
    *reinterpret_cast<float4*>(svn + q) = make_float4(ex[0], ex[1], ex[2], ex[3]);
    *reinterpret_cast<float4*>(sdv + q) = make_float4(m[0], m[1], m[2], m[3]);
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < kRounds; ++e) {
    const int t = e * 256 + tid;
    if (t < n) {
      if (s_ex_out) s_ex_out[poff + p0 + t] = svn[t];
      s_comp[poff + p0 + t] = sdv[t];
    }
  }
}

// ------------------------------------------------------------------- threshold search
// Order-preserving map float -> uint32 (larger float, larger key); -0 is folded into +0 so
// that equal floats have equal keys.
__device__ __forceinline__ unsigned order_key(float f) {
  unsigned u = __float_as_uint(f);
  if (u == 0x80000000u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

constexpr int kSelBinBits = 11, kSelBins = 1 << kSelBinBits;
constexpr int kSelListCap = 256;   // candidates ranked directly
constexpr int kSelMaxCluster = kMaxCluster;

// The keys that a round of a search counts, [base, base + span], in bins of 2^shift keys.  Never past the largest key there is:
// the last bin of a range would else reach over 2^32, and keys below all others (k_budget's padding is key 0) be counted in it.
struct SelRange {
  unsigned base, span;
  int shift;
};
// The first round's: all keys, lo the smallest and hi the largest.
__host__ __device__ __forceinline__ SelRange sel_range(const unsigned lo, const unsigned hi) {
  SelRange r{lo, hi - lo, 0};
#ifdef __CUDA_ARCH__
  const int bits = 32 - __clz(r.span);
#else
  const int bits = r.span ? 32 - __builtin_clz(r.span) : 0;
#endif
  if (bits > kSelBinBits) r.shift = bits - kSelBinBits;
  return r;
}
// The keys of one bin, not yet binned again.
__host__ __device__ __forceinline__ SelRange sel_bin(const SelRange& r, const unsigned bin, const unsigned hi) {
  const unsigned base = r.base + (bin << r.shift), size = (1u << r.shift) - 1u;
  return {base, size < hi - base ? size : hi - base, r.shift};
}
__host__ __device__ __forceinline__ int sel_next_shift(const int shift) { return shift > kSelBinBits ? shift - kSelBinBits : 0; }

struct SelSmem {
  int hist[2][kSelBins];
  unsigned list[kSelListCap];    // this CTA's candidates
  int pos[kSelListCap];          // and which of its keys they are
  unsigned all[kSelListCap];     // those of every CTA of the cluster, in rank order (written by all of them)
  unsigned wlo[32], whi[32];
  uint2 range[kSelMaxCluster];   // smallest and largest key of every CTA (each written by that CTA)
  int scan[32];
  int nlist;                     // this CTA's candidates
  int bin, remaining, count;     // bin that holds the threshold, keys still needed from it, keys in it
  int above_before, bin_before;  // keys above the bin and in it in the CTAs of lower rank
  unsigned tau;
  int need_eq, eq_total;
};
// What the CTAs of a cluster send each other in the rounds of a search, two rounds in turn: every rank's counts in
// groups of 32 bins.
constexpr int kSelGroups = kSelBins / 32;
struct SelMail {
  int groups[2][kSelMaxCluster][kSelGroups];
};

struct Threshold {
  unsigned tau;              // the want-th largest key
  int need_eq, eq_total;     // keys equal to it that are wanted / that there are
  int gt_before, eq_before;  // keys above it and equal to it in the CTAs of lower rank
  bool listed;               // above(j) was called for this CTA's keys above the last bin, whose sm.nlist keys
                             // are in sm.list / sm.pos
};

// Sum of v over the threads after the caller (suffix = true) or before it; every thread of the CTA takes
// part.  Ends with every warp past its reads of `scan` only after the caller's next CTA barrier.
template <int T, bool SUFFIX>
__device__ __forceinline__ int block_scan(const int v, int* scan, const int lane, const int warp) {
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = SUFFIX ? __shfl_down_sync(0xffffffffu, incl, o) : __shfl_up_sync(0xffffffffu, incl, o);
    if (SUFFIX ? lane + o < 32 : lane >= o) incl += x;
  }
  if (lane == (SUFFIX ? 0 : 31)) scan[warp] = incl;
  __syncthreads();
  const bool other = lane < T / 32 && (SUFFIX ? lane > warp : lane < warp);
  return incl - v + __reduce_add_sync(0xffffffffu, other ? scan[lane] : 0);
}

// Threshold of the `want` largest keys (1 <= want < number of keys) of a set spread over the CTAs of a
// cluster (cs == 1: one CTA).  All T threads of all CTAs take part; key_at(j), j < n, gives this CTA's keys,
// lo / hi are the smallest and largest of those this thread has seen (all of them together: the CTA's).
//
// The keys are binned linearly between the smallest and the largest of all: 2048 bins over the range in
// use put the keys of a head, which share sign and most of their exponent, into hundreds of bins, so the
// counting is one shared-memory add per key without contention, and the bin of the threshold holds a few
// dozen keys, which are listed and ranked against each other.  One sweep to count, one to list, where digits of
// the raw key bits took two to four sweeps and as many exchanges across the cluster.  A bin with more keys
// than the list takes is binned again (three rounds reach single key values), so any distribution, all-equal
// keys included, ends after a bounded number of sweeps.  The listing sweep calls above(j) for the keys that
// are wanted in any case.  sm.hist must be zero on entry (visible to the CTA).
//
// Across a cluster a search is bound by its exchanges, three barriers with what has to be known behind each.  A CTA
// sends that into its peers' shared memory ahead of the barrier (range; counts per group of 32 bins; candidates, whose place
// in the common list the counts give), because a load from there costs another half a microsecond behind it; only the 32 counts
// of the one group that holds the threshold are fetched, by one warp.  (Eight CTAs of 4096 keys: 7.6 us, fetched
// from the peers behind the barriers, now 5.6; one layer of 4 x 32768 keys 47.6 -> 45.8.)
// On entry every CTA of the cluster has started.  mail: not used when cs == 1.
template <int T, typename KeyAt, typename Above>
__device__ __forceinline__ Threshold threshold_search(const KeyAt& key_at, const Above& above_bin, const int n,
                                                      const int want, unsigned lo, unsigned hi, SelSmem& sm,
                                                      SelMail& mail, cg::cluster_group& cluster, const int cs,
                                                      const int crank) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = T / 32, PER = kSelBins / T;
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) sm.wlo[warp] = lo, sm.whi[warp] = hi;
  if (tid == 0) sm.nlist = 0;
  __syncthreads();
  lo = __reduce_min_sync(0xffffffffu, lane < NW ? sm.wlo[lane] : 0xffffffffu);
  hi = __reduce_max_sync(0xffffffffu, lane < NW ? sm.whi[lane] : 0u);
  if (cs > 1) {
    if (tid < cs) *cluster.map_shared_rank(&sm.range[crank], tid) = make_uint2(lo, hi);
    cluster.sync();
    const uint2 mine = lane < cs ? sm.range[lane] : make_uint2(0xffffffffu, 0u);
    lo = mine.x, hi = mine.y;
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
  }
  SelRange r = sel_range(lo, hi);   // of the candidates
  int remaining = want, gt_before = 0;
  for (int round = 0;; ++round) {
    int* hist = sm.hist[round & 1];
    for (int j = tid; j < n; j += T) {
      const unsigned d = key_at(j) - r.base;
      if (d <= r.span) atomicAdd(&hist[d >> r.shift], 1);
    }
    __syncthreads();
    // thread t owns bins PER t .. PER t + PER - 1
    int h[PER], mine = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) h[k] = hist[PER * tid + k], mine += h[k];
    if (cs > 1) {
      constexpr int GL = 32 / PER;   // lanes that own a group of 32 bins; they send its count to the ranks in turn
      int sum = mine;
#pragma unroll
      for (int o = 1; o < GL; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      int* slot = &mail.groups[round & 1][crank][tid / GL];
      for (int to = lane % GL; to < cs; to += GL) *cluster.map_shared_rank(slot, to) = sum;
      cluster.sync();
      if (warp == 0) {
        // two groups per lane, of all CTAs and of those of lower rank
        int2 tot = make_int2(0, 0), low = tot;
#pragma unroll
        for (int of = 0; of < kSelMaxCluster; ++of) {
          const int2 v = of < cs ? *reinterpret_cast<const int2*>(&mail.groups[round & 1][of][2 * lane]) : make_int2(0, 0);
          tot.x += v.x, tot.y += v.y;
          if (of < crank) low.x += v.x, low.y += v.y;
        }
        auto keys_above = [&](const int v) {   // sum of v over the higher lanes
          int incl = v;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_down_sync(0xffffffffu, incl, o);
            if (lane + o < 32) incl += x;
          }
          return incl - v;
        };
        int above = keys_above(tot.x + tot.y);
        const bool in_y = above < remaining && remaining <= above + tot.y;
        const bool in_x = above + tot.y < remaining && remaining <= above + tot.y + tot.x;
        int src = __ffs(__ballot_sync(0xffffffffu, in_x || in_y)) - 1;
        const int group = __shfl_sync(0xffffffffu, 2 * lane + (in_y ? 1 : 0), src);
        above = __shfl_sync(0xffffffffu, in_y ? above : above + tot.y, src);
        int before = __reduce_add_sync(0xffffffffu, (2 * lane > group ? low.x : 0) + (2 * lane + 1 > group ? low.y : 0));
        // the bins of that group, one per lane
        int v[kSelMaxCluster], all = 0, lower = 0;
#pragma unroll
        for (int of = 0; of < kSelMaxCluster; ++of) v[of] = of < cs ? *cluster.map_shared_rank(&hist[32 * group + lane], of) : 0;
#pragma unroll
        for (int of = 0; of < kSelMaxCluster; ++of) all += v[of], lower += of < crank ? v[of] : 0;
        above += keys_above(all);
        src = __ffs(__ballot_sync(0xffffffffu, above < remaining && remaining <= above + all)) - 1;
        before += __reduce_add_sync(0xffffffffu, lane > src ? lower : 0);
        if (lane == src) {
          sm.bin = 32 * group + lane;
          sm.remaining = remaining - above;
          sm.count = all;
          sm.above_before = before;
          sm.bin_before = lower;
        }
      }
    } else {
      int above = block_scan<T, true>(mine, sm.scan, lane, warp);
      if (above < remaining && remaining <= above + mine) {
#pragma unroll
        for (int k = PER - 1; k >= 0; --k) {
          if (above < remaining && remaining <= above + h[k]) {
            sm.bin = PER * tid + k;
            sm.remaining = remaining - above;
            sm.count = h[k];
          }
          above += h[k];
        }
      }
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) sm.hist[(round & 1) ^ 1][PER * tid + k] = 0;   // every CTA is past its reads of it
    __syncthreads();
    if (cs > 1) gt_before += sm.above_before;
    r = sel_bin(r, (unsigned)sm.bin, hi);
    remaining = sm.remaining;
    if (r.shift == 0 || sm.count <= kSelListCap) break;
    r.shift = sel_next_shift(r.shift);
  }
  const int count = sm.count;
  const int before = cs > 1 ? sm.bin_before : 0;   // candidates of the lower ranks
  Threshold th;
  th.gt_before = gt_before;
  th.eq_before = 0;
  th.listed = r.shift != 0;
  if (r.shift == 0) {   // the bin is one key value
    th.tau = r.base, th.need_eq = remaining, th.eq_total = count, th.eq_before = before;
    return th;
  }
  // list the candidates; the keys above them are wanted in any case
  for (int j = tid; j < n; j += T) {
    const unsigned key = key_at(j);
    if (key >= r.base) {
      if (key - r.base <= r.span) {
        const int at = atomicAdd(&sm.nlist, 1);
        sm.list[at] = key, sm.pos[at] = j;
        if (cs > 1)
          for (int to = 0; to < cs; ++to) *cluster.map_shared_rank(&sm.all[before + at], to) = key;
      } else {
        above_bin(j);
      }
    }
  }
  const unsigned* all = sm.list;
  if (cs > 1) {
    all = sm.all;
    cluster.sync();
  } else {
    __syncthreads();
  }
  for (int k = tid; k < count; k += T) {
    const unsigned key = all[k];
    int g = 0, e = 0;
#pragma unroll 4
    for (int x = 0; x < count; ++x) {
      const unsigned y = all[x];
      g += y > key;
      e += y == key;
    }
    if (g < remaining && remaining <= g + e) sm.tau = key, sm.need_eq = remaining - g, sm.eq_total = e;
  }
  __syncthreads();
  th.tau = sm.tau, th.need_eq = sm.need_eq, th.eq_total = sm.eq_total;
  if (cs > 1) {
    int g = 0, e = 0;
    for (int x = lane; x < before; x += 32) {
      g += all[x] > th.tau;
      e += all[x] == th.tau;
    }
    th.gt_before += __reduce_add_sync(0xffffffffu, g);
    th.eq_before = __reduce_add_sync(0xffffffffu, e);
  }
  return th;
}

constexpr int kBudgetCluster = kMaxCluster;
constexpr int kBudgetThreads = 1024;
// (0 is the padding's; order_key gives it to one NaN)
__device__ __forceinline__ unsigned budget_key(const float f) { return max(order_key(f), 1u); }

// Head budgets of one sequence under the adaptive rule (see mixkv.h).  One CTA per (sequence,
// layer) when the call has many of them, else a cluster of up to kBudgetCluster CTAs, each with a
// slice of the positions of every head.  A CTA turns its H * n pooled scores into
// order-preserving keys once and keeps them in shared memory when they fit (cache_cap keys);
// otherwise every sweep reads them from global memory.
// Bound by its chain of block-wide (cluster-wide) steps, not by the scores it reads: 28 layers x 8 ragged
// sequences of 4 heads, 2 to 7 thousand candidates each, 65 us with digit passes over the raw keys, 35 us with
// threshold_search.  In a cluster that chain also crosses six barriers or more (start, range, counts of each round, candidates,
// heads' counts, end), with what a CTA needs of the others sent ahead of them but for the heads' counts.  Clusters of two and
// half the threads were no faster (measured when it was fetched behind four barriers).
__global__ void __launch_bounds__(kBudgetThreads)
k_budget(const SeqTable st, const float* __restrict__ scores, int* __restrict__ counts,
         const int Bp, const int floor_slots, const int cache_cap) {
  extern __shared__ unsigned bkeys[];   // [cache_cap] keys
  __shared__ __align__(16) SelSmem sm;
  __shared__ int s_gt[64], s_eq[64], t_gt[64], t_eq[64];
  __shared__ __align__(16) SelMail mail;
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks(), crank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_launch_dependents();
  if (cs > 1) cluster.sync();   // every CTA has started: its peers may write to it
  for (int t = tid; t < 2 * kSelBins; t += kBudgetThreads) (&sm.hist[0][0])[t] = 0;
  if (tid < 64) s_gt[tid] = 0, s_eq[tid] = 0;
  pdl_wait();
  const int b = blockIdx.x / cs, layer = blockIdx.y, H = st.H;
  counts += (size_t)layer * st.batch * H;
  const int P = st.cu[b + 1] - st.cu[b] - st.W;
  const long long total = (long long)H * P;
  long long N = (long long)H * (Bp - floor_slots);
  if (N > total) N = total;
  const float* base = scores + ppos(st, layer, 0, b, 0);
  const size_t stride = (size_t)st.Ptot;
  if (N <= 0 || N == total) {   // nothing to share, or everything: the same in every CTA of the cluster
    if (crank == 0)
      for (int h = tid; h < H; h += kBudgetThreads) counts[b * H + h] = N <= 0 ? min(floor_slots, P) : P;
    return;
  }
  // This CTA's slice of every head: positions [p0, p0 + n).  Its keys stand head after head, every head padded
  // to whole words of 32 with key 0 (below every score's), so that a word belongs to one head.
  const int chunk = (P + cs - 1) / cs;
  const int p0 = min(crank * chunk, P), n = min(chunk, P - p0);
  const int npad = (n + 31) & ~31, local = H * npad;
  const bool cached = local <= cache_cap;
  unsigned lo = 0xffffffffu, hi = 0u;
  for (int i0 = 0; i0 < npad; i0 += 2 * kBudgetThreads) {   // up to eight loads in flight per thread
    for (int h0 = 0; h0 < H; h0 += 4) {
      float v[2][4];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int i = i0 + u * kBudgetThreads + tid;
          v[u][k] = i < n && h0 + k < H ? base[(size_t)(h0 + k) * stride + p0 + i] : 0.f;
        }
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int i = i0 + u * kBudgetThreads + tid;
          if (i < npad && h0 + k < H) {
            const unsigned key = i < n ? budget_key(v[u][k]) : 0u;
            if (cached) bkeys[(h0 + k) * npad + i] = key;
            if (i < n) lo = min(lo, key), hi = max(hi, key);
          }
        }
    }
  }
  __syncthreads();
  auto key_at = [&](const int e) -> unsigned {
    if (cached) return bkeys[e];
    const int h = e / npad, i = e - h * npad;
    return i < n ? budget_key(base[(size_t)h * stride + p0 + i]) : 0u;
  };
  const Threshold th =
      threshold_search<kBudgetThreads>(key_at, [](int) {}, local, (int)N, lo, hi, sm, mail, cluster, cs, crank);
  // a vote per word of 32; most words hold nothing that counts
  for (int h = 0; h < H; ++h) {
    for (int i0 = warp * 32; i0 < npad; i0 += kBudgetThreads) {
      const unsigned key = key_at(h * npad + i0 + lane);
      const int gt = __popc(__ballot_sync(0xffffffffu, key > th.tau)),
                eq = __popc(__ballot_sync(0xffffffffu, key == th.tau));
      if (lane == 0 && (gt | eq)) {
        if (gt) atomicAdd(&s_gt[h], gt);
        if (eq) atomicAdd(&s_eq[h], eq);
      }
    }
  }
  // every CTA's per-head counts are complete
  if (cs > 1) cluster.sync();
  else __syncthreads();
  if (crank == 0) {
    for (int h = tid; h < H; h += kBudgetThreads) {
      int g = 0, q = 0;
      for (int r = 0; r < cs; ++r) {
        g += *cluster.map_shared_rank(&s_gt[h], r);
        q += *cluster.map_shared_rank(&s_eq[h], r);
      }
      t_gt[h] = g, t_eq[h] = q;
    }
    __syncthreads();
    if (tid == 0) {
      int rem = th.need_eq;  // equal-to-threshold elements go to the lower (head, position) first
      for (int h = 0; h < H; ++h) {
        const int take = min(t_eq[h], rem);
        rem -= take;
        counts[b * H + h] = min(floor_slots + t_gt[h] + take, P);
      }
    }
  }
  if (cs > 1) cluster.sync();   // the peers' shared memory stays alive until rank 0 has read it
}

// Word at which the keys of a slice start in k_tail's dynamic shared memory: behind the two bitmaps, on a
// 16-byte boundary.
__host__ __device__ __forceinline__ int tail_keys_at(const int chunk) { return ((chunk >> 4) + 3) & ~3; }
// Positions per CTA when cs CTAs share the P candidates of a head: whole words of 32.
__host__ __device__ __forceinline__ int tail_chunk(const int P, const int cs) {
  return (((P + cs - 1) / cs) + 31) & ~31;
}

// ------------------------------------------------------------------------------ tail
constexpr int kTailMaxCluster = kMaxCluster;
constexpr int kTailCacheCap = 40960;       // positions a CTA keeps in shared memory
constexpr int kTailCacheCapFull = 16384;   // the same in a cluster of eight: few, very long heads go unfused beyond
constexpr size_t kTailSmem = 203 * 1024;   // dynamic shared memory at most
constexpr int kTailRowCap = 1024;          // selected rows of a CTA listed in shared memory for the gather

struct TailKernelArgs {
  const float* scores;        // select on these (FUSED == false)
  const float* s_div;         // FUSED: parts of the mix
  const float* rbar_in;
  float* s_comp_out;          // FUSED: mixed scores are written here (nullptr: nobody wants them)
  const int* counts_dev;      // adaptive budgets; nullptr = fixed
  int* counts_out;
  int* idx;
  int* idx_offsets;
  int* out_row_offsets;       // may be nullptr
  const __nv_bfloat16* K;     // gather when K_out != nullptr
  const __nv_bfloat16* V;
  __nv_bfloat16* K_out;
  __nv_bfloat16* V_out;
  int Bp;                     // B - W
  int floor_slots;            // ADAPT: rows that every head gets
  int cached;                 // keys of the slice fit the shared-memory cache
  long long kv_layer_stride;  // elements between consecutive layers of K (V)
  int idx_cap;                // index-list entries reserved per layer
  int out_rows_cap;           // output rows reserved per layer
  int* status_clear;          // optional word set to 0
  MixParams mp;
};

// Selected rows of (b', h') pairs before bh, fixed budgets.
__device__ __forceinline__ int fixed_offset(const SeqTable& st, int bh, int Bp) {
  const int b = bh / st.H, h = bh % st.H;
  int off = 0;
  for (int x = 0; x < b; ++x) off += st.H * min(Bp, st.cu[x + 1] - st.cu[x] - st.W);
  if (b < st.batch) off += h * min(Bp, st.cu[b + 1] - st.cu[b] - st.W);
  return off;
}

// T threads per CTA, cs CTAs (a cluster, read from the launch) per (layer, sequence, head): see tail_shape.
//
// Latency bound: a unit is a chain of short phases.  Mix (or load) the slice's scores into shared memory as
// keys; threshold (threshold_search); one vote per 32 positions turns the keys into a bitmap whose prefix sums
// place every kept position; gather.  28 layers x 4 heads x 32736 candidates: 35 us (57 with digit passes over the
// raw keys and a position per thread and step in the mix); 896 heads of 2 to 7 thousand candidates (selection and
// gather only): 47 us (119).
// CL: launched as a cluster (else one CTA per unit, and none of the cluster's code is there to be stepped over).
// ADAPT: a cluster is the heads of a sequence, a CTA each, and shares the sequence's budget out first (the rule of
// k_budget, from the keys that the CTAs hold anyway): a search across the cluster, then every CTA its own.  It stands for
// mix, budget and tail kernels that each read again what the one before wrote, where tail_adapts says so.
template <bool FUSED, int T, bool CL, bool ADAPT>
__global__ void __launch_bounds__(T, 1024 / T)
k_tail(const SeqTable st, const Workspace ws, const TailKernelArgs a) {
  extern __shared__ __align__(16) unsigned char tail_smem[];
  __shared__ __align__(16) SelSmem sm;
  __shared__ int s_off, s_want;
  __shared__ float sc[8];
  __shared__ __align__(16) int s_rows[kTailRowCap];   // (ahead of the compaction: what the search exchanges)
  static_assert(sizeof(SelMail) <= sizeof(s_rows));
  SelMail& mail = reinterpret_cast<SelMail&>(s_rows);
  __shared__ int s_gt[32], s_eq[32];   // (ADAPT)
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = CL && !ADAPT ? (int)cluster.block_rank() : 0;   // (in ADAPT a unit is one CTA's)
  const int cs = CL && !ADAPT ? (int)cluster.num_blocks() : 1;
  const int BH = st.batch * st.H;
  const int unit = blockIdx.x / cs;                    // (layer, sequence, head)
  const int layer = unit / BH, bh = unit % BH, b = bh / st.H, h = bh % st.H;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int W = st.W;
  const int P = st.cu[b + 1] - st.cu[b] - W;
  const size_t poff = ppos(st, layer, h, b, 0);
  // this layer's slices of the per-layer arrays
  const int* counts_dev = a.counts_dev ? a.counts_dev + (size_t)layer * BH : nullptr;
  int* counts_out = a.counts_out ? a.counts_out + (size_t)layer * BH : nullptr;
  int* idx_offsets = a.idx_offsets + (size_t)layer * (BH + 1);
  int* out_row_offsets = a.out_row_offsets ? a.out_row_offsets + (size_t)layer * (BH + 1) : nullptr;
  // slice of this CTA: positions [c0, c0 + n), whole words of 32 positions
  const int chunk = tail_chunk(P, cs);
  const int c0 = min(crank * chunk, P);
  const int n = min(chunk, P - c0);
  const int nwords = (n + 31) >> 5;
  unsigned* words = reinterpret_cast<unsigned*>(tail_smem);            // [chunk / 32] bitmap of kept positions
  unsigned* eqw = words + (chunk >> 5);                                // [chunk / 32] positions equal to the threshold
  unsigned* skeys = reinterpret_cast<unsigned*>(tail_smem) + tail_keys_at(chunk);   // [chunk] when cached
  float* sraw = reinterpret_cast<float*>(skeys + chunk);               // FUSED: [4 T + 64] raw scores of a block
  float* sdv = sraw + 4 * T + 64;                                      // FUSED: [4 T] diversity scores

  if (CL) cluster.barrier_arrive();   // this CTA has started: its peers may write to it
  for (int t = tid; t < 2 * kSelBins; t += T) (&sm.hist[0][0])[t] = 0;
  const SegList sl2 = pass2_segments(st, layer, b, h);   // (divisions: ahead of the wait)
  const int fixed_off = fixed_offset(st, bh, a.Bp);
  pdl_wait();

  if (a.status_clear && blockIdx.x == 0 && tid == 0) *a.status_clear = 0;
  // ---- budget and output offsets of this (b, h)
  if (warp == 0) {
    int off = 0, cnt;
    if (counts_dev) {
      for (int t = lane; t < bh; t += 32) off += counts_dev[t];
      off = __reduce_add_sync(0xffffffffu, off);
      cnt = counts_dev[bh];
    } else {
      off = fixed_off;
      cnt = min(a.Bp, P);
    }
    if (lane == 0 && !ADAPT) {
      s_off = off;
      s_want = cnt;
      if (crank == 0) {
        idx_offsets[bh] = off;
        if (counts_out) counts_out[bh] = cnt;
        if (out_row_offsets) out_row_offsets[bh] = off + bh * W;
        if (bh == BH - 1) {
          idx_offsets[BH] = off + cnt;
          if (out_row_offsets) out_row_offsets[BH] = off + cnt + BH * W;
        }
      }
    }
  }
  const bool cached = FUSED || a.cached;
  unsigned klo = 0xffffffffu, khi = 0u;   // smallest and largest key this thread has made
  if (FUSED) {
    // ---- pooling and mix of this slice (Eq. 2, Eq. 5) in blocks of 4 T positions.  A block is read from
    // global memory one block ahead (consecutive threads, consecutive positions), staged in shared memory
    // (raw scores with the pooling halo; value norms in the slots of the block's keys), and every
    // thread then takes four CONSECUTIVE positions: a window of up to nine raw scores around them is three
    // 16-byte loads instead of four times the window.
    constexpr int BL = 4 * T;
    const int half = a.mp.pool_k >> 1;
    const bool avg = a.mp.pool_mode == MIXKV_POOL_AVG, vnorm_on = a.mp.use_vnorm != 0;
    const float pad = avg ? 0.f : -INFINITY;
    const float invk = 1.0f / (float)a.mp.pool_k;
    const float* g_raw = ws.s_ex_raw + poff;
    const float* g_vn = ws.vnorm + poff + c0;
    const float* g_dv = a.s_div + poff + c0;
    float* svn = reinterpret_cast<float*>(skeys);
    float raw[5], vn[4], dv[4];   // the fifth raw score: the halo (62 positions at most)
    auto load_block = [&](const int j0) {
      const int nb = min(BL, n - j0), i0 = c0 + j0 - half;
      if (nb == BL && i0 >= 0 && i0 + BL + 2 * half <= P) {   // inside the sequence: nothing to test
        const float* r = g_raw + i0 + tid;
        const float* d = g_dv + j0 + tid;
        const float* v = g_vn + j0 + tid;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          raw[e] = r[e * T];
          dv[e] = d[e * T];
          vn[e] = vnorm_on ? v[e * T] : 0.f;
        }
        if (tid < 2 * half) raw[4] = r[4 * T];
        return;
      }
#pragma unroll
      for (int e = 0; e < 5; ++e) {
        const int t = e * T + tid, i = i0 + t;
        raw[e] = (t < nb + 2 * half && i >= 0 && i < P) ? g_raw[i] : pad;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int t = e * T + tid;
        vn[e] = (vnorm_on && t < nb) ? g_vn[j0 + t] : 0.f;
        dv[e] = t < nb ? g_dv[j0 + t] : 0.f;
      }
    };
    HeadParts hp;
    if (warp == 1) first_head_parts(hp, ws, sl2, unit, a.mp.use_vnorm, a.rbar_in, lane);
    if (n > 0) load_block(0);
    if (warp == 1)
      head_scalars(hp, st, ws, sl2, layer, b, h, a.mp.pool_k, a.mp.pool_mode, a.mp.use_vnorm, a.mp.eps, lane, sc);
    for (int j0 = 0; j0 < n; j0 += BL) {
      const int nb = min(BL, n - j0);   // positions of this block
      __syncthreads();                  // the previous block's readers of the stage are done
      if (nb == BL) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          sraw[e * T + tid] = raw[e], sdv[e * T + tid] = dv[e], svn[j0 + e * T + tid] = vn[e];
        if (tid < 2 * half) sraw[BL + tid] = raw[4];
      } else {
#pragma unroll
        for (int e = 0; e < 5; ++e) {
          const int t = e * T + tid;
          if (t < nb + 2 * half) sraw[t] = raw[e];
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int t = e * T + tid;
          if (t < nb) sdv[t] = dv[e], svn[j0 + t] = vn[e];
        }
      }
      if (j0 + BL < n) load_block(j0 + BL);
      __syncthreads();
      const int q = 4 * tid;            // this thread's positions q .. q + 3 of the block
      if (q < nb) {
        float ex[4], m[4];
        pool4(sraw + q, a.mp.pool_k, avg, a.mp.pool_mode, invk, ex);
        mix4(ex, *reinterpret_cast<const float4*>(svn + j0 + q), *reinterpret_cast<const float4*>(sdv + q), sc,
             a.mp.use_vnorm, a.mp.mix_mode, m);
        unsigned key[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          key[e] = order_key(m[e]);
          if (q + e < nb) {
            klo = min(klo, key[e]);
            khi = max(khi, key[e]);
          }
        }
        if (a.s_comp_out) {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (q + e < nb) a.s_comp_out[poff + c0 + j0 + q + e] = m[e];
        }
        *reinterpret_cast<uint4*>(skeys + j0 + q) = make_uint4(key[0], key[1], key[2], key[3]);
      }
    }
  } else {
    for (int j0 = 0; j0 < n; j0 += 4 * T) {   // four loads in flight per thread
      float v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = j0 + e * T + tid;
        v[e] = j < n ? a.scores[poff + c0 + j] : 0.f;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = j0 + e * T + tid;
        if (j < n) {
          const unsigned key = order_key(v[e]);
          if (cached) skeys[j] = key;
          klo = min(klo, key);
          khi = max(khi, key);
        }
      }
    }
  }
  __syncthreads();
  if (CL) cluster.barrier_wait();
  auto key_at = [&](int j) -> unsigned { return cached ? skeys[j] : order_key(a.scores[poff + c0 + j]); };
  if constexpr (ADAPT) {
    // ---- this head's share: the floor, and the keys among the H * (Bp - floor) largest of all heads (equal ones to the
    // lower head, then position).  No head can run out of candidates (tail_adapts), so a sequence fills H * Bp rows.
    const int rank = (int)cluster.block_rank(), H = st.H;
    const int N = H * (a.Bp - a.floor_slots);
    int share = 0;
    if (N > 0) {
      const Threshold th = threshold_search<T>(key_at, [](int) {}, n, N, klo, khi, sm, mail, cluster, H, rank);
      int gt = 0, eq = 0;
      for (int j = tid; j < n; j += T) {
        const unsigned key = key_at(j);
        gt += key > th.tau;
        eq += key == th.tau;
      }
      gt = __reduce_add_sync(0xffffffffu, gt);
      eq = __reduce_add_sync(0xffffffffu, eq);
      if (lane == 0) s_gt[warp] = gt, s_eq[warp] = eq;
      __syncthreads();
      gt = __reduce_add_sync(0xffffffffu, lane < T / 32 ? s_gt[lane] : 0);
      eq = __reduce_add_sync(0xffffffffu, lane < T / 32 ? s_eq[lane] : 0);
      share = gt + max(0, min(eq, th.need_eq - th.eq_before));
    }
    if (tid == 0) s_want = a.floor_slots + share;
    cluster.sync();   // the shares are there, and nobody reads another's search any more
    const int mine = lane < H ? *cluster.map_shared_rank(&s_want, lane) : 0;
    const int off = b * H * a.Bp + __reduce_add_sync(0xffffffffu, lane < rank ? mine : 0);
    const int cnt = a.floor_slots + share;
    if (tid == 0) {
      s_off = off;
      idx_offsets[bh] = off;
      if (counts_out) counts_out[bh] = cnt;
      if (out_row_offsets) out_row_offsets[bh] = off + bh * W;
      if (bh == BH - 1) {
        idx_offsets[BH] = off + cnt;
        if (out_row_offsets) out_row_offsets[BH] = off + cnt + BH * W;
      }
    }
    cluster.barrier_arrive();   // past this CTA's last remote read
    for (int t = tid; t < 2 * kSelBins; t += T) (&sm.hist[0][0])[t] = 0;   // for this head's own search
    __syncthreads();
  }
  const int want = s_want;

  int kept = 0, before = 0;   // positions this CTA keeps, and the CTAs of lower rank
  if (want >= P) {            // every candidate
    for (int w = tid; w < nwords; w += T) words[w] = n - 32 * w >= 32 ? 0xffffffffu : (1u << (n - 32 * w)) - 1u;
    before = c0;
  } else if (want > 0) {
    for (int w = tid; w < nwords; w += T) words[w] = 0u;   // visible after the search's first barrier
    auto keep = [&](const int j) { atomicOr(&words[j >> 5], 1u << (j & 31)); };
    const Threshold th = threshold_search<T>(key_at, keep, n, want, klo, khi, sm, mail, cluster, cs, crank);
    const bool all_eq = th.need_eq == th.eq_total;   // no tie to split: keep every key from tau on
    if (all_eq && th.listed) {
      for (int k = tid; k < sm.nlist; k += T)
        if (sm.list[k] >= th.tau) keep(sm.pos[k]);
    } else {
      // a warp votes on 32 consecutive positions
      __syncthreads();
      for (int j0 = 0; j0 < n; j0 += T) {
        const int j = j0 + tid;
        const unsigned key = j < n ? key_at(j) : 0u;
        const unsigned m = __ballot_sync(0xffffffffu, j < n && (all_eq ? key >= th.tau : key > th.tau));
        const unsigned q = __ballot_sync(0xffffffffu, j < n && key == th.tau);
        if (lane == 0 && (j >> 5) < nwords) {
          words[j >> 5] = m;
          eqw[j >> 5] = q;
        }
      }
    }
    __syncthreads();
    before = th.gt_before + min(th.eq_before, th.need_eq);
    if (!all_eq) {   // the first need_eq equal keys in position order
      int seen = th.eq_before;
      for (int w0 = 0; w0 < nwords; w0 += T) {
        const int w = w0 + tid;
        unsigned q = w < nwords ? eqw[w] : 0u;
        const int first = seen + block_scan<T, false>(__popc(q), sm.scan, lane, warp);
        int take = max(0, min(__popc(q), th.need_eq - first));
        unsigned keep = 0u;
        for (; take > 0; --take) {
          keep |= q & (0u - q);
          q &= q - 1u;
        }
        if (w < nwords) words[w] |= keep;
        __syncthreads();
        if (tid < 32) {   // total of this round
          const int tot = __reduce_add_sync(0xffffffffu, lane < T / 32 ? sm.scan[lane] : 0);
          if (lane == 0) sm.bin = tot;
        }
        __syncthreads();
        seen += sm.bin;
        __syncthreads();
      }
    }
  }
  // ---- compaction: prefix sums over the words of the bitmap place every kept position
  int* out = a.idx + (size_t)layer * a.idx_cap + s_off;
  if (want > 0) {
    __syncthreads();   // the words are complete
    for (int w0 = 0; w0 < nwords; w0 += T) {
      const int w = w0 + tid;
      unsigned m = w < nwords ? words[w] : 0u;
      int k = kept + block_scan<T, false>(__popc(m), sm.scan, lane, warp);
      kept += __reduce_add_sync(0xffffffffu, lane < T / 32 ? sm.scan[lane] : 0);
      for (; m; m &= m - 1u, ++k) {
        const int i = c0 + 32 * w + __ffs(m) - 1;
        out[before + k] = i;
        if (k < kTailRowCap) s_rows[k] = i;
      }
      __syncthreads();
    }
  }
  if (cs > 1 && want > 0 && want < P) cluster.barrier_arrive();   // past this CTA's last remote read

  pdl_launch_dependents();

  // ---- gather: the rows this CTA keeps in ascending position order; the last CTA adds the W window rows
  if (a.K_out) {
    const int rows = kept + (crank == cs - 1 ? W : 0);
    const __nv_bfloat16* Ksrc = a.K + (size_t)layer * a.kv_layer_stride;
    const __nv_bfloat16* Vsrc = a.V + (size_t)layer * a.kv_layer_stride;
    const size_t srow0 = (size_t)h * st.Ltot + st.cu[b];
    const size_t drow0 = (size_t)layer * a.out_rows_cap + (size_t)(s_off + bh * W + before);
    const int hw = tid >> 4, l = tid & 15;                       // half-warps, 16 B per lane
    constexpr int kSweep = T / 16;
    auto source = [&](const int r) {
      return r >= kept ? P + (r - kept) : r < kTailRowCap ? s_rows[r] : __ldcg(out + before + r);
    };
    for (int r0 = hw; r0 < rows; r0 += 4 * kSweep) {   // four rows of K and V in flight
      uint4 kk[4], vv[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = r0 + e * kSweep;
        if (r < rows) {
          const size_t src = (srow0 + source(r)) * kHeadDim;
          kk[e] = __ldg(reinterpret_cast<const uint4*>(Ksrc + src) + l);
          vv[e] = __ldg(reinterpret_cast<const uint4*>(Vsrc + src) + l);
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = r0 + e * kSweep;
        if (r < rows) {
          reinterpret_cast<uint4*>(a.K_out + (drow0 + r) * kHeadDim)[l] = kk[e];
          reinterpret_cast<uint4*>(a.V_out + (drow0 + r) * kHeadDim)[l] = vv[e];
        }
      }
    }
  }
  // a CTA's shared memory stays alive until its peers have read it
  if (cs > 1 && want > 0 && want < P) cluster.barrier_wait();
  if constexpr (ADAPT) cluster.barrier_wait();
}

int floor_slots(const mixkv_params& p) {
  const int Bp = p.budget - p.window;
  int f = (int)floor((double)p.ada_floor * (double)Bp);
  if (f > Bp) f = Bp;
  if (f < 0) f = 0;
  return f;
}

MixParams mix_params(const mixkv_params& p) {
  MixParams mp;
  mp.pool_k = p.pool_kernel;
  mp.pool_mode = p.pool_mode;
  mp.use_vnorm = p.use_vnorm;
  mp.mix_mode = p.mix_mode;
  mp.eps = p.eps;
  return mp;
}

}  // namespace

cudaError_t launch_poolsum(const LaunchCtx& c) {
  return launch_pdl(k_poolsum, dim3(c.st.pchunks_total, c.st.H, c.st.layers), dim3(1024), 0,
                    c.stream, 1, c.st,
                    c.ws, c.p.pool_kernel);
}

cudaError_t launch_mixpool(const LaunchCtx& c, const float* s_div, const float* rbar_in,
                           float* s_ex_out, float* s_comp) {
  const long long chunks = (long long)c.st.pchunks_total * c.st.H * c.st.layers;
  if (chunks < device_sm_count())
    return launch_pdl(k_mixpool<512>, dim3(c.st.pchunks_total * 4, c.st.H, c.st.layers), dim3(256), 0, c.stream, 1, c.st, c.ws,
                      s_div, rbar_in, s_ex_out, s_comp, mix_params(c.p));
  return launch_pdl(k_mixpool<kPChunk>, dim3(c.st.pchunks_total, c.st.H, c.st.layers), dim3(256), 0, c.stream, 1, c.st,
                    c.ws, s_div, rbar_in, s_ex_out, s_comp, mix_params(c.p));
}

// Budgets chosen by the caller (rows to keep per (layer, sequence, head), window included) ->
// candidates to select: minus the window, at least 0, at most B - W and the candidates there are.
__global__ void __launch_bounds__(256)
k_given_budgets(const SeqTable st, const int* __restrict__ budgets, int* __restrict__ counts,
                const int Bp) {
  pdl_launch_dependents();
  pdl_wait();
  const int layer = blockIdx.x, BH = st.batch * st.H;
  for (int t = threadIdx.x; t < BH; t += blockDim.x) {
    const int b = t / st.H;
    const int P = st.cu[b + 1] - st.cu[b] - st.W;
    const int c = budgets[(size_t)layer * BH + t] - st.W;
    counts[(size_t)layer * BH + t] = max(0, min(c, min(Bp, P)));
  }
}

cudaError_t launch_given_budgets(const LaunchCtx& c, const int* budgets, int* counts) {
  return launch_pdl(k_given_budgets, dim3(c.st.layers), dim3(256), 0, c.stream, 1, c.st, budgets,
                    counts, c.p.budget - c.p.window);
}

namespace {
// Clusters of `size` CTAs that the device holds at once with an SM to each CTA (k_tail and k_budget with 1024 threads;
// 120 KB make sure of it).
int alone_clusters(const int size) {
  static std::atomic<bool> done[kMaxDevices];
  static ClusterFit fit;
  (void)answered(ensure_smem(k_tail<true, 1024, true, false>, kTailSmem, done));   // (a failure shows at the launch)
  return fit.ask(k_tail<true, 1024, true, false>, 1024, 120 * 1024, size);
}
// The same with two CTAs to an SM, of 512 threads and half of its shared memory each (adapt_pairs_fit).
int paired_clusters(const int size) {
  static std::atomic<bool> done[kMaxDevices];
  static ClusterFit fit;
  (void)answered(ensure_smem(k_tail<true, 512, true, true>, kTailSmem, done));
  return fit.ask(k_tail<true, 512, true, true>, 512, 113 * 1024 - 24576, size);
}

// CTAs per (sequence, layer) pair: one while it has 8192 keys or less of all heads (the exchanges cost as much as
// the sweeps they save), else as many as leave each that much and are all resident at once, one per SM (15 clusters of
// eight are, 33 of four, 74 of two).  One CTA each / this, whole calls, pairs of 16 heads x keys, us: 4 of 3000 72.7 / 59.5,
// 15 of 4000 245 / 156, 17, 20, 28 of 6000 381 / 248, 433 / 294, 526 / 392, 28, 56 of 2000 163 / 159, 290 / 291, one of
// 30000 806 / 187; 17 of 12 x 2000 92.4 / 87.5.
template <typename Fit>
int budget_clusters(const int pairs, const long long keys, const Fit& alone) {
  int cs = 1;
  while (cs < kBudgetCluster && keys > 8192LL * cs && pairs <= alone(2 * cs)) cs *= 2;
  return cs;
}
}  // namespace

cudaError_t launch_budget(const LaunchCtx& c, const float* scores, int* counts) {
  const int cs = budget_clusters(c.st.batch * c.st.layers, (long long)c.st.H * c.max_prefix, alone_clusters);
  const size_t chunk = ((size_t)c.max_prefix + cs - 1) / cs;
  // the keys of a CTA's slice of the longest sequence in shared memory when they fit
  const size_t want = (size_t)c.st.H * ((chunk + 31) / 32) * 128;
  const size_t cap_bytes = 200 * 1024;
  const size_t smem = want <= cap_bytes ? want : 0;
  if (smem > 20 * 1024) {   // on top of the static shared memory of the search
    static std::atomic<bool> done[kMaxDevices];
    const cudaError_t e = ensure_smem(k_budget, cap_bytes, done);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(k_budget, dim3(c.st.batch * cs, c.st.layers), dim3(kBudgetThreads), smem, c.stream, cs,
                    c.st, scores, counts, c.p.budget - c.p.window, floor_slots(c.p), (int)(smem / 4));
}

// Launch shape of k_tail for the longest sequence of the call.
struct TailShape {
  int cs, threads, chunk;
  bool cached;
};

// CTAs per unit.  One when there are many units or a unit is a block of positions or less (an exchange across a
// cluster costs more than another block).  Few long ones: more of them, always so that all clusters are resident at
// once with an SM to each CTA, and as long as pairs leave an SM over and clusters of four and eight a fifth of them: beyond
// that the exchange costs more than it saves (selection alone, 74 units of 6000 positions on pairs 10.4 us, on one CTA
// each 7.0; 31 of 12000 on four 10.1, on two 8.9; 15 of 30000 on eight 12.3, on four 9.9).
template <typename Fit>
int tail_clusters(const long long units, const int P, const int sms, const Fit& alone) {
  int cs = 1;
  while (cs < kTailMaxCluster && tail_chunk(P, cs) > 4096 && units * 2 * cs <= (cs == 1 ? sms - 1 : sms * 4 / 5) &&
         units <= alone(2 * cs))
    cs *= 2;
  return cs;
}

TailShape tail_shape(const LaunchCtx& c) {
  const long long units = (long long)c.st.layers * c.st.batch * c.st.H;
  const int P = c.max_prefix, sms = device_sm_count();
  TailShape t;
  t.cs = tail_clusters(units, P, sms, alone_clusters);
  // What does not fit shared memory in that many CTAs takes more of them, where there is a place for such a cluster.
  while (t.cs < kTailMaxCluster && tail_chunk(P, t.cs) > kTailCacheCap && alone_clusters(2 * t.cs) > 0) t.cs *= 2;
  t.chunk = tail_chunk(P, t.cs);
  // A CTA alone on its SM: 1024 threads (a block of 4096 positions), fewer when the slice is shorter.  More
  // CTAs than SMs: smaller ones side by side, as many as there are and as shared memory holds (heads of
  // 7300: 256 threads 47 us, 1024 70; 256 heads of 16352: 512 threads 41 us, 1024 47).
  const long long per_sm = (units * t.cs + sms - 1) / sms;
  t.threads = per_sm >= 3 ? 256 : per_sm == 2 ? 512 : t.chunk <= 1024 ? 256 : t.chunk <= 2048 ? 512 : 1024;
  if (per_sm > 1)
    while (t.threads < 1024 &&
           (1024 / t.threads) * (24576 + (size_t)t.chunk * 17 / 4 + (size_t)t.threads * 32) > 226 * 1024)
      t.threads *= 2;
  t.cached = t.chunk <= (t.cs == kTailMaxCluster ? kTailCacheCapFull : kTailCacheCap);
  return t;
}

bool tail_can_fuse(const LaunchCtx& c) { return tail_shape(c).cached; }

// Whether two CTAs of 512 threads share an SM (its shared memory) with a head of P candidates each.
bool adapt_pairs_fit(const int P) {
  return 2 * (24576 + (size_t)tail_chunk(P, 1) * 17 / 4 + 512 * 32) <= 226 * 1024;
}

// Threads of a CTA when the heads of a sequence are a cluster that shares its budget out (k_tail with ADAPT), 0: where
// mix, budget and tail kernels are as good.  What all threads do (sweeps, counts sent to the other heads) is most of it on
// long heads, so 1024 threads, as long as all clusters are resident with an SM to each CTA.  Where they are not, 512 threads
// and two CTAs to an SM, all resident that way.  Heads too long for two to share an SM take 1024 threads in more than one
// wave.  (Layer, sequence) pairs of heads x keys, whole calls, three kernels / this, us:
//   all resident, 1024 (512 threads in brackets): 4 of 8 x 760 32.2 / 27.7 (28.0), 33 of 4 x 760 41.5 / 37.5 (38.6), 1 of
//     4 x 4300 34.8 / 28.3 (27.5), 15 of 8 x 9000 167 / 157 (163), 74 of 2 x 17000 352 / 338 (346), 15 of 8 x 24500 413 /
//     399 (399)
//   not resident (1024 threads in a second wave in brackets): 36 of 4 x 760 42.2 / 39.5 (51.3), 110 of 2 x 4300
//     149 / 138 (154), 23 of 6 x 2300 73.5 / 65.2 (76.3), 38 of 6 x 9000 302 / 285 (296), 60 of 4 x 17000 573 / 551 (564),
//     17 of 8 x 9000 191 / 179 (193), x 17000 335 / 324 (339), 29 of 8 x 17000 561 / 536 (548)
//   too long for pairs: 17 of 8 x 24500 476 / 478, 60 of 4 820 / 801, 23 of 6 476 / 483
// Seven and eight heads of 8192 keys or less in more clusters than are resident one to an SM keep the three kernels: that line
// was drawn when a search fetched its counts from the peers (17 of 8 x 760 48.9 / 52.0).  With the counts sent, 512 threads
// are ahead there as well: 17 of 8 x 760 44.5 / 39.5, x 2300 72.6 / 64.9, 16 of 8 x 8000 161 / 154, 29 of 8 x 4300 164 / 150.
template <typename Alone, typename Paired>
int adapt_threads(const long long sequences, const int heads, const int P, const Alone& alone, const Paired& paired) {
  if (sequences <= alone(heads)) return 1024;
  if (!adapt_pairs_fit(P)) return alone(heads) > 0 ? 1024 : 0;
  return sequences <= paired(heads) && (heads <= 6 || P > 8192) ? 512 : 0;
}

// Whole calls, three kernels against this, us.  One layer: longer heads want more than a CTA each (4 of 32768 67.1 / 67.3,
// 2 of 40000 62.4 / 68.3); more CTAs than are resident together lose what the launches cost (288 units 206 / 211, 896, 28
// layers x 8 ragged sequences, 889 / 924).
constexpr int kAdaptMaxKeys = 24576;
static_assert(kAdaptMaxKeys <= kTailCacheCap, "the keys of a head stay in one CTA");
TailShape adapt_shape(const LaunchCtx& c) {
  return {1, adapt_threads((long long)c.st.layers * c.st.batch, c.st.H, c.max_prefix, alone_clusters, paired_clusters),
          tail_chunk(c.max_prefix, 1), true};
}
bool tail_adapts(const LaunchCtx& c) {
  const int H = c.st.H, Bp = c.p.budget - c.p.window, f = floor_slots(c.p);
  if (c.p.budget_mode != MIXKV_BUDGET_ADAPTIVE || H < 2 || H > kMaxCluster || c.max_prefix > kAdaptMaxKeys) return false;
  if ((long long)c.st.layers * c.st.batch * H > device_sm_count() * 13LL / 8) return false;
  int shortest = c.max_prefix;
  for (int b = 0; b < c.st.batch; ++b) shortest = std::min(shortest, c.st.cu[b + 1] - c.st.cu[b] - c.st.W);
  if ((long long)f + (long long)H * (Bp - f) > shortest) return false;
  return adapt_shape(c).threads != 0;
}

template <bool FUSED, int T, bool CL, bool ADAPT>
cudaError_t launch_tail_t(const LaunchCtx& c, const TailKernelArgs& a, const TailShape& sh,
                          size_t smem) {
  if (smem > 20 * 1024) {   // on top of the static part
    static std::atomic<bool> done[kMaxDevices];
    const cudaError_t e = ensure_smem(k_tail<FUSED, T, CL, ADAPT>, kTailSmem, done);
    if (e != cudaSuccess) return e;
  }
  const dim3 grid(c.st.layers * c.st.batch * c.st.H * sh.cs);
  return launch_pdl(k_tail<FUSED, T, CL, ADAPT>, grid, dim3(T), smem, c.stream, ADAPT ? c.st.H : sh.cs, c.st, c.ws, a);
}

cudaError_t launch_tail(const LaunchCtx& c, const TailArgs& t) {
  TailKernelArgs a;
  a.scores = t.scores;
  a.s_div = t.s_div;
  a.rbar_in = t.rbar_in;
  a.s_comp_out = t.s_comp_out;
  a.counts_dev = t.counts_dev;
  a.counts_out = t.counts_out;
  a.idx = t.idx;
  a.idx_offsets = t.idx_offsets;
  a.out_row_offsets = t.out_row_offsets;
  a.K = (const __nv_bfloat16*)t.K;
  a.V = (const __nv_bfloat16*)t.V;
  a.K_out = (__nv_bfloat16*)t.K_out;
  a.V_out = (__nv_bfloat16*)t.V_out;
  a.Bp = c.p.budget - c.p.window;
  a.floor_slots = floor_slots(c.p);
  a.kv_layer_stride = c.kv_layer_stride;
  a.idx_cap = c.idx_cap;
  a.out_rows_cap = c.out_rows_cap;
  a.status_clear = t.status_clear;
  a.mp = mix_params(c.p);
  const TailShape sh = t.adapt ? adapt_shape(c) : tail_shape(c);
  const bool fused = t.scores == nullptr;
  a.cached = sh.cached ? 1 : 0;
  if (fused && !a.cached) return cudaErrorInvalidValue;   // callers check tail_can_fuse() first
  // bitmaps of kept and of equal positions, the keys, the pooling stage
  size_t smem = (size_t)tail_keys_at(sh.chunk) * 4;
  if (a.cached) smem += (size_t)sh.chunk * 4;
  if (fused) smem += ((size_t)8 * sh.threads + 64) * 4;
  auto launch = [&](auto threads) {
    constexpr int T = decltype(threads)::value;
    if constexpr (T >= 512)
      if (t.adapt)
        return fused ? launch_tail_t<true, T, true, true>(c, a, sh, smem) : launch_tail_t<false, T, true, true>(c, a, sh, smem);
    if (sh.cs > 1)
      return fused ? launch_tail_t<true, T, true, false>(c, a, sh, smem) : launch_tail_t<false, T, true, false>(c, a, sh, smem);
    return fused ? launch_tail_t<true, T, false, false>(c, a, sh, smem) : launch_tail_t<false, T, false, false>(c, a, sh, smem);
  };
  switch (sh.threads) {
    case 256: return launch(std::integral_constant<int, 256>());
    case 512: return launch(std::integral_constant<int, 512>());
    default: return launch(std::integral_constant<int, 1024>());
  }
}

}  // namespace mixkv

extern "C" int mixkv_internal_tail_clusters(int64_t units, int32_t candidates, int32_t sms, const int32_t* alone) {
  return mixkv::tail_clusters(units, candidates, sms, [&](const int n) { return alone[n]; });
}
extern "C" int mixkv_internal_adapt_threads(int64_t sequences, int32_t heads, int32_t candidates, const int32_t* alone,
                                            const int32_t* paired) {
  return mixkv::adapt_threads(sequences, heads, candidates, [&](const int n) { return alone[n]; },
                              [&](const int n) { return paired[n]; });
}
extern "C" int mixkv_internal_search_rounds(uint32_t lo, uint32_t hi, uint32_t key, uint32_t* base, uint32_t* span,
                                            int32_t* shift) {
  mixkv::SelRange r = mixkv::sel_range(lo, hi);
  for (int n = 0;; ++n) {
    base[n] = r.base, span[n] = r.span, shift[n] = r.shift;
    if (r.shift == 0) return n + 1;
    r = mixkv::sel_bin(r, (key - r.base) >> r.shift, hi);
    r.shift = mixkv::sel_next_shift(r.shift);
  }
}
extern "C" int mixkv_internal_budget_clusters(int32_t pairs, int64_t keys_per_pair, const int32_t* alone) {
  return mixkv::budget_clusters(pairs, keys_per_pair, [&](const int n) { return alone[n]; });
}
