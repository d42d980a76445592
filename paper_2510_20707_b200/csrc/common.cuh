// Shared declarations of the MixKV CUDA library (sm_100a): problem description handed to
// every kernel, the workspace carve-up, and small device helpers.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "mixkv.h"

namespace mixkv {

constexpr int kHeadDim = 128;        // d, fixed
constexpr int kMaxBatch = 64;        // sequences per call
constexpr int kMaxLayers = 1024;     // layers per call
constexpr int kMaxNQ = 240;          // G*W upper bound (16 spare rows carry the mean key)
constexpr int kTile = 128;           // keys per tensor-core tile
constexpr int kPChunk = 2048;        // candidate positions per CTA in pool / mix
constexpr int kExtraRows = 16;       // rows appended to the query tile in pass 2
constexpr int kMaxCluster = 8;       // CTAs of a cluster (the portable limit)
constexpr float kLog2e = 1.4426950408889634f;

// Tiles split contiguously over g CTAs, in (layer, sequence, head) order.  Runs of n tiles are shared out over p CTAs each
// (p <= n): the first r of them take q + 1 tiles, the others q.  Either one run of all tiles over all CTAs, or, where
// that makes no CTA's share longer than split_tiles() allows, a run per head, so that no CTA works on two of them.
struct Split {
  int n, p, q, r, g;
};
// First tile of CTA c.
__host__ __device__ __forceinline__ int cta_first_tile(const int c, const Split& sp) {
  const int run = c / sp.p, k = c - run * sp.p;
  return run * sp.n + k * sp.q + (k < sp.r ? k : sp.r);
}
// CTA whose contiguous range contains tile t.
__host__ __device__ __forceinline__ int tile_owner(const int t, const Split& sp) {
  const int run = t / sp.n, k = t - run * sp.n, big = sp.r * (sp.q + 1);
  return run * sp.p + (k < big ? k / (sp.q + 1) : sp.r + (k - big) / sp.q);
}

// Everything a kernel needs to find its slice of the ragged batch.
struct SeqTable {
  int layers;                        // layers handled by one call (an outer batch dimension)
  int batch, H, G, W, NQ;
  int Ltot, Ptot;
  int pchunks_total;                 // sum over sequences of ceil(P_b / kPChunk)
  int cu[kMaxBatch + 1];             // sequence offsets into Ltot
  int pchunk_start[kMaxBatch + 1];   // prefix sum of candidate chunks
  // persistent 128-key tile schedules of the two tensor-core passes, (b, h, t) order
  // Tiles of one layer: nt1 over all L keys (pass 1), nt2 over the P candidate keys (pass 2).
  int nt1, nt2;
  Split sp1, sp2;                    // of the tiles of all layers over the CTAs of the passes
  int tile1_start[kMaxBatch + 1];    // prefix sum of H * ceil(L_b / 128)
  int tile2_start[kMaxBatch + 1];    // prefix sum of H * ceil(P_b / 128)
};

// Device workspace carve-up (all pointers into the caller's workspace).
struct Workspace {
  // every array below has a leading [layers] dimension
  float* kinv;        // [H, Ltot]   1 / |K_i|  (0 for a zero key)
  float* vnorm;       // [H, Ptot]   |V_i|
  float* s_ex_raw;    // [H, Ptot]   window attention score before pooling
  float* s_div;       // [H, Ptot]
  float* s_comp;      // [H, Ptot]
  // per-segment partial results; a segment is a run of tiles of one (b, h) inside one CTA's
  // range and its slot is the id of its first tile
  float2* rowstat;    // [nt1, NQ]  softmax (reference, sum) of each window row, log2 units
  float* ksum;        // [nt1, d]      sum of unit keys
  float4* vstat;      // [nt2]         (min, max, sum, -) of |V_i| over candidates
  float4* dstat;      // [nt2, 2]      per pair of epilogue warpgroups: (min, max, sum) of s_div, window-count-weighted sum of s_ex_raw
  float* exsum;       // [H, pchunks_total]   per-chunk sum of pooled s_ex (max pooling only)
  float* rbar;        // [batch*H]   redundancy of Eq. 4, left by pass 2
  int* counts;        // [batch*H]
  int* idx_offsets;   // [batch*H + 1]
  int* idx;           // [batch*H*(B-W)]
  size_t bytes;
};

struct LaunchCtx {
  SeqTable st;
  Workspace ws;
  mixkv_params p;
  long long kv_layer_stride;   // elements between the K (V) tensors of consecutive layers
  long long q_layer_stride;    // elements between the window queries of consecutive layers
  int idx_cap;                 // selected rows one layer can produce (capacity of its index list)
  int out_rows_cap;            // output rows reserved per layer: batch * H * B
  float scale_log2e;   // softmax scale * log2(e)
  int max_seq_len;
  int max_prefix;
  cudaStream_t stream;
  void* const* trace_events;  // optional measurement hook: events recorded between kernels
  int n_trace_events;
  mutable int stage;
  bool clear_status;          // the first kernel sets the status word to 0

  // Records the event that marks the start of the next kernel (or the end of the last).
  void mark() const {
    if (trace_events && stage < n_trace_events && trace_events[stage])
      cudaEventRecord((cudaEvent_t)trace_events[stage], stream);
    ++stage;
  }
};

// ---- kernels (defined in the .cu files) ------------------------------------------
cudaError_t launch_pass1(const LaunchCtx& c, const void* K, const void* Q, int* status);
cudaError_t launch_pass2(const LaunchCtx& c, const void* K, const void* V, const void* Q,
                         float* s_div_out, float* rbar_out, int* status);
constexpr int kMaxDevices = 64;   // what is looked up or set once per device is remembered for so many
int device_sm_count();
// Whether a question to the runtime was answered.  For those that a call can do without the answer of: their error is
// not left behind as the thread's last one, where the caller's next check would take it for its own.
inline bool answered(const cudaError_t e) {
  if (e != cudaSuccess) (void)cudaGetLastError();
  return e == cudaSuccess;
}
// The current device as an index into what is remembered per device; -1: none, or one past the end.
inline int device_slot() {
  int dev = -1;
  return answered(cudaGetDevice(&dev)) && dev >= 0 && dev < kMaxDevices ? dev : -1;
}
// Lets `kernel` have `smem` bytes of dynamic shared memory on the current device, once per device; `done` is the
// kernel's own array (static: entry points may run in several threads at once).
template <typename F>
cudaError_t ensure_smem(F kernel, size_t smem, std::atomic<bool> (&done)[kMaxDevices], const int dev = device_slot()) {
  if (dev >= 0 && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess && dev >= 0) done[dev].store(true, std::memory_order_release);
  return e;
}
// Clusters of 1 .. 8 CTAs of one kernel that the current device holds at once.  A cluster lies in one group of SMs, and
// how the SMs of a chip fall into groups differs between chips of one model, so the runtime is asked, once per device
// and size (0.2 us a question); `kernel` may already have its shared memory.  No answer counts as none and is not
// remembered.  Without a device: as if SMs were all alike.
struct ClusterFit {
  std::atomic<int> known[kMaxDevices][kMaxCluster + 1];   // 0: not asked, else the answer + 1
  template <typename F>
  int ask(F kernel, int threads, size_t smem, int size, const int dev = device_slot()) {
    if (dev >= 0)
      if (const int k = known[dev][size].load(std::memory_order_relaxed)) return k - 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)size);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)size;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (!answered(cudaOccupancyMaxActiveClusters(&n, kernel, &cfg))) return dev >= 0 ? 0 : device_sm_count() / size;
    if (dev >= 0) known[dev][size].store(n + 1, std::memory_order_relaxed);
    return n;
  }
};
// Fills a CUtensorMap (passed as void*) for a tensor of 16-bit elements of the given rank: dims innermost first,
// strides in bytes of dimensions 1 .. rank-1, box extents; 128-byte swizzle, zero fill outside.
bool encode_map_16bit(void* tm, const void* base, int rank, const unsigned long long* dims,
                     const unsigned long long* strides_bytes, const unsigned* box);
// MIXKV_OK on a compute-capability 10.x device, MIXKV_ERR_UNSUPPORTED on any other,
// MIXKV_ERR_CUDA when none can be queried; *major_out (optional) receives the major number.
int device_check(int* major_out);
cudaError_t launch_poolsum(const LaunchCtx& c);
cudaError_t launch_mixpool(const LaunchCtx& c, const float* s_div, const float* rbar_in,
                           float* s_ex_out, float* s_comp);
cudaError_t launch_budget(const LaunchCtx& c, const float* scores, int* counts);
// Index of (layer, head h, sequence b, position i) in a [layers, H, Ltot] / [layers, H, Ptot]
// array.
__host__ __device__ __forceinline__ size_t kpos(const SeqTable& st, int layer, int h, int b,
                                                int i) {
  return ((size_t)layer * st.H + h) * st.Ltot + st.cu[b] + i;
}
__host__ __device__ __forceinline__ size_t ppos(const SeqTable& st, int layer, int h, int b,
                                                int i) {
  return ((size_t)layer * st.H + h) * st.Ptot + (st.cu[b] - b * st.W) + i;
}

// Gram matrix of the block sums of a similarity map (similarity_tc.cu).
struct GramArgs {
  const void* parts;   // [2][heads][T][d] fp16 (block 1: bf16): the scaled block sums as value and remainder
  float inv_scale2;    // one over the square of the scale
  const int* nz;       // [heads][T]       non-zero rows of a block
  const float* us;     // [heads][slices][d]  partial sums of all unit rows of a head
  const int* nzs;      // [heads][slices]
  int slices, heads, L, block, T;
  float* cells;        // [heads][T][T]
  float* mean;         // [heads] or nullptr
};
cudaError_t launch_gram(const GramArgs& g, cudaStream_t s);

// Selection (and optionally the mix before it and the gather after it), one CTA or cluster per
// (layer, sequence, head).  scores != nullptr: select on them; else mix first (s_div, rbar_in) and
// write the mixed scores to s_comp_out.  counts_dev == nullptr: fixed budgets.
struct TailArgs {
  const float* scores;
  const float* s_div;
  const float* rbar_in;
  float* s_comp_out;
  const int* counts_dev;
  int* counts_out;
  int* idx;
  int* idx_offsets;
  int* out_row_offsets;
  const void* K;
  const void* V;
  void* K_out;
  void* V_out;
  int* status_clear;   // optional word set to 0
  bool adapt;          // adaptive budgets shared out by this kernel (tail_adapts)
};
// counts [layers, batch*H] <- candidates to select for budgets [layers, batch*H] given by the caller
cudaError_t launch_given_budgets(const LaunchCtx& c, const int* budgets, int* counts);
cudaError_t launch_tail(const LaunchCtx& c, const TailArgs& a);
// Whether the longest sequence is short enough for the fused mix + select + gather kernel.
bool tail_can_fuse(const LaunchCtx& c);
// Whether that kernel can share adaptive budgets out itself: the heads of a sequence make a cluster, every head's
// candidates fit one CTA, and even a head that got all shared rows would not run out of candidates (the rows of a
// sequence are then known without looking at the others).
bool tail_adapts(const LaunchCtx& c);
// Whether pass 2 is launched with the spare warp's folds, from the splits of both passes, the tiles of pass 2, the heads of the
// call ((layer, sequence, head) units) and the pass-1 tiles of the longest.
bool pass2_spare(const Split& sp1, const Split& sp2, int tiles2, int heads, int longest);

// Launch with programmatic dependent launch (and an optional cluster size): the kernel may
// start while its predecessor in the stream drains; every kernel calls pdl_wait() before it
// touches global memory that an earlier one may still write or read (pass 2 loads the call's inputs without).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t stream, int cluster, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  int n = 0;
  attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[n].val.programmaticStreamSerializationAllowed = 1;
  ++n;
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = (unsigned)n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ---- device helpers ----------------------------------------------------------------
__device__ __forceinline__ int find_seq(const int* start, int batch, int x) {
  int b = 0;
  while (b + 1 < batch && x >= start[b + 1]) ++b;
  return b;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_min(const float v) {   // (one instruction where five exchanges and comparisons did it)
  float r;
  asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float warp_max(const float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

// Programmatic dependent launch: let the next kernel of the stream be scheduled, and wait
// until everything before this kernel in the stream has completed and is visible.
//
// Where a kernel lets the next one start costs more than what that one gains by being there early: the passes do it with
// the last tile but one, the tail ahead of its gather.  At the top of all three / behind their waits / once the passes' last
// MMA was issued, us a call: one layer of 4 x 1024 keys 20.7 / 20.6 / 18.5, of 4 x 32768 50.0 / 48.0 / 47.4, 28 layers of
// 4 x 4096 108.7 / 107.4 / 103.3, scores and selection of three sequences 58.6 / 57.3 / 54.8; never (at the end of a CTA)
// 20.9, 49.6, 104.9, 56.3.  A tile earlier than that: 18.2 -> 18.1, 45.7 -> 45.5, level, 54.9 -> 54.3 (two and three
// tiles earlier 56.5 on the last).
// The mix, budget, decode and similarity kernels gain nothing or lose by it (4 x 32768 rows in blocks of 16 30.6 at the top,
// 30.9 to 32.3 later) and keep theirs at the top.
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Packed fp32 pairs (one instruction for two lanes of arithmetic).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// The two bf16 of a word as a packed fp32 pair (low half first), built in place in the 64-bit
// register (a pair assembled from two separate floats costs moves).
__device__ __forceinline__ f32x2 bf16x2_wide(const uint32_t w) {
  return ((unsigned long long)(w & 0xffff0000u) << 32) | (unsigned long long)(w << 16);
}

}  // namespace mixkv
