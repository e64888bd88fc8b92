// Shared device/host helpers of the MoIN CUDA library (sm_100a only).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <limits.h>
#include <stdint.h>

#include "../../include/moin.h"

namespace moin {

// ----------------------------------------------------------------------------------------
// Device status block (one per process; its device address is passed to kernels).
// ----------------------------------------------------------------------------------------
struct DeviceStatus {
  int timeout_flag;
  int timeout_site;
  int invalid_expert_ids;
  int reserved[5];
};

// Plan buffer layout (int32 words).  Header first, then the arrays.
constexpr int kPlanHeaderWords = 16;
enum PlanHeader { PH_NSEG = 0, PH_NTILES = 1, PH_NLORA = 2, PH_MAXSEG = 3, PH_T = 4, PH_E = 5, PH_NCHUNK = 6, PH_NGEMM = 7 };
constexpr int kSegChunk = 8;      // token columns of one warp MMA: what a work item of the stream kernels covers
constexpr int kPlanChunk = 256;   // tokens per histogram chunk
constexpr int kTileRows = 128;    // rows per tile
constexpr int kTileRuns = 4;      // runs a row tile of the long-run GEMM covers at most

struct PlanView {   // pointers into the plan buffer
  int* header;
  int* perm;         // [T]   token indices ordered by (expert, token)
  int* seg_expert;   // [Smax]
  int* seg_start;    // [Smax + 1]
  int4* seg_tab;     // [Smax + 1] packed (expert, start, length, 0): one 16-byte load per segment
  int4* chunk_tab;   // [Cmax] the segments cut into pieces of at most kSegChunk tokens: (expert, start, length, 0)
  int* tile_row0;    // [T + 1]
  int* tile_rows;    // [T]
  int* tile_expert;  // [T]
  // Row tiles of the long-run GEMM: the regular grid of kTileRows rows, whatever runs of one expert it cuts (a grid tile
  // of more than kTileRuns runs is cut at run boundaries): (first row, rows, first run, runs).
  int4* gemm_tab;    // [T]
  int* run_expert;   // [T]   runs in token order: expert or -1
  int* run_row0;     // [T + 1] their first rows
  int* grid_run;     // [grid tiles] run of the grid tile's first row
  int* grid_nrun;    // [grid tiles] runs in it
  int* rank;         // [T]   scratch
  int* key;          // [T]   scratch
  int* keybase;      // [E+1] scratch
  int* chunkbase;    // [E+1] scratch
  int* hist;         // [n_chunks * (E+1)] scratch
  int T, E, Smax, Cmax, n_chunks;
};

__host__ __device__ inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

inline PlanView plan_view(void* buffer, int T, int E, size_t* total_words = nullptr) {
  PlanView v;
  v.T = T; v.E = E;
  v.Smax = T < E ? T : E;
  v.Cmax = T / kSegChunk + v.Smax;
  v.n_chunks = (T + kPlanChunk - 1) / kPlanChunk;
  int* base = reinterpret_cast<int*>(buffer);
  size_t off = 0;
  auto take = [&](size_t n) { size_t o = off; off += align_up(n, 4); return base ? base + o : nullptr; };
  v.header = take(kPlanHeaderWords);
  v.perm = take(T);
  v.seg_expert = take(v.Smax + 1);
  v.seg_start = take(v.Smax + 2);
  v.seg_tab = reinterpret_cast<int4*>(take(4 * (size_t)(v.Smax + 1)));
  v.chunk_tab = reinterpret_cast<int4*>(take(4 * (size_t)(v.Cmax + 1)));
  v.tile_row0 = take(T + 1);
  v.tile_rows = take(T + 1);
  v.tile_expert = take(T + 1);
  v.gemm_tab = reinterpret_cast<int4*>(take(4 * (size_t)(T + 1)));
  v.run_expert = take(T + 1);
  v.run_row0 = take(T + 2);
  v.grid_run = take(T / kTileRows + 2);
  v.grid_nrun = take(T / kTileRows + 2);
  v.rank = take(T);
  v.key = take(T);
  v.keybase = take(E + 2);
  v.chunkbase = take(E + 2);
  v.hist = take((size_t)v.n_chunks * (size_t)(E + 1));
  if (total_words) *total_words = off;
  return v;
}
inline size_t plan_bytes(int T, int E) {
  size_t words = 0;
  plan_view(nullptr, T, E, &words);
  return words * sizeof(int);
}

// ----------------------------------------------------------------------------------------
// Small device utilities
// ----------------------------------------------------------------------------------------
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Four 8-bit float codes (e4m3) -> bf16(fp32(value * scale)), in order: two to a word.
__device__ __forceinline__ void fp8x4_to_bf16(uint32_t codes, float scale, uint32_t& lo, uint32_t& hi) {
  uint32_t h0, h1;   // the values as fp16 (exact)
  asm("{\n .reg .b16 a, b;\n mov.b32 {a, b}, %2;\n cvt.rn.f16x2.e4m3x2 %0, a;\n cvt.rn.f16x2.e4m3x2 %1, b;\n}\n"
      : "=r"(h0), "=r"(h1) : "r"(codes));
  const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&h0)), f1 = __half22float2(*reinterpret_cast<const __half2*>(&h1));
  lo = pack_bf16(f0.x * scale, f0.y * scale);
  hi = pack_bf16(f1.x * scale, f1.y * scale);
}

// Streaming 16-byte load that does not allocate in L1 (adapter weights are read once).
__device__ __forceinline__ uint4 ldg_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ uint4 ldg_cached(const void* p) {
  return __ldg(reinterpret_cast<const uint4*>(p));
}

// mma.sync m16n8k16, bf16 x bf16 -> fp32 (warp-level tensor-core path for the skinny LoRA products)
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Function between the two low-rank matrices (MOIN_ACT_*).
__device__ __forceinline__ float lora_act(float v, int act) {
  switch (act) {
    case MOIN_ACT_RELU: return fmaxf(v, 0.f);
    case MOIN_ACT_SILU: return v / (1.f + __expf(-v));
    case MOIN_ACT_GELU: return 0.5f * v * (1.f + erff(v * 0.70710678118654752f));
    default: return v;
  }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Router: (similarity, index) as a 64-bit key whose maximum is the best similarity, among equals the lowest index.
__device__ __forceinline__ unsigned long long route_key(float sim, int k) {
  uint32_t u = __float_as_uint(sim);
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ((unsigned long long)u << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)k);
}
__device__ __forceinline__ float key_to_float(uint32_t u) {   // upper half of a key
  u = (u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u;
  return __uint_as_float(u);
}

// Programmatic dependent launch: the next kernel of the stream may start once every CTA has got here / this CTA goes
// on once the kernels before it are complete and their writes visible (no-ops in an ordinary launch).  The kernels of a
// call are launched this way, so that a kernel's launch latency and set-up lie under the tail of the one before it
// (about 2 us each).  Rule: a kernel waits before it touches global memory and lets the next one start only after that
// - then everything before a running kernel is complete but the kernel right before it.  Four kernels differ, and say
// beside their code how the order is kept: the adapter shrink beside the decode GEMM, which does not wait at its start
// (its last CTA waits at its end); the expand behind it, which reads the plan and starts on the adapters before it waits,
// and lets the next kernel start at once; route_parts_kernel, which reads the queries before it waits; and the decode GEMM
// of a forward (w_early), which reads weights before it waits, and so must not stand behind a kernel that lets it start
// before waiting itself: never right behind the shrink or the expand.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void pdl_begin() {
  pdl_wait();
  pdl_launch_dependents();
}
// Launch as the programmatic dependent of the kernel before it in the stream.
template <class... P, class... A>
inline cudaError_t launch_pdl(void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, P(args)...);
}

// Launchers implemented in the .cu files (host side).
int plan_launches(int T, int E);   // kernels launch_plan_build issues for this shape
cudaError_t launch_plan_build(const int* token_expert, const PlanView& v, DeviceStatus* status, bool want_tiles,
                              cudaStream_t stream);
// Register-fed short-segment kernels: one launch covers up to kMaxStreamJobs projections sharing a plan.
constexpr int kMaxStreamJobs = 4;
struct ShrinkJobs {
  const __nv_bfloat16* x[kMaxStreamJobs];
  const __nv_bfloat16* A[kMaxStreamJobs];
  float* h[kMaxStreamJobs];
  const int* slot_of_expert[kMaxStreamJobs];
  const int* slot_rank[kMaxStreamJobs];   // per-slot rank (nullptr: the pool's r)
  int r[kMaxStreamJobs], d_in[kMaxStreamJobs], per_seg[kMaxStreamJobs];
  int n;
};
struct ExpandJobs {
  const float* h[kMaxStreamJobs];
  const __nv_bfloat16* B[kMaxStreamJobs];
  const float* y0[kMaxStreamJobs];
  __nv_bfloat16* y[kMaxStreamJobs];
  const int* slot_of_expert[kMaxStreamJobs];
  const int* slot_rank[kMaxStreamJobs];   // per-slot rank (nullptr: the pool's r)
  int act[kMaxStreamJobs];                // MOIN_ACT_* applied to h
  int r[kMaxStreamJobs], d_out[kMaxStreamJobs], per_seg[kMaxStreamJobs];
  int n;
};
cudaError_t launch_lora_shrink_stream(const PlanView& pv, ShrinkJobs jobs, int n_sms, cudaStream_t stream);
cudaError_t launch_lora_expand_stream(const PlanView& pv, ExpandJobs jobs, float scale, int n_sms,
                                      cudaStream_t stream);
cudaError_t launch_gemm_warp(const __nv_bfloat16* x, const __nv_bfloat16* W, __nv_bfloat16* y, float* y0, int T,
                             int d_in, int d_out, cudaStream_t stream);
cudaError_t launch_route_top2_simple(const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm,
                                     const int* cmap, int Q, int K, int D, int* out_expert, int* out_centroid,
                                     int* out_second, float* out_best, float* out_margin, cudaStream_t stream);
cudaError_t launch_route_finish_top2(const unsigned long long* keys, const unsigned long long* keys2,
                                     const __nv_bfloat16* q, const int* cmap, int Q, int D, int* out_expert,
                                     int* out_centroid, int* out_second, float* out_best, float* out_margin,
                                     cudaStream_t stream);
bool kmeans_update_split(int K, int D, int n_sms);   // column groups apart, norms in a second launch
cudaError_t launch_kmeans_update(const PlanView& pv, const __nv_bfloat16* x, const __nv_bfloat16* c_old,
                                 __nv_bfloat16* c_new, float* inv_new, int D, int n_sms, cudaStream_t stream);
cudaError_t launch_inv_norm(const __nv_bfloat16* c, int K, int D, float* inv_norm, cudaStream_t stream);
cudaError_t launch_route_simple(const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm,
                                const int* cmap, int Q, int K, int D, int* out_expert, int* out_centroid,
                                float* out_best, cudaStream_t stream);
bool route_cluster_supported(int Q, int K, int D);
bool route_few_topics(int Q, int K, int D);   // left to the CUDA-core kernel
cudaError_t launch_route_cluster(const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm,
                                 const int* cmap, int Q, int K, int D, int* out_expert, int* out_centroid,
                                 float* out_best, unsigned long long* part_keys, cudaStream_t stream);
// Parts the cluster kernel cuts the table into: a cluster each, given route_parts(Q, K, D) * Q keys of scratch (top-2:
// twice as many); with part_keys == nullptr one cluster walks them all, with the same results to the bit.
constexpr int kRouteMaxParts = 12;
constexpr int kRouteMaxPartKeys = 12 * 32;   // queries x parts where there is more than one: at most 12 clusters of up to 32 queries
int route_parts(int Q, int K, int D);
cudaError_t launch_route_top2_cluster(const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm,
                                      const int* cmap, int Q, int K, int D, int* out_expert, int* out_centroid,
                                      int* out_second, float* out_best, float* out_margin,
                                      unsigned long long* part_keys, cudaStream_t stream);
// keys[0 .. n) = 0: a kernel of the chain rather than a memset, which neither starts under the kernel before it nor lets
// the next one set up under it (K-means iteration 83 -> 80.6 us, 200
// queries x 5000 x 768 12.3 -> 11.8 us).
cudaError_t launch_clear_keys(unsigned long long* keys, size_t n, cudaStream_t stream);
// out_best[i] /= |q_i| (-inf stays)
cudaError_t launch_route_cosine(const __nv_bfloat16* q, int Q, int D, float* out_best, cudaStream_t stream);
cudaError_t launch_route_finish(const unsigned long long* keys, const __nv_bfloat16* q, const int* cmap, int Q, int D,
                                int* out_expert, int* out_centroid, float* out_best, cudaStream_t stream);

// Host state of the entry points (api.cu): one record per device ordinal, filled on the first call made with
// that device current.  The status block's address and the kernels' shared-memory opt-ins belong to one device, so
// nothing here is shared between devices.
constexpr int kMaxDevices = 64;
constexpr int kOptinSlots = 19;
struct HostState {
  DeviceStatus* status = nullptr;  // device address of the status block
  int device = -1;
  int n_sms = 0;
  int gemm_impl = 0;               // MOIN_OPT_GEMM_IMPL (process-wide option, copied in on every call)
  size_t smem_optin[kOptinSlots] = {};   // dynamic shared memory already opted in, per kernel (see ensure_smem_optin)
};
moin_status host_state(HostState** out);      // lazily initialised for the current device
moin_status record_cuda(cudaError_t e);       // MOIN_OK or MOIN_ERR_CUDA (remembers e)

// Kernels that need more than 48 KB of dynamic shared memory opt in with cudaFuncSetAttribute; the driver keeps
// that attribute per device, so the "already done" note is kept per device too (slot = one id per kernel).
enum {
  OPTIN_ROUTE_CLUSTER = 0, /* .. 7 */ OPTIN_ROUTE_SIMPLE = 8, OPTIN_ATTENTION = 9, OPTIN_DECODE_GEMM = 10,
  OPTIN_DECODE_GEMM_FP8 = 11, OPTIN_TC_SHRINK = 12, OPTIN_TC_PAIR = 13, /* .. 17 */ OPTIN_DECODE_GEMM_EARLY = 18
};
template <class Fn>
inline cudaError_t ensure_smem_optin(int slot, Fn* fn, size_t bytes) {
  HostState* hs = nullptr;
  if (host_state(&hs) != MOIN_OK) return cudaErrorInvalidDevice;
  if (hs->smem_optin[slot] >= bytes) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) hs->smem_optin[slot] = bytes;
  return e;
}

// Brackets the launches issued during its lifetime with two CUDA events when profiling is enabled.
struct ProfScope {
  ProfScope(int kernel, int launches, cudaStream_t stream);
  ~ProfScope();
  int slot;
  cudaStream_t stream;
  bool nvtx;
};

}  // namespace moin
