// tcgen05 / TMEM / TMA GEMM family (host-side interface).
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace moin {

// 2-D row-major bf16 tensor [rows, cols] -> TMA map with a [box_rows x 64] box, 128-byte swizzle, zero fill
// (columns of the box beyond `cols` read as zero).
moin_status make_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows);

// The same for bytes: a [box_rows x 64] box, 64-byte swizzle.
moin_status make_map_u8(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows);

// bf16 [T][n_heads][64]: a box of box_t tokens x box_heads heads.
moin_status make_map_heads(CUtensorMap* map, const void* base, uint64_t T, uint32_t n_heads, uint32_t box_heads, uint32_t box_t);

// Shape predicates (host): can the tcgen05 kernels take this problem?
bool tc_gemm_supported(int T, int d_in, int d_out);
bool tc_router_supported(int Q, int K, int D);
bool tc_fused_supported(int r);

// y = x W^T (bf16) and optionally y0 = x W^T (fp32) for few tokens, up to kMaxStreamJobs projections in one launch
// (gemm_decode.cu).
// w_scale != nullptr: W is 8-bit float codes with a scale per row (all jobs of a launch alike), T <= kDecodeFp8MaxT without
// adapters, kDecodeSegMaxT beside those of short segments.
struct DecodeGemmJob { const __nv_bfloat16* x; const void* W; __nv_bfloat16* y; float* y0; int d_in, d_out; const float* w_scale; };
constexpr int kDecodeGemmMaxT = 512, kDecodeFp8MaxT = 512;
// Beside the adapters of short segments it takes more tokens: one launch for a group and the shrink under it, where CTA pairs take
// a launch a projection, store the fp32 copy from registers and leave the shrink no SM.  Forwards in segments of 12 tokens by
// pairs / by this kernel, ms: rank 64 636 tokens 7.41 / 5.64, 1020 9.43 / 7.83, 2004 14.7 / 13.2; rank 16 4.85 / 4.01, 5.82 / 5.50,
// 10.4 / 8.8; 8-bit base, rank 64 8.28 / 5.78, 10.2 / 8.40, 15.6 / 13.9.  Beyond 2048 tokens it gives nothing at rank 8 (2400 to 4000
// tokens x 0.96 to 1.01) and 128 (0.96 to 1.06), 2 to 8 % between.  With an adapter for three requests in ten the gain is smaller
// (rank 64 5.46 / 5.57 at 800 tokens, 6.04 / 6.37 at 1024, 8.98 / 7.60 at 1400).
// A forward's groups only, which together gain: a layer call may be one projection by itself, or of a batch of which few tokens
// have an adapter, and loses (1024 tokens in runs of 12, pairs / this kernel, us: 2048 -> 2048 of rank 16 25.9 / 31.2, of rank 64
// with an adapter for a tenth of the tokens 20.7 / 26.8; 704 -> 760 14.5 / 18.6).
constexpr int kDecodeSegMaxT = 2048;
// small_tiles: the rule for narrow adapters (see there).  w_early: W may be read before this kernel waits (8-bit codes always are).
// Only where the kernel right before in the stream writes no weights and waits before it lets this one start, so that all older
// ones (a copy or a conversion of W) are complete by then: behind a norm, an attention or a SwiGLU of this library, not behind the
// adapter shrink or expand, which let the next kernel start first, and not in a call whose neighbours are not known.
moin_status launch_decode_gemm(HostState* hs, const DecodeGemmJob* jobs, int n_jobs, int T, bool small_tiles, bool w_early, cudaStream_t stream);
// moin_lora_linear_group, and what a decoder forward says beside it (nullptr: a layer call).  w_scale != nullptr: a base of 8-bit
// codes, jobs[j].W points to them and w_scale[j] to their row scales; short segments and few tokens only.
struct ForwardGroup { const float* const* w_scale; bool w_early; };
inline bool decode_fp8_supported(const HostState* hs, int T, bool segments) {
  return hs->gemm_impl != 1 && T <= (segments ? kDecodeSegMaxT : kDecodeFp8MaxT);
}
moin_status lora_linear_group(const moin_plan* plan, const moin_lora_job* jobs, int n_jobs, const ForwardGroup* forward, float scale,
                              void* workspace, size_t workspace_bytes, moin_stream stream);
// Long-run GEMMs on CTA pairs (tc_pair.cu): y_j = x_j W_j^T for up to kPairJobs projections of one K; with a plan the
// low-rank term s x A_e^T B_e^T is added from hb (hi / lo parts of s x A_e^T, [2][M][r], all jobs of the same r).
constexpr int kPairJobs = 3;
struct PairJob { const __nv_bfloat16 *x, *W, *hb; __nv_bfloat16* y; float* y0; const moin_pool* pool; int N; };   // y0: fp32 copy or nullptr
moin_status launch_pair_gemm(HostState* hs, const PlanView* pv, const PairJob* jobs, int n_jobs, int M, int K,
                             cudaStream_t stream);
// jobs[0].y = silu(x Wg^T + ..) * (x Wu^T + ..): gate and up projection (of one x, N and rank) in one launch.
moin_status launch_pair_swiglu(HostState* hs, const PlanView* pv, const PairJob* jobs, int M, int K, cudaStream_t stream);
// Can a block's gate and up projections take that path (pools: both, or nullptr without adapters)?
bool swiglu_supported(const HostState* hs, const moin_plan* plan, const moin_pool* pools, int T, int d_in, int d_out);
// ... and the path: the shrinks, then launch_pair_swiglu.  jobs[0].y is the result, jobs[1].y is not written.
moin_status lora_swiglu(HostState* hs, const moin_plan* plan, const moin_lora_job* jobs, float scale, int T, int d_in,
                        int d_out, void* workspace, size_t workspace_bytes, cudaStream_t stream);
// keys[i] = max over k of (orderable(<q_i,c_k> * inv_norm[k]) << 32 | (0xFFFFFFFF - k)), merged with atomicMax.
moin_status launch_pair_router(HostState* hs, const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm, int Q,
                               int K, int D, unsigned long long* keys, cudaStream_t stream,
                               unsigned long long* keys2 = nullptr);   // keys2 != nullptr: also the runner-up
// Without scratch: the outputs, out_best (nullable, as out_centroid) not yet divided by |q| (launch_route_cosine does).
moin_status launch_pair_router_rows(HostState* hs, const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm,
                                    const int* cmap, int Q, int K, int D, int* out_expert, int* out_centroid, float* out_best,
                                    cudaStream_t stream);
// Tile mode: hb = hi/lo bf16 parts of s * x A_e^T ([2][T][r]); launch_pair_gemm adds hb B_e^T.
moin_status launch_tc_shrink_group(HostState* hs, const PlanView& pv, const moin_pool* const* pools,
                                   const __nv_bfloat16* const* xs, __nv_bfloat16* const* hbs, int n_jobs, float scale,
                                   cudaStream_t stream);
constexpr int kTcMaxShrinkJobs = 3;   // projections one grouped shrink launch can take

// Causal GQA attention on tcgen05 (attention_tc.cu).  q not rotated, k rotated.
bool attention_tc_supported(int n_heads, int n_kv_heads, int head_dim);
moin_status launch_attention_tc(HostState* hs, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                const int* cu, __nv_bfloat16* out, const float2* rope, int R,
                                int T, int max_seqlen, int n_heads, int n_kv_heads, float scale_log2,
                                cudaStream_t stream);

}  // namespace moin
