// Base GEMM y = x W^T for few tokens (decode) on tcgen05 / TMEM / TMA, several projections in one launch.
//
// With few rows the GEMM is a stream over the weights, so the operands are swapped against the long-run kernel: 128
// OUTPUT FEATURES are the M side of a tile (A = rows of W) and the tokens, up to 256, the N side (B = rows of x), so
// every byte of W is read once per call whatever the number of tokens, and 24 tokens cost a tile of 32 and not of
// 128.  The reduction of a narrow projection (2048 -> 256 is two tiles) is cut over `ks` CTAs of a cluster.  The
// partial sums meet through distributed shared memory - every CTA owns 1/ks of the tokens and adds the parts in rank
// order, so the result does not depend on timing; a job's ks depends on its own shape, the tokens and the token tile of the
// launch, so with the same tile a projection gives the same bits alone and in a group.
//   warp 0     TMA producer (one thread): [128 x 64] box of W and [nt x 64] box of x per stage
//   warp 1     allocates TMEM, issues the MMAs (one elected lane)
//   warps 2-5  read the accumulator (TMEM lane = feature, column = token); all warps store
// What bounds it: at small T the HBM stream of W plus ~4 us of set-up and first round trip; at T = 256 the 32 KB of x
// that every 16 KB block of W brings along (an SM takes about 64 bytes per clock from L2).
//
// 8-bit weights (FP8): warps 2-5, idle until the epilogue otherwise, turn each stage's codes into the bf16 weights that
// the stand-alone conversion makes - a thread has one row of the tile, so one scale - and put them into tensor memory as
// the A operand (32 columns a stage).  HBM reads one byte a weight and nothing is written; a tile takes at most 128
// tokens, so that tensor memory holds the accumulator and four stages or more with two CTAs on an SM, and more tokens
// convert a tile again from L2.  Bound by the conversion, 128 threads at about six instructions for two codes.  Forward on
// the 8-bit base with a converted copy per group / this: 112 tokens 2499 / 1871 us, 303 3746 / 2665, 495 4525 / 3525.
#include <cuda.h>

#include "ptx.cuh"
#include "tc_gemm.cuh"

namespace moin {

constexpr int kDgThreads = 192, kDgM = 128, kDgK = 64, kDgMaxN = 256, kDgMaxStages = 8, kDgMaxSplit = 8;
constexpr int kDgFp8MaxN = 128, kDgFp8Cols = 256, kDgFp8Smem = 104 * 1024;

struct DgMaps { CUtensorMap w[kMaxStreamJobs], x[kMaxStreamJobs]; };
struct DgParams {
  int n_jobs, T, nt, n_chunks, stages, tmem_cols, cluster;   // nt tokens per tile, n_chunks tiles over the tokens
  int cta_end[kMaxStreamJobs];   // CTAs of jobs 0 .. j (each job's padded to whole clusters)
  int ks[kMaxStreamJobs], tiles[kMaxStreamJobs], K[kMaxStreamJobs], d_out[kMaxStreamJobs];
  __nv_bfloat16* y[kMaxStreamJobs];
  float* y0[kMaxStreamJobs];     // fp32 copy, nullable
  const float* w_scale[kMaxStreamJobs];   // FP8: scale per row of W
  DeviceStatus* status;
};

template <bool FP8, bool EARLY>
__global__ void __launch_bounds__(kDgThreads)
decode_gemm_kernel(const __grid_constant__ DgMaps maps, const DgParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t ring = (raw + 1023u) & ~1023u;
  const int S = p.stages;
  constexpr uint32_t kWBytes = kDgM * kDgK * (FP8 ? 1 : 2);
  const uint32_t stage_bytes = kWBytes + (uint32_t)p.nt * kDgK * 2;
  const uint32_t bars = ring + (uint32_t)S * stage_bytes;
  uint8_t* bar_ptr = smem_raw + (bars - raw);
  const uint32_t full0 = bars, empty0 = bars + 8 * kDgMaxStages, done = bars + 16 * kDgMaxStages;
  const uint32_t conv0 = bars + 16 * kDgMaxStages + 32;   // FP8: the stage's weights are in tensor memory
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_ptr + 16 * kDgMaxStages + 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_ptr + 16 * kDgMaxStages + 16);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  int job = 0;
#pragma unroll
  for (int j = 0; j + 1 < kMaxStreamJobs; ++j)
    if (j + 1 < p.n_jobs && (int)blockIdx.x >= p.cta_end[j]) job = j + 1;
  int K = p.K[0], d_out = p.d_out[0], ks = p.ks[0], n_tiles = p.tiles[0], first = 0;
  __nv_bfloat16* y = p.y[0];
  float* y0 = p.y0[0];
  const float* w_scale = p.w_scale[0];
#pragma unroll
  for (int j = 1; j < kMaxStreamJobs; ++j)
    if (job == j) {
      K = p.K[j]; d_out = p.d_out[j]; ks = p.ks[j]; n_tiles = p.tiles[j]; y = p.y[j]; y0 = p.y0[j];
      w_scale = p.w_scale[j];
      first = p.cta_end[j - 1];
    }
  // ks consecutive CTAs of a cluster share an item = (feature tile, token chunk)
  const int idx = (int)blockIdx.x - first, item = idx / ks, rank = idx - item * ks;
  const int group0 = (int)(blockIdx.x % (unsigned)p.cluster) - rank;   // cluster rank of the item's first CTA
  const int tile = item / p.n_chunks;
  const bool on = tile < n_tiles;                                      // (the last cluster of a job may be padded)
  const int tok0 = (item - tile * p.n_chunks) * p.nt, f0 = tile * kDgM;
  const int nkb = on ? K / kDgK : 0, kb0 = nkb * rank / ks, kb1 = nkb * (rank + 1) / ks;
  const int n_early = EARLY ? min(S, kb1 - kb0) : 0;   // k-blocks whose weights do not wait for the kernel before

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
      if (FP8) mbar_init(conv0 + 8 * s, 4);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // Weights that the kernel before this one leaves alone (see w_early): the first stages' are on their way while that one
    // ends.  Forwards of 16 / 112 / 260 / 1000 tokens, rank 16: bf16 base 1334 -> 1289, 1763 -> 1745, 2495 -> 2479, 5722 -> 5694
    // us; 8-bit base 1326 -> 1303, 1834 -> 1790, 2550 -> 2525, 5956 -> 5926.
    for (int s = 0; s < n_early; ++s) {
      mbar_expect_tx(full0 + 8 * s, stage_bytes);
      tma_load_2d(ring + s * stage_bytes, &maps.w[job], full0 + 8 * s, (kb0 + s) * kDgK, f0);
    }
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();                // x and whatever else ran before (the set-up above overlaps the tail of it)
  pdl_launch_dependents();   // the adapter shrink does not read this kernel's results: it may take the free SM slots

  bool ok = true;
  const uint32_t a_col = ((uint32_t)p.nt + 31u) & ~31u;   // FP8: first tensor-memory column of the converted weights
  if (warp == 0) {
    if (lane == 0) {
      const CUtensorMap* mw = &maps.w[job];
      const CUtensorMap* mx = &maps.x[job];
      uint32_t s = 0, ph = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait(empty0 + 8 * s, ph ^ 1u, abort_flag, p.status, 51)) break;
        const uint32_t sa = ring + s * stage_bytes, full = full0 + 8 * s;
        if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
        if (!EARLY || kb - kb0 >= n_early) {
          mbar_expect_tx(full, stage_bytes);
          tma_load_2d(sa, mw, full, kb * kDgK, f0);
        }
        tma_load_2d(sa + kWBytes, mx, full, kb * kDgK, tok0);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    const uint32_t idesc = idesc_bf16(kDgM, p.nt);
    const bool leader = elect_one();
    uint32_t s = 0, ph = 0;
    for (int kb = kb0; kb < kb1 && ok; ++kb) {
      if (!(ok = mbar_wait_warp(full0 + 8 * s, ph, abort_flag, p.status, 52))) break;
      if (FP8 && !(ok = mbar_wait_warp(conv0 + 8 * s, ph, abort_flag, p.status, 54))) break;
      tc_fence_after();
      const uint32_t sa = ring + s * stage_bytes, empty = empty0 + 8 * s, ta = tmem + a_col + s * (kDgK / 2);
      if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
      const uint64_t da = sdesc_k128(sa), db = sdesc_k128(sa + kWBytes);
      if (leader) {
#pragma unroll
        for (int k = 0; k < kDgK / 16; ++k) {
          const uint32_t acc = (kb > kb0 || k > 0) ? 1u : 0u;
          if (FP8) tc_mma_bf16_ta(tmem, ta + 8 * k, db + (uint64_t)(2 * k), idesc, acc);
          else tc_mma_bf16(tmem, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, acc);
        }
        tc_commit(empty);
      }
    }
    if (ok && leader) tc_commit(done);
    __syncwarp();
  } else {
    if (FP8) {   // a thread converts one row (TMEM lane) of the stage's codes; its scale stays in a register
      const int row = (warp & 3) * 32 + lane;
      const float sc = on && f0 + row < d_out ? __ldg(w_scale + f0 + row) : 0.f;
      const uint32_t swz = (uint32_t)(row >> 1) & 3u;   // 64-byte swizzle: 16-byte piece c of a row lies at c ^ swz
      uint32_t s = 0, ph = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!(ok = mbar_wait_warp(full0 + 8 * s, ph, abort_flag, p.status, 55))) break;
        tc_fence_after();
        const uint32_t sa = ring + s * stage_bytes + (uint32_t)row * kDgK;
        const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) + a_col + s * (kDgK / 2);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t v[16];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const uint4 w = lds_u4(sa + (((uint32_t)(2 * h + c) ^ swz) << 4));
            fp8x4_to_bf16(w.x, sc, v[8 * c], v[8 * c + 1]);
            fp8x4_to_bf16(w.y, sc, v[8 * c + 2], v[8 * c + 3]);
            fp8x4_to_bf16(w.z, sc, v[8 * c + 4], v[8 * c + 5]);
            fp8x4_to_bf16(w.w, sc, v[8 * c + 6], v[8 * c + 7]);
          }
          tmem_st16(ta + 16 * h, v);
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(conv0 + 8 * s);
        if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
      }
    }
    ok = ok && mbar_wait_warp(done, 0, abort_flag, p.status, 53);
    tc_fence_after();
  }
  // ---------------------------------------------------------------- epilogue
  // The tile goes to shared memory as [token][128 features] fp32 (the ring is free: every stage has been consumed) and
  // leaves from there a token row at a time, so that a warp's store is one whole 256-byte (bf16) or 512-byte (fp32)
  // line.  With a split reduction every CTA of the item sums its 1/ks of the tokens over the parts, read from the
  // other CTAs' shared memory in rank order.  (Scalar stores straight from TMEM lanes, or pushed one float at a time
  // into the other CTAs, took 12 us of a 20 us launch at 256 tokens.)
  if (warp >= 2 && ok && on) {
    const int q = warp & 3, f = q * 32 + lane;             // TMEM lane quarter of this warp, feature of this thread
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    for (int c = 0; c < p.nt; c += 16) {
      uint32_t v[16];
      tmem_ld16(lane_addr + c, v);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; ++i)
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(ring + (uint32_t)((c + i) * kDgM + f) * 4u), "r"(v[i]) : "memory");
    }
  }
  if (p.cluster > 1) {
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }
  if (on && f0 + 4 * lane < d_out) {                       // (d_out is a multiple of 8)
    const int own = p.nt / ks, c0 = rank * own;            // tokens this CTA adds up and stores
    uint32_t base[kDgMaxSplit];
#pragma unroll
    for (int r = 0; r < kDgMaxSplit; ++r) base[r] = (ks > 1 && r < ks) ? map_rank(ring, (uint32_t)(group0 + r)) : ring;
    for (int cc = c0 + warp; cc < c0 + own; cc += kDgThreads / 32) {
      const int tok = tok0 + cc;
      if (tok >= p.T) break;
      const uint32_t off = (uint32_t)(cc * kDgM + 4 * lane) * 4u;
      float4 v[kDgMaxSplit];
#pragma unroll
      for (int r = 0; r < kDgMaxSplit; ++r)
        if (r < ks) v[r] = ks > 1 ? ld_cluster_f4(base[r] + off) : lds_f4(base[r] + off);
      float4 acc = v[0];
#pragma unroll
      for (int r = 1; r < kDgMaxSplit; ++r)
        if (r < ks) { acc.x += v[r].x; acc.y += v[r].y; acc.z += v[r].z; acc.w += v[r].w; }
      const size_t o = (size_t)tok * d_out + f0 + 4 * lane;
      *reinterpret_cast<uint2*>(y + o) = make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
      if (y0) *reinterpret_cast<float4*>(y0 + o) = acc;
    }
  }
  if (p.cluster > 1) {   // no CTA leaves while another may still read its part
    cluster_arrive();
    cluster_wait();
  }
  if (*abort_flag) {   // a wait ran out: let copies / MMAs in flight land before shared and tensor memory are released
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < 2000000ull) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, p.tmem_cols);
  }
}

moin_status launch_decode_gemm(HostState* hs, const DecodeGemmJob* jobs, int n_jobs, int T, bool small_tiles, bool w_early, cudaStream_t stream) {
  DgMaps maps;
  DgParams p = {};
  p.n_jobs = n_jobs; p.T = T; p.status = hs->status;
  // Split a projection's reduction until its own CTAs fill their share of the SM slots or a CTA is down to four 64-wide
  // blocks (its own, whatever else is in the group).  Beside many tokens' adapters the share is half of the
  // SMs (decode step of 256 tokens with half / all / a quarter: 237 / 264 / 248 us); up to 64 tokens two CTAs fit an SM
  // and there is little to stream beside them (step of 24 tokens with half / all: 88 / 87 us).  8-bit codes: once all
  // SMs, whatever the tokens (forwards of 112 / 303 / 495 tokens with half 1933 / 3263 / 4020 us, all 1871 / 2665 /
  // 3525, twice 1992 / 2795 / 3516).
  const bool fp8 = jobs[0].w_scale != nullptr;
  // Narrow adapters leave the memory to the GEMM, and its tiles of 64 tokens, two CTAs an SM, the epilogues short: forwards of 300
  // to 512 tokens in segments of 1 to 24, tiles of 64 over tiles of up to 256: rank 8 0.85 to 0.93, 16 0.87 to 0.97, 32 0.89 to
  // 1.01, 40 0.92 to 1.10, 64 0.97 to 1.23.  Segments of 12, up to 256 / of 64, ms: rank 16 1020 tokens 5.96 / 5.50, 1404 7.05 / 6.89,
  // 2004 8.84 / 9.90; rank 32 6.29 / 6.18, 7.70 / 7.94, 9.92 / 11.4; rank 64 7.83 / 8.08, 9.98 / 11.3, 13.2 / 14.8.
  const int max_n = small_tiles ? 64 : fp8 ? kDgFp8MaxN : kDgMaxN;
  const int chunks0 = (T + max_n - 1) / max_n;
  const bool small = (T + chunks0 - 1) / chunks0 <= 64;
  const int limit = fp8 || (small_tiles && T > 512) ? hs->n_sms : small ? 2 * hs->n_sms : hs->n_sms / 2;
  int items = 0;   // CTAs with one token tile per 256 tokens
  p.cluster = 1;
  for (int j = 0; j < n_jobs; ++j) {
    p.tiles[j] = (jobs[j].d_out + kDgM - 1) / kDgM;
    p.ks[j] = 1;
    while (p.ks[j] < kDgMaxSplit && p.tiles[j] * chunks0 * p.ks[j] * 2 <= limit && jobs[j].d_in / kDgK >= 4 * p.ks[j] * 2) p.ks[j] *= 2;
    if (p.ks[j] > p.cluster) p.cluster = p.ks[j];
    items += p.tiles[j] * chunks0 * p.ks[j];
  }
  // A small launch cuts the tokens finer as well: its time is the epilogue of one tile (264 x 256 -> 256: 9.6 us with
  // four CTAs of 144 tokens, 4.8 us with the single-CTA GEMM of 128 x 64 tiles, 4.3 us with CTAs of 32 tokens).
  p.n_chunks = chunks0;
  p.nt = ((T + p.n_chunks - 1) / p.n_chunks + 15) / 16 * 16;
  while (p.nt > 32 && items * 2 <= hs->n_sms / 2) {
    items *= 2;
    p.n_chunks *= 2;
    p.nt = ((T + p.n_chunks - 1) / p.n_chunks + 15) / 16 * 16;
  }
  for (int j = 0; j < n_jobs; ++j) {
    moin_status st = fp8 ? make_map_u8(&maps.w[j], jobs[j].W, jobs[j].d_out, jobs[j].d_in, kDgM)
                         : make_map(&maps.w[j], jobs[j].W, jobs[j].d_out, jobs[j].d_in, kDgM);
    if (!st) st = make_map(&maps.x[j], jobs[j].x, T, jobs[j].d_in, p.nt);
    if (st) return st;
    p.K[j] = jobs[j].d_in; p.d_out[j] = jobs[j].d_out;
    p.y[j] = jobs[j].y; p.y0[j] = jobs[j].y0;
    p.w_scale[j] = jobs[j].w_scale;
  }
  int ctas = 0;
  for (int j = 0; j < n_jobs; ++j) {
    ctas += (int)align_up((size_t)p.tiles[j] * p.n_chunks * p.ks[j], p.cluster);
    p.cta_end[j] = ctas;
  }
  // Shared memory: the stream kernels beside this one feed on L1, which gets what shared memory leaves (228 KB in all):
  // 150 KB an SM against 192: decode step of 256 tokens 237 / 254 us.
  const int stage = kDgM * kDgK * (fp8 ? 1 : 2) + p.nt * kDgK * 2;
  const int budget = fp8 ? kDgFp8Smem : 150 * 1024 / (p.nt <= 64 ? 2 : 1);
  p.stages = budget / stage < kDgMaxStages ? budget / stage : kDgMaxStages;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.nt) p.tmem_cols *= 2;
  if (fp8) {
    const int slots = (kDgFp8Cols - (p.nt + 31) / 32 * 32) / (kDgK / 2);   // tensor-memory buffers of converted weights
    if (p.stages > slots) p.stages = slots;
    p.tmem_cols = kDgFp8Cols;
  }
  // the ring is also the fp32 staging of the epilogue
  const size_t out = (size_t)p.nt * kDgM * sizeof(float);
  while ((size_t)p.stages * stage < out) ++p.stages;
  size_t smem = (size_t)p.stages * stage + 1024 /*align*/ + 256 /*barriers*/;
  // (codes come from forwards only, whose neighbours are known.  A kernel of its own for layer calls: with the early loads under a
  // run-time flag they took 0.2 to 0.4 us a launch longer.)
  auto* kernel = fp8 ? decode_gemm_kernel<true, true> : w_early ? decode_gemm_kernel<false, true> : decode_gemm_kernel<false, false>;
  // Half of the tensor memory for less than half of the shared memory would let a third CTA in, which then waits in the
  // allocation for CTAs that may wait for its own cluster: two at most.
  if (fp8 && smem < kDgFp8Smem) smem = kDgFp8Smem;
  cudaError_t e = ensure_smem_optin(fp8 ? OPTIN_DECODE_GEMM_FP8 : w_early ? OPTIN_DECODE_GEMM_EARLY : OPTIN_DECODE_GEMM, kernel, 160 * 1024);
  if (e != cudaSuccess) return record_cuda(e);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3(kDgThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)p.cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return record_cuda(cudaLaunchKernelEx(&cfg, kernel, maps, p));
}

}  // namespace moin
