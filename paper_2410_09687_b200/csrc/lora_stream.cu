// Segmented LoRA shrink / expand for short segments (decode): every distinct adapter is
// streamed from HBM exactly once per call, straight from global memory into warp-MMA
// fragments.
//
// Both products are skinny (8 token columns per MMA), so they are HBM-bound on the adapter
// bytes; the tensor-core instruction used is the warp-level m16n8k16 one, which does the
// reduction over the long dimension without shuffles.  Operand fragments are loaded with one
// 16-byte load per thread and row: the MMA's k index is only a summation index, so the
// 8 consecutive elements a thread loads are assigned to the k slots it owns in two
// consecutive MMAs - as long as the other operand uses the same assignment the dot product
// is unchanged.  A warp-wide load then covers 8 rows x 64 contiguous bytes (full sectors).
#include "common.cuh"

namespace moin {

// Four warps split the reduction, 32-wide k steps dealt to them in turn.  Many items: 16 adapter rows an item and four steps a warp
// in flight, so that six CTAs share an SM.  Up to kShrinkFewT tokens the items leave the SMs empty and the time is a warp's chain
// of loads: half the rows an item (the other half of the MMA's rows idle) and twice the steps in flight, the sums of a row in the
// same order.  Decode steps, us, many / few: 6 tokens of rank 16 54.8 / 53.1, of rank 64 61.4 / 57.9, 16 of rank 64 80.6 / 74.2, 1 of
// rank 128 60.1 / 55.3; forward of 14 tokens on the 8-bit base 1440 / 1360, of 6 1379 / 1239.  (Eight warps: as fast, but another
// order of the sums; with more tokens they are slower: 256 tokens 230 -> 246.)
constexpr int kShrinkWarps = 4, kShrinkFewT = 16;
constexpr int kExpandThreads = 128;      // 4 warps
constexpr int kExpandFirst = 4;          // 16-row tiles prefetched while a warp waits for the shrink

// The unit both kernels work on is a CHUNK of the plan: at most 8 tokens (the columns of one MMA) of one expert.  A
// longer segment is several chunks that run side by side and find the adapter in L2; walking them one after the other
// in one CTA cost a round trip each (264 tokens over 8 experts, 256 -> 256: shrink 10.6 us, expand 17 us; a call of the layer 21.9 us, now 8.7).
// Work items of a launch span up to kMaxStreamJobs projections that share one batch plan: item index ->
// (job, chunk, sub-block), jobs laid out one after the other, `per_seg[j]` items per chunk in job j.
// Kernel parameters are only ever indexed with compile-time indices (a run-time index would force a
// local-memory copy of the parameter block): pick(arr, j) selects arr[j] with a compare chain.
template <class V>
__device__ __forceinline__ V pick(const V (&arr)[kMaxStreamJobs], int j) {
  V v = arr[0];
#pragma unroll
  for (int i = 1; i < kMaxStreamJobs; ++i)
    if (j == i) v = arr[i];
  return v;
}

__device__ __forceinline__ void l2_prefetch(const void* p, uint32_t bytes) {   // 16-byte aligned, a multiple of 16
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
struct ItemRef { int job, seg, sub; };
template <class Jobs>
__device__ __forceinline__ ItemRef decode_item(int item, int nchunk, const Jobs& jobs) {
  ItemRef it = {0, 0, 0};
  int rem = item;
#pragma unroll
  for (int j = 0; j + 1 < kMaxStreamJobs; ++j) {
    if (it.job == j && j + 1 < jobs.n && rem >= nchunk * jobs.per_seg[j]) {
      rem -= nchunk * jobs.per_seg[j];
      it.job = j + 1;
    }
  }
  const int ps = pick(jobs.per_seg, it.job);
  it.seg = rem / ps;
  it.sub = rem - it.seg * ps;
  return it;
}

struct SegMeta { int slot, s0, n, job, sub, r_use; };   // r_use: rank of the slot's adapter (<= the stored rank)
template <class Jobs>
__device__ __forceinline__ SegMeta load_seg(const int4* __restrict__ chunk_tab, const Jobs& jobs, int item, int items,
                                            int nchunk) {
  SegMeta m = {-1, 0, 0, 0, 0, 0};
  if (item < items) {
    const ItemRef it = decode_item(item, nchunk, jobs);
    const int4 e = __ldg(chunk_tab + it.seg);   // (expert, start, length, -)
    m.slot = __ldg(pick(jobs.slot_of_expert, it.job) + e.x);
    const int* rank_tab = pick(jobs.slot_rank, it.job);
    m.r_use = (m.slot >= 0 && rank_tab) ? min(__ldg(rank_tab + m.slot), pick(jobs.r, it.job)) : pick(jobs.r, it.job);
    m.s0 = e.y;
    m.n = e.z;
    m.job = it.job;
    m.sub = it.sub;
  }
  return m;
}

// h[pos][rho] = sum_i A[slot][rho][i] * x[perm[pos]][i]      (fp32, pos = position in sorted order)
// Work item = (job, chunk, group of ROWS adapter rows: 16, or 8); the CTA's warps interleave over k.
// Small CTAs (4 warps, 80 registers: six per SM, and room beside a base-GEMM CTA) and one CTA per item:
// the hardware's block scheduler hands the items out as slots free up, so a launch ends evenly whatever
// the base GEMM beside it occupies, and a CTA's metadata hops (segment count, table entry,
// slot) hide behind the streams of the other CTAs on its SM.
template <int ROWS, int UNROLL>
__global__ void __launch_bounds__(kShrinkWarps * 32, UNROLL == 4 ? 6 : 3)
lora_shrink_stream_kernel(const int* __restrict__ header, const int* __restrict__ perm,
                          const int4* __restrict__ chunk_tab, const ShrinkJobs jobs) {
  __shared__ float red[kShrinkWarps][32][4];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  pdl_launch_dependents();
  const int nchunk = header[PH_NCHUNK];
  int items = 0;
#pragma unroll
  for (int j = 0; j < kMaxStreamJobs; ++j)
    if (j < jobs.n) items += nchunk * jobs.per_seg[j];
  int item = blockIdx.x;
  SegMeta nxt = load_seg(chunk_tab, jobs, item, items, nchunk);
  for (; item < items; item += gridDim.x) {
    const SegMeta cur = nxt;
    nxt = load_seg(chunk_tab, jobs, item + gridDim.x, items, nchunk);  // lookahead
    if (cur.slot < 0 || cur.sub * ROWS >= cur.r_use) continue;  // uniform per CTA: no adapter, or rows beyond its rank
    const int r = pick(jobs.r, cur.job), d_in = pick(jobs.d_in, cur.job);
    const __nv_bfloat16* __restrict__ x = pick(jobs.x, cur.job);
    const __nv_bfloat16* __restrict__ A = pick(jobs.A, cur.job);
    float* __restrict__ h = pick(jobs.h, cur.job);
    const int steps = d_in >> 5;  // 32 k per step
    const int rho0 = cur.sub * ROWS + g, rho1 = rho0 + 8;
    const bool v0 = rho0 < cur.r_use, v1 = ROWS == 16 && rho1 < cur.r_use;   // rows beyond the slot's rank are not read
    const __nv_bfloat16* a_row0 = A + ((size_t)cur.slot * r + (v0 ? rho0 : 0)) * (size_t)d_in + 8 * t;
    const __nv_bfloat16* a_row1 = A + ((size_t)cur.slot * r + (v1 ? rho1 : 0)) * (size_t)d_in + 8 * t;
    {
      const bool vx = g < cur.n;
      float c[4] = {0.f, 0.f, 0.f, 0.f};
      const __nv_bfloat16* x_row = nullptr;
      for (int base = 0; base < steps; base += kShrinkWarps * UNROLL) {
        uint4 a0[UNROLL], a1[UNROLL], xv[UNROLL];
        const uint4 z = make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {  // adapter bytes first: they come from HBM
          const int i = base + u * kShrinkWarps + warp;
          const bool vi = i < steps;
          a0[u] = (vi && v0) ? ldg_stream(a_row0 + i * 32) : z;
          a1[u] = (vi && v1) ? ldg_stream(a_row1 + i * 32) : z;
        }
        if (x_row == nullptr) x_row = x + (size_t)(vx ? perm[cur.s0 + g] : 0) * (size_t)d_in + 8 * t;
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
          const int i = base + u * kShrinkWarps + warp;
          xv[u] = (i < steps && vx) ? ldg_cached(x_row + i * 32) : z;
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
          mma_bf16_16816(c, a0[u].x, a1[u].x, a0[u].y, a1[u].y, xv[u].x, xv[u].y);
          mma_bf16_16816(c, a0[u].z, a1[u].z, a0[u].w, a1[u].w, xv[u].z, xv[u].w);
        }
      }
      // fixed-order reduction over the warps (deterministic)
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 4; ++j) red[warp][lane][j] = c[j];
      __syncthreads();
      if (warp == 0) {
        float s[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float acc = red[0][lane][j];
#pragma unroll
          for (int w = 1; w < kShrinkWarps; ++w) acc += red[w][lane][j];
          s[j] = acc;
        }
        // c0:(rho0, col 2t) c1:(rho0, col 2t+1) c2:(rho1, col 2t) c3:(rho1, col 2t+1)
        const int col = 2 * t;
        if (col < cur.n) {
          float* hp = h + (size_t)(cur.s0 + col) * r;
          if (v0) hp[rho0] = s[0];
          if (v1) hp[rho1] = s[2];
        }
        if (col + 1 < cur.n) {
          float* hp = h + (size_t)(cur.s0 + col + 1) * r;
          if (v0) hp[rho0] = s[1];
          if (v1) hp[rho1] = s[3];
        }
      }
    }
  }
  // One CTA ends only after the base GEMM launched before this kernel: whoever waits for this grid (the expand, in
  // stream order) has waited for the GEMM too, although the two run side by side.
  if (blockIdx.x == gridDim.x - 1) pdl_wait();
}

// y[perm[pos]][j] = bf16( y0[perm[pos]][j] + scale * sum_rho B[slot][j][rho] * h[pos][rho] )
// h is split into bf16 hi + lo parts (two MMAs) so the low-rank term keeps ~fp32 accuracy.
//
// The unit of work is one 16-row tile of B for one (chunk, job); units are ordered (chunk, job, tile)
// and every warp of the grid takes one contiguous, equally long range of them (tiles need no reduction
// across each other, so a range may start and end anywhere).  All warps therefore stream the same number
// of adapter bytes, whatever the mix of projection widths in the launch, and a warp's range is contiguous
// in memory inside a (chunk, job).  A warp walks its range some tiles at a time with the adapter rows and the base
// values y0 of a batch loaded together.  `jobs.per_seg[j]` = tiles of job j.

// Tiles tile0 .. tile1 - 1 of one (chunk, job), TB of them in flight; P: 32-wide groups of the rank, ceil(r_use / 32).
struct ExpandPiece {
  const __nv_bfloat16* Bs;   // the adapter's B
  const float *h, *y0;
  __nv_bfloat16* y;
  int r, r_use, d_out, act, s0, n, my_row;   // my_row: token row of column g (-1: none)
};
template <int P, int TB, bool VAR>
__device__ __forceinline__ void expand_piece(const ExpandPiece& e, int tile0, int tile1, float scale, int g, int t) {
  // token operand (MMA "B" fragment): column g = token g, k slots <- rho 32p + 8t .. +7
  uint32_t hh[P][4], hl[P][4];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int rb = 32 * p + 8 * t;
    float v[8];
    if (g < e.n && rb < e.r_use) {
      const float4 f0 = *reinterpret_cast<const float4*>(e.h + (size_t)(e.s0 + g) * e.r + rb);
      const float4 f1 = *reinterpret_cast<const float4*>(e.h + (size_t)(e.s0 + g) * e.r + rb + 4);
      v[0] = f0.x; v[1] = f0.y; v[2] = f0.z; v[3] = f0.w; v[4] = f1.x; v[5] = f1.y; v[6] = f1.z; v[7] = f1.w;
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = 0.f;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float s0v = (VAR ? lora_act(v[2 * q], e.act) : v[2 * q]) * scale;
      const float s1v = (VAR ? lora_act(v[2 * q + 1], e.act) : v[2 * q + 1]) * scale;
      const uint32_t hi = pack_bf16(s0v, s1v);
      hh[p][q] = hi;
      hl[p][q] = pack_bf16(s0v - bf16_lo(hi), s1v - bf16_hi(hi));
    }
  }
  const int row_c0 = __shfl_sync(0xffffffffu, e.my_row, (2 * t) * 4);
  const int row_c1 = __shfl_sync(0xffffffffu, e.my_row, (2 * t + 1) * 4);
  const int r = e.r, d_out = e.d_out;
  for (int tb = tile0; tb < tile1; tb += TB) {
    uint4 a0[TB][P], a1[TB][P];
    float b0[TB][4];
#pragma unroll
    for (int i = 0; i < TB; ++i) {
      const int ja = (tb + i) * 16 + g, jc = ja + 8;
      const bool va = (tb + i) < tile1 && ja < d_out, vc = (tb + i) < tile1 && jc < d_out;
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const int rb = 32 * p + 8 * t;
        const uint4 z = make_uint4(0, 0, 0, 0);
        a0[i][p] = (va && rb < e.r_use) ? ldg_stream(e.Bs + (size_t)ja * r + rb) : z;
        a1[i][p] = (vc && rb < e.r_use) ? ldg_stream(e.Bs + (size_t)jc * r + rb) : z;
      }
      b0[i][0] = (va && row_c0 >= 0) ? __ldg(e.y0 + (size_t)row_c0 * d_out + ja) : 0.f;
      b0[i][1] = (va && row_c1 >= 0) ? __ldg(e.y0 + (size_t)row_c1 * d_out + ja) : 0.f;
      b0[i][2] = (vc && row_c0 >= 0) ? __ldg(e.y0 + (size_t)row_c0 * d_out + jc) : 0.f;
      b0[i][3] = (vc && row_c1 >= 0) ? __ldg(e.y0 + (size_t)row_c1 * d_out + jc) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < TB; ++i) {
      const int ja = (tb + i) * 16 + g, jc = ja + 8;
      const bool va = (tb + i) < tile1 && ja < d_out, vc = (tb + i) < tile1 && jc < d_out;
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int p = 0; p < P; ++p) {
        mma_bf16_16816(c, a0[i][p].x, a1[i][p].x, a0[i][p].y, a1[i][p].y, hl[p][0], hl[p][1]);
        mma_bf16_16816(c, a0[i][p].z, a1[i][p].z, a0[i][p].w, a1[i][p].w, hl[p][2], hl[p][3]);
        mma_bf16_16816(c, a0[i][p].x, a1[i][p].x, a0[i][p].y, a1[i][p].y, hh[p][0], hh[p][1]);
        mma_bf16_16816(c, a0[i][p].z, a1[i][p].z, a0[i][p].w, a1[i][p].w, hh[p][2], hh[p][3]);
      }
      // c0:(ja, col 2t) c1:(ja, col 2t+1) c2:(jc, col 2t) c3:(jc, col 2t+1)
      if (row_c0 >= 0) {
        const size_t o = (size_t)row_c0 * d_out;
        if (va) e.y[o + ja] = __float2bfloat16_rn(b0[i][0] + c[0]);
        if (vc) e.y[o + jc] = __float2bfloat16_rn(b0[i][2] + c[2]);
      }
      if (row_c1 >= 0) {
        const size_t o = (size_t)row_c1 * d_out;
        if (va) e.y[o + ja] = __float2bfloat16_rn(b0[i][1] + c[1]);
        if (vc) e.y[o + jc] = __float2bfloat16_rn(b0[i][3] + c[3]);
      }
    }
  }
}

// VAR: some pool of the launch has a rank per slot or an activation; without it the kernel is the plain layer's
// (the rank is the stored rank, h is used as it is) and carries none of the variant's bookkeeping.  A variant launch
// takes each piece by its own rank, so that narrow adapters keep as many bytes in flight as wide ones.
// P: number of 32-wide rho groups, ceil(max r / 32).
template <int P, bool VAR>
__global__ void __launch_bounds__(kExpandThreads, 4)
lora_expand_stream_kernel(const int* __restrict__ header, const int* __restrict__ perm,
                          const int4* __restrict__ chunk_tab, const ExpandJobs jobs, float scale, int tps) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const long long wid = (long long)blockIdx.x * (kExpandThreads / 32) + warp;
  const long long nw = (long long)gridDim.x * (kExpandThreads / 32);
  pdl_launch_dependents();
  // The plan and the adapters are older than the shrink before this kernel; h (shrink) and y0 (base GEMM, which the
  // shrink's completion covers) are not: the wait comes after the first piece's metadata and the start of its adapter
  // rows (decode step of 24 tokens 83.7 -> 78.1 us, of 256 tokens 236.5 -> 230.5 us; prefetching further ahead or all
  // along the range only disturbs the streams: 237-260 us).
  bool waited = false;
  const int nchunk = __ldg(header + PH_NCHUNK);
  const long long units = (long long)nchunk * tps;
  long long u = units * wid / nw;
  const long long u_end = units * (wid + 1) / nw;
  while (u < u_end) {
    // ---- chunk: expert, rows, adapter slots of all jobs (one hop after the table entry)
    const int seg = (int)(u / tps);
    const int4 e = __ldg(chunk_tab + seg);   // (expert, start, length, -)
    const int s0 = e.y, n = e.z;
    int slots[kMaxStreamJobs];
#pragma unroll
    for (int j = 0; j < kMaxStreamJobs; ++j) slots[j] = (j < jobs.n) ? __ldg(jobs.slot_of_expert[j] + e.x) : -1;
    int ranks[kMaxStreamJobs];   // rank of the slot's adapter: columns of B and entries of h beyond it are not read
#pragma unroll
    for (int j = 0; j < kMaxStreamJobs; ++j)
      ranks[j] = (VAR && j < jobs.n && slots[j] >= 0 && jobs.slot_rank[j]) ? min(__ldg(jobs.slot_rank[j] + slots[j]), jobs.r[j])
                                                                     : (j < jobs.n ? jobs.r[j] : 0);
    const int my_row = g < n ? __ldg(perm + s0 + g) : -1;
    const long long seg_end = (long long)(seg + 1) * tps;
    int rem = (int)(u - (long long)seg * tps);
    int job = 0;
#pragma unroll
    for (int j = 0; j + 1 < kMaxStreamJobs; ++j) {
      if (job == j && j + 1 < jobs.n && rem >= jobs.per_seg[j]) {
        rem -= jobs.per_seg[j];
        job = j + 1;
      }
    }
    // ---- (chunk, job) pieces of the range
    while (u < u_end && u < seg_end) {
      const int tiles_j = pick(jobs.per_seg, job);
      const int tile0 = rem;
      const long long left = u_end - u;
      const int tile1 = (left < (long long)(tiles_j - tile0)) ? tile0 + (int)left : tiles_j;
      const int slot = pick(slots, job);
      if (slot >= 0) {
        ExpandPiece pc;
        pc.r = pick(jobs.r, job);
        pc.d_out = pick(jobs.d_out, job);
        pc.r_use = VAR ? pick(ranks, job) : pc.r;
        pc.act = VAR ? pick(jobs.act, job) : MOIN_ACT_NONE;
        pc.h = pick(jobs.h, job);
        pc.y0 = pick(jobs.y0, job);
        pc.y = pick(jobs.y, job);
        pc.Bs = pick(jobs.B, job) + (size_t)slot * (size_t)pc.d_out * (size_t)pc.r;
        pc.s0 = s0; pc.n = n; pc.my_row = my_row;
        if (!waited) {
          if (!VAR && lane == 0) {   // the first rows on their way to L2 meanwhile
            const int rows = min(pc.d_out, min(tile1, tile0 + kExpandFirst) * 16) - tile0 * 16;
            l2_prefetch(pc.Bs + (size_t)tile0 * 16 * pc.r, (uint32_t)(rows * pc.r * 2));
          }
          pdl_wait();
          waited = true;
        }
        if (VAR) {
          if (P >= 4 && pc.r_use > 64) expand_piece<4, 1, VAR>(pc, tile0, tile1, scale, g, t);
          else if (P >= 2 && pc.r_use > 32) expand_piece<2, 2, VAR>(pc, tile0, tile1, scale, g, t);
          else expand_piece<1, 2, VAR>(pc, tile0, tile1, scale, g, t);
        } else {
          expand_piece<P, (P > 2 ? 1 : 2), VAR>(pc, tile0, tile1, scale, g, t);
        }
      }
      u += tile1 - tile0;
      rem = 0;
      ++job;
    }
  }
  if (!waited) pdl_wait();   // (a kernel that waits for this one counts on everything before being complete)
}

static int stream_grid(long max_items, int n_sms, int ctas_per_sm) {
  long g = max_items < (long)n_sms * ctas_per_sm ? max_items : (long)n_sms * ctas_per_sm;
  return g < 1 ? 1 : (int)g;
}

cudaError_t launch_lora_shrink_stream(const PlanView& pv, ShrinkJobs jobs, int n_sms, cudaStream_t stream) {
  const bool few = pv.T <= kShrinkFewT;
  const int rows = few ? 8 : 16;
  long items = 0;
  for (int j = 0; j < jobs.n; ++j) {
    jobs.per_seg[j] = (jobs.r[j] + rows - 1) / rows;
    items += (long)pv.Cmax * jobs.per_seg[j];
  }
  // one CTA per item (capped; CTAs stride over the items beyond the cap)
  auto go = [&](auto* fn) {
    return launch_pdl(fn, stream_grid(items, n_sms, 1024), 32 * kShrinkWarps, 0, stream, pv.header, pv.perm, pv.chunk_tab, jobs);
  };
  return few ? go(lora_shrink_stream_kernel<8, 8>) : go(lora_shrink_stream_kernel<16, 4>);
}

cudaError_t launch_lora_expand_stream(const PlanView& pv, ExpandJobs jobs, float scale, int n_sms,
                                      cudaStream_t stream) {
  int tps = 0, rmax = 0;
  for (int j = 0; j < jobs.n; ++j) {
    jobs.per_seg[j] = (jobs.d_out[j] + 15) / 16;   // 16-row tiles per chunk
    tps += jobs.per_seg[j];
    rmax = jobs.r[j] > rmax ? jobs.r[j] : rmax;
  }
  // one warp per 2 tiles at least; at most one CTA per resident slot (4 per SM)
  const long max_ctas = ((long)pv.Cmax * tps + 2 * (kExpandThreads / 32) - 1) / (2 * (kExpandThreads / 32));
  const int grid = stream_grid(max_ctas, n_sms, 4);
  bool var = false;
  for (int j = 0; j < jobs.n; ++j) var = var || jobs.slot_rank[j] != nullptr || jobs.act[j] != MOIN_ACT_NONE;
  auto go = [&](auto* fn) {
    return launch_pdl(fn, grid, kExpandThreads, 0, stream, pv.header, pv.perm, pv.chunk_tab, jobs, scale, tps);
  };
  if (rmax <= 32) return var ? go(lora_expand_stream_kernel<1, true>) : go(lora_expand_stream_kernel<1, false>);
  if (rmax <= 64) return var ? go(lora_expand_stream_kernel<2, true>) : go(lora_expand_stream_kernel<2, false>);
  return var ? go(lora_expand_stream_kernel<4, true>) : go(lora_expand_stream_kernel<4, false>);
}

}  // namespace moin
