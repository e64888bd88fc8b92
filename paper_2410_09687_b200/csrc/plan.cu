// Batch plan: grouping of tokens by expert id (integer work only).
//
// Batches of up to 1024 tokens take one single-CTA launch (plan_small_kernel: a bitonic sort of
// (expert id, token) keys in shared memory).  Larger ones take a few small launches:
//   plan_rank_kernel    per 256-token chunk: sanitise ids, stable in-chunk rank, per-chunk histogram
//   plan_prefix_kernel  (batches of more than one chunk) per expert id: prefix of its counts over the chunks
//   plan_scan_kernel    one CTA: prefix over expert ids -> segment list; run tiles
//   plan_scatter_kernel per chunk: position = expert base + chunk prefix + in-chunk rank -> perm
// The result is a stable counting sort (token order is kept inside every expert segment), so
// the plan is deterministic.
#include "common.cuh"

namespace moin {

__global__ void __launch_bounds__(kPlanChunk) plan_rank_kernel(const int* __restrict__ token_expert, int T, int E,
                                                               int* __restrict__ key, int* __restrict__ rank,
                                                               int* __restrict__ hist, DeviceStatus* status) {
  __shared__ __align__(16) int skey[kPlanChunk];
  const int tid = threadIdx.x;
  pdl_begin();
  int* row = hist + (size_t)blockIdx.x * (size_t)(E + 1);   // this chunk's counts: cleared here, no separate launch
  for (int i = tid; i <= E; i += kPlanChunk) row[i] = 0;
  const int t = blockIdx.x * kPlanChunk + tid;
  int k = -2;  // padding lanes never match
  if (t < T) {
    int e = token_expert[t];
    if (e >= 0 && e < E) {
      k = e;
    } else {
      k = E;  // "no adapter" bucket
      if (e != -1) atomicAdd(&status->invalid_expert_ids, 1);
    }
  }
  skey[tid] = k;
  __syncthreads();
  const unsigned in_batch = __ballot_sync(0xffffffffu, t < T);
  if (t >= T) return;
  // equal keys before and after this one: four keys a read in the other warps, a match inside the own (key by key over
  // the whole chunk: 40000 tokens 6.2 us, so 4.0)
  const int w0 = tid & ~31, lane = tid & 31;
  const unsigned same = __match_any_sync(in_batch, k);
  int before = __popc(same & ((1u << lane) - 1u)), after = __popc(same >> lane) - 1;
  auto count = [&](int i) {
    const int4 q = *reinterpret_cast<const int4*>(skey + i);
    return (q.x == k) + (q.y == k) + (q.z == k) + (q.w == k);
  };
#pragma unroll 8
  for (int i = 0; i < w0; i += 4) before += count(i);
#pragma unroll 8
  for (int i = w0 + 32; i < kPlanChunk; i += 4) after += count(i);
  key[t] = k;
  rank[t] = before;
  if (after == 0) row[k] = before + 1;
}

// Block-wide scans for NT threads (a multiple of 32, at most 1024).  `smem` must hold 33 ints.
template <int NT>
__device__ __forceinline__ int block_excl_sum(int v, int* smem, int* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += n;
  }
  __syncthreads();  // protect smem reuse between calls
  if (lane == 31) smem[w] = inc;
  __syncthreads();
  if (w == 0) {
    int s = (lane < NT / 32) ? smem[lane] : 0;
    int si = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int n = __shfl_up_sync(0xffffffffu, si, o);
      if (lane >= o) si += n;
    }
    smem[lane] = si - s;  // exclusive prefix of warp totals
    if (lane == 31) smem[32] = si;
  }
  __syncthreads();
  *total = smem[32];
  return smem[w] + inc - v;
}
template <int NT>
__device__ __forceinline__ int block_incl_max(int v, int* smem) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc = max(inc, n);
  }
  __syncthreads();
  if (lane == 31) smem[w] = inc;
  __syncthreads();
  if (w == 0) {
    int s = (lane < NT / 32) ? smem[lane] : INT_MIN;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int n = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s = max(s, n);
    }
    smem[lane] = s;  // inclusive max over warps 0..lane
  }
  __syncthreads();
  int prev = (w > 0) ? smem[w - 1] : INT_MIN;
  return max(inc, prev);
}

// Per expert id: exclusive prefix of its per-chunk counts over the chunks (in place) and the total.
// A CTA covers 64 expert ids (threadIdx.x, so the loads of a chunk row are coalesced) and cuts the chunks into
// kPrefixGroups consecutive ranges (threadIdx.y); a thread sums its range with its loads in flight in batches,
// the ranges' totals meet in shared memory, and a second pass over the (now cached) counts writes the prefixes.
constexpr int kPrefixIds = 64, kPrefixGroups = 4, kPrefixBatch = 16;
__global__ void __launch_bounds__(kPrefixIds * kPrefixGroups) plan_prefix_kernel(PlanView v) {
  __shared__ int s_sum[kPrefixGroups][kPrefixIds];
  pdl_begin();
  const int k = blockIdx.x * kPrefixIds + threadIdx.x, g = threadIdx.y;
  const bool on = k <= v.E;
  const size_t pitch = (size_t)(v.E + 1);
  const int per = (v.n_chunks + kPrefixGroups - 1) / kPrefixGroups;
  const int c_lo = g * per, c_hi = min(v.n_chunks, c_lo + per);
  int total = 0;
  for (int c0 = c_lo; on && c0 < c_hi; c0 += kPrefixBatch) {
    int n[kPrefixBatch];
#pragma unroll
    for (int j = 0; j < kPrefixBatch; ++j) n[j] = (c0 + j < c_hi) ? __ldcg(v.hist + (size_t)(c0 + j) * pitch + k) : 0;
#pragma unroll
    for (int j = 0; j < kPrefixBatch; ++j) total += n[j];
  }
  s_sum[g][threadIdx.x] = total;
  __syncthreads();
  int run = 0;
  for (int gg = 0; gg < g; ++gg) run += s_sum[gg][threadIdx.x];
  for (int c0 = c_lo; on && c0 < c_hi; c0 += kPrefixBatch) {
    int n[kPrefixBatch];
#pragma unroll
    for (int j = 0; j < kPrefixBatch; ++j) n[j] = (c0 + j < c_hi) ? __ldcg(v.hist + (size_t)(c0 + j) * pitch + k) : 0;
#pragma unroll
    for (int j = 0; j < kPrefixBatch; ++j) {
      if (c0 + j < c_hi) v.hist[(size_t)(c0 + j) * pitch + k] = run;
      run += n[j];
    }
  }
  if (on && g == kPrefixGroups - 1) v.keybase[k] = run;
}

// Row tiles of the long-run GEMM (see PlanView) from the runs that plan_tiles has numbered: a thread per grid tile.
template <int NT>
__device__ __forceinline__ void plan_gemm_tiles(const PlanView& v, int* smem, int n_runs) {
  const int tid = threadIdx.x, T = v.T;
  const int G = (T + kTileRows - 1) / kTileRows, per = (G + NT - 1) / NT;
  const int g_lo = min(G, tid * per), g_hi = min(G, g_lo + per);
  int count = 0;
  for (int g = g_lo; g < g_hi; ++g) {
    int last = n_runs - 1;
    if (g + 1 < G) {
      last = v.grid_run[g + 1];
      if (v.run_row0[last] == (g + 1) * kTileRows) --last;   // that run begins with the next tile
    }
    const int nr = last - v.grid_run[g] + 1;
    v.grid_nrun[g] = nr;
    count += (nr + kTileRuns - 1) / kTileRuns;
  }
  int total;
  int idx = block_excl_sum<NT>(count, smem, &total);
  for (int g = g_lo; g < g_hi; ++g) {
    const int f = v.grid_run[g], nr = v.grid_nrun[g];
    for (int r = 0; r < nr; r += kTileRuns) {
      const int row0 = r == 0 ? g * kTileRows : v.run_row0[f + r];
      const int end = r + kTileRuns < nr ? v.run_row0[f + r + kTileRuns] : min(T, (g + 1) * kTileRows);
      v.gemm_tab[idx++] = make_int4(row0, end - row0, f + r, min(kTileRuns, nr - r));
    }
  }
  if (tid == 0) v.header[PH_NGEMM] = total;
}

// Row tiles: maximal runs of equal expert id in token order, cut every kTileRows rows.  One CTA of NT
// threads; `key[t]` is the sanitised id of token t (shared or global memory).  smem: 33 ints.
// `row0` is where the tile starts are read back from to form the tile lengths: v.tile_row0 itself, or a
// shared-memory copy ([T + 1] ints) when the caller has one.
// Every thread takes one contiguous range of the tokens (a multiple of 4, read 16 bytes at a time), so the whole batch
// needs two block-wide scans; two scans per NT tokens made the kernel 27 us long at 16 384 tokens.
template <int NT>
__device__ __forceinline__ void plan_tiles(const PlanView& v, const int* key, int* smem, int* row0) {
  const int tid = threadIdx.x;
  const int T = v.T, E = v.E;
  const int per = ((T + NT - 1) / NT + 3) / 4 * 4;
  const int lo = min(T, tid * per), hi = min(T, lo + per);
  auto load4 = [&](int t, int (&k)[4]) {   // ids of tokens t .. t + 3 (t is a multiple of 4; -3 beyond the batch)
    if (t + 4 <= T) {
      const int4 w = *reinterpret_cast<const int4*>(key + t);
      k[0] = w.x; k[1] = w.y; k[2] = w.z; k[3] = w.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) k[i] = (t + i < T) ? key[t + i] : -3;
    }
  };
  const int before = (lo > 0 && lo < T) ? key[lo - 1] : -4;   // id of the token in front of the range
  // 1. last run start inside the range; its maximum over the earlier ranges is the run this range begins in
  int last = -1, prev = before;
  for (int t = lo; t < hi; t += 4) {
    int k[4];
    load4(t, k);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (t + i < hi) {
        if (k[i] != prev) last = t + i;
        prev = k[i];
      }
  }
  const int incl = block_incl_max<NT>(last, smem);
  int run = __shfl_up_sync(0xffffffffu, incl, 1);   // exclusive: the lane before, or the last lane of the warp before
  if ((tid & 31) == 0) run = tid > 0 ? smem[(tid >> 5) - 1] : -1;
  // 2. tiles and runs that start inside the range
  int count = 0, n_run = 0, rs = run;
  prev = before;
  for (int t = lo; t < hi; t += 4) {
    int k[4];
    load4(t, k);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (t + i < hi) {
        if (k[i] != prev) {
          rs = t + i;
          ++n_run;
        }
        prev = k[i];
        count += ((t + i - rs) % kTileRows) == 0;
      }
  }
  int total, n_runs;
  int idx = block_excl_sum<NT>(count, smem, &total);
  int ord = block_excl_sum<NT>(n_run, smem, &n_runs);
  // 3. the lists
  rs = run;
  prev = before;
  for (int t = lo; t < hi; t += 4) {
    int k[4];
    load4(t, k);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (t + i < hi) {
        if (k[i] != prev) {
          rs = t + i;
          v.run_expert[ord] = (k[i] == E) ? -1 : k[i];
          v.run_row0[ord] = rs;
          ++ord;
        }
        prev = k[i];
        if ((t + i) % kTileRows == 0) v.grid_run[(t + i) / kTileRows] = ord - 1;
        if (((t + i - rs) % kTileRows) == 0) {
          v.tile_row0[idx] = t + i;
          if (row0 != v.tile_row0) row0[idx] = t + i;
          v.tile_expert[idx] = (k[i] == E) ? -1 : k[i];
          ++idx;
        }
      }
  }
  if (tid == 0) {
    v.tile_row0[total] = T;
    v.run_row0[n_runs] = T;
    if (row0 != v.tile_row0) row0[total] = T;
    v.header[PH_NTILES] = total;
  }
  __syncthreads();
  for (int i = tid; i < total; i += NT) v.tile_rows[i] = row0[i + 1] - row0[i];
  plan_gemm_tiles<NT>(v, smem, n_runs);
}

__global__ void __launch_bounds__(1024) plan_scan_kernel(PlanView v, int do_prefix, int want_tiles) {
  constexpr int NT = 1024;
  __shared__ int smem[33];
  pdl_begin();
  const int tid = threadIdx.x;
  const int T = v.T, E = v.E, nc = v.n_chunks;
  const size_t pitch = (size_t)(E + 1);

  // 1. per expert id: prefix over chunks (in place) and total (done by plan_prefix_kernel for multi-chunk batches)
  for (int k = tid; do_prefix && k <= E; k += 1024) {
    int run = 0;
    for (int c = 0; c < nc; ++c) {
      int* p = v.hist + (size_t)c * pitch + k;
      int n = *p;
      *p = run;
      run += n;
    }
    v.keybase[k] = run;
  }
  __syncthreads();

  // 2. prefix over expert ids -> segment list (ascending expert id), "no adapter" bucket last; a contiguous range of
  // ids per thread, so one set of scans whatever E
  const int per = (E + NT - 1) / NT, k_lo = min(E, tid * per), k_hi = min(E, k_lo + per);
  int n_tok = 0, n_seg = 0, n_chunk = 0, max_seg = 0;
  for (int k = k_lo; k < k_hi; ++k) {
    const int n = v.keybase[k];
    n_tok += n;
    n_seg += n > 0;
    n_chunk += (n + kSegChunk - 1) / kSegChunk;
    max_seg = max(max_seg, n);
  }
  int carry_tok, carry_seg, carry_chunk;
  int tok = block_excl_sum<NT>(n_tok, smem, &carry_tok);
  int seg = block_excl_sum<NT>(n_seg, smem, &carry_seg);
  int chunk = block_excl_sum<NT>(n_chunk, smem, &carry_chunk);
  for (int k = k_lo; k < k_hi; ++k) {
    const int n = v.keybase[k];
    v.keybase[k] = tok;
    v.chunkbase[k] = chunk;   // (plan_scatter_kernel writes the chunks)
    if (n > 0) {
      v.seg_expert[seg] = k;
      v.seg_start[seg] = tok;
      v.seg_tab[seg] = make_int4(k, tok, n, 0);
      ++seg;
    }
    tok += n;
    chunk += (n + kSegChunk - 1) / kSegChunk;
  }
  max_seg = block_incl_max<NT>(max_seg, smem);
  if (tid == 1023) {
    v.seg_start[carry_seg] = carry_tok;
    v.keybase[E] = carry_tok;
    v.header[PH_NSEG] = carry_seg;
    v.header[PH_NCHUNK] = carry_chunk;
    v.header[PH_NLORA] = carry_tok;
    v.header[PH_MAXSEG] = max_seg;
    v.header[PH_T] = T;
    v.header[PH_E] = E;
  }

  // 3. row tiles (only the long-run kernels read them)
  if (want_tiles) {
    plan_tiles<NT>(v, v.key, smem, v.tile_row0);
  } else if (tid == 0) {
    v.header[PH_NTILES] = v.header[PH_NGEMM] = 0;
  }
}

// Whole plan of a batch of at most 1024 tokens in one CTA.  The tokens are sorted by the key
// (sanitised expert id << 10 | token index) with a bitonic network in shared memory: the low bits make
// the order stable, the sorted position of a token is its place in `perm`, and the segments are the
// runs of equal id in the sorted sequence (ascending id, the "no adapter" bucket E last).
constexpr int kPlanSmallT = 1024;
constexpr int kPlanSmallE = 1 << 20;   // the id must fit above the 10 token bits of a 31-bit key
template <int NT>   // threads = sort width: the power of two at or above T, at least 128
__global__ void __launch_bounds__(NT) plan_small_kernel(const int* __restrict__ token_expert, PlanView v,
                                                        DeviceStatus* status, int want_tiles) {
  __shared__ __align__(16) int s_key[NT];   // sanitised id by token
  __shared__ int s_sort[NT + 1];   // sort keys, then the segment starts plus one end marker (NT segments at most)
  __shared__ int s_row0[NT + 1];   // tile starts
  __shared__ int smem[33];
  pdl_begin();
  const int tid = threadIdx.x;
  const int T = v.T, E = v.E;
  int k = 0x1FFFFF;  // padding sorts last
  if (tid < T) {
    int e = token_expert[tid];
    if (e >= 0 && e < E) {
      k = e;
    } else {
      k = E;  // "no adapter" bucket
      if (e != -1) atomicAdd(&status->invalid_expert_ids, 1);
    }
  }
  s_key[tid] = (tid < T) ? k : -2;
  // A thread keeps its element in a register: partners in the same warp exchange by shuffle, others through the one of two
  // buffers that nobody reads any more (one barrier a step; every step through shared memory with two: 24 / 256 / 264 tokens
  // 4.6 / 5.1 / 6.1 us a launch, so 3.6 / 3.7 / 4.1).
  int v_sort = (k << 10) | tid, flip = 0;
#pragma unroll
  for (int size = 2; size <= NT; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      int other;
      if (stride >= 32) {
        int* buf = flip ? s_row0 : s_sort;
        flip ^= 1;
        buf[tid] = v_sort;
        __syncthreads();
        other = buf[tid ^ stride];
      } else {
        other = __shfl_xor_sync(0xffffffffu, v_sort, stride);
      }
      const bool keep_min = ((tid & stride) == 0) == ((tid & size) == 0);
      v_sort = keep_min ? min(v_sort, other) : max(v_sort, other);
    }
  }
  __syncthreads();
  s_sort[tid] = v_sort;
  __syncthreads();
  // sorted position p holds (id, token): perm, run starts, segment list
  const int mine = s_sort[tid];
  const int id = mine >> 10;
  if (tid < T) v.perm[tid] = mine & 1023;
  const int prev_id = (tid > 0) ? (s_sort[tid - 1] >> 10) : -1;
  const int is_start = (tid < T) && id < E && (tid == 0 || prev_id != id);
  int n_seg, n_lora;
  const int seg = block_excl_sum<NT>(is_start, smem, &n_seg);
  block_excl_sum<NT>((tid < T) && id < E, smem, &n_lora);   // tokens with an adapter sort first
  __syncthreads();                                           // every thread has read its neighbour's key
  if (is_start) s_sort[seg] = tid;                           // reuse as the segment-start list
  if (tid == 0) s_sort[n_seg] = n_lora;
  __syncthreads();
  int len = 0;
  if (is_start) {
    len = s_sort[seg + 1] - tid;
    v.seg_expert[seg] = id;
    v.seg_start[seg] = tid;
    v.seg_tab[seg] = make_int4(id, tid, len, 0);
  }
  if (tid == 0) v.seg_start[n_seg] = n_lora;
  // chunks: every kSegChunk-th position of a segment starts one
  const int my_seg = seg + is_start - 1;                     // segment of this sorted position (seg counts the starts before it)
  const int in_seg = tid < n_lora ? tid - s_sort[my_seg] : 1;
  int n_chunk;
  const int chunk = block_excl_sum<NT>((in_seg % kSegChunk) == 0, smem, &n_chunk);
  if ((in_seg % kSegChunk) == 0) v.chunk_tab[chunk] = make_int4(id, tid, min(kSegChunk, s_sort[my_seg + 1] - tid), 0);
  const int max_seg = block_incl_max<NT>(len, smem);
  if (tid == NT - 1) {
    v.header[PH_NSEG] = n_seg;
    v.header[PH_NCHUNK] = n_chunk;
    v.header[PH_NLORA] = n_lora;
    v.header[PH_MAXSEG] = max_seg;
    v.header[PH_T] = T;
    v.header[PH_E] = E;
  }
  if (want_tiles) {
    plan_tiles<NT>(v, s_key, smem, s_row0);
  } else if (tid == 0) {
    v.header[PH_NTILES] = v.header[PH_NGEMM] = 0;
  }
}

__global__ void __launch_bounds__(kPlanChunk) plan_scatter_kernel(PlanView v) {
  pdl_begin();
  const int t = blockIdx.x * kPlanChunk + threadIdx.x;
  if (t >= v.T) return;
  const int k = v.key[t];
  const int pos = v.keybase[k] + v.hist[(size_t)blockIdx.x * (size_t)(v.E + 1) + k] + v.rank[t];
  v.perm[pos] = t;
  if (k < v.E) {
    const int in_seg = pos - v.keybase[k];
    if ((in_seg % kSegChunk) == 0)
      v.chunk_tab[v.chunkbase[k] + in_seg / kSegChunk] = make_int4(k, pos, min(kSegChunk, v.keybase[k + 1] - pos), 0);
  }
}

int plan_launches(int T, int E) {
  if (T <= kPlanSmallT && E < kPlanSmallE) return 1;
  return T > kPlanChunk ? 4 : 3;
}

cudaError_t launch_plan_build(const int* token_expert, const PlanView& v, DeviceStatus* status, bool want_tiles,
                              cudaStream_t stream) {
  if (v.T <= kPlanSmallT && v.E < kPlanSmallE) {
    const int tiles = want_tiles;
    if (v.T <= 128) return launch_pdl(plan_small_kernel<128>, 1, 128, 0, stream, token_expert, v, status, tiles);
    if (v.T <= 256) return launch_pdl(plan_small_kernel<256>, 1, 256, 0, stream, token_expert, v, status, tiles);
    if (v.T <= 512) return launch_pdl(plan_small_kernel<512>, 1, 512, 0, stream, token_expert, v, status, tiles);
    return launch_pdl(plan_small_kernel<1024>, 1, 1024, 0, stream, token_expert, v, status, tiles);
  }
  launch_pdl(plan_rank_kernel, v.n_chunks, kPlanChunk, 0, stream, token_expert, v.T, v.E, v.key, v.rank, v.hist, status);
  if (v.n_chunks > 1)
    launch_pdl(plan_prefix_kernel, (v.E + 1 + kPrefixIds - 1) / kPrefixIds, dim3(kPrefixIds, kPrefixGroups), 0, stream, v);
  launch_pdl(plan_scan_kernel, 1, 1024, 0, stream, v, v.n_chunks > 1 ? 0 : 1, (int)want_tiles);
  launch_pdl(plan_scatter_kernel, v.n_chunks, kPlanChunk, 0, stream, v);
  return cudaGetLastError();
}

}  // namespace moin
