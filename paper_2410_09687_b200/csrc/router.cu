// Query router kernels: centroid inverse norms, the CUDA-core cosine-argmax kernel used for
// small problems and odd shapes, and the finishing pass shared with the tensor-core router.
#include <cooperative_groups.h>

#include "tc_gemm.cuh"

namespace cg = cooperative_groups;

namespace moin {

// inv_norm[k] = 1/|c_k| (0 for a zero row).  One warp per centroid.
__global__ void __launch_bounds__(256)
centroid_inv_norm_kernel(const __nv_bfloat16* __restrict__ c, int K, int D, float* __restrict__ inv_norm) {
  pdl_begin();
  const int k = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (k >= K) return;
  const __nv_bfloat16* row = c + (size_t)k * D;
  float s = 0.f;
  for (int ch = lane; ch < D / 8; ch += 32) {
    const uint4 v = ldg_cached(row + ch * 8);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float a = bf16_lo(w[q]), b = bf16_hi(w[q]);
      s = fmaf(a, a, s);
      s = fmaf(b, b, s);
    }
  }
  s = warp_sum(s);
  if (lane == 0) inv_norm[k] = (s > 0.f) ? rsqrtf(s) : 0.f;
}

constexpr int kRouteQB = 8;  // queries per CTA

// One CTA = 8 queries (bf16 in shared memory), 4 warps striding over centroids.
// sim = <q, c_k> * inv_norm[k]; strict '>' keeps the lowest index on ties; NaN never wins.
__global__ void __launch_bounds__(128)
route_simple_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ c,
                    const float* __restrict__ inv_norm, const int* __restrict__ cmap, int Q, int K, int D,
                    int* __restrict__ out_expert, int* __restrict__ out_centroid, float* __restrict__ out_best) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint4* sq = reinterpret_cast<uint4*>(smem_raw);  // [8][D/8]
  __shared__ float s_best[4][kRouteQB];
  __shared__ int s_id[4][kRouteQB];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_begin();
  const int q0 = blockIdx.x * kRouteQB;
  const int nch = D / 8;
  for (int i = tid; i < kRouteQB * nch; i += 128) {
    const int qi = i / nch, ch = i - qi * nch;
    sq[i] = (q0 + qi < Q) ? ldg_cached(q + (size_t)(q0 + qi) * D + ch * 8) : make_uint4(0, 0, 0, 0);
  }
  __syncthreads();
  float best = -INFINITY;
  int best_id = 0;
  for (int k = warp; k < K; k += 4) {
    float acc[kRouteQB];
#pragma unroll
    for (int j = 0; j < kRouteQB; ++j) acc[j] = 0.f;
    const __nv_bfloat16* crow = c + (size_t)k * D;
    for (int ch = lane; ch < nch; ch += 32) {
      const uint4 cv = ldg_cached(crow + ch * 8);
      const uint32_t cw[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
      for (int j = 0; j < kRouteQB; ++j) {
        const uint4 qv = sq[j * nch + ch];
        const uint32_t qw[4] = {qv.x, qv.y, qv.z, qv.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[j] = fmaf(bf16_lo(cw[e]), bf16_lo(qw[e]), acc[j]);
          acc[j] = fmaf(bf16_hi(cw[e]), bf16_hi(qw[e]), acc[j]);
        }
      }
    }
    const float inv = inv_norm[k];
#pragma unroll
    for (int j = 0; j < kRouteQB; ++j) {
      const float dot = warp_sum(acc[j]);
      const float sim = (inv > 0.f) ? dot * inv : -INFINITY;
      if (lane == j && sim > best) {
        best = sim;
        best_id = k;
      }
    }
  }
  if (lane < kRouteQB) {
    s_best[warp][lane] = best;
    s_id[warp][lane] = best_id;
  }
  __syncthreads();
  if (tid < kRouteQB && q0 + tid < Q) {
    float b = -INFINITY;
    int id = INT_MAX;
    for (int w = 0; w < 4; ++w) {
      const float s = s_best[w][tid];
      const int i = s_id[w][tid];
      if (s > b || (s == b && s > -INFINITY && i < id)) {
        b = s;
        id = i;
      }
    }
    if (!(b > -INFINITY)) id = 0;  // nothing won (all similarities -inf or NaN)
    if (out_centroid) out_centroid[q0 + tid] = id;
    out_expert[q0 + tid] = cmap ? cmap[id] : id;
    if (out_best) {
      // divide by |q| so the reported value is the cosine
      float ss = 0.f;
      for (int ch = 0; ch < nch; ++ch) {
        const uint4 qv = sq[tid * nch + ch];
        const uint32_t qw[4] = {qv.x, qv.y, qv.z, qv.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          ss = fmaf(bf16_lo(qw[e]), bf16_lo(qw[e]), ss);
          ss = fmaf(bf16_hi(qw[e]), bf16_hi(qw[e]), ss);
        }
      }
      out_best[q0 + tid] = b * rsqrtf(ss);
    }
  }
}

// Finishing pass of the tensor-core router: unpack the per-query (similarity, index) key that
// the GEMM epilogues merged with 64-bit atomicMax, apply the centroid->expert map, and turn
// the winning value into a cosine by dividing by |q|.  One warp per query.
__global__ void __launch_bounds__(256)
route_finish_kernel(const unsigned long long* __restrict__ keys, const __nv_bfloat16* __restrict__ q,
                    const int* __restrict__ cmap, int Q, int D, int* __restrict__ out_expert,
                    int* __restrict__ out_centroid, float* __restrict__ out_best) {
  pdl_begin();
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= Q) return;
  const unsigned long long key = keys[i];
  int id = (key == 0ull) ? 0 : (int)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));
  if (lane == 0) {
    if (out_centroid) out_centroid[i] = id;
    out_expert[i] = cmap ? cmap[id] : id;
  }
  if (out_best) {
    float ss = 0.f;
    for (int ch = lane; ch < D / 8; ch += 32) {
      const uint4 v = ldg_cached(q + (size_t)i * D + ch * 8);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        ss = fmaf(bf16_lo(w[e]), bf16_lo(w[e]), ss);
        ss = fmaf(bf16_hi(w[e]), bf16_hi(w[e]), ss);
      }
    }
    ss = warp_sum(ss);
    if (lane == 0) out_best[i] = (key == 0ull) ? -INFINITY : key_to_float((uint32_t)(key >> 32)) * rsqrtf(ss);
  }
}

// ----------------------------------------------------------------------------------------
// Small-batch router.
//
// A cluster of 8 CTAs serves NQ queries against one part of the centroid table.  The part is cut into 16-row
// tiles, dealt round-robin to the cluster's warps; a warp holds its tile's rows as the A operand of m16n8k16 (loaded
// straight from global memory, 16 bytes per lane: lane t of a row group takes k-elements 8t..8t+7 of every 32, and the
// queries, staged once in shared memory, are read with the same k assignment, so the contraction is unchanged) and the
// NQ queries as NQ/8 B operands.  Every lane keeps the best candidate of its rows over all its tiles; they meet per CTA
// in shared memory with a 64-bit max on the (similarity, index) key, and after a cluster barrier CTA 0 reads the other
// CTAs' keys through distributed shared memory.  A table in one part (up to 512 centroids) is finished right there:
// one launch, no scratch.  Larger tables are cut into parts, one cluster each, whose keys go to
// scratch and meet in a small second launch.  Without scratch (WALK) one cluster takes the whole table, a tile per warp; it
// adds up the two halves of a row that two warps of a part would have had apart, so that the bits are the same (1 x 5000 x
// 768: 7.7 us in ten parts, 21.7 without scratch).
//
// What bounds it: a few dependent memory round trips, and what the SMs of one cluster can pull - one cluster of 16
// needs 15.3 us for 1 x 5000 x 768 (480 KB per SM), ten clusters and the second launch 7.4 us (the CUDA-core kernel
// with its one CTA per eight queries: 1446 us).  The centroid loads run one batch of kRcBatch k-steps ahead of
// the products, across tiles too (deeper register rings measured slower: 16.5 us), and the queries' rows are skewed to
// 64 bytes past a multiple of 128, so that the eight rows of a fragment sit on distinct banks.  NQ = 8 for up to eight
// queries: 5.8 us at 500 centroids against 9.1 us for a 32-wide query block.
// ----------------------------------------------------------------------------------------
constexpr int kRcWarps = 8, kRcBatch = 6;

__device__ __forceinline__ unsigned long long shfl_xor_u64(unsigned long long v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o);
}
// best two of two (best, second) pairs of distinct keys (0 = none)
__device__ __forceinline__ void merge_top2(unsigned long long& b, unsigned long long& s, unsigned long long ob,
                                           unsigned long long os) {
  const unsigned long long hi = b > ob ? b : ob, lo = b > ob ? ob : b, se = s > os ? s : os;
  b = hi;
  s = lo > se ? lo : se;
}
__host__ __device__ inline int route_pitch(int D) {   // bytes of a query row in shared memory, 64 mod 128
  const int row = (D + 31) / 32 * 64;
  return (row & 127) ? row : row + 64;
}
__device__ __forceinline__ void add_sq8(const uint4& v, float& ss) {   // ss += the squares of eight bf16
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    ss = fmaf(bf16_lo(w[e]), bf16_lo(w[e]), ss);
    ss = fmaf(bf16_hi(w[e]), bf16_hi(w[e]), ss);
  }
}

struct RouteOut { int *expert, *centroid, *second; float *best, *margin; };

// keys -> outputs of query i (ss = |q_i|^2)
template <bool TOP2>
__device__ __forceinline__ void route_write(const RouteOut& out, const int* cmap, int i, unsigned long long k1,
                                            unsigned long long k2, float ss) {
  const int id = (k1 == 0ull) ? 0 : (int)(0xFFFFFFFFu - (uint32_t)(k1 & 0xFFFFFFFFull));
  const float rq = rsqrtf(ss), s1 = key_to_float((uint32_t)(k1 >> 32)), s2 = key_to_float((uint32_t)(k2 >> 32));
  if (out.centroid) out.centroid[i] = id;
  if (out.expert) out.expert[i] = cmap ? cmap[id] : id;
  if (out.best) out.best[i] = (k1 == 0ull) ? -INFINITY : s1 * rq;
  if (TOP2) {
    if (out.second) out.second[i] = (k2 == 0ull) ? -1 : (int)(0xFFFFFFFFu - (uint32_t)(k2 & 0xFFFFFFFFull));
    if (out.margin) out.margin[i] = (k1 == 0ull || k2 == 0ull) ? INFINITY : (s1 - s2) * rq;
  }
}

// part_keys (nullptr when parts == 1 or WALK): [parts][Q] keys, and with TOP2 [parts][Q] runner-up keys behind them
template <int NQ, bool TOP2, bool WALK>
__global__ void __launch_bounds__(kRcWarps * 32)
route_cluster_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ c,
                     const float* __restrict__ inv_norm, const int* __restrict__ cmap, int Q, int K, int D, int parts,
                     unsigned long long* __restrict__ part_keys, const RouteOut out) {
  constexpr int NJ = NQ / 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned long long s_keys[NQ], s_keys2[NQ];
  __shared__ float s_part[kRcWarps / 2][NJ][4][32];
  pdl_begin();
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int rank = (int)cluster.block_rank(), csize = (int)cluster.num_blocks();
  const int cl = blockIdx.x / csize, part = WALK ? 0 : cl % parts, q0 = (WALK ? cl : cl / parts) * NQ;
  const int pitch = route_pitch(D);
  const int nch = D / 8, steps = (nch + 3) / 4, all_tiles = (K + 15) / 16;
  const int tile_lo = WALK ? 0 : (int)((long long)all_tiles * part / parts);
  const int tile_hi = WALK ? all_tiles : (int)((long long)all_tiles * (part + 1) / parts);
  // few tiles: two warps share one, half of the k range each (the halves are added in shared memory in a fixed order)
  const bool halves = (all_tiles + parts - 1) / parts <= csize * (kRcWarps / 2);   // (the same in every part)
  const int ksplit = halves && !WALK ? 2 : 1, tile_warps = kRcWarps / ksplit;
  const int tw = warp % tile_warps, kpart = warp / tile_warps;
  const int steps_part = (steps + ksplit - 1) / ksplit;
  const int s_lo = kpart * steps_part, s_hi = min(steps, s_lo + steps_part);
  const int nb = (steps_part + kRcBatch - 1) / kRcBatch;   // batches per tile
  const int second = WALK && halves ? (steps + 1) / 2 : INT_MAX;   // first step of the second half

  uint4 a[2][kRcBatch][2];
  auto load = [&](uint4 (&r)[kRcBatch][2], int tl, int b) {
    const int r0 = tl * 16 + g, r1 = r0 + 8;
    // rows past K read row K-1 (in bounds) and are masked at the end
    const __nv_bfloat16* p0 = c + (size_t)min(r0, K - 1) * D;
    const __nv_bfloat16* p1 = c + (size_t)min(r1, K - 1) * D;
#pragma unroll
    for (int u = 0; u < kRcBatch; ++u) {
      const int st = s_lo + b * kRcBatch + u, ch = st * 4 + t;
      const bool on = tl < tile_hi && st < s_hi && ch < nch;
      r[u][0] = on ? ldg_cached(p0 + ch * 8) : make_uint4(0, 0, 0, 0);
      r[u][1] = on ? ldg_cached(p1 + ch * 8) : make_uint4(0, 0, 0, 0);
    }
  };
  // the first centroid rows are requested before the queries are staged: one round trip for both
  int tile = tile_lo + rank * tile_warps + tw;
  const int stride = csize * tile_warps;
  load(a[0], tile, 0);
  const int row_ch = steps * 4;   // chunks of a staged row, zero beyond the embedding
  for (int i0 = 0; i0 < NQ * row_ch; i0 += kRcWarps * 32 * 12) {
    uint4 v[12];
#pragma unroll
    for (int u = 0; u < 12; ++u) {
      const int i = i0 + u * kRcWarps * 32 + tid;
      const int qi = i / row_ch, ch = i - qi * row_ch;
      v[u] = (i < NQ * row_ch && q0 + qi < Q && ch < nch) ? ldg_cached(q + (size_t)(q0 + qi) * D + ch * 8) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int u = 0; u < 12; ++u) {
      const int i = i0 + u * kRcWarps * 32 + tid;
      const int qi = i / row_ch, ch = i - qi * row_ch;
      if (i < NQ * row_ch) *reinterpret_cast<uint4*>(smem_raw + (size_t)qi * pitch + ch * 16) = v[u];
    }
  }
  if (tid < NQ) {
    s_keys[tid] = 0ull;
    s_keys2[tid] = 0ull;
  }
  __syncthreads();

  // candidates of this lane: queries j*8 + 2t + e; rows in increasing order, strict '>' keeps the lowest index
  float best[NJ][2], runner[NJ][2];
  int best_k[NJ][2], runner_k[NJ][2];
#pragma unroll
  for (int j = 0; j < NJ; ++j)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      best[j][e] = runner[j][e] = -INFINITY;
      best_k[j][e] = runner_k[j][e] = 0;
    }
  float acc[NJ][4];
#pragma unroll
  for (int j = 0; j < NJ; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
  float acc0[NJ][4];   // WALK: of the first half
  auto multiply = [&](uint4 (&r)[kRcBatch][2], int b) {
#pragma unroll
    for (int u = 0; u < kRcBatch; ++u) {
      const int st = s_lo + b * kRcBatch + u;
      if (st >= s_hi) break;
      if (WALK && st == second) {
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            acc0[j][e] = acc[j][e];
            acc[j][e] = 0.f;
          }
      }
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const uint4 bv = *reinterpret_cast<const uint4*>(smem_raw + (size_t)(j * 8 + g) * pitch + st * 64 + t * 16);
        mma_bf16_16816(acc[j], r[u][0].x, r[u][1].x, r[u][0].y, r[u][1].y, bv.x, bv.y);
        mma_bf16_16816(acc[j], r[u][0].z, r[u][1].z, r[u][0].w, r[u][1].w, bv.z, bv.w);
      }
    }
  };
  auto take = [&](float sim, int k, int j, int e) {
    if (sim > best[j][e]) {
      if (TOP2) { runner[j][e] = best[j][e]; runner_k[j][e] = best_k[j][e]; }
      best[j][e] = sim;
      best_k[j][e] = k;
    } else if (TOP2 && sim > runner[j][e]) {
      runner[j][e] = sim;
      runner_k[j][e] = k;
    }
  };
  auto finish_tile = [&]() {   // (CTA-uniform trip count when two warps share a tile)
    if (ksplit == 2) {
      if (kpart > 0) {
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) s_part[tw][j][e][lane] = acc[j][e];
      }
      __syncthreads();
      if (kpart == 0) {
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[j][e] += s_part[tw][j][e][lane];
      }
    }
    if (WALK && second < steps) {
#pragma unroll
      for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] += acc0[j][e];
    }
    if (kpart == 0 && tile < tile_hi) {
      // acc[j][0..1]: centroid r0, queries j*8 + 2t, 2t+1;  acc[j][2..3]: centroid r1
      const int r0 = tile * 16 + g, r1 = r0 + 8;
      const float inv0 = (r0 < K) ? inv_norm[r0] : 0.f, inv1 = (r1 < K) ? inv_norm[r1] : 0.f;
#pragma unroll
      for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (inv0 > 0.f) take(acc[j][e] * inv0, r0, j, e);
          if (inv1 > 0.f) take(acc[j][2 + e] * inv1, r1, j, e);
        }
    }
#pragma unroll
    for (int j = 0; j < NJ; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
  };
  if (ksplit == 2) {   // at most one tile per warp: every warp walks the same number of batches
    for (int b = 0; b < nb; b += 2) {
      if (b + 1 < nb) load(a[1], tile, b + 1);
      multiply(a[0], b);
      if (b + 2 < nb) load(a[0], tile, b + 2);
      if (b + 1 < nb) multiply(a[1], b + 1);
    }
    finish_tile();
  } else {             // (tile, batch) pairs in sequence, two per turn so that the buffers are static
    int b = 0;
    auto advance = [&](int& tl, int& bb) {
      if (++bb == nb) { bb = 0; tl += stride; }
    };
    while (tile < tile_hi) {
      int tl = tile, bb = b;
      advance(tl, bb);
      load(a[1], tl, bb);
      multiply(a[0], b);
      if (b == nb - 1) finish_tile();
      tile = tl; b = bb;
      if (tile >= tile_hi) break;
      advance(tl, bb);
      load(a[0], tl, bb);
      multiply(a[1], b);
      if (b == nb - 1) finish_tile();
      tile = tl; b = bb;
    }
  }
  // the eight row groups of a warp meet by shuffles, the warps in shared memory, the CTAs below
  if (kpart == 0) {
#pragma unroll
    for (int j = 0; j < NJ; ++j)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        // key 0 = no candidate (zero-norm or padding row, NaN or -inf similarity)
        unsigned long long k1 = best[j][e] > -INFINITY ? route_key(best[j][e], best_k[j][e]) : 0ull;
        unsigned long long k2 = (TOP2 && runner[j][e] > -INFINITY) ? route_key(runner[j][e], runner_k[j][e]) : 0ull;
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          const unsigned long long o1 = shfl_xor_u64(k1, o);
          if (TOP2) merge_top2(k1, k2, o1, shfl_xor_u64(k2, o));
          else k1 = o1 > k1 ? o1 : k1;
        }
        if (g == 0 && k1 != 0ull) {
          // two-slot merge: whatever loses a comparison for the first slot is offered to the second
          unsigned long long old = atomicMax(&s_keys[j * 8 + 2 * t + e], k1);
          if (TOP2) {
            old = old < k1 ? old : k1;
            if (old != 0ull) atomicMax(&s_keys2[j * 8 + 2 * t + e], old);
            if (k2 != 0ull) atomicMax(&s_keys2[j * 8 + 2 * t + e], k2);
          }
        }
      }
  }
  cluster.sync();
  if (rank == 0) {
    // eight lanes per query fetch the CTAs' keys and share the norm
    const int qi = tid >> 3, sub = tid & 7;
    const bool on = qi < NQ && q0 + qi < Q;
    unsigned long long k1 = 0ull, k2 = 0ull;
    if (on) {
      for (int r = sub; r < csize; r += 8) {
        const unsigned long long o1 = *cluster.map_shared_rank(&s_keys[qi], r);
        if (TOP2) merge_top2(k1, k2, o1, *cluster.map_shared_rank(&s_keys2[qi], r));
        else k1 = o1 > k1 ? o1 : k1;
      }
    }
    float ss = 0.f;
    if (on && (parts == 1 || WALK) && (out.best || out.margin))
      for (int ch = sub; ch < nch; ch += 8) add_sq8(*reinterpret_cast<const uint4*>(smem_raw + (size_t)qi * pitch + ch * 16), ss);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const unsigned long long o1 = shfl_xor_u64(k1, o);
      if (TOP2) merge_top2(k1, k2, o1, shfl_xor_u64(k2, o));
      else k1 = o1 > k1 ? o1 : k1;
      ss += __shfl_xor_sync(0xffffffffu, ss, o);
    }
    if (on && sub == 0) {
      if (parts > 1 && !WALK) {
        part_keys[(size_t)part * Q + q0 + qi] = k1;
        if (TOP2) part_keys[(size_t)(parts + part) * Q + q0 + qi] = k2;
      } else {
        route_write<TOP2>(out, cmap, q0 + qi, k1, k2, ss);
      }
    }
  }
  cluster.sync();  // the other CTAs' shared memory stays alive until CTA 0 has read it
}

// The parts of a table meet: eight lanes per query.
template <bool TOP2>
__global__ void __launch_bounds__(128)
route_parts_kernel(const unsigned long long* __restrict__ part_keys, int parts, const __nv_bfloat16* __restrict__ q,
                   const int* __restrict__ cmap, int Q, int D, const RouteOut out) {
  const int i = blockIdx.x * 16 + (threadIdx.x >> 3), sub = threadIdx.x & 7;
  const bool on = i < Q;
  float ss = 0.f;
  if (on && (out.best || out.margin))
    for (int ch = sub; ch < D / 8; ch += 8) add_sq8(ldg_cached(q + (size_t)i * D + ch * 8), ss);
  pdl_begin();   // the parts' keys (the queries above are older: the kernel before this one has waited for them)
  unsigned long long k1 = 0ull, k2 = 0ull;
  if (on) {
    for (int r = sub; r < parts; r += 8) {
      const unsigned long long o1 = __ldcg(part_keys + (size_t)r * Q + i);
      if (TOP2) merge_top2(k1, k2, o1, __ldcg(part_keys + (size_t)(parts + r) * Q + i));
      else k1 = o1 > k1 ? o1 : k1;
    }
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    const unsigned long long o1 = shfl_xor_u64(k1, o);
    if (TOP2) merge_top2(k1, k2, o1, shfl_xor_u64(k2, o));
    else k1 = o1 > k1 ? o1 : k1;
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
  }
  if (on && sub == 0) route_write<TOP2>(out, cmap, i, k1, k2, ss);
}

__global__ void __launch_bounds__(256)
clear_keys_kernel(unsigned long long* __restrict__ keys, size_t n) {   // keys is 16-byte aligned
  pdl_begin();
  const size_t i = 2 * ((size_t)blockIdx.x * 256 + threadIdx.x);
  if (i + 1 < n) *reinterpret_cast<ulonglong2*>(keys + i) = make_ulonglong2(0ull, 0ull);
  else if (i < n) keys[i] = 0ull;
}
cudaError_t launch_clear_keys(unsigned long long* keys, size_t n, cudaStream_t stream) {
  return launch_pdl(clear_keys_kernel, (unsigned)((n + 511) / 512), 256, 0, stream, keys, n);
}

// How a problem is cut: queries per cluster, CTAs per cluster, parts of the table; fast = the rule picks this kernel.
struct RouteCut { int nq, csize, parts, groups; bool fast; };
// A handful of topics: the CUDA-core kernel has them done before a cluster is set up (D = 768, 1 to 384 queries x 1 topic
// 5.4-8.7 us by the cluster kernel, 3.1-3.8 so; x 8 5.6-8.6 / 4.4-5.0; 512 x 16 8.1 by the GEMM, 7.2 so).
bool route_few_topics(int Q, int K, int D) { return K <= 16 && K * D <= 16 * 768 && (long long)Q * K < (1ll << 16); }
static RouteCut route_cut(int Q, int K, int D) {
  RouteCut r = {0, 8, 1, 0, false};
  if (Q < 1 || K < 1 || (D % 8) != 0 || 8 * route_pitch(D) > 200 * 1024) return r;
  const int nq = r.nq = (Q > 8 && 32 * route_pitch(D) <= 200 * 1024) ? 32 : 8;
  r.groups = (Q + nq - 1) / nq;
  // One tile per warp pair of a cluster of 8 = 512 centroids per part, while all clusters are resident at once: a
  // cluster of 8 one-per-SM CTAs needs 8 free SMs of one GPC, and 16 of them take two waves (500 centroids x 768,
  // 256 queries = 8 clusters 9.8 us, 512 queries = 16 clusters 18.4 us).
  constexpr int kResident = kRouteMaxPartKeys / 32;
  while (r.parts < kRouteMaxParts && K > 512 * r.parts && r.groups * (r.parts + 1) <= kResident) ++r.parts;
  const int tiles = (K + 512 * r.parts - 1) / (512 * r.parts);   // tiles per warp pair
  // Against the tensor-core GEMM with its clearing and finishing launches (11.8 us up to 128 queries, 14.4 at 256 x
  // 5000 x 768): 7.3 us for up to 8 queries and 9.8-10.6 us for up to 32 per cluster with one tile per warp pair,
  // 13.3 and 18.7 with two.
  r.fast = r.groups * r.parts <= kResident && tiles <= (nq == 8 ? 2 : 1);
  // Too narrow for the GEMM: against the CUDA-core kernel (2.2 us + 0.18 us a centroid) a wave of clusters takes 6.3 us
  // (D = 40: 512 queries x 30 12.6 / 6.9 us, 1500 x 100 25.9 / 20.2, 1500 x 300 27 / 60).
  if (!tc_router_supported(Q, K, D)) r.fast = r.fast || (r.groups <= 64 && K > 35 * ((r.groups + kResident - 1) / kResident));
  if (route_few_topics(Q, K, D)) r.fast = false;
  return r;
}
bool route_cluster_supported(int Q, int K, int D) { return route_cut(Q, K, D).fast; }
int route_parts(int Q, int K, int D) {
  const RouteCut r = route_cut(Q, K, D);
  return r.fast ? r.parts : 1;
}
template <int NQ, bool TOP2, bool WALK>
static cudaError_t launch_rc(int optin, const RouteCut& cut, const __nv_bfloat16* q, const __nv_bfloat16* c,
                             const float* inv_norm, const int* cmap, int Q, int K, int D, const RouteOut& out,
                             unsigned long long* part_keys, cudaStream_t stream) {
  const size_t smem = (size_t)NQ * route_pitch(D);
  const int clusters = WALK ? 1 : cut.parts;   // per group of queries
  cudaError_t ce = ensure_smem_optin(optin, route_cluster_kernel<NQ, TOP2, WALK>, smem > 64 * 1024 ? smem : 64 * 1024);
  if (ce != cudaSuccess) return ce;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cut.csize;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(cut.groups * clusters * cut.csize));
  cfg.blockDim = dim3(kRcWarps * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  ce = cudaLaunchKernelEx(&cfg, route_cluster_kernel<NQ, TOP2, WALK>, q, c, inv_norm, cmap, Q, K, D, cut.parts, part_keys, out);
  if (ce != cudaSuccess || clusters == 1) return ce;
  return launch_pdl(route_parts_kernel<TOP2>, (Q + 15) / 16, 128, 0, stream, part_keys, cut.parts, q, cmap, Q, D, out);
}
template <bool TOP2>
static cudaError_t launch_rc(const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm, const int* cmap, int Q,
                             int K, int D, const RouteOut& out, unsigned long long* part_keys, cudaStream_t stream) {
  const RouteCut cut = route_cut(Q, K, D);
  const bool walk = cut.parts > 1 && part_keys == nullptr;
  const int slot = OPTIN_ROUTE_CLUSTER + 4 * TOP2 + 2 * walk + (cut.nq == 8);
  if (cut.nq == 32)
    return walk ? launch_rc<32, TOP2, true>(slot, cut, q, c, inv_norm, cmap, Q, K, D, out, part_keys, stream)
                : launch_rc<32, TOP2, false>(slot, cut, q, c, inv_norm, cmap, Q, K, D, out, part_keys, stream);
  return walk ? launch_rc<8, TOP2, true>(slot, cut, q, c, inv_norm, cmap, Q, K, D, out, part_keys, stream)
              : launch_rc<8, TOP2, false>(slot, cut, q, c, inv_norm, cmap, Q, K, D, out, part_keys, stream);
}

cudaError_t launch_route_cluster(const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm,
                                 const int* cmap, int Q, int K, int D, int* out_expert, int* out_centroid,
                                 float* out_best, unsigned long long* part_keys, cudaStream_t stream) {
  const RouteOut out = {out_expert, out_centroid, nullptr, out_best, nullptr};
  return launch_rc<false>(q, c, inv_norm, cmap, Q, K, D, out, part_keys, stream);
}
cudaError_t launch_route_top2_cluster(const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm,
                                      const int* cmap, int Q, int K, int D, int* out_expert, int* out_centroid,
                                      int* out_second, float* out_best, float* out_margin,
                                      unsigned long long* part_keys, cudaStream_t stream) {
  const RouteOut out = {out_expert, out_centroid, out_second, out_best, out_margin};
  return launch_rc<true>(q, c, inv_norm, cmap, Q, K, D, out, part_keys, stream);
}

// ----------------------------------------------------------------------------------------
// K-means update: centroid of every non-empty cluster = mean of its member rows, its inverse norm with it; a cluster
// without members keeps its centroid.  One CTA per segment of the plan built from the assignments (segment = cluster
// id, start, length in `perm`, members in increasing point order); the CTAs behind those copy the clusters without a
// segment, a warp for each kMeanEmpties clusters, so one launch covers the table however the points are spread.  (The
// empty clusters next to a segment copied by the segment's CTA: 40000 points in the first 500 of 1000 clusters 77 us,
// no point in any 134 us, now 16 and 8.)
//
// HBM-bound (every point is read once) as long as enough rows are in flight: warp (g, p) of a CTA adds part p of the
// members in column group g (256 columns, 8 a lane; up to 128 columns several members at once), eight rows in flight,
// and the parts' sums are added in order.  P grows with the members per cluster.  One warp per column group walking
// all the members four at a time took 26.5 us for 40000 x 768 in 1000 clusters and 66.7 us for 6141 in 28, now 19.3
// and 9.0 us, with the copy of the table and the norms (4.4 us, two launches) in the same launch.
// ----------------------------------------------------------------------------------------
constexpr int kMeanRows = 8, kMeanMaxWarps = 16, kMeanEmpties = 8;
__global__ void __launch_bounds__(kMeanMaxWarps * 32, 2)
kmeans_update_kernel(const int* __restrict__ header, const int* __restrict__ perm, const int4* __restrict__ seg_tab,
                     const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* c_old, __nv_bfloat16* c_new,
                     float* __restrict__ inv_new, int K, int D, int G, int P, int seg_ctas) {
  __shared__ float4 s_acc[kMeanMaxWarps][2][32];
  __shared__ float s_ss[kMeanMaxWarps];
  pdl_begin();
  const int nseg = header[PH_NSEG];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_warps = blockDim.x >> 5;
  const int g = warp % G, part = warp / G, nch = D / 8;
  const int lpr = nch <= 8 ? 8 : nch <= 16 ? 16 : 32, rows = 32 / lpr;   // lanes per row, members taken at once
  const int sub = lane / lpr, lc = lane % lpr;
  if ((int)blockIdx.x >= seg_ctas) {   // clusters m0 .. m0 + kMeanEmpties - 1 as far as they are empty
    const int m0 = (((int)blockIdx.x - seg_ctas) * n_warps + warp) * kMeanEmpties;
    if (m0 >= K || blockIdx.y > 0) return;
    int lo = 0, hi = nseg;   // first segment of a cluster >= m0: the lanes probe 32 places at a time
    while (lo < hi) {
      const int step = (hi - lo + 32) / 33, at = lo + (lane + 1) * step - 1;
      const int below = __popc(__ballot_sync(0xffffffffu, at < hi && __ldg(seg_tab + min(at, hi - 1)).x < m0));
      lo = min(hi, lo + below * step);
      if (below < 32) hi = min(hi, lo + step - 1);
    }
    const int k = lo + lane < nseg && lane < kMeanEmpties ? __ldg(seg_tab + lo + lane).x : K;
    const uint32_t full = __reduce_or_sync(0xffffffffu, k < m0 + kMeanEmpties ? 1u << (k - m0) : 0u);
    for (int m = m0; m < min(K, m0 + kMeanEmpties); ++m) {
      if ((full >> (m - m0)) & 1u) continue;
      float s2 = 0.f;
      for (int ch = lane; ch < nch; ch += 32) {
        const uint4 v = *reinterpret_cast<const uint4*>(c_old + (size_t)m * D + ch * 8);
        if (c_new != c_old) *reinterpret_cast<uint4*>(c_new + (size_t)m * D + ch * 8) = v;
        add_sq8(v, s2);
      }
      s2 = warp_sum(s2);
      if (inv_new != nullptr && lane == 0) inv_new[m] = s2 > 0.f ? rsqrtf(s2) : 0.f;
    }
    return;
  }
  for (int seg = blockIdx.x; seg < nseg; seg += seg_ctas) {
    const int4 e = __ldg(seg_tab + seg);   // (cluster, start, length, -)
    const int k = e.x, lo = e.y + (int)((long long)e.z * part / P), hi = e.y + (int)((long long)e.z * (part + 1) / P);
    float ss = 0.f;
    const int c_step = 32 * G * gridDim.y;   // (gridDim.y > 1: the column groups are spread over CTAs, norms come later)
    for (int c0 = 32 * G * blockIdx.y; c0 < nch; c0 += c_step) {
      const int ch = c0 + g * 32 + lc;
      const bool on = ch < nch;
      float acc[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] = 0.f;
      for (int j0 = lo; j0 < hi; j0 += 32) {
        const int nb = min(32, hi - j0);
        const int idx = lane < nb ? __ldg(perm + j0 + lane) : 0;
        for (int j = 0; j < nb; j += kMeanRows * rows) {
          uint4 v[kMeanRows];
#pragma unroll
          for (int u = 0; u < kMeanRows; ++u) {
            const int m = j + u * rows + sub, row = __shfl_sync(0xffffffffu, idx, m & 31);
            v[u] = (on && m < nb) ? ldg_stream(x + (size_t)row * D + ch * 8) : make_uint4(0, 0, 0, 0);
          }
#pragma unroll
          for (int u = 0; u < kMeanRows; ++u) {   // absent rows add zero
            const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              acc[2 * q] += bf16_lo(w[q]);
              acc[2 * q + 1] += bf16_hi(w[q]);
            }
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
        for (int o = lpr; o < 32; o <<= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
      s_acc[warp][0][lane] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      s_acc[warp][1][lane] = make_float4(acc[4], acc[5], acc[6], acc[7]);
      __syncthreads();
      if (part == 0 && on && sub == 0) {
        for (int p = 1; p < P; ++p) {
          const float4 u = s_acc[p * G + g][0][lane], w = s_acc[p * G + g][1][lane];
          acc[0] += u.x; acc[1] += u.y; acc[2] += u.z; acc[3] += u.w;
          acc[4] += w.x; acc[5] += w.y; acc[6] += w.z; acc[7] += w.w;
        }
        const float n = (float)e.z;
        uint4 o;
        o.x = pack_bf16(acc[0] / n, acc[1] / n);
        o.y = pack_bf16(acc[2] / n, acc[3] / n);
        o.z = pack_bf16(acc[4] / n, acc[5] / n);
        o.w = pack_bf16(acc[6] / n, acc[7] / n);
        *reinterpret_cast<uint4*>(c_new + (size_t)k * D + ch * 8) = o;
        add_sq8(o, ss);
      }
      __syncthreads();
    }
    if (inv_new != nullptr) {
      ss = warp_sum(ss);
      if (lane == 0) s_ss[warp] = ss;
      __syncthreads();
      if (tid == 0) {
        float t = s_ss[0];
        for (int i = 1; i < G; ++i) t += s_ss[i];   // (the warps of part 0)
        inv_new[k] = t > 0.f ? rsqrtf(t) : 0.f;
      }
      __syncthreads();
    }
  }
}

// Enough clusters to fill the GPU: a CTA takes whole rows and the norm with them.  Fewer: its column groups go to
// CTAs of their own (65536 x 768 in 20 clusters: 446 us whole rows, 92 us) and the norms to a second launch.
bool kmeans_update_split(int K, int D, int n_sms) { return K < 2 * n_sms && D > 256; }
cudaError_t launch_kmeans_update(const PlanView& pv, const __nv_bfloat16* x, const __nv_bfloat16* c_old,
                                 __nv_bfloat16* c_new, float* inv_new, int D, int n_sms, cudaStream_t stream) {
  const int nch = D / 8, groups = (nch + 31) / 32;
  const bool split = kmeans_update_split(pv.E, D, n_sms);
  const int G = split ? 1 : groups < 4 ? groups : 4;
  int P = pv.T / pv.E / 16;   // sixteen members per warp
  P = P < 1 ? 1 : P > kMeanMaxWarps / G ? kMeanMaxWarps / G : P;
  const int seg_ctas = pv.Smax < n_sms * 16 ? pv.Smax : n_sms * 16;
  const int empty_warps = (pv.E + kMeanEmpties - 1) / kMeanEmpties, empty_ctas = (empty_warps + G * P - 1) / (G * P);
  launch_pdl(kmeans_update_kernel, dim3((unsigned)(seg_ctas + empty_ctas), split ? (unsigned)groups : 1u), 32 * G * P, 0, stream,
             pv.header, pv.perm, pv.seg_tab, x, c_old, c_new, split ? nullptr : inv_new, pv.E, D, G, P, seg_ctas);
  if (split && inv_new != nullptr) return launch_inv_norm(c_new, pv.E, D, inv_new, stream);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------------------
// Best and runner-up (top-2) router on the CUDA cores: one warp per query, lanes stride over the
// embedding, centroids in increasing order (strict '>' keeps the lowest index among equals for both
// places).  Small problems and odd shapes; the tensor-core path covers the rest.
// ----------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
route_top2_simple_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ c,
                         const float* __restrict__ inv_norm, const int* __restrict__ cmap, int Q, int K, int D,
                         int* __restrict__ out_expert, int* __restrict__ out_centroid, int* __restrict__ out_second,
                         float* __restrict__ out_best, float* __restrict__ out_margin) {
  pdl_begin();
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= Q) return;
  const int nch = D / 8;
  float best = -INFINITY, second = -INFINITY, qq = 0.f;
  int best_k = 0, second_k = -1;
  for (int k = 0; k < K; ++k) {
    float acc = 0.f;
    for (int ch = lane; ch < nch; ch += 32) {
      const uint4 qv = ldg_cached(q + (size_t)i * D + ch * 8), cv = ldg_cached(c + (size_t)k * D + ch * 8);
      const uint32_t qw[4] = {qv.x, qv.y, qv.z, qv.w}, cw[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc = fmaf(bf16_lo(qw[e]), bf16_lo(cw[e]), acc);
        acc = fmaf(bf16_hi(qw[e]), bf16_hi(cw[e]), acc);
        if (k == 0) {
          qq = fmaf(bf16_lo(qw[e]), bf16_lo(qw[e]), qq);
          qq = fmaf(bf16_hi(qw[e]), bf16_hi(qw[e]), qq);
        }
      }
    }
    acc = warp_sum(acc);
    const float inv = inv_norm[k];
    const float sim = acc * inv;
    if (inv > 0.f && sim > best) {
      second = best; second_k = (best > -INFINITY) ? best_k : -1;
      best = sim; best_k = k;
    } else if (inv > 0.f && sim > second) {
      second = sim; second_k = k;
    }
  }
  qq = warp_sum(qq);
  if (lane == 0) {
    const float rq = rsqrtf(qq);
    const int id = (best > -INFINITY) ? best_k : 0;
    if (out_centroid) out_centroid[i] = id;
    if (out_expert) out_expert[i] = cmap ? cmap[id] : id;
    if (out_second) out_second[i] = (second > -INFINITY) ? second_k : -1;
    if (out_best) out_best[i] = (best > -INFINITY) ? best * rq : -INFINITY;
    if (out_margin) out_margin[i] = (second > -INFINITY) ? (best - second) * rq : INFINITY;
  }
}

// Finishing pass of the tensor-core top-2 router: unpack both keys, divide by |q|.  One warp per query.
__global__ void __launch_bounds__(256)
route_finish_top2_kernel(const unsigned long long* __restrict__ keys, const unsigned long long* __restrict__ keys2,
                         const __nv_bfloat16* __restrict__ q, const int* __restrict__ cmap, int Q, int D,
                         int* __restrict__ out_expert, int* __restrict__ out_centroid, int* __restrict__ out_second,
                         float* __restrict__ out_best, float* __restrict__ out_margin) {
  pdl_begin();
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= Q) return;
  const unsigned long long k1 = keys[i], k2 = keys2[i];
  float ss = 0.f;
  for (int ch = lane; ch < D / 8; ch += 32) {
    const uint4 v = ldg_cached(q + (size_t)i * D + ch * 8);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      ss = fmaf(bf16_lo(w[e]), bf16_lo(w[e]), ss);
      ss = fmaf(bf16_hi(w[e]), bf16_hi(w[e]), ss);
    }
  }
  ss = warp_sum(ss);
  if (lane == 0) {
    const float rq = rsqrtf(ss);
    const int id = (k1 == 0ull) ? 0 : (int)(0xFFFFFFFFu - (uint32_t)(k1 & 0xFFFFFFFFull));
    const float s1 = key_to_float((uint32_t)(k1 >> 32)), s2 = key_to_float((uint32_t)(k2 >> 32));
    if (out_centroid) out_centroid[i] = id;
    if (out_expert) out_expert[i] = cmap ? cmap[id] : id;
    if (out_second) out_second[i] = (k2 == 0ull) ? -1 : (int)(0xFFFFFFFFu - (uint32_t)(k2 & 0xFFFFFFFFull));
    if (out_best) out_best[i] = (k1 == 0ull) ? -INFINITY : s1 * rq;
    if (out_margin) out_margin[i] = (k1 == 0ull || k2 == 0ull) ? INFINITY : (s1 - s2) * rq;
  }
}

cudaError_t launch_route_top2_simple(const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm,
                                     const int* cmap, int Q, int K, int D, int* out_expert, int* out_centroid,
                                     int* out_second, float* out_best, float* out_margin, cudaStream_t stream) {
  return launch_pdl(route_top2_simple_kernel, (Q + 7) / 8, 256, 0, stream, q, c, inv_norm, cmap, Q, K, D, out_expert,
                    out_centroid, out_second, out_best, out_margin);
}
cudaError_t launch_route_finish_top2(const unsigned long long* keys, const unsigned long long* keys2,
                                     const __nv_bfloat16* q, const int* cmap, int Q, int D, int* out_expert,
                                     int* out_centroid, int* out_second, float* out_best, float* out_margin,
                                     cudaStream_t stream) {
  launch_pdl(route_finish_top2_kernel, (Q + 7) / 8, 256, 0, stream, keys, keys2, q, cmap, Q, D, out_expert, out_centroid, out_second,
                                                           out_best, out_margin);
  return cudaGetLastError();
}

cudaError_t launch_inv_norm(const __nv_bfloat16* c, int K, int D, float* inv_norm, cudaStream_t stream) {
  launch_pdl(centroid_inv_norm_kernel, (K + 7) / 8, 256, 0, stream, c, K, D, inv_norm);
  return cudaGetLastError();
}

cudaError_t launch_route_simple(const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm,
                                const int* cmap, int Q, int K, int D, int* out_expert, int* out_centroid,
                                float* out_best, cudaStream_t stream) {
  const size_t smem = (size_t)kRouteQB * D * 2;
  cudaError_t ce = ensure_smem_optin(OPTIN_ROUTE_SIMPLE, route_simple_kernel, 8 * 8192 * 2);
  if (ce != cudaSuccess) return ce;
  return launch_pdl(route_simple_kernel, (Q + kRouteQB - 1) / kRouteQB, 128, smem, stream, q, c, inv_norm, cmap, Q, K, D,
                    out_expert, out_centroid, out_best);
}

// The same without the cosine output: nothing to reduce, so one thread per query (coalesced keys and ids).
__global__ void __launch_bounds__(256)
route_finish_ids_kernel(const unsigned long long* __restrict__ keys, const int* __restrict__ cmap, int Q,
                        int* __restrict__ out_expert, int* __restrict__ out_centroid) {
  pdl_begin();
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= Q) return;
  const unsigned long long key = keys[i];
  const int id = (key == 0ull) ? 0 : (int)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));
  if (out_centroid) out_centroid[i] = id;
  out_expert[i] = cmap ? cmap[id] : id;
}

// best[i] / |q_i| for the router without scratch, added up as in route_finish_kernel.
__global__ void __launch_bounds__(256)
route_cosine_kernel(const __nv_bfloat16* __restrict__ q, int Q, int D, float* __restrict__ best) {
  pdl_begin();
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= Q) return;
  float ss = 0.f;
  for (int ch = lane; ch < D / 8; ch += 32) add_sq8(ldg_cached(q + (size_t)i * D + ch * 8), ss);
  ss = warp_sum(ss);
  if (lane == 0 && best[i] > -INFINITY) best[i] *= rsqrtf(ss);
}
cudaError_t launch_route_cosine(const __nv_bfloat16* q, int Q, int D, float* out_best, cudaStream_t stream) {
  return launch_pdl(route_cosine_kernel, (unsigned)((Q + 7) / 8), 256, 0, stream, q, Q, D, out_best);
}

cudaError_t launch_route_finish(const unsigned long long* keys, const __nv_bfloat16* q, const int* cmap, int Q, int D,
                                int* out_expert, int* out_centroid, float* out_best, cudaStream_t stream) {
  if (out_best == nullptr)
    launch_pdl(route_finish_ids_kernel, (Q + 255) / 256, 256, 0, stream, keys, cmap, Q, out_expert, out_centroid);
  else
    launch_pdl(route_finish_kernel, (Q + 7) / 8, 256, 0, stream, keys, q, cmap, Q, D, out_expert, out_centroid, out_best);
  return cudaGetLastError();
}

}  // namespace moin
