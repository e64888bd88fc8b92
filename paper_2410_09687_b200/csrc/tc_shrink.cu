// Long-run LoRA shrink  h = s act(x A_e^T)  on tcgen05 / TMEM / TMA, stored as bf16 hi + lo parts.
//
// A work item is one row tile of the batch plan (a run of one expert, at most 128 rows) for a SET of projections that
// share x (a launch each): their adapters' rows stand side by side in the B operand, so x is read once.  The product is skinny (N = the
// set's ranks together), and its time is latency: 128 rows x K of x through one SM at a time.  The reduction is
// therefore cut over the `ks` CTAs of a cluster - as many as fill the GPU - and the parts meet in shared memory: every
// CTA of the cluster adds its share of the rows over the parts in rank order (independent of timing), applies the
// function, the scale and the slot's rank, and writes whole rows.
//   warp 0     TMA producer (one thread): [128 x 64] box of x, [r x 64] box of A per projection
//   warp 1     allocates TMEM, issues the MMAs (one elected lane)
//   warps 2-9  TMEM -> shared memory (row pitch N + 4 floats: no bank conflicts), two warps per lane quarter
// Against one CTA per row tile (calls of 3392 tokens in runs of 106, rank 64, to 256 columns, projection included):
// K = 2048 26.6 -> 23.2 us, K = 5632 52 -> 42 us, three projections 46.5 -> 32.7 us; 16384 tokens fill the SMs with one
// CTA per row tile and are bound by reading x (rank 16, K = 5632: 41 us, 28 us of them at the copy bandwidth).
#include <cuda.h>

#include "ptx.cuh"
#include "tc_gemm.cuh"

namespace moin {

constexpr int kTsThreads = 320, kTsM = 128, kTsK = 64, kTsMaxN = 256, kTsMaxStages = 8;

struct TsMaps { CUtensorMap x, a[kTcMaxShrinkJobs]; };
struct TsParams {
  int T, K, r, n_jobs, N;                   // N: the jobs' ranks together, a multiple of 16
  int stages, stage_bytes, tmem_cols, ks;
  const int *header, *tile_row0, *tile_rows, *tile_expert;
  const int* slot_of_expert[kTcMaxShrinkJobs];
  const int* slot_rank[kTcMaxShrinkJobs];   // nullable: the stored rank
  __nv_bfloat16* hb[kTcMaxShrinkJobs];      // [2][T][r]: hi, lo (rows without an adapter are not written)
  int act;
  float scale;
  DeviceStatus* status;
};

// Where a projection's h goes for the tile in hand.
struct TsOut { int slot, r_use; __nv_bfloat16* hb; };
__device__ __forceinline__ TsOut ts_out(const TsParams& p, const int (&slot)[kTcMaxShrinkJobs], int job) {
  TsOut o = {slot[0], p.r, p.hb[0]};
  const int* ranks = p.slot_rank[0];
#pragma unroll
  for (int j = 1; j < kTcMaxShrinkJobs; ++j)
    if (job == j) { o.slot = slot[j]; ranks = p.slot_rank[j]; o.hb = p.hb[j]; }
  if (ranks && o.slot >= 0) o.r_use = min(__ldg(ranks + o.slot), p.r);
  return o;
}
// Columns cj .. cj + 7 of row `row` of the job's h: function, scale, nothing beyond the adapter's rank, hi and lo parts.
__device__ __forceinline__ void ts_put(const TsParams& p, const TsOut& o, int row, int cj, float (&f)[8]) {
  if (p.act != MOIN_ACT_NONE) {
#pragma unroll
    for (int k = 0; k < 8; ++k) f[k] = lora_act(f[k], p.act);
  }
  const bool in = cj < o.r_use;   // (ranks are multiples of 8)
#pragma unroll
  for (int k = 0; k < 8; ++k) f[k] = in ? f[k] * p.scale : 0.f;
  uint4 h, l;
  h.x = pack_bf16(f[0], f[1]); h.y = pack_bf16(f[2], f[3]); h.z = pack_bf16(f[4], f[5]); h.w = pack_bf16(f[6], f[7]);
  l.x = pack_bf16(f[0] - bf16_lo(h.x), f[1] - bf16_hi(h.x));   // hi + lo carries the value to ~fp32 accuracy
  l.y = pack_bf16(f[2] - bf16_lo(h.y), f[3] - bf16_hi(h.y));
  l.z = pack_bf16(f[4] - bf16_lo(h.z), f[5] - bf16_hi(h.z));
  l.w = pack_bf16(f[6] - bf16_lo(h.w), f[7] - bf16_hi(h.w));
  __nv_bfloat16* dst = o.hb + (size_t)row * (size_t)p.r + cj;
  *reinterpret_cast<uint4*>(dst) = h;
  *reinterpret_cast<uint4*>(dst + (size_t)p.T * (size_t)p.r) = l;
}

__global__ void __launch_bounds__(kTsThreads, 1)
tc_shrink_kernel(const __grid_constant__ TsMaps maps, const __grid_constant__ TsParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t ring = (raw + 1023u) & ~1023u;
  const int S = p.stages;
  const uint32_t bars = ring + (uint32_t)S * (uint32_t)p.stage_bytes;
  uint8_t* bar_ptr = smem_raw + (bars - raw);
  const uint32_t full0 = bars, empty0 = bars + 8 * kTsMaxStages, done = bars + 16 * kTsMaxStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_ptr + 16 * kTsMaxStages + 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_ptr + 16 * kTsMaxStages + 16);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = p.ks > 1 ? (int)cluster_rank() : 0;
  const int cluster = (int)blockIdx.x / p.ks, n_clusters = (int)gridDim.x / p.ks;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_begin();   // (the set-up above overlaps the tail of the kernel before)

  // the first tile's entries together with the number of tiles (one round trip less; in bounds: no more clusters than tokens)
  int4 nxt = make_int4(__ldg(p.tile_row0 + cluster), __ldg(p.tile_rows + cluster), __ldg(p.tile_expert + cluster), 0);
  const int total = __ldg(p.header + PH_NTILES), N = p.N, pitch = N + 4;
  const int nkb = p.K / kTsK, kb0 = nkb * rank / p.ks, kb1 = nkb * (rank + 1) / p.ks;
  auto sync_cluster = [&]() {
    if (p.ks > 1) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  };
  uint32_t st = 0, ph = 0, n_done = 0;   // ring position and phase (of the producer and of the MMA warp)
  bool ok = true;
  for (int tm = cluster; tm < total; tm += n_clusters) {
    const int row0 = nxt.x, rows = nxt.y, e = nxt.z;
    if (tm + n_clusters < total)
      nxt = make_int4(__ldg(p.tile_row0 + tm + n_clusters), __ldg(p.tile_rows + tm + n_clusters), __ldg(p.tile_expert + tm + n_clusters), 0);
    int slot[kTcMaxShrinkJobs];
    bool any = false;
#pragma unroll
    for (int j = 0; j < kTcMaxShrinkJobs; ++j) {
      slot[j] = j < p.n_jobs && e >= 0 ? __ldg(p.slot_of_expert[j] + e) : -1;
      any = any || slot[j] >= 0;
    }
    if (!any) {   // no product; (the same for the whole cluster)
    } else if (warp == 0) {
      if (lane == 0) {
        const uint32_t tx = (uint32_t)(kTsM + p.n_jobs * p.r) * kTsK * 2;
        for (int kb = kb0; kb < kb1 && ok; ++kb) {
          if (!(ok = mbar_wait(empty0 + 8 * st, ph ^ 1u, abort_flag, p.status, 71))) break;
          const uint32_t sa = ring + st * p.stage_bytes, sb = sa + kTsM * kTsK * 2, full = full0 + 8 * st;
          if (++st == (uint32_t)S) { st = 0; ph ^= 1u; }
          mbar_expect_tx(full, tx);
          tma_load_2d(sa, &maps.x, full, kb * kTsK, row0);
#pragma unroll
          for (int j = 0; j < kTcMaxShrinkJobs; ++j)
            if (j < p.n_jobs)   // (a projection without this adapter loads slot 0: its columns are not stored)
              tma_load_2d(sb + (uint32_t)(j * p.r) * (kTsK * 2), &maps.a[j], full, kb * kTsK, max(slot[j], 0) * p.r);
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      const uint32_t idesc = idesc_bf16(kTsM, N);
      const bool leader = elect_one();
      for (int kb = kb0; kb < kb1 && ok; ++kb) {
        if (!(ok = mbar_wait_warp(full0 + 8 * st, ph, abort_flag, p.status, 72))) break;
        tc_fence_after();
        const uint32_t sa = ring + st * p.stage_bytes, empty = empty0 + 8 * st;
        if (++st == (uint32_t)S) { st = 0; ph ^= 1u; }
        const uint64_t da = sdesc_k128(sa), db = sdesc_k128(sa + kTsM * kTsK * 2);
        if (leader) {
#pragma unroll
          for (int k = 0; k < kTsK / 16; ++k)
            tc_mma_bf16(tmem, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, (kb > kb0 || k > 0) ? 1u : 0u);
          tc_commit(empty);
        }
      }
      if (ok && leader) tc_commit(done);
      __syncwarp();
    } else {
      // this CTA's part to shared memory (the ring is free: every stage has been consumed), [row][pitch] fp32
      if (ok && (ok = mbar_wait_warp(done, n_done & 1u, abort_flag, p.status, 73))) {
        tc_fence_after();
        const int q = warp & 3, wh = (warp - 2) >> 2;
        const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
        const uint32_t dst = ring + (uint32_t)((q * 32 + lane) * pitch) * 4u;
        for (int c = 16 * wh; c < N; c += 32) {
          uint32_t v[16];
          tmem_ld16(lanes + c, v);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; i += 4)
            asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(dst + 4u * (c + i)), "r"(v[i]), "r"(v[i + 1]), "r"(v[i + 2]),
                         "r"(v[i + 3]) : "memory");
        }
        tc_fence_before();
      }
    }
    if (any) {
      ++n_done;
      sync_cluster();
      // This CTA's share of the rows: eight columns of a row per lane, as many rows as fit a warp, so that a warp stores whole
      // lines and nothing is worked out anew for each piece.  (A division for every piece of a row: 64 x 256 tokens 18.5 /
      // 13.5 / 7 us of the launch for ranks of 192 / 128 / 64 together, now 3.6 / 2.3 / 2.6; a thread per row straight from
      // its accumulator 7 / 4.5 / 2.3.)  With parts of other CTAs it is bound by the reads through the cluster: one row a time.
      const int own = kTsM / p.ks, r8 = p.r / 8, per_row = p.n_jobs * r8, rpw = 32 / per_row;
      const int sub = lane / per_row, c8 = lane - sub * per_row, job = c8 >= 2 * r8 ? 2 : c8 >= r8 ? 1 : 0, cj = (c8 - job * r8) * 8;
      const TsOut o = ts_out(p, slot, job);
      const int end = min(own, rows - rank * own);
      if (sub < rpw && o.slot >= 0 && !*abort_flag) {
        for (int rr = warp * rpw + sub; rr < end; rr += rpw * (kTsThreads / 32)) {
          const uint32_t off = (uint32_t)((rank * own + rr) * pitch + c8 * 8) * 4u;
          float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
          auto add = [&](const float4& a, const float4& b) {
            f[0] += a.x; f[1] += a.y; f[2] += a.z; f[3] += a.w;
            f[4] += b.x; f[5] += b.y; f[6] += b.z; f[7] += b.w;
          };
          if (p.ks == 1) {
            add(lds_f4(ring + off), lds_f4(ring + off + 16));
          } else {
            for (int k0 = 0; k0 < p.ks; k0 += 4) {
              float4 va[4], vb[4];
#pragma unroll
              for (int k = 0; k < 4; ++k)
                if (k0 + k < p.ks) {
                  const uint32_t part = map_rank(ring, (uint32_t)(k0 + k)) + off;
                  va[k] = ld_cluster_f4(part);
                  vb[k] = ld_cluster_f4(part + 16);
                }
#pragma unroll
              for (int k = 0; k < 4; ++k)
                if (k0 + k < p.ks) add(va[k], vb[k]);
            }
          }
          ts_put(p, o, row0 + rank * own + rr, cj, f);
        }
      }
      // the parts have been read everywhere: the next item's copies may overwrite them
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      sync_cluster();
    }
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

// One set: projections of one K, rank and activation that share x, ranks together at most 256.
static moin_status launch_set(HostState* hs, const PlanView& pv, const moin_pool* const* pools, const __nv_bfloat16* x,
                              __nv_bfloat16* const* hbs, int n_jobs, float scale, cudaStream_t stream) {
  const int T = pv.T, K = pools[0]->d_in, r = pools[0]->r;
  TsMaps maps;
  TsParams p = {};
  p.T = T; p.K = K; p.r = r; p.n_jobs = n_jobs; p.N = (n_jobs * r + 15) / 16 * 16;
  p.scale = scale; p.act = pools[0]->activation; p.status = hs->status;
  p.header = pv.header; p.tile_row0 = pv.tile_row0; p.tile_rows = pv.tile_rows; p.tile_expert = pv.tile_expert;
  moin_status st = make_map(&maps.x, x, T, K, kTsM);
  for (int j = 0; j < n_jobs && !st; ++j) {
    st = make_map(&maps.a[j], pools[j]->A, (uint64_t)pools[j]->n_slots * r, K, r);   // one slot's rows
    p.slot_of_expert[j] = pools[j]->slot_of_expert;
    p.slot_rank[j] = pools[j]->slot_rank;
    p.hb[j] = hbs[j];
  }
  if (st) return st;
  // the ring is also the fp32 staging of the parts
  p.stage_bytes = (kTsM + p.N) * kTsK * 2;
  p.stages = 200 * 1024 / p.stage_bytes < kTsMaxStages ? 200 * 1024 / p.stage_bytes : kTsMaxStages;
  while (p.stages * p.stage_bytes < kTsM * (p.N + 4) * 4) ++p.stages;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.N) p.tmem_cols *= 2;
  // Cut the reduction while the row tiles leave SMs free and a CTA keeps at least four 64-wide blocks; clusters of eight
  // only for a handful of tiles (a GPC holds few of them).
  const long items = (T + kTsM - 1) / kTsM;
  const int ks_max = items <= 12 ? 8 : 4;
  p.ks = 1;
  while (p.ks < ks_max && items * p.ks * 2 <= hs->n_sms && K / kTsK >= 4 * p.ks * 2) p.ks *= 2;
  long clusters = hs->n_sms / p.ks;
  if (clusters > T) clusters = T;   // (at most one row tile per token)
  const size_t smem = (size_t)p.stages * p.stage_bytes + 1024 /*align*/ + 256 /*barriers*/;
  cudaError_t e = ensure_smem_optin(OPTIN_TC_SHRINK, tc_shrink_kernel, 210 * 1024);
  if (e != cudaSuccess) return record_cuda(e);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * p.ks));
  cfg.blockDim = dim3(kTsThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)p.ks;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  ProfScope prof(MOIN_K_SHRINK_TC, 1, stream);
  return record_cuda(cudaLaunchKernelEx(&cfg, tc_shrink_kernel, maps, p));
}

moin_status launch_tc_shrink_group(HostState* hs, const PlanView& pv, const moin_pool* const* pools,
                                   const __nv_bfloat16* const* xs, __nv_bfloat16* const* hbs, int n_jobs, float scale,
                                   cudaStream_t stream) {
  if (n_jobs < 1 || n_jobs > kTcMaxShrinkJobs) return MOIN_ERR_INVALID_ARG;
  for (int j0 = 0; j0 < n_jobs;) {
    int n = 1;
    while (j0 + n < n_jobs && xs[j0 + n] == xs[j0] && (n + 1) * pools[j0]->r <= kTsMaxN) ++n;
    moin_status st = launch_set(hs, pv, pools + j0, xs[j0], hbs + j0, n, scale, stream);
    if (st) return st;
    j0 += n;
  }
  return MOIN_OK;
}

}  // namespace moin
