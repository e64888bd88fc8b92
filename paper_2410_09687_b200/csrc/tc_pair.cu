// Long-run GEMMs on CTA pairs: tcgen05 with cta_group::2, sm_100a.
//
// Two CTAs on neighbouring SMs work on one [256 x BN] tile of  A[M,K] B[N,K]^T : each holds 128 rows of A, HALF of the
// B rows and 128 rows of the accumulator, and the first CTA issues the MMAs for both.  Why pairs: an SM receives about
// 64 bytes per clock from L2.  A single-CTA 128 x 256 tile needs 48 KB per 64-wide k-block (96 bytes per clock at the
// tensor rate, so two thirds of it at best); in a pair the same MMA work needs 32 KB per SM, which the fill rate covers.
//
// Roles per CTA: warp 0 TMA producer (its own A rows and its half of B; completion of both CTAs' copies is counted on
// the FIRST CTA's barrier), warp 1 TMEM allocation and - first CTA only - MMA issue, warps 2-9 epilogue of the CTA's
// own 128 rows.  A commit arrives on both CTAs' barriers (stage free, accumulator ready); both epilogues release an
// accumulator on the first CTA's barrier.  Two accumulators in TMEM: the epilogue of tile i overlaps the MMAs of i + 1.
//
// Row tiles are the regular grid of 128 rows, also with a batch plan: a tile may hold up to kTileRuns runs of one expert
// (the plan cuts a grid tile of more).  With adapters every tile ends with extra K blocks [hi(s h) | lo(s h)] x
// [B_e ; B_e], one pass per run, that add the low-rank term inside the accumulator; a pass's MMAs leave out the
// accumulator rows of the other runs (disable-output-lane), whatever lies in their h and whatever B_e holds: an adapter
// with an infinity or a NaN in it spoils the rows of its own run only.  Tiles that began anew with each
// run instead multiplied up to a fifth of padding: 11 prompts of 65 to 600 tokens, forward 10.34 -> 8.98 ms; nine, a
// block's projections 464 -> 400 us.
//
// A launch covers up to kPairJobs projections that share the plan and the reduction length (the column tiles of all of
// them side by side under one row tile, so an x they share comes from L2): one ramp and one partial last wave per group.
// Every wait on an mbarrier is bounded; on expiry the kernel raises the status flag and returns.
#include <cuda.h>
#include <float.h>

#include "tc_gemm.cuh"
#include "ptx.cuh"

namespace moin {

constexpr int kPairThreads = 320, kPairM = 128, kPairK = 64;
// PAIR_ROUTER_ROWS: a pair takes all column tiles of its rows and so needs no keys to meet in (see launch_pair_router_rows)
enum { PAIR_STORE = 0, PAIR_ROUTER = 1, PAIR_ROUTER2 = 2, PAIR_SWIGLU = 3, PAIR_ROUTER_ROWS = 4 };

struct PairMaps { CUtensorMap x[kPairJobs], w[kPairJobs], b[kPairJobs], h[kPairJobs], y[kPairJobs]; };
struct PairParams {
  int M, K, n_jobs, bn, cols;            // bn: tile width, a multiple of 16 up to 256; cols: output columns of it
  int N[kPairJobs], tn_end[kPairJobs];   // columns, column tiles of jobs 0 .. j
  const int *header, *run_expert, *run_row0;   // plan (header == nullptr: regular grid over M, no runs)
  const int4* gemm_tab;
  int tail_r;                            // stored rank of the appended low-rank blocks (0 = none)
  const int* slot_of_expert[kPairJobs];
  const int* slot_rank[kPairJobs];       // nullable: the stored rank
  __nv_bfloat16* y[kPairJobs];
  float* y0[kPairJobs];                  // fp32 copy, nullable (then the rows are written straight from registers)
  const float* inv_norm;                 // PAIR_ROUTER*
  unsigned long long *keys, *keys2;
  const int* cmap;                       // PAIR_ROUTER_ROWS: outputs, the cosine still to be divided by |q|
  int *out_expert, *out_centroid;
  float* out_best;
  DeviceStatus* status;
};

constexpr int kPairMaxN = 256, kPairStageBytes = (kPairM + kPairMaxN / 2) * kPairK * 2, kPairStages = 6;
constexpr int kPairOutBytes = 8 * 32 * 128;   // epilogue staging: [32 rows x 64 columns] bf16 per warp
constexpr size_t kPairSmem = (size_t)kPairStages * kPairStageBytes + 1024 /*align*/ + 1024 /*barriers*/ + kPairOutBytes;

// What a tile is: its job, first column, and for both CTAs of the pair the rows and the runs in them.
struct PairTile { int job, n0, row0[2], rows[2], run0[2], n_run[2]; };

__device__ __forceinline__ PairTile pair_tile(const PairParams& p, int tile, int tiles_m) {
  PairTile t;
  const int tn_all = p.tn_end[p.n_jobs - 1];
  const int pm = tile / tn_all;
  int tn = tile - pm * tn_all;
  t.job = 0;
#pragma unroll
  for (int j = 0; j + 1 < kPairJobs; ++j)
    if (j + 1 < p.n_jobs && tn >= p.tn_end[j]) t.job = j + 1;
  int first = 0;
#pragma unroll
  for (int j = 1; j < kPairJobs; ++j)
    if (t.job == j) first = p.tn_end[j - 1];
  t.n0 = (tn - first) * p.cols;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int tm = 2 * pm + c;
    int4 g = make_int4(p.M, 0, 0, 0);   // no such row tile: the copy fills zeros, nothing is stored
    if (tm < tiles_m) {
      if (p.header != nullptr) g = __ldg(p.gemm_tab + tm);
      else g = make_int4(tm * kPairM, min(kPairM, p.M - tm * kPairM), 0, 0);
    }
    t.row0[c] = g.x; t.rows[c] = g.y; t.run0[c] = g.z; t.n_run[c] = g.w;
  }
  return t;
}
// Low-rank passes of a tile: one per run of the first CTA's rows, then the second's; the run in which both meet takes one
// pass for both.  Finding a pass's adapter is a chain of three loads: an epilogue warp does it a tile ahead, lane i for
// pass i (SWIGLU: lanes 8 .. 15 for the up projection), and leaves the result in shared memory.  (In the producer and the
// MMA warp themselves, at the start of a tile or in steps between the quarters of its main loop, it cost 2 to 5 percent.)
constexpr int kPairPasses = 2 * kTileRuns;
// What the passes leave out stands there word for word as the MMAs take it.
struct PairTable {
  struct { int slot, rank; } pass[2 * kPairPasses];   // adapter or -1, its rank
  uint32_t out[kPairPasses][8];                       // accumulator rows of other runs, first CTA's then second's
  int n, has[2], pad;                                 // passes; bit i: the CTA has rows of pass i's run
};
// disable-output-lane word of 32 accumulator rows of which first .. end - 1 (counted from the word's first row) take part
__device__ __forceinline__ uint32_t lanes_out(int first, int end) {
  const uint32_t below_end = end <= 0 ? 0u : end >= 32 ? ~0u : (1u << end) - 1u;
  const uint32_t below_first = first <= 0 ? 0u : first >= 32 ? ~0u : (1u << first) - 1u;
  return ~(below_end & ~below_first);
}
__device__ __forceinline__ void pair_passes(const PairParams& p, const PairTile& t, bool two_jobs, int lane, PairTable* tab) {
  const int shared = t.n_run[0] > 0 && t.n_run[1] > 0 && t.run0[0] + t.n_run[0] - 1 == t.run0[1];
  const int n = t.n_run[0] + t.n_run[1] - shared;
  const int i = lane % kPairPasses, job = two_jobs ? lane / kPairPasses : t.job;
  const int run = i < t.n_run[0] ? t.run0[0] + i : t.run0[1] + i - t.n_run[0] + shared;
  bool has = false;
  if (lane < (two_jobs ? 2 : 1) * kPairPasses && i < n) {
    int slot = -1, rank = p.tail_r;
    const int* slots = p.slot_of_expert[0];
    const int* ranks = p.slot_rank[0];
#pragma unroll
    for (int j = 1; j < kPairJobs; ++j)
      if (job == j) { slots = p.slot_of_expert[j]; ranks = p.slot_rank[j]; }
    const int e = __ldg(p.run_expert + run);
    if (e >= 0) slot = __ldg(slots + e);
    if (slot >= 0 && ranks) rank = min(__ldg(ranks + slot), p.tail_r);
    tab->pass[lane].slot = slot;
    tab->pass[lane].rank = rank;
  } else if (lane >= 2 * kPairPasses && i < n) {   // lanes 16 .. 23: the first CTA's rows, 24 .. 31: the second's
    const int c = lane >= 3 * kPairPasses;
    const int row0 = c ? t.row0[1] : t.row0[0], rows = c ? t.rows[1] : t.rows[0];
    const int first = __ldg(p.run_row0 + run) - row0, end = min(__ldg(p.run_row0 + run + 1) - row0, rows);
#pragma unroll
    for (int w = 0; w < 4; ++w) tab->out[i][4 * c + w] = lanes_out(first - 32 * w, end - 32 * w);
    has = first < rows && end > 0;
  }
  const uint32_t in = __ballot_sync(0xffffffffu, has);
  if (lane == 0) {
    tab->n = n;
    tab->has[0] = (int)(in >> (2 * kPairPasses)) & ((1 << kPairPasses) - 1);
    tab->has[1] = (int)(in >> (3 * kPairPasses));
  }
}

// g / (1 + e^-g) without a branch: the quotient by an approximate reciprocal (good to its last place, also where it is
// subnormal), corrected by its own remainder (Markstein's method), which leaves half a last place and a rounding error of
// 2^-45 or so.  A divisor that overflowed gives -0, infinities and NaN what a division gives.  The division operator's
// branch to its exceptional cases kept the elements of a row from being worked on side by side: gate / up launch of 9
// requests of 116 to 464 tokens 103.3 us with it, 96.7 so.  (For bf16 gates the same bits but for the sign of a zero.)
__device__ __forceinline__ float pair_silu(float g) {
  const float d = 1.f + __expf(-g);
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(d));
  const float q = g * r, rest = fmaf(-q, fminf(d, FLT_MAX), g);
  return fmaf(fabsf(g) < INFINITY ? rest : 0.f, r, q);
}

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
tc_pair_kernel(const __grid_constant__ PairMaps maps, const PairParams p) {
  constexpr int S = kPairStages;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t ring = (raw + 1023u) & ~1023u;
  const uint32_t out0 = ring + (uint32_t)S * kPairStageBytes;   // 1024-byte aligned: the swizzle is a function of the address
  const uint32_t bars = out0 + kPairOutBytes;
  uint8_t* bar_ptr = smem_raw + (bars - raw);
  const uint32_t full0 = bars, empty0 = bars + 8 * S, tfull0 = bars + 16 * S, tempty0 = tfull0 + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_ptr + 16 * S + 32);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_ptr + 16 * S + 40);
  constexpr bool kTail = EPI == PAIR_STORE || EPI == PAIR_SWIGLU;   // low-rank blocks at the end of a tile
  // pass tables of this and the next tile, their barriers: written, and read to the end by this CTA's producer
  const uint32_t tab0 = bars + 16 * S + 48, tabread0 = tab0 + 16;
  PairTable* tabs = reinterpret_cast<PairTable*>(bar_ptr + 192);
  static_assert(16 * S + 80 <= 192 && 192 + 2 * sizeof(PairTable) <= 1024 && sizeof(PairTable) % 16 == 0, "barrier block");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full0 + 8 * s, 1);     // used in the first CTA: its producer's arrival plus both CTAs' bytes
      mbar_init(empty0 + 8 * s, 1);    // each CTA's own, by commit
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull0 + 8 * a, 1);    // each CTA's own, by commit
      mbar_init(tempty0 + 8 * a, 16);  // used in the first CTA: one arrival per epilogue warp of the pair
      mbar_init(tab0 + 8 * a, 1);
      mbar_init(tabread0 + 8 * a, 1);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(tmem_slot), 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_arrive();   // the other CTA's barriers exist before anything is signalled there
  cluster_wait();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_begin();   // (the set-up above overlaps the tail of the kernel before)

  const int tiles_m = p.header != nullptr ? p.header[PH_NGEMM] : (p.M + kPairM - 1) / kPairM;
  const int total = (tiles_m + 1) / 2 * p.tn_end[p.n_jobs - 1];
  const int nkb_main = (p.K + kPairK - 1) / kPairK;
  const int nrb = (p.tail_r + kPairK - 1) / kPairK;   // 64-wide blocks of the rank
  const int pair = (int)blockIdx.x >> 1, n_pairs = (int)gridDim.x >> 1;
  const int tn_all = p.tn_end[p.n_jobs - 1];
  const int tile_first = EPI == PAIR_ROUTER_ROWS ? pair * tn_all : pair;
  auto next_tile = [&](int tile) {
    if (EPI != PAIR_ROUTER_ROWS) return tile + n_pairs;
    return (tile + 1) % tn_all ? tile + 1 : tile + 1 + (n_pairs - 1) * tn_all;
  };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      // both CTAs' copies of a stage: the operands, the low-rank blocks (SWIGLU: of half the columns at a time)
      const uint32_t tx = (uint32_t)(2 * kPairM + p.bn) * kPairK * 2;
      const uint32_t tx_tail = EPI == PAIR_SWIGLU ? (uint32_t)(2 * kPairM + p.bn / 2) * kPairK * 2 : tx;
      uint32_t it = 0, lt = 0;
      bool ok = true;
      for (int tile = tile_first; tile < total && ok; tile = next_tile(tile), ++lt) {
        const PairTile t = pair_tile(p, tile, tiles_m);
        const int row0 = rank == 0 ? t.row0[0] : t.row0[1];
        const CUtensorMap* mx = &maps.x[t.job];
        const CUtensorMap* mw = &maps.w[EPI == PAIR_SWIGLU ? (int)rank : t.job];
        const int w0 = EPI == PAIR_SWIGLU ? t.n0 : t.n0 + (int)rank * (p.bn / 2);
        for (int kb = 0; kb < nkb_main; ++kb, ++it) {
          const uint32_t s = it % S, ph = (it / S) & 1u;
          if (!(ok = mbar_wait(empty0 + 8 * s, ph ^ 1u, abort_flag, p.status, 61))) break;
          const uint32_t sa = ring + s * kPairStageBytes, sb = sa + kPairM * kPairK * 2;
          const uint32_t bar = map_rank(full0 + 8 * s, 0);
          if (rank == 0) mbar_expect_tx(full0 + 8 * s, tx);
          tma_load_2d_pair(sa, mx, bar, kb * kPairK, row0);
          tma_load_2d_pair(sb, mw, bar, kb * kPairK, w0);
        }
        if (!kTail || p.tail_r == 0 || !ok) continue;
        if (!(ok = mbar_wait(tab0 + 8 * (lt & 1u), (lt >> 1) & 1u, abort_flag, p.status, 65))) break;
        const volatile PairTable* tab = tabs + (lt & 1u);
        const int n_pass = tab->n, has = tab->has[rank];
        for (int g = 0; g < (EPI == PAIR_SWIGLU ? 2 : 1) && ok; ++g) {
          const int job = EPI == PAIR_SWIGLU ? g : t.job;
          int n = p.N[0];
#pragma unroll
          for (int jj = 1; jj < kPairJobs; ++jj)
            if (job == jj) n = p.N[jj];
          for (int i = 0; i < n_pass && ok; ++i) {
            const int slot = tab->pass[g * kPairPasses + i].slot;
            if (slot < 0) continue;
            const int b0 = slot * n + t.n0 + (int)rank * (p.cols / 2);
            for (int j = 0; j < 2 * nrb; ++j, ++it) {
              const uint32_t s = it % S, ph = (it / S) & 1u;
              if (!(ok = mbar_wait(empty0 + 8 * s, ph ^ 1u, abort_flag, p.status, 61))) break;
              const uint32_t sa = ring + s * kPairStageBytes, sb = sa + kPairM * kPairK * 2;
              const uint32_t bar = map_rank(full0 + 8 * s, 0);
              if (rank == 0) mbar_expect_tx(full0 + 8 * s, tx_tail);
              const int lo = j >= nrb ? 1 : 0, rb = j - lo * nrb;   // hi blocks first, then lo blocks
              // all rows of the tile: the MMAs choose; a CTA without any of the run's starts past the last: nothing is read
              // (14 prompts of 202 to 262 tokens, rank 8, gate/up launch 121 us when it reads them, 117 so)
              tma_load_2d_pair(sa, &maps.h[job], bar, rb * kPairK, (has >> i) & 1 ? lo * p.M + row0 : 2 * p.M);
              tma_load_2d_pair(sb, &maps.b[job], bar, rb * kPairK, b0);
            }
          }
        }
        if (ok) mbar_arrive(tabread0 + 8 * (lt & 1u));
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (first CTA, for both)
    if (rank == 0) {   // the whole warp walks the loop, one elected lane issues (see elect_one)
      const uint32_t idesc = idesc_bf16(2 * kPairM, p.bn);
      const uint32_t idesc_tail = EPI == PAIR_SWIGLU ? idesc_bf16(2 * kPairM, p.bn / 2) : idesc;
      const bool leader = elect_one();
      uint32_t it = 0, lt = 0;
      bool ok = true;
      for (int tile = tile_first; tile < total && ok; tile = next_tile(tile), ++lt) {
        const uint32_t acc = lt & 1u, aph = (lt >> 1) & 1u;
        if (!(ok = mbar_wait_cluster_warp(tempty0 + 8 * acc, aph ^ 1u, abort_flag, p.status, 62))) break;
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + acc * kPairMaxN;
        for (int kb = 0; kb < nkb_main; ++kb, ++it) {
          const uint32_t s = it % S, ph = (it / S) & 1u;
          if (!(ok = mbar_wait_cluster_warp(full0 + 8 * s, ph, abort_flag, p.status, 63))) break;
          tc_fence_after();
          const uint32_t sa = ring + s * kPairStageBytes, sb = sa + kPairM * kPairK * 2;
          const uint64_t da = sdesc_k128(sa), db = sdesc_k128(sb);
          const int nk16 = (min(kPairK, p.K - kb * kPairK) + 15) / 16;
          if (leader) {
            if (nk16 == 4) {
#pragma unroll
              for (int k = 0; k < 4; ++k)
                tc_mma_bf16_pair(tmem_d, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, (kb > 0 || k > 0) ? 1u : 0u);
            } else {
              for (int k = 0; k < nk16; ++k)
                tc_mma_bf16_pair(tmem_d, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, (kb > 0 || k > 0) ? 1u : 0u);
            }
            tc_commit_pair(empty0 + 8 * s);
          }
        }
        if (kTail && p.tail_r > 0 && ok) {
          if (!(ok = mbar_wait_warp(tab0 + 8 * (lt & 1u), (lt >> 1) & 1u, abort_flag, p.status, 66))) break;
          const volatile PairTable* tab = tabs + (lt & 1u);
          const int n_pass = tab->n;
          for (int g = 0; g < (EPI == PAIR_SWIGLU ? 2 : 1) && ok; ++g) {
            const uint32_t tmem_g = tmem_d + g * (p.bn / 2);
            for (int i = 0; i < n_pass && ok; ++i) {
              const int slot = tab->pass[g * kPairPasses + i].slot, rk = tab->pass[g * kPairPasses + i].rank;
              if (slot < 0) continue;
              const uint32_t words = bars + 192 + (lt & 1u) * (uint32_t)sizeof(PairTable) + (uint32_t)offsetof(PairTable, out) + 32u * i;
              const uint4 first = lds_u4(words), second = lds_u4(words + 16);
              const uint32_t out[8] = {first.x, first.y, first.z, first.w, second.x, second.y, second.z, second.w};
              for (int j = 0; j < 2 * nrb; ++j, ++it) {
                const uint32_t s = it % S, ph = (it / S) & 1u;
                if (!(ok = mbar_wait_cluster_warp(full0 + 8 * s, ph, abort_flag, p.status, 63))) break;
                tc_fence_after();
                const uint32_t sa = ring + s * kPairStageBytes, sb = sa + kPairM * kPairK * 2;
                const uint64_t da = sdesc_k128(sa), db = sdesc_k128(sb);
                const int rb = j >= nrb ? j - nrb : j;
                const int nk16 = (min(kPairK, rk - rb * kPairK) + 15) / 16;   // beyond the rank: no MMA
                if (leader) {
                  for (int k = 0; k < nk16; ++k)
                    tc_mma_bf16_pair_rows(tmem_g, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc_tail, out);
                  tc_commit_pair(empty0 + 8 * s);
                }
              }
            }
          }
        }
        __syncwarp();   // every lane has read the tile's passes
        if (ok && leader) tc_commit_pair(tfull0 + 8 * acc);
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9), this CTA's 128 rows
    const int q = warp & 3;             // TMEM lane quarter this warp may read
    const int trow = q * 32 + lane;     // row of the tile owned by this thread
    const int wh = (warp - 2) >> 2;     // two warps per quarter, every other 64 columns each
    const uint32_t buf = out0 + (uint32_t)(wh * 4 + q) * 4096u;
    uint32_t lt = 0, n_st = 0;
    unsigned long long row_key = 0ull;   // PAIR_ROUTER_ROWS: of this thread's row, over the column tiles so far
    bool ok = true;
    // Passes of tile i into table i & 1.  The readers of tile i - 2's passes there are through: the MMA warp, whose
    // reads come before the commit of the accumulator that this warp has waited for, and the producer, whose last entries
    // may be passes without an adapter, which no copy and so no accumulator depends on: it says when it has read them.
    auto scout = [&](const PairTile& n, uint32_t i) -> bool {
      if (!mbar_wait_warp(tabread0 + 8 * (i & 1u), ((i >> 1) & 1u) ^ 1u, abort_flag, p.status, 67)) return false;
      pair_passes(p, n, EPI == PAIR_SWIGLU, lane, tabs + (i & 1u));
      __syncwarp();
      if (lane == 0) mbar_arrive(tab0 + 8 * (i & 1u));
      return true;
    };
    if (kTail && warp == 2 && p.tail_r > 0 && pair < total) ok = scout(pair_tile(p, pair, tiles_m), 0);
    for (int tile = tile_first; tile < total && ok; tile = next_tile(tile), ++lt) {
      const PairTile t = pair_tile(p, tile, tiles_m);
      if (kTail && warp == 2 && p.tail_r > 0 && tile + n_pairs < total &&
          !(ok = scout(pair_tile(p, tile + n_pairs, tiles_m), lt + 1))) break;
      const int row0 = rank == 0 ? t.row0[0] : t.row0[1], rows = rank == 0 ? t.rows[0] : t.rows[1];
      int n = p.N[0];
      __nv_bfloat16* y = p.y[0];
      float* y0 = p.y0[0];
#pragma unroll
      for (int j = 1; j < kPairJobs; ++j)
        if (t.job == j) { n = p.N[j]; y = p.y[j]; y0 = p.y0[j]; }
      const uint32_t acc = lt & 1u, aph = (lt >> 1) & 1u;
      // 1/|c_k| of the columns of half h; NaN where there is no candidate: it loses every maximum
      auto stage_norms = [&](int h) {
        const int k0 = t.n0 + h * (p.bn / 2) + 4 * lane;
        float4 v;
        float* e = reinterpret_cast<float*>(&v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float inv = (4 * lane < p.bn / 2 && k0 + i < n) ? __ldg(p.inv_norm + k0 + i) : 0.f;
          e[i] = inv > 0.f ? inv : __int_as_float(0x7FC00000);
        }
        __syncwarp();   // the other lanes have read the last values
        *reinterpret_cast<float4*>(smem_raw + (buf - raw) + 16 * lane) = v;
        __syncwarp();
      };
      if (EPI == PAIR_ROUTER || EPI == PAIR_ROUTER2) stage_norms(wh);
      if (!(ok = mbar_wait_warp(tfull0 + 8 * acc, aph, abort_flag, p.status, 64))) break;
      tc_fence_after();
      const bool row_ok = trow < rows;
      const size_t grow = (size_t)(row0 + trow);
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + acc * kPairMaxN;
      float best = -INFINITY, second = -INFINITY;
      int best_k = 0, second_k = 0;
      auto release = [&]() {   // the accumulator has been read
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_rank(tempty0 + 8 * acc, 0));
      };
      auto row_best = [&](int h, bool last) {   // best (and second) score of this thread's row among the columns of half h
        // The row's (up to) 128 scores go to registers at once, which frees the accumulator; then the maximum (two
        // columns per instruction) and the first column that holds it.  A running (maximum, index) pair column by
        // column takes eight instructions a column and bounded the launch: 65536 x 5000 x 768 400 us with 128 x 256 tiles
        // of single CTAs, 455 us with pairs, now 305 us alone (1.65 PFLOP/s) and 365 us in a loop at the power limit.
        uint32_t f[4][32];
#pragma unroll
        for (int g = 0; g < 4; ++g)
          if (32 * g < p.bn / 2) tmem_ld32(taddr + h * (p.bn / 2) + 32 * g, f[g]);
        tmem_ld_wait();
        if (last) release();
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if (32 * g < p.bn / 2) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
              const float4 inv = lds_f4(buf + 4u * (32 * g + j));
              const float f0 = __uint_as_float(f[g][j]) * inv.x, f1 = __uint_as_float(f[g][j + 1]) * inv.y;
              const float f2 = __uint_as_float(f[g][j + 2]) * inv.z, f3 = __uint_as_float(f[g][j + 3]) * inv.w;
              best = fmax3(best, fmax3(f0, f1, f2), f3);
              f[g][j] = __float_as_uint(f0); f[g][j + 1] = __float_as_uint(f1);
              f[g][j + 2] = __float_as_uint(f2); f[g][j + 3] = __float_as_uint(f3);
            }
          }
        }
#pragma unroll
        for (int g = 3; g >= 0; --g) {
          if (32 * g < p.bn / 2) {
#pragma unroll
            for (int j = 31; j >= 0; --j) best_k = (__uint_as_float(f[g][j]) == best) ? 32 * g + j : best_k;   // lowest index wins
          }
        }
        if (EPI == PAIR_ROUTER2) {   // the same once more without the winner
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            if (32 * g < p.bn / 2) {
#pragma unroll
              for (int j = 0; j < 32; j += 2) {
                if (32 * g + j == best_k) f[g][j] = 0x7FC00000u;
                if (32 * g + j + 1 == best_k) f[g][j + 1] = 0x7FC00000u;
                second = fmax3(second, __uint_as_float(f[g][j]), __uint_as_float(f[g][j + 1]));
              }
            }
          }
#pragma unroll
          for (int g = 3; g >= 0; --g) {
            if (32 * g < p.bn / 2) {
#pragma unroll
              for (int j = 31; j >= 0; --j) second_k = (__uint_as_float(f[g][j]) == second) ? 32 * g + j : second_k;
            }
          }
          second_k += t.n0 + h * (p.bn / 2);
        }
        best_k += t.n0 + h * (p.bn / 2);
      };
      if (EPI == PAIR_STORE || EPI == PAIR_SWIGLU) {
        // Full 32-row groups leave through shared memory (128-byte swizzled rows) as tiled stores of whole lines: a
        // warp's 16-byte pieces straight from registers are 32 partial-line requests per instruction, beside the
        // operand loads in L2.  Partial row groups of a plan tile and the rest of a tile
        // whose width is no multiple of 64 are written row by row (a tiled store cannot be clipped).
        const int col_end = min(n, t.n0 + p.cols);
#pragma unroll 1
        for (int c = 64 * wh; c < p.cols; c += 128) {
          if (t.n0 + c >= n || q * 32 >= rows) break;
          const bool staged = q * 32 + 32 <= rows && c + 64 <= p.cols && y0 == nullptr;
          if (staged && n_st >= 1) {               // the store that last read this buffer
            if (lane == 0) bulk_wait_read<0>();
            __syncwarp();
          }
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            uint32_t v[32];
            tmem_ld32(taddr + c + 32 * hh, v);
            if (EPI == PAIR_SWIGLU) {   // silu(gate) * up, both rounded to bf16 first as the separate projections are
              uint32_t u[32];
              tmem_ld32(taddr + p.cols + c + 32 * hh, u);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 32; j += 2) {
                const uint32_t gw = pack_bf16(__uint_as_float(v[j]), __uint_as_float(v[j + 1]));
                const uint32_t uw = pack_bf16(__uint_as_float(u[j]), __uint_as_float(u[j + 1]));
                const float g0 = bf16_lo(gw), g1 = bf16_hi(gw);
                v[j] = __float_as_uint(pair_silu(g0) * bf16_lo(uw));
                v[j + 1] = __float_as_uint(pair_silu(g1) * bf16_hi(uw));
              }
            } else {
              tmem_ld_wait();
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              uint4 o;
              o.x = pack_bf16(__uint_as_float(v[8 * j]), __uint_as_float(v[8 * j + 1]));
              o.y = pack_bf16(__uint_as_float(v[8 * j + 2]), __uint_as_float(v[8 * j + 3]));
              o.z = pack_bf16(__uint_as_float(v[8 * j + 4]), __uint_as_float(v[8 * j + 5]));
              o.w = pack_bf16(__uint_as_float(v[8 * j + 6]), __uint_as_float(v[8 * j + 7]));
              const int col = t.n0 + c + 32 * hh + 8 * j;      // N is a multiple of 8
              if (staged) {
                const uint32_t dst = buf + (uint32_t)lane * 128u + ((uint32_t)((4 * hh + j) ^ (lane & 7)) << 4);
                asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(o.x), "r"(o.y), "r"(o.z), "r"(o.w) : "memory");
              } else if (row_ok && col < col_end) {
                *reinterpret_cast<uint4*>(y + grow * (size_t)n + col) = o;
                if (y0 != nullptr) {
                  uint4* d0 = reinterpret_cast<uint4*>(y0 + grow * (size_t)n + col);
                  d0[0] = make_uint4(v[8 * j], v[8 * j + 1], v[8 * j + 2], v[8 * j + 3]);
                  d0[1] = make_uint4(v[8 * j + 4], v[8 * j + 5], v[8 * j + 6], v[8 * j + 7]);
                }
              }
            }
          }
          if (staged) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&maps.y[t.job], buf, t.n0 + c, row0 + q * 32);
              bulk_commit();
            }
            ++n_st;
          }
        }
      }
      if (EPI == PAIR_STORE || EPI == PAIR_SWIGLU) release();
      if (EPI == PAIR_ROUTER || EPI == PAIR_ROUTER2) row_best(wh, true);
      if (EPI == PAIR_ROUTER_ROWS) {   // both halves by one warp, whose keys stay in registers
        if (wh != 0) {
          release();
          continue;
        }
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          stage_norms(h);
          best = -INFINITY;
          best_k = 0;
          row_best(h, h == 1);
          if (best > -INFINITY) {
            const unsigned long long key = route_key(best, best_k);
            row_key = key > row_key ? key : row_key;
          }
        }
        if ((tile + 1) % tn_all == 0) {
          if (row_ok) {
            const int id = row_key == 0ull ? 0 : (int)(0xFFFFFFFFu - (uint32_t)(row_key & 0xFFFFFFFFull));
            if (p.out_centroid) p.out_centroid[grow] = id;
            p.out_expert[grow] = p.cmap ? p.cmap[id] : id;
            if (p.out_best) p.out_best[grow] = row_key == 0ull ? -INFINITY : key_to_float((uint32_t)(row_key >> 32));
          }
          row_key = 0ull;
        }
      }
      if (EPI == PAIR_ROUTER && row_ok && best > -INFINITY)
        atomicMax(p.keys + grow, route_key(best, best_k));
      if (EPI == PAIR_ROUTER2 && row_ok) {
        // Two-slot merge: the max goes to keys; whatever loses a comparison there (the value it displaced, or the
        // candidate itself) is offered to keys2.  Keys are distinct and both slots are maxima: order independent.
        const float cand[2] = {best, second};
        const int cand_k[2] = {best_k, second_k};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (cand[i] > -INFINITY) {
            const unsigned long long key = route_key(cand[i], cand_k[i]);
            const unsigned long long old = atomicMax(p.keys + grow, key);
            const unsigned long long loser = old < key ? old : key;
            if (loser != 0ull) atomicMax(p.keys2 + grow, loser);
          }
        }
      }
    }
    if ((EPI == PAIR_STORE || EPI == PAIR_SWIGLU) && lane == 0) bulk_wait_all();   // this thread's tiled stores are complete
  }
  // ------------------------------------------------------------------ teardown
  if (*abort_flag) {
    // a wait ran out somewhere: give copies / MMAs still in flight time to land before memory is released
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < 2000000ull) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  cluster_arrive();   // neither CTA leaves, or frees its tensor memory, while the other may still signal or multiply
  cluster_wait();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
template <int EPI>
static moin_status launch_pair(HostState* hs, const PairMaps& maps, const PairParams& p, long max_tiles, cudaStream_t stream) {
  cudaError_t e = ensure_smem_optin(OPTIN_TC_PAIR + EPI, tc_pair_kernel<EPI>, kPairSmem);
  if (e != cudaSuccess) return record_cuda(e);
  long pairs = max_tiles < hs->n_sms / 2 ? max_tiles : hs->n_sms / 2;
  if (pairs < 1) pairs = 1;
  return record_cuda(launch_pdl(tc_pair_kernel<EPI>, (unsigned)(2 * pairs), kPairThreads, kPairSmem, stream, maps, p));
}

// Tile width: the one with the least (waves of pair tiles over the SM pairs) x (time of one tile).  Per k-block an SM
// takes in 128 + bn / 2 rows of 128 bytes at about 64 bytes a clock = 256 + bn clocks, and multiplies for 2 bn: the
// fill is the longer below bn = 256.  3392 rows x 2048 columns (14 x 8 tiles of 256 on 74 pairs: two waves, the second
// half empty) take 14 x 10 tiles of 208.
static int pick_pair_bn(long tiles_m, const int* N, int n_jobs, int n_sms, int step) {
  int best = 256;
  long best_cost = -1;
  for (int bn = 256; bn >= 64; bn -= step) {
    long tn = 0;
    for (int j = 0; j < n_jobs; ++j) tn += (N[j] + bn - 1) / bn;
    const long tiles = (tiles_m + 1) / 2 * tn, pairs = n_sms / 2;
    const long cost = ((tiles + pairs - 1) / pairs) * (bn + 256);
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best = bn;
    }
  }
  return best;
}

moin_status launch_pair_gemm(HostState* hs, const PlanView* pv, const PairJob* jobs, int n_jobs, int M, int K,
                             cudaStream_t stream) {
  if (n_jobs < 1 || n_jobs > kPairJobs) return MOIN_ERR_INVALID_ARG;
  int N[kPairJobs];
  for (int j = 0; j < n_jobs; ++j) N[j] = jobs[j].N;
  const long tiles_m = (M + kPairM - 1) / kPairM;
  const int bn = pick_pair_bn(tiles_m, N, n_jobs, hs->n_sms, 16);
  PairMaps maps;
  PairParams p = {};
  p.M = M; p.K = K; p.n_jobs = n_jobs; p.bn = p.cols = bn; p.status = hs->status;
  if (pv) {
    p.header = pv->header; p.gemm_tab = pv->gemm_tab; p.run_expert = pv->run_expert; p.run_row0 = pv->run_row0;
    p.tail_r = jobs[0].pool->r;
  }
  int tn = 0;
  for (int j = 0; j < n_jobs; ++j) {
    const PairJob& g = jobs[j];
    moin_status st = make_map(&maps.x[j], g.x, M, K, kPairM);
    if (!st) st = make_map(&maps.w[j], g.W, g.N, K, bn / 2);
    if (!st) st = make_map(&maps.y[j], g.y, M, g.N, 32);
    if (!st && pv) {
      const int r = g.pool->r;
      st = make_map(&maps.h[j], g.hb, 2ull * M, r, kPairM);
      if (!st) st = make_map(&maps.b[j], g.pool->B, (uint64_t)g.pool->n_slots * g.N, r, bn / 2);
      p.slot_of_expert[j] = g.pool->slot_of_expert;
      p.slot_rank[j] = g.pool->slot_rank;
    }
    if (st) return st;
    tn += (g.N + bn - 1) / bn;
    p.N[j] = g.N; p.tn_end[j] = tn; p.y[j] = g.y; p.y0[j] = g.y0;
  }
  // upper bound on the row tiles of a plan without reading it back; the grid is capped at the SM pairs
  const long max_tiles = (pv ? (long)M : (tiles_m + 1) / 2) * tn;
  return launch_pair<PAIR_STORE>(hs, maps, p, max_tiles, stream);
}

// The gate and up projections of a block with the product of the two: one launch, act[M][F] instead of two matrices.
// The first CTA holds cols rows of the gate weight and the second the same rows of the up weight, so one MMA gives both
// (accumulator columns 0 .. cols - 1 and cols .. 2 cols - 1); the low-rank blocks multiply the gate's and the up
// projection's halves of the columns one after the other.  16384 x 2048 -> 2 x 5632: the two projections 510 us and the
// product's own pass 94 us (553 MB), now 507 us together.
moin_status launch_pair_swiglu(HostState* hs, const PlanView* pv, const PairJob* jobs, int M, int K, cudaStream_t stream) {
  const int F = jobs[0].N, N2 = 2 * F;
  const long tiles_m = (M + kPairM - 1) / kPairM;
  const int bn = pick_pair_bn(tiles_m, &N2, 1, hs->n_sms, 64);   // (the halves start at multiples of 32 columns)
  PairMaps maps;
  PairParams p = {};
  p.M = M; p.K = K; p.n_jobs = 1; p.bn = bn; p.cols = bn / 2; p.status = hs->status;
  p.N[0] = p.N[1] = F;
  p.tn_end[0] = (F + p.cols - 1) / p.cols;
  p.y[0] = jobs[0].y;
  moin_status st = make_map(&maps.x[0], jobs[0].x, M, K, kPairM);
  if (!st) st = make_map(&maps.y[0], jobs[0].y, M, F, 32);
  if (pv) {
    p.header = pv->header; p.gemm_tab = pv->gemm_tab; p.run_expert = pv->run_expert; p.run_row0 = pv->run_row0;
    p.tail_r = jobs[0].pool->r;
  }
  for (int j = 0; j < 2 && !st; ++j) {
    const PairJob& g = jobs[j];
    st = make_map(&maps.w[j], g.W, F, K, p.cols);
    if (!st && pv) {
      const int r = g.pool->r;
      st = make_map(&maps.h[j], g.hb, 2ull * M, r, kPairM);
      if (!st) st = make_map(&maps.b[j], g.pool->B, (uint64_t)g.pool->n_slots * F, r, p.cols / 2);
      p.slot_of_expert[j] = g.pool->slot_of_expert;
      p.slot_rank[j] = g.pool->slot_rank;
    }
  }
  if (st) return st;
  return launch_pair<PAIR_SWIGLU>(hs, maps, p, (pv ? (long)M : (tiles_m + 1) / 2) * p.tn_end[0], stream);
}

moin_status launch_pair_router(HostState* hs, const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm, int Q,
                               int K, int D, unsigned long long* keys, cudaStream_t stream, unsigned long long* keys2) {
  const long tiles_m = (Q + kPairM - 1) / kPairM;
  const int bn = pick_pair_bn(tiles_m, &K, 1, hs->n_sms, 64);
  PairMaps maps;
  PairParams p = {};
  p.M = Q; p.K = D; p.n_jobs = 1; p.bn = p.cols = bn; p.status = hs->status; p.inv_norm = inv_norm; p.keys = keys; p.keys2 = keys2;
  p.N[0] = K; p.tn_end[0] = (K + bn - 1) / bn;
  moin_status st = make_map(&maps.x[0], q, Q, D, kPairM);
  if (!st) st = make_map(&maps.w[0], c, K, D, bn / 2);
  if (st) return st;
  const long tiles = (tiles_m + 1) / 2 * p.tn_end[0];
  if (keys2 != nullptr) return launch_pair<PAIR_ROUTER2>(hs, maps, p, tiles, stream);
  return launch_pair<PAIR_ROUTER>(hs, maps, p, tiles, stream);
}

// The same without scratch: outputs written by the pair, except that out_best still lacks the division by |q|.  For few
// queries only, as a pair then walks the table alone (the keys' way has a clearing and a finishing launch and more SMs:
// 400 x 500 x 768 8.8 us with keys, 13.3 without, 1024 x 1000 x 768 9.9 and 20.6; the cluster kernel in waves 10 and 37).
// The scores and their order of merging are those of launch_pair_router, and so are the results, to the bit.
moin_status launch_pair_router_rows(HostState* hs, const __nv_bfloat16* q, const __nv_bfloat16* c, const float* inv_norm,
                                    const int* cmap, int Q, int K, int D, int* out_expert, int* out_centroid, float* out_best,
                                    cudaStream_t stream) {
  PairMaps maps;
  PairParams p = {};
  p.M = Q; p.K = D; p.n_jobs = 1; p.status = hs->status; p.inv_norm = inv_norm;
  p.bn = p.cols = K > 192 ? 256 : (K + 63) / 64 * 64;
  p.N[0] = K; p.tn_end[0] = (K + p.bn - 1) / p.bn;
  p.cmap = cmap; p.out_expert = out_expert; p.out_centroid = out_centroid; p.out_best = out_best;
  moin_status st = make_map(&maps.x[0], q, Q, D, kPairM);
  if (!st) st = make_map(&maps.w[0], c, K, D, p.bn / 2);
  if (st) return st;
  return launch_pair<PAIR_ROUTER_ROWS>(hs, maps, p, (Q + 2 * kPairM - 1) / (2 * kPairM), stream);
}

}  // namespace moin
