// Causal grouped-query attention inside each request on tcgen05 / TMEM (head_dim 64).
//
// One work item = (request, kv head, block of query positions).  The g = n_heads / n_kv_heads query heads
// that share a kv head are stacked into one 128-row tile: row r holds position q0 + r / g of head kvh * g + r % g,
// so a block covers 128 / g positions and every staged K / V tile serves all g heads.  Persistent CTAs (two per
// SM) walk the items, longest first.
//
// The time of an item is a chain of hand-overs (scores, softmax, product), not any unit's throughput, so a CTA keeps two
// chains going: the even key tiles are one STREAM, the odd ones another, each with its own four softmax warps, scores,
// running maximum, row sum and accumulator; the two meet once at the end of the item.  A stream takes a thread per row and
// one pass over its key tiles (the scores of a tile are read from tensor memory twice, once for their maximum): p = 2^(s - m)
// against a maximum m that may lag behind by a factor of up to 2^8 (p is bf16 and
// its sum fp32: the relative accuracy is the same), so the accumulator is rescaled only when a row outgrows that.  P goes
// back into tensor memory over the scores it came from, as the A operand of the second product: nothing of it passes
// through shared memory.  Warp roles:
//   warp 0      TMA producer: K and V tiles [64 keys x 64 dims] into rings of four.  K is a K-major operand of the
//               form the GEMMs use; V, whose rows run along the output dimension of the second product, is read
//               as an MN-major operand (same staged bytes, the other operand layout), so no transposed copy exists
//   warp 1      MMA issuer: polls both streams and issues whatever is ready, S_h = Q K^T or O_h += P_h V
//   warps 2-5   stream 0, warps 6-9 stream 1; between two items they rotate and stage the next Q (128-byte swizzled rows,
//               written by hand, two buffers: its first scores are computed while this item's O is merged and stored)
// Tensor memory: S_h / P_h at columns 64 h, O_h at 128 + 64 h; two CTAs fill an SM's 512 columns.
// Key tiles start at the request's first token (only the innermost coordinate of a TMA copy has an alignment rule, and
// that is the head's first dimension); the mask is key <= query position.
// Every mbarrier wait is bounded; on expiry the CTA raises the status flag, drains and returns.
// A tile takes a stream about 3 us (at 16 such warps an SM a warp issues an instruction every eight cycles or so; the
// exponentials alone would take a quarter of it), an item's end another 3: four chains an SM are what tensor memory holds.
// Per block of 64 requests of 256 tokens 99 -> 80 us, of 11 requests of 65 to 600 tokens 42.5 -> 34.8 us, against one chain
// per CTA (two threads a row, two passes over the keys: a tile's maximum first, scores computed twice beyond 256 keys).
// One barrier arrival per warp instead of per thread: 82 / 35.5 us.
#include <cuda.h>

#include "ptx.cuh"
#include "tc_gemm.cuh"

namespace moin {

constexpr int kAtThreads = 320;                  // producer warp, MMA warp, 8 softmax warps
constexpr int kAtKeys = 64;                      // keys per tile
constexpr int kAtTile = 128 * 64 * 2;            // Q tile: 128 rows x 128 bytes
constexpr int kAtKV = kAtKeys * 64 * 2;          // K and V tiles: 64 keys x 128 bytes
constexpr int kAtRing = 4;                       // stages of K and of V
constexpr int kAtCuMax = 1024;                   // request offsets kept in shared memory when there are at most this many
constexpr int kAtRopeBytes = 4096;               // (cos, sin) rows of an item's positions, when they fit (<= 16 positions)
constexpr int kAtMerge = 4096;                   // (maximum, sum) of every row by stream, for two items
constexpr int kAtSmem = 2 * kAtTile /*Q*/ + 2 * kAtRing * kAtKV + 1024 /*align*/ + 256 /*barriers*/ + kAtMerge +
                        kAtCuMax * 4 + kAtRopeBytes;
constexpr int kAtTmemCols = 256;
constexpr float kAtLag = 8.f;                    // powers of two by which a running maximum may lag behind

struct AttParams {
  __nv_bfloat16* out;          // [T, n_heads * 64]
  const int* cu;               // [R + 1]
  const float2* rope;          // [max_seqlen, 32] (cos, sin)
  int R, n_heads, n_kv, g, ppt, n_qb;   // g heads per kv head, ppt = 128 / g positions per tile, n_qb query blocks
  int max_pos;                 // rows of the rope table
  int rope_smem, cu_smem;      // an item's rope rows / the request offsets are staged in shared memory
  float scale_log2;
  DeviceStatus* status;
};

constexpr uint32_t kAtIdesc = idesc_bf16(128, 64);
// the same with B MN-major (V tile: one 128-byte row per key, the 64 output dims contiguous); a 16-key step of
// such a tile is two 8-key groups = 2048 bytes further on
constexpr uint32_t kAtIdescPV = kAtIdesc | (1u << 16);
constexpr uint64_t kAtVStep = 2048 >> 4;

__device__ __forceinline__ float fast_exp2(float x) {   // x <= kAtLag here: 2^x up to 256, below 2^-126 zero
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Two-lane fp32 arithmetic (one instruction for a pair of scores): the softmax threads are bound by the number of
// instructions they issue, not by any one pipe.
__device__ __forceinline__ uint64_t pair_f32(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpair_f32(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// byte offset of 16-byte chunk c of row r in a swizzled [rows x 128 bytes] tile
__device__ __forceinline__ uint32_t at_swz(int r, int c) {
  return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4));
}

struct AttItem { int req, kvh, q0, t0, L, n_tiles; bool on; };
__device__ __forceinline__ AttItem at_item(const AttParams& p, const int* cu, int idx) {
  AttItem it;
  const int per_qb = p.R * p.n_kv;
  const int qb = p.n_qb - 1 - idx / per_qb;     // longest blocks first
  const int rem = idx % per_qb;
  it.req = rem / p.n_kv;
  it.kvh = rem % p.n_kv;
  it.q0 = qb * p.ppt;
  it.t0 = cu[it.req];
  it.L = cu[it.req + 1] - it.t0;
  it.on = it.q0 < it.L;
  const int kv_end = min(it.L, it.q0 + p.ppt);   // keys of the request this block can see
  it.n_tiles = it.on ? (kv_end + kAtKeys - 1) / kAtKeys : 0;
  return it;
}

__global__ void __launch_bounds__(kAtThreads, 2)
attention_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const AttParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - raw);
  const uint32_t sQ = base, sK = base + 2 * kAtTile, sV = sK + kAtRing * kAtKV;
  const uint32_t bars = sV + kAtRing * kAtKV;
  uint8_t* bar_ptr = base_ptr + (bars - base);
  // barriers (8 bytes each)
  const uint32_t kfull = bars, kempty = bars + 32, vfull = bars + 64, vempty = bars + 96, sready = bars + 128,
                 pready = bars + 144, pvdone = bars + 160, oready = bars + 176, ofree = bars + 184, qready = bars + 192,
                 rfull = bars + 200, rempty = bars + 208, qraw = bars + 240;
  int* cu_s = reinterpret_cast<int*>(bar_ptr + 256 + kAtMerge);
  const uint32_t sRope = bars + 256 + kAtMerge + kAtCuMax * 4;
  const int* cu = p.cu_smem ? cu_s : p.cu;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_ptr + 216);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_ptr + 224);
  volatile int* sm_fail = reinterpret_cast<volatile int*>(bar_ptr + 228);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kAtRing; ++i) {
      mbar_init(kfull + 8 * i, 1); mbar_init(kempty + 8 * i, 1);
      mbar_init(vfull + 8 * i, 1); mbar_init(vempty + 8 * i, 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(sready + 8 * h, 1); mbar_init(pready + 8 * h, 128); mbar_init(pvdone + 8 * h, 1);
    }
    mbar_init(oready, 1);
    mbar_init(ofree, 256);
    mbar_init(qready, 256);
    mbar_init(qraw, 1);
    mbar_init(rfull, 1);
    mbar_init(rempty, 256);
    *abort_flag = 0;
    sm_fail[0] = sm_fail[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), kAtTmemCols);
    tmem_relinquish();
  }
  pdl_begin();   // (the set-up above overlaps the tail of the kernel before)
  if (p.cu_smem)
    for (int i = threadIdx.x; i <= p.R; i += kAtThreads) cu_s[i] = __ldg(p.cu + i);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int n_items = p.n_qb * p.R * p.n_kv;
  auto next_item = [&](int& i, AttItem& out) -> bool {   // the next item of this CTA that has any query row
    for (i += gridDim.x; i < n_items; i += gridDim.x) {
      out = at_item(p, cu, i);
      if (out.on) return true;
    }
    return false;
  };

  if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      uint32_t tq = 0, rq = 0;   // tiles, rope blocks so far
      bool ok = true;
      int idx = (int)blockIdx.x - (int)gridDim.x;
      AttItem it;
      bool have = next_item(idx, it);
      auto load_rope = [&](const AttItem& n) -> bool {   // (cos, sin) rows of the item's positions, for its Q staging
        if (!p.rope_smem) return true;
        if (!mbar_wait(rempty, (rq & 1u) ^ 1u, abort_flag, p.status, 44)) return false;
        const uint32_t bytes = (uint32_t)min(p.ppt, p.max_pos - n.q0) * 256u;
        mbar_expect_tx(rfull, bytes);
        bulk_load_1d(sRope, p.rope + (size_t)n.q0 * 32, bytes, rfull);
        ++rq;
        return true;
      };
      if (have) ok = load_rope(it);
      while (have && ok) {
        AttItem nx;
        int nidx = idx;
        const bool have_nx = next_item(nidx, nx);
        if (have_nx) ok = load_rope(nx);   // wanted after this item's first tiles (the buffer: since the item before's)
        for (int j = 0; j < it.n_tiles && ok; ++j, ++tq) {
          const uint32_t s = tq % kAtRing, ph = (tq / kAtRing) & 1u;
          if (!(ok = mbar_wait(kempty + 8 * s, ph ^ 1u, abort_flag, p.status, 31))) break;
          mbar_expect_tx(kfull + 8 * s, kAtKV);
          tma_load_2d(sK + s * kAtKV, &tmK, kfull + 8 * s, it.kvh * 64, it.t0 + j * kAtKeys);
          if (!(ok = mbar_wait(vempty + 8 * s, ph ^ 1u, abort_flag, p.status, 32))) break;
          mbar_expect_tx(vfull + 8 * s, kAtKV);
          tma_load_2d(sV + s * kAtKV, &tmV, vfull + 8 * s, it.kvh * 64, it.t0 + j * kAtKeys);
        }
        it = nx;
        idx = nidx;
        have = have_nx;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    {   // the whole warp walks the loop, one elected lane issues (as in the GEMMs)
      const bool leader = elect_one();
      uint32_t tq = 0, nit = 0;
      uint32_t n_p[2] = {0, 0};   // products issued per stream: phases of sready / pready / pvdone
      bool ok = true;
      for (int idx = blockIdx.x; idx < n_items && ok; idx += gridDim.x) {
        const AttItem it = at_item(p, cu, idx);
        if (!it.on) continue;
        if (!(ok = mbar_wait_warp(qready, nit & 1u, abort_flag, p.status, 35))) break;
        tc_fence_after();
        const uint64_t dq = sdesc_k128(sQ + (nit & 1u) * kAtTile);
        int tile[2] = {0, 1}, left = it.n_tiles;   // next tile of each stream; products to go
        bool scores[2] = {false, false};           // its scores have been issued
        bool o_free = false;
        unsigned long long t0 = 0;
        uint32_t spins = 0;
        while (left > 0) {
          bool moved = false;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (tile[h] >= it.n_tiles) continue;
            const uint32_t g = tq + (uint32_t)tile[h], s = g % kAtRing, ph = (g / kAtRing) & 1u;
            if (!scores[h]) {
              // P of the product before lies where these scores go
              if (!__all_sync(0xffffffffu, (n_p[h] == 0 || mbar_test_wait(pvdone + 8 * h, (n_p[h] - 1) & 1u)) &&
                                               mbar_test_wait(kfull + 8 * s, ph))) continue;
              tc_fence_after();
              const uint64_t dk = sdesc_k128(sK + s * kAtKV);
              if (leader) {
#pragma unroll
                for (int k = 0; k < 4; ++k) tc_mma_bf16(tmem + h * 64, dq + (uint64_t)(2 * k), dk + (uint64_t)(2 * k), kAtIdesc, k > 0 ? 1u : 0u);
                tc_commit(kempty + 8 * s);
                tc_commit(sready + 8 * h);
              }
              scores[h] = true;
              moved = true;
            } else {
              // the accumulators are free once the O of the item before has been read
              if (!o_free && !(o_free = __all_sync(0xffffffffu, mbar_test_wait(ofree, (nit & 1u) ^ 1u)))) continue;
              if (!__all_sync(0xffffffffu, mbar_test_wait(pready + 8 * h, n_p[h] & 1u) && mbar_test_wait(vfull + 8 * s, ph))) continue;
              tc_fence_after();
              const uint64_t dv = sdesc_k128(sV + s * kAtKV);
              const uint32_t first = tile[h] == h ? 0u : 1u;
              if (leader) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                  tc_mma_bf16_ta(tmem + 128 + h * 64, tmem + h * 64 + 8 * k, dv + kAtVStep * k, kAtIdescPV, k > 0 ? 1u : first);
                tc_commit(vempty + 8 * s);
                tc_commit(pvdone + 8 * h);
              }
              ++n_p[h];
              scores[h] = false;
              tile[h] += 2;
              --left;
              moved = true;
            }
          }
          if (moved) {
            spins = 0;
            t0 = 0;
          } else if ((++spins & 0x3FFu) == 0) {   // bounded, as every wait
            int stop = *abort_flag;
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > kWaitLimitNs) {
              stop = *abort_flag = 1;
              atomicExch(&p.status->timeout_flag, 1);
              atomicExch(&p.status->timeout_site, 33);
            }
            if (__any_sync(0xffffffffu, stop != 0)) {
              ok = false;
              break;
            }
          }
        }
        if (ok && leader) tc_commit(oready);
        tq += (uint32_t)it.n_tiles;
        ++nit;
      }
    }
  } else {
    // ------------------------------------------------------------------ softmax / epilogue: a thread per row and stream
    // The streams of an item meet through shared memory at a named barrier that all 256 threads reach whatever happened
    // before (a thread whose wait ran out skips the work, not the barrier); the decision to give up is taken from the
    // item's flag, which is only written before it (two flags in turn: the next item may fail before all have read).
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const int qd = p.n_heads * 64;
    float2* xml = reinterpret_cast<float2*>(bar_ptr + 256);   // [item parity][stream][row]: (maximum, sum)
    uint32_t n_s = 0, nit = 0, rq = 0;                        // score tiles of this stream, items, rope blocks
    bool ok = true;
    // Q rows: the raw tile comes by TMA (in the swizzled layout); a thread rotates 16-byte chunks 2 half, 2 half + 1 of its
    // row and their partners 4 further on in place (pairs (d, d + 32), position inside the request).  Rows past the
    // request are whatever lies there: nothing of a row reaches another.
    const int i0c = 2 * half;
    const int row_pos = row / p.g, row_head = row % p.g;   // position inside the block and head inside the group
    auto q_load = [&](const AttItem& n, uint32_t buf) {    // one thread
      mbar_expect_tx(qraw, kAtTile);
      tma_load_3d(sQ + buf * kAtTile, &tmQ, qraw, 0, n.kvh * p.g, n.t0 + n.q0);
    };
    uint32_t nq = 0;   // Q tiles staged
    auto q_stage = [&](const AttItem& n) {
      uint8_t* qrow = base_ptr + (sQ - base) + (nq & 1u) * kAtTile;
      ok = mbar_wait_warp(qraw, nq & 1u, abort_flag, p.status, 46) && ok;
      ++nq;
      const int npos = n.q0 + row_pos;
      const bool nlive = npos < n.L;
      uint4 c[4];
      c[0] = *reinterpret_cast<const uint4*>(qrow + at_swz(row, i0c));
      c[1] = *reinterpret_cast<const uint4*>(qrow + at_swz(row, i0c + 1));
      c[2] = *reinterpret_cast<const uint4*>(qrow + at_swz(row, i0c + 4));
      c[3] = *reinterpret_cast<const uint4*>(qrow + at_swz(row, i0c + 5));
      // the (cos, sin) rows of the item's positions: staged by the producer when they fit, else from the table
      if (p.rope_smem) ok = mbar_wait_warp(rfull, rq & 1u, abort_flag, p.status, 45) && ok;
      if (nlive) {
        const float4* rt = p.rope_smem ? reinterpret_cast<const float4*>(base_ptr + (sRope - base) + row_pos * 256)
                                       : reinterpret_cast<const float4*>(p.rope + (size_t)npos * 32);
#pragma unroll
        for (int i = 0; i < 2; ++i) {          // chunk i0c + i holds dims 8 (i0c + i) .., its partner the same + 32
          uint32_t* lo = reinterpret_cast<uint32_t*>(&c[i]);
          uint32_t* hi = reinterpret_cast<uint32_t*>(&c[i + 2]);
#pragma unroll
          for (int w = 0; w < 4; ++w) {        // word w: two consecutive dims
            const float4 cs = rt[(8 * (i0c + i) + 2 * w) / 2];   // (cos, sin) of those two dims
            const float a0 = bf16_lo(lo[w]), a1 = bf16_hi(lo[w]), b0 = bf16_lo(hi[w]), b1 = bf16_hi(hi[w]);
            lo[w] = pack_bf16(a0 * cs.x - b0 * cs.y, a1 * cs.z - b1 * cs.w);
            hi[w] = pack_bf16(b0 * cs.x + a0 * cs.y, b1 * cs.z + a1 * cs.w);
          }
        }
      }
      *reinterpret_cast<uint4*>(qrow + at_swz(row, i0c)) = c[0];
      *reinterpret_cast<uint4*>(qrow + at_swz(row, i0c + 1)) = c[1];
      *reinterpret_cast<uint4*>(qrow + at_swz(row, i0c + 4)) = c[2];
      *reinterpret_cast<uint4*>(qrow + at_swz(row, i0c + 5)) = c[3];
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(qready);
      if (p.rope_smem) {
        mbar_arrive(rempty);
        ++rq;
      }
    };
    int idx = (int)blockIdx.x - (int)gridDim.x;
    AttItem it;
    bool have = next_item(idx, it);
    if (have) {
      if (threadIdx.x == 64) q_load(it, 0);
      q_stage(it);
    }
    const uint32_t s_addr = tmem + lane_addr + half * 64;
    while (have) {
      const int pos = it.q0 + row_pos;
      // The next item's Q buffer is free: O of the item before this one was waited for, so all its products are complete.
      AttItem nx;
      const bool have_nx = next_item(idx, nx);
      if (have_nx && threadIdx.x == 64) q_load(nx, (nit + 1) & 1u);
      if (have_nx && half >= it.n_tiles) q_stage(nx);
      // Keys are counted from the request's first token; row `pos` sees key <= pos.  A group of 16 is visible to every
      // row of the item when it ends before the item's first position, to none when it starts after the item's last one
      // (both the same for all threads), and is masked key by key otherwise.
      const int q_last = it.q0 + p.ppt - 1;
      float m = -INFINITY, l = 0.f;   // running maximum of the raw scores (the scale is positive), sum of p
      for (int j = half; j < it.n_tiles && ok; j += 2, ++n_s) {
        if (!(ok = mbar_wait_warp(sready + 8 * half, n_s & 1u, abort_flag, p.status, 39))) break;
        tc_fence_after();
        // twice over the scores in groups of 16 keys, the next group's read in flight (a thread that keeps all 64 spills)
        const int kr0 = j * kAtKeys;
        uint32_t va[16], vb[16];
        float ma = -INFINITY, mc = -INFINITY;
        auto group_max = [&](const uint32_t (&v)[16], int kr) {
          if (kr + 15 <= it.q0) {
#pragma unroll
            for (int c = 0; c < 16; c += 4) {
              ma = fmax3(ma, __uint_as_float(v[c]), __uint_as_float(v[c + 1]));
              mc = fmax3(mc, __uint_as_float(v[c + 2]), __uint_as_float(v[c + 3]));
            }
          } else if (kr <= q_last) {
#pragma unroll
            for (int c = 0; c < 16; ++c)
              if (kr + c <= pos) ma = fmaxf(ma, __uint_as_float(v[c]));
          }
        };
        tmem_ld16(s_addr, va);
        tmem_ld16(s_addr + 16, vb);
        tmem_ld_wait();
        group_max(va, kr0);
        group_max(vb, kr0 + 16);
        tmem_ld16(s_addr + 32, va);
        tmem_ld16(s_addr + 48, vb);
        tmem_ld_wait();
        group_max(va, kr0 + 32);
        group_max(vb, kr0 + 48);
        tmem_ld16(s_addr, va);
        const float mx = fmaxf(ma, mc);
        if (j == half) {
          m = mx;
        } else {
          const bool grow = (mx - m) * p.scale_log2 > kAtLag;
          if (__any_sync(0xffffffffu, grow)) {   // (these scores exist only because the product before is complete)
            const float m_new = grow ? mx : m;
            const float corr = grow ? fast_exp2((m - m_new) * p.scale_log2) : 1.f;
            m = m_new;
            l *= corr;
#pragma unroll
            for (int c = 0; c < 64; c += 16) {
              uint32_t o[16];
              tmem_ld16(s_addr + 128 + c, o);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * corr);
              tmem_st16(s_addr + 128 + c, o);
            }
          }
        }
        const float mb = (m == -INFINITY) ? 0.f : m * p.scale_log2;
        const uint64_t nmb2 = pair_f32(-mb, -mb), scale2 = pair_f32(p.scale_log2, p.scale_log2);
        uint64_t l2 = pair_f32(l, 0.f);
        auto group_p = [&](const uint32_t (&v)[16], int kr, uint32_t* w) {
          if (kr + 15 <= it.q0) {
#pragma unroll
            for (int c = 0; c < 16; c += 2) {
              float x0, x1;
              unpair_f32(fma2(pair_f32(__uint_as_float(v[c]), __uint_as_float(v[c + 1])), scale2, nmb2), x0, x1);
              const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
              l2 = add2(l2, pair_f32(p0, p1));
              w[c >> 1] = pack_bf16(p0, p1);
            }
          } else if (kr <= q_last) {
#pragma unroll
            for (int c = 0; c < 16; c += 2) {
              const float p0 = kr + c <= pos ? fast_exp2(fmaf(__uint_as_float(v[c]), p.scale_log2, -mb)) : 0.f;
              const float p1 = kr + c + 1 <= pos ? fast_exp2(fmaf(__uint_as_float(v[c + 1]), p.scale_log2, -mb)) : 0.f;
              l2 = add2(l2, pair_f32(p0, p1));
              w[c >> 1] = pack_bf16(p0, p1);
            }
          } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) w[c] = 0u;
          }
        };
#pragma unroll
        for (int hq = 0; hq < 2; ++hq) {   // P of 32 keys into columns whose scores have been read
          uint32_t w[16];
          tmem_ld_wait();
          tmem_ld16(s_addr + 32 * hq + 16, vb);
          group_p(va, kr0 + 32 * hq, w);
          tmem_ld_wait();
          if (hq == 0) tmem_ld16(s_addr + 32, va);
          group_p(vb, kr0 + 32 * hq + 16, w + 8);
          tmem_st16(s_addr + 16 * hq, w);
        }
        float la, lb;
        unpair_f32(l2, la, lb);
        l = la + lb;
        tmem_st_wait();
        tc_fence_before();
        mbar_arrive(pready + 8 * half);
        if (have_nx && j == half) q_stage(nx);   // under this tile's product and the next one's scores
      }
      float2* mine = xml + (nit & 1u) * 256;
      mine[half * 128 + row] = make_float2(m, l);
      if (!ok) sm_fail[nit & 1u] = 1;
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (sm_fail[nit & 1u]) break;              // the same for all 256 threads
      const float2 other = mine[(half ^ 1) * 128 + row];
      const float top = fmaxf(m, other.x);
      const float a_me = fast_exp2((m - top) * p.scale_log2), a_ot = fast_exp2((other.x - top) * p.scale_log2);
      const float sum = l * a_me + other.y * a_ot;
      const float inv = sum > 0.f ? 1.f / sum : 0.f;
      const float f0 = (half == 0 ? a_me : a_ot) * inv, f1 = (half == 0 ? a_ot : a_me) * inv;
      // ---- (O_0 f_0 + O_1 f_1) -> out: this thread's 32 of the row's 64 dims
      if ((ok = mbar_wait_warp(oready, nit & 1u, abort_flag, p.status, 42))) {
        tc_fence_after();
        const bool live = it.q0 + row_pos < it.L;
        __nv_bfloat16* dst = p.out + (size_t)(it.t0 + (live ? it.q0 + row_pos : 0)) * qd + (it.kvh * p.g + row_head) * 64 + half * 32;
        uint32_t v[16], u[16];
#pragma unroll
        for (int c = 0; c < 32; c += 16) {
          tmem_ld16(tmem + lane_addr + 128 + half * 32 + c, v);
          if (it.n_tiles > 1) {
            tmem_ld16(tmem + lane_addr + 192 + half * 32 + c, u);
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) u[i] = 0u;   // (nothing was ever accumulated there)
          }
          tmem_ld_wait();
          if (c == 16) {                          // O is in registers: the accumulators may be written again
            tc_fence_before();
            mbar_arrive(ofree);
          }
          uint32_t o[8];
#pragma unroll
          for (int i = 0; i < 16; i += 2)
            o[i >> 1] = pack_bf16(fmaf(__uint_as_float(u[i]), f1, __uint_as_float(v[i]) * f0),
                                  fmaf(__uint_as_float(u[i + 1]), f1, __uint_as_float(v[i + 1]) * f0));
          if (live) {
            *reinterpret_cast<uint4*>(dst + c) = make_uint4(o[0], o[1], o[2], o[3]);
            *reinterpret_cast<uint4*>(dst + c + 8) = make_uint4(o[4], o[5], o[6], o[7]);
          }
        }
      }
      ++nit;
      it = nx;
      have = have_nx;
    }
  }
  // ------------------------------------------------------------------ teardown
  if (*abort_flag) {
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < 2000000ull) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kAtTmemCols);
  }
}

bool attention_tc_supported(int n_heads, int n_kv_heads, int head_dim) {
  if (head_dim != 64 || n_kv_heads < 1 || (n_heads % n_kv_heads) != 0) return false;
  const int g = n_heads / n_kv_heads;
  return g >= 1 && g <= 128 && (128 % g) == 0;
}

// q [T, n_heads*64] (not rotated), k [T, n_kv*64] (rotated), v [T, n_kv*64] -> out [T, n_heads*64].
moin_status launch_attention_tc(HostState* hs, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                const int* cu, __nv_bfloat16* out, const float2* rope, int R,
                                int T, int max_seqlen, int n_heads, int n_kv_heads, float scale_log2,
                                cudaStream_t stream) {
  const int kvd = n_kv_heads * 64, g = n_heads / n_kv_heads;
  CUtensorMap mq, mk, mv;
  moin_status st = make_map_heads(&mq, q, (uint64_t)T, (uint32_t)n_heads, (uint32_t)g, (uint32_t)(128 / g));
  if (!st) st = make_map(&mk, k, (uint64_t)T, (uint64_t)kvd, kAtKeys);
  if (!st) st = make_map(&mv, v, (uint64_t)T, (uint64_t)kvd, kAtKeys);
  if (st) return st;
  AttParams p = {};
  p.out = out; p.cu = cu; p.rope = rope; p.R = R; p.n_heads = n_heads; p.n_kv = n_kv_heads; p.g = g;
  p.ppt = 128 / g; p.n_qb = (max_seqlen + p.ppt - 1) / p.ppt; p.scale_log2 = scale_log2; p.status = hs->status;
  p.max_pos = max_seqlen;
  p.rope_smem = p.ppt * 256 <= kAtRopeBytes;
  p.cu_smem = R + 1 <= kAtCuMax;
  cudaError_t e = ensure_smem_optin(OPTIN_ATTENTION, attention_tc_kernel, kAtSmem);
  if (e != cudaSuccess) return record_cuda(e);
  const long items = (long)p.n_qb * R * n_kv_heads;
  long grid = items < 2L * hs->n_sms ? items : 2L * hs->n_sms;
  if (grid < 1) grid = 1;
  return record_cuda(launch_pdl(attention_tc_kernel, (unsigned)grid, kAtThreads, kAtSmem, stream, mq, mk, mv, p));
}

}  // namespace moin
