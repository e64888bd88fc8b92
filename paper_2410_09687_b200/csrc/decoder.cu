// Decoder forward: glue kernels (embedding, RMSNorm, rotary embedding, causal GQA attention,
// SwiGLU) around the routed LoRA projections, and the host-side sequencing.
#include "common.cuh"
#include "tc_gemm.cuh"

namespace moin {

// token -> (position inside its request, its expert: the caller's per-token id if given, else the expert of its
// request).  One CTA per request.
__global__ void __launch_bounds__(256)
token_meta_kernel(const int* __restrict__ cu, const int* __restrict__ req_expert,
                  const int* __restrict__ token_expert_in, int R, int* __restrict__ pos,
                  int* __restrict__ token_expert, int* __restrict__ last_row) {
  pdl_begin();
  const int r = blockIdx.x;
  if (r >= R) return;
  const int t0 = cu[r], t1 = cu[r + 1];
  const int e = req_expert ? req_expert[r] : -1;
  for (int t = t0 + threadIdx.x; t < t1; t += blockDim.x) {
    pos[t] = t - t0;
    token_expert[t] = token_expert_in ? token_expert_in[t] : e;
  }
  if (threadIdx.x == 0) last_row[r] = (t1 > t0) ? t1 - 1 : -1;
}

// W[j][i] = bf16(fp32(value(code[j][i]) * scale[j])): 8-bit float codes (4 exponent bits, bias 7, 3 mantissa bits,
// no infinities, 0x7F / 0xFF = NaN) -> the bf16 weight the GEMMs read, for the matrices of one projection group.  A warp
// converts a row: eight codes a lane and load, so that loads and stores are whole lines, four loads in flight.  Bound by
// the traffic (one byte in, two out).  One launch per matrix, a thread per 16 codes with a 64-bit division for its row
// and the fields put together bit by bit: forward of 112 tokens on the 8-bit base 2.98 ms, with this 2.50.
struct DequantJobs {
  const uint2* codes[MOIN_MAX_GROUP];
  const float* scale[MOIN_MAX_GROUP];
  uint4* out[MOIN_MAX_GROUP];
  int row_end[MOIN_MAX_GROUP];   // rows of jobs 0 .. j
  int n;
};
__global__ void __launch_bounds__(256)
dequant_fp8_kernel(const DequantJobs jobs, int d_in8) {
  pdl_begin();
  int row = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (row >= jobs.row_end[jobs.n - 1]) return;
  const uint2* codes = jobs.codes[0];
  const float* scale = jobs.scale[0];
  uint4* out = jobs.out[0];
  int first = 0;
#pragma unroll
  for (int j = 1; j < MOIN_MAX_GROUP; ++j)
    if (j < jobs.n && row >= jobs.row_end[j - 1]) {
      codes = jobs.codes[j]; scale = jobs.scale[j]; out = jobs.out[j]; first = jobs.row_end[j - 1];
    }
  row -= first;
  const float sc = __ldg(scale + row);
  codes += (size_t)row * d_in8;
  out += (size_t)row * d_in8;
  for (int c0 = threadIdx.x & 31; c0 < d_in8; c0 += 4 * 32) {
    uint2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c0 + 32 * u < d_in8) v[u] = __ldg(codes + c0 + 32 * u);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c0 + 32 * u < d_in8) {
        uint4 o;
        fp8x4_to_bf16(v[u].x, sc, o.x, o.y);
        fp8x4_to_bf16(v[u].y, sc, o.z, o.w);
        out[c0 + 32 * u] = o;
      }
  }
}
static moin_status launch_dequant(const DequantJobs& jobs, int d_in, cudaStream_t stream) {
  ProfScope prof(MOIN_K_GLUE, 1, stream);
  return record_cuda(launch_pdl(dequant_fp8_kernel, (unsigned)((jobs.row_end[jobs.n - 1] + 7) / 8), 256, 0, stream, jobs, d_in / 8));
}

// cos/sin of pos * base^(-2i/hd), computed in double once per call.
__global__ void rope_table_kernel(float2* __restrict__ table, int n_pos, int half, double base) {
  pdl_begin();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_pos * half) return;
  const int p = idx / half, i = idx - p * half;
  const double ang = (double)p * pow(base, -(double)i / (double)half);
  table[idx] = make_float2((float)cos(ang), (float)sin(ang));
}

__global__ void __launch_bounds__(256)
embed_kernel(const int* __restrict__ tokens, const __nv_bfloat16* __restrict__ embed, int hidden, int vocab,
             float* __restrict__ res) {
  pdl_begin();
  const int t = blockIdx.x;
  int tok = tokens[t];
  tok = tok < 0 ? 0 : (tok >= vocab ? vocab - 1 : tok);
  const __nv_bfloat16* row = embed + (size_t)tok * hidden;
  for (int i = threadIdx.x * 8; i < hidden; i += blockDim.x * 8) {
    const uint4 v = ldg_cached(row + i);
    float4 a = make_float4(bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y));
    float4 b = make_float4(bf16_lo(v.z), bf16_hi(v.z), bf16_lo(v.w), bf16_hi(v.w));
    *reinterpret_cast<float4*>(res + (size_t)t * hidden + i) = a;
    *reinterpret_cast<float4*>(res + (size_t)t * hidden + i + 4) = b;
  }
}

// res[t] += add[t] (bf16, optional);  out[t] = bf16(res[t] / sqrt(mean(res[t]^2) + eps) * gain)  (optional)
// rows (nullable): gather list - CTA b normalises row rows[b] into out row b (used for last-token logits).
// Bound by the traffic of the row (res in and out, add, out).  A thread's pieces of rows up to 2048 wide stay in
// registers, all loads issued before the first use; the rest of a wider row is read again for the second pass.
constexpr int kNormKeep = 2;   // 16-byte pieces a thread keeps (more of them would cost rows in flight on an SM)
__global__ void __launch_bounds__(256, 6)
add_rmsnorm_kernel(float* __restrict__ res, const __nv_bfloat16* __restrict__ add,
                   const __nv_bfloat16* __restrict__ gain, __nv_bfloat16* __restrict__ out, int hidden, float eps,
                   const int* __restrict__ rows) {
  __shared__ float s_part[8];
  pdl_begin();
  const int b = blockIdx.x;
  const int t = rows ? rows[b] : b;
  if (t < 0) return;
  float* rrow = res + (size_t)t * hidden;
  const __nv_bfloat16* arow = add ? add + (size_t)t * hidden : nullptr;
  const int i0 = threadIdx.x * 4, step = 256 * 4;
  float4 v[kNormKeep];
  uint2 a[kNormKeep], gv[kNormKeep];
#pragma unroll
  for (int k = 0; k < kNormKeep; ++k) {
    const int i = i0 + k * step;
    v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    a[k] = gv[k] = make_uint2(0u, 0u);
    if (i < hidden) {
      v[k] = *reinterpret_cast<const float4*>(rrow + i);
      if (arow) a[k] = *reinterpret_cast<const uint2*>(arow + i);
      if (out) gv[k] = __ldg(reinterpret_cast<const uint2*>(gain + i));
    }
  }
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < kNormKeep; ++k) {
    const int i = i0 + k * step;
    if (arow && i < hidden) {
      v[k].x += bf16_lo(a[k].x); v[k].y += bf16_hi(a[k].x); v[k].z += bf16_lo(a[k].y); v[k].w += bf16_hi(a[k].y);
      *reinterpret_cast<float4*>(rrow + i) = v[k];
    }
    ss += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
  }
  for (int i = i0 + kNormKeep * step; i < hidden; i += step) {
    float4 w = *reinterpret_cast<const float4*>(rrow + i);
    if (arow) {
      const uint2 aw = *reinterpret_cast<const uint2*>(arow + i);
      w.x += bf16_lo(aw.x); w.y += bf16_hi(aw.x); w.z += bf16_lo(aw.y); w.w += bf16_hi(aw.y);
      *reinterpret_cast<float4*>(rrow + i) = w;
    }
    ss += w.x * w.x + w.y * w.y + w.z * w.z + w.w * w.w;
  }
  if (!out) return;
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) tot += s_part[w];
  const float inv = rsqrtf(tot / (float)hidden + eps);
  auto norm = [&](const float4& w, const uint2& g) {
    uint2 o;
    o.x = pack_bf16(w.x * inv * bf16_lo(g.x), w.y * inv * bf16_hi(g.x));
    o.y = pack_bf16(w.z * inv * bf16_lo(g.y), w.w * inv * bf16_hi(g.y));
    return o;
  };
  __nv_bfloat16* orow = out + (size_t)b * hidden;
#pragma unroll
  for (int k = 0; k < kNormKeep; ++k)
    if (i0 + k * step < hidden) *reinterpret_cast<uint2*>(orow + i0 + k * step) = norm(v[k], gv[k]);
  for (int i = i0 + kNormKeep * step; i < hidden; i += step)
    *reinterpret_cast<uint2*>(orow + i) = norm(*reinterpret_cast<const float4*>(rrow + i), *reinterpret_cast<const uint2*>(gain + i));
}

// In-place rotary embedding on v[T][n_h * 64], pairing (i, i + 32).
__global__ void __launch_bounds__(256)
rope_kernel(__nv_bfloat16* __restrict__ v, const int* __restrict__ pos, const float2* __restrict__ table, int T,
            int n_h) {
  pdl_begin();
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;  // (t, head, i)
  const long total = (long)T * n_h * 32;
  if (idx >= total) return;
  const int i = (int)(idx & 31);
  const long th = idx >> 5;
  const int t = (int)(th / n_h);
  __nv_bfloat16* p = v + th * 64;
  const float2 cs = table[pos[t] * 32 + i];
  const float a = __bfloat162float(p[i]), b = __bfloat162float(p[i + 32]);
  p[i] = __float2bfloat16_rn(a * cs.x - b * cs.y);
  p[i + 32] = __float2bfloat16_rn(b * cs.x + a * cs.y);
}

__global__ void __launch_bounds__(256)
swiglu_kernel(__nv_bfloat16* __restrict__ gate, const __nv_bfloat16* __restrict__ up, long n8) {
  pdl_begin();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n8) return;
  const uint4 gv = *reinterpret_cast<const uint4*>(gate + i * 8);
  const uint4 uv = *reinterpret_cast<const uint4*>(up + i * 8);
  const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w}, uw[4] = {uv.x, uv.y, uv.z, uv.w};
  uint32_t o[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float g0 = bf16_lo(gw[e]), g1 = bf16_hi(gw[e]);
    o[e] = pack_bf16(g0 / (1.f + __expf(-g0)) * bf16_lo(uw[e]), g1 / (1.f + __expf(-g1)) * bf16_hi(uw[e]));
  }
  *reinterpret_cast<uint4*>(gate + i * 8) = make_uint4(o[0], o[1], o[2], o[3]);
}

// Causal grouped-query attention inside each request, head_dim 64.
// Grid (query block of 64 rows, head, request); 4 warps x 16 query rows; keys and values staged 64 at a
// time, row-major [key][dim], in a two-buffer shared-memory ring filled with 16-byte asynchronous copies
// (the next tile is on its way while the current one is used); K fragments come from ldmatrix, V
// fragments from ldmatrix.trans (the transpose P V needs); online softmax in the exp2 domain.
constexpr int kAttPitch = 72;   // elements: 144-byte rows keep the 8 rows of an ldmatrix tile on distinct banks
__device__ __forceinline__ void cp_async_16(uint32_t dst, const void* src, bool valid) {
  const int n = valid ? 16 : 0;   // 0 source bytes: the 16 destination bytes are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_plain(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}

__global__ void __launch_bounds__(128)
attention_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k,
                 const __nv_bfloat16* __restrict__ v, const int* __restrict__ cu, __nv_bfloat16* __restrict__ out,
                 int n_heads, int n_kv_heads, float scale_log2, const float2* __restrict__ rope) {
  __shared__ __align__(16) uint16_t Ks[2][64 * kAttPitch];
  __shared__ __align__(16) uint16_t Vs[2][64 * kAttPitch];
  const int req = blockIdx.z, head = blockIdx.y, qb = blockIdx.x;
  const int t0 = cu[req], L = cu[req + 1] - t0;
  if (qb * 64 >= L) return;
  const int kvh = head / (n_heads / n_kv_heads);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int qd = n_heads * 64, kvd = n_kv_heads * 64;
  const int r0 = qb * 64 + warp * 16 + g, r1 = r0 + 8;  // query rows (within request) of this thread
  const int kv_end = min(L, qb * 64 + 64);
  const uint32_t ks_base = (uint32_t)__cvta_generic_to_shared(&Ks[0][0]);
  const uint32_t vs_base = (uint32_t)__cvta_generic_to_shared(&Vs[0][0]);
  constexpr uint32_t kBufBytes = 64 * kAttPitch * 2;

  auto stage = [&](int kb, int buf) {   // keys kb .. kb+63 -> buffer `buf`; rows past the request are zero-filled
#pragma unroll
    for (int i = tid; i < 64 * 8; i += 128) {
      const int key = i >> 3, ch = i & 7;
      const bool ok = kb + key < L;
      const size_t row = (size_t)(t0 + (ok ? kb + key : L - 1)) * kvd + kvh * 64 + ch * 8;
      const uint32_t off = (uint32_t)buf * kBufBytes + (uint32_t)(key * kAttPitch + ch * 8) * 2;
      cp_async_16(ks_base + off, k + row, ok);
      cp_async_16(vs_base + off, v + row, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  stage(0, 0);

  uint32_t qa[4][4];
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    const int d = ks * 16 + 2 * t;
    const __nv_bfloat16* p0 = q + (size_t)(t0 + r0) * qd + head * 64 + d;
    const __nv_bfloat16* p1 = q + (size_t)(t0 + r1) * qd + head * 64 + d;
    qa[ks][0] = (r0 < L) ? *reinterpret_cast<const uint32_t*>(p0) : 0u;
    qa[ks][1] = (r1 < L) ? *reinterpret_cast<const uint32_t*>(p1) : 0u;
    qa[ks][2] = (r0 < L) ? *reinterpret_cast<const uint32_t*>(p0 + 8) : 0u;
    qa[ks][3] = (r1 < L) ? *reinterpret_cast<const uint32_t*>(p1 + 8) : 0u;
  }
  if (rope != nullptr) {
    // rotary embedding of the query rows on the fly (pairing (d, d + 32): k-steps ks and ks + 2 of the same
    // thread; position = row index inside the request), rounded to bf16 as the stand-alone kernel does
#pragma unroll
    for (int ks = 0; ks < 2; ++ks)
#pragma unroll
      for (int idx = 0; idx < 4; ++idx) {
        const int row = (idx & 1) ? r1 : r0;
        if (row < L) {
          const int d0 = ks * 16 + 2 * t + ((idx & 2) ? 8 : 0);
          const float4 cc = __ldg(reinterpret_cast<const float4*>(rope + (size_t)row * 32 + d0));   // d0 is even
          const float2 c0 = make_float2(cc.x, cc.y), c1 = make_float2(cc.z, cc.w);
          const uint32_t lo = qa[ks][idx], hi = qa[ks + 2][idx];
          const float a0 = bf16_lo(lo), a1 = bf16_hi(lo), b0 = bf16_lo(hi), b1 = bf16_hi(hi);
          qa[ks][idx] = pack_bf16(a0 * c0.x - b0 * c0.y, a1 * c1.x - b1 * c1.y);
          qa[ks + 2][idx] = pack_bf16(b0 * c0.x + a0 * c0.y, b1 * c1.x + a1 * c1.y);
        }
      }
  }
  float o[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) o[i][j] = 0.f;
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
  // ldmatrix lane roles: lane l addresses row (l & 7) of matrix (l >> 3)
  const int lm_row = lane & 7, lm_mat = lane >> 3;
  for (int kb = 0, it = 0; kb < kv_end; kb += 64, ++it) {
    const int buf = it & 1;
    __syncthreads();                       // the other buffer's readers (previous tile) are done
    if (kb + 64 < kv_end) {
      stage(kb + 64, buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();                       // every thread's copies of this tile have landed
    const uint32_t kbuf = ks_base + (uint32_t)buf * kBufBytes, vbuf = vs_base + (uint32_t)buf * kBufBytes;
    float s[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
#pragma unroll
      for (int j = 0; j < 4; ++j) s[nt][j] = 0.f;
#pragma unroll
      for (int kp = 0; kp < 2; ++kp) {
        // matrices: keys nt*8.., dim chunks kp*32 + {0, 8, 16, 24}  ->  (b0, b1) of k-step 2kp and of 2kp+1
        uint32_t b0, b1, b2, b3;
        ldmatrix_x4_plain(kbuf + (uint32_t)((nt * 8 + lm_row) * kAttPitch + kp * 32 + lm_mat * 8) * 2, b0, b1, b2, b3);
        mma_bf16_16816(s[nt], qa[2 * kp][0], qa[2 * kp][1], qa[2 * kp][2], qa[2 * kp][3], b0, b1);
        mma_bf16_16816(s[nt], qa[2 * kp + 1][0], qa[2 * kp + 1][1], qa[2 * kp + 1][2], qa[2 * kp + 1][3], b2, b3);
      }
    }
    // scale, causal mask, running max
    float mx0 = m0, mx1 = m1;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int key = kb + nt * 8 + 2 * t + (j & 1);
        const int row = (j < 2) ? r0 : r1;
        const float val = (key <= row && key < L) ? s[nt][j] * scale_log2 : -INFINITY;
        s[nt][j] = val;
        if (j < 2) mx0 = fmaxf(mx0, val); else mx1 = fmaxf(mx1, val);
      }
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
    const float base0 = (mx0 == -INFINITY) ? 0.f : mx0, base1 = (mx1 == -INFINITY) ? 0.f : mx1;
    const float corr0 = exp2f(m0 - base0), corr1 = exp2f(m1 - base1);  // m = -inf -> 0
    m0 = mx0; m1 = mx1;
    l0 *= corr0; l1 *= corr1;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      o[i][0] *= corr0; o[i][1] *= corr0; o[i][2] *= corr1; o[i][3] *= corr1;
    }
    uint32_t pa[4][4];  // P as A fragments: 4 k16 steps over the 64 keys
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const float p0 = exp2f(s[nt][0] - base0), p1 = exp2f(s[nt][1] - base0);
      const float p2 = exp2f(s[nt][2] - base1), p3 = exp2f(s[nt][3] - base1);
      l0 += p0 + p1;
      l1 += p2 + p3;
      const int ks = nt >> 1, hi = nt & 1;
      pa[ks][hi * 2 + 0] = pack_bf16(p0, p1);
      pa[ks][hi * 2 + 1] = pack_bf16(p2, p3);
    }
#pragma unroll
    for (int dp = 0; dp < 4; ++dp)
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        // matrices: keys ks*16 + {0, 8} x dims (2dp)*8.., then the same keys x dims (2dp+1)*8..; transposed on load
        uint32_t b0, b1, b2, b3;
        ldmatrix_x4_trans(vbuf + (uint32_t)((ks * 16 + (lm_mat & 1) * 8 + lm_row) * kAttPitch + (2 * dp + (lm_mat >> 1)) * 8) * 2,
                          b0, b1, b2, b3);
        mma_bf16_16816(o[2 * dp], pa[ks][0], pa[ks][1], pa[ks][2], pa[ks][3], b0, b1);
        mma_bf16_16816(o[2 * dp + 1], pa[ks][0], pa[ks][1], pa[ks][2], pa[ks][3], b2, b3);
      }
  }
  l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
  l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
  const float i0 = l0 > 0.f ? 1.f / l0 : 0.f, i1 = l1 > 0.f ? 1.f / l1 : 0.f;
#pragma unroll
  for (int dt = 0; dt < 8; ++dt) {
    const int d = head * 64 + dt * 8 + 2 * t;
    if (r0 < L) *reinterpret_cast<uint32_t*>(out + (size_t)(t0 + r0) * qd + d) = pack_bf16(o[dt][0] * i0, o[dt][1] * i0);
    if (r1 < L) *reinterpret_cast<uint32_t*>(out + (size_t)(t0 + r1) * qd + d) = pack_bf16(o[dt][2] * i1, o[dt][3] * i1);
  }
}

struct DecoderWorkspace {
  float* res; __nv_bfloat16 *xn, *q, *k, *v, *att, *o, *gate, *up, *xlast;
  __nv_bfloat16* wq[3];   // dequantised weights of the projection group in flight (quantised base only)
  int *pos, *token_expert, *last_row;
  float2* rope;
  void* plan; size_t plan_bytes;
  void* lora; size_t lora_bytes;
  size_t total;
};

static DecoderWorkspace carve(const moin_model* m, int R, int T, int max_seqlen, void* base) {
  DecoderWorkspace w;
  char* p = reinterpret_cast<char*>(base);
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += align_up(bytes, 256); return base ? (void*)(p + o) : nullptr; };
  const size_t H = m->hidden, qd = (size_t)m->n_heads * m->head_dim, kvd = (size_t)m->n_kv_heads * m->head_dim;
  const size_t F = m->ffn, TT = T;
  w.res = (float*)take(TT * H * 4);
  w.xn = (__nv_bfloat16*)take(TT * (H > qd ? H : qd) * 2);
  w.q = (__nv_bfloat16*)take(TT * qd * 2);
  w.k = (__nv_bfloat16*)take(TT * kvd * 2);
  w.v = (__nv_bfloat16*)take(TT * kvd * 2);
  w.att = (__nv_bfloat16*)take(TT * qd * 2);
  w.o = (__nv_bfloat16*)take(TT * H * 2);
  w.gate = (__nv_bfloat16*)take(TT * F * 2);
  w.up = (__nv_bfloat16*)take(TT * F * 2);
  w.xlast = (__nv_bfloat16*)take((size_t)R * H * 2);
  for (int i = 0; i < 3; ++i) w.wq[i] = m->W8 ? (__nv_bfloat16*)take(F * (H > qd ? H : qd) * 2) : nullptr;
  w.pos = (int*)take(TT * 4);
  w.token_expert = (int*)take(TT * 4);
  w.last_row = (int*)take((size_t)R * 4 + 4);
  w.rope = (float2*)take((size_t)(max_seqlen > 0 ? max_seqlen : T) * 32 * sizeof(float2));
  w.plan_bytes = moin_plan_bytes(T, m->E > 0 ? m->E : 1);
  w.plan = take(w.plan_bytes);
  size_t lb = 0;
  int r = 8;
  if (m->pools) r = m->pools[0].r;
  auto one = [&](size_t din, size_t dout) { return moin_lora_linear_workspace_bytes(T, (int)din, (int)dout, r); };
  const size_t groups[5] = {one(H, qd) + 2 * one(H, kvd), one(qd, H), 2 * one(H, F), one(F, H), one(H, (size_t)m->vocab)};
  for (size_t b : groups) lb = b > lb ? b : lb;
  w.lora_bytes = lb;
  w.lora = take(lb);
  w.total = off;
  return w;
}

// Tiles or segments for T tokens of R requests, one expert each?  Segments read an adapter again for every eight tokens: what
// they cost over tiles grows with the tokens.  Tiles pay a pass over a row tile for every run in it (about a request; the lower
// the rank, the less segments lose to make up for it), a fixed part a launch that weighs less the wider the model, and on an 8-bit
// base the conversion of all weights.  Measured on 2400 forwards of hidden size 2048 (14 to 260 tokens a request, equal and ragged,
// ranks 8 to 128, both bases, some requests without an adapter): over the better of the two 0.3 % a forward, at the worst 21 %
// (tiles for requests of about 32 tokens, five of which fall into many row tiles and cost a second one); always tiles 25 %, always
// segments 18 %, tiles from 64 tokens a request on 10 %.  880 of sizes 512 to 4096: 0.9 %, 26 %.  Segments and tiles meet, ranks 16; 64, in all
// tokens: requests of 140 410; 320, of 64 520; 330, of 48 560; 350, of 36 1300; 600, of 28 beyond 2048; 1000, on the 8-bit base of 64
// 790; 540, in models of half the width of 64 650; 510.
static bool forward_tiles(const moin_model* m, int T, int R) {
  int r = 8;
  for (int p = 0; p < 7 && m->n_layers > 0; ++p) r = m->pools[p].r > r ? m->pools[p].r : r;
  const int fixed = 620000 / (m->hidden > 1024 ? m->hidden : 1024);
  const int convert = m->W8 ? (r < 130 ? 330 - 2 * r : 70) : 0;
  return T >= fixed + convert + (long long)(14 + 160 / r) * R;
}

}  // namespace moin

using namespace moin;

extern "C" size_t moin_decoder_workspace_bytes(const moin_model* model, int32_t R, int32_t T) {
  if (!model || R < 0 || T < 0) return 0;
  return carve(model, R, T, T, nullptr).total + 256;
}

static moin_status decoder_forward_impl(const moin_model* m, const int32_t* tokens, const int32_t* cu_seqlens,
                                        const int32_t* req_expert, const int32_t* token_expert_in, int32_t R,
                                        int32_t T, int32_t max_seqlen, void* logits, int32_t logits_mode,
                                        const moin_decoder_taps* taps, void* workspace, size_t workspace_bytes,
                                        moin_stream stream) {
  if (!m || R < 0 || T < 0) return MOIN_ERR_INVALID_ARG;
  if (R == 0 || T == 0) return MOIN_OK;
  if (!cu_seqlens || !m->W || !m->attn_norm || !m->mlp_norm || !m->final_norm) return MOIN_ERR_INVALID_ARG;
  if (m->head_dim != 64 || m->n_kv_heads < 1 || (m->n_heads % m->n_kv_heads) != 0) return MOIN_ERR_BAD_SHAPE;
  if ((m->hidden % 64) != 0 || (m->ffn % 64) != 0 || (m->vocab % 8) != 0) return MOIN_ERR_BAD_SHAPE;
  if (logits_mode < MOIN_LOGITS_ALL || logits_mode > MOIN_LOGITS_NONE) return MOIN_ERR_INVALID_ARG;
  if (logits_mode != MOIN_LOGITS_NONE && (!logits || !m->lm_head)) return MOIN_ERR_INVALID_ARG;
  if (max_seqlen < 1 || max_seqlen > T) max_seqlen = T;
  const int lb = taps ? taps->layer_begin : 0, le = taps ? taps->layer_end : m->n_layers;
  if (lb < 0 || le > m->n_layers || lb > le) return MOIN_ERR_INVALID_ARG;
  const bool from_hidden = taps && taps->hidden_in;
  if (!from_hidden && (!tokens || !m->embed)) return MOIN_ERR_INVALID_ARG;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return MOIN_ERR_WORKSPACE;
  DecoderWorkspace w = carve(m, R, T, T, workspace);
  if (workspace_bytes < w.total) return MOIN_ERR_WORKSPACE;
  HostState* hs;
  moin_status st = host_state(&hs);
  if (st) return st;
  cudaStream_t s = (cudaStream_t)stream;
  const int H = m->hidden, nh = m->n_heads, nkv = m->n_kv_heads, F = m->ffn;
  const int qd = nh * 64, kvd = nkv * 64;

  { ProfScope prof(MOIN_K_GLUE, 2, s);
  launch_pdl(token_meta_kernel, R, 256, 0, s, cu_seqlens, req_expert, token_expert_in, R, w.pos, w.token_expert, w.last_row);
  launch_pdl(rope_table_kernel, (max_seqlen * 32 + 255) / 256, 256, 0, s, w.rope, max_seqlen, 32, (double)m->rope_base); }
  moin_plan plan;
  memset(&plan, 0, sizeof(plan));
  const bool lora = m->pools != nullptr && (req_expert != nullptr || token_expert_in != nullptr);
  if (lora) {
    plan.buffer = w.plan; plan.buffer_bytes = w.plan_bytes; plan.T = T; plan.E = m->E;
    // one expert per request: the run lengths are the request lengths; one per token: they depend on the ids, so
    // the plan decides after it has grouped them (reads its header back: one synchronisation of the stream)
    plan.mode = token_expert_in ? MOIN_PLAN_AUTO : (forward_tiles(m, T, R) ? MOIN_PLAN_TILES : MOIN_PLAN_SEGMENTS);
    st = moin_plan_build(w.token_expert, &plan, stream);
    if (st) return st;
    // Ids that change no more often than the requests do (as many tiles as R runs have at the most): the rule of one expert per
    // request, so that the same batch takes the same kernels however it is given.  Else the plan's own choice.
    if (token_expert_in && plan.n_tiles <= R + T / kTileRows) plan.mode = forward_tiles(m, T, R) ? MOIN_PLAN_TILES : MOIN_PLAN_SEGMENTS;
  }
  if (from_hidden) {
    cudaError_t e = cudaMemcpyAsync(w.res, taps->hidden_in, (size_t)T * H * 4, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return record_cuda(e);
  } else {
    ProfScope prof(MOIN_K_GLUE, 1, s);
    launch_pdl(embed_kernel, T, 256, 0, s, tokens, (const __nv_bfloat16*)m->embed, H, m->vocab, w.res);
  }
  // weights of the projections p0 .. p0 + n - 1, which share d_in: the caller's bf16 matrices, or - quantised base - their
  // codes dequantised into the scratch slots by one launch on the call's stream (the group before has read its slots
  // by then)
  auto weights = [&](int layer, int p0, int n, int d_in, const int* d_out, const void** W) -> moin_status {
    DequantJobs dq = {};
    for (int j = 0; j < n; ++j) {
      const int i = layer * 7 + p0 + j;
      W[j] = m->W[i];
      if (!m->W8 || !m->W8[i]) continue;
      if (!m->W_scale || !m->W_scale[i]) return MOIN_ERR_INVALID_ARG;
      if (!aligned16(m->W8[i])) return MOIN_ERR_MISALIGNED;
      dq.codes[dq.n] = (const uint2*)m->W8[i];
      dq.scale[dq.n] = m->W_scale[i];
      dq.out[dq.n] = (uint4*)w.wq[j];
      dq.row_end[dq.n] = (dq.n ? dq.row_end[dq.n - 1] : 0) + d_out[j];
      W[j] = w.wq[j];
      ++dq.n;
    }
    return dq.n ? launch_dequant(dq, d_in, s) : MOIN_OK;
  };
  // projections of a block that read the same input and do not depend on one another go out as one group, right behind a norm,
  // the attention or the SwiGLU, which wait before they let it start: its GEMM may read the caller's weights at once (w_early)
  auto proj_group = [&](int layer, int p0, int n, const void* in, int d_in, const int* d_out, void* const* outs) -> moin_status {
    // few tokens in short segments: the GEMM converts the codes itself (gemm_decode.cu has both sides' times)
    bool coded = m->W8 && decode_fp8_supported(hs, T, lora) && (!lora || plan.mode == MOIN_PLAN_SEGMENTS);
    for (int j = 0; j < n && coded; ++j) coded = m->W8[layer * 7 + p0 + j] && m->W_scale && m->W_scale[layer * 7 + p0 + j];
    if (coded) {
      moin_lora_job jobs[MOIN_MAX_GROUP];
      DecodeGemmJob gemm[MOIN_MAX_GROUP];
      for (int j = 0; j < n; ++j) {
        const int i = layer * 7 + p0 + j;
        if (!aligned16(m->W8[i])) return MOIN_ERR_MISALIGNED;
        if (lora) jobs[j] = {in, m->W8[i], &m->pools[i], outs[j]};
        else gemm[j] = {(const __nv_bfloat16*)in, m->W8[i], (__nv_bfloat16*)outs[j], nullptr, d_in, d_out[j], m->W_scale[i]};
      }
      const ForwardGroup fwd = {m->W_scale + layer * 7 + p0, true};
      if (lora) return lora_linear_group(&plan, jobs, n, &fwd, m->lora_scale, w.lora, w.lora_bytes, stream);
      ProfScope prof(MOIN_K_GEMM_TC, 1, s);
      return launch_decode_gemm(hs, gemm, n, T, false, true, s);
    }
    const void* W[MOIN_MAX_GROUP];
    moin_status e = weights(layer, p0, n, d_in, d_out, W);
    bool converted = false;   // by the kernel right before
    for (int j = 0; j < n; ++j) converted = converted || W[j] != m->W[layer * 7 + p0 + j];
    if (e) return e;
    moin_lora_job jobs[MOIN_MAX_GROUP];
    for (int i = 0; i < n; ++i) {
      if (!lora) {
        e = moin_lora_linear(nullptr, in, W[i], nullptr, 0.f, T, d_in, d_out[i], outs[i], w.lora, w.lora_bytes, stream);
        if (e) return e;
      } else {
        jobs[i] = {in, W[i], &m->pools[layer * 7 + p0 + i], outs[i]};
      }
    }
    const ForwardGroup fwd = {nullptr, !converted};
    return lora ? lora_linear_group(&plan, jobs, n, &fwd, m->lora_scale, w.lora, w.lora_bytes, stream) : MOIN_OK;
  };
  const float scale_log2 = 1.4426950408889634f / sqrtf(64.f);
  const __nv_bfloat16* pending = nullptr;
  for (int l = lb; l < le; ++l) {
    { ProfScope prof(MOIN_K_GLUE, 1, s);
      launch_pdl(add_rmsnorm_kernel, T, 256, 0, s, w.res, pending, (const __nv_bfloat16*)m->attn_norm[l], w.xn, H, m->rms_eps, nullptr); }
    {
      const int dout[3] = {qd, kvd, kvd};
      void* const outs[3] = {w.q, w.k, w.v};
      if ((st = proj_group(l, 0, 3, w.xn, H, dout, outs))) return st;
    }
    // rotary embedding: the keys are rotated in place once (every query head and every later query reads them);
    // the queries are rotated inside the attention kernel as it loads them
    { ProfScope prof(MOIN_K_GLUE, 1, s);
      launch_pdl(rope_kernel, (int)(((long)T * nkv * 32 + 255) / 256), 256, 0, s, w.k, w.pos, w.rope, T, nkv); }
    if (hs->gemm_impl != 1 && attention_tc_supported(nh, nkv, m->head_dim)) {   // tcgen05 kernel
      ProfScope prof(MOIN_K_ATTENTION, 1, s);
      if ((st = launch_attention_tc(hs, w.q, w.k, w.v, cu_seqlens, w.att, w.rope, R, T, max_seqlen, nh, nkv,
                                    scale_log2, s)))
        return st;
    } else {   // warp-MMA kernel: other head groupings, or forced by MOIN_OPT_GEMM_IMPL = 1
      ProfScope prof(MOIN_K_ATTENTION, 1, s);
      attention_kernel<<<dim3((max_seqlen + 63) / 64, nh, R), 128, 0, s>>>(w.q, w.k, w.v, cu_seqlens, w.att, nh, nkv, scale_log2,
                                                                         w.rope);
    }
    void* const o_out[1] = {w.o};   // (also the down projection's)
    if ((st = proj_group(l, 3, 1, w.att, qd, &H, o_out))) return st;
    { ProfScope prof(MOIN_K_GLUE, 1, s);
      launch_pdl(add_rmsnorm_kernel, T, 256, 0, s, w.res, w.o, (const __nv_bfloat16*)m->mlp_norm[l], w.xn, H, m->rms_eps, nullptr); }
    const int dout_f[2] = {F, F};
    const moin_pool* mlp_pools = lora ? &m->pools[l * 7 + 4] : nullptr;
    if (swiglu_supported(hs, lora ? &plan : nullptr, mlp_pools, T, H, F)) {   // long runs: the product in the GEMM's epilogue
      const void* W[2];
      if ((st = weights(l, 4, 2, H, dout_f, W))) return st;
      const moin_lora_job jobs[2] = {{w.xn, W[0], mlp_pools, w.gate}, {w.xn, W[1], lora ? mlp_pools + 1 : nullptr, w.up}};
      if ((st = lora_swiglu(hs, lora ? &plan : nullptr, jobs, m->lora_scale, T, H, F, w.lora, w.lora_bytes, s)))
        return st;
    } else {
      void* const outs[2] = {w.gate, w.up};
      if ((st = proj_group(l, 4, 2, w.xn, H, dout_f, outs))) return st;
      ProfScope prof(MOIN_K_GLUE, 1, s);
      launch_pdl(swiglu_kernel, (int)(((long)T * F / 8 + 255) / 256), 256, 0, s, w.gate, w.up, (long)T * F / 8);
    }
    if ((st = proj_group(l, 6, 1, w.gate, F, &H, o_out))) return st;
    pending = w.o;
  }
  if (pending) { ProfScope prof(MOIN_K_GLUE, 1, s);
    launch_pdl(add_rmsnorm_kernel, T, 256, 0, s, w.res, pending, nullptr, nullptr, H, m->rms_eps, nullptr); }
  if (taps && taps->hidden_out) {
    cudaError_t e = cudaMemcpyAsync(taps->hidden_out, w.res, (size_t)T * H * 4, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return record_cuda(e);
  }
  if (logits_mode == MOIN_LOGITS_ALL) {
    { ProfScope prof(MOIN_K_GLUE, 1, s);
      launch_pdl(add_rmsnorm_kernel, T, 256, 0, s, w.res, nullptr, (const __nv_bfloat16*)m->final_norm, w.xn, H, m->rms_eps, nullptr); }
    st = moin_lora_linear(nullptr, w.xn, m->lm_head, nullptr, 0.f, T, H, m->vocab, logits, w.lora, w.lora_bytes, stream);
    if (st) return st;
  } else if (logits_mode == MOIN_LOGITS_LAST) {
    cudaError_t e = cudaMemsetAsync(w.xlast, 0, (size_t)R * H * 2, s);
    if (e != cudaSuccess) return record_cuda(e);
    { ProfScope prof(MOIN_K_GLUE, 1, s);
      launch_pdl(add_rmsnorm_kernel, R, 256, 0, s, w.res, nullptr, (const __nv_bfloat16*)m->final_norm, w.xlast, H, m->rms_eps, w.last_row); }
    st = moin_lora_linear(nullptr, w.xlast, m->lm_head, nullptr, 0.f, R, H, m->vocab, logits, w.lora, w.lora_bytes, stream);
    if (st) return st;
  }
  return record_cuda(cudaGetLastError());
}

extern "C" moin_status moin_decoder_forward(const moin_model* m, const int32_t* tokens, const int32_t* cu_seqlens,
                                            const int32_t* req_expert, int32_t R, int32_t T, int32_t max_seqlen,
                                            void* logits, int32_t logits_mode, const moin_decoder_taps* taps,
                                            void* workspace, size_t workspace_bytes, moin_stream stream) {
  return decoder_forward_impl(m, tokens, cu_seqlens, req_expert, nullptr, R, T, max_seqlen, logits, logits_mode, taps,
                              workspace, workspace_bytes, stream);
}

extern "C" moin_status moin_decoder_forward_per_token(const moin_model* m, const int32_t* tokens,
                                                      const int32_t* cu_seqlens, const int32_t* token_expert, int32_t R,
                                                      int32_t T, int32_t max_seqlen, void* logits, int32_t logits_mode,
                                                      const moin_decoder_taps* taps, void* workspace,
                                                      size_t workspace_bytes, moin_stream stream) {
  if (!token_expert) return MOIN_ERR_INVALID_ARG;
  return decoder_forward_impl(m, tokens, cu_seqlens, nullptr, token_expert, R, T, max_seqlen, logits, logits_mode, taps,
                              workspace, workspace_bytes, stream);
}

extern "C" moin_status moin_dequant_fp8(const void* codes, const float* scale, int32_t d_out, int32_t d_in, void* W,
                                        moin_stream stream) {
  if (!codes || !scale || !W || d_out < 0 || d_in < 0) return MOIN_ERR_INVALID_ARG;
  if ((d_in % 16) != 0) return MOIN_ERR_BAD_SHAPE;
  if (!aligned16(codes) || !aligned16(W)) return MOIN_ERR_MISALIGNED;
  if (d_out == 0 || d_in == 0) return MOIN_OK;
  HostState* hs;
  moin_status st = host_state(&hs);
  if (st) return st;
  DequantJobs jobs = {};
  jobs.n = 1;
  jobs.codes[0] = (const uint2*)codes; jobs.scale[0] = scale; jobs.out[0] = (uint4*)W; jobs.row_end[0] = d_out;
  return launch_dequant(jobs, d_in, (cudaStream_t)stream);
}
