// Kernels of the teacher-forced forward of Section 3.3 (Eq. 6): the whole target of every sequence in one
// pass, every token attending to the tokens the dependency rule of Section 3.2 lets it see - evaluated per
// (query, key) pair from (subsequence, timestamp) and never stored as a mask - and to the sequence's context.  Off the decode
// hot path (scoring, perplexity).
#include "mma_tile.cuh"
#include "pd_internal.h"

namespace pd {

namespace {

// Self-attention of up to 128 query rows of one sequence and head (one CTA; W warps of 16 rows each) over 64-key tiles that all
// warps share: a three-slot ring filled with 16-byte asynchronous copies (rows of 128 bytes, chunks swizzled), scores and
// P.V on mma.sync, online softmax in the log2 domain; a warp owns its rows, so nothing is merged.  The keys are the sequence's own
// target rows, with the dependency rule and the T5 bias applied to the accumulator fragment; the key walk ends at the first tile of a
// later subsequence.
// With a bias, whose table bounds the timestamps, a row's subsequence and timestamp share a word (8 and 24 bits) with a guard bit above each: one
// subtraction tells whether a query sees a key - both guard bits stand - and the bias is read whatever it tells, at a place that is always in the
// table, so that no pair branches.  Without one the two stand by themselves, and the signs of two differences tell.
// What bounds it: the mask and the bias, evaluated per pair.  11.5 k rows of 32 sequences, 16 heads, per layer: 203 us in groups of 32 rows
// (every group reads its keys again), 160 us with 16 rows per warp, two comparisons and a branch per pair and the tiles to walk found by
// search, 234 us with 32 (the mask needs the registers); 96 us here.  Where 128-row blocks would leave SMs without one, 64-row blocks.
constexpr int TK = 64, TSLOTS = 3, TMAXD = 640;
constexpr int TSLOT_BYTES = TK * 256;            // 64 key rows, then 64 value rows
constexpr int TATTN_SMEM = TSLOTS * TSLOT_BYTES + 128;

__device__ __forceinline__ void t_cp_async16(uint32_t dst, const void *src, bool on) {
  const int n = on ? 16 : 0;                     // 0 source bytes: the destination is zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void t_cp_async8(uint32_t dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
constexpr uint32_t kSees = 0x80800000u;          // guard bits above the timestamp (24 bits) and the subsequence (8 bits)

template <int W, bool BIAS>
__global__ void __launch_bounds__(W * 32, 16 / W) teacher_self_kernel(DenseAttnArgs a) {
  using namespace mt;
  constexpr int TT = W * 32;
  extern __shared__ uint8_t t_raw[];
  __shared__ __align__(16) int2 key_s[TSLOTS][TK];      // BIAS: (subsequence << 24 | timestamp, 4 x position), else (subsequence, timestamp)
  __shared__ float bias_s[BIAS ? TMAXD : 1];
  const int grp = blockIdx.x, h = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tig = lane & 3;
  const int q0 = a.grp_row0[grp], nq = a.grp_n[grp];
  const uint32_t base = (smem_u32(t_raw) + 127u) & ~127u;
  const size_t ld = 3 * (size_t)a.d;
  const int k0 = a.grp_key_row0[grp], nk = a.grp_keys[grp];
  const __nv_bfloat16 *kp = a.q + (size_t)k0 * ld + a.d + (size_t)h * kDh, *vp = kp + a.d;      // row 0 of this head's keys and values
  if (BIAS)
    for (int dd = tid; dd < a.n_dist; dd += TT) bias_s[dd] = a.bias_tab[(size_t)h * a.n_dist + dd];

  auto fetch = [&](int tile) {
    const int slot = tile % TSLOTS, first = tile * TK;
    const uint32_t dst = base + slot * TSLOT_BYTES;
#pragma unroll
    for (int i = 0; i < TK * 16 / TT; ++i) {     // chunks 0-7 of a row: keys, 8-15: values
      const int c = tid + i * TT, r = c >> 4, p = c & 15;
      const bool on = first + r < nk;            // absent keys: zero rows
      const __nv_bfloat16 *src = (p < 8 ? kp : vp) + (on ? (size_t)(first + r) * ld : 0) + (p & 7) * 8;
      t_cp_async16(dst + (p >> 3) * (TK * 128) + swz(r, p & 7), src, on);
    }
    for (int i = tid; i < TK; i += TT) {
      if (first + i < nk) t_cp_async8(smem_u32(&key_s[slot][i]), a.row_key + k0 + first + i);
      else key_s[slot][i] = make_int2(BIAS ? 0x7f << 24 : 0x7fffffff, 0);      // a subsequence no row reaches
    }
  };
  const int n_tiles = a.grp_tiles[grp];          // keys are sorted by subsequence: nothing of a later one than the block's last row's is visible
#pragma unroll
  for (int t = 0; t < TSLOTS - 1; ++t) {
    if (t < n_tiles) fetch(t);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // this warp's query rows: 16 warp + g, + 8
  const int w0 = warp * 16;
  const int r_lo = w0 + g, r_hi = r_lo + 8;
  const __nv_bfloat16 *q_lo = a.q + (size_t)(q0 + r_lo) * ld + (size_t)h * kDh + 2 * tig, *q_hi = q_lo + 8 * ld;
  uint32_t qf[4][4];
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) {
    qf[kk][0] = r_lo < nq ? *reinterpret_cast<const uint32_t *>(q_lo + kk * 16) : 0u;
    qf[kk][1] = r_hi < nq ? *reinterpret_cast<const uint32_t *>(q_hi + kk * 16) : 0u;
    qf[kk][2] = r_lo < nq ? *reinterpret_cast<const uint32_t *>(q_lo + kk * 16 + 8) : 0u;
    qf[kk][3] = r_hi < nq ? *reinterpret_cast<const uint32_t *>(q_hi + kk * 16 + 8) : 0u;
  }
  // BIAS: subsequence and timestamp of the rows under their guard bits (no row: sees nothing), 4 x position; else the two by themselves
  const int2 none = make_int2(BIAS ? (int)((0x7fu << 24) - kSees) : -1, 0);
  const int2 k_lo = r_lo < nq ? a.row_key[q0 + r_lo] : none, k_hi = r_hi < nq ? a.row_key[q0 + r_hi] : none;
  const uint32_t qk[2] = {(uint32_t)k_lo.x + (BIAS ? kSees : 0u), (uint32_t)k_hi.x + (BIAS ? kSees : 0u)};
  const int qp[2] = {k_lo.y, k_hi.y};
  auto subsequence = [](int x) { return BIAS ? x >> 24 : x; };
  const int warp_i_max = w0 < nq ? subsequence(a.row_key[q0 + min(w0 + 15, nq - 1)].x) : -1;
  TileAcc A;
  A.clear();
  const float sl2 = a.scale_log2e;

  for (int tile = 0; tile < n_tiles; ++tile) {
    asm volatile("cp.async.wait_group %0;" ::"n"(TSLOTS - 2) : "memory");
    __syncthreads();                             // tile landed for everybody; everybody is through with the tile before
    if (tile + TSLOTS - 1 < n_tiles) fetch(tile + TSLOTS - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int slot = tile % TSLOTS;
    if (w0 >= nq || subsequence(key_s[slot][0].x) > warp_i_max) continue;      // no row of this warp sees the tile
    const uint32_t kbase = base + slot * TSLOT_BYTES, vbase = kbase + TK * 128;
    float sc[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
#pragma unroll
      for (int kq = 0; kq < 2; ++kq) {
        uint32_t b0, b1, b2, b3;
        ldsm_x4(kbase + swz(nt * 8 + (lane & 7), kq * 4 + (lane >> 3)), b0, b1, b2, b3);
        mma_bf16(sc[nt], qf[2 * kq][0], qf[2 * kq][1], qf[2 * kq][2], qf[2 * kq][3], b0, b1);
        mma_bf16(sc[nt], qf[2 * kq + 1][0], qf[2 * kq + 1][1], qf[2 * kq + 1][2], qf[2 * kq + 1][3], b2, b3);
      }
    }
    // ---- scale, the dependency rule per pair (i' <= i and tau' <= tau), bias on the Manhattan distance (log2 domain).  A pair that is not
    // visible may have any distance down to minus a position: it reads the table's start, and the value is dropped.
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const int4 k2 = *reinterpret_cast<const int4 *>(&key_s[slot][nt * 8 + 2 * tig]);
#pragma unroll
      for (int kx = 0; kx < 2; ++kx)
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const uint32_t di = qk[hh] - (uint32_t)(kx ? k2.z : k2.x);
          const bool vis = BIAS ? (di & kSees) == kSees : ((int)di | (qp[hh] - (kx ? k2.w : k2.y))) >= 0;
          float v = sc[nt][2 * hh + kx] * sl2;
          if (BIAS) v += *reinterpret_cast<const float *>(reinterpret_cast<const char *>(bias_s) + max(qp[hh] - (kx ? k2.w : k2.y), 0));
          sc[nt][2 * hh + kx] = vis ? v : -INFINITY;
        }
    }
    uint32_t pf[4][4];
    float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      mx0 = fmaxf(mx0, fmaxf(sc[nt][0], sc[nt][1]));
      mx1 = fmaxf(mx1, fmaxf(sc[nt][2], sc[nt][3]));
    }
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1)); mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1)); mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
    const float mn0 = fmaxf(A.m0, mx0), mn1 = fmaxf(A.m1, mx1);
    const float ref0 = mn0 == -INFINITY ? 0.f : mn0, ref1 = mn1 == -INFINITY ? 0.f : mn1;
    const float c0 = ex2f(A.m0 - ref0), c1 = ex2f(A.m1 - ref1);
    A.m0 = mn0; A.m1 = mn1;
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const float p0 = ex2f(sc[nt][0] - ref0), p1 = ex2f(sc[nt][1] - ref0);
      const float p2 = ex2f(sc[nt][2] - ref1), p3 = ex2f(sc[nt][3] - ref1);
      s0 += p0 + p1; s1 += p2 + p3;
      pf[nt >> 1][(nt & 1) * 2] = pack_bf16(p0, p1);
      pf[nt >> 1][(nt & 1) * 2 + 1] = pack_bf16(p2, p3);
    }
    A.l0 = A.l0 * c0 + s0; A.l1 = A.l1 * c1 + s1;
    if (__any_sync(0xffffffffu, c0 != 1.f || c1 != 1.f)) {   // some row's running maximum moved
#pragma unroll
      for (int dn = 0; dn < 8; ++dn) { A.o[dn][0] *= c0; A.o[dn][1] *= c0; A.o[dn][2] *= c1; A.o[dn][3] *= c1; }
    }
    // ---- O += P (16 x 64 keys) . V (64 keys x 64)
#pragma unroll
    for (int kq = 0; kq < 4; ++kq) {
      const int key = kq * 16 + ((lane >> 3) & 1) * 8 + (lane & 7);
#pragma unroll
      for (int dp = 0; dp < 4; ++dp) {
        uint32_t b0, b1, b2, b3;
        ldsm_x4_t(vbase + swz(key, dp * 2 + (lane >> 4)), b0, b1, b2, b3);
        mma_bf16(A.o[2 * dp], pf[kq][0], pf[kq][1], pf[kq][2], pf[kq][3], b0, b1);
        mma_bf16(A.o[2 * dp + 1], pf[kq][0], pf[kq][1], pf[kq][2], pf[kq][3], b2, b3);
      }
    }
  }
  A.l0 += __shfl_xor_sync(0xffffffffu, A.l0, 1); A.l0 += __shfl_xor_sync(0xffffffffu, A.l0, 2);
  A.l1 += __shfl_xor_sync(0xffffffffu, A.l1, 1); A.l1 += __shfl_xor_sync(0xffffffffu, A.l1, 2);
  const float i0 = 1.f / A.l0, i1 = 1.f / A.l1;
  __nv_bfloat16 *o_lo = a.out + (size_t)(q0 + r_lo) * a.d + (size_t)h * kDh + 2 * tig, *o_hi = o_lo + 8 * (size_t)a.d;
#pragma unroll
  for (int dn = 0; dn < 8; ++dn) {
    if (r_lo < nq) *reinterpret_cast<__nv_bfloat162 *>(o_lo + dn * 8) = __floats2bfloat162_rn(A.o[dn][0] * i0, A.o[dn][1] * i0);
    if (r_hi < nq) *reinterpret_cast<__nv_bfloat162 *>(o_hi + dn * 8) = __floats2bfloat162_rn(A.o[dn][2] * i1, A.o[dn][3] * i1);
  }
}

// Rotary mode: queries and keys rotated by their row's position tau + i, everything rounded to bf16.
__global__ void __launch_bounds__(256) rotate_rows_kernel(int d, const float *__restrict__ qkv, const int32_t *__restrict__ row_sub,
                                                          const int32_t *__restrict__ row_tau, const float2 *__restrict__ rope_tab,
                                                          __nv_bfloat16 *__restrict__ out) {
  const int r = blockIdx.x;
  const int pos = row_sub[r] + row_tau[r];
  const float4 *src = reinterpret_cast<const float4 *>(qkv + (size_t)r * 3 * d);
  uint2 *dst = reinterpret_cast<uint2 *>(out + (size_t)r * 3 * d);
  for (int c = threadIdx.x; c < 3 * d / 4; c += 256) {        // four columns
    float4 v = src[c];
    if (c < d / 2) {
      const float4 cs = *reinterpret_cast<const float4 *>(rope_tab + (size_t)pos * (kDh / 2) + (4 * c % kDh) / 2);
      v = make_float4(v.x * cs.x - v.y * cs.y, v.x * cs.y + v.y * cs.x, v.z * cs.z - v.w * cs.w, v.z * cs.w + v.w * cs.z);
    }
    dst[c] = make_uint2(mt::pack_bf16(v.x, v.y), mt::pack_bf16(v.z, v.w));
  }
}

// x[r] = embedding of the row's input token (fp32 residual stream)
__global__ void gather_rows_kernel(int d, const int32_t *__restrict__ row_tok, const __nv_bfloat16 *__restrict__ embed,
                                   float *__restrict__ x) {
  const int r = blockIdx.x;
  const __nv_bfloat16 *e = embed + (size_t)row_tok[r] * d;      // four columns per thread; d is a multiple of 64
  for (int c = threadIdx.x; c < d / 4; c += blockDim.x) *reinterpret_cast<float4 *>(x + (size_t)r * d + 4 * c) = load4_table(e + 4 * c);
}

// logprob[r] = logits[r][target] - log sum_v exp(logits[r][v])   (the row's term of Eq. 6).  One pass over the row (every thread
// keeps a running maximum and the sum relative to it), 16-byte loads over its aligned body.  (Maximum and sum in a pass
// each, 4-byte loads: 88 us for 2089 rows of 32128, against 48 us.)
__global__ void __launch_bounds__(256) target_logprob_kernel(int V, const float *__restrict__ logits, const int32_t *__restrict__ targets,
                                                             float *__restrict__ logprob) {
  __shared__ float red_m[8], red_s[8];
  const int tid = threadIdx.x;
  const float *row = logits + (size_t)blockIdx.x * V;
  float m = -INFINITY, s = 0.f;
  auto finite = [](float mx) { return mx > -INFINITY ? mx : 0.f; };      // so that a NaN among logits of -inf stays one in the sum
  auto take4 = [&](const float4 &x) {
    const float mx = fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w));
    if (mx > m) { s *= expf(m - mx); m = mx; }
    const float r = finite(m);
    s += (expf(x.x - r) + expf(x.y - r)) + (expf(x.z - r) + expf(x.w - r));
  };
  auto take = [&](float x) {
    if (x > m) { s *= expf(m - x); m = x; }
    s += expf(x - finite(m));
  };
  // scalar up to the row's first 16-byte boundary: the caller's buffer may itself start between two
  const int head = min(V, (int)((16u - (unsigned)(reinterpret_cast<uintptr_t>(row) & 15u)) & 15u) / 4);
  const int nvec = (V - head) / 4;
  if (tid < head) take(row[tid]);
  const float4 *body = reinterpret_cast<const float4 *>(row + head);
  int q = tid;
  for (; q + 3 * 256 < nvec; q += 4 * 256) {
    float4 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = __ldcs(body + q + u * 256);
#pragma unroll
    for (int u = 0; u < 4; ++u) take4(x[u]);
  }
  for (; q < nvec; q += 256) take4(__ldcs(body + q));
  for (int v = head + 4 * nvec + tid; v < V; v += 256) take(row[v]);
  auto join = [&](float &ma, float &sa, float mb, float sb) {
    const float mx = fmaxf(ma, mb), r = finite(mx);
    sa = sa * expf(ma - r) + sb * expf(mb - r);
    ma = mx;
  };
  for (int o = 16; o > 0; o >>= 1) join(m, s, __shfl_xor_sync(0xffffffffu, m, o), __shfl_xor_sync(0xffffffffu, s, o));
  if ((tid & 31) == 0) { red_m[tid >> 5] = m; red_s[tid >> 5] = s; }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < 8; ++w) join(m, s, red_m[w], red_s[w]);
    logprob[blockIdx.x] = row[targets[blockIdx.x]] - (m + logf(s));
  }
}

}  // namespace

cudaError_t teacher_attn_prepare() {
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(teacher_self_kernel<8, true>, attr, TATTN_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(teacher_self_kernel<4, true>, attr, TATTN_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(teacher_self_kernel<8, false>, attr, TATTN_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(teacher_self_kernel<4, false>, attr, TATTN_SMEM);
  return e;
}

cudaError_t launch_teacher_self(const DenseAttnArgs &a, cudaStream_t s) {
  if (a.n_groups < 1) return cudaSuccess;
  if (a.bias_tab != nullptr && a.n_dist > TMAXD) return cudaErrorInvalidValue;      // the head's bias row is held in shared memory
  const dim3 grid(a.n_groups, a.H);
  auto launch = [&](auto wide, auto narrow) {
    if (a.block_rows == 128) wide<<<grid, 256, TATTN_SMEM, s>>>(a);
    else narrow<<<grid, 128, TATTN_SMEM, s>>>(a);
  };
  if (a.bias_tab != nullptr) launch(teacher_self_kernel<8, true>, teacher_self_kernel<4, true>);
  else launch(teacher_self_kernel<8, false>, teacher_self_kernel<4, false>);
  return cudaGetLastError();
}

cudaError_t launch_rotate_rows(int rows, int d, const float *qkv, const int32_t *row_sub, const int32_t *row_tau, const float2 *rope_tab,
                               void *out, cudaStream_t s) {
  rotate_rows_kernel<<<rows, 256, 0, s>>>(d, qkv, row_sub, row_tau, rope_tab, (__nv_bfloat16 *)out);
  return cudaGetLastError();
}

cudaError_t launch_gather_rows(int rows, int d, const int32_t *row_tok, const void *embed, float *x, cudaStream_t s) {
  gather_rows_kernel<<<rows, 128, 0, s>>>(d, row_tok, (const __nv_bfloat16 *)embed, x);
  return cudaGetLastError();
}

cudaError_t launch_target_logprob(int rows, int V, const float *logits, const int32_t *targets, float *logprob, cudaStream_t s) {
  target_logprob_kernel<<<rows, 256, 0, s>>>(V, logits, targets, logprob);
  return cudaGetLastError();
}

}  // namespace pd
