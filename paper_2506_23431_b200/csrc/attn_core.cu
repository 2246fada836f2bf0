// CUDA-core attention kernels (fp32 arithmetic) for both storage types:
//   * pipelined self-attention over the paged per-subsequence KV cache, with the visibility
//     rule of Section 3.2 evaluated from (subsequence, start step, entry) metadata per page;
//   * cross-attention over the shared context keys/values (all context rows < ctx_len visible);
//   * the split-K merge.
// These are the fp32 path of every configuration and the bf16 path when a sequence has more
// than 32 rows; otherwise bf16 runs the tensor-core kernels in self_attn_tc.cu and
// cross_attn_tma.cu.
#include <type_traits>

#include "pd_internal.h"

namespace pd {

template <typename T> __device__ __forceinline__ void st_f(T *p, float v);
template <> __device__ __forceinline__ void st_f<float>(float *p, float v) { *p = v; }
template <> __device__ __forceinline__ void st_f<__nv_bfloat16>(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ void st_f2(float *p, float x, float y) { *reinterpret_cast<float2 *>(p) = make_float2(x, y); }
__device__ __forceinline__ void st_f2(__nv_bfloat16 *p, float x, float y) { *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(x, y); }
template <typename T> __device__ __forceinline__ float2 ld_f2(const T *p);
template <> __device__ __forceinline__ float2 ld_f2<float>(const float *p) { return *reinterpret_cast<const float2 *>(p); }
template <> __device__ __forceinline__ float2 ld_f2<__nv_bfloat16>(const __nv_bfloat16 *p) { return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p)); }

constexpr int TK = 32;            // keys per tile: one per lane
constexpr int NW = 8;             // warps per CTA at most
constexpr int REG_WARPS = 12;     // warps the registers are shared out for: 168 each, three warps per quarter of an SM (two with any more)
constexpr int MAXD = 512;         // longest distance table held in shared memory
constexpr int PP = TK + 4;        // floats per row of a warp's weights

template <typename T> __host__ __device__ constexpr int row_bytes() { return kDh * (int)sizeof(T) + 16; }      // padded: lanes read rows of their own without conflicts
template <typename T> __host__ __device__ constexpr int ring_bytes() { return 2 * TK * row_bytes<T>(); }      // per warp: one tile of keys and one of values
template <typename T> constexpr int core_smem(int warps) { return warps * (ring_bytes<T>() + kCoreRows * PP * 4); }
static_assert(ring_bytes<__nv_bfloat16>() >= kCoreRows * (kDh + 2) * 4, "a warp's (O, m, l) fits over its ring");

__device__ __forceinline__ void c_cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void c_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void c_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// values 4 c .. 4 c + 3 of key row e in shared memory (SWZ: a 2-byte cache row, whose 16-byte chunks are stored swizzled)
template <bool SWZ> __device__ __forceinline__ float4 key4(const float *row, int, int c) { return *reinterpret_cast<const float4 *>(row + 4 * c); }
template <bool SWZ> __device__ __forceinline__ float4 key4(const __nv_bfloat16 *row, int e, int c) {
  const int col = SWZ ? ((((4 * c) >> 3) ^ (e & 7)) << 3) + ((4 * c) & 7) : 4 * c;
  const uint2 w = *reinterpret_cast<const uint2 *>(row + col);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

// A maximum as the point of reference of exponentials: with nothing visible yet (-inf) any finite one gives them weight 0, and a score that is
// no number keeps a weight that is none, whichever warp or split meets it.
__device__ __forceinline__ float finite(float m) { return m == -INFINITY ? 0.f : m; }

// One CTA = one (split, head, sequence, chunk of up to 16 rows).  Its warps, eight at most, work alone on every eighth 32-key tile: a lane
// holds one key for the scores (queries come as broadcasts from shared memory) and two columns of the output for
// P.V; online softmax per warp, one merge at the end.  Each warp has room for one tile of keys and one of values: the
// next keys travel while the weights meet the values, the next values while the next scores are taken.
// What bounds it at decode sizes is the chain of latencies of a tile, so nothing in the walk waits for another warp.  (Tiles
// staged for the whole CTA with five barriers each: 19.3 us for 4 rows over 256 fp32 keys, against 7.9 us;
// 16 x 12 heads x 1000 keys, 9 rows: 87 us against 62-65 us.)
// FULL = all NW warps (the count then folds into every address and loop), else as many as the launch has.
template <typename T, bool SELF, bool FULL>
__global__ void __launch_bounds__(REG_WARPS * 32) attn_core_kernel(AttnArgs a) {
  const Dims &dm = a.dm;
  const int n_chunk = (dm.C + kCoreRows - 1) / kCoreRows;
  const int split = blockIdx.x / n_chunk, h = blockIdx.y, b = blockIdx.z, c0 = (blockIdx.x % n_chunk) * kCoreRows;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = FULL ? NW : (int)blockDim.x >> 5, nt = nw * 32;
  __shared__ __align__(16) float Qs[kCoreRows][kDh];
  extern __shared__ __align__(16) uint8_t core_raw[];   // the warps' tiles (then their (O, m, l)), the warps' weights
  __shared__ float bias_d[SELF ? MAXD : 1];
  __shared__ int sub_s[kCoreRows];

  // ---- ahead of the dependency wait: what older kernels left (the stand-alone op reads caller-written counts: clamped, so that
  // no access leaves the tensors)
  const int S_all = min(max(a.st.n_active[b], 0), min(dm.C, kMaxRows));
  const int S = min(kCoreRows, S_all - c0);             // rows of this chunk
  const int row0 = b * dm.C + c0;
  const int t = SELF ? a.st.hdr[HDR_STEP_T] - a.st.t0[b] : 0;        // the sequence's own step
  const bool use_bias = SELF && dm.pos_mode == PD_POS_T5_BIAS;
  if (use_bias)
    for (int dd = tid; dd < dm.n_dist && dd < MAXD; dd += nt)
      bias_d[dd] = a.rel_bias[h * a.rel_buckets + a.dist_bucket[dd]] * 1.4426950408889634f;  // log2 domain
  if (tid < kCoreRows) sub_s[tid] = (SELF && tid < S) ? a.st.row_sub[row0 + tid] : 0;
  int n_tiles, ctx_len = 0;
  if (SELF) {
    n_tiles = S > 0 ? a.st.row_sub[row0 + S - 1] * dm.PPS : 0;   // rows are in increasing subsequence order;                 one tile per page (page_tokens <= TK); later subsequences are invisible
  } else {
    ctx_len = min(max(a.st.ctx_len[b], 1), dm.ctx);
    n_tiles = (ctx_len + TK - 1) / TK;
  }
  constexpr int RB = row_bytes<T>();
  constexpr bool SWZ = SELF && sizeof(T) == 2;
  uint8_t *ring = core_raw + warp * ring_bytes<T>();
  const uint32_t ring_k = (uint32_t)__cvta_generic_to_shared(ring), ring_v = ring_k + TK * RB;
  float *ps = reinterpret_cast<float *>(core_raw + nw * ring_bytes<T>()) + warp * kCoreRows * PP;

  struct Tile { int n_valid, k_sub, k_tau0; const T *kp; };      // keys that exist (0: the walk is over), subsequence, first timestamp
  int at = split * nw + warp;
  const size_t v_off = SELF ? kDh : (size_t)dm.ctx * kDh, kstride = SELF ? 2 * kDh : kDh;
  auto next_tile = [&]() {
    Tile x;
    x.n_valid = 0; x.k_sub = 0; x.k_tau0 = 0; x.kp = nullptr;
    for (; at < n_tiles && x.n_valid <= 0; at += a.splits * nw) {
      if (SELF) {
        const int ksub = at / dm.PPS + 1, j = at % dm.PPS;
        const int sidx = b * dm.SM + ksub - 1, e0 = j * dm.P;
        x.n_valid = min(dm.P, a.st.len[sidx] + 1 - e0);   // bos + content tokens, including this step's input
        if (x.n_valid <= 0) { x.n_valid = 0; continue; }
        const int page = a.st.page_table[(size_t)sidx * dm.PPS + j];
        x.kp = (const T *)a.kv + kv_block_offset(a.layer, dm.pool, page, dm.H, h, dm.P);      // a value row follows its key row
        x.k_sub = ksub;
        x.k_tau0 = a.st.start[sidx] - 1 + e0;             // timestamp of the tile's first entry
      } else {
        x.n_valid = min(TK, ctx_len - at * TK);
        x.kp = (const T *)a.kv + ctx_kv_offset(a.layer, dm.B, b, dm.H, h, 0, dm.ctx) + (size_t)at * TK * kDh;
      }
    }
    return x;
  };
  constexpr int CPR = kDh * (int)sizeof(T) / 16;          // 16-byte chunks of a row
  auto fetch = [&](uint32_t dst, const T *src, int n) {
#pragma unroll 4
    for (int c = lane; c < n * CPR; c += 32) c_cp_async16(dst + (c / CPR) * RB + (c % CPR) * 16, reinterpret_cast<const uint8_t *>(src + (c / CPR) * kstride) + (c % CPR) * 16);
    c_commit();
  };
  Tile cur;
  cur.n_valid = 0; cur.kp = nullptr; cur.k_sub = cur.k_tau0 = 0;
  auto fetch_first = [&]() {
    fetch(ring_k, cur.kp, cur.n_valid);
    fetch(ring_v, cur.kp + v_off, cur.n_valid);
  };
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (!SELF && S > 0) { cur = next_tile(); fetch_first(); }           // the context is older than the kernel before
  asm volatile("griddepcontrol.wait;" ::: "memory");
  T *out = (T *)a.out;
  if (split == 0)                                       // rows beyond the active ones stay zero
    for (int idx = tid; idx < (min(kCoreRows, dm.C - c0) - max(S, 0)) * kDh; idx += nt)
      st_f<T>(out + (size_t)(row0 + max(S, 0) + idx / kDh) * dm.d + h * kDh + idx % kDh, 0.f);
  if (S <= 0) return;
  for (int idx = tid; idx < kCoreRows * kDh / 4; idx += nt) {        // four columns at a time: a CTA may have only one warp
    const int r = idx / (kDh / 4), c = 4 * (idx % (kDh / 4));
    *reinterpret_cast<float4 *>(&Qs[r][c]) = r < S ? key4<false>((const T *)a.q + (size_t)(row0 + r) * dm.d + h * kDh, 0, c / 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();

  float o[kCoreRows][2];
#pragma unroll
  for (int s = 0; s < kCoreRows; ++s) o[s][0] = o[s][1] = 0.f;
  float m_run = -INFINITY, l_run = 0.f;                 // lane s: maximum and sum of row s
  if (SELF) { cur = next_tile(); fetch_first(); }
  while (cur.n_valid > 0) {
    const Tile nxt = next_tile();
    const int n_valid = cur.n_valid;
    c_wait1();
    __syncwarp();
    const int e = min(lane, n_valid - 1);
    float k[kDh];
    const T *krow = reinterpret_cast<const T *>(ring + e * RB);
#pragma unroll
    for (int c = 0; c < kDh / 4; ++c) *reinterpret_cast<float4 *>(&k[4 * c]) = key4<SWZ>(krow, e, c);
    __syncwarp();
    fetch(ring_k, nxt.kp, nxt.n_valid);
    // ---- scores in the log2 domain, online softmax: row by row, a key per lane
    float corr = 1.f;                                     // lane s: factor of row s's old state
    for (int s0 = 0; s0 < S; s0 += 4) {                   // four rows at a time: their chains of multiply-adds and shuffles overlap
      float sc[4], mx[4], p[4], sum[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) sc[u] = 0.f;
#pragma unroll
      for (int c = 0; c < kDh / 4; ++c)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 q = *reinterpret_cast<const float4 *>(&Qs[s0 + u][4 * c]);
          sc[u] = fmaf(q.x, k[4 * c], sc[u]); sc[u] = fmaf(q.y, k[4 * c + 1], sc[u]); sc[u] = fmaf(q.z, k[4 * c + 2], sc[u]); sc[u] = fmaf(q.w, k[4 * c + 3], sc[u]);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        bool vis = lane < n_valid;
        sc[u] *= dm.scale_log2e;
        if (SELF) {
          // dependency rule: subsequence index not larger than the query's, timestamp not later
          const int sub = sub_s[s0 + u];
          vis = vis && cur.k_sub <= sub && cur.k_tau0 + lane <= t - 1;
          if (use_bias && vis) sc[u] += bias_d[(t - 1 + sub) - (cur.k_tau0 + lane + cur.k_sub)];   // = |dtau| + |di| on a visible pair
        }
        if (!vis) sc[u] = -INFINITY;
        mx[u] = sc[u];
      }
#pragma unroll
      for (int w = 16; w > 0; w >>= 1)
#pragma unroll
        for (int u = 0; u < 4; ++u) mx[u] = fmaxf(mx[u], __shfl_xor_sync(0xffffffffu, mx[u], w));
      float m_old[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        m_old[u] = __shfl_sync(0xffffffffu, m_run, s0 + u);
        mx[u] = fmaxf(m_old[u], mx[u]);
        p[u] = exp2f(sc[u] - finite(mx[u]));
        sum[u] = p[u];
        ps[(s0 + u) * PP + lane] = p[u];
      }
#pragma unroll
      for (int w = 16; w > 0; w >>= 1)
#pragma unroll
        for (int u = 0; u < 4; ++u) sum[u] += __shfl_xor_sync(0xffffffffu, sum[u], w);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (lane == s0 + u) {
          corr = exp2f(m_old[u] - finite(mx[u]));
          m_run = mx[u]; l_run = l_run * corr + sum[u];
        }
    }
    c_wait1();
    __syncwarp();
    // ---- O = O corr + P V: two columns per lane, four keys at a time
#pragma unroll
    for (int s = 0; s < kCoreRows; ++s) { const float f = __shfl_sync(0xffffffffu, corr, s); o[s][0] *= f; o[s][1] *= f; }
#pragma unroll 2
    for (int e4 = 0; e4 < n_valid; e4 += 4) {
      float2 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int ee = min(e4 + u, n_valid - 1);          // (absent keys have weight 0)
        const int col = SWZ ? ((((2 * lane) >> 3) ^ (ee & 7)) << 3) + ((2 * lane) & 7) : 2 * lane;
        v[u] = ld_f2<T>(reinterpret_cast<const T *>(ring + (TK + ee) * RB) + col);
      }
#pragma unroll
      for (int s = 0; s < kCoreRows; ++s) {
        if (s < S) {
          const float4 p = *reinterpret_cast<const float4 *>(&ps[s * PP + e4]);
          o[s][0] = fmaf(p.x, v[0].x, o[s][0]); o[s][1] = fmaf(p.x, v[0].y, o[s][1]);
          o[s][0] = fmaf(p.y, v[1].x, o[s][0]); o[s][1] = fmaf(p.y, v[1].y, o[s][1]);
          o[s][0] = fmaf(p.z, v[2].x, o[s][0]); o[s][1] = fmaf(p.z, v[2].y, o[s][1]);
          o[s][0] = fmaf(p.w, v[3].x, o[s][0]); o[s][1] = fmaf(p.w, v[3].y, o[s][1]);
        }
      }
    }
    __syncwarp();
    fetch(ring_v, nxt.kp + v_off, nxt.n_valid);
    cur = nxt;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  // ---- merge of the warps
  __syncthreads();
  float *mo = reinterpret_cast<float *>(core_raw), *mm = mo + nw * kCoreRows * kDh, *ml = mm + nw * kCoreRows;
#pragma unroll
  for (int s = 0; s < kCoreRows; ++s)
    if (s < S) *reinterpret_cast<float2 *>(&mo[(warp * kCoreRows + s) * kDh + 2 * lane]) = make_float2(o[s][0], o[s][1]);
  if (lane < S) { mm[warp * kCoreRows + lane] = m_run; ml[warp * kCoreRows + lane] = l_run; }
  __syncthreads();
  for (int s = warp; s < S; s += nw) {                  // a row per warp, two columns per lane
    const int r = row0 + s;
    float m[NW], M = -INFINITY, L = 0.f;               // (absent warps: -inf, weight 0; their loads do not wait for one another's test)
#pragma unroll
    for (int w = 0; w < NW; ++w) { m[w] = w < nw ? mm[w * kCoreRows + s] : -INFINITY; M = fmaxf(M, m[w]); }
    float2 O = make_float2(0.f, 0.f);
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float f = exp2f(m[w] - finite(M)), l = w < nw ? ml[w * kCoreRows + s] : 0.f;
      const float2 u = w < nw ? *reinterpret_cast<const float2 *>(&mo[(w * kCoreRows + s) * kDh + 2 * lane]) : make_float2(0.f, 0.f);
      L += l * f;
      O.x += u.x * f; O.y += u.y * f;
    }
    if (a.splits == 1) {
      st_f2(out + (size_t)r * dm.d + h * kDh + 2 * lane, O.x / L, O.y / L);
    } else {
      const size_t pi = ((size_t)r * dm.H + h) * a.splits + split;
      *reinterpret_cast<float2 *>(a.part_o + pi * kDh + 2 * lane) = O;
      if (lane == 0) { a.part_ml[pi * 2] = M; a.part_ml[pi * 2 + 1] = L; }
    }
  }
}

template <typename T, bool SELF>
static cudaError_t prepare_core() {
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const cudaError_t e = cudaFuncSetAttribute(attn_core_kernel<T, SELF, true>, attr, core_smem<T>(NW));
  return e != cudaSuccess ? e : cudaFuncSetAttribute(attn_core_kernel<T, SELF, false>, attr, core_smem<T>(NW));
}
cudaError_t attn_core_prepare(int dtype, bool self) {
  if (dtype == PD_DTYPE_BF16) return self ? prepare_core<__nv_bfloat16, true>() : prepare_core<__nv_bfloat16, false>();
  return self ? prepare_core<float, true>() : prepare_core<float, false>();
}

// The tiles of a round of eight warps per split: with fewer, a split adds a launch and takes no tile off any warp's walk.
int attn_core_splits_useful(int ctx) { return (ctx + NW * TK - 1) / (NW * TK); }

// a.pdl: launched as a programmatic dependent of the kernel before it - only where that kernel writes none of the state, and
// what it writes is read behind the wait (queries, the step's keys/values).
cudaError_t launch_attn_core(const AttnArgs &a, int dtype, bool self, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  // Chunks share a dimension with the splits: the sequences alone may fill theirs (the entry points take 65535).
  const int chunks = (a.dm.C + kCoreRows - 1) / kCoreRows;
  cfg.gridDim = dim3(a.splits * chunks, a.dm.H, a.batch);
  // Warps: with a CTA per SM at most, all eight (they share the loads ahead of the walk).  Beyond that no more than there are tiles for, and as
  // few as keep the number of rounds: a warp without a tile holds 12 - 20 KB of shared memory that another CTA could use.  64 sequences x
  // 12 heads, fp32: 20 rows over 64 keys 92 us with eight warps each, 33 with two; 33 rows over 300 keys 269 us, 162 with five.
  const int tiles = self ? a.dm.SM * a.dm.PPS : (a.dm.ctx + TK - 1) / TK, each = (tiles + a.splits - 1) / a.splits;
  const int rounds = (each + NW - 1) / NW;
  const int warps = (long long)a.splits * chunks * a.dm.H * a.batch <= kSms ? NW : (each + rounds - 1) / rounds;
  cfg.blockDim = dim3(32 * warps, 1, 1);
  cfg.dynamicSmemBytes = dtype == PD_DTYPE_BF16 ? core_smem<__nv_bfloat16>(warps) : core_smem<float>(warps);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = a.pdl ? 1 : 0;
  auto launch = [&](auto full) {
    constexpr bool F = decltype(full)::value;
    if (dtype == PD_DTYPE_BF16)
      return self ? cudaLaunchKernelEx(&cfg, attn_core_kernel<__nv_bfloat16, true, F>, a) : cudaLaunchKernelEx(&cfg, attn_core_kernel<__nv_bfloat16, false, F>, a);
    return self ? cudaLaunchKernelEx(&cfg, attn_core_kernel<float, true, F>, a) : cudaLaunchKernelEx(&cfg, attn_core_kernel<float, false, F>, a);
  };
  return warps == NW ? launch(std::true_type()) : launch(std::false_type());
}

// Merge of the split-K partials (m, l, o) of one row and head: the usual log-sum-exp rescale.
template <typename T>
__global__ void attn_merge_kernel(AttnArgs a) {
  const Dims &dm = a.dm;
  int r = blockIdx.x;
  int b = r / dm.C, c = r % dm.C;
  if (c >= min(a.st.n_active[b], dm.C)) return;       // the attention kernel already zeroed unused rows
  T *out = (T *)a.out;
  for (int idx = threadIdx.x; idx < dm.d; idx += blockDim.x) {
    int h = idx / kDh, dim = idx % kDh;
    size_t p0 = ((size_t)r * dm.H + h) * a.splits;
    float M = -INFINITY;
    for (int s = 0; s < a.splits; ++s) M = fmaxf(M, a.part_ml[(p0 + s) * 2]);
    float L = 0.f, O = 0.f;
    for (int s = 0; s < a.splits; ++s) {
      float w = exp2f(a.part_ml[(p0 + s) * 2] - finite(M));
      L += a.part_ml[(p0 + s) * 2 + 1] * w;
      O += a.part_o[(p0 + s) * kDh + dim] * w;
    }
    st_f<T>(out + (size_t)r * dm.d + idx, O / L);
  }
}

cudaError_t launch_attn_merge(const AttnArgs &a, int dtype, cudaStream_t s) {
  int rows = a.batch * a.dm.C;
  if (dtype == PD_DTYPE_BF16) attn_merge_kernel<__nv_bfloat16><<<rows, 256, 0, s>>>(a);
  else attn_merge_kernel<float><<<rows, 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace pd
