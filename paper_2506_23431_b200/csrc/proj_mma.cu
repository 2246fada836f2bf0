// The linear layers of a decode step (Eq. 3: a stacked transformer decoder) over the step's active rows, packed back to back:
//
//   acc[m][n] = sum_k A[m][k] * W[k][n]        A bf16 [rows][K] packed, W bf16 [K][N] as the caller stores it
//
// with everything between two products in the epilogue: the scale of the RMSNorm in front of the layer (applied after
// the product; the producer of A left x * gain in bf16 and the partial sums of x^2), ReLU, rotary positions and the
// KV-append of the self-attention projection, or the residual add that leaves the next layer's A and sums.
//
// What bounds it: a step has a few to about a hundred rows (of narrow layers several hundred, see proj_tc_better) and
// 1-8 MB of weights per product, so a product is a chain of latencies.  The kernel keeps that chain short: everything that
// does not depend on the kernel before it happens ahead of the programmatic-dependency wait - the CTA's whole slice of W (32 columns) travels through shared memory into mma
// fragments in REGISTERS, split along K over the warps.  Behind the wait there are left: one round of 16-byte loads of
// the rows straight into fragment registers (the order of the 32 k of a unit is permuted alike on both sides, which
// a contraction does not see), the mma chain, one sum over the warps through shared memory, the epilogue.
// A reduction longer than a CTA's warps hold (1024) is split over a thread-block cluster: every CTA pushes its sums into
// the shared memory of the CTA that owns the row, which adds them in rank order (results do not depend on timing).
// Measured per launch in a captured chain of layers (B200, weights from HBM): 2.6 us at 6 rows of width 768 where cuBLAS
// and its share of the norm kernels take 5.1 us; 3.9-4.1 against 5.6 us at 28 rows of width 1024, 5.2 against 5.6 us at 60; 5.0 against 5.2 us
// at 90 rows of width 768.  (Tried for these sizes and slower: tcgen05 with the weights as M operand, 4.8-6 us at 6-60
// rows - tensor-memory set-up and read-out are links of the chain, and N = 16 to 64 does not feed the pipe.)
#include "pd_internal.h"

namespace pd {

constexpr int PJ_KU_MAX = 4;                     // 32-wide K units per warp
constexpr int PJ_WARPS = 8, PJ_T = PJ_WARPS * 32;
constexpr int PJ_NB = 4, PJ_NT = PJ_NB * 8;      // 8-column tiles, columns per CTA
constexpr int PJ_BATCH = 8;                      // 16-row tiles per batch (row scales and, in a cluster, sums are kept per batch)
constexpr int PJ_PITCH = PJ_NT * 2 + 16;         // bytes per k row of the W slice (spreads ldmatrix rows over the banks)
constexpr int PJ_RP = PJ_NT + 8;                 // floats per row of a partial tile
constexpr int PJ_RED = PJ_WARPS * 16 * PJ_RP;    // floats of one buffer of partial tiles
constexpr int PJ_SUMS = (PJ_BATCH * 16 + 8) * PJ_NT;   // floats: the cluster's sums of a batch for the rows this CTA owns
// dynamic shared memory: the W slice on its way into registers, then the warps' partial tiles (double buffered); the sums behind
__host__ __device__ constexpr int pj_lead(int ku) {
  const int w = PJ_WARPS * ku * 32 * PJ_PITCH, red = 2 * PJ_RED * 4;
  return w > red ? w : red;
}
__host__ __device__ constexpr int pj_smem(int ku, bool cluster) { return pj_lead(ku) + (cluster ? PJ_SUMS * 4 : 0); }

__device__ __forceinline__ void j_cp_async16(uint32_t dst, const void *src, bool on) {
  const int n = on ? 16 : 0;                     // 0 source bytes: the destination is zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void j_ldsm_x4_t(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr) : "memory");
}
__device__ __forceinline__ void j_mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t j_pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ void j_cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void j_cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void j_st_peer(uint32_t local, uint32_t rank, float2 v) {
  uint32_t addr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(local), "r"(rank));
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}

// What the epilogue of one (row, column pair) needs beside the product.
struct PjExtra { float2 x; int4 meta; float2 cs; };

// Grid (columns / 32, row groups, K splits = cluster size).
template <int EPI, int KU, bool CLUSTER>
__global__ void __launch_bounds__(PJ_T, 2) proj_mma_kernel(ProjArgs a) {
  extern __shared__ __align__(16) uint8_t j_smem[];
  __shared__ int rows_s[PJ_WARPS];
  __shared__ float inv_s[PJ_BATCH * 16];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tig = lane & 3;
  const int n0 = (int)blockIdx.x * PJ_NT, ks = CLUSTER ? (int)gridDim.z : 1;
  const int rank = CLUSTER ? (int)blockIdx.z : 0;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // ---- ahead of the dependency wait: the number of rows (left by the previous step's scheduler), this warp's W slice
  int n = 0;
  for (int b = tid; b < a.batch; b += PJ_T) n += a.n_active[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  if (lane == 0) rows_s[warp] = n;
  // row groups in use: no more than give every CTA the same number of 16-row tiles; the others leave before they fetch
  int gy = (int)gridDim.y, rows = 0, n_mt = 0;
  auto count = [&]() {
    rows = 0;
#pragma unroll
    for (int w = 0; w < PJ_WARPS; ++w) rows += rows_s[w];
    rows = min(rows, a.rows_cap);
    n_mt = (rows + 15) / 16;
    const int each = max(1, (n_mt + gy - 1) / gy);    // tiles of the busiest CTA
    gy = max(1, (n_mt + each - 1) / each);
  };
  if (blockIdx.y > 0) {
    __syncthreads();
    count();
    if ((int)blockIdx.y >= gy) {
      if (CLUSTER) { j_cluster_arrive(); j_cluster_wait(); }
      asm volatile("griddepcontrol.wait;" ::: "memory");
      return;
    }
  }
  const uint32_t wbuf = (uint32_t)__cvta_generic_to_shared(j_smem) + warp * KU * 32 * PJ_PITCH;
  const int u0 = (rank * PJ_WARPS + warp) * KU;       // first 32-wide K unit of this warp
#pragma unroll
  for (int j = 0; j < KU; ++j) {
    // row k of the unit lies at place 16 [k & 4] + 8 [k & 2] + 2 (k / 8) + (k & 1): eight consecutive places are the k
    // of one fragment half, so that ldmatrix rows fall into different banks
#pragma unroll
    for (int i = 0; i < PJ_NB; ++i) {
      const int c = i * 32 + lane, k = c / PJ_NB, ch = c % PJ_NB;
      const int place = ((k >> 2) & 1) * 16 + ((k >> 1) & 1) * 8 + (k >> 3) * 2 + (k & 1);
      const int kk = (u0 + j) * 32 + k, nn = n0 + ch * 8;
      const bool on = kk < a.K && nn < a.N;
      j_cp_async16(wbuf + j * 32 * PJ_PITCH + place * PJ_PITCH + ch * 16, a.w + (on ? (size_t)kk * a.N + nn : 0), on);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  if (CLUSTER) j_cluster_arrive();                    // (waited for behind the dependency wait: every peer has started)
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  uint32_t wf[KU][2][PJ_NB][2];
#pragma unroll
  for (int j = 0; j < KU; ++j)
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int nb = 0; nb < PJ_NB; nb += 2)           // lanes 0-15: both halves of column tile nb, 16-31: of nb + 1
        j_ldsm_x4_t(wbuf + j * 32 * PJ_PITCH + (m * 16 + (lane & 15)) * PJ_PITCH + (nb + (lane >> 4)) * 16, wf[j][m][nb][0], wf[j][m][nb][1],
                    wf[j][m][nb + 1][0], wf[j][m][nb + 1][1]);
  __syncthreads();                                    // the W slice is in registers everywhere: its memory takes the partial tiles
  if (blockIdx.y == 0) count();
  const int ce = 2 * (tid & 15);                      // this thread's pair of columns in the epilogue (sixteen threads per row)
  float2 gn = make_float2(0.f, 0.f);
  if (EPI == PROJ_RESID) gn = make_float2(__bfloat162float(a.gain_next[n0 + ce]), __bfloat162float(a.gain_next[n0 + ce + 1]));      // (the caller's, aligned to one value)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (CLUSTER) j_cluster_wait();

  float *red = reinterpret_cast<float *>(j_smem);
  float *sums = reinterpret_cast<float *>(j_smem + pj_lead(KU));
  const int per = (PJ_BATCH * 16 + ks - 1) / ks;      // rows of a batch a CTA of the cluster owns
  const int mine = n_mt > (int)blockIdx.y ? (n_mt - (int)blockIdx.y + gy - 1) / gy : 0;      // row tiles blockIdx.y, + gy, ...
  uint4 af[KU][2];
  auto load_a = [&](int mt) {
#pragma unroll
    for (int j = 0; j < KU; ++j)
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const int r = mt * 16 + g + 8 * hh, kk = (u0 + j) * 32 + 8 * tig;
        af[j][hh] = r < rows && kk < a.K ? __ldcg(reinterpret_cast<const uint4 *>(a.act + (size_t)r * a.K + kk)) : make_uint4(0u, 0u, 0u, 0u);
      }
  };
  auto load_extra = [&](int r, PjExtra &x) {          // what the epilogue needs of row r
    const bool on = r < rows;
    if (EPI == PROJ_RESID) x.x = on ? __ldcg(reinterpret_cast<const float2 *>(a.x + (size_t)r * a.N + n0 + ce)) : make_float2(0.f, 0.f);
    if (EPI == PROJ_QKV) {
      x.meta = on ? __ldcg(a.row_meta + r) : make_int4(0, 0, 0, 0);    // (page, slot, position tau + i, subsequence)
      if (a.rope_tab != nullptr) x.cs = a.rope_tab[(size_t)x.meta.z * (kDh / 2) + ((n0 & (kDh - 1)) + ce) / 2];
    }
  };
  auto finish = [&](int r, float inv, float2 s, const PjExtra &x) {
    const int col = n0 + ce;
    const bool on = r < rows && col < a.N;
    if (EPI == PROJ_RESID) {
      float ss = 0.f;
      if (on) {
        s.x += x.x.x; s.y += x.x.y;
        *reinterpret_cast<float2 *>(a.x + (size_t)r * a.N + col) = s;
        *reinterpret_cast<uint32_t *>(a.out + (size_t)r * a.N + col) = j_pack2(s.x * gn.x, s.y * gn.y);
        ss = s.x * s.x + s.y * s.y;
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);      // sixteen neighbouring lanes share a row
      if (on && ce == 0) a.ssq_out[(size_t)r * a.ssq_stride + blockIdx.x] = ss;
    } else if (on) {
      s.x *= inv; s.y *= inv;
      if (EPI == PROJ_RELU) { s.x = fmaxf(s.x, 0.f); s.y = fmaxf(s.y, 0.f); }
      if (EPI != PROJ_QKV) {
        *reinterpret_cast<uint32_t *>(a.out + (size_t)r * a.N + col) = j_pack2(s.x, s.y);
      } else {
        const int d = a.N / 3, which = n0 / d, h = (n0 - which * d) / kDh, cc = col - which * d - h * kDh;
        if (a.raw != nullptr) {
          if (a.raw_f32) *reinterpret_cast<float2 *>(reinterpret_cast<float *>(a.raw) + (size_t)r * a.N + col) = s;
          else *reinterpret_cast<uint32_t *>(reinterpret_cast<__nv_bfloat16 *>(a.raw) + (size_t)r * a.N + col) = j_pack2(s.x, s.y);
        }
        if (a.rope_tab != nullptr && which < 2) s = make_float2(s.x * x.cs.x - s.y * x.cs.y, s.x * x.cs.y + s.y * x.cs.x);
        const uint32_t pk = j_pack2(s.x, s.y);
        if (which == 0) {
          *reinterpret_cast<uint32_t *>(a.out + (size_t)r * d + h * kDh + cc) = pk;
        } else {
          __nv_bfloat16 *blk = a.kv_pool + kv_block_offset(a.layer, a.pool, x.meta.x, d / kDh, h, a.P);
          *reinterpret_cast<uint32_t *>(blk + kv_entry_offset<__nv_bfloat16>(x.meta.y, cc, which - 1)) = pk;
        }
      }
    }
  };
  if (mine > 0) load_a(blockIdx.y);
  PjExtra ex;
  if (!CLUSTER && mine > 0) load_extra((int)blockIdx.y * 16 + (tid >> 4), ex);
  int buf = 0;
  // (128 rows are one batch.  With more, a wide layer of a short reduction - 300 rows of 64 by 4800 - leaves room for one row group, which takes
  // three; a reduction over a cluster has no more rows than one batch, see proj_tc_better.)
  for (int t0 = 0; t0 < mine; t0 += PJ_BATCH) {
    const int tb = min(PJ_BATCH, mine - t0);
    if (t0 > 0) {                                     // the previous batch's scales and sums are read by now
      if (CLUSTER) { j_cluster_arrive(); j_cluster_wait(); } else __syncthreads();
    }
    if (EPI != PROJ_RESID) {                          // scales of the norm in front: two rows of every tile per warp, sixteen lanes each
#pragma unroll
      for (int t = 0; t < PJ_BATCH; ++t) {
        const int rl = warp * 2 + (lane >> 4), r = ((int)blockIdx.y + (t0 + t) * gy) * 16 + rl;
        float s = 0.f;
        if (t < tb && r < rows)
          for (int p = lane & 15; p < a.parts_in; p += 16) s += __ldcg(a.ssq_in + (size_t)r * a.ssq_stride + p);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (t < tb && (lane & 15) == 0) inv_s[t * 16 + rl] = rsqrtf(s * a.inv_width + a.eps);
        if (t + 1 >= tb) break;
      }
    }
    for (int t = 0; t < tb; ++t, buf ^= 1) {
      const int mt = (int)blockIdx.y + (t0 + t) * gy;
      float acc[PJ_NB][4];
#pragma unroll
      for (int nb = 0; nb < PJ_NB; ++nb) acc[nb][0] = acc[nb][1] = acc[nb][2] = acc[nb][3] = 0.f;
#pragma unroll
      for (int j = 0; j < KU; ++j) {
#pragma unroll
        for (int nb = 0; nb < PJ_NB; ++nb) j_mma(acc[nb], af[j][0].x, af[j][1].x, af[j][0].y, af[j][1].y, wf[j][0][nb][0], wf[j][0][nb][1]);
#pragma unroll
        for (int nb = 0; nb < PJ_NB; ++nb) j_mma(acc[nb], af[j][0].z, af[j][1].z, af[j][0].w, af[j][1].w, wf[j][1][nb][0], wf[j][1][nb][1]);
      }
      if (t0 + t + 1 < mine) load_a(mt + gy);
      float *rb = red + buf * PJ_RED;
#pragma unroll
      for (int nb = 0; nb < PJ_NB; ++nb) {
        *reinterpret_cast<float2 *>(rb + (warp * 16 + g) * PJ_RP + nb * 8 + 2 * tig) = make_float2(acc[nb][0], acc[nb][1]);
        *reinterpret_cast<float2 *>(rb + (warp * 16 + g + 8) * PJ_RP + nb * 8 + 2 * tig) = make_float2(acc[nb][2], acc[nb][3]);
      }
      __syncthreads();
      const int rl = tid >> 4;
      float2 s = make_float2(0.f, 0.f);
#pragma unroll
      for (int w = 0; w < PJ_WARPS; ++w) {
        const float2 u = *reinterpret_cast<const float2 *>(rb + (w * 16 + rl) * PJ_RP + ce);
        s.x += u.x; s.y += u.y;
      }
      if (CLUSTER) {
        const int q = t * 16 + rl;                    // row q of the batch belongs to CTA q % ks: push, nobody reads a peer
        j_st_peer((uint32_t)__cvta_generic_to_shared(sums + ((rank * per) + q / ks) * PJ_NT + ce), (uint32_t)(q % ks), s);
      } else {
        const PjExtra now = ex;
        if (t0 + t + 1 < mine) load_extra((mt + gy) * 16 + rl, ex);
        finish(mt * 16 + rl, EPI != PROJ_RESID ? inv_s[t * 16 + rl] : 1.f, s, now);
      }
    }
    if (CLUSTER) {
      // rows rank, rank + ks, ... of the batch: the CTAs' sums in rank order
      auto row_of = [&](int q) { return ((int)blockIdx.y + (t0 + (q >> 4)) * gy) * 16 + (q & 15); };
      j_cluster_arrive();
      int i = tid >> 4;
      if (i * ks + rank < tb * 16) load_extra(row_of(i * ks + rank), ex);
      j_cluster_wait();
      for (int i0 = 0; i0 * ks < tb * 16; i0 += 16, i += 16) {      // (whole warps stay together)
        const int q = i * ks + rank;
        const bool in = q < tb * 16;
        float2 s = make_float2(0.f, 0.f);
        if (in) {
#pragma unroll
          for (int p = 0; p < 8; ++p)
            if (p < ks) {
              const float2 u = *reinterpret_cast<const float2 *>(sums + (p * per + i) * PJ_NT + ce);
              s.x += u.x; s.y += u.y;
            }
        }
        const PjExtra now = ex;
        if (q + 16 * ks < tb * 16) load_extra(row_of(q + 16 * ks), ex);
        finish(in ? row_of(q) : rows, EPI != PROJ_RESID && in ? inv_s[q] : 1.f, s, now);
      }
    }
  }
}

// ---- host side ------------------------------------------------------------------------------------
template <int EPI, bool CLUSTER>
static cudaError_t launch_ku(const ProjArgs &a, int ku, const cudaLaunchConfig_t *cfg_in) {      // cfg_in null: set the attributes
  auto one = [&](auto kernel, int smem) {
    if (cfg_in == nullptr) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaLaunchConfig_t cfg = *cfg_in;
    cfg.dynamicSmemBytes = smem;
    return cudaLaunchKernelEx(&cfg, kernel, a);
  };
  cudaError_t e = cudaSuccess;
  const bool all = cfg_in == nullptr;
  if (all || ku == 1) e = one(proj_mma_kernel<EPI, 1, CLUSTER>, pj_smem(1, CLUSTER));
  if (e == cudaSuccess && (all || ku == 2)) e = one(proj_mma_kernel<EPI, 2, CLUSTER>, pj_smem(2, CLUSTER));
  if (e == cudaSuccess && (all || ku == 3)) e = one(proj_mma_kernel<EPI, 3, CLUSTER>, pj_smem(3, CLUSTER));
  if (e == cudaSuccess && (all || ku == 4)) e = one(proj_mma_kernel<EPI, 4, CLUSTER>, pj_smem(4, CLUSTER));
  return e;
}
template <bool CLUSTER>
static cudaError_t launch_epi(int epi, const ProjArgs &a, int ku, const cudaLaunchConfig_t *cfg) {
  const bool all = cfg == nullptr;
  cudaError_t e = cudaSuccess;
  if (all || epi == PROJ_STORE) e = launch_ku<PROJ_STORE, CLUSTER>(a, ku, cfg);
  if (e == cudaSuccess && (all || epi == PROJ_RELU)) e = launch_ku<PROJ_RELU, CLUSTER>(a, ku, cfg);
  if (e == cudaSuccess && (all || epi == PROJ_RESID)) e = launch_ku<PROJ_RESID, CLUSTER>(a, ku, cfg);
  if (e == cudaSuccess && (all || epi == PROJ_QKV)) e = launch_ku<PROJ_QKV, CLUSTER>(a, ku, cfg);
  return e;
}

// A reduction takes at most eight CTAs of 1024 (the portable cluster size); 16-byte accesses throughout.
bool proj_mma_supported(int K, int N, const void *w) {
  return K >= 8 && K % 8 == 0 && K <= 8 * PJ_WARPS * PJ_KU_MAX * 32 && N % 8 == 0 && reinterpret_cast<uintptr_t>(w) % 16 == 0;
}
int proj_mma_parts(int N) { return (N + PJ_NT - 1) / PJ_NT; }

cudaError_t proj_mma_prepare() {
  ProjArgs a;
  cudaError_t e = launch_epi<false>(0, a, 0, nullptr);
  return e != cudaSuccess ? e : launch_epi<true>(0, a, 0, nullptr);
}

cudaError_t launch_proj_mma(int epi, const ProjArgs &a, cudaStream_t s) {
  const int units = (a.K + 31) / 32, per_cta = PJ_WARPS * PJ_KU_MAX;
  const int ks = (units + per_cta - 1) / per_cta, ku = (units + PJ_WARPS * ks - 1) / (PJ_WARPS * ks);
  const int tiles = proj_mma_parts(a.N);
  // Row groups: as many as two CTAs per SM hold (the kernel uses fewer where they would not shorten the longest walk).
  // 60 rows of width 1024: 5.2 us per launch against 6.3 us with one CTA per SM and 6.4 us with three.
  int gy = 2 * kSms / (tiles * ks);
  if (gy > (a.rows_cap + 15) / 16) gy = (a.rows_cap + 15) / 16;
  if (gy < 1) gy = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles, gy, ks);
  cfg.blockDim = dim3(PJ_T, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[n].val.programmaticStreamSerializationAllowed = 1;
  ++n;
  if (ks > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = 1; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = ks;
    ++n;
  }
  cfg.attrs = attr; cfg.numAttrs = n;
  return ks > 1 ? launch_epi<true>(epi, a, ku, &cfg) : launch_epi<false>(epi, a, ku, &cfg);
}

}  // namespace pd
