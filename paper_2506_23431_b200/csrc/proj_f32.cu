// The linear layers of a decode step in fp32 for few rows (one or two sequences of a small model: latency is all there is):
//
//   acc[m][n] = sum_k A[m][k] * W[k][n]        A fp32 [rows][K], W fp32 [K][N] as the caller stores it, fp32 throughout
//
// The shape of proj_mma.cu on the plain ALUs: a CTA holds its 32 columns of W in registers (a lane = a column, the warps split
// K), fetched ahead of the programmatic-dependency wait; behind it travel only the rows, which every lane then
// reads as broadcasts from shared memory.  Epilogues as there: the norm's scale behind the product, ReLU, rotation and cache append,
// or residual add with the next layer's input and the partial sums of squares.  Reductions beyond 1024 are split over a
// cluster, whose CTAs push their sums to the CTA that owns the row (added in rank order: results do not depend on timing).
// Four rows, width 256: about 2.2 us per launch in a captured chain, where cuBLAS's kernels take 4.1 us, with a norm kernel of
// 1.6 us in front of every second one.
#include "pd_internal.h"

namespace pd {

constexpr int PF_WARPS = 8, PF_T = PF_WARPS * 32, PF_NT = 32;
constexpr int PF_KU_MAX = 4;                     // 32-wide K units per warp
constexpr int PF_TILES = 2;                      // 16-row tiles at most
constexpr int PF_RP = PF_NT + 8;
constexpr int PF_RED = PF_WARPS * 16 * PF_RP;
constexpr int PF_SUMS = (PF_TILES * 16 + 8) * PF_NT;
__host__ __device__ constexpr int pf_apitch(int ku) { return ku * 32 + 4; }
__host__ __device__ constexpr int pf_smem(int ku) { return (PF_WARPS * 16 * pf_apitch(ku) + PF_RED + PF_SUMS) * 4; }

__device__ __forceinline__ void f_cp_async16(uint32_t dst, const void *src, bool on) {
  const int n = on ? 16 : 0;                     // 0 source bytes: the destination is zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void f_cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void f_cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void f_st_peer(uint32_t local, uint32_t rank, float2 v) {
  uint32_t addr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(local), "r"(rank));
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}

// Grid (columns / 32, 1, K splits = cluster size).
template <int EPI, int KU, bool CLUSTER>
__global__ void __launch_bounds__(PF_T, 1) proj_f32_kernel(ProjF32Args a) {
  extern __shared__ __align__(16) float f_smem[];
  __shared__ float inv_s[PF_TILES * 16];
  constexpr int KW = KU * 32, AP = pf_apitch(KU);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n0 = (int)blockIdx.x * PF_NT, ks = CLUSTER ? (int)gridDim.z : 1, rank = CLUSTER ? (int)blockIdx.z : 0;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  float *abuf = f_smem + warp * 16 * AP, *red = f_smem + PF_WARPS * 16 * AP, *sums = red + PF_RED;
  const int k0 = (rank * PF_WARPS + warp) * KW, rows = a.rows;
  // ---- ahead of the dependency wait: this warp's slice of W
  float w[KW];
#pragma unroll
  for (int k = 0; k < KW; ++k) w[k] = k0 + k < a.K && n0 + lane < a.N ? __ldg(a.w + (size_t)(k0 + k) * a.N + n0 + lane) : 0.f;
  if (CLUSTER) f_cluster_arrive();                    // (waited for behind the dependency wait: every peer has started)
  const int ce = 2 * (tid & 15), rl = tid >> 4;       // this thread's pair of columns and row of a tile in the epilogue
  const int col = n0 + ce;
  float2 gn = make_float2(0.f, 0.f);
  if (EPI == PROJ_RESID) gn = make_float2(a.gain_next[col], a.gain_next[col + 1]);      // (the caller's, aligned to one value)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (CLUSTER) f_cluster_wait();

  const int n_mt = (rows + 15) / 16;
  auto load_a = [&](int mt) {
#pragma unroll
    for (int i = 0; i < KU * 4; ++i) {                // 16 rows x KW / 4 chunks
      const int c = i * 32 + lane, r = c / (KW / 4), q = c % (KW / 4);
      const bool on = mt * 16 + r < rows && k0 + 4 * q < a.K;
      f_cp_async16((uint32_t)__cvta_generic_to_shared(abuf + r * AP + 4 * q), a.act + (on ? (size_t)(mt * 16 + r) * a.K + k0 + 4 * q : 0), on);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (n_mt > 0) load_a(0);
  float2 x0[PF_TILES];
  int4 meta[PF_TILES];
#pragma unroll
  for (int t = 0; t < PF_TILES; ++t) {
    const int r = t * 16 + rl;
    if (EPI == PROJ_RESID) x0[t] = r < rows ? __ldcg(reinterpret_cast<const float2 *>(a.x + (size_t)r * a.N + col)) : make_float2(0.f, 0.f);
    if (EPI == PROJ_QKV) meta[t] = r < rows ? __ldcg(a.row_meta + r) : make_int4(0, 0, 0, 0);     // (page, slot, position tau + i, subsequence or 0)
  }
  if (EPI != PROJ_RESID) {                            // scales of the norm in front: two rows of every tile per warp, sixteen lanes each
#pragma unroll
    for (int t = 0; t < PF_TILES; ++t) {
      const int rr = t * 16 + warp * 2 + (lane >> 4);
      float s = 0.f;
      if (a.ssq_in != nullptr && rr < rows)
        for (int p = lane & 15; p < a.parts_in; p += 16) s += __ldcg(a.ssq_in + (size_t)rr * a.ssq_stride + p);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if ((lane & 15) == 0) inv_s[rr] = a.ssq_in != nullptr ? rsqrtf(s * a.inv_width + a.eps) : 1.f;
    }
  }
  auto finish = [&](int t, float2 s, bool mine) {
    const int r = t * 16 + rl;
    const bool on = mine && r < rows && col < a.N;
    if (EPI == PROJ_RESID) {
      float ss = 0.f;
      if (on) {
        float2 xo = x0[0];
#pragma unroll
        for (int u = 1; u < PF_TILES; ++u) if (u == t) xo = x0[u];
        s.x += xo.x; s.y += xo.y;
        *reinterpret_cast<float2 *>(a.x + (size_t)r * a.N + col) = s;
        *reinterpret_cast<float2 *>(a.out + (size_t)r * a.N + col) = make_float2(s.x * gn.x, s.y * gn.y);
        ss = s.x * s.x + s.y * s.y;
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);      // sixteen neighbouring lanes share a row
      if (on && ce == 0) a.ssq_out[(size_t)r * a.ssq_stride + blockIdx.x] = ss;
    } else if (on) {
      const float inv = inv_s[r];
      s.x *= inv; s.y *= inv;
      if (EPI == PROJ_RELU) { s.x = s.x > 0.f ? s.x : 0.f; s.y = s.y > 0.f ? s.y : 0.f; }
      if (EPI != PROJ_QKV) {
        *reinterpret_cast<float2 *>(a.out + (size_t)r * a.N + col) = s;
      } else {
        int4 mt = meta[0];
#pragma unroll
        for (int u = 1; u < PF_TILES; ++u) if (u == t) mt = meta[u];
        const int d = a.N / 3, which = n0 / d, h = (n0 - which * d) / kDh, cc = col - which * d - h * kDh;
        if (a.raw != nullptr) *reinterpret_cast<float2 *>(a.raw + (size_t)r * a.N + col) = s;
        if (mt.w <= 0) return;                        // an unused row
        if (a.rope_tab != nullptr && which < 2) {
          const float2 cs = a.rope_tab[(size_t)mt.z * (kDh / 2) + cc / 2];
          s = make_float2(s.x * cs.x - s.y * cs.y, s.x * cs.y + s.y * cs.x);
        }
        float *to = which == 0 ? a.out + (size_t)r * d + h * kDh + cc
                               : a.kv_pool + kv_block_offset(a.layer, a.pool, mt.x, d / kDh, h, a.P) + kv_entry_offset<float>(mt.y, cc, which - 1);
        *reinterpret_cast<float2 *>(to) = s;
      }
    }
  };
  const int per = (PF_TILES * 16 + ks - 1) / ks;      // rows a CTA of the cluster owns
  for (int t = 0; t < n_mt; ++t) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    const int nr = min(16, rows - t * 16);
    for (int r = 0; r < nr; r += 4) {                 // (rows beyond the last are zero)
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int k = 0; k < KW; k += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 q = *reinterpret_cast<const float4 *>(abuf + (r + u) * AP + k);
          acc[u] = fmaf(q.x, w[k], acc[u]); acc[u] = fmaf(q.y, w[k + 1], acc[u]); acc[u] = fmaf(q.z, w[k + 2], acc[u]); acc[u] = fmaf(q.w, w[k + 3], acc[u]);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u) red[(warp * 16 + r + u) * PF_RP + lane] = acc[u];
    }
    __syncthreads();
    if (t + 1 < n_mt) load_a(t + 1);
    float2 s = make_float2(0.f, 0.f);
    if (rl < nr) {
#pragma unroll
      for (int v = 0; v < PF_WARPS; ++v) {
        const float2 u = *reinterpret_cast<const float2 *>(red + (v * 16 + rl) * PF_RP + ce);
        s.x += u.x; s.y += u.y;
      }
    }
    if (CLUSTER) {
      const int q = t * 16 + rl;                      // row q belongs to CTA q % ks: push, nobody reads a peer
      f_st_peer((uint32_t)__cvta_generic_to_shared(sums + (rank * per + q / ks) * PF_NT + ce), (uint32_t)(q % ks), s);
    } else {
      finish(t, s, true);
    }
    __syncthreads();                                  // the partial tile is read: the next one may be written
  }
  if (CLUSTER) {
    f_cluster_arrive();
    f_cluster_wait();
    for (int t = 0; t < n_mt; ++t) {
      const int q = t * 16 + rl;
      float2 s = make_float2(0.f, 0.f);
      const bool mine = q % ks == rank;
      if (mine) {
#pragma unroll
        for (int p = 0; p < 8; ++p)
          if (p < ks) {
            const float2 u = *reinterpret_cast<const float2 *>(sums + (p * per + q / ks) * PF_NT + ce);
            s.x += u.x; s.y += u.y;
          }
      }
      finish(t, s, mine);                             // (every lane takes part: sixteen share a row's sum of squares)
    }
  }
}

// ---- host side ------------------------------------------------------------------------------------
template <int EPI, bool CLUSTER>
static cudaError_t launch_ku(const ProjF32Args &a, int ku, const cudaLaunchConfig_t *cfg_in) {      // cfg_in null: set the attributes
  auto one = [&](auto kernel, int smem) {
    if (cfg_in == nullptr) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaLaunchConfig_t cfg = *cfg_in;
    cfg.dynamicSmemBytes = smem;
    return cudaLaunchKernelEx(&cfg, kernel, a);
  };
  cudaError_t e = cudaSuccess;
  const bool all = cfg_in == nullptr;
  if (all || ku == 1) e = one(proj_f32_kernel<EPI, 1, CLUSTER>, pf_smem(1));
  if (e == cudaSuccess && (all || ku == 2)) e = one(proj_f32_kernel<EPI, 2, CLUSTER>, pf_smem(2));
  if (e == cudaSuccess && (all || ku == 3)) e = one(proj_f32_kernel<EPI, 3, CLUSTER>, pf_smem(3));
  if (e == cudaSuccess && (all || ku == 4)) e = one(proj_f32_kernel<EPI, 4, CLUSTER>, pf_smem(4));
  return e;
}
template <bool CLUSTER>
static cudaError_t launch_epi(int epi, const ProjF32Args &a, int ku, const cudaLaunchConfig_t *cfg) {
  const bool all = cfg == nullptr;
  cudaError_t e = cudaSuccess;
  if (all || epi == PROJ_STORE) e = launch_ku<PROJ_STORE, CLUSTER>(a, ku, cfg);
  if (e == cudaSuccess && (all || epi == PROJ_RELU)) e = launch_ku<PROJ_RELU, CLUSTER>(a, ku, cfg);
  if (e == cudaSuccess && (all || epi == PROJ_RESID)) e = launch_ku<PROJ_RESID, CLUSTER>(a, ku, cfg);
  if (e == cudaSuccess && (all || epi == PROJ_QKV)) e = launch_ku<PROJ_QKV, CLUSTER>(a, ku, cfg);
  return e;
}

// A reduction takes at most eight CTAs of 1024 (the portable cluster size); 16-byte rows.
bool proj_f32_supported(int K, int N, int rows, const void *w) {
  return rows <= PF_TILES * 16 && K % 4 == 0 && K <= 8 * PF_WARPS * PF_KU_MAX * 32 && N % 2 == 0 && reinterpret_cast<uintptr_t>(w) % 16 == 0;
}

cudaError_t proj_f32_prepare() {
  ProjF32Args a;
  cudaError_t e = launch_epi<false>(0, a, 0, nullptr);
  return e != cudaSuccess ? e : launch_epi<true>(0, a, 0, nullptr);
}

cudaError_t launch_proj_f32(int epi, const ProjF32Args &a, cudaStream_t s) {
  const int units = (a.K + 31) / 32, per_cta = PF_WARPS * PF_KU_MAX;
  const int ks = (units + per_cta - 1) / per_cta, ku = (units + PF_WARPS * ks - 1) / (PF_WARPS * ks);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((a.N + PF_NT - 1) / PF_NT, 1, ks);
  cfg.blockDim = dim3(PF_T, 1, 1);
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
