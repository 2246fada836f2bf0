// The linear layers of a decode step over more packed rows than proj_mma.cu is for, on the 5th-generation tensor cores:
//
//   acc[n][m] = sum_k W[k][n] * A[m][k]        A bf16 [rows][K] packed, W bf16 [K][N] as the caller stores it
//
// with the same epilogues as proj_mma.cu (norm scale behind the product, ReLU, rotation + cache append, residual add + the next
// layer's input and sums of squares).
//
// A pair of CTAs (two SMs, tcgen05 cta_group::2) takes 128 columns of W - the M dimension, 64 per CTA, read MN-major in the caller's
// layout - and a group of up to 128 rows as the N dimension, of which each CTA fetches half.  So a CTA brings in 64 columns of W and
// R / 2 rows, where a CTA alone would need the same columns and R rows: behind the dependency wait the rows are what is waited for.
// The weights do not depend on the kernel before: their tiles are requested ahead of that wait, as many as the ring holds.  A CTA
// takes at most half an SM's shared memory, so that this works while the kernel before still holds the other half (with the whole of it,
// decodes are slower by a tenth).  Tensor memory is taken ahead of the wait as well (behind it: 72.3 ms against 68.3 for the decode of 32 sequences
// below), by pairs that have rows only.
// Tensor memory of a pair is taken and given back by instructions that belong to both CTAs, and nothing orders one CTA against the other by
// itself.  A form that took it before it knew its rows, and gave it back at once where there were none, ended in a launch failure once; the cause was
// never established.  By reading, a CTA of it could give back, and exit, while its peer was still taking.  So the CTAs meet behind the taking, and
// compare addresses there (a product writes both CTAs' tensor memory at one), and meet again behind the giving back before either exits: 0.1 us
// per launch.  Pairs of two launches, like pairs of one launch of more pairs than the chip has pairs of SMs, may take at the same time; shared
// memory lets no third one onto their SMs, and columns never run out: two pairs take 128 of 512, the other kernels that fit beside one of them 256.
// (With the next launch started only behind the taking a decode takes 1.9 % longer, and pairs of one launch still take at the same time.)
// The lanes of tensor memory are columns of W, its columns rows of A: an epilogue warp holds 32 neighbouring columns of one row at
// a time, reads the residual stream in whole lines, and pairs of lanes pack two rows' stores into one.
// Reductions beyond 1024 are split over a cluster of pairs: every CTA copies its sums of the rows another CTA owns into that CTA's
// shared memory (one bulk copy per peer), which adds them in rank order (results do not depend on timing).
// What bounds it: a launch is a chain of latencies - release of the launch before 1.2 us, first rows 0.5, products and the weights the
// ring did not hold, accumulators out, 0.6 to the exit.  What a launch advances a decode of 32 sequences by (204 rows active of 512, width 1024): 7.1 us
// for queries, keys and values, 5.2-5.7 for the square products, 6.7 up, 9.2 down, where the library took 5.6, 4.3-4.6, 6.3 and 8.3 and
// 2.4 for a norm in front of every other one, without overlap.  Fewer or more row groups, K splits of 1536 or 2048: slower or the same.
// Every mbarrier wait is bounded: on expiry the kernel records PD_ERR_TIMEOUT, stops waiting, falls through to the
// common exit and frees its tensor memory.
#include <algorithm>

#include "pd_internal.h"

namespace pd {

constexpr int PT_BK = 64;                        // K of a block: 128 bytes of a row of A, 64 rows of W
constexpr int PT_COLS = 64;                      // columns of W per CTA
constexpr int PT_W_BYTES = PT_BK * PT_COLS * 2;  // 8 KB
constexpr int PT_R_MAX = 128;                    // most rows of a group
constexpr int PT_TMEM = PT_R_MAX / 2;            // columns of tensor memory: half the rows of a group
constexpr int PT_STAGES_MAX = 8;
constexpr int PT_EPI_WARPS = 8, PT_EPI_T = PT_EPI_WARPS * 32;
constexpr int PT_THREADS = 96 + PT_EPI_T;        // weights warp, product warp, rows warp, epilogue warps
constexpr int PT_RING = 104 * 1024;              // behind the products it takes the partial sums of a split reduction
constexpr int PT_SMEM = PT_RING + 256 /*barriers*/ + 1024 /*alignment slack*/;
constexpr uint32_t PT_SPIN_LIMIT = 1u << 24;
static_assert(8 * (2 * PT_STAGES_MAX + 6) <= 256, "barriers");
// 64-wide blocks of K per stage and copy: a copy costs its issue and a round trip, so small boxes are taken several at a time
__host__ __device__ constexpr int pt_blocks(int R) { return R <= 64 ? 4 : 2; }

__device__ __forceinline__ uint32_t t_smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void t_mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void t_mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Arrival at a barrier of any CTA of the cluster.
__device__ __forceinline__ void t_mbar_arrive_peer(uint32_t bar_cluster) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}
// Bounded wait: false when the phase did not complete within the spin limit.
template <bool CLUSTER = false>
__device__ __forceinline__ bool t_mbar_wait(uint32_t bar, uint32_t parity) {
  for (uint32_t it = 0; it < PT_SPIN_LIMIT; ++it) {
    uint32_t ok;
    if (CLUSTER)
      asm volatile(
          "{\n\t.reg .pred p;\n\t"
          "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(ok)
          : "r"(bar), "r"(parity)
          : "memory");
    else
      asm volatile(
          "{\n\t.reg .pred p;\n\t"
          "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(ok)
          : "r"(bar), "r"(parity)
          : "memory");
    if (ok) return true;
  }
  return false;
}
// The same by a whole warp: one answer for all its lanes, so that none goes on without the others also where the limit runs out.  (Asked behind
// the loop: lanes that take every turn together cost 1.5 % of a decode with 8-bit context.)
template <bool CLUSTER = false>
__device__ __forceinline__ bool t_mbar_wait_warp(uint32_t bar, uint32_t parity) { return __all_sync(0xffffffffu, t_mbar_wait<CLUSTER>(bar, parity)); }
__device__ __forceinline__ uint32_t t_peer(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
// `bytes` of this CTA's shared memory into another CTA's, whose barrier counts them.
__device__ __forceinline__ void t_copy_peer(uint32_t dst_cluster, uint32_t src, uint32_t bytes, uint32_t bar_cluster) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst_cluster), "r"(src), "r"(bytes), "r"(bar_cluster) : "memory");
}
// A tile into this CTA's shared memory; the completion goes to the barrier `bar` of the pair's first CTA.
__device__ __forceinline__ void t_tma_load(uint32_t dst, const CUtensorMap *tmap, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(tmap), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
// The map itself on its way: a first copy with it would wait for a round trip more.
__device__ __forceinline__ void t_map_prefetch(const CUtensorMap *tmap) { asm volatile("prefetch.tensormap [%0];" ::"l"(tmap) : "memory"); }
__device__ __forceinline__ void t_tma_load3(uint32_t dst, const CUtensorMap *tmap, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(tmap), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
__device__ __forceinline__ void t_tma_prefetch(const CUtensorMap *tmap, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(tmap), "r"(x), "r"(y) : "memory");
}
// Shared-memory matrix descriptor of rows of 128 bytes, 128-byte swizzle, 1024 B between groups of eight rows: a K-major operand
// (rows = rows of A) as well as one 64-wide span of an MN-major one (rows = K).  Low word: address >> 4; the high word is constant.
constexpr uint32_t PT_DESC_HI = 64u | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t t_desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (64u << 16); }
// kind::f16: D fp32, A and B bf16; bit 15: A is MN-major; N >> 3 at bit 17; M (128 over the pair) >> 4 at bit 24
__device__ __forceinline__ uint32_t t_idesc(int n) { return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uint32_t)(n >> 3) << 17) | (8u << 24); }
__device__ __forceinline__ void t_mma(uint32_t tmem_d, uint32_t alo, uint32_t blo, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %5};\n\t"
      "mov.b64 db, {%2, %5};\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(alo), "r"(blo), "r"(idesc), "r"(accumulate), "n"(PT_DESC_HI)
      : "memory");
}
// One lane of a converged warp.
__device__ __forceinline__ bool t_elect() {
  uint32_t on;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(on));
  return on != 0;
}
// The barrier at this offset in both CTAs of the pair gets one arrival once every product issued so far by this thread has finished.
__device__ __forceinline__ void t_commit(uint32_t bar, uint16_t mask) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"(mask) : "memory");
}
// 8 columns (rows of A) of this warp's quarter of tensor memory, one lane per column of W
__device__ __forceinline__ void t_tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    asm volatile("" : "+r"(r[i]));                   // nothing reads it ahead of the wait
    v[i] = __uint_as_float(r[i]);
  }
}
__device__ __forceinline__ void t_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void t_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// The product warp tells the epilogue warps where tensor memory is (they ask behind the products, and never wait here).
__device__ __forceinline__ void t_tmem_told() { asm volatile("bar.arrive 2, %0;" ::"n"(PT_EPI_T + 32) : "memory"); }
__device__ __forceinline__ void t_tmem_ask() { asm volatile("bar.sync 2, %0;" ::"n"(PT_EPI_T + 32) : "memory"); }
__device__ __forceinline__ void t_epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(PT_EPI_T) : "memory"); }
__device__ __forceinline__ void t_cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void t_cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t t_pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

struct ProjTcArgs : ProjArgs {
  int groups;                // row groups that give every SM one CTA
  int32_t *status;           // error word (PD_ERR_TIMEOUT on an expired wait)
};

// Grid (2 x column slices, row groups, K splits), cluster (2, 1, K splits).
template <int EPI, bool SPLIT>
__global__ void __launch_bounds__(PT_THREADS, 2)
proj_tc_kernel(const __grid_constant__ ProjTcWeightMaps wmaps, const __grid_constant__ ProjTcActMaps maps, ProjTcArgs a) {
  extern __shared__ uint8_t t_raw[];
  __shared__ uint32_t tmem_base_s, peer_base_s;
  __shared__ int same_s;                             // the pair's tensor memory is at one address
  __shared__ int rows_s[PT_THREADS / 32];
  __shared__ float inv_s[PT_R_MAX];
  __shared__ int4 meta_s[EPI == PROJ_QKV ? PT_R_MAX : 1];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int half = (int)blockIdx.x & 1;              // this CTA's half of the pair's columns and rows
  const int ks = SPLIT ? (int)gridDim.z : 1, z = SPLIT ? (int)blockIdx.z : 0;
  const uint32_t leader = 2u * z, peer = leader + (uint32_t)(half ^ 1);      // first CTA of this pair in the cluster, the other one of it
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // ---- ahead of the dependency wait: the number of rows (left by the previous step's scheduler), barriers, tensor memory, weights
  const uint32_t ring = (t_smem_u32(t_raw) + 1023u) & ~1023u;
  const uint32_t full = ring + PT_RING, empty = full + 8 * PT_STAGES_MAX, acc_full = empty + 8 * PT_STAGES_MAX, red_full = acc_full + 8,
                 red_free = red_full + 8, acc_read = red_free + 8, peer_has = acc_read + 8, peer_gave = peer_has + 8;
  int cnt = 0;
  for (int b = tid; b < a.batch; b += PT_THREADS) cnt += a.n_active[b];
  if (tid < 2) t_map_prefetch(&wmaps.k[tid]);
  if (tid == 0) {
    for (int s = 0; s < PT_STAGES_MAX; ++s) { t_mbar_init(full + 8 * s, 1); t_mbar_init(empty + 8 * s, 1); }
    t_mbar_init(acc_full, 1);
    t_mbar_init(red_full, 1);
    t_mbar_init(red_free, (uint32_t)ks);
    t_mbar_init(acc_read, (uint32_t)(2 * PT_EPI_WARPS + (SPLIT ? ks : 0)));
    t_mbar_init(peer_has, 1);
    t_mbar_init(peer_gave, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  t_cluster_arrive();                                // this CTA's barriers stand
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  if (lane == 0) rows_s[warp] = cnt;
  __syncthreads();
  int rows = 0;
#pragma unroll
  for (int w = 0; w < PT_THREADS / 32; ++w) rows += rows_s[w];
  rows = min(rows, a.rows_cap);
  // row groups in use: as many as give every SM one CTA, more where a group would not fit; none smaller than 16 rows
  const int gy = max(1, min(min((int)gridDim.y, (rows + 15) / 16), max(a.groups, (rows + PT_R_MAX - 1) / PT_R_MAX)));
  const int per = ((rows + gy - 1) / gy + 7) / 8 * 8;
  const int row0 = (int)blockIdx.y * per, n_rows = min(per, rows - row0);
  if ((int)blockIdx.y >= gy || n_rows <= 0) {        // (the whole cluster; it takes no tensor memory)
    t_cluster_wait();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return;
  }
  const int R = min(PT_R_MAX, (n_rows + 31) / 32 * 32);
  const int CH = pt_blocks(R);
  const int w_bytes = CH * PT_W_BYTES, stage_bytes = w_bytes + CH * R * 64;       // 64 columns of W and R / 2 rows
  const int S = min(PT_STAGES_MAX, PT_RING / stage_bytes);
  const int kb_all = a.K / PT_BK, kb_per = (kb_all + ks - 1) / ks;
  const int kb0 = z * kb_per, nkb = min(kb_per, kb_all - kb0), nch = (nkb + CH - 1) / CH;    // (the launcher leaves no split without a block)
  t_cluster_wait();                                  // every barrier of the cluster stands
  const int n0 = (int)blockIdx.x * PT_COLS;
  bool ok = true, same = true;

  if (warp == 0) {
    // ------------------------------------------------------------------ weights (one lane)
    if (lane == 0) {
      const uint32_t lead_full = t_peer(full, leader);
      const CUtensorMap *map_w = &wmaps.k[CH >> 2];
      const bool lead = half == 0;
      const uint32_t tx = 2u * (uint32_t)stage_bytes, ring_end = ring + S * stage_bytes;
      uint32_t dst = ring, bar = 0, parity = 1u;
      int x = kb0 * PT_BK;
      for (int it = 0; it < nch; ++it, x += CH * PT_BK) {
        if (dst == ring_end) {
          if (it == S && blockIdx.y == 0)            // what the ring does not hold yet: into L2 (one row group asks for all)
            for (int i = it, xp = x; i < nch; ++i, xp += CH * PT_BK) t_tma_prefetch(map_w, n0, xp);
          dst = ring; bar = 0; parity ^= 1u;
        }
        if (it >= S && !t_mbar_wait(empty + bar, parity)) { ok = false; break; }
        if (lead) t_mbar_expect_tx(full + bar, tx);
        t_tma_load(dst, map_w, lead_full + bar, n0, x);
        dst += stage_bytes; bar += 8;
      }
      asm volatile("griddepcontrol.wait;" ::: "memory");
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ products (one lane of the pair).  The whole warp walks: a loop that
    // one lane walks keeps descriptors out of the uniform registers the products read, and a product then costs 128 cycles to issue
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(t_smem_u32(&tmem_base_s)), "r"(PT_TMEM) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    __syncwarp();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(&tmem_base_s);
    // The two CTAs tell each other where: neither goes on before the pair's allocation is complete in both.
    if (lane == 0) {
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(t_peer(t_smem_u32(&peer_base_s), peer)), "r"(tmem) : "memory");
      t_mbar_arrive_peer(t_peer(peer_has, peer));
    }
    ok = t_mbar_wait_warp<true>(peer_has, 0u);
    same = !ok || *reinterpret_cast<volatile uint32_t *>(&peer_base_s) == tmem;
    if (lane == 0) *reinterpret_cast<volatile int *>(&same_s) = same;
    __syncwarp();
    t_tmem_told();
    if (half == 0) {
      const uint32_t idesc = t_idesc(R);
      const uint16_t mask = (uint16_t)(3u << leader);
      int s = 0;
      uint32_t u = 0, lo = t_desc_lo(ring);
      for (int ch = 0; ch < nch && ok; ++ch) {
        if (!t_mbar_wait_warp(full + 8 * s, u & 1u)) { ok = false; break; }
        t_fence_after();
        if (t_elect()) {
          const int nb = same ? min(CH, nkb - ch * CH) : 0;    // (a product writes both CTAs' tensor memory, at one address)
          for (int b = 0; b < nb; ++b) {
#pragma unroll
            for (int k4 = 0; k4 < PT_BK / 16; ++k4)  // 16 of K: two groups of eight rows of W, 32 bytes of a row of A
              t_mma(tmem, lo + b * (PT_W_BYTES >> 4) + k4 * (2048 >> 4), lo + (w_bytes >> 4) + b * (R * 64 >> 4) + k4 * (32 >> 4), idesc,
                    ch > 0 || b > 0 || k4 > 0 ? 1u : 0u);
          }
          if (ch + S < nch) t_commit(empty + 8 * s, mask);     // (a stage that is not filled again needs none)
        }
        lo += (uint32_t)stage_bytes >> 4;
        if (++s == S) { s = 0; ++u; lo = t_desc_lo(ring); }
      }
      if (ok && t_elect()) t_commit(acc_full, mask);
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ rows (one lane)
    if (lane == 0) {
      const uint32_t lead_full = t_peer(full, leader);
      const uint32_t ring_end = ring + S * stage_bytes;
      const CUtensorMap *map_a = &maps.box[R / 32 - 1];
      const int y = row0 + half * (R / 2);
      uint32_t dst = ring, bar = 0, parity = 1u;
      t_map_prefetch(map_a);
      asm volatile("griddepcontrol.wait;" ::: "memory");
      for (int it = 0, kb = kb0; it < nch; ++it, kb += CH) {
        if (dst == ring_end) { dst = ring; bar = 0; parity ^= 1u; }
        if (it >= S && !t_mbar_wait(empty + bar, parity)) { ok = false; break; }
        t_tma_load3(dst + w_bytes, map_a, lead_full + bar, 0, y, kb);
        dst += stage_bytes; bar += 8;
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue: a warp holds 32 columns, one row after the other
    const int e = warp - 3, q = warp & 3;            // lanes 32 q .. of tensor memory
    const int RQ = R / 4;                            // rows per warp: column halves (q & 1) x row halves (q >> 1) x two warps each
    const int r0w = (q >> 1) * (R / 2) + (e >> 2) * RQ;      // first of this warp's rows in the group
    const int c = (q & 1) * 32 + lane, col = n0 + c;
    const bool col_on = col < a.N;
    const int own = SPLIT ? ((RQ + ks - 1) / ks + 3) / 4 * 4 : RQ;      // rows of a warp a CTA of the cluster owns, in fours
    const int j0 = SPLIT ? z * own : 0, j1 = min(RQ, j0 + own);
    const int lim = row0 + n_rows;
    constexpr int OWN_MAX = SPLIT ? 16 : 32;
    float gain = 0.f;
    if (EPI == PROJ_RESID && col_on) gain = __bfloat162float(a.gain_next[col]);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float xv[OWN_MAX];
    if (EPI == PROJ_RESID) {
#pragma unroll
      for (int j = 0; j < OWN_MAX; ++j) {
        const int r = row0 + r0w + j0 + j;
        xv[j] = j0 + j < j1 && r < lim && col_on ? __ldcg(a.x + (size_t)r * a.N + col) : 0.f;
      }
    } else {
      // scales of the norm in front: eight lanes per row, every load of the group's rows on its way at once
      const int t = tid - (PT_THREADS - PT_EPI_T), l8 = t & 7;
      float sum[PT_R_MAX / 32];
#pragma unroll
      for (int i = 0; i < PT_R_MAX / 32; ++i) sum[i] = 0.f;
      for (int p0 = 0; p0 < a.parts_in; p0 += 32) {
#pragma unroll
        for (int i = 0; i < PT_R_MAX / 32; ++i)
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int r = row0 + i * 32 + (t >> 3), pp = p0 + k * 8 + l8;
            if (r < lim && pp < a.parts_in) sum[i] += __ldcg(a.ssq_in + (size_t)r * a.ssq_stride + pp);
          }
      }
#pragma unroll
      for (int i = 0; i < PT_R_MAX / 32; ++i) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
        if (l8 == 0) inv_s[i * 32 + (t >> 3)] = rsqrtf(sum[i] * a.inv_width + a.eps);
      }
      // (all of it: a split's warp asks for the positions of whole chunks, which may end beyond the group's rows)
      if (EPI == PROJ_QKV && t < PT_R_MAX) meta_s[t] = row0 + t < lim ? __ldcg(a.row_meta + row0 + t) : make_int4(0, 0, 0, 0);
      t_epi_sync();
    }
    // (cos, sin) of a chunk of eight rows, requested a chunk ahead: even lanes hold the even rows', odd lanes the odd rows'
    const bool odd = lane & 1, rope = EPI == PROJ_QKV && a.rope_tab != nullptr && n0 < 2 * (a.N / 3);
    float2 cs[4];
    auto load_cs = [&](int jb) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        cs[k] = __ldg(a.rope_tab + (size_t)meta_s[EPI == PROJ_QKV ? (r0w + j0 + jb + 2 * k + odd) & (PT_R_MAX - 1) : 0].z * (kDh / 2) + c / 2);
    };
    if (rope && j0 < j1) load_cs(0);
    ok = t_mbar_wait_warp(acc_full, 0u);
    t_tmem_ask();
    same = *reinterpret_cast<volatile int *>(&same_s) != 0;
    ok = ok && same;
    t_fence_after();
    const uint32_t taddr = tmem_base_s + ((uint32_t)(q * 32) << 16) + (uint32_t)((e >> 2) * RQ);
    const float *red = reinterpret_cast<const float *>(t_raw + (ring - t_smem_u32(t_raw)));
    const uint32_t blk = (uint32_t)own * (PT_EPI_WARPS * 128);      // bytes of one owner's rows: [warp][fours of rows][32 columns][4]
    auto read_done = [&]() {                         // this warp has read its accumulators
      t_fence_before();
      __syncwarp();
      if (lane < 2) t_mbar_arrive_peer(t_peer(acc_read, leader + lane));
    };
    if (SPLIT) {
      // The ring is free: it takes this CTA's sums, one block per owner, and behind them the peers' sums of the rows it owns.
      // Row j of a warp belongs to CTA j / own of the splits, same half.
      if (e == 0) {
        if (lane == 0) t_mbar_expect_tx(red_full, (uint32_t)(ks - 1) * blk);
        __syncwarp();
        if (lane < ks) t_mbar_arrive_peer(t_peer(red_free, 2u * lane + half));
      }
      float4 *dst = reinterpret_cast<float4 *>(t_raw + (ring - t_smem_u32(t_raw))) + e * own * 8 + lane;
      for (int jb = 0, o = 0, jj = 0; ok && jb < RQ; jb += 8) {
        float v[8];
        t_tmem_ld8(taddr + jb, v);
#pragma unroll
        for (int i = 0; i < 8; i += 4) {             // four rows at a time
          dst[(size_t)o * (blk >> 4) + jj * 8] = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
          jj += 4;
          if (jj == own) { jj = 0; ++o; }
        }
      }
      read_done();
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      t_epi_sync();
      if (e == 0 && lane < ks && lane != z) {
        if (t_mbar_wait<true>(red_free, 0u)) t_copy_peer(t_peer(ring + (uint32_t)(ks + z) * blk, 2u * lane + half), ring + lane * blk, blk, t_peer(red_full, 2u * lane + half));
        else ok = false;
      }
      __syncwarp();
      const bool sums = t_mbar_wait_warp<true>(red_full, 0u);      // (whatever else happened: nobody leaves under a copy)
      ok = __all_sync(0xffffffffu, ok && sums);
      if (e == 0 && lane < ks) t_mbar_arrive_peer(t_peer(acc_read, 2u * lane + half));     // (the peers' sums are here: they may leave)
    } else if (!ok) {
      read_done();
    }
#pragma unroll
    for (int jb = 0; jb < OWN_MAX; jb += 8) {
      if (!ok || j0 + jb >= j1) break;
      float v[8];
      if (SPLIT) {
#pragma unroll
        for (int i = 0; i < 8; i += 4) {
          float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
          if (jb + i < own)
#pragma unroll
            for (int s = 0; s < 4; ++s)              // rank order
              if (s < ks) {
                const float4 u = *reinterpret_cast<const float4 *>(red + (size_t)(s == z ? s : ks + s) * (blk >> 2) + (e * own + jb + i) * 32 + lane * 4);
                t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
              }
          v[i] = t.x; v[i + 1] = t.y; v[i + 2] = t.z; v[i + 3] = t.w;
        }
      } else {
        t_tmem_ld8(taddr + jb, v);
        if (j0 + jb + 8 >= j1) read_done();
      }
      const int rl = r0w + j0 + jb, r = row0 + rl;   // row of v[0] in the group, among the packed rows
      auto on = [&](int i) { return j0 + jb + i < j1 && r + i < lim; };
      if (EPI == PROJ_RESID) {
        float f[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          v[i] += xv[jb + i];
          if (on(i) && col_on) a.x[(size_t)(r + i) * a.N + col] = v[i];
          f[i] = v[i] * v[i];                        // (columns beyond N are zero)
          v[i] *= gain;
        }
        // sums of the squares over the warp's 32 columns, eight rows at once: after three halvings a lane holds one row
#pragma unroll
        for (int o = 4, n = 4; o > 0; o >>= 1, n >>= 1) {
          const bool up = lane & o;
#pragma unroll
          for (int i = 0; i < n; ++i) {
            const float keep = up ? f[i + n] : f[i], give = up ? f[i] : f[i + n];
            f[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
          }
        }
        f[0] += __shfl_xor_sync(0xffffffffu, f[0], 8);
        f[0] += __shfl_xor_sync(0xffffffffu, f[0], 16);
        if (lane < 8 && on(lane) && n0 + (q & 1) * 32 < a.N) a.ssq_out[(size_t)(r + lane) * a.ssq_stride + (n0 + (q & 1) * 32) / 32] = f[0];
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] *= inv_s[(rl + i) & (PT_R_MAX - 1)];
        if (EPI == PROJ_RELU) {
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = fmaxf(v[i], 0.f);
        }
      }
      if (EPI == PROJ_QKV) {
        const int d = a.N / 3, which = n0 / d, hcol = n0 - which * d;      // (64 columns of one head)
        if (a.raw != nullptr) {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (on(i) && col_on) {
              if (a.raw_f32) reinterpret_cast<float *>(a.raw)[(size_t)(r + i) * a.N + col] = v[i];
              else reinterpret_cast<__nv_bfloat16 *>(a.raw)[(size_t)(r + i) * a.N + col] = __float2bfloat16(v[i]);
            }
        }
        if (rope) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float2 mine = cs[i >> 1];
            const float ox = __shfl_xor_sync(0xffffffffu, mine.x, 1), oy = __shfl_xor_sync(0xffffffffu, mine.y, 1);
            const bool own_row = odd == (bool)(i & 1);
            const float2 t = make_float2(own_row ? mine.x : ox, own_row ? mine.y : oy);
            const float other = __shfl_xor_sync(0xffffffffu, v[i], 1);
            v[i] = odd ? other * t.y + v[i] * t.x : v[i] * t.x - other * t.y;
          }
          if (jb + 8 < OWN_MAX && j0 + jb + 8 < j1) load_cs(jb + 8);
        }
#pragma unroll
        for (int i = 0; i < 8; i += 2) {             // even lanes take row i, odd lanes row i + 1, two columns each
          const float got = __shfl_xor_sync(0xffffffffu, odd ? v[i] : v[i + 1], 1);
          const uint32_t pk = odd ? t_pack2(got, v[i + 1]) : t_pack2(v[i], got);
          if (!on(i + odd) || !col_on) continue;
          if (which == 0) {
            *reinterpret_cast<uint32_t *>(a.out + (size_t)(r + i + odd) * d + hcol + (c & ~1)) = pk;
          } else {
            const int4 m = meta_s[rl + i + odd];
            __nv_bfloat16 *dst = a.kv_pool + kv_block_offset(a.layer, a.pool, m.x, d / kDh, hcol / kDh, a.P);
            *reinterpret_cast<uint32_t *>(dst + kv_entry_offset<__nv_bfloat16>(m.y, c & ~1, which - 1)) = pk;
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
          const float got = __shfl_xor_sync(0xffffffffu, odd ? v[i] : v[i + 1], 1);
          const uint32_t pk = odd ? t_pack2(got, v[i + 1]) : t_pack2(v[i], got);
          if (on(i + odd) && col_on) *reinterpret_cast<uint32_t *>(a.out + (size_t)(r + i + odd) * a.N + (col & ~1)) = pk;
        }
      }
    }
  }
  if (!same) atomicExch(a.status, (int)PD_ERR_DEVICE);
  else if (!ok) atomicExch(a.status, (int)PD_ERR_TIMEOUT);
  if (warp == 1) {
    // every warp of both CTAs is through with the accumulators, and the peers with this CTA's sums (nobody leaves while another
    // CTA reaches into it)
    __syncwarp();
    if (!t_mbar_wait_warp<true>(acc_read, 0u)) atomicExch(a.status, (int)PD_ERR_TIMEOUT);
    __syncwarp();
    t_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base_s), "r"(PT_TMEM) : "memory");
    // neither CTA leaves while the other has a pair-wide instruction to finish
    if (lane == 0) t_mbar_arrive_peer(t_peer(peer_gave, peer));
    if (!t_mbar_wait_warp<true>(peer_gave, 0u)) atomicExch(a.status, (int)PD_ERR_TIMEOUT);
  }
}

// ---- host side ------------------------------------------------------------------------------------
namespace {
struct Plan { int slices, ks, groups, gy; };
// K splits of at most 1024 each, at most four; row groups: one CTA per SM, more where a group would not fit.
Plan plan(int K, int N, int rows_cap) {
  Plan p;
  p.slices = (N + 2 * PT_COLS - 1) / (2 * PT_COLS);
  p.ks = std::min((K / PT_BK + 15) / 16, 4);
  p.groups = std::max(1, kSms / 2 / (p.slices * p.ks));
  p.gy = std::max(std::min(p.groups, (rows_cap + 15) / 16), (rows_cap + PT_R_MAX - 1) / PT_R_MAX);
  return p;
}

template <typename F>
cudaError_t each_kernel(int epi, bool split, bool all, F f) {
  cudaError_t e = cudaSuccess;
  auto one = [&](int ep, bool sp, auto kernel) { if (e == cudaSuccess && (all || (ep == epi && sp == split))) e = f(kernel); };
  one(PROJ_STORE, false, proj_tc_kernel<PROJ_STORE, false>);
  one(PROJ_RELU, false, proj_tc_kernel<PROJ_RELU, false>);
  one(PROJ_RESID, false, proj_tc_kernel<PROJ_RESID, false>);
  one(PROJ_QKV, false, proj_tc_kernel<PROJ_QKV, false>);
  one(PROJ_STORE, true, proj_tc_kernel<PROJ_STORE, true>);
  one(PROJ_RELU, true, proj_tc_kernel<PROJ_RELU, true>);
  one(PROJ_RESID, true, proj_tc_kernel<PROJ_RESID, true>);
  one(PROJ_QKV, true, proj_tc_kernel<PROJ_QKV, true>);
  return e;
}
}  // namespace

// Whole blocks of K, 16-byte tensor-map rows.
bool proj_tc_supported(int K, int N) { return K >= PT_BK && K % PT_BK == 0 && N % 8 == 0; }

// Against the register products of proj_mma.cu, whole decodes of four layers, 512 keys, every product on the one or the other, "register /
// tensor memory" with about two thirds and with about 0.42 of the allocated rows active, inner sides of four widths:
//   width    130 rows       256           384           512           640           768
//    256   0.813 0.785   0.864 0.832   0.898 0.860   0.933 0.895   0.991 0.912   1.022 0.931
//    512   0.901 0.861   0.982 0.935   1.075 0.997   1.146 1.057   1.206 1.111   1.237 1.151
//    768   1.007 0.935   1.205 1.061   1.369 1.206   1.490 1.318   1.631 1.400   1.744 1.490
//   1024   1.077 0.973   1.263 1.117   1.437 1.276   1.615 1.391   1.594 1.438   1.708 1.509
// and with other inner sides:
//   512 x 512    0.816 0.784 at 130 rows, 0.992 0.933 at 512, 1.054 1.000 at 768
//   256 x 8192   0.996 0.910 at 130 rows, 1.413 1.220 at 512, 1.593 1.315 at 768
//    64 x 8192   0.918 0.854 at 130 rows, 1.220 1.084 at 512, 1.359 1.165 at 768
// A register product walks its rows at a rate that falls with its weights, one on tensor memory hardly notices either: the line where both
// take the same is rows = 60 + 1.5e8 / weights.  (A side below 128 counts as 128: 64 x 4096, 1.081 at 512 rows, would seem alike only at 632.)
// Whole decodes by this rule, each product by itself, are between 0.95 and 1.12 times as fast as with the better of the two for all products.
bool proj_tc_better(int K, int N, int rows_cap) {
  return rows_cap > 128 && (long long)(rows_cap - 60) * std::max(K, 128) * std::max(N, 128) > 150000000;
}

cudaError_t proj_tc_prepare() {
  return each_kernel(0, false, true, [](auto kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PT_SMEM); });
}

cudaError_t encode_proj_tc_weight_maps(ProjTcWeightMaps *out, const void *w, uint64_t K, uint64_t N) {
  const uint64_t gdim[2] = {N, K}, gstride[1] = {N * 2};
  for (int i = 0; i < 2; ++i) {
    const uint32_t box[2] = {PT_COLS, (uint32_t)PT_BK << (i + 1)};
    cudaError_t e = encode_tensor_map(&out->k[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, w, gdim, gstride, box, nullptr);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
cudaError_t encode_proj_tc_act_maps(ProjTcActMaps *out, const void *act, uint64_t rows, uint64_t K) {
  const uint64_t gdim[3] = {PT_BK, rows, K / PT_BK}, gstride[2] = {K * 2, PT_BK * 2};
  for (int i = 0; i < PT_R_MAX / 32; ++i) {
    const uint32_t box[3] = {PT_BK, 16u * (i + 1), (uint32_t)pt_blocks(32 * (i + 1))};
    cudaError_t e = encode_tensor_map(&out->box[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, act, gdim, gstride, box, nullptr);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_proj_tc(int epi, const ProjTcWeightMaps &map_w, const ProjTcActMaps &maps, const ProjArgs &a_in, int32_t *status, cudaStream_t s) {
  ProjTcArgs a;
  static_cast<ProjArgs &>(a) = a_in;
  const Plan p = plan(a.K, a.N, a.rows_cap);
  a.groups = p.groups; a.status = status;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * p.slices, p.gy, p.ks);
  cfg.blockDim = dim3(PT_THREADS, 1, 1);
  cfg.dynamicSmemBytes = PT_SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = p.ks;
  cfg.attrs = attr; cfg.numAttrs = 2;
  return each_kernel(epi, p.ks > 1, false, [&](auto kernel) { return cudaLaunchKernelEx(&cfg, kernel, map_w, maps, a); });
}

}  // namespace pd
