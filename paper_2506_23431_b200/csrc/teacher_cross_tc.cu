// Cross-attention of the teacher-forced forward (every target row of a sequence against its whole context) on the
// 5th-generation tensor cores.
//
// One CTA per block of up to 128 query rows of one sequence and head, two CTAs per SM.  Warp 0 fetches the queries and streams 128-key
// tiles of keys and values through a ring with TMA; one lane of warp 1 issues the products: S = Q K^T of a whole tile into 128
// columns of tensor memory (as soon as the second half of the tile before has been read out of them), O += P V per half; warps 2-5
// hold one row per thread: no shuffles, a half's 64 scores come with tcgen05.ld, its weights go back as bf16 with tcgen05.st, the A operand
// of P V (through shared memory instead, with 64-key products, both operands' reads and the fences cost 16 us of 205).
// The running maximum lags: O is rescaled only when a row's maximum has grown by more than 2^8, so that the usual
// half leaves O alone (weights up to 2^8 lose nothing in bf16, and the same stale maximum divides out).
// What bounds it: the loads and products and their hand-overs between the warps - without the exponentials a launch takes 176 of its
// 190 us.  Two CTAs per SM, so that one's exponentials (64 x 128 per half, 512 cycles at 16 a cycle) run under the other's products.  11.5 k rows, 32
// contexts of 2048, 16 heads, per layer: 190 us, where mma.sync (32 rows per warp, 64-key tiles) took 389 us; 3 documents of 1000 in 64-row
// blocks, 12 heads: 13.9 us against 17.5 us.
// Every mbarrier wait is bounded: on expiry the kernel records PD_ERR_TIMEOUT, stops waiting, falls through to the
// common exit and frees its tensor memory.
#include <float.h>

#include "pd_internal.h"

namespace pd {

namespace {

constexpr int XC_M = 128, XC_K = 128, XC_H = 64;   // query rows per CTA, keys per tile and per half
constexpr int XC_STAGES = 2;
constexpr int XC_TILE = XC_K * kDh * 2;            // keys (or values) of a tile: 16 KB
constexpr int XC_STAGE = 2 * XC_TILE;
constexpr int XC_Q = XC_M * kDh * 2;
constexpr int XC_THREADS = 192;
constexpr int XC_SMEM = XC_Q + XC_STAGES * XC_STAGE + 256 /*barriers*/ + 1024 /*alignment slack*/;
constexpr int XC_TMEM = 256, XC_O = 128, XC_W = 192;       // scores at columns 0 - 127, O from 128, the halves' weights from 192 and 224
constexpr float XC_LAG = 8.f;
constexpr uint32_t XC_SPIN_LIMIT = 1u << 24;

__device__ __forceinline__ uint32_t c_smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void c_mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void c_mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void c_mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool c_mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: false when the phase did not complete within the spin limit.
__device__ __forceinline__ bool c_mbar_wait(uint32_t bar, uint32_t parity) {
  for (uint32_t it = 0; it < XC_SPIN_LIMIT; ++it)
    if (c_mbar_try(bar, parity)) return true;
  return false;
}
// The same by a whole warp, whose lanes take every turn together: also where the limit runs out none goes on without the others.
__device__ __forceinline__ bool c_mbar_wait_warp(uint32_t bar, uint32_t parity) {
  for (uint32_t it = 0; it < XC_SPIN_LIMIT; ++it)
    if (__all_sync(0xffffffffu, c_mbar_try(bar, parity))) return true;
  return false;
}
__device__ __forceinline__ void c_tma_load_2d(uint32_t dst, const CUtensorMap *tmap, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(tmap), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
// Shared-memory matrix descriptor of rows of 128 bytes, 128-byte swizzle, 1024 B between groups of eight rows.  The same words serve
// a K-major operand (rows = M or N) and, with one 64-wide span of it, an MN-major one (rows = K).  Low word: address >> 4; the high one is constant.
constexpr uint32_t XC_DESC_HI = 64u | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t c_desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (64u << 16); }
// One lane of a converged warp.
__device__ __forceinline__ bool c_elect() {
  uint32_t on;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(on));
  return on != 0;
}
// instruction descriptor of kind::f16: D fp32, A and B bf16, N >> 3 at bit 17, M >> 4 at bit 24; bit 16: B is MN-major
constexpr uint32_t xc_idesc(int n) { return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(XC_M >> 4) << 24); }
__device__ __forceinline__ void c_mma_bf16(uint32_t tmem_d, uint32_t alo, uint32_t blo, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %5};\n\t"
      "mov.b64 db, {%2, %5};\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(alo), "r"(blo), "r"(idesc), "r"(accumulate), "n"(XC_DESC_HI)
      : "memory");
}
// A from tensor memory: two consecutive K values per 32-bit column, one row per lane
__device__ __forceinline__ void c_mma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint32_t blo, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
      "mov.b64 db, {%2, %5};\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(tmem_a), "r"(blo), "r"(idesc), "r"(accumulate), "n"(XC_DESC_HI)
      : "memory");
}
__device__ __forceinline__ void c_mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 32 columns of this warp's quarter of tensor memory, one row per lane (complete after c_tmem_ld_wait)
template <int O>
__device__ __forceinline__ void c_tmem_ld32(uint32_t taddr, uint32_t (&r)[64]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[O + 0]), "=r"(r[O + 1]), "=r"(r[O + 2]), "=r"(r[O + 3]), "=r"(r[O + 4]), "=r"(r[O + 5]), "=r"(r[O + 6]), "=r"(r[O + 7]),
        "=r"(r[O + 8]), "=r"(r[O + 9]), "=r"(r[O + 10]), "=r"(r[O + 11]), "=r"(r[O + 12]), "=r"(r[O + 13]), "=r"(r[O + 14]),
        "=r"(r[O + 15]), "=r"(r[O + 16]), "=r"(r[O + 17]), "=r"(r[O + 18]), "=r"(r[O + 19]), "=r"(r[O + 20]), "=r"(r[O + 21]),
        "=r"(r[O + 22]), "=r"(r[O + 23]), "=r"(r[O + 24]), "=r"(r[O + 25]), "=r"(r[O + 26]), "=r"(r[O + 27]), "=r"(r[O + 28]),
        "=r"(r[O + 29]), "=r"(r[O + 30]), "=r"(r[O + 31])
      : "r"(taddr)
      : "memory");
}
// The registers pass through the second statement, so that nothing reads them ahead of the wait.
__device__ __forceinline__ void c_tmem_ld_wait(uint32_t (&r)[64]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 64; i += 16)
    asm volatile("" : "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3]), "+r"(r[i + 4]), "+r"(r[i + 5]), "+r"(r[i + 6]), "+r"(r[i + 7]),
                      "+r"(r[i + 8]), "+r"(r[i + 9]), "+r"(r[i + 10]), "+r"(r[i + 11]), "+r"(r[i + 12]), "+r"(r[i + 13]), "+r"(r[i + 14]), "+r"(r[i + 15]));
}
// Two fp32 operations in one instruction (each rounded as its own).
__device__ __forceinline__ uint64_t c_f2(float lo, float hi) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
__device__ __forceinline__ uint64_t c_fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t v;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
  return v;
}
__device__ __forceinline__ uint64_t c_add2(uint64_t a, uint64_t b) {
  uint64_t v;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ float2 c_u2(uint64_t v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
template <int O, int N>
__device__ __forceinline__ void c_tmem_st32(uint32_t taddr, const uint32_t (&r)[N]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[O + 0]), "r"(r[O + 1]), "r"(r[O + 2]), "r"(r[O + 3]), "r"(r[O + 4]), "r"(r[O + 5]), "r"(r[O + 6]), "r"(r[O + 7]),
        "r"(r[O + 8]), "r"(r[O + 9]), "r"(r[O + 10]), "r"(r[O + 11]), "r"(r[O + 12]), "r"(r[O + 13]), "r"(r[O + 14]), "r"(r[O + 15]),
        "r"(r[O + 16]), "r"(r[O + 17]), "r"(r[O + 18]), "r"(r[O + 19]), "r"(r[O + 20]), "r"(r[O + 21]), "r"(r[O + 22]), "r"(r[O + 23]),
        "r"(r[O + 24]), "r"(r[O + 25]), "r"(r[O + 26]), "r"(r[O + 27]), "r"(r[O + 28]), "r"(r[O + 29]), "r"(r[O + 30]), "r"(r[O + 31])
      : "memory");
}
__device__ __forceinline__ void c_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void c_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ float c_ex2(float x) {   // 2^x; ex2(-inf) = 0
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t c_pack(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

__global__ void __launch_bounds__(XC_THREADS, 2) teacher_cross_kernel(const __grid_constant__ CUtensorMap map_q,
                                                                      const __grid_constant__ CUtensorMap map_kv, DenseAttnArgs a) {
  extern __shared__ uint8_t c_raw[];
  __shared__ uint32_t tmem_base_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = blockIdx.x, h = blockIdx.y;
  const int q0 = a.grp_row0[grp], nq = a.grp_n[grp], nk = a.grp_keys[grp];
  const int n_tiles = (nk + XC_K - 1) / XC_K, n_halves = (nk + XC_H - 1) / XC_H;
  const uint32_t base = (c_smem_u32(c_raw) + 1023u) & ~1023u;
  const uint32_t q_s = base, ring = q_s + XC_Q;
  const uint32_t bar_q = ring + XC_STAGES * XC_STAGE, bar_full = bar_q + 8, bar_empty = bar_full + 8 * XC_STAGES, bar_s = bar_empty + 8 * XC_STAGES,
                 bar_read = bar_s + 8, bar_p = bar_read + 8, bar_pv = bar_p + 16;
  if (tid == 0) {
    const uint32_t warps = (uint32_t)(nq + 31) / 32;       // softmax warps that have rows
    c_mbar_init(bar_q, 1);
    for (int s = 0; s < XC_STAGES; ++s) { c_mbar_init(bar_full + 8 * s, 1); c_mbar_init(bar_empty + 8 * s, 1); }
    c_mbar_init(bar_s, 1);
    c_mbar_init(bar_read, warps);
    c_mbar_init(bar_p, warps); c_mbar_init(bar_p + 8, warps);
    c_mbar_init(bar_pv, 1); c_mbar_init(bar_pv + 8, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(c_smem_u32(&tmem_base_s)), "r"(XC_TMEM) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  c_fence_before();
  __syncthreads();
  c_fence_after();
  const uint32_t tmem = tmem_base_s;
  bool ok = true;

  if (warp == 0) {
    // ------------------------------------------------------------------ producer (one lane)
    if (lane == 0) {
      c_mbar_expect_tx(bar_q, XC_Q);
      c_tma_load_2d(q_s, &map_q, bar_q, h * kDh, q0);       // rows beyond the block belong to nobody's output
      const int y = (int)(ctx_kv_offset(a.layer, a.B, a.grp_seq[grp], a.H, h, 0, a.ctx) / kDh);
      int s = 0;
      uint32_t u = 0;
      for (int j = 0; j < n_tiles; ++j) {
        if (!c_mbar_wait(bar_empty + 8 * s, (u & 1u) ^ 1u)) { ok = false; break; }
        c_mbar_expect_tx(bar_full + 8 * s, XC_STAGE);
        const uint32_t dst = ring + s * XC_STAGE;
        c_tma_load_2d(dst, &map_kv, bar_full + 8 * s, 0, y + j * XC_K);
        c_tma_load_2d(dst + XC_TILE, &map_kv, bar_full + 8 * s, 0, y + a.ctx + j * XC_K);
        if (++s == XC_STAGES) { s = 0; ++u; }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ products (one lane).  The whole warp walks: in a loop that a single lane
    // walks the descriptors stay out of the uniform registers the products read, and a product costs 128 cycles to issue where it takes 52 to 68
    const uint32_t q_lo = c_desc_lo(q_s), ring_lo = c_desc_lo(ring);
    auto scores = [&](int tile) {
      const int s = tile % XC_STAGES;
      if (!c_mbar_wait_warp(bar_full + 8 * s, (uint32_t)(tile / XC_STAGES) & 1u)) { ok = false; return; }
      c_fence_after();
      if (c_elect()) {
#pragma unroll
        for (int k = 0; k < kDh / 16; ++k)
          c_mma_bf16(tmem, q_lo + k * 2, ring_lo + s * (XC_STAGE >> 4) + k * 2, xc_idesc(XC_K), k > 0 ? 1u : 0u);
        c_mma_commit(bar_s);
      }
    };
    ok = c_mbar_wait_warp(bar_q, 0);
    if (ok) scores(0);
    for (int j = 0; j < n_halves && ok; ++j) {
      const int tile = j >> 1, s = tile % XC_STAGES;
      if ((j & 1) != 0 && tile + 1 < n_tiles) {             // the tile's scores are all read: the next one's
        if (!c_mbar_wait_warp(bar_read, (uint32_t)tile & 1u)) { ok = false; break; }
        c_fence_after();
        scores(tile + 1);
      }
      if (!ok || !c_mbar_wait_warp(bar_p + 8 * (j & 1), (uint32_t)(j >> 1) & 1u)) { ok = false; break; }
      c_fence_after();
      if (c_elect()) {
        const uint32_t v_lo = ring_lo + s * (XC_STAGE >> 4) + (XC_TILE >> 4) + (j & 1) * (XC_TILE / 2 >> 4);
#pragma unroll
        for (int k = 0; k < XC_H / 16; ++k)                 // 16 keys = 8 columns of weights, 16 rows of values
          c_mma_bf16_ta(tmem + XC_O, tmem + XC_W + (uint32_t)((j & 1) * 32 + k * 8), v_lo + k * (2048 >> 4), xc_idesc(kDh) | (1u << 16),
                        (j > 0 || k > 0) ? 1u : 0u);
        if ((j & 1) != 0) c_mma_commit(bar_empty + 8 * s);
        c_mma_commit(bar_pv + 8 * (j & 1));
      }
    }
  } else if ((warp & 3) * 32 < nq) {
    // ------------------------------------------------------------------ softmax: one row per thread
    const int row = (warp & 3) * 32 + lane;                 // tensor-memory lanes 32 (warp & 3) .. + 31 belong to this warp
    const uint32_t tm = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const float sl2 = a.scale_log2e;
    float m_used = 0.f, l = 0.f;
    uint32_t r[64];                                         // the row's scores of a half
    auto fetch = [&](int j) {
      if ((j & 1) == 0) {
        if (!c_mbar_wait(bar_s, (uint32_t)(j >> 1) & 1u)) { ok = false; return; }
        __syncwarp();
        c_fence_after();
      }
      c_tmem_ld32<0>(tm + (uint32_t)(j & 1) * 64u, r);
      c_tmem_ld32<32>(tm + (uint32_t)(j & 1) * 64u + 32u, r);
    };
    fetch(0);
    for (int j = 0; j < n_halves && ok; ++j) {
      c_tmem_ld_wait(r);
      if (j & 1) {
        c_fence_before();
        __syncwarp();
        if (lane == 0) c_mbar_arrive(bar_read);
      }
      const int nv = nk - j * XC_H;
      if (nv < XC_H) {                                      // the last half: absent keys weigh nothing, and their value rows, which hold
#pragma unroll                                              // whatever follows in memory, are cleared (no copy into this stage follows)
        for (int i = 0; i < 64; ++i) if (i >= nv) r[i] = 0xff800000u;
        const int s = (j >> 1) % XC_STAGES;
        if (!c_mbar_wait(bar_full + 8 * s, (uint32_t)((j >> 1) / XC_STAGES) & 1u)) { ok = false; break; }
        for (int i = nv * 8 + row; i < XC_H * 8; i += (nq + 31) / 32 * 32)
          asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(ring + s * XC_STAGE + XC_TILE + (j & 1) * (XC_TILE / 2) + i * 16), "r"(0u) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int i = 0; i < 64; ++i) mx[i & 3] = fmaxf(mx[i & 3], __uint_as_float(r[i]));
      const float m = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sl2;
      if (j == 0) {
        m_used = fmaxf(m, -FLT_MAX);                        // (finite also where all 64 scores have overflowed to -inf: they weigh 0)
      } else if (__any_sync(0xffffffffu, m > m_used + XC_LAG)) {      // some row's maximum has moved too far: rescale this warp's rows of O
        if (!c_mbar_wait(bar_pv + 8 * ((j - 1) & 1), (uint32_t)((j - 1) >> 1) & 1u)) { ok = false; break; }
        __syncwarp();
        c_fence_after();
        const float m_new = fmaxf(m_used, m), c = c_ex2(m_used - m_new);
        uint32_t o[64];
        c_tmem_ld32<0>(tm + XC_O, o);
        c_tmem_ld32<32>(tm + XC_O + 32u, o);
        c_tmem_ld_wait(o);
#pragma unroll
        for (int i = 0; i < 64; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * c);
        c_tmem_st32<0>(tm + XC_O, o);
        c_tmem_st32<32>(tm + XC_O + 32u, o);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        l *= c;
        m_used = m_new;
      }
      uint32_t pk[32];
      const uint64_t scale2 = c_f2(sl2, sl2), ref2 = c_f2(-m_used, -m_used);
      uint64_t sum2[4] = {0, 0, 0, 0};
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float2 x = c_u2(c_fma2(c_f2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1])), scale2, ref2));
        const float p0 = c_ex2(x.x), p1 = c_ex2(x.y);
        sum2[i & 3] = c_add2(sum2[i & 3], c_f2(p0, p1));
        pk[i] = c_pack(p0, p1);
      }
      const float2 sum = c_u2(c_add2(c_add2(sum2[0], sum2[1]), c_add2(sum2[2], sum2[3])));
      l += sum.x + sum.y;
      if (j + 1 < n_halves) fetch(j + 1);                   // on its way while the weights leave
      if (j > 1 && !c_mbar_wait(bar_pv + 8 * (j & 1), (uint32_t)((j >> 1) - 1) & 1u)) { ok = false; break; }      // the weights two halves back are consumed
      __syncwarp();
      c_tmem_st32<0>(tm + XC_W + (uint32_t)(j & 1) * 32u, pk);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      c_fence_before();
      __syncwarp();
      // A barrier each for even and odd halves: a warp arrives for half j behind its wait for the products of half j - 2, which start when
      // every warp has arrived for that one, so no arrival is ever counted into the half before.  (With one barrier for all halves a
      // warp could arrive for j while another still rescales O for j - 1, whose products then started on unfinished weights.)
      if (lane == 0) c_mbar_arrive(bar_p + 8 * (j & 1));
    }
    if (ok && !c_mbar_wait(bar_pv + 8 * ((n_halves - 1) & 1), (uint32_t)((n_halves - 1) >> 1) & 1u)) ok = false;
    if (__all_sync(0xffffffffu, ok)) {
      c_fence_after();
      uint32_t o[64];
      c_tmem_ld32<0>(tm + XC_O, o);
      c_tmem_ld32<32>(tm + XC_O + 32u, o);
      c_tmem_ld_wait(o);
      if (row < nq) {
        const float inv = 1.f / l;
        uint4 *dst = reinterpret_cast<uint4 *>(a.out + (size_t)(q0 + row) * a.d + (size_t)h * kDh);
        auto two = [&](int i) { return c_pack(__uint_as_float(o[i]) * inv, __uint_as_float(o[i + 1]) * inv); };
#pragma unroll
        for (int c = 0; c < 8; ++c) dst[c] = make_uint4(two(8 * c), two(8 * c + 2), two(8 * c + 4), two(8 * c + 6));
      }
    }
  }
  if (!ok && lane == 0) atomicExch(a.status, (int)PD_ERR_TIMEOUT);
  __syncwarp();
  c_fence_before();
  __syncthreads();
  if (warp == 1) {
    c_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(XC_TMEM) : "memory");
  }
}

}  // namespace

cudaError_t teacher_cross_tc_prepare() {
  return cudaFuncSetAttribute(teacher_cross_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, XC_SMEM);
}

// Tensor maps: queries [rows][d] in boxes of 128 rows x one head; the context keys/values as rows of one position of one
// (layer, sequence, head, K or V), in boxes of one tile.
cudaError_t encode_teacher_cross_maps(CUtensorMap *map_q, CUtensorMap *map_kv, const void *q, uint64_t rows, uint64_t d, const void *kv_c,
                                      uint64_t kv_rows) {
  const uint64_t qdim[2] = {d, rows}, qstride[1] = {d * 2};
  const uint32_t qbox[2] = {kDh, XC_M};
  cudaError_t e = encode_tensor_map(map_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, q, qdim, qstride, qbox, nullptr);
  if (e != cudaSuccess) return e;
  const uint64_t kdim[2] = {kDh, kv_rows}, kstride[1] = {kDh * 2};
  const uint32_t kbox[2] = {kDh, XC_K};
  return encode_tensor_map(map_kv, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, kv_c, kdim, kstride, kbox, nullptr);
}

cudaError_t launch_teacher_cross_tc(const CUtensorMap &map_q, const CUtensorMap &map_kv, const DenseAttnArgs &a, cudaStream_t s) {
  if (a.n_groups < 1) return cudaSuccess;
  teacher_cross_kernel<<<dim3(a.n_groups, a.H), XC_THREADS, XC_SMEM, s>>>(map_q, map_kv, a);
  return cudaGetLastError();
}

}  // namespace pd
