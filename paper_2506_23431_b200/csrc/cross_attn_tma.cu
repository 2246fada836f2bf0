// Batched cross-attention for the bf16 path (sm_100a): every active subsequence of a sequence
// is a query row against the shared encoder keys/values (all context positions < ctx_len
// visible, no positional term).  This is the one part of the step that is a dense S x L_ctx
// contraction, so it runs on tensor cores; it stays HBM-bound (about S flop per byte).
//
// A (sequence, head) pair - its queries against its context - is a segment; a cluster of 1, 2, 4 or 8 CTAs
// takes one, every CTA an equal share of its 128-key tiles, two CTAs per SM (8-bit: four).  In every CTA a producer warp
// streams the K and V tiles of its share (16 KB each, contiguous) through a ring of shared-memory stages
// with TMA (cp.async.bulk.tensor.2d, 128-byte swizzle, completion on an mbarrier); four consumer warps each
// take 32 keys of every tile: S = Q K^T with mma.sync m16n8k16 (bf16 in, fp32 accumulate), online softmax in
// the log2 domain with quad shuffles, O += P V.  At the end the warps' (m, l, O) are tree-merged through
// shared memory into warp 0; in a cluster the other CTAs push that state into the first one's shared memory,
// which merges them in rank order (deterministic) and writes the output.  A segment without an active
// row ends at once, and the hardware's block scheduler fills its place.
// Per launch, us, bf16, sequences x heads x context x rows: 1 x 12 x 777 x 8 6.2, 4 x 12 x 777 x 8 8.3, 8 x 16 x 4096 x 10 26.7,
// 16 x 12 x 1000 x 9 13.9, 32 x 16 x 2048 x 12 45.4, 64 x 12 x 1024 x 7 37.9.
// Every mbarrier wait is bounded: on expiry the kernel records PD_ERR_TIMEOUT and drains.
//
// 8-bit variant (FP8 = true): the context keys/values are E4M3 codes with one scale per (layer,
// sequence, head, keys | values) - half the bytes of the dominant term of a decode step.  Keys are
// stored [position][64] (a 128-key tile is 64 lines of 128 bytes), values transposed [dim][position],
// so that both reach the tensor cores through plain ldmatrix: a thread's 32-bit fragment word holds
// four consecutive codes (four dims of a key, or four keys of a dim), widened to two f16 pairs in
// registers (cvt.rn.f16x2.e4m3x2, exact).  The order of the sixteen dims (keys) inside a k16 step is
// therefore 4 tig + {0, 1} | 4 tig + {2, 3} instead of 2 tig + {0, 1} | 2 tig + 8 + {0, 1}; queries
// (score columns) are loaded with the same permutation, which a contraction does not see.  Queries and
// softmax weights go through f16 (exact for bf16 queries in f16's range; 11 bits for the weights), the
// key scale is folded into the score scale and the value scale into the final 1 / l.  Stages are 16 KB.
#include <cuda_fp16.h>

#include "pd_internal.h"

namespace pd {

constexpr int XK = 128;                   // keys per tile
// CTAs per SM and the ring: two with three 32 KB stages (bf16), four with three 16 KB stages (8-bit, up to 16 rows).  The 8-bit
// kernel waits on its own arithmetic between tiles more than on memory, so it wants warps rather than depth: 32 sequences x 16 heads x 2048
// keys 33.5 us with two CTAs (96 KB rings), 36.8 with three (512 segments leave a thin second wave), 29.2 with four, the same with
// two stages; its loads alone take 25.7 us.  The bf16 kernel is within 2 us of its loads alone (44.6 us there).  Two row tiles need the
// registers of two CTAs per SM.
__host__ __device__ constexpr int xctas(int mt, bool fp8) { return fp8 && mt == 1 ? 4 : 2; }      // CTAs per SM
__host__ __device__ constexpr int xring_bytes(int mt, bool fp8) { return fp8 && mt == 1 ? 48 * 1024 : 96 * 1024; }
// consumer warps, each taking 32 keys of a tile.  (Eight warps of 16 keys each were measured in both
// variants and lost: 50.3 against 49.2 us per full bf16 launch, 31.9 against 28.7 us per 8-bit launch.)
constexpr int XCW = 4, XTHREADS = (XCW + 1) * 32;
constexpr int XREC_WORDS = 36;            // per lane and 16-row tile: 32 output values, 2 maxima, 2 sums
constexpr int XREC_FLOATS = XREC_WORDS * 32;
__host__ __device__ constexpr int xsmem(int mt, bool fp8) { return xring_bytes(mt, fp8) + 128 /*barriers*/ + 1024 /*alignment slack*/; }
constexpr uint32_t XSPIN_LIMIT = 1u << 24;

bool cross_attn_tma_supported(const Dims &dm) { return dm.C <= 32; }

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
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
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (uint32_t it = 0; it < XSPIN_LIMIT; ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *tmap, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(tmap), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *tmap, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(tmap), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                        uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
  __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}
// two E4M3 codes (the low or the high half of a fragment word) -> f16 pair; every E4M3 value is an f16 value.
// (Widening with integer instructions instead - byte permute, shift, mask: the codes' values times 2^-8 -
// gave the same results and a slower kernel: 39 against 30 us per launch.)
__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint32_t word, int high) {
  uint32_t r;
  const unsigned short v = (unsigned short)(high ? (word >> 16) : (word & 0xffffu));
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(r) : "h"(v));
  return r;
}
__device__ __forceinline__ uint32_t bf16x2_to_f16x2(uint32_t w) {
  const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162 *>(&w);
  const __half2 hh = __float22half2_rn(__bfloat1622float2(b));
  return *reinterpret_cast<const uint32_t *>(&hh);
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}
template <int THREADS> __device__ __forceinline__ void consumer_bar_sync() { asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory"); }

// Everything the kernel before wrote (queries) is read behind this; keys, values, row counts and context lengths are
// older, so the producer streams ahead of it.
__device__ __forceinline__ void x_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Byte offset of (row, 16-byte chunk) inside a 128-byte-swizzled tile whose rows are 128 bytes.
__device__ __forceinline__ uint32_t swz(int row, int chunk) { return (uint32_t)(row * 128 + ((chunk ^ (row & 7)) << 4)); }

__device__ __forceinline__ float ex2f(float x) {   // 2^x; ex2(-inf) = 0
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// One warp's (or one CTA's) state for a 16-row query tile in mma fragment layout: this lane holds
// columns dn*8 + 2*tig, +1 of rows g (o[dn][0..1], m0, l0) and g + 8 (o[dn][2..3], m1, l1).
struct TileAcc {
  float o[8][4];
  float m0, m1, l0, l1;
  __device__ __forceinline__ void clear() {
    m0 = m1 = -INFINITY; l0 = l1 = 0.f;
#pragma unroll
    for (int dn = 0; dn < 8; ++dn) o[dn][0] = o[dn][1] = o[dn][2] = o[dn][3] = 0.f;
  }
  // record layout [word][lane]: consecutive lanes touch consecutive words (coalesced, no bank conflicts)
  __device__ __forceinline__ void store(float *rec, int lane) const {
#pragma unroll
    for (int dn = 0; dn < 8; ++dn)
#pragma unroll
      for (int x = 0; x < 4; ++x) rec[(dn * 4 + x) * 32 + lane] = o[dn][x];
    rec[32 * 32 + lane] = m0; rec[33 * 32 + lane] = m1; rec[34 * 32 + lane] = l0; rec[35 * 32 + lane] = l1;
  }
  // acc <- acc (+) record, the log-sum-exp merge of two partial softmax states
  __device__ __forceinline__ void merge(const float *rec, int lane) {
    auto ld = [&](int w) { return rec[w * 32 + lane]; };
    const float om0 = ld(32), om1 = ld(33), ol0 = ld(34), ol1 = ld(35);
    const float M0 = fmaxf(m0, om0), M1 = fmaxf(m1, om1);
    const float r0 = M0 == -INFINITY ? 0.f : M0, r1 = M1 == -INFINITY ? 0.f : M1;
    const float a0 = ex2f(m0 - r0), b0 = ex2f(om0 - r0), a1 = ex2f(m1 - r1), b1 = ex2f(om1 - r1);
    m0 = M0; m1 = M1;
    l0 = l0 * a0 + ol0 * b0; l1 = l1 * a1 + ol1 * b1;
#pragma unroll
    for (int dn = 0; dn < 8; ++dn) {
      o[dn][0] = o[dn][0] * a0 + ld(dn * 4 + 0) * b0;
      o[dn][1] = o[dn][1] * a0 + ld(dn * 4 + 1) * b0;
      o[dn][2] = o[dn][2] * a1 + ld(dn * 4 + 2) * b1;
      o[dn][3] = o[dn][3] * a1 + ld(dn * 4 + 3) * b1;
    }
  }
};

// Query fragments of the sequence's S rows from row0 on.  (Plain loads: neighbouring lanes share sectors, and loads past L1 made
// a launch 1-3 us slower.)
template <int MT, bool FP8>
__device__ __forceinline__ void load_queries(uint32_t (&qf)[MT][4][4], const __nv_bfloat16 *qbuf, int row0, int S, int d, int h, int g, int tig) {
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    int r_lo = mt * 16 + g, r_hi = r_lo + 8;
    if (FP8) {
      // f16 queries, dims 4 tig + {0, 1} | 4 tig + {2, 3} of every 16: the order the key codes come in
      const __nv_bfloat16 *q_lo = qbuf + (size_t)(row0 + r_lo) * d + h * kDh + 4 * tig;
      const __nv_bfloat16 *q_hi = qbuf + (size_t)(row0 + r_hi) * d + h * kDh + 4 * tig;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const uint2 lo = r_lo < S ? *reinterpret_cast<const uint2 *>(q_lo + kk * 16) : make_uint2(0u, 0u);
        const uint2 hi = r_hi < S ? *reinterpret_cast<const uint2 *>(q_hi + kk * 16) : make_uint2(0u, 0u);
        qf[mt][kk][0] = bf16x2_to_f16x2(lo.x); qf[mt][kk][2] = bf16x2_to_f16x2(lo.y);
        qf[mt][kk][1] = bf16x2_to_f16x2(hi.x); qf[mt][kk][3] = bf16x2_to_f16x2(hi.y);
      }
    } else {
      const __nv_bfloat16 *q_lo = qbuf + (size_t)(row0 + r_lo) * d + h * kDh + 2 * tig;
      const __nv_bfloat16 *q_hi = qbuf + (size_t)(row0 + r_hi) * d + h * kDh + 2 * tig;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        qf[mt][kk][0] = r_lo < S ? *reinterpret_cast<const uint32_t *>(q_lo + kk * 16) : 0u;
        qf[mt][kk][1] = r_hi < S ? *reinterpret_cast<const uint32_t *>(q_hi + kk * 16) : 0u;
        qf[mt][kk][2] = r_lo < S ? *reinterpret_cast<const uint32_t *>(q_lo + kk * 16 + 8) : 0u;
        qf[mt][kk][3] = r_hi < S ? *reinterpret_cast<const uint32_t *>(q_hi + kk * 16 + 8) : 0u;
      }
    }
  }
}

// One tile for one consumer warp: scores of its keys (the first one at context position key0, place kb of the tile), online softmax,
// O += P V.
template <int MT, bool FP8>
__device__ __forceinline__ void tile_step(TileAcc (&acc)[MT], const uint32_t (&qf)[MT][4][4], uint32_t kbase, uint32_t vbase, int key0, int kb,
                                          int ctx_len, float seg_sl2, int lane) {
  constexpr int KPW = XK / XCW, NTW = KPW / 8, KSW = KPW / 16;      // keys per warp and tile; 8-key score tiles, 16-key P.V steps
  const int tig = lane & 3;
  const bool ragged = key0 + KPW > ctx_len;
  // Rows at or beyond ctx_len hold whatever follows in memory.  Their weights are exactly 0 below;
  // the value fragments of those keys are cleared in registers after ldmatrix, so that 0 never
  // multiplies a non-finite.
  // ---- scores: S[mt][nt] = Q (16 x 64) . K^T (64 x 8 keys)
  float sc[MT][NTW][4];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int nt = 0; nt < NTW; ++nt) sc[mt][nt][0] = sc[mt][nt][1] = sc[mt][nt][2] = sc[mt][nt][3] = 0.f;
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt) {
    if (FP8) {
      // column c of score tile nt = 2 ks + u is key 16 ks + 4 (c >> 1) + 2 u + (c & 1) of this warp's 32: the
      // order in which the value codes of a 16-key step come out of ldmatrix (see the P.V loop).  The keys
      // of every group of 16 are STORED in that order (tile u's eight keys in lines 4 u .. 4 u + 3), so that
      // the eight rows of an ldmatrix fall into eight different 16-byte bank groups.
      const int key = kb + nt * 8 + (lane & 7);                                 // position in stored order
      const int line = key >> 1, chunk = ((key & 1) << 2) + (lane >> 3);       // two keys per 128-byte line
      uint32_t r[4];
      ldsm_x4(kbase + (uint32_t)(line * 128 + ((chunk ^ (line & 7)) << 4)), r[0], r[1], r[2], r[3]);   // all 64 dims of 8 keys
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t b0 = e4m3x2_to_f16x2(r[j], 0), b1 = e4m3x2_to_f16x2(r[j], 1);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) mma_f16(sc[mt][nt], qf[mt][j][0], qf[mt][j][1], qf[mt][j][2], qf[mt][j][3], b0, b1);
      }
    } else {
      const int key = kb + nt * 8 + (lane & 7);
#pragma unroll
      for (int kp = 0; kp < 2; ++kp) {      // two k16 steps per ldmatrix.x4
        uint32_t b0, b1, b2, b3;
        ldsm_x4(kbase + swz(key, kp * 4 + (lane >> 3)), b0, b1, b2, b3);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          mma_bf16(sc[mt][nt], qf[mt][2 * kp][0], qf[mt][2 * kp][1], qf[mt][2 * kp][2], qf[mt][2 * kp][3], b0, b1);
          mma_bf16(sc[mt][nt], qf[mt][2 * kp + 1][0], qf[mt][2 * kp + 1][1], qf[mt][2 * kp + 1][2],
                   qf[mt][2 * kp + 1][3], b2, b3);
        }
      }
    }
  }
  // ---- scale, mask the ragged end of the context, online softmax
  uint32_t pf[MT][KSW][4];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < NTW; ++nt) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float v = sc[mt][nt][e] * seg_sl2;
        const int kidx = FP8 ? key0 + 16 * (nt >> 1) + 4 * tig + 2 * (nt & 1) + (e & 1) : key0 + nt * 8 + 2 * tig + (e & 1);
        if (ragged && kidx >= ctx_len) v = -INFINITY;
        sc[mt][nt][e] = v;
      }
      mx0 = fmaxf(mx0, fmaxf(sc[mt][nt][0], sc[mt][nt][1]));
      mx1 = fmaxf(mx1, fmaxf(sc[mt][nt][2], sc[mt][nt][3]));
    }
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
    TileAcc &A = acc[mt];
    const float mn0 = fmaxf(A.m0, mx0), mn1 = fmaxf(A.m1, mx1);
    const float ref0 = mn0 == -INFINITY ? 0.f : mn0, ref1 = mn1 == -INFINITY ? 0.f : mn1;
    const float c0 = ex2f(A.m0 - ref0), c1 = ex2f(A.m1 - ref1);
    A.m0 = mn0; A.m1 = mn1;
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int nt = 0; nt < NTW; ++nt) {
      float p0 = ex2f(sc[mt][nt][0] - ref0), p1 = ex2f(sc[mt][nt][1] - ref0);
      float p2 = ex2f(sc[mt][nt][2] - ref1), p3 = ex2f(sc[mt][nt][3] - ref1);
      s0 += p0 + p1; s1 += p2 + p3;
      pf[mt][nt >> 1][(nt & 1) * 2 + 0] = FP8 ? pack_f16(p0, p1) : pack_bf16(p0, p1);
      pf[mt][nt >> 1][(nt & 1) * 2 + 1] = FP8 ? pack_f16(p2, p3) : pack_bf16(p2, p3);
    }
    A.l0 = A.l0 * c0 + s0;
    A.l1 = A.l1 * c1 + s1;
    if (__any_sync(0xffffffffu, c0 != 1.f || c1 != 1.f)) {   // some row's running maximum moved
#pragma unroll
      for (int dn = 0; dn < 8; ++dn) { A.o[dn][0] *= c0; A.o[dn][1] *= c0; A.o[dn][2] *= c1; A.o[dn][3] *= c1; }
    }
  }
  // ---- O += P (16 x 32 keys) . V (32 keys x 64)
  if (FP8) {
    // transposed values: a line is one dim, a 16-byte chunk sixteen keys; positions at or beyond ctx_len
    // hold zero codes (written so, or filled by the copy beyond max_ctx), so nothing needs masking
#pragma unroll
    for (int ks = 0; ks < KSW; ++ks) {
      const int chunk = (kb + ks * 16) >> 4;
#pragma unroll
      for (int dq = 0; dq < 2; ++dq) {      // four 8-wide slices of the head per ldmatrix.x4
        const int dim = (dq * 4 + (lane >> 3)) * 8 + (lane & 7);
        uint32_t r[4];
        ldsm_x4(vbase + (uint32_t)(dim * 128 + ((chunk ^ (dim & 7)) << 4)), r[0], r[1], r[2], r[3]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t b0 = e4m3x2_to_f16x2(r[j], 0), b1 = e4m3x2_to_f16x2(r[j], 1);
#pragma unroll
          for (int mt = 0; mt < MT; ++mt)
            mma_f16(acc[mt].o[dq * 4 + j], pf[mt][ks][0], pf[mt][ks][1], pf[mt][ks][2], pf[mt][ks][3], b0, b1);
        }
      }
    }
  } else {
#pragma unroll
  for (int ks = 0; ks < KSW; ++ks) {
    const int key = kb + ks * 16 + ((lane >> 3) & 1) * 8 + (lane & 7);
    // this lane's fragment halves hold keys k0, k0 + 1 (b0, b2) and k0 + 8, k0 + 9 (b1, b3)
    uint32_t keep_a = 0xffffffffu, keep_b = 0xffffffffu;
    if (ragged) {
      const int k0 = key0 + ks * 16 + 2 * tig;
      keep_a = (k0 < ctx_len ? 0x0000ffffu : 0u) | (k0 + 1 < ctx_len ? 0xffff0000u : 0u);
      keep_b = (k0 + 8 < ctx_len ? 0x0000ffffu : 0u) | (k0 + 9 < ctx_len ? 0xffff0000u : 0u);
    }
#pragma unroll
    for (int dp = 0; dp < 4; ++dp) {      // two 8-wide slices of the head per ldmatrix.x4
      uint32_t b0, b1, b2, b3;
      ldsm_x4_t(vbase + swz(key, dp * 2 + (lane >> 4)), b0, b1, b2, b3);
      if (ragged) { b0 &= keep_a; b1 &= keep_b; b2 &= keep_a; b3 &= keep_b; }
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        mma_bf16(acc[mt].o[2 * dp], pf[mt][ks][0], pf[mt][ks][1], pf[mt][ks][2], pf[mt][ks][3], b0, b1);
        mma_bf16(acc[mt].o[2 * dp + 1], pf[mt][ks][0], pf[mt][ks][1], pf[mt][ks][2], pf[mt][ks][3], b2, b3);
      }
    }
  }
  }
}

template <int MT>
__device__ __forceinline__ void store_rows(const TileAcc (&acc)[MT], __nv_bfloat16 *out, int row0, int S, int d, int h, float seg_vscale, int g, int tig) {
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    const TileAcc &A = acc[mt];
    const int r_lo = mt * 16 + g, r_hi = r_lo + 8;
    const float i0 = seg_vscale / A.l0, i1 = seg_vscale / A.l1;
    __nv_bfloat16 *o_lo = out + (size_t)(row0 + r_lo) * d + h * kDh + 2 * tig;
    __nv_bfloat16 *o_hi = out + (size_t)(row0 + r_hi) * d + h * kDh + 2 * tig;
#pragma unroll
    for (int dn = 0; dn < 8; ++dn) {
      if (r_lo < S) *reinterpret_cast<__nv_bfloat162 *>(o_lo + dn * 8) = __floats2bfloat162_rn(A.o[dn][0] * i0, A.o[dn][1] * i0);
      if (r_hi < S) *reinterpret_cast<__nv_bfloat162 *>(o_hi + dn * 8) = __floats2bfloat162_rn(A.o[dn][2] * i1, A.o[dn][3] * i1);
    }
  }
}

// MT = 16-row query tiles (rows per sequence <= 16 * MT); FP8 = keys/values are E4M3 codes (tmap: the keys'
// 128-byte lines, tmap_v: the transposed values), else bf16 (tmap alone: rows of 64 values)
template <int MT, bool FP8>
__global__ void __launch_bounds__(XTHREADS, xctas(MT, FP8)) cross_attn_tma_kernel(const __grid_constant__ CUtensorMap tmap,
                                                                                       const __grid_constant__ CUtensorMap tmap_v, AttnArgs a) {
  constexpr int KPW = XK / XCW;
  constexpr int XTILE_BYTES = XK * kDh * (FP8 ? 1 : 2), XSTAGE_BYTES = 2 * XTILE_BYTES, XSTAGES = xring_bytes(MT, FP8) / XSTAGE_BYTES;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int before_s[XCW];
  const Dims &dm = a.dm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tig = lane & 3;
  const int ns = gridDim.x, rank = blockIdx.x, h = blockIdx.y, b = blockIdx.z, H = dm.H;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t *smem_al = smem_raw + (base - smem_u32(smem_raw));
  float *scratch = reinterpret_cast<float *>(smem_al);        // half the consumer warps' records for the tree merge, over the ring
  const uint32_t bar_full = base + XSTAGES * XSTAGE_BYTES, bar_empty = bar_full + 8 * XSTAGES, bar_part = bar_empty + 8 * XSTAGES;
  const float *recv = reinterpret_cast<const float *>(smem_al);      // states of ranks 1 .. ns - 1, over the ring: [rank - 1][row tile][XREC_FLOATS]

  if (tid == 0) {
    for (int s = 0; s < XSTAGES; ++s) { mbar_init(bar_full + 8 * s, 1); mbar_init(bar_empty + 8 * s, XCW); }
    mbar_init(bar_part, (uint32_t)(ns > 1 ? ns - 1 : 1));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // (counts the caller of the stand-alone op wrote are clamped to the tensors' extents)
  const int S = min(max(a.st.n_active[b], 0), min(dm.C, 16 * MT)), ctx_len = min(max(a.st.ctx_len[b], 1), dm.ctx);
  int before = 0;                                       // packed rows: active rows of the sequences before this one
  if (a.packed && warp < XCW) {
    for (int bb = tid; bb < b; bb += XCW * 32) before += min(max(a.st.n_active[bb], 0), min(dm.C, 16 * MT));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    if (lane == 0) before_s[warp] = before;
  }
  __syncthreads();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int kv_b = a.kv_seq != nullptr ? a.kv_seq[b] : b;      // the sequence whose context this group reads
  int row0 = a.row_base != nullptr ? a.row_base[b] : b * dm.C;
  if (a.packed) {
    row0 = 0;
#pragma unroll
    for (int w = 0; w < XCW; ++w) row0 += before_s[w];
  }
  __nv_bfloat16 *out = (__nv_bfloat16 *)a.out;
  if (a.clear_status && rank == 0 && h == 0 && b == 0 && tid == 0) a.st.hdr[HDR_STATUS] = 0;      // stand-alone op: its scratch comes as it is; a wait can expire only long after this
  if (!a.packed && a.row_base == nullptr && rank == 0)  // rows of the sequence beyond its active ones come back as zeros
    for (int idx = tid; idx < (dm.C - S) * (kDh / 8); idx += XTHREADS)
      *reinterpret_cast<uint4 *>(out + (size_t)(row0 + S + idx / (kDh / 8)) * dm.d + h * kDh + (idx % (kDh / 8)) * 8) = make_uint4(0u, 0u, 0u, 0u);
  const int nt = S > 0 ? (ctx_len + XK - 1) / XK : 0;
  const int lo = nt * rank / ns, hi = nt * (rank + 1) / ns;

  bool ok = true;
  TileAcc acc[MT];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) acc[mt].clear();
  float seg_sl2 = dm.scale_log2e, seg_vscale = 1.f;     // 8-bit: the key scale joins the score scale, the value scale the final 1 / l
  if (FP8) {
    const float2 sc2 = *reinterpret_cast<const float2 *>(a.kv_scale + ((((size_t)a.layer * dm.B + kv_b) * H + h) << 1));
    seg_sl2 *= sc2.x; seg_vscale = sc2.y;
  }
  if (warp == XCW) {
    if (lane == 0) {                                    // producer: ahead of the dependency wait, the context is older than the kernel before
      for (int it = 0; it < hi - lo; ++it) {
        const int s = it % XSTAGES;
        if (!mbar_wait(bar_empty + 8 * s, (((uint32_t)(it / XSTAGES)) & 1u) ^ 1u)) { ok = false; break; }
        // The stage was read through the generic proxy and is filled through the async one.  Without this fence a copy overtook the last
        // ldmatrix of the slowest warp: a 32-byte sector of the values, one decode in a few where the launches before and after overlap
        // this one.  (In the consumer warps, ahead of their arrival, it holds as well, and costs them 36 cycles a tile.)
        if (it >= XSTAGES) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(bar_full + 8 * s, XSTAGE_BYTES);
        const uint32_t dst = base + s * XSTAGE_BYTES;
        if (FP8) {
          const int blk = (((a.layer * dm.B + kv_b) * H + h) << 1);    // block = max_ctx * 64 bytes of keys, then as many of transposed values
          tma_load_2d(dst, &tmap, bar_full + 8 * s, 0, blk * (dm.ctx >> 1) + (lo + it) * (XK / 2));    // 64 lines = 128 keys
          tma_load_3d(dst + XTILE_BYTES, &tmap_v, bar_full + 8 * s, (lo + it) * XK, 0, blk + 1);       // 64 dims x 128 keys
        } else {
          const int y = (int)(ctx_kv_offset(a.layer, dm.B, kv_b, H, h, 0, dm.ctx) / kDh) + (lo + it) * XK;
          tma_load_2d(dst, &tmap, bar_full + 8 * s, 0, y);                         // K tile
          tma_load_2d(dst + XTILE_BYTES, &tmap, bar_full + 8 * s, 0, y + dm.ctx);  // V tile
        }
      }
    }
    __syncwarp();
    x_dependency_wait();
  } else {
    x_dependency_wait();
    if (hi > lo) {
      uint32_t qf[MT][4][4];
      load_queries<MT, FP8>(qf, (const __nv_bfloat16 *)a.q, row0, S, dm.d, h, g, tig);
      const int kb = warp * KPW;
      for (int it = 0; it < hi - lo; ++it) {
        const int s = it % XSTAGES;
        if (ok && !mbar_wait(bar_full + 8 * s, ((uint32_t)(it / XSTAGES)) & 1u)) ok = false;
        if (!ok) break;
        const uint32_t kbase = base + s * XSTAGE_BYTES;
        tile_step<MT, FP8>(acc, qf, kbase, kbase + XTILE_BYTES, (lo + it) * XK + kb, kb, ctx_len, seg_sl2, lane);
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_empty + 8 * s);
      }
    }
    consumer_bar_sync<XCW * 32>();                      // the last tile is consumed: the ring is free
    // row sums across the quad, the warps' states into warp 0's
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
      TileAcc &A = acc[mt];
      A.l0 += __shfl_xor_sync(0xffffffffu, A.l0, 1); A.l0 += __shfl_xor_sync(0xffffffffu, A.l0, 2);
      A.l1 += __shfl_xor_sync(0xffffffffu, A.l1, 1); A.l1 += __shfl_xor_sync(0xffffffffu, A.l1, 2);
#pragma unroll
      for (int stride = XCW / 2; stride >= 1; stride >>= 1) {
        if (warp >= stride && warp < 2 * stride) A.store(scratch + (warp - stride) * XREC_FLOATS, lane);
        consumer_bar_sync<XCW * 32>();
        if (warp < stride) A.merge(scratch + warp * XREC_FLOATS, lane);
        consumer_bar_sync<XCW * 32>();
      }
    }
  }
  __syncwarp();
  if (ns > 1) {                                         // every tile of the segment is consumed: the first CTA's ring is free
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  if (warp == 0 && S > 0) {
    if (rank > 0) {
      uint32_t dst;
      asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst) : "r"(base + (uint32_t)((rank - 1) * MT * XREC_FLOATS + lane) * 4u));
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        const TileAcc &A = acc[mt];
        auto put = [&](int w, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + (uint32_t)(mt * XREC_FLOATS + w * 32) * 4u), "f"(v) : "memory"); };
#pragma unroll
        for (int dn = 0; dn < 8; ++dn)
#pragma unroll
          for (int x = 0; x < 4; ++x) put(dn * 4 + x, A.o[dn][x]);
        put(32, A.m0); put(33, A.m1); put(34, A.l0); put(35, A.l1);
      }
      __syncwarp();
      if (lane == 0) {
        uint32_t bar;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(bar) : "r"(bar_part));
        asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
      }
    } else {
      if (ns > 1) {
        bool got = false;
        for (uint32_t it = 0; it < XSPIN_LIMIT && !got; ++it) {
          uint32_t done;
          asm volatile(
              "{\n\t.reg .pred p;\n\t"
              "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
              "selp.u32 %0, 1, 0, p;\n\t}"
              : "=r"(done)
              : "r"(bar_part)
              : "memory");
          got = done != 0;
        }
        ok = ok && got;
        for (int r = 1; r < ns && ok; ++r)              // rank order: the result does not depend on arrival order
#pragma unroll
          for (int mt = 0; mt < MT; ++mt) acc[mt].merge(recv + ((r - 1) * MT + mt) * XREC_FLOATS, lane);
      }
      store_rows<MT>(acc, out, row0, S, dm.d, h, seg_vscale, g, tig);
    }
  }
  if (!ok && lane == 0) atomicExch(&a.st.hdr[HDR_STATUS], (int)PD_ERR_TIMEOUT);
}

// Tensor map of the context keys/values seen as a 2-D bf16 array [rows, 64] (row = one context
// position of one (layer, sequence, head, K or V)): boxes of 128 rows x 64 columns (one head's
// keys or values of one tile, 16 KB contiguous), 128-byte swizzle.  *driver_code gets the CUresult
// when the encode itself fails.
cudaError_t encode_ctx_kv_tensor_map(CUtensorMap *out, const void *base, uint64_t rows, int *driver_code) {
  const uint64_t gdim[2] = {kDh, rows}, gstride[1] = {kDh * 2};
  const uint32_t box[2] = {kDh, XK};
  return encode_tensor_map(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, gdim, gstride, box, driver_code);
}

// Tensor maps of the 8-bit context keys/values, n_blocks = layers * sequences * heads blocks of
// max_ctx * 64 bytes of keys followed by max_ctx * 64 bytes of transposed values.  Keys: the whole buffer
// as lines of 128 bytes (two keys each), boxes of 64 lines; values: [block][64 dims][max_ctx], boxes of
// 128 keys x 64 dims.  Both with the 128-byte swizzle; reads beyond max_ctx are filled with zeros.
cudaError_t encode_ctx_kv8_tensor_maps(CUtensorMap *map_k, CUtensorMap *map_v, const void *base, uint64_t n_blocks, uint64_t ctx,
                                       int *driver_code) {
  const uint64_t kdim[2] = {128, n_blocks * 2 * ctx * kDh / 128}, kstride[1] = {128};
  const uint32_t kbox[2] = {128, XK / 2};
  cudaError_t e = encode_tensor_map(map_k, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, base, kdim, kstride, kbox, driver_code);
  if (e != cudaSuccess) return e;
  const uint64_t vdim[3] = {ctx, kDh, n_blocks * 2}, vstride[2] = {ctx, ctx * kDh};
  const uint32_t vbox[3] = {XK, kDh, 1u};
  return encode_tensor_map(map_v, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, base, vdim, vstride, vbox, driver_code);
}

// CTAs per segment: the power of two that gives at most one CTA per SM, as long as every CTA has a tile.  (48 segments of 777
// keys: 2 -> 8.3, 3 -> 10.0, 4 -> 8.6, 6 -> 12.4 us - clusters of other sizes leave SMs of a GPC over; 120 segments of 1024 keys:
// 1 -> 11.4, 2 -> 12.3; 192 of 1000: 1 -> 13.9, 2 -> 18.6; 24 of 1024: 2 -> 7.0, 4 -> 6.2, 8 -> 8.2.)
static int cross_cluster_size(const AttnArgs &a) {
  const long long segs = (long long)a.batch * a.dm.H;
  const int tiles = (a.dm.ctx + XK - 1) / XK;
  int ns = 1;
  while (ns < 8 && 2 * ns <= tiles && 2 * ns * segs <= kSms) ns *= 2;
  return ns;
}
static_assert(7 * XREC_FLOATS * 4 <= xring_bytes(1, true) && 7 * 2 * XREC_FLOATS * 4 <= xring_bytes(2, true), "the states of a cluster fit over the ring");

// 8-bit launches begin under the kernel before from this many segments on, and with no more places on an SM than the launch needs if it is spread
// evenly: their CTAs are small, and pile up, four on each of the SMs that the kernel before has left already.  Decodes of four layers, segments x
// keys, ms: begun behind the kernel before / under it, piled up / under it, spread:
//   8 x 96   4.10 / 4.32 / 4.43       16 x 4096  6.53 / 7.31 / 7.35     32 x 4096  6.89 / 7.66 / 6.76      48 x 784   6.68 / 7.12 / 6.52
//   64 x 96  4.84 / 4.84 / 4.70       128 x 4096 10.89 / 14.25 / 10.59  144 x 2048 9.33 / 10.80 / 9.00     192 x 1024 9.87 / 10.32 / 9.52
//   256 x 2048 12.58 / 13.39 / 12.15  384 x 2048 14.34 / 14.80 / 14.00  512 x 2048 16.31 / 15.84 / 15.81   768 x 1024 (another path) alike
// Dynamic shared memory of such a launch of `ctas` CTAs:
constexpr long long kX8EarlySegs = 48;
constexpr int kSmSmem = 228 * 1024, kCtaSmem = 1024;      // shared memory of an SM; what a CTA takes beside its own
static int x8_smem(int mt, long long ctas) {
  const int places = (int)((ctas + kSms - 1) / kSms);
  const int one_more = kSmSmem / (places + 1) - kCtaSmem + 16;      // places + 1 CTAs of this size do not fit
  return places < xctas(mt, true) && one_more > xsmem(mt, true) ? one_more : xsmem(mt, true);
}

// rows_per_seq, fp8: the variant to prepare
cudaError_t cross_attn_tma_prepare(int rows_per_seq, bool fp8) {
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if (rows_per_seq <= 16)
    return fp8 ? cudaFuncSetAttribute(cross_attn_tma_kernel<1, true>, attr, x8_smem(1, 1)) : cudaFuncSetAttribute(cross_attn_tma_kernel<1, false>, attr, xsmem(1, false));
  return fp8 ? cudaFuncSetAttribute(cross_attn_tma_kernel<2, true>, attr, x8_smem(2, 1)) : cudaFuncSetAttribute(cross_attn_tma_kernel<2, false>, attr, xsmem(2, false));
}

// 8-bit keys/values (a.kv_scale set): tmap = the keys' lines, tmap_v = the transposed values; else tmap alone.
// a.pdl: launched as a programmatic dependent of the query projection before it, which writes none of the keys,
// values, row counts and context lengths, so the first tiles travel while that kernel runs (8-bit: not with few segments).
cudaError_t launch_cross_attn_tma(const AttnArgs &a, const CUtensorMap &tmap, const CUtensorMap &tmap_v, cudaStream_t s) {
  const int mt = (a.dm.C + 15) / 16;
  const bool fp8 = a.kv_scale != nullptr;
  if (mt < 1 || mt > 2 || a.batch > 65535) return cudaErrorInvalidValue;
  const int ns = cross_cluster_size(a);
  const bool early = a.pdl && (!fp8 || (long long)a.batch * a.dm.H >= kX8EarlySegs);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ns, a.dm.H, a.batch);
  cfg.blockDim = dim3(XTHREADS, 1, 1);
  cfg.dynamicSmemBytes = fp8 && early ? x8_smem(mt, (long long)ns * a.dm.H * a.batch) : xsmem(mt, fp8);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ns; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = early ? 2 : 1;
  if (mt == 1) return fp8 ? cudaLaunchKernelEx(&cfg, cross_attn_tma_kernel<1, true>, tmap, tmap_v, a) : cudaLaunchKernelEx(&cfg, cross_attn_tma_kernel<1, false>, tmap, tmap_v, a);
  return fp8 ? cudaLaunchKernelEx(&cfg, cross_attn_tma_kernel<2, true>, tmap, tmap_v, a) : cudaLaunchKernelEx(&cfg, cross_attn_tma_kernel<2, false>, tmap, tmap_v, a);
}

}  // namespace pd
