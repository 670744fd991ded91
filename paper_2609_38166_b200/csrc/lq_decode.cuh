// Decode: one token for one (sequence, value head), done by a CTA of two warps with different roles.
//
// Eq. 10 (readout of the smoothed, compensated window representation) evaluated for x = alpha.k and
// x = alpha.q in one pass over the 8-bit codes:
//   S_{l-1}^T (alpha.x) = (B/127) Z^T (C Gamma_{1:l} x) + Uc (Kc^T Gamma_{1:l} x) + sum_j u_j (kt_j^T Gamma_{j+1:l} x)
// then u = v - S_{l-1}^T(alpha.k) (Eq. 3), o = S_{l-1}^T(alpha.q) + u (kt^T q), and the record is appended.
//
// Data movement: a head's block (16 KiB of codes, the two scale vectors, the compensators: 19 KiB) and
// its n buffered record rows are each contiguous in memory and are brought into the CTA's shared-memory slot
// by TWO TMA bulk copies, each completing on its own mbarrier: a few large bulk requests keep the memory
// system busy where thousands of 16-byte loads could not (plain loads are limited per warp), and about 64 KB
// in flight per SM saturate HBM.  The slot is small enough for six CTAs per SM.  CTAs are persistent and walk
// over the heads with a grid stride.  No load sits on a head's critical path (with the memory system kept
// full a load takes microseconds to return): the token's vectors are loaded into registers one head ahead,
// the per-head scalars (window position, beta, scalar alpha) for 32 heads at a time, one per lane; whatever
// needs only the token (the scalar-gate decay chain, kt^T q) is computed before the wait for the slot.
//
// Roles: the STREAM warp turns C Gamma x into fixed-point digits, runs the tensor-core pass over the codes,
// adds the compensator terms, requests the next head's block as soon as nobody needs this one's any more,
// adds the record terms and finishes u and o; the DOT warp meanwhile projects onto the compensators, walks
// the buffered records (projections and the records' terms of the readout in one pass), requests the next
// head's records, appends the new record and makes the window-position arrival.  They meet at named barriers
// (three per head, four with the diagonal gate, whose decays both warps read from the records).
//
// Arithmetic: the first term is a dense int8 contraction, Z^T [128 x 128] against the two vectors.  The
// vectors are put on a 30-bit block fixed-point grid and split into four signed base-256 digits each, which
// gives an int8 operand of 128 x 8; the tensor cores (mma.sync m16n8k32, s8 x s8 -> s32) produce exact
// integer sums, recombined in 64-bit integers and rounded to fp32 once, so the result does not depend on
// the order of accumulation.  The codes are stored value-channel major (Z^T, [d_v][d_k]): the contraction
// index is then contiguous, as the MMA operand layout needs.  The small dot products against records and
// compensators run on the fp32 pipes in the library's fixed summation order.
#pragma once
#include <type_traits>

#include "lq_common.cuh"

namespace lq {

// Long windows: the records come in segments of this many rows, newest first, two of which the slot holds at a time: while
// one is walked the next is on its way (a multiple of four: the walk takes eight or four records at a time from the newest back).
// Rows of 1 to 1.5 KB (fp32) and of half that (fp16); diagonal gate, W = 64, us per step at 256 x 32 heads: fp32 8 rows 132,
// 4: 148, 12: 149, 16: 146; fp16 12 rows 125, 8: 130, 16: 123 (with records walked four at a time; eight at a time, 116 and 114).
__host__ __device__ constexpr int rec_seg(bool rec16) { return rec16 ? 12 : 8; }

// ---- shared-memory slot of one CTA ----
struct DecodeSlot {
  // byte offsets inside the slot; every region starts on a 16-byte boundary
  int head, rec, bas, digits, y, pj, pk, pq, mbar, bytes;
  __host__ __device__ DecodeSlot(int W, int r, bool diag, bool rec16, bool bf16, int seg) {
    // a window holds at most W-1 records when a token arrives; seg > 0: two segments of that many at a time
    const int rows = seg > 0 ? 2 * seg : W > 1 ? W - 1 : 1;
    int o = 0;
    head = o; o += bf16 ? BF16W_HEAD_BYTES : head_bytes(r);   // codes | col_scale | row_smooth | comp_k | comp_u, or S0^T
    rec = o; o += (rec16 ? 2 : 4) * record_floats(diag) * rows;   // buffered record rows (fp32 or fp16)
    bas = o; o += diag ? 0 : 2 * 4 * MAX_W;         // scalar gate: the records' decays, one copy per warp
    digits = o; o += 8 * D;               // digit planes: plane 4v+d = digit d of vector v (0: k, 1: q); bf16: record terms
    y = o; o += 2 * 4 * D;                // [2][128]: the rounded sums of the state stream, later the record terms
    pj = o; o += 4 * 16;                  // [2][8]: projections of a group of records, on their way to all lanes of the dot warp
    pk = o; o += (4 * (r + 2) + 15) / 16 * 16;      // compensator projections against Gamma k
    pq = o; o += (4 * (r + 2) + 15) / 16 * 16;      // ... against Gamma q; pq[r], pq[r+1] hold kt^T q of alternate heads with a token
    mbar = o; o += 32;                    // head block, records (two)
    bytes = (o + 127) / 128 * 128;
  }
};

// D(16x8, s32) += A(16x32, s8, row-major) * B(32x8, s8, column-major)
__device__ __forceinline__ void mma_s8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                       uint32_t b1) {
  asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Block fixed point of a 128-vector whose largest magnitude is xmax: scale = 2^(29-e), back = 2^(e-29) with
// 2^e <= xmax < 2^(e+1); both zero when xmax < 2^-96 (the vector then counts as zero).
__device__ __forceinline__ void fixed_point_scales(float xmax, float &scale, float &back) {
  if (!(xmax >= 0x1p-96f)) { scale = 0.0f; back = 0.0f; return; }
  const int e = static_cast<int>((__float_as_uint(xmax) >> 23) & 0xFF) - 127;
  scale = __uint_as_float(static_cast<uint32_t>(29 - e + 127) << 23);
  back = __uint_as_float(static_cast<uint32_t>(e - 29 + 127) << 23);
}

__device__ __forceinline__ void widen8_bf16(const uint4 w, float (&x)[8]) {
  const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int e = 0; e < 4; e++) {
    x[2 * e] = __uint_as_float(ws[e] << 16);
    x[2 * e + 1] = __uint_as_float(ws[e] & 0xFFFF0000u);
  }
}
// the same as four (even, odd) pairs
__device__ __forceinline__ void widen8_bf16(const uint4 w, float2 (&x)[4]) {
  const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int e = 0; e < 4; e++) x[e] = make_float2(__uint_as_float(ws[e] << 16), __uint_as_float(ws[e] & 0xFFFF0000u));
}
__device__ __forceinline__ void widen8_f16(const uint4 w, float (&x)[8]) {
  const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int e = 0; e < 4; e++) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&ws[e]));
    x[2 * e] = f.x;
    x[2 * e + 1] = f.y;
  }
}

// sums of four values over sixteen neighbouring lanes each, the four shuffle chains interleaved
__device__ __forceinline__ void tree16x4(float (&x)[4]) {
#pragma unroll
  for (int s = 1; s <= 8; s <<= 1) {
#pragma unroll
    for (int v = 0; v < 4; v++) x[v] = x[v] + __shfl_xor_sync(FULL, x[v], s);
  }
}

// Columns j0 .. j0 + 63 of the products of a bfloat16 state (S0T: [d_v][d_k] in shared memory) with two vectors, into
// y[0][.] and y[1][.]; lane c (and its twin c + 16) holds block c of the vectors.  Eight columns at a time per half-warp: the
// sixteen sums are taken over the sixteen lanes by halving exchanges (15 shuffles instead of 64), neighbouring blocks first.
__device__ __forceinline__ void bf16_columns(const uint16_t *S0T, int j0, const float2 (&xk)[4], const float2 (&xq)[4], float *y, int lane) {
  const int c = lane & 15, half = lane >> 4;
  const bool u0 = lane & 1, u1 = lane & 2, u2 = lane & 4, u3 = lane & 8;
#pragma unroll 1
  for (int j = j0 + 8 * half; j < j0 + 64; j += 16) {
    float vk[8], vq[8], x8[8], x4[4], x2[2];
#pragma unroll
    for (int m = 0; m < 8; m++) {
      float2 s2[4];
      widen8_bf16(*reinterpret_cast<const uint4 *>(S0T + (j + m) * D + 8 * c), s2);
      vk[m] = block8(s2, xk);
      vq[m] = block8(s2, xq);
    }
#pragma unroll
    for (int e = 0; e < 8; e++) x8[e] = (u0 ? vq[e] : vk[e]) + __shfl_xor_sync(FULL, u0 ? vk[e] : vq[e], 1);
#pragma unroll
    for (int e = 0; e < 4; e++) x4[e] = (u1 ? x8[e + 4] : x8[e]) + __shfl_xor_sync(FULL, u1 ? x8[e] : x8[e + 4], 2);
#pragma unroll
    for (int e = 0; e < 2; e++) x2[e] = (u2 ? x4[e + 2] : x4[e]) + __shfl_xor_sync(FULL, u2 ? x4[e] : x4[e + 2], 4);
    const float x = (u3 ? x2[1] : x2[0]) + __shfl_xor_sync(FULL, u3 ? x2[0] : x2[1], 8);
    y[(u0 ? D : 0) + j + (u1 ? 4 : 0) + (u2 ? 2 : 0) + (u3 ? 1 : 0)] = x;
  }
}

// Compensator keys against Gamma_{1:l} k and Gamma_{1:l} q, by one warp: the projections go to pk[h], pq[h].  A dot product of 128
// terms is taken by sixteen lanes (lane c owns block c of eight terms); the two halves of the warp work on different vectors, two
// per half and trip, so that four shuffle trees overlap.  Both halves make the same number of trips (the shuffles name all 32
// lanes); an index outside the range recomputes a valid item and is not stored.
__device__ __forceinline__ void project_compensators(const uint16_t *ckh, int r, const float2 (&gam)[4], const float2 (&k2)[4],
                                                     const float2 (&q2)[4], float *pk, float *pq, int lane) {
  const int c = lane & 15, half = lane >> 4;
  float2 gk2[4], gq2[4];
#pragma unroll
  for (int cc = 0; cc < 4; cc++) { gk2[cc] = __fmul2_rn(gam[cc], k2[cc]); gq2[cc] = __fmul2_rn(gam[cc], q2[cc]); }
#pragma unroll 1
  for (int hb = 0; hb < r; hb += 4) {
    float s4[4];
    int ho[2];
#pragma unroll
    for (int u = 0; u < 2; u++) {
      ho[u] = hb + 2 * u + half;
      const int h = ho[u] < r ? ho[u] : r - 1;
      float x8[8];
      widen8_f16(*reinterpret_cast<const uint4 *>(ckh + h * D + 8 * c), x8);
      float2 x2[4];
#pragma unroll
      for (int cc = 0; cc < 4; cc++) x2[cc] = make_float2(x8[2 * cc], x8[2 * cc + 1]);
      s4[2 * u] = block8(x2, gk2);
      s4[2 * u + 1] = block8(x2, gq2);
    }
    tree16x4(s4);
#pragma unroll
    for (int u = 0; u < 2; u++)
      if (c == 0 && ho[u] < r) { pk[ho[u]] = s4[2 * u]; pq[ho[u]] = s4[2 * u + 1]; }
  }
}

// 2 NP records jt, jt-1, ...: half 0 projects the first, third, ... of them, half 1 the others.  The sums over the sixteen
// lanes are taken by halving exchanges (eight values: 4 + 2 + 1 + 1 shuffles), after which a lane holds one of them;
// through pj every lane gets all.  A group of four may run past record `base`; what lies below is computed from that record and
// dropped.  `seg`: the rows at hand, beginning with record `base`; bas: the records' decays (scalar gate); g2 or (scalar gate) g1:
// Gamma_{jt+1:l}, kept up (and past record `base` exactly at the end).  With one number in place of the scalar gate's vector the walk
// takes about 30 instructions less for a pair of records: with the waits not unrolled (mbar_wait) 1024 x 32 heads, W = 32, 259 -> 252 us a step.
template <int GATE, int NP, typename rec_t>
__device__ __forceinline__ void walk_group(const rec_t *seg, const int base, const float *bas, float *pj, const int jt, const int lane,
                                           const float2 (&k2)[4], const float2 (&q2)[4], float2 (&g2)[4], float &g1,
                                           float2 (&rk_rec)[2], float2 (&rq_rec)[2]) {
  constexpr bool DIAG = GATE == LQ_GATE_DIAG, MASKED = NP == 2;
  constexpr int RF = record_floats(DIAG);
  const int c = lane & 15, half = lane >> 4;
  float v[2 * NP];
#pragma unroll
  for (int u = 0; u < NP; u++) {
    // the decays of the two records of this pair; the half that owns the older one steps over the newer
    const int jn = jt - 2 * u, jold = jn - 1;  // newer, older
    const int in = MASKED ? max(jn, base) : jn, iold = MASKED ? max(jold, base) : jold;
    float2 gmine[4];
    // past both records, as far as they are there (selects: a branch for the last trip of a long head was slower)
    if constexpr (DIAG) {
      float2 an[4], ao[4];
      load8p(seg + (in - base) * RF + REC_A + 8 * c, an);
      load8p(seg + (iold - base) * RF + REC_A + 8 * c, ao);
#pragma unroll
      for (int cc = 0; cc < 4; cc++) {
        const float2 gn = g2[cc], go = __fmul2_rn(gn, an[cc]);   // Gamma_{jn+1:l}, Gamma_{jold+1:l}
        gmine[cc] = half ? go : gn;
        g2[cc] = !MASKED || jold >= base ? __fmul2_rn(go, ao[cc]) : jn >= base ? go : gn;
      }
    } else {
      const float gn = g1, go = gn * bas[in], past = go * bas[iold];
      g1 = !MASKED || jold >= base ? past : jn >= base ? go : gn;
#pragma unroll
      for (int cc = 0; cc < 4; cc++) gmine[cc] = pair(half ? go : gn);
    }
    const int j = half ? iold : in;
    float2 x2[4], yk2[4], yq2[4];
    load8p(seg + (j - base) * RF + REC_KT + 8 * c, x2);
#pragma unroll
    for (int cc = 0; cc < 4; cc++) { yk2[cc] = __fmul2_rn(gmine[cc], k2[cc]); yq2[cc] = __fmul2_rn(gmine[cc], q2[cc]); }
    v[2 * u] = block8(x2, yk2);
    v[2 * u + 1] = block8(x2, yq2);
  }
  // halving exchanges over lane bits 0, 1, (2), then plain ones; lane c ends with value `mine` of its half
  const bool u0 = lane & 1, u1 = lane & 2, u2 = lane & 4;
  float x;
  int mine;
  if constexpr (NP == 4) {
    float x4[4], x2_[2];
#pragma unroll
    for (int e = 0; e < 4; e++) x4[e] = (u0 ? v[e + 4] : v[e]) + __shfl_xor_sync(FULL, u0 ? v[e] : v[e + 4], 1);
#pragma unroll
    for (int e = 0; e < 2; e++) x2_[e] = (u1 ? x4[e + 2] : x4[e]) + __shfl_xor_sync(FULL, u1 ? x4[e] : x4[e + 2], 2);
    x = (u2 ? x2_[1] : x2_[0]) + __shfl_xor_sync(FULL, u2 ? x2_[0] : x2_[1], 4);
    mine = (u0 ? 4 : 0) + (u1 ? 2 : 0) + (u2 ? 1 : 0);
  } else {
    float x2_[2];
#pragma unroll
    for (int e = 0; e < 2; e++) x2_[e] = (u0 ? v[e + 2] : v[e]) + __shfl_xor_sync(FULL, u0 ? v[e] : v[e + 2], 1);
    x = (u1 ? x2_[1] : x2_[0]) + __shfl_xor_sync(FULL, u1 ? x2_[0] : x2_[1], 2);
    x = x + __shfl_xor_sync(FULL, x, 4);
    mine = (u0 ? 2 : 0) + (u1 ? 1 : 0);
  }
  x = x + __shfl_xor_sync(FULL, x, 8);
  __syncwarp();                                // (the group before has been read)
  if (c < 2 * NP) pj[(mine & 1) * 8 + (mine & ~1) + half] = x;     // pj[vector][record]
  __syncwarp();
  float pk_[2 * NP], pq_[2 * NP];
#pragma unroll
  for (int e = 0; e < NP / 2; e++) {
    const float4 a = *reinterpret_cast<const float4 *>(pj + 4 * e), b = *reinterpret_cast<const float4 *>(pj + 8 + 4 * e);
    pk_[4 * e] = a.x; pk_[4 * e + 1] = a.y; pk_[4 * e + 2] = a.z; pk_[4 * e + 3] = a.w;
    pq_[4 * e] = b.x; pq_[4 * e + 1] = b.y; pq_[4 * e + 2] = b.z; pq_[4 * e + 3] = b.w;
  }
#pragma unroll
  for (int e = 0; e < 2 * NP; e++) {
    const int j = jt - e;
    if (MASKED && j < base) break;             // the same for every lane
    const float4 u4 = load4(seg + (j - base) * RF + REC_U + 4 * lane);
    const float2 lo = make_float2(u4.x, u4.y), hi = make_float2(u4.z, u4.w), pk2 = pair(pk_[e]), pq2 = pair(pq_[e]);
    rk_rec[0] = __ffma2_rn(lo, pk2, rk_rec[0]); rq_rec[0] = __ffma2_rn(lo, pq2, rq_rec[0]);
    rk_rec[1] = __ffma2_rn(hi, pk2, rk_rec[1]); rq_rec[1] = __ffma2_rn(hi, pq2, rq_rec[1]);
  }
}
// The records from jt back to `base`: eight at a time while they last, then four.
template <int GATE, typename rec_t>
__device__ __forceinline__ void walk_records(const rec_t *seg, const int base, const float *bas, float *pj, int jt, const int lane,
                                             const float2 (&k2)[4], const float2 (&q2)[4], float2 (&g2)[4], float &g1,
                                             float2 (&rk_rec)[2], float2 (&rq_rec)[2]) {
#pragma unroll 1
  for (; jt - 7 >= base; jt -= 8) walk_group<GATE, 4>(seg, base, bas, pj, jt, lane, k2, q2, g2, g1, rk_rec, rq_rec);
#pragma unroll 1
  for (; jt >= base; jt -= 4) walk_group<GATE, 2>(seg, base, bas, pj, jt, lane, k2, q2, g2, g1, rk_rec, rq_rec);
}

// C Gamma k (lanes 0..15) and C Gamma q (lanes 16..31) on their fixed-point grids, as digit planes; back_*: what a unit of the
// grids is worth
__device__ __forceinline__ void digit_planes(const float *cs, const float (&gam)[8], const float (&k8)[8], const float (&q8)[8],
                                             int8_t *digits, int lane, float &back_k, float &back_q) {
  const int c = lane & 15, half = lane >> 4;
  float back_own;
  {
    float c8[8], x8[8];
    load8(cs + 8 * c, c8);
    float m = 0.0f;
#pragma unroll
    for (int e = 0; e < 8; e++) {
      x8[e] = c8[e] * (gam[e] * (half ? q8[e] : k8[e]));
      m = fmaxf(m, fabsf(x8[e]));
    }
#pragma unroll
    for (int s = 1; s <= 8; s <<= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, s));
    float scale;
    fixed_point_scales(m, scale, back_own);
    // X = d0 + 256 d1 + 65536 d2 + 2^24 d3 with digits in [-128, 127]: the digit is the low byte read as
    // signed, and taking it off is (X + 128) >> 8.  The bytes of the four stages of an element are the
    // four digits; prmt gathers the same digit of four elements into one word.
    uint32_t st[8][4];
#pragma unroll
    for (int e = 0; e < 8; e++) {
      int X = __float2int_rn(x8[e] * scale);
#pragma unroll
      for (int d = 0; d < 4; d++) { st[e][d] = static_cast<uint32_t>(X); X = (X + 128) >> 8; }
    }
#pragma unroll
    for (int d = 0; d < 4; d++) {
      const uint32_t lo = __byte_perm(__byte_perm(st[0][d], st[1][d], 0x0040), __byte_perm(st[2][d], st[3][d], 0x0040), 0x5410);
      const uint32_t hi = __byte_perm(__byte_perm(st[4][d], st[5][d], 0x0040), __byte_perm(st[6][d], st[7][d], 0x0040), 0x5410);
      *reinterpret_cast<uint2 *>(digits + (4 * half + d) * D + 8 * c) = make_uint2(lo, hi);
    }
  }
  const float back_other = __shfl_xor_sync(FULL, back_own, 16);
  back_k = half ? back_other : back_own;
  back_q = half ? back_own : back_other;
}

// The state stream on the tensor cores: eight 16-row tiles of Z^T, K = 128 as four k-blocks.  A
// thread's 16 bytes of a row hold key channels 64p+16t..64p+16t+15 and serve two k-blocks; the digit
// planes are read with the same permutation of the key index.  The two 64-channel halves of a tile
// accumulate separately (exact integers: any split gives the same sum), which halves the dependent
// chain of MMAs.  Digit pairs are recombined in int32 (|sum| < 2^30), the two pairs in int64 (the total has
// 47 bits), and one rounding takes it to fp32.
// GROUPS: the tiles are taken in so many groups (registers); y may lie where the digits are.
template <int GROUPS>
__device__ __forceinline__ void code_sums(const int8_t *zt, const int8_t *digits, float *y, int lane) {
  const int g = lane >> 2, t = lane & 3;
  constexpr int h0 = 0, h1 = 64;         // the two 64-channel halves (the same split for every lane)
  const uint4 bfa = *reinterpret_cast<const uint4 *>(digits + g * D + h0 + 16 * t);
  const uint4 bfb = *reinterpret_cast<const uint4 *>(digits + g * D + h1 + 16 * t);
  constexpr int TILES = 8 / GROUPS;
#pragma unroll 1
  for (int mg = 0; mg < 8; mg += TILES) {
    int pair_lo[TILES], pair_hi[TILES];  // digit-pair sums of rows g and g+8 of each tile
#pragma unroll
    for (int mt = 0; mt < TILES; mt++) {
      int ca[4] = {0, 0, 0, 0}, cb[4] = {0, 0, 0, 0};
      const int j = 16 * (mg + mt) + g;
      const uint4 alo = *reinterpret_cast<const uint4 *>(zt + j * D + h0 + 16 * t);
      const uint4 ahi = *reinterpret_cast<const uint4 *>(zt + (j + 8) * D + h0 + 16 * t);
      const uint4 blo = *reinterpret_cast<const uint4 *>(zt + j * D + h1 + 16 * t);
      const uint4 bhi = *reinterpret_cast<const uint4 *>(zt + (j + 8) * D + h1 + 16 * t);
      mma_s8(ca, alo.x, ahi.x, alo.y, ahi.y, bfa.x, bfa.y);
      mma_s8(cb, blo.x, bhi.x, blo.y, bhi.y, bfb.x, bfb.y);
      mma_s8(ca, alo.z, ahi.z, alo.w, ahi.w, bfa.z, bfa.w);
      mma_s8(cb, blo.z, bhi.z, blo.w, bhi.w, bfb.z, bfb.w);
      // c[0], c[1]: row g, planes 2t, 2t+1;  c[2], c[3]: row g+8.  Planes 4v..4v+3 are the digits of
      // vector v: lanes t = 0, 1 carry the k sums and t = 2, 3 the q sums, even t the low digit pair.
      pair_lo[mt] = (ca[0] + cb[0]) + ((ca[1] + cb[1]) << 8);
      pair_hi[mt] = (ca[2] + cb[2]) + ((ca[3] + cb[3]) << 8);
    }
    int oth_lo[TILES], oth_hi[TILES];
#pragma unroll
    for (int mt = 0; mt < TILES; mt++) {
      oth_lo[mt] = __shfl_xor_sync(FULL, pair_lo[mt], 1);
      oth_hi[mt] = __shfl_xor_sync(FULL, pair_hi[mt], 1);
    }
    if (!(t & 1)) {                      // this lane has the low pairs, its neighbour sent the high pairs
      float *dst = y + (t >> 1) * D + g + 16 * mg;
#pragma unroll
      for (int mt = 0; mt < TILES; mt++) {
        dst[16 * mt] = __ll2float_rn(static_cast<long long>(oth_lo[mt]) * 65536 + pair_lo[mt]);
        dst[16 * mt + 8] = __ll2float_rn(static_cast<long long>(oth_hi[mt]) * 65536 + pair_hi[mt]);
      }
    }
  }
}

// Named barriers of the CTA (64 threads each): one side arrives, the other waits.
//   1: dot warp -> stream warp, "the record terms (and the ticket) are in shared memory"
//   2: stream warp -> dot warp, "its sums are out of y"
//   3: dot warp -> stream warp, "the compensator projections are in shared memory"
//   4, 5: stream warp -> dot warp, "the records' decays have been read" (diagonal gate; one for each half of the record area:
//      with two segments there the stream warp may be through with both before the dot warp is with the first)
__device__ __forceinline__ void named_arrive(int id) {
  __threadfence_block();
  asm volatile("bar.arrive %0, 64;\n" ::"r"(id) : "memory");
}
__device__ __forceinline__ void named_wait(int id) { asm volatile("bar.sync %0, 64;\n" ::"r"(id) : "memory"); }

// The token's vectors as raw bf16 bits, loaded one head ahead: lane c (and its twin c+16) owns key
// channels 8c..8c+7, lane l value channels 4l..4l+3.
struct TokenRaw {
  uint4 k, q, a;        // a: diagonal-gate alpha
  uint2 v;
  float ba_lo, ba_hi;   // scalar gate: decays of buffered records `lane` and `lane + 32` (stale beyond n)
  uint16_t beta, alpha; // (SCALARS: the head's scalars come with its vectors)
};

// A head index with its sequence and value-head parts, stepped without divisions.
struct HeadIdx {
  unsigned bh, b, hv;
  __device__ __forceinline__ void step(unsigned dbh, unsigned db, unsigned dhv, unsigned heads_v) {
    bh += dbh; b += db; hv += dhv;
    if (hv >= heads_v) { hv -= heads_v; b += 1; }
  }
};

template <int GATE, bool SCALARS = false>
__device__ __forceinline__ void load_token(const Params &p, const HeadIdx h, int group, int lane, int role, TokenRaw &tk) {
  const int c = lane & 15;
  const size_t bh = h.bh;
  const size_t qk_off = ((size_t)h.b * p.heads_qk + h.hv / group) * D;
  tk.k = *reinterpret_cast<const uint4 *>(p.k + qk_off + 8 * c);
  tk.q = *reinterpret_cast<const uint4 *>(p.q + qk_off + 8 * c);
  if (role == 0) tk.v = *reinterpret_cast<const uint2 *>(p.v + bh * D + 4 * lane);
  if (SCALARS && role == 1) tk.beta = p.beta[bh];
  if (SCALARS && GATE == LQ_GATE_SCALAR) tk.alpha = p.alpha[bh];
  if (GATE == LQ_GATE_DIAG) {
    tk.a = *reinterpret_cast<const uint4 *>(p.alpha + bh * D + 8 * c);
  } else {
    if (lane < p.W) tk.ba_lo = p.decays[bh * (size_t)p.W + lane];
    if (lane + 32 < p.W) tk.ba_hi = p.decays[bh * (size_t)p.W + lane + 32];
  }
}

// The work of one pair of warps (role 0: stream warp, role 1: dot warp) on its shared-memory slot: heads
// first, first + G, first + 2G, ...
// LONGW: the records come in segments (launch_decode_t says when); in the other instances everything to do with a second
// segment drops out at compile time.
// BF16: the per-window BF16 state (lq_shape.state_bf16): the head block is S0^T in bfloat16, its product with Gamma x is
// taken in binary32 by both warps, half of the columns each; there are no scales and no compensators.
// ONCE: one head and no more, and the caller makes the window-position arrival.
template <int GATE, bool R16, bool LONGW, bool BF16, bool ONCE = false>
__device__ __forceinline__ void decode_slot(const Params &p, unsigned char *slot, const int lane, const int role,
                                            const unsigned first, const unsigned G) {
  uint32_t parA = 0, parR = 0;               // phase of the head block's copy barrier; bit b: of the records' barrier b
  int buf = 0;                               // (long windows) the half of the record area that the next segment to be walked is in
  constexpr bool DIAG = GATE == LQ_GATE_DIAG;
  constexpr int RF = record_floats(DIAG);
  const int W = p.W, r = p.r;
  using rec_t = typename std::conditional<R16, __half, float>::type;   // element type of the record rows
  constexpr int SEG = LONGW ? rec_seg(R16) : 0;
  const DecodeSlot L(W, r, DIAG, R16, BF16, SEG);
  const uint32_t block_bytes = BF16 ? BF16W_HEAD_BYTES : head_bytes(r);
  const int c = lane & 15, half = lane >> 4;
  const int8_t *zt = reinterpret_cast<const int8_t *>(slot + L.head + HB_CODES);
  const float *bs = reinterpret_cast<const float *>(slot + L.head + HB_COL_SCALE);
  const float *cs = reinterpret_cast<const float *>(slot + L.head + HB_ROW_SMOOTH);
  const uint16_t *ckh = reinterpret_cast<const uint16_t *>(slot + L.head + HB_COMP_K);
  const uint16_t *cuh = reinterpret_cast<const uint16_t *>(slot + L.head + hb_comp_u(r));
  const rec_t *rec = reinterpret_cast<const rec_t *>(slot + L.rec);     // rows of RF elements: kt | u | (alpha)
  float *bas = reinterpret_cast<float *>(slot + L.bas) + role * MAX_W;   // this warp's copy of the decays
  int8_t *digits = reinterpret_cast<int8_t *>(slot + L.digits);
  float *y = reinterpret_cast<float *>(slot + L.y), *pk = reinterpret_cast<float *>(slot + L.pk);
  float *pq = reinterpret_cast<float *>(slot + L.pq), *pj = reinterpret_cast<float *>(slot + L.pj);
  const uint32_t barA = smem_addr(slot + L.mbar), barR = barA + 8, slot_a = smem_addr(slot);   // head block, records

  const unsigned nh = static_cast<unsigned>(p.batch) * p.heads_v, Hv = p.heads_v;
  const unsigned G_b = G / Hv, G_hv = G % Hv;       // one grid stride in (sequence, head) steps
  const int group = p.heads_v / p.heads_qk;

#ifdef LQ_TIMING
  long long tick_ = clock64();
  unsigned acc_[12] = {0};
#endif
  // The slot is filled by two bulk copies with a barrier each, because its two parts become free at different
  // times.  The head block (codes, scales, compensators) of the next head is requested by the stream warp as soon
  // as both warps have taken the last thing they need from it (the compensator rows), the records by the dot
  // warp as soon as it has walked them: about half of a head's work later the wait for the next head starts, and
  // by then the copies have been on their way for a while.
  // The regions the copies overwrite were only READ through ordinary loads, whose values have been used
  // before the call; the warps write only their scratch regions.  So nothing written by the generic proxy is
  // at stake and no cross-proxy fence is needed (it costs over a thousand cycles here).
  // A head at its last free record (n == W - 1) goes through the window boundary right after this kernel, which
  // reads the same head block and records again: its lines are asked to stay in the L2 until then.
  const uint64_t keep = l2_keep_policy(), stream = l2_stream_policy();
  auto request_head = [&](unsigned bh, int n) {
    if (lane == 0) {
      const uint8_t *block = p.heads + bh * (size_t)block_bytes;
      mbar_expect_tx(barA, block_bytes);
      if (n == W - 1) bulk_g2s_hint(slot_a + L.head, block, block_bytes, barA, keep);
      else bulk_g2s_hint(slot_a + L.head, block, block_bytes, barA, stream);
    }
  };
  // first record of the segment that ends before record `hi`
  auto seg_base = [&](int hi) { return (LONGW && hi > SEG) ? hi - SEG : 0; };
  // records [seg_base(hi), hi) of head bh, n of which are buffered in all, into half `to` of the record area
  auto request_segment = [&](unsigned bh, int n, int hi, int to) {
    if (lane == 0) {
      const int lo = seg_base(hi);
      const uint32_t rb = static_cast<uint32_t>(sizeof(rec_t)) * RF * (hi - lo), bar_to = barR + 8 * to;
      const uint32_t dst = slot_a + L.rec + to * static_cast<uint32_t>(sizeof(rec_t)) * RF * SEG;
      mbar_expect_tx(bar_to, rb);            // with no records the phase completes at once
      if (hi > lo) {
        if (n == W - 1) bulk_g2s_hint(dst, p.record<rec_t>(bh, lo, DIAG), rb, bar_to, keep);
        else bulk_g2s_hint(dst, p.record<rec_t>(bh, lo, DIAG), rb, bar_to, stream);
      }
    }
  };
  // the newest records of a head: with long windows the two newest segments
  auto request_records = [&](unsigned bh, int n) {
    request_segment(bh, n, n, buf);
    if (LONGW && n > SEG) request_segment(bh, n, n - SEG, buf ^ 1);
  };
  // Bounded wait for one of the two.  A copy that never lands must not hang the GPU: when the limit runs out the
  // error flag is set and the warp goes on (its results are garbage, the flag says so); the other warp, which
  // meets this one at the named barriers, is not left waiting.
  auto wait_for = [&](uint32_t bar_, uint32_t &par) {
    if (!mbar_wait(bar_, par) && lane == 0) atomicOr(&g_device_error, 1);
    par ^= 1u;
    __syncwarp();
  };
  auto wait_records = [&]() {                // the segment in half `buf`
    if (!mbar_wait(barR + 8 * buf, (parR >> buf) & 1u) && lane == 0) atomicOr(&g_device_error, 1);
    parR ^= 1u << buf;
    __syncwarp();
  };

  // Equal shares do not take equal time: pairs that share an SM with fewer others, or sit nearer the memory they
  // read, are through with ten heads when others have done eight.  With scratch words in the state (lq_state.work)
  // every pair therefore takes only its first S heads in turn (DRAWN_ROUNDS rounds fewer than would fall to it), and
  // the heads that are left (S G + t, t < pool) go to whoever gets there first: from its last turn but one on, the dot
  // warp draws a ticket t in every trip, for the head two trips on (word 0 of the scratch words counts the tickets;
  // the boundary kernel behind this one puts it back to zero), hands it to the stream warp with the record terms
  // (barrier 1), and at the end of the trip both warps ask for that head's scalars, which they look at for the first
  // time half a trip later (ext_*) and move to the lane registers of the other heads' at the end of the next trip.
  // A pair stops when a ticket is beyond the pool.
  const int rounds_all = ONCE ? 1 : static_cast<int>(nh / G);  // rounds in which every pair has a head
  const int DRAWN_ROUNDS = rounds_all >= 6 ? 2 : 1;            // (with few rounds, more of them in turn)
  const bool draw = !ONCE && p.work != nullptr && rounds_all >= 3;
  const int S = draw ? rounds_all - DRAWN_ROUNDS : 0;
  const unsigned pool = draw ? nh - static_cast<unsigned>(S) * G : 0;
  // Per-head scalars of this CTA's heads, 32 heads at a time: lane l holds those of the CTA's (32*batch+l)-th head
  int sc_n = 0;
  uint32_t sc_beta = 0, sc_alpha = 0;
  auto load_scalars = [&](unsigned first_bh) {
    const unsigned bh = first_bh + lane * G;  // (once per 32 heads: a division is fine here)
    if (bh < (draw ? static_cast<unsigned>(S) * G : nh)) {     // (the heads taken in turn)
      sc_n = p.win_pos[bh / Hv];             // bits 16.. are the arrival counter of this launch: masked at use
      sc_beta = p.beta[bh];
      if (!DIAG) sc_alpha = p.alpha[bh];
    }
  };

  // Arrival on win_pos (see arrive_and_set): the counter says how many heads of the sequence have READ the old
  // value, which this head did when its scalars were loaded.  The dot warp makes the arrival, at the end of its
  // work: it has slack, the stream warp (the longer of the two) has none to sit out the atomic's round trip.
  // A head whose window is already full (n >= W) gets no token: it is neither requested nor waited for.
  auto wanted = [&](int n_) { return n_ < W; };
  load_scalars(first);
  TokenRaw nxt;                               // the token of the head about to start
  nxt.ba_lo = nxt.ba_hi = 1.0f;
  HeadIdx hd{first, first / Hv, first % Hv};  // this head and the next one
  HeadIdx hd1 = hd;
  hd1.step(G, G_b, G_hv, Hv);
  {
    const int n0 = __shfl_sync(FULL, sc_n, 0) & 0xFFFF;
    if (first < nh && wanted(n0)) {
      load_token<GATE>(p, hd, group, lane, role, nxt);
      if (role == 0) request_head(first, n0);
      else request_records(first, n0);
    }
  }
#ifdef LQ_TIMING
  tick_ = clock64();
#endif
  unsigned *qidx = reinterpret_cast<unsigned *>(pk + r);      // (a spare word of the projection area)
  unsigned ticket = 0xFFFFFFFFu;             // (dot warp, lane 0) what was drawn in this trip
  bool drawing = draw;                       // no ticket has been beyond the pool yet
  int ext_n = 0;                             // scalars of the head drawn a trip ago, on their way
  uint32_t ext_beta = 0, ext_alpha = 0;
  int idx = 0;                               // position of the head in this slot's list
  int odd = 0;                               // parity of the heads with a token so far
  // end of a trip
  auto finish_trip = [&]() {
    // the next head, if it was drawn: its scalars, asked for a trip ago, go where the others' are
    if (draw && idx + 1 >= S && lane == ((idx + 1) & 31)) { sc_n = ext_n; sc_beta = ext_beta; sc_alpha = ext_alpha; }
    unsigned extra = nh;                     // the head after the next one, if it is a drawn one
    if (drawing && idx + 2 >= S) {
      const unsigned tk = role == 1 ? __shfl_sync(FULL, ticket, 0) : *reinterpret_cast<volatile unsigned *>(qidx);
      if (tk < pool) {
        extra = static_cast<unsigned>(S) * G + tk;
        ext_n = p.win_pos[extra / Hv];
        ext_beta = p.beta[extra];
        if (!DIAG) ext_alpha = p.alpha[extra];
      } else {
        drawing = false;
      }
    }
    hd = hd1;
    idx++;
    if (!draw || idx + 1 < S) {
      hd1.step(G, G_b, G_hv, Hv);
    } else if (extra < nh) {
      const unsigned b_ = extra / Hv;
      hd1 = HeadIdx{extra, b_, extra - b_ * Hv};
    } else {
      hd1 = HeadIdx{nh, 0u, 0u};
    }
  };
  for (; hd.bh < nh; finish_trip()) {
    const bool draws = drawing && idx + 2 >= S;                 // a ticket is drawn in this trip
    if (p.overlap && role == 1 && !draws && hd1.bh >= nh) grid_dependents_may_start();
    if (draws && role == 1 && lane == 0) ticket = static_cast<unsigned>(atomicAdd(p.work, 1));
    const size_t bh = hd.bh;
    const int n = __shfl_sync(FULL, sc_n, idx & 31) & 0xFFFF;
    const float beta = __uint_as_float(__shfl_sync(FULL, sc_beta, idx & 31) << 16);
    const float alpha_s = __uint_as_float(__shfl_sync(FULL, sc_alpha, idx & 31) << 16);
    // the next head's scalars: from the next batch when this head is the last of its batch
    const unsigned bh_next = hd1.bh;
    if ((idx & 31) == 31) load_scalars(bh_next);
    // The next head's window position.  Of a drawn head it is still on its way (ext_n, asked for at the end of the
    // trip before): it is looked at only where the head's data is requested, half a trip from here; until then the
    // head counts as one that gets a token (its token is loaded, which does no harm if it gets none).
    const bool next_drawn = draw && idx + 1 >= S;
    const int n_next_turn = bh_next < nh ? (__shfl_sync(FULL, sc_n, (idx + 1) & 31) & 0xFFFF) : W;
    auto n_next_now = [&]() { return next_drawn ? (bh_next < nh ? (ext_n & 0xFFFF) : W) : n_next_turn; };
    const bool next_token = next_drawn ? bh_next < nh : wanted(n_next_turn);
    const bool active = wanted(n);
    const int b = static_cast<int>(hd.b);
    LQ_TICK(0);

    if (!active) {                           // nothing was requested for this head; keep the pipeline going
      const int n_next = n_next_now();
      if (wanted(n_next)) {
        load_token<GATE>(p, hd1, group, lane, role, nxt);
        if (role == 0) request_head(bh_next, n_next);
        else request_records(bh_next, n_next);
      }
      // The ticket changes hands outside the usual place.  As in a trip with a token, barrier 2 (the stream warp is through
      // with the trip before) comes ahead of barrier 1: without it the dot warp could arrive at barrier 1 in two such trips
      // before the stream warp came there once, which would complete the barrier without it and leave it waiting for good.
      if (draws) {
        if (role == 1) {
          named_wait(2);
          if (lane == 0) *qidx = ticket;
          __syncwarp();
          named_arrive(1);
        } else {
          named_arrive(2);
          named_wait(1);
        }
      }
      continue;
    }

    // ---- this head's token (loaded while the previous head was being worked on); once it is unpacked
    // the registers are free for the next head's, whose load is then issued ----
    float k8[8], q8[8], a8[8];
    widen8_bf16(nxt.k, k8);
    widen8_bf16(nxt.q, q8);
    const uint2 v_raw = nxt.v;
    if (DIAG) {
      widen8_bf16(nxt.a, a8);
    } else {
#pragma unroll
      for (int e = 0; e < 8; e++) a8[e] = alpha_s;
      bas[lane] = nxt.ba_lo;
      bas[lane + 32] = nxt.ba_hi;
    }
    if (next_token) load_token<GATE>(p, hd1, group, lane, role, nxt);        // used one trip from now
    // scalar gate: Gamma_{1:l}, the chain of decays from the newest record back (Appendix B.2), needs nothing
    // from the slot, so the stream warp takes it before it waits
    float gsc = alpha_s;
    if (!DIAG) {
      __syncwarp();
#pragma unroll 4
      for (int j = role == 0 ? n - 1 : -1; j >= 0; j--) gsc = gsc * bas[j];
    }
    // kt^T q needs only the token: the dot warp takes it before the wait as well.  It goes to one of two places
    // in turn, because the stream warp may still be reading the previous head's.  In turn over the heads WITH a token: the
    // barriers of the head in between are what keeps a word from being written before the head two back has read it, and a
    // head whose window came in full meets at none.
    const int ktq_at = r + odd;
    odd ^= 1;
    if (role == 1) {
      float2 k2p[4], q2p[4];
#pragma unroll
      for (int cc = 0; cc < 4; cc++) {
        k2p[cc] = __fmul2_rn(pair(beta), make_float2(k8[2 * cc], k8[2 * cc + 1]));
        q2p[cc] = make_float2(q8[2 * cc], q8[2 * cc + 1]);
      }
      const float ktq_pre = tree16(block8(k2p, q2p));
      if (lane == 0) pq[ktq_at] = ktq_pre;
    }
    LQ_TICK(1);

    // ---- the stream warp waits for the head block; the dot warp first takes the records, which it asked for
    // earlier and which need nothing from the head block, and waits for the block when it gets to the compensators ----
    if (role == 0 && !DIAG) wait_for(barA, parA);  // (diagonal gate: after its own walk of the records' decays)
    LQ_TICK(2);
    if (idx == 0) LQ_STAMP(0, 2);

    if (role == 1) {
      // =========================== DOT WARP ===========================
      // Records are walked from the newest back, with g8 = Gamma_{j+1:l} kept up on the way (Appendix B.2).
      float2 k2[4], q2[4], a2[4], g2[4], kt2[4];
#pragma unroll
      for (int cc = 0; cc < 4; cc++) {
        k2[cc] = make_float2(k8[2 * cc], k8[2 * cc + 1]);
        q2[cc] = make_float2(q8[2 * cc], q8[2 * cc + 1]);
        a2[cc] = make_float2(a8[2 * cc], a8[2 * cc + 1]);
        g2[cc] = a2[cc];
        kt2[cc] = __fmul2_rn(pair(beta), k2[cc]);
      }
      wait_records();                        // the newest segment of the records
      // The record terms sum_j u_j (kt_j^T Gamma k) and the same for q, channels 4 lane .. 4 lane + 3, as one chain from the
      // newest record back.
      float2 rk_rec[2] = {{0.0f, 0.0f}, {0.0f, 0.0f}}, rq_rec[2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
      int n_left = n, base = seg_base(n);            // the segment at hand begins with record `base`, its newest is n_left - 1
      float g1 = alpha_s;
      const rec_t *seg = rec + buf * SEG * RF;       // and lies here
      for (;;) {
        walk_records<GATE>(seg, base, bas, pj, n_left - 1, lane, k2, q2, g2, g1, rk_rec, rq_rec);
        if (!LONGW || base == 0) break;
        // the segment is walked: on to the one before it
        __syncwarp();
        if (DIAG) named_wait(4 + buf);               // (the stream warp has taken this segment's decays as well)
        if (base > SEG) request_segment(bh, n, base - SEG, buf);        // (the one after that is on its way to the other half)
        n_left = base;
        base = seg_base(base);
        buf ^= 1;
        seg = rec + buf * SEG * RF;
        wait_records();
      }
      if (!DIAG) gsc = g1;                           // (the walk has come past record 0)
      const int walked = 4 + buf;                    // the barrier of the last segment
      if (LONGW) buf ^= 1;                           // the next head's segments follow on in turn
      LQ_TICK(3);
      if constexpr (BF16) {                  // this warp's half of the columns; then all goes to the stream warp
        if (DIAG) named_wait(walked);        // (the stream warp has read the records' decays too)
        else __syncwarp();                   // (every lane has read its last row)
        {
          const int n_next = n_next_now();
          if (wanted(n_next)) request_records(bh_next, n_next);
        }
        float2 xk[4], xq[4];
#pragma unroll
        for (int cc = 0; cc < 4; cc++) {
          const float2 gm = DIAG ? g2[cc] : pair(gsc);
          xk[cc] = __fmul2_rn(gm, k2[cc]);
          xq[cc] = __fmul2_rn(gm, q2[cc]);
        }
        named_wait(2);                       // the stream warp has taken the head before out of y and the terms
        wait_for(barA, parA);
        bf16_columns(reinterpret_cast<const uint16_t *>(zt), 64, xk, xq, y, lane);
        float *terms = reinterpret_cast<float *>(digits);
        *reinterpret_cast<float4 *>(terms + 4 * lane) = make_float4(rk_rec[0].x, rk_rec[0].y, rk_rec[1].x, rk_rec[1].y);
        *reinterpret_cast<float4 *>(terms + D + 4 * lane) = make_float4(rq_rec[0].x, rq_rec[0].y, rq_rec[1].x, rq_rec[1].y);
        if (draws && lane == 0) *qidx = ticket;
        __syncwarp();
        named_arrive(1);                     // (this warp is done with the head block as well)
      } else {
      // Now the head block: the compensators are projected with Gamma_{1:l}, which for the diagonal gate is where
      // the walk's chain of decays has arrived (g2), for the scalar gate the product taken before the wait.
      wait_for(barA, parA);
      if (r > 0) {
        if (DIAG) {
          project_compensators(ckh, r, g2, k2, q2, pk, pq, lane);
        } else {
          float2 gam[4];
#pragma unroll
          for (int cc = 0; cc < 4; cc++) gam[cc] = pair(gsc);
          project_compensators(ckh, r, gam, k2, q2, pk, pq, lane);
        }
      }
      __syncwarp();
      named_arrive(3);                       // the compensator projections are in pk, pq; this warp is done with the head block
      LQ_TICK(4);
      if (DIAG) named_wait(walked);          // diagonal gate: the stream warp read the records' decays too
      {
        const int n_next = n_next_now();
        if (wanted(n_next)) request_records(bh_next, n_next);
      }
      named_wait(2);                         // the stream warp has taken its sums out of y
      *reinterpret_cast<float4 *>(y + 4 * lane) = make_float4(rk_rec[0].x, rk_rec[0].y, rk_rec[1].x, rk_rec[1].y);
      *reinterpret_cast<float4 *>(y + D + 4 * lane) = make_float4(rq_rec[0].x, rq_rec[0].y, rq_rec[1].x, rq_rec[1].y);
      if (draws && lane == 0) *qidx = ticket;
      __syncwarp();
      named_arrive(1);                       // the record terms are in shared memory (and the ticket)
      }
      LQ_TICK(5);
      // append the key side of the record (and its decay)
      {
        rec_t *row = p.record<rec_t>(bh, n, DIAG);
        if (half == 0) {
          store8p(row + REC_KT + 8 * c, kt2);
          if (DIAG) store8(row + REC_A + 8 * c, a8);
          else if (lane == 0) p.decays[bh * (size_t)W + n] = a8[0];
        }
      }
      if (!ONCE && lane == 0) arrive_and_set(p.win_pos, b, p.heads_v, n + 1);
      LQ_TICK(7);
    } else {
      // =========================== STREAM WARP ===========================
      // Gamma_{1:l}: the chain of decays from the newest record back (Appendix B.2)
      float gam[8];
#pragma unroll
      for (int e = 0; e < 8; e++) gam[e] = a8[e];
      if (DIAG) {
        for (int hi = n;;) {                        // segment after segment, in step with the dot warp
          const int lo = seg_base(hi);
          const rec_t *seg = rec + buf * SEG * RF;
          wait_records();
#pragma unroll 2
          for (int j = hi - 1; j >= lo; j--) {
            float aj[8];
            load8(seg + (j - lo) * RF + REC_A + 8 * c, aj);
#pragma unroll
            for (int e = 0; e < 8; e++) gam[e] = gam[e] * aj[e];
          }
          __syncwarp();
          named_arrive(4 + buf);             // this warp is done with the segment
          if (LONGW) buf ^= 1;
          if (lo == 0) break;
          hi = lo;
        }
        wait_for(barA, parA);
      } else {
#pragma unroll
        for (int e = 0; e < 8; e++) gam[e] = gsc;
      }
      LQ_TICK(3);
      float rk[4], rq[4];
      const float v4[4] = {__uint_as_float(v_raw.x << 16), __uint_as_float(v_raw.x & 0xFFFF0000u),
                           __uint_as_float(v_raw.y << 16), __uint_as_float(v_raw.y & 0xFFFF0000u)};
      if constexpr (BF16) {
        float2 xk[4], xq[4];
#pragma unroll
        for (int cc = 0; cc < 4; cc++) {
          const float2 gm = make_float2(gam[2 * cc], gam[2 * cc + 1]);
          xk[cc] = __fmul2_rn(gm, make_float2(k8[2 * cc], k8[2 * cc + 1]));
          xq[cc] = __fmul2_rn(gm, make_float2(q8[2 * cc], q8[2 * cc + 1]));
        }
        named_arrive(2);                     // the head before is out of y and the terms
        bf16_columns(reinterpret_cast<const uint16_t *>(zt), 0, xk, xq, y, lane);
        __syncwarp();
        named_wait(1);                       // the other half of the columns and the record terms
        {
          const int n_next = n_next_now();
          if (wanted(n_next)) request_head(bh_next, n_next);
        }
        const float *terms = reinterpret_cast<const float *>(digits);
        const float4 yk = *reinterpret_cast<const float4 *>(y + 4 * lane), yq = *reinterpret_cast<const float4 *>(y + D + 4 * lane);
        const float4 tk = *reinterpret_cast<const float4 *>(terms + 4 * lane), tq = *reinterpret_cast<const float4 *>(terms + D + 4 * lane);
        rk[0] = yk.x + tk.x; rk[1] = yk.y + tk.y; rk[2] = yk.z + tk.z; rk[3] = yk.w + tk.w;
        rq[0] = yq.x + tq.x; rq[1] = yq.y + tq.y; rq[2] = yq.z + tq.z; rq[3] = yq.w + tq.w;
      } else {
      float back_k, back_q;
      digit_planes(cs, gam, k8, q8, digits, lane, back_k, back_q);
      __syncwarp();                          // the digit planes are visible to the warp
      LQ_TICK(4);

      code_sums<1>(zt, digits, y, lane);
      __syncwarp();
      LQ_TICK(5);

      // Per value channel (lane l: channels 4l..4l+3): scale the sums, then add the compensator and record
      // terms with the projections of the dot warp
      {
        const float4 yk4 = *reinterpret_cast<const float4 *>(y + 4 * lane);
        const float4 yq4 = *reinterpret_cast<const float4 *>(y + D + 4 * lane);
        const float4 s4 = *reinterpret_cast<const float4 *>(bs + 4 * lane);      // code steps B_j / 127
        rk[0] = s4.x * (yk4.x * back_k); rk[1] = s4.y * (yk4.y * back_k); rk[2] = s4.z * (yk4.z * back_k); rk[3] = s4.w * (yk4.w * back_k);
        rq[0] = s4.x * (yq4.x * back_q); rq[1] = s4.y * (yq4.y * back_q); rq[2] = s4.z * (yq4.z * back_q); rq[3] = s4.w * (yq4.w * back_q);
        LQ_TICK(6);
        named_arrive(2);                     // y has been read: the dot warp may put the record terms there
        named_wait(3);                       // the compensator projections are complete
        LQ_TICK(7);
#pragma unroll 2
        for (int h = 0; h < r; h++) {
          const uint2 w = *reinterpret_cast<const uint2 *>(cuh + h * D + 4 * lane);
          const float2 f01 = __half22float2(*reinterpret_cast<const __half2 *>(&w.x));
          const float2 f23 = __half22float2(*reinterpret_cast<const __half2 *>(&w.y));
          const float uc[4] = {f01.x, f01.y, f23.x, f23.y};
          const float pkh = pk[h], pqh = pq[h];
#pragma unroll
          for (int e = 0; e < 4; e++) { rk[e] = fmaf(uc[e], pkh, rk[e]); rq[e] = fmaf(uc[e], pqh, rq[e]); }
        }
        __syncwarp();                        // nobody reads the head block any more (the dot warp finished with
        {
          const int n_next = n_next_now();
          if (wanted(n_next)) request_head(bh_next, n_next);   // it before barrier 3): the next head's may land
        }
        named_wait(1);                       // the record terms are complete
        {
          const float4 tk = *reinterpret_cast<const float4 *>(y + 4 * lane);
          const float4 tq = *reinterpret_cast<const float4 *>(y + D + 4 * lane);
          rk[0] = rk[0] + tk.x; rk[1] = rk[1] + tk.y; rk[2] = rk[2] + tk.z; rk[3] = rk[3] + tk.w;
          rq[0] = rq[0] + tq.x; rq[1] = rq[1] + tq.y; rq[2] = rq[2] + tq.z; rq[3] = rq[3] + tq.w;
        }
      }
      }
      {
        const float ktq = pq[ktq_at];
        float u[4], o[4];
#pragma unroll
        for (int e = 0; e < 4; e++) { u[e] = p.delta ? v4[e] - rk[e] : v4[e]; o[e] = fmaf(u[e], ktq, rq[e]); }
        LQ_TICK(8);
        *reinterpret_cast<float4 *>(p.o + bh * D + 4 * lane) = make_float4(o[0], o[1], o[2], o[3]);
        store4(p.record<rec_t>(bh, n, DIAG) + REC_U + 4 * lane, u[0], u[1], u[2], u[3]);
      }
      LQ_TICK(9);
    }
  }
#ifdef LQ_TIMING
  if (lane == 0)
    for (int i = 0; i < 12; i++) atomicAdd(&g_phase_cycles[16 * role + i], (unsigned long long)acc_[i]);
#endif
}

// Persistent kernel of two-warp CTAs: CTA `blockIdx.x` takes heads blockIdx.x, blockIdx.x + gridDim.x, ...
template <int GATE, bool R16, bool LONGW, bool BF16>
__global__ void __launch_bounds__(64, 6) decode_kernel(const Params p) {
  extern __shared__ __align__(128) unsigned char lq_slot[];
  LQ_STAMP(0, 0);
  // Resident while the kernel ahead drains: the CTA asks the L2 for its first head block meanwhile (a prefetch returns
  // no data, so it does not matter that the kernel ahead may still be writing that block: the L2 is where its writes
  // go).  The first head of a CTA is the only one whose copy nothing hides.
  if (threadIdx.x == 0 && blockIdx.x < static_cast<unsigned>(p.batch) * p.heads_v)
    bulk_prefetch_l2(p.heads + blockIdx.x * (size_t)(BF16 ? BF16W_HEAD_BYTES : head_bytes(p.r)), BF16 ? BF16W_HEAD_BYTES : head_bytes(p.r));
  const int lane = threadIdx.x & 31, role = threadIdx.x >> 5;
  if (threadIdx.x == 0) {                    // the slot's two copy barriers (shared memory only)
    const uint32_t bar = smem_addr(lq_slot + DecodeSlot(p.W, p.r, GATE == LQ_GATE_DIAG, R16, BF16, LONGW ? rec_seg(R16) : 0).mbar);
    mbar_init(bar, 1);
    mbar_init(bar + 8, 1);
    if (LONGW) mbar_init(bar + 16, 1);
  }
  __syncthreads();
  grid_dependency_wait();                    // no data in global memory is read or written above this line
  LQ_STAMP(0, 1);
  decode_slot<GATE, R16, LONGW, BF16>(p, lq_slot, lane, role, blockIdx.x, gridDim.x);
  LQ_STAMP(0, 3);
#ifdef LQ_TIMING
  if (threadIdx.x == 0 && blockIdx.x < 1024) {
    unsigned smid_;
    asm volatile("mov.u32 %0, %smid;" : "=r"(smid_));
    g_timeline[p.gen & 3][0][4][blockIdx.x] = smid_;
  }
  if (threadIdx.x == 32 && blockIdx.x < 1024) {          // the dot warp's last instruction
    unsigned long long t_;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t_));
    g_timeline[p.gen & 3][0][5][blockIdx.x] = t_;
  }
#endif
}

}  // namespace lq
