// The window boundary of a head: rebuild the dense state from the window representation (Eq. 7), refit the Compensator
// Tokens by power iteration on all r vectors at once (Eqs. 5-6), smooth the residual (Sec. 3.4), requantize it to 8 bits
// per value channel (Appendix B.3) and write the head back.
//
// Layout.  Eight warps hold the 128x128 state in registers: a warp owns 16 columns (value channels) of all 128 rows, lane
// (ty, tx) = (lane >> 1, lane & 1) the 8x8 tile of rows 8 ty .. 8 ty + 7 and eight of the columns, kept as column pairs
// (two FMAs per instruction).  So everything that belongs to a column - the products with the keys, the value sides, the
// scales, the codes - stays inside a warp, and only row sums (the products with the start vectors, the smoothing scales)
// go through shared memory and a barrier.  Two CTAs fill the register file of an SM.
//
// What bounds it: a flush (W = 16, r = 4) takes 23 K cycles with two CTAs on the SM (27 K before two records and two start
// vectors were in flight at a time); 9 K of them are the fp32 pipes (about 1150 packed FMAs per warp, two cycles each, four
// warps to a scheduler), the rest the waits between its dependent phases, of which only the other CTA fills some.  Issue slots
// are 48 % busy.  Against tiles of 8 rows x 128 columns per half-warp, where every column sum crossed the CTA (13 barriers a
// head, now 8), and copies by all threads into two staging buffers: 2048 dense states quantized in 55.2 us (91.4 before),
// 2048 states dequantized in 45.6 us (54.0); a step of 256 x 32 heads, 512 of them due, 73 -> 61 us.
//
// With NW = 4 four warps hold the state, 32 columns each and 16 to a lane (launch_boundary_t says where).
#pragma once
#include <type_traits>

#include "lq_common.cuh"
#include "lq_decode.cuh"

namespace lq {

// Shared memory of a CTA, byte offsets: working arrays at fixed places (sized for RM vectors), then one or two slots, which
// are filled by bulk copies: the head block and the records, or (quantizing) a dense state.  A slot is free again when the
// products with the start vectors have been taken; with two of them the next head is asked for when this one is begun.
// A dense state lies in groups of eight rows, DENSE_GROUP bytes apart and shifted against one another by 16-byte units, so
// that the four row groups that a quarter of a warp reads at a time fall on different banks.
constexpr int TOKEN_SLOT = 128;              // a step in one launch: where the slot of its token lies, behind the barriers
constexpr int DENSE_GROUP = 8 * D * 4 + 128;
template <int NW>
__host__ __device__ constexpr int dense_group_at(int g) { return g * DENSE_GROUP + ((g & 1) ? 16 : 0) + ((g & 2) ? (NW == 4 ? 32 : 64) : 0); }
// FIT = false: only what it takes to rebuild a state.
template <int RM, int NW, bool FIT = true>
struct BoundarySmem {
  static constexpr int bar = 0;                              // [2] copy barriers
  static constexpr int invc = 16;                            // [128]      1 / code step, per warp
  static constexpr int ic = invc + 4 * D;                    // [128]      1 / c
  static constexpr int gam = ic + 4 * D;                     // [128]      Gamma_{1:n}
  static constexpr int gram = gam + 4 * D;                   // [RM][RM]   Gram matrix (lower triangle), later K^T K (a > b)
  static constexpr int chol = gram + 4 * RM * RM;            // L [RM][RM], 1 / L_hh [RM], alive [RM] (more than four vectors)
  static constexpr int ub = chol + (RM > 4 ? 4 * (RM * RM + 2 * RM) : 0);      // [RM][128]  value sides as stored, per warp
  static constexpr int T = ub + 4 * D * RM;                  // [RM][128]  S w_h, then the keys as stored
  // Row sums go through here eight vectors at a time (r is more than eight where RM is): all sixteen at once are 64 KB, with which one CTA fits on an SM instead of
  // two (2048 heads, W = 16, r = 16 flushed in 325 us, 239 with eight at a time).
  static constexpr int PV = RM > 8 ? 8 : RM > 0 ? RM : 1;
  static constexpr int part = T + 4 * D * RM;                // [NW][PV][128] per-warp row sums; later [NW][128] those of |R|
  static constexpr int head = FIT ? part + 4 * D * NW * PV : gram;       // the slots
  int rec, slot, dec, kd, Wv, out, bytes;
  __host__ __device__ BoundarySmem(int mode, int W, int r, bool diag, bool rec16, bool bf16, bool iterate, int slots, bool staged_out = false) {
    rec = bf16 ? BF16W_HEAD_BYTES : head_bytes(r);           // within a slot: [W] record rows behind the head block
    slot = mode == 1 ? (RM <= 8 ? 16 * DENSE_GROUP : 0) : rec + (rec16 ? 2 : 4) * record_floats(diag) * W;
    dec = head + slots * slot;                               // [W] scalar gate: the records' decays
    kd = dec + (mode != 1 && !diag ? (4 * W + 15) / 16 * 16 : 0);   // [W][128] fp16 records: Gamma_{j+1:n} kt_j (fp32: in place)
    Wv = kd + (mode != 1 && rec16 ? 4 * D * W : 0);          // [r][128] several rounds: S^T q_h
    out = (Wv + (iterate ? 4 * D * r : 0) + 127) / 128 * 128; // (dequantizing) a dense state on its way out
    bytes = out + (staged_out ? 16 * DENSE_GROUP : 0);
  }
};

// Barrier of the warps that hold a state: all of the CTA, or (GROUP) its first ones (the others of such a CTA have barriers 1 to 8)
template <bool GROUP, int NW>
__device__ __forceinline__ void boundary_sync() {
  if constexpr (GROUP) asm volatile("bar.sync 15, %0;\n" ::"n"(32 * NW) : "memory");
  else __syncthreads();
}

// A state is held by NW warps; of a lane's columns there are tile_cols(NW), in pairs.
__host__ __device__ constexpr int tile_cols(int nw) { return 64 / nw; }
// M += x y^T on the tile
template <int NP>
__device__ __forceinline__ void rank1_pairs(float2 (&M)[8][NP], const float (&x)[8], const float2 (&y)[NP]) {
#pragma unroll
  for (int a = 0; a < 8; a++) {
    const float2 xa = pair(x[a]);
#pragma unroll
    for (int c = 0; c < NP; c++) M[a][c] = __ffma2_rn(xa, y[c], M[a][c]);
  }
}
// the lane's columns of a row (of floats, or fp16 values)
template <int NP, typename T>
__device__ __forceinline__ void load_cols(const T *src, float2 (&x)[NP]) {
#pragma unroll
  for (int b = 0; b < NP / 4; b++) {
    float2 v[4];
    load8p(src + 8 * b, v);
#pragma unroll
    for (int e = 0; e < 4; e++) x[4 * b + e] = v[e];
  }
}
// sum over the lane's columns of one row, block by block
template <int NP>
__device__ __forceinline__ float row_blocks(const float2 (&m)[NP], const float2 (&w)[NP]) {
  float s[NP / 4];
#pragma unroll
  for (int b = 0; b < NP / 4; b++) {
    float2 acc = __fmul2_rn(m[4 * b], w[4 * b]);
#pragma unroll
    for (int c = 1; c < 4; c++) acc = __ffma2_rn(m[4 * b + c], w[4 * b + c], acc);
    s[b] = acc.x + acc.y;
  }
  if constexpr (NP == 8) return s[0] + s[1];
  else return s[0];
}

// Eight floats of a dense state's row.  One 32-byte access (a whole sector) where the base allows it: the lanes of a warp
// touch pieces of 16 rows, and with 16-byte accesses every sector goes to the L2 twice.
__device__ __forceinline__ void load_row8(const float *src, bool wide, float2 (&x)[4]) {
  if (wide)
    asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=f"(x[0].x), "=f"(x[0].y), "=f"(x[1].x), "=f"(x[1].y), "=f"(x[2].x), "=f"(x[2].y), "=f"(x[3].x), "=f"(x[3].y)
                 : "l"(src));
  else
    load8p(src, x);
}
__device__ __forceinline__ void store_row8(float *dst, bool wide, const float2 (&x)[4]) {
  if (wide)
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"l"(dst), "f"(x[0].x), "f"(x[0].y), "f"(x[1].x),
                 "f"(x[1].y), "f"(x[2].x), "f"(x[2].y), "f"(x[3].x), "f"(x[3].y)
                 : "memory");
  else
    store8p(dst, x);
}

template <int NP>
__device__ __forceinline__ void load_row(const float *src, bool wide, float2 (&x)[NP]) {
#pragma unroll
  for (int b = 0; b < NP / 4; b++) {
    float2 v[4];
    load_row8(src + 8 * b, wide, v);
#pragma unroll
    for (int e = 0; e < 4; e++) x[4 * b + e] = v[e];
  }
}
template <int NP>
__device__ __forceinline__ void store_row(float *dst, bool wide, const float2 (&x)[NP]) {
#pragma unroll
  for (int b = 0; b < NP / 4; b++) {
    const float2 v[4] = {x[4 * b], x[4 * b + 1], x[4 * b + 2], x[4 * b + 3]};
    store_row8(dst + 8 * b, wide, v);
  }
}

// eight bfloat16 values
__device__ __forceinline__ void load8_bf16(const uint16_t *src, float (&x)[8]) {
  const uint4 w = *reinterpret_cast<const uint4 *>(src);
  const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int e = 0; e < 4; e++) { x[2 * e] = __uint_as_float(ws[e] << 16); x[2 * e + 1] = __uint_as_float(ws[e] & 0xFFFF0000u); }
}

// Which of the lane's columns a column_tree leaves with it (eight columns: the same one with lanes that differ in bit 4)
template <int NC>
__device__ __forceinline__ int column_of(int lane) {
  if constexpr (NC == 16) return (lane & 2 ? 8 : 0) + (lane & 4 ? 4 : 0) + (lane & 8 ? 2 : 0) + (lane & 16 ? 1 : 0);
  else return (lane & 2 ? 4 : 0) + (lane & 4 ? 2 : 0) + (lane & 8 ? 1 : 0);
}
// one level of halving exchanges: N values of two lanes (differing in lane bit MASK) become N / 2 each
template <int N, int MASK, typename Op>
__device__ __forceinline__ void halve(const float (&p)[N], float (&q)[N / 2], int lane, Op op) {
  const bool up = lane & MASK;
#pragma unroll
  for (int e = 0; e < N / 2; e++) {
    const float keep = up ? p[e + N / 2] : p[e], send = up ? p[e] : p[e + N / 2];
    q[e] = op(keep, __shfl_xor_sync(FULL, send, MASK));
  }
}
// Combine the per-column values p over the 16 lanes ty (lane bits 1..4), neighbouring blocks first, by halving
// exchanges; returns the result of column column_of(lane).
template <int NC, typename Op>
__device__ __forceinline__ float column_tree(const float (&p)[NC], int lane, Op op) {
  if constexpr (NC == 16) {
    float q8[8], q4[4], q2[2], q1[1];
    halve<16, 2>(p, q8, lane, op);
    halve<8, 4>(q8, q4, lane, op);
    halve<4, 8>(q4, q2, lane, op);
    halve<2, 16>(q2, q1, lane, op);
    return q1[0];
  } else {
    float q4[4], q2[2], q1[1];
    halve<8, 2>(p, q4, lane, op);
    halve<4, 4>(q4, q2, lane, op);
    halve<2, 8>(q2, q1, lane, op);
    return op(q1[0], __shfl_xor_sync(FULL, q1[0], 16));
  }
}
// S^T x for the lane's columns: even and odd rows as two chains of the block
template <int NP>
__device__ __forceinline__ void column_blocks(const float2 (&M)[8][NP], const float (&x)[8], float (&pc)[2 * NP]) {
#pragma unroll
  for (int c = 0; c < NP; c++) {
    float2 even = __fmul2_rn(pair(x[0]), M[0][c]), odd = __fmul2_rn(pair(x[1]), M[1][c]);
#pragma unroll
    for (int a = 2; a < 8; a += 2) {
      even = __ffma2_rn(pair(x[a]), M[a][c], even);
      odd = __ffma2_rn(pair(x[a + 1]), M[a + 1][c], odd);
    }
    const float2 s = __fadd2_rn(even, odd);
    pc[2 * c] = s.x; pc[2 * c + 1] = s.y;
  }
}
// Row values of the two lanes tx added; the lane keeps rows 8 ty + 4 tx .. + 3 and puts them into dst[128]
__device__ __forceinline__ void store_row_pairs(const float (&p)[8], int ty, int tx, float *dst) {
  float q[4];
#pragma unroll
  for (int e = 0; e < 4; e++) {
    const float keep = tx ? p[e + 4] : p[e], send = tx ? p[e] : p[e + 4];
    q[e] = keep + __shfl_xor_sync(FULL, send, 1);
  }
  *reinterpret_cast<float4 *>(dst + 8 * ty + 4 * tx) = make_float4(q[0], q[1], q[2], q[3]);
}
// the sum of what the warps left for one row (rows of the warps `stride` floats apart)
template <int NW>
__device__ __forceinline__ float sum_warps(const float *c, int stride) {
  if constexpr (NW == 4) return (c[0] + c[stride]) + (c[2 * stride] + c[3 * stride]);
  return ((c[0] + c[stride]) + (c[2 * stride] + c[3 * stride])) + ((c[4 * stride] + c[5 * stride]) + (c[6 * stride] + c[7 * stride]));
}

// Entry j of start vector h where no buffered record supplies one: -1 where h and j share an odd number of bits
__device__ __forceinline__ float walsh_entry(int h, int j) { return (__popc(h & j) & 1) ? -1.0f : 1.0f; }

// Lower triangle of the Gram matrix of the r vectors X (rows of 128 floats in shared memory), one dot product per
// half-warp and trip.
template <int RM, int NW>
__device__ __forceinline__ void gram_lower(const float *X, int r, float *G, bool with_diagonal) {
  const int hw = threadIdx.x >> 4, c = threadIdx.x & 15;
  const int npairs = with_diagonal ? r * (r + 1) / 2 : r * (r - 1) / 2;
  for (int base = 0; base < npairs; base += 2 * NW) {            // the same trip count for every thread
    const int idx = base + hw;
    const int ii = idx < npairs ? idx : 0;
    int a = 0;                                               // ii = a (a + 1) / 2 + b with b <= a
#pragma unroll
    for (int e = 1; e < RM; e++) a += ii >= e * (e + 1) / 2;
    const int b = ii - a * (a + 1) / 2;
    if (!with_diagonal) a += 1;                              // pairs b < a only
    const float d = dot128_shared(X + a * D, X + b * D, c);
    if (idx < npairs && c == 0) G[a * RM + b] = d;
  }
}

// Cholesky factor of the Gram matrix, by one warp: lane h owns row h of L.  Column by column: lane j finishes
// L_jj from its own row, the lanes below it their entry of column j (the entries of row j they need come by
// shuffle from lane j); the arithmetic of an entry is  s = G_hj; s = fma(-L_hm, L_jm, s) for m < j; L_hj = s / L_jj.
// Writes L (strictly lower part), then inv[h] = 1 / L_hh and alive[h], to shared memory.
// A vector whose squared length is below 1e-30, or of which the vectors before it leave no more than 1e-6 of its
// squared length, is dropped: inv = 0, which makes its orthonormalised vector and all its L entries zero.
// RM: the largest number of vectors this instance is compiled for (nv <= RM), the row length of G and L.
template <int RM>
__device__ __forceinline__ void cholesky_lower_warp(const float *G, int nv, float *L, int lane) {
  float *inv = L + RM * RM, *alive = inv + RM;
  const int h = lane;
  float g[RM], l[RM];
#pragma unroll
  for (int j = 0; j < RM; j++) {
    g[j] = (h < nv && j <= h) ? G[h * RM + j] : 0.0f;
    l[j] = 0.0f;
  }
  float inv_h = 0.0f;
  bool ok_h = false;
#pragma unroll
  for (int j = 0; j < RM; j++) {
    if (j < nv) {                                            // (the same for every lane)
      float d = g[j];                                        // meaningful in lane j: G_jj minus the squares of row j
#pragma unroll
      for (int m = 0; m < j; m++) d = fmaf(-l[m], l[m], d);
      const bool ok = g[j] >= 1e-30f && d > 1e-6f * g[j];
      const float iv = ok ? 1.0f / sqrtf(d) : 0.0f;
      const float inv_j = __shfl_sync(FULL, iv, j);
      if (lane == j) { inv_h = iv; ok_h = ok; }
      float sacc = g[j];                                     // meaningful in lanes h > j: G_hj
#pragma unroll
      for (int m = 0; m < j; m++) sacc = fmaf(-l[m], __shfl_sync(FULL, l[m], j), sacc);
      if (h > j) l[j] = sacc * inv_j;
    }
  }
  if (h < nv) {
#pragma unroll
    for (int j = 0; j < RM; j++)
      if (j < h) L[h * RM + j] = l[j];
    inv[h] = inv_h;
    alive[h] = ok_h ? 1.0f : 0.0f;
  }
}

// Orthonormalise the r vectors X (rows of 128 floats in shared memory) in place, in order:
// q_h = (x_h - sum_{j<h} L_hj q_j) / L_hh, one thread per element index (four warps).  With FINAL the results are rounded to
// fp16 (what is stored as compensator keys), written to keys and kept in X as stored.  Up to four vectors: each of these
// threads computes the factor itself, in registers (no barrier around a chain of four 1/sqrt; the other four warps leave the
// issue slots to them); more: one warp does, through shared memory.
// Returns the bit mask of the vectors that were not dropped.  Begins and ends with a barrier; `behind_first` is called behind
// the first.
template <bool FINAL, int RM, bool GROUP, int NW, typename F>
__device__ __forceinline__ uint32_t orthonormalize(float *X, int r, float *gram, float *chol, uint16_t *keys, F behind_first) {
  __shared__ uint32_t alive_mask;
  const int tid = threadIdx.x, i = tid;
  boundary_sync<GROUP, NW>();
  behind_first();
  gram_lower<RM, NW>(X, r, gram, true);
  boundary_sync<GROUP, NW>();
  LQ_BTICK(7);
  if constexpr (RM > 4) {
    if (tid < 32) cholesky_lower_warp<RM>(gram, r, chol, tid);
    boundary_sync<GROUP, NW>();
  }
  if (tid < D) {
    uint32_t alive = 0;
    float x[RM];
#pragma unroll
    for (int h = 0; h < RM; h++) x[h] = h < r ? X[h * D + i] : 0.0f;
    if constexpr (RM <= 4) {
      float l[4][4], iv[4];
#pragma unroll
      for (int h = 0; h < 4; h++) {
        float gr[4];
#pragma unroll
        for (int j = 0; j <= h; j++) gr[j] = h < r ? gram[h * RM + j] : 0.0f;
#pragma unroll
        for (int j = 0; j < h; j++) {
          float s = gr[j];
#pragma unroll
          for (int m = 0; m < j; m++) s = fmaf(-l[h][m], l[j][m], s);
          l[h][j] = s * iv[j];
        }
        float d = gr[h];
#pragma unroll
        for (int m = 0; m < h; m++) d = fmaf(-l[h][m], l[h][m], d);
        const bool ok = gr[h] >= 1e-30f && d > 1e-6f * gr[h];
        alive |= ok ? 1u << h : 0u;
        iv[h] = ok ? 1.0f / sqrtf(d) : 0.0f;
#pragma unroll
        for (int j = 0; j < h; j++) x[h] = fmaf(-l[h][j], x[j], x[h]);
        x[h] = x[h] * iv[h];
      }
    } else {
      const float *iv = chol + RM * RM;
#pragma unroll
      for (int h = 0; h < RM; h++) {
        if (h < r) {
#pragma unroll
          for (int j = 0; j < h; j++) x[h] = fmaf(-chol[h * RM + j], x[j], x[h]);
          x[h] = x[h] * iv[h];
          alive |= iv[RM + h] != 0.0f ? 1u << h : 0u;
        }
      }
    }
    LQ_BTICK(8);
#pragma unroll
    for (int h = 0; h < RM; h++) {
      if (h < r) {
        float out = x[h];
        if (FINAL) {
          const uint16_t bits = (alive >> h) & 1u ? to_f16_bits_sat(out) : static_cast<uint16_t>(0);
          keys[h * D + i] = bits;
          out = f16_bits(bits);
        }
        X[h * D + i] = out;
      }
    }
    if (FINAL && tid == 0) alive_mask = alive;
  }
  boundary_sync<GROUP, NW>();
  return FINAL ? alive_mask : 0u;
}

// Working arrays of the warps that take a state through its boundary (shared memory)
struct BoundaryArrays {
  float *dec, *gam;                          // [W] the records' decays (scalar gate), [128] Gamma_{1:n}
  float *kd;                                 // [W][128] fp16 records: Gamma_{j+1:n} kt_j (fp32: in place of kt_j)
  float *part, *abs_part;                    // [NW][PV][128] per-warp row sums, [NW][128] those of |R|
  float *T, *Wv, *gram, *chol;               // see BoundarySmem
  float *ub, *ic, *invc;                     // ub, invc: this warp's
  unsigned char *rows = nullptr, *newest = nullptr;           // (GROUP) the record rows but the last one, and that
  unsigned char *out = nullptr;              // (dequantizing) where the state is put together for bulk stores, or null
};

// One head through its boundary (MODE, RM, BF16, EXACT, ROUNDS: see boundary_kernel): `slot` holds its head block and, behind it, its n
// records, or a dense state.  GROUP: the eight warps are the first of a larger CTA, and the row sums lie in the slot, where the codes
// were (PV = 4 vectors at a time: each warp's sums take the place of the 2 KB of codes that only this warp reads).
// slot_is_free() is called by every thread, behind a barrier after which nobody reads the slot.
template <int GATE, int MODE, bool R16, int RM, bool BF16, bool EXACT, bool ROUNDS, bool GROUP, int PV, int NW, typename F>
__device__ __forceinline__ void boundary_head(const Params &p, const BoundaryArrays &A, unsigned char *slot, const size_t bh, const int n,
                                              const int r, const int rT, const bool wide, F slot_is_free) {
  // Exactly four vectors: registers are left for deeper unrolling, step 61.3 -> 60.8 us and 74.2 -> 73.0 at W = 8; for exactly
  // eight it is slower, 234.3 -> 236.5 us at 512 x 32 heads, diagonal gate, W = 64.  Not with four warps, whose code is twice as long to
  // begin with: behind other kernels it comes from the L2 or beyond, and that is where it runs in a model.  256 x 32 heads, scalar gate,
  // us per step, in a loop of steps / with a projection, norms and a softmax in front of each: records 4, start vectors 4 at a time and
  // the loops over the rounds in between 59.1 / 69.7, W = 8 72.1 / 83.9; one at a time and no such loops (ROUNDS) 59.3 / 64.4 and
  // 71.8 / 76.9; eight warps 59.6 / 64.0 and 73.5 / 78.3.
  constexpr bool FOUR = EXACT && RM == 4 && MODE == 0, DEEP = FOUR && NW == 8 && !GROUP;
  constexpr bool DIAG = GATE == LQ_GATE_DIAG, RECORDS = MODE != 1, STAGED = MODE != 1 || RM <= 8;
  constexpr int RF = record_floats(DIAG);
  using rec_t = typename std::conditional<R16, __half, float>::type;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, ty = lane >> 1, tx = lane & 1;
  constexpr int NT = 32 * NW, NC = tile_cols(NW), NP = NC / 2, CW = 2 * NC;   // threads, columns of a lane, pairs of them, columns of a warp
  const int v0 = CW * warp + NC * tx;        // the lane's first column
  float *dec = A.dec, *gam = A.gam, *part = A.part, *abs_part = A.abs_part, *T = A.T, *Wv = A.Wv, *gram = A.gram, *chol = A.chol;
  float *ub = A.ub, *ic_s = A.ic, *invc = A.invc;
  rec_t *rec = reinterpret_cast<rec_t *>(slot + (BF16 ? BF16W_HEAD_BYTES : head_bytes(r)));
  auto rec_row = [&](int j) -> rec_t * {
    if constexpr (GROUP) return reinterpret_cast<rec_t *>(j == n - 1 ? A.newest : A.rows + j * (RF * sizeof(rec_t)));
    else return rec + j * RF;
  };
  auto kd_row = [&](int j) -> float * {                   // Gamma_{j+1:n} kt_j
    if constexpr (R16) return A.kd + j * D;
    else return rec_row(j) + REC_KT;
  };
  if (RECORDS) {
    // cumulative decays, newest record first (Appendix B.2): kd_j = Gamma_{j+1:n} kt_j, gam = Gamma_{1:n}
    if (tid < D) {
      auto kt_at = [&](int j) { return static_cast<float>(rec_row(j)[REC_KT + tid]); };
      auto a_at = [&](int j) { return DIAG ? static_cast<float>(rec_row(j)[REC_A + tid]) : dec[j]; };
      float g = 1.0f;
      int j = n - 1;
      for (; j >= 3; j -= 4) {                            // four records per trip: the loads go out together
        float kt[4], a[4];
#pragma unroll
        for (int e = 0; e < 4; e++) { kt[e] = kt_at(j - e); a[e] = a_at(j - e); }
#pragma unroll
        for (int e = 0; e < 4; e++) { kd_row(j - e)[tid] = g * kt[e]; g = g * a[e]; }
      }
      for (; j >= 0; j--) { const float kt = kt_at(j); kd_row(j)[tid] = g * kt; g = g * a_at(j); }
      gam[tid] = g;
    }
    boundary_sync<GROUP, NW>();
    LQ_BTICK(2);
  }

  float2 M[8][NP];                                        // rows 8 ty + a, columns v0 + 2 c, v0 + 2 c + 1
  // ---- the dense state (Eq. 7) ----
  if constexpr (RECORDS) {
    const uint8_t *zt = slot + HB_CODES;
    const uint16_t *ckh = reinterpret_cast<const uint16_t *>(slot + HB_COMP_K), *cuh = ckh + r * D;
    if constexpr (BF16) {
#pragma unroll
      for (int c = 0; c < NP; c++) {
        float lo[8], hi[8];                               // columns v0 + 2 c, v0 + 2 c + 1
        load8_bf16(reinterpret_cast<const uint16_t *>(slot) + (v0 + 2 * c) * D + 8 * ty, lo);
        load8_bf16(reinterpret_cast<const uint16_t *>(slot) + (v0 + 2 * c + 1) * D + 8 * ty, hi);
#pragma unroll
        for (int a = 0; a < 8; a++) M[a][c] = make_float2(lo[a], hi[a]);
      }
    } else {
      float ci[8];
      float2 sj[NP];
      load8(reinterpret_cast<const float *>(slot + HB_ROW_SMOOTH) + 8 * ty, ci);
      load_cols(reinterpret_cast<const float *>(slot + HB_COL_SCALE) + v0, sj);
      uint2 zz[NC];
#pragma unroll
      for (int b = 0; b < NC; b++) {
        zz[b] = *reinterpret_cast<const uint2 *>(zt + (v0 + b) * D + 8 * ty);
        zz[b].x ^= 0x80808080u; zz[b].y ^= 0x80808080u;
      }
      // int8 -> fp32 without the conversion unit: byte + 128 in the low mantissa bits of 2^23, minus 2^23 + 128
#pragma unroll
      for (int a = 0; a < 8; a++)
#pragma unroll
        for (int c = 0; c < NP; c++) {
          const float2 raw = make_float2(
              __uint_as_float(__byte_perm(a < 4 ? zz[2 * c].x : zz[2 * c].y, 0x4B000000u, 0x7540 | (a & 3))),
              __uint_as_float(__byte_perm(a < 4 ? zz[2 * c + 1].x : zz[2 * c + 1].y, 0x4B000000u, 0x7540 | (a & 3))));
          M[a][c] = __fmul2_rn(pair(ci[a]), __fmul2_rn(__fadd2_rn(raw, pair(-8388736.0f)), sj[c]));
        }
    }
#pragma unroll (FOUR && !GROUP ? 2 : 1)
    for (int h = 0; h < r; h++) {
      float kc[8];
      float2 uc[NP];
      load8(reinterpret_cast<const __half *>(ckh + h * D + 8 * ty), kc);
      load_cols(reinterpret_cast<const __half *>(cuh + h * D + v0), uc);
      rank1_pairs(M, kc, uc);
    }
    {
      float gi[8];
      load8(gam + 8 * ty, gi);
#pragma unroll
      for (int a = 0; a < 8; a++)
#pragma unroll
        for (int c = 0; c < NP; c++) M[a][c] = __fmul2_rn(pair(gi[a]), M[a][c]);
    }
    constexpr int AHEAD = MODE == 2 ? 1 : DEEP ? 4 : FOUR || GROUP ? 1 : 2;   // (dequantizing spills with two records at a time)
#pragma unroll AHEAD
    for (int j = 0; j < n; j++) {
      float kj[8];
      float2 uj[NP];
      load8(kd_row(j) + 8 * ty, kj);
      load_cols(rec_row(j) + REC_U + v0, uj);
      rank1_pairs(M, kj, uj);
    }
    LQ_BTICK(3);
  } else if constexpr (STAGED) {
    const float *S = reinterpret_cast<const float *>(slot + dense_group_at<NW>(ty)) + v0;
#pragma unroll
    for (int a = 0; a < 8; a++) load_cols(S + a * D, M[a]);
  } else {
    const float *S = p.S + bh * (size_t)(D * D) + 8 * ty * D + v0;
#pragma unroll
    for (int a = 0; a < 8; a++) load_row(S + a * D, wide, M[a]);
  }
  if constexpr (MODE == 2) {
    if (A.out) {
      if (warp == 0) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");      // (the state before has left)
    } else {
      float *S = p.S + bh * (size_t)(D * D) + 8 * ty * D + v0;
#pragma unroll
      for (int a = 0; a < 8; a++) store_row(S + a * D, wide, M[a]);
    }
  } else if constexpr (RM > 0) {
    // T_h = S w_h; w_h is the value side of the (h+1)-th newest record, or Walsh function h
    auto start_vector = [&](int h, float2 (&w)[NP]) {
      if (RECORDS && h < n) {
        load_cols(rec_row(n - 1 - h) + REC_U + v0, w);
      } else {
#pragma unroll
        for (int c = 0; c < NP; c++) w[c] = make_float2(walsh_entry(h, v0 + 2 * c), walsh_entry(h, v0 + 2 * c + 1));
      }
    };
    auto row_sums = [&](const float2 (&w)[NP], int at) {
      float pr[8];
#pragma unroll
      for (int a = 0; a < 8; a++) pr[a] = row_blocks(M[a], w);
      store_row_pairs(pr, ty, tx, part + (warp * PV + at) * D);
    };
    if constexpr (RM > PV) {
#pragma unroll 2
      for (int h = 0; h < rT; h++) {
        if (h == PV) {                                    // more than eight (up to sixteen): the first eight are summed here
          boundary_sync<GROUP, NW>();
          for (int idx = tid; idx < PV * D; idx += NT) T[idx] = sum_warps<NW>(part + idx, PV * D);
          boundary_sync<GROUP, NW>();
        }
        float2 w[NP];
        start_vector(h, w);
        row_sums(w, h % PV);
      }
    } else {
#pragma unroll (DEEP ? 4 : GROUP || (NW == 4 && EXACT) ? 1 : 2)
      for (int h = 0; h < rT; h++) {
        float2 w[NP];
        start_vector(h, w);
        row_sums(w, h);
      }
    }
  }
  // without row sums in it the slot is free when all have come here: the next head may land while this one is worked on
  constexpr bool SUMS_IN_SLOT = GROUP && RM > 0;
  if (STAGED && !SUMS_IN_SLOT) asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  boundary_sync<GROUP, NW>();
  if (!SUMS_IN_SLOT) slot_is_free();
  if constexpr (MODE == 2) {
    if (A.out) {
      float *rows = reinterpret_cast<float *>(A.out + dense_group_at<NW>(ty)) + v0;
#pragma unroll
      for (int a = 0; a < 8; a++) {
#pragma unroll
        for (int b = 0; b < NP / 2; b++)
          *reinterpret_cast<float4 *>(rows + a * D + 4 * b) = make_float4(M[a][2 * b].x, M[a][2 * b].y, M[a][2 * b + 1].x, M[a][2 * b + 1].y);
      }
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      boundary_sync<GROUP, NW>();
      if (warp == 0) {
        if (lane < 16) bulk_s2g(p.S + bh * (size_t)(D * D) + lane * 8 * D, smem_addr(A.out) + dense_group_at<NW>(lane), 8 * D * 4);
        asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
      }
    }
  }

  if constexpr (BF16 && MODE != 2) {                      // round and store: that is the new boundary state
    uint16_t *S0T = reinterpret_cast<uint16_t *>(p.heads + bh * (size_t)BF16W_HEAD_BYTES) + v0 * D + 8 * ty;
#pragma unroll
    for (int c = 0; c < NP; c++) {
      uint32_t lo[4], hi[4];
#pragma unroll
      for (int e = 0; e < 4; e++) {
        lo[e] = (uint32_t)to_bf16_bits(M[2 * e][c].x) | ((uint32_t)to_bf16_bits(M[2 * e + 1][c].x) << 16);
        hi[e] = (uint32_t)to_bf16_bits(M[2 * e][c].y) | ((uint32_t)to_bf16_bits(M[2 * e + 1][c].y) << 16);
      }
      *reinterpret_cast<uint4 *>(S0T + (2 * c) * D) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      *reinterpret_cast<uint4 *>(S0T + (2 * c + 1) * D) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    }
    if (MODE == 1 && tid == 0) p.win_pos[bh / p.heads_v] = 0;
  } else if constexpr (MODE != 2) {
    uint32_t alive = 0;
    if constexpr (RM > 0) {
      constexpr int T0 = RM > PV ? PV * D : 0;            // (those before are there)
      for (int idx = T0 + tid; idx < r * D; idx += NT) T[idx] = sum_warps<NW>(part + idx - T0, PV * D);
      LQ_BTICK(10);
      // further rounds: W_h = S^T q_h, orthonormalise, T_h = S q_h
      for (int it = 1; ROUNDS && it < p.n_iter; it++) {
        orthonormalize<false, RM, GROUP, NW>(T, r, gram, chol, nullptr, [] {});
#pragma unroll 1
        for (int h = 0; h < r; h++) {
          float x[8], pc[NC];
          load8(T + h * D + 8 * ty, x);
          column_blocks(M, x, pc);
          const float s = column_tree(pc, lane, [](float a, float b) { return a + b; });
          if (NC == 16 || lane < 16) Wv[h * D + v0 + column_of<NC>(lane)] = s;
        }
        orthonormalize<false, RM, GROUP, NW>(Wv, r, gram, chol, nullptr, [] {});
#pragma unroll 1
        for (int h = 0; h < r; h++) {
          if (RM > PV && h == PV) {
            boundary_sync<GROUP, NW>();
            for (int idx = tid; idx < PV * D; idx += NT) T[idx] = sum_warps<NW>(part + idx, PV * D);
            boundary_sync<GROUP, NW>();
          }
          float2 w[NP];
          load_cols(Wv + h * D + v0, w);
          float pr[8];
#pragma unroll
          for (int a = 0; a < 8; a++) pr[a] = row_blocks(M[a], w);
          store_row_pairs(pr, ty, tx, part + (warp * PV + (RM > PV ? h % PV : h)) * D);
        }
        boundary_sync<GROUP, NW>();
        for (int idx = T0 + tid; idx < r * D; idx += NT) T[idx] = sum_warps<NW>(part + idx - T0, PV * D);
      }
      if (SUMS_IN_SLOT) asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      alive = orthonormalize<true, RM, GROUP, NW>(T, r, gram, chol, p.comp_k(bh), [&] {   // T then holds the keys as stored
        if (SUMS_IN_SLOT) slot_is_free();
      });
      LQ_BTICK(11);
      gram_lower<RM, NW>(T, r, gram, false);                  // k_a^T k_h (published by the barrier in front of the value sides)

      // ---- value sides and removal of the stored tokens ----
      float x[RM];                                        // S^T k_h for the lane's column
      const int col = column_of<NC>(lane);
      auto column_sum = [&](int h) {
        float kf[8], pc[NC];
        load8(T + h * D + 8 * ty, kf);
        column_blocks(M, kf, pc);
        return column_tree(pc, lane, [](float a, float b) { return a + b; });
      };
      if constexpr (GROUP) {                              // (one after the other through ub: one copy of the code, see step_kernel)
#pragma unroll 1
        for (int h = 0; h < r; h++) {
          const float sum = column_sum(h);
          if (NC == 16 || lane < 16) ub[CW * h + NC * tx + col] = sum;
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < RM; h++) x[h] = h < r ? ub[CW * h + NC * tx + col] : 0.0f;
        __syncwarp();
      } else {
#pragma unroll
        for (int h = 0; h < RM; h++) x[h] = h < r ? column_sum(h) : 0.0f;
      }
      boundary_sync<GROUP, NW>();                                    // K^T K is complete
      LQ_BTICK(13);
      // u_h = S^T k_h - sum_{a<h} u_a (k_a^T k_h) with the stored values: what tokens 0..h-1 leave
      float uf[RM];
      uint16_t *cu_out = p.comp_u(bh) + v0 + col;
#pragma unroll
      for (int h = 0; h < RM; h++) {
        uf[h] = 0.0f;
        if (h < r) {
#pragma unroll
          for (int a = 0; a < h; a++) x[h] = fmaf(-uf[a], gram[h * RM + a], x[h]);
          const uint16_t bits = (alive >> h) & 1u ? to_f16_bits_sat(x[h]) : static_cast<uint16_t>(0);
          uf[h] = f16_bits(bits);
          if (NC == 16 || lane < 16) {
            cu_out[h * D] = bits;
            ub[CW * h + NC * tx + col] = uf[h];
          }
        }
      }
      __syncwarp();
      LQ_BTICK(14);
#pragma unroll ((FOUR && !GROUP) || NW == 4 ? 2 : 1)
      for (int h = 0; h < r; h++) {                       // M -= k u^T with the stored values
        float kf[8];
        float2 uv[NP];
        load8(T + h * D + 8 * ty, kf);
        load_cols(ub + CW * h + NC * tx, uv);
#pragma unroll
        for (int a = 0; a < 8; a++) kf[a] = -kf[a];
        rank1_pairs(M, kf, uv);
      }
    }
    LQ_BTICK(4);
    // ---- residual smoothing: c_i = max(sqrt(mean_j |R_ij|), 1e-6) ----
    {
      float pr[8];
#pragma unroll
      for (int a = 0; a < 8; a++) {                       // even and odd columns as two chains
        float s[NP / 4];
#pragma unroll
        for (int b = 0; b < NP / 4; b++) {
          float even = fabsf(M[a][4 * b].x), odd = fabsf(M[a][4 * b].y);
#pragma unroll
          for (int c = 1; c < 4; c++) { even = even + fabsf(M[a][4 * b + c].x); odd = odd + fabsf(M[a][4 * b + c].y); }
          s[b] = even + odd;
        }
        if constexpr (NP == 8) pr[a] = s[0] + s[1];
        else pr[a] = s[0];
      }
      store_row_pairs(pr, ty, tx, abs_part + warp * D);
    }
    boundary_sync<GROUP, NW>();
    if (tid < D) {
      const float ci = p.smooth ? fmaxf(sqrtf(sum_warps<NW>(abs_part + tid, D) / static_cast<float>(D)), 1e-6f) : 1.0f;
      ic_s[tid] = p.smooth ? 1.0f / ci : 1.0f;
      p.row_smooth(bh)[tid] = ci;
    }
    boundary_sync<GROUP, NW>();
    LQ_BTICK(5);

    // ---- code steps and codes ----
    {
      float ic[8];
      load8(ic_s + 8 * ty, ic);
#pragma unroll
      for (int a = 0; a < 8; a++)
#pragma unroll
        for (int c = 0; c < NP; c++) M[a][c] = __fmul2_rn(M[a][c], pair(ic[a]));
    }
    float m[NC];
#pragma unroll
    for (int c = 0; c < NP; c++) {
      m[2 * c] = fabsf(M[0][c].x); m[2 * c + 1] = fabsf(M[0][c].y);
#pragma unroll
      for (int a = 1; a < 8; a++) {
        m[2 * c] = fmaxf(m[2 * c], fabsf(M[a][c].x));
        m[2 * c + 1] = fmaxf(m[2 * c + 1], fabsf(M[a][c].y));
      }
    }
    const float amax = column_tree(m, lane, [](float a, float b) { return fmaxf(a, b); });
    if (NC == 16 || lane < 16) {
      const int col = column_of<NC>(lane);
      p.col_scale(bh)[v0 + col] = amax / 127.0f;          // stored as the step of the code, B_j / 127
      invc[NC * tx + col] = amax > 0.0f ? 127.0f / amax : 0.0f;
    }
    __syncwarp();
    LQ_BTICK(6);
    float2 inv[NP];
    load_cols(invc + NC * tx, inv);
    int8_t *ZT = p.codes(bh) + v0 * D + 8 * ty;
#pragma unroll
    for (int c = 0; c < NP; c++) {
      // |X * inv| <= 127 (1 + 2^-23): adding 1.5 * 2^23 leaves the nearest integer (ties to even) in the low byte
      // (product and sum are rounded one after the other; written as a packed addition the two would get fused)
      float2 z[8];
#pragma unroll
      for (int a = 0; a < 8; a++) z[a] = __ffma2_rn(__fmul2_rn(M[a][c], inv[c]), pair(1.0f), pair(12582912.0f));
      auto bytes4 = [](float x0, float x1, float x2, float x3) {
        return __byte_perm(__byte_perm(__float_as_uint(x0), __float_as_uint(x1), 0x0040),
                           __byte_perm(__float_as_uint(x2), __float_as_uint(x3), 0x0040), 0x5410);
      };
      *reinterpret_cast<uint2 *>(ZT + (2 * c) * D) =
          make_uint2(bytes4(z[0].x, z[1].x, z[2].x, z[3].x), bytes4(z[4].x, z[5].x, z[6].x, z[7].x));
      *reinterpret_cast<uint2 *>(ZT + (2 * c + 1) * D) =
          make_uint2(bytes4(z[0].y, z[1].y, z[2].y, z[3].y), bytes4(z[4].y, z[5].y, z[6].y, z[7].y));
    }
    if (MODE == 1 && tid == 0) p.win_pos[bh / p.heads_v] = 0;      // (nobody reads win_pos in this mode)
  }
}

// MODE 0 flush (window representation -> dense -> new window representation), 1 quantize dense fp32 states,
// 2 dequantize to dense fp32 states.  RM: the largest r the instance handles; 0: no compensators at all (an instance of its
// own: told apart inside the others, the two ways cost those 400 bytes of spills; in the one for r = 0 the compiler still spills
// 280 bytes: 256 x 32 heads, W = 16, r = 0, 53.0 us a step, 71.7 with the former layout, which spilled none).
// BF16: the per-window BF16 state (lq_shape.state_bf16, RM = 0): the dense state is rounded to bfloat16, and that is all.
// slots: 1 or 2.  staged_out (dequantizing): a state leaves by bulk stores from shared memory.
// EXACT: r is RM, known at compile time: without a test per vector the compiler interleaves the four or eight column sums
// (flush at 256 x 32 heads: step 62.2 -> 61.4 us, W = 8 75.6 -> 74.4; quantizing 2048 states, r = 4: 57.5 -> 55.2 us, where only
// the products with the start vectors must not know r: the vectors, the same for every head, would be kept in registers and
// others spilled, 69.9 us; with eight vectors it spills all the same).
// ROUNDS: p.n_iter may be more than one.  Without, the loops over the further rounds, a third of the code on the way, are not there.
// STEP (a flush): a whole decode step of few heads in one launch.  Every CTA has one head: two of its warps take it through the
// token (decode_slot), then, if that filled the window, the CTA through the boundary.  What bounds it: the latency of a token and
// of a boundary, and the host time of a launch, of which it needs one instead of two (figures: one_launch).
template <int GATE, int MODE, bool R16, int RM, bool BF16, bool EXACT, bool ROUNDS, bool STEP, int NW>
__global__ void __launch_bounds__(32 * NW, STEP ? 1 : 2) boundary_kernel(const Params p, const int slots, const int staged_out) {
  constexpr bool DIAG = GATE == LQ_GATE_DIAG, RECORDS = MODE != 1, STAGED = MODE != 1 || RM <= 8;
  static_assert(!BF16 || RM == 0, "the per-window BF16 state has no compensators");
  constexpr int RF = record_floats(DIAG);
  using rec_t = typename std::conditional<R16, __half, float>::type;
  using Lay = BoundarySmem<MODE == 2 ? 0 : RM, NW, MODE != 2>;
  constexpr int PV = Lay::PV;                // vectors whose row sums `part` holds at a time
  extern __shared__ __align__(128) unsigned char lq_bsm[];
  __shared__ unsigned todo_bh[32], due_counts[2][8];
  __shared__ int todo_n[32], todo_count, lead_due[8];
  const int W = p.W, rT = MODE == 1 ? p.r : EXACT ? RM : p.r, r = EXACT ? RM : RM > 0 ? p.r : 0, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (RM > 0 && r < 1) return;               // (not launched)
  const unsigned nh = static_cast<unsigned>(p.batch) * p.heads_v;
  const Lay L(MODE, W, r, DIAG, R16, BF16, MODE != 2 && RM > 0 && p.n_iter > 1, slots);
  float *dec = reinterpret_cast<float *>(lq_bsm + L.dec);
  auto at_bytes = [&](int offset) { return reinterpret_cast<float *>(lq_bsm + offset); };
  BoundaryArrays A{dec, at_bytes(Lay::gam), at_bytes(L.kd), at_bytes(Lay::part), at_bytes(Lay::part), at_bytes(Lay::T), at_bytes(L.Wv),
                         at_bytes(Lay::gram), at_bytes(Lay::chol), at_bytes(Lay::ub) + warp * (D / NW) * RM, at_bytes(Lay::ic), at_bytes(Lay::invc) + D / NW * warp};
  if (MODE == 2 && RM > 0 && NW == 4 && staged_out) A.out = lq_bsm + L.out;
  const uint32_t bar = smem_addr(lq_bsm + Lay::bar);
  const bool wide = (reinterpret_cast<uintptr_t>(p.S) & 31) == 0;
  LQ_STAMP(1, 0);
  if (STAGED && tid == 0) { mbar_init(bar, 1); mbar_init(bar + 8, 1); }
  unsigned char *token_slot = lq_bsm + TOKEN_SLOT;     // (the boundary's arrays and slot take its place)
  if constexpr (STEP) {
    if (tid == 0) {
      const uint32_t token_bar = smem_addr(token_slot + DecodeSlot(W, p.r, DIAG, R16, BF16, 0).mbar);
      mbar_init(token_bar, 1);
      mbar_init(token_bar + 8, 1);
    }
    __syncthreads();
  }
  grid_dependency_wait();                    // everything the kernel before this one wrote is visible from here on
  if (STEP) grid_dependents_may_start();     // (up to half as many heads as SMs, the next step's CTAs find room beside these)
  LQ_STAMP(1, 1);
#ifdef LQ_TIMING
  if (tid == 0) { for (int i = 0; i < 16; i++) lq_bacc[i] = 0; lq_btick = clock64(); }
#endif
  // the decode kernels ahead of a flush count the tickets of their pools of heads in the state's scratch words
  if (MODE == 0 && !STEP && p.work != nullptr && blockIdx.x == 0 && tid < LQ_WORK_WORDS) p.work[tid] = 0;

  uint32_t parity = 0;                       // bit b: phase of copy barrier b
  int at = 0;                                // the slot of the head at hand
  float dec_next = 0.0f;                     // this thread's decay of the head on its way (scalar gate, tid < n)
  auto request = [&](size_t bh, int n, int to) {             // bring head bh and its n records, or its dense state, into slot `to`
    const uint32_t dst = smem_addr(lq_bsm + Lay::head) + to * L.slot, bar_to = bar + 8 * to;
    if constexpr (RECORDS) {
      if (!DIAG && tid < n) dec_next = p.decays[bh * (size_t)W + tid];
      if (tid == 0) {
        const uint32_t rb = static_cast<uint32_t>(sizeof(rec_t)) * RF * n;
        mbar_expect_tx(bar_to, L.rec + rb);
        bulk_g2s(dst, p.heads + bh * (size_t)L.rec, L.rec, bar_to);
        if (n > 0) bulk_g2s(dst + L.rec, p.record<rec_t>(bh, 0, DIAG), rb, bar_to);
      }
    } else if (warp == 0) {
      if (lane == 0) mbar_expect_tx(bar_to, 4 * D * D);
      __syncwarp();
      if (lane < 16) bulk_g2s(dst + dense_group_at<NW>(lane), p.S + bh * (size_t)(D * D) + lane * 8 * D, 8 * D * 4, bar_to);
    }
  };

  // The CTA puts together its next 32 heads (a flush: of those that are due, see list_due_heads; otherwise warp 0, every
  // gridDim-th head) and how many records each holds; then the CTA takes them one after the other.
  int count = 32;
  for (unsigned first = blockIdx.x; count == 32; first += 32 * gridDim.x) {
    if constexpr (STEP) {
      const int b = blockIdx.x / p.heads_v, n_in = p.win_pos[b] & 0xFFFF;
      if (warp < 2) {
        decode_slot<GATE, R16, false, BF16, true>(p, token_slot, lane, warp, blockIdx.x, gridDim.x);
        asm volatile("fence.proxy.async;\n" ::: "memory");    // the record is written; a bulk copy may read it next
      }
      // (the barrier is where the whole CTA has read win_pos, ahead of its arrival)
      const bool due = __syncthreads_or(n_in == W - 1 || n_in == W);
      // (a sequence beyond W gets no token and keeps its entry, upper bits included)
      if (tid == 0 && n_in <= W) arrive_and_set(p.win_pos, b, p.heads_v, due ? 0 : n_in + 1);
      if (!due) return;
      if (tid == 0) {
        const uint32_t token_bar = smem_addr(token_slot + DecodeSlot(W, p.r, DIAG, R16, BF16, 0).mbar);
        mbar_inval(token_bar);
        mbar_inval(token_bar + 8);
        // (the two words may lie where a bulk copy of the boundary lands: the warps' fences came before these accesses)
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        todo_bh[0] = blockIdx.x;
        todo_n[0] = W;
        todo_count = 1;
      }
    } else if constexpr (MODE == 0) {
      if (warp < due_scan_warps<NW>(p)) {
        int lead;
        const int c = list_due_heads<NW>(p, first, gridDim.x, due_scan_warps<NW>(p), due_counts, todo_bh, todo_n, lead);
        if (lane == 0) lead_due[warp] = lead;
        if (tid == 0) todo_count = c;
      }
    } else if (warp == 0) {
      const unsigned bh_mine = first + lane * gridDim.x;
      const bool have = bh_mine < nh;
      const int n_mine = MODE == 2 && have ? p.win_pos[bh_mine / p.heads_v] & 0xFFFF : 0;
      const int c = __popc(__ballot_sync(FULL, have));
      todo_bh[lane] = bh_mine;
      todo_n[lane] = n_mine > W ? W : n_mine;
      if (lane == 0) todo_count = c;
    }
    __syncthreads();
    count = todo_count;
    if (STAGED && count > 0) request(todo_bh[0], todo_n[0], at);
    // report that this CTA has seen all of win_pos, once the first head's copies are on their way (the round trip hides behind
    // them), part by part; with nothing due in a part there is nothing to restart
    if (MODE == 0 && !STEP && count < 32) {
      const int warps = due_scan_warps<NW>(p), w = (warp + 1) % NW;     // (the last warp for part 0)
      if (w < warps && lead_due[w] >= 0) restart_due_windows(p, lead_due[w], w, warps);
    }
    LQ_BTICK(0);

    for (int k = 0; k < count; k++) {
      const size_t bh = todo_bh[k];
      if (MODE == 0 && p.overlap && count < 32 && k == count - 1) grid_dependents_may_start();
      const int n = todo_n[k];                                // (never 0 when due)
      unsigned char *slot = lq_bsm + Lay::head + at * L.slot;
      if (RECORDS && !DIAG && tid < n) dec[tid] = dec_next;
      if (STAGED) {
        if (slots > 1 && k + 1 < count) request(todo_bh[k + 1], todo_n[k + 1], at ^ 1);
        if (!mbar_wait(bar + 8 * at, (parity >> at) & 1u) && lane == 0) atomicOr(&g_device_error, 1);
        parity ^= 1u << at;
      }
      if (RECORDS) {
        if (!DIAG) __syncthreads();
        if (k == 0) LQ_STAMP(1, 2);
        LQ_BTICK(1);
      }
      boundary_head<GATE, MODE, R16, RM, BF16, EXACT, ROUNDS, false, PV, NW>(p, A, slot, bh, n, r, rT, wide, [&] {
        if (STAGED && slots == 1 && k + 1 < count) request(todo_bh[k + 1], todo_n[k + 1], at);
        if (!STAGED && k + 1 < count && tid < 8)              // (dense states: at least into the L2)
          bulk_prefetch_l2(p.S + todo_bh[k + 1] * (size_t)(D * D) + tid * (D * D / 8), D * D / 2);
        if (slots > 1) at ^= 1;
      });
      if (k == 0) LQ_STAMP(1, 3);
      LQ_BTICK(9);
    }
    __syncthreads();                         // the list is rewritten by the next round
  }
  if (MODE == 2 && RM > 0 && NW == 4 && staged_out && warp == 0) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
  LQ_STAMP(1, 4);
#ifdef LQ_TIMING
  if (tid == 0)
    for (int i = 0; i < 16; i++) atomicAdd(&g_phase_cycles[32 + i], (unsigned long long)lq_bacc[i]);
#endif
}

}  // namespace lq
