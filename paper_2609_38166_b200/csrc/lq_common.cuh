// Device helpers shared by the sm_100a kernels of the per-window 8-bit decode step.
//
// Everything is compiled with -fmad=false: a product is fused with an addition only where fmaf() is
// written, so that every value is reproducible bit for bit.  Sums over a channel index follow one
// fixed order: the terms are taken in blocks of eight; inside a block the even- and the odd-numbered
// terms form two chains, each accumulated left to right (first product rounded, the rest folded in with
// fmaf), and the two chains are added; block results are added as a balanced binary tree over the block
// index.  The thread mappings below are chosen so that this order is the natural one: a thread owns one
// block of eight (where registers allow, as four float2 pairs, so that one packed fused multiply-add,
// FFMA2 on sm_100, advances both chains); neighbouring lanes own neighbouring blocks, and butterfly
// exchanges with lane masks 1, 2, 4, ... walk up the tree.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/lq.h"

namespace lq {

constexpr int D = 128;       // d_k = d_v of the supported shape
constexpr int MAX_W = 64;
constexpr int MAX_R = 16;
constexpr unsigned FULL = 0xffffffffu;

// Byte offsets inside a head block and float offsets inside a record row (d_k = d_v = 128).
constexpr int HB_CODES = 0;
constexpr int HB_COL_SCALE = D * D;
constexpr int HB_ROW_SMOOTH = HB_COL_SCALE + 4 * D;
constexpr int HB_COMP_K = HB_ROW_SMOOTH + 4 * D;
__host__ __device__ constexpr int hb_comp_u(int r) { return HB_COMP_K + 2 * D * r; }
__host__ __device__ constexpr int head_bytes(int r) { return HB_COMP_K + 4 * D * r; }
constexpr int BF16W_HEAD_BYTES = 2 * D * D;   // per-window BF16: S0^T
__host__ __device__ constexpr int record_floats(bool diag) { return diag ? 3 * D : 2 * D; }
constexpr int REC_KT = 0, REC_U = D, REC_A = 2 * D;

// Launch-time description of one call, passed to the kernels by value.
struct Params {
  int batch, heads_v, heads_qk, W, r, n_iter, smooth, delta, rec16, force;
  int overlap;       // let the next kernel of the stream start when every CTA is at its last head (else when all have ended)
  uint8_t *heads;    // [B*Hv] head blocks of head_bytes(r)
  void *records;     // [B*Hv][W] record rows of record_floats(gate) elements, fp32 or (rec16) fp16
  float *decays;     // scalar gate: [B*Hv][W]
  int32_t *win_pos;
  int32_t *work;     // lq_state.work (scratch words, zero between calls), or null
  const uint16_t *q, *k, *v, *beta, *alpha;
  float *o;
  float *S;          // dense fp32 states (quantize / dequantize / fp32 baseline)
  uint16_t *S16;     // dense bf16 states (bf16 baseline)
#ifdef LQ_TIMING
  int gen;           // development aid: which of the four generations of time stamps this launch writes
#endif

  __device__ __forceinline__ uint8_t *head(size_t bh) const { return heads + bh * (size_t)head_bytes(r); }
  __device__ __forceinline__ int8_t *codes(size_t bh) const { return reinterpret_cast<int8_t *>(head(bh) + HB_CODES); }
  __device__ __forceinline__ float *col_scale(size_t bh) const { return reinterpret_cast<float *>(head(bh) + HB_COL_SCALE); }
  __device__ __forceinline__ float *row_smooth(size_t bh) const { return reinterpret_cast<float *>(head(bh) + HB_ROW_SMOOTH); }
  __device__ __forceinline__ uint16_t *comp_k(size_t bh) const { return reinterpret_cast<uint16_t *>(head(bh) + HB_COMP_K); }
  __device__ __forceinline__ uint16_t *comp_u(size_t bh) const { return reinterpret_cast<uint16_t *>(head(bh) + hb_comp_u(r)); }
  // row of record j of head bh; `diag` selects the row length, T the element type (float, or __half with rec16)
  template <typename T>
  __device__ __forceinline__ T *record(size_t bh, int j, bool diag) const {
    return static_cast<T *>(records) + (bh * W + j) * (size_t)record_floats(diag);
  }
};

__device__ __forceinline__ float bf16_bits(uint16_t h) { return __uint_as_float(static_cast<uint32_t>(h) << 16); }
__device__ __forceinline__ float f16_bits(uint16_t h) { return __half2float(__ushort_as_half(h)); }
// binary32 -> binary16 bits, nearest even, clamped to the finite range first
__device__ __forceinline__ uint16_t to_f16_bits_sat(float x) {
  x = fminf(fmaxf(x, -65504.0f), 65504.0f);
  return __half_as_ushort(__float2half_rn(x));
}
// binary32 -> bfloat16 bits, nearest even (finite inputs)
__device__ __forceinline__ uint16_t to_bf16_bits(float x) {
  uint32_t u = __float_as_uint(x);
  u += 0x7FFFu + ((u >> 16) & 1u);
  return static_cast<uint16_t>(u >> 16);
}

// L2 eviction priorities: lines that will not be read again soon / lines another kernel reads next
__device__ __forceinline__ uint64_t l2_stream_policy() {
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(policy));
  return policy;
}
__device__ __forceinline__ uint64_t l2_keep_policy() {
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;\n" : "=l"(policy));
  return policy;
}
// ---- mbarrier / TMA bulk copy (1-D) ----
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_inval(uint32_t bar) { asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(bar) : "memory"); }
// The arrival that announces the bytes of the next copies.  Relaxed: nothing this thread wrote has to be
// visible to anybody through this barrier (the copies' own completion is what the waiters acquire), and the
// default release form stalls the warp for about 800 cycles here.
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.relaxed.cta.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
// global -> shared bulk copy; addresses and size are multiples of 16 bytes
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// The same with an L2 eviction priority for the lines the copy brings in.
__device__ __forceinline__ void bulk_g2s_hint(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;\n" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(policy)
      : "memory");
}
// shared -> global bulk copy of the issuing thread's bulk group; addresses and size are multiples of 16 bytes
__device__ __forceinline__ void bulk_s2g(void *dst, uint32_t src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
// Ask the L2 for a piece of global memory (no data comes back, nothing waits for it).
__device__ __forceinline__ void bulk_prefetch_l2(const void *src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(src), "r"(bytes) : "memory");
}
// Bounded wait for phase `parity`; false if the limit of LIMIT polls ran out (the caller then reports and bails out).
template <int LIMIT = (1 << 20)>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
#pragma unroll 1                             // (unrolled, the waits were a fifth of the decode kernel's code)
  for (int spin = 0; spin < LIMIT; spin++) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Set when a bounded wait gave up (bit 0: a wait for bulk copies; bit 3: the wait of lq_selftest_bounded_wait).  Never cleared
// by kernels: lq_clear_device_flags.
__device__ int g_device_error = 0;

// ---- sum of sixteen block results held by sixteen neighbouring lanes (tree levels 1, 2, 4, 8) ----
__device__ __forceinline__ float tree16(float x) {
  x = x + __shfl_xor_sync(FULL, x, 1);
  x = x + __shfl_xor_sync(FULL, x, 2);
  x = x + __shfl_xor_sync(FULL, x, 4);
  x = x + __shfl_xor_sync(FULL, x, 8);
  return x;
}

__device__ __forceinline__ float2 pair(float x) { return make_float2(x, x); }

// Block result of eight products a[e]*b[e] given as four pairs: the .x components are the even-numbered
// terms, the .y components the odd-numbered ones; each chain runs left to right, then the two are added.
__device__ __forceinline__ float block8(const float2 (&a)[4], const float2 (&b)[4]) {
  float2 acc = __fmul2_rn(a[0], b[0]);
#pragma unroll
  for (int c = 1; c < 4; c++) acc = __ffma2_rn(a[c], b[c], acc);
  return acc.x + acc.y;
}

__device__ __forceinline__ void load8p(const float *src, float2 (&x)[4]) {
  const float4 lo = *reinterpret_cast<const float4 *>(src), hi = *reinterpret_cast<const float4 *>(src + 4);
  x[0] = make_float2(lo.x, lo.y); x[1] = make_float2(lo.z, lo.w);
  x[2] = make_float2(hi.x, hi.y); x[3] = make_float2(hi.z, hi.w);
}
__device__ __forceinline__ void store8p(float *dst, const float2 (&x)[4]) {
  *reinterpret_cast<float4 *>(dst) = make_float4(x[0].x, x[0].y, x[1].x, x[1].y);
  *reinterpret_cast<float4 *>(dst + 4) = make_float4(x[2].x, x[2].y, x[3].x, x[3].y);
}

// Dot product of two 128-vectors in shared memory, computed by sixteen neighbouring lanes
// (lane c = lane & 15 owns block c); every one of the sixteen lanes returns the sum.
__device__ __forceinline__ float dot128_shared(const float *a, const float *b, int c) {
  float2 a2[4], b2[4];
  load8p(a + 8 * c, a2);
  load8p(b + 8 * c, b2);
  return tree16(block8(a2, b2));
}

// Programmatic dependent launch: a kernel launched with the stream-serialization attribute may become resident
// before the kernel ahead of it has finished; this is where it waits for that kernel's completion and writes
// (a no-op for an ordinary launch).
// When the dependents may start: allowed at the very beginning, their CTAs come up one by one wherever room appears, so that
// the few with work to do share an SM and the decode CTAs fill the gaps that boundary CTAs of another size leave.  With little
// work (fewer boundaries than boundary CTAs, Params.overlap == 0) they start when the kernel ahead has ended, evenly over the
// SMs: step at 32 x 32 heads 24.5 -> 19.0 us, 77 x 12 heads (W = 13) 22.0 -> 17.6 us.  With more, when every CTA has come to
// its last head, which hides their start: 256 x 32 heads 64.7 us at the beginning or the end, 63.9 us at the last head.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependents_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Phase timing (development aid, compiled in with -DLQ_TIMING only): clock cycles per phase of the decode
// warps, summed over all heads by lane 0 of each warp (slots 0..15: stream warp, 16..31: dot warp; 32..: thread 0 of the boundary kernel's CTAs).
#ifdef LQ_TIMING
__device__ unsigned long long g_phase_cycles[64];
// cycles are summed in registers and flushed once per warp at the end of the kernel, so that the probe
// itself puts no traffic on the memory system while the kernel runs
// (-DLQ_STAMPS_ONLY: the per-CTA time stamps below without the per-phase counters, which cost ≈ 10 % of the time)
#ifdef LQ_STAMPS_ONLY
#define LQ_TICK(slot) do { } while (0)
#else
#define LQ_TICK(slot)                                     \
  do {                                                    \
    const long long now_ = clock64();                     \
    acc_[slot] += static_cast<unsigned>(now_ - tick_);    \
    tick_ = now_;                                         \
  } while (0)
#endif
// the boundary kernel's variant: thread 0 of the CTA keeps its sums in shared memory
__shared__ unsigned lq_bacc[16];
__shared__ long long lq_btick;
#ifdef LQ_STAMPS_ONLY
#define LQ_BTICK(slot) do { } while (0)
#else
#define LQ_BTICK(slot)                                          \
  do {                                                          \
    if (threadIdx.x == 0) {                                     \
      const long long now_ = clock64();                         \
      lq_bacc[slot] += static_cast<unsigned>(now_ - lq_btick);  \
      lq_btick = now_;                                          \
    }                                                           \
  } while (0)
#endif
// time stamps (ns, the GPU's global timer) of thread 0 of every CTA: [generation][kernel][stamp][CTA]
__device__ unsigned long long g_timeline[4][2][6][1024];
#define LQ_STAMP(kernel, slot)                                                                   \
  do {                                                                                           \
    if (threadIdx.x == 0 && blockIdx.x < 1024) {                                                 \
      unsigned long long t_;                                                                     \
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t_));                                      \
      g_timeline[p.gen & 3][kernel][slot][blockIdx.x] = t_;                                      \
    }                                                                                            \
  } while (0)
#else
#define LQ_TICK(slot) do { } while (0)
#define LQ_BTICK(slot) do { } while (0)
#define LQ_STAMP(kernel, slot) do { } while (0)
#endif

// =====================================================================================
// 8x8 register tiles: a CTA of 256 threads holds one 128x128 state, thread (ty, tx) owning rows
// 8ty..8ty+7 and columns 8tx..8tx+7, with tx = lane & 15 and ty = 2*warp + (lane >> 4).
// =====================================================================================
struct Tile {
  int tid, lane, warp, tx, ty;
  __device__ __forceinline__ Tile() {
    tid = threadIdx.x; lane = tid & 31; warp = tid >> 5; tx = lane & 15; ty = tid >> 4;
  }
};

__device__ __forceinline__ void load8(const float *src, float (&x)[8]) {
  const float4 lo = *reinterpret_cast<const float4 *>(src), hi = *reinterpret_cast<const float4 *>(src + 4);
  x[0] = lo.x; x[1] = lo.y; x[2] = lo.z; x[3] = lo.w; x[4] = hi.x; x[5] = hi.y; x[6] = hi.z; x[7] = hi.w;
}
__device__ __forceinline__ void store8(float *dst, const float (&x)[8]) {
  *reinterpret_cast<float4 *>(dst) = make_float4(x[0], x[1], x[2], x[3]);
  *reinterpret_cast<float4 *>(dst + 4) = make_float4(x[4], x[5], x[6], x[7]);
}

// ---- record rows kept in fp16: the same accessors on __half rows (widening is exact; narrowing saturates to
// the finite range and rounds to nearest even, like the compensators) ----
__device__ __forceinline__ void load8p(const __half *src, float2 (&x)[4]) {
  const uint4 raw = *reinterpret_cast<const uint4 *>(src);
  const __half2 *h = reinterpret_cast<const __half2 *>(&raw);
#pragma unroll
  for (int i = 0; i < 4; i++) x[i] = __half22float2(h[i]);
}
__device__ __forceinline__ void load8(const __half *src, float (&x)[8]) {
  float2 v[4];
  load8p(src, v);
#pragma unroll
  for (int i = 0; i < 4; i++) { x[2 * i] = v[i].x; x[2 * i + 1] = v[i].y; }
}
__device__ __forceinline__ float4 load4(const float *src) { return *reinterpret_cast<const float4 *>(src); }
__device__ __forceinline__ float4 load4(const __half *src) {
  const uint2 raw = *reinterpret_cast<const uint2 *>(src);
  const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&raw.x));
  const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&raw.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ uint32_t pack2_f16_sat(float a, float b) {
  return (uint32_t)to_f16_bits_sat(a) | ((uint32_t)to_f16_bits_sat(b) << 16);
}
__device__ __forceinline__ void store8p(__half *dst, const float2 (&x)[4]) {
  *reinterpret_cast<uint4 *>(dst) = make_uint4(pack2_f16_sat(x[0].x, x[0].y), pack2_f16_sat(x[1].x, x[1].y),
                                               pack2_f16_sat(x[2].x, x[2].y), pack2_f16_sat(x[3].x, x[3].y));
}
__device__ __forceinline__ void store8(__half *dst, const float (&x)[8]) {
  *reinterpret_cast<uint4 *>(dst) = make_uint4(pack2_f16_sat(x[0], x[1]), pack2_f16_sat(x[2], x[3]),
                                               pack2_f16_sat(x[4], x[5]), pack2_f16_sat(x[6], x[7]));
}
__device__ __forceinline__ void store4(float *dst, float a, float b, float c, float d) {
  *reinterpret_cast<float4 *>(dst) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void store4(__half *dst, float a, float b, float c, float d) {
  *reinterpret_cast<uint2 *>(dst) = make_uint2(pack2_f16_sat(a, b), pack2_f16_sat(c, d));
}

// Column sums.  In: p[b] = this thread's block result for column 8tx+b (block index ty).
// part: 8*128 floats and out: 128 floats of shared memory.  Returns w[b] = full sum of column 8tx+b in
// every thread.  Tree levels: ty^1 inside the warp (lane^16), then warps (0,1)(2,3)(4,5)(6,7), pairs of
// pairs, halves.  Contains two __syncthreads(); `part` and `out` may be rewritten after the CTA's next barrier.
__device__ __forceinline__ void col_tree(const float (&p)[8], float *part, float *out, const Tile &t, float (&w)[8]) {
  const bool up = t.lane & 16;
  {
    float r[4];
#pragma unroll
    for (int e = 0; e < 4; e++) {
      const float keep = up ? p[e + 4] : p[e], send = up ? p[e] : p[e + 4];
      r[e] = keep + __shfl_xor_sync(FULL, send, 16);      // rows 16w..16w+7 with rows 16w+8..16w+15
    }
    *reinterpret_cast<float4 *>(part + t.warp * D + 8 * t.tx + (up ? 4 : 0)) = make_float4(r[0], r[1], r[2], r[3]);
  }
  __syncthreads();
  if (t.tid < D) {
    const float *c = part + t.tid;
    out[t.tid] = ((c[0] + c[D]) + (c[2 * D] + c[3 * D])) + ((c[4 * D] + c[5 * D]) + (c[6 * D] + c[7 * D]));
  }
  __syncthreads();
  load8(out + 8 * t.tx, w);
}

// p[b] = block result over this thread's eight rows of  sum_a M[a][b] * x[a]: rows 0,2,4,6 and rows
// 1,3,5,7 are the two chains of the block.  (Scalar operations: a packed one would need the per-row
// multiplier duplicated into a register pair, and the 64-register tile leaves no room for that.)
__device__ __forceinline__ void col_blocks(const float (&M)[8][8], const float (&x)[8], float (&p)[8]) {
#pragma unroll
  for (int b = 0; b < 8; b++) {
    float even = M[0][b] * x[0], odd = M[1][b] * x[1];
#pragma unroll
    for (int a = 2; a < 8; a += 2) {
      even = fmaf(M[a][b], x[a], even);
      odd = fmaf(M[a + 1][b], x[a + 1], odd);
    }
    p[b] = even + odd;
  }
}
// ---- the heads that are due for a window boundary ----
// Position of the k-th set bit of m (k < popc(m)).
__device__ __forceinline__ int nth_set_bit(uint32_t m, unsigned k) {
  int pos = 0;
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    const unsigned c = __popc(m & ((1u << s) - 1u));
    if (k >= c) { k -= c; m >>= s; pos += s; }
  }
  return pos;
}

// The due heads, in an order of their sequences that every CTA sees alike, belong to CTA i mod gridDim: with the windows of a
// serving batch in no particular order, heads handed out by their own index pile up on some CTAs (256 sequences x 32 heads in
// random order, W = 16: up to five boundaries on one CTA and none on others; a step of 100 us, 73 us with equal shares).
// The CTA lists up to 32 of its heads in one pass over win_pos: due heads number first, first + stride, ..., `todo_bh` and
// `todo_n` the head and its buffered records.  What bounds it is the round trip of the loads, of which a lane has eight in flight,
// and where few are due, the instructions, which a CTA fetches for itself: up to 256 sequences warp 0 does it alone, in one
// trip; more of them take all NW warps of the CTA, 256 NW sequences to a trip, warp w those whose index / 32 is w modulo NW.
// W = 16, eight warps, us per step with one warp at all sizes / as it is: 512 x 2 heads 22.6 / 18.7, 1024 x 8 66.7 / 61.7, 8192 x 1 141 / 66,
// 32768 x 1 644 / 246; with eight warps at all sizes 32 x 32 heads take 18.7 instead of 18.4.
// Called by the `warps` first warps (due_scan_warps).  Returns how many heads are listed.  `lead`: a due sequence among those
// this warp looks at, the same for the warp of this number in every CTA (-1: none).  `counts`: shared memory.  Ends without a
// barrier.
__device__ __forceinline__ bool window_due(const Params &p, int v) { return v == p.W || (p.force && v > 0); }
template <int NW>
__device__ __forceinline__ int due_scan_warps(const Params &p) { return p.batch <= 256 ? 1 : NW; }
template <int NW>
__device__ __forceinline__ int list_due_heads(const Params &p, unsigned first, unsigned stride, int warps, unsigned (*counts)[8],
                                              unsigned *todo_bh, int *todo_n, int &lead) {
  constexpr int U = 8;                       // loads in flight per lane
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, span = 32 * warps;
  const unsigned item = first + lane * stride;
  const unsigned want = item / static_cast<unsigned>(p.heads_v);       // rank of the head's sequence among the due ones
  unsigned base = 0;
  int turn = 0;
  lead = -1;
#pragma unroll 1
  for (int b0 = 0; b0 < p.batch; b0 += span * U, turn ^= 1) {
    const int mine0 = b0 + 32 * warp;
    int v[U];
    uint32_t m[U];
    unsigned c = 0;
#pragma unroll
    for (int u = 0; u < U; u++) v[u] = mine0 + span * u + lane < p.batch ? p.win_pos[mine0 + span * u + lane] & 0xFFFF : 0;
#pragma unroll
    for (int u = 0; u < U; u++) {
      m[u] = __ballot_sync(FULL, window_due(p, v[u]));
      c += __popc(m[u]);
    }
    unsigned at = base;
    if (warps == 1) {
      base += c;
    } else {
      if (lane == 0) counts[turn][warp] = c;
      __syncthreads();                       // (in turn: the counts of the trip before may still be read)
#pragma unroll
      for (int w = 0; w < NW; w++) {
        const unsigned x = counts[turn][w];
        if (w < warp) at += x;
        base += x;
      }
    }
    if (c == 0) continue;
    // the sequence of rank `want`, if it is one of this trip: the word it is in, then the bit; and the first due one
    unsigned left = want - at;               // (unsigned: beyond all words for ranks below `at`)
    uint32_t word = 0;
    int bit0 = 0, lead_word = 0;
    uint32_t lead_bits = 0;
#pragma unroll
    for (int u = 0; u < U; u++) {
      const unsigned cu = __popc(m[u]);
      if (word == 0) {
        if (left < cu) { word = m[u]; bit0 = u; }
        else left -= cu;
      }
      if (lead_bits == 0) { lead_bits = m[u]; lead_word = u; }
    }
    if (word != 0) {
      const int b = mine0 + span * bit0 + nth_set_bit(word, left);
      todo_bh[lane] = static_cast<unsigned>(b) * p.heads_v + (item - want * p.heads_v);
      todo_n[lane] = p.force ? min(p.win_pos[b] & 0xFFFF, p.W) : p.W;
    }
    if (lead < 0) lead = mine0 + span * lead_word + __ffs(lead_bits) - 1;
  }
  return __popc(__ballot_sync(FULL, want < base));
}

// A CTA whose part `w` of win_pos (of `warps` parts, as above) has been seen says so on the upper bits of the entry of a due
// sequence of that part; the last CTA starts the windows of the due sequences of the part afresh (nobody reads these entries any
// more, and the boundaries themselves do not need them).  The other entries are not touched, whatever a caller keeps there: a
// sequence without a request may be parked at any position from W up, 2^31 - 1 or -1 included, with whose upper bits nothing
// could be counted.  One warp calls this.
__device__ __forceinline__ void restart_due_windows(const Params &p, int lead, int w, int warps) {
  constexpr int U = 8;
  const int lane = threadIdx.x & 31, span = 32 * warps;
  if (p.force) {                             // (which also takes the parked ones: count on another one where there is one)
    int ok = p.batch;
    for (int b = 32 * w + lane; b < p.batch; b += span) {
      const int v = p.win_pos[b] & 0xFFFF;
      if (v > 0 && v <= p.W) { ok = b; break; }
    }
    ok = __reduce_min_sync(FULL, ok);
    if (ok < p.batch) lead = ok;
  }
  int old = 0;
  if (lane == 0) old = atomicAdd(p.win_pos + lead, 0x10000);
  old = __shfl_sync(FULL, old, 0);
  if ((old >> 16) != static_cast<int>(gridDim.x) - 1) return;
#pragma unroll 1
  for (int b0 = 32 * w + lane; b0 < p.batch; b0 += span * U) {
    int v[U];
#pragma unroll
    for (int u = 0; u < U; u++) v[u] = b0 + span * u < p.batch ? __ldcg(p.win_pos + b0 + span * u) & 0xFFFF : 0;
#pragma unroll
    for (int u = 0; u < U; u++)
      if (window_due(p, v[u])) p.win_pos[b0 + span * u] = 0;
  }
}

// Last-arrival bookkeeping on win_pos[b]: bits 16.. count the heads of sequence b that are done with
// the value in bits 0..15.  The head that arrives last (all heads_v have read the old value by then)
// stores the new value and thereby clears the counter.  Call from one thread per head, after a
// __syncthreads() that follows the head's last global write.
__device__ __forceinline__ void arrive_and_set(int32_t *win_pos, int b, int heads_v, int new_value) {
  const int old = atomicAdd(win_pos + b, 0x10000);
  if ((old >> 16) == heads_v - 1) win_pos[b] = new_value;
}

}  // namespace lq
