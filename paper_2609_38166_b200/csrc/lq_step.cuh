// A whole decode step of many heads in one launch: tokens and window boundaries side by side on every SM.
//
// The token of a head is bound by memory, a boundary by its own dependent phases and the fp32 pipes; one after the other, as
// two kernels, each leaves idle what the other needs.  Here a persistent CTA per SM has eight warps that take states through
// their boundaries (boundary_head) and up to four pairs of warps that take heads through the token, with the same device
// routines and the same division of the work as in the decode kernel.  A due head is taken through its token by a pair like any
// other; then the shared-memory slot it is in goes over to the eight warps, which read nothing of it from memory again, and ask for
// the slot's next head as soon as they need the slot no longer.
//
// Which sequences are due is known when the kernel starts, so every CTA looks over win_pos once, lists the sequences in an
// order that all CTAs see alike, and has its share of the due heads; its pairs take them up early enough that the eight
// warps have one to go on with.  The last CTA to have looked moves all window positions on.
//
// What bounds it: with a due head to an SM the chain of launch (a CTA fills its SM, so it comes up when the one before has ended),
// look over win_pos, copies, token and boundary: 32 x 32 heads, W = 16, 16.5 us, of which the boundary is 7.9 and the way there 3.4
// from the moment the sequences are listed (18.0 as two launches).  With more, the issue slots, which both sorts of work use half of by
// themselves: together they take about as long as one after the other.  Two things decide how well they go together.  Instructions:
// an SM keeps some 32 KB of them, and a straight line beyond that is fetched at 6 cycles an instruction instead of 3.4, so loops
// stay rolled where the unrolled ones gain little (256 x 32 heads 74 -> 62 us with the waits, the products of the codes and the
// projections rolled).  And a launch brings only the first of a kernel's code along; behind other kernels what lies beyond comes from the L2
// or the memory when it is reached: of a boundary (15.2 K cycles) the phases behind the products with the start vectors then took 14.6 K
// cycles instead of 7.8.  So the boundary's loops over records, start vectors and columns are rolled as well, and one round has an instance
// without the loops over further ones: 32 x 32 heads, W = 16, behind a projection, norms and a softmax 21.0 -> 19.1 us (two launches 18.8),
// in a loop of steps 16.6 -> 16.4.  Registers: a spilled value comes back from the L2, because the slots leave little of the L1; 128 of them
// (four pairs) spill nothing, 96 (six pairs) up to 180 bytes: diagonal gate, 64 x 32 heads, W = 16 24.7 / 29.2 us.
#pragma once
#include "lq_boundary.cuh"
#include "lq_decode.cuh"

namespace lq {

constexpr int STEP_MAX_BATCH = 2048;         // sequences that the boundary's warps look over in one trip
constexpr int STEP_MAX_R = 8;
constexpr int STEP_WARPS = 8, STEP_PAIRS = 4, STEP_THREADS = 32 * STEP_WARPS + 64 * STEP_PAIRS;      // (of 128 registers)
constexpr unsigned NO_ITEM = 0xFFFFFFFFu;
// Due heads that the pairs may be ahead of the boundary's warps, the one at hand included (two: 64 x 32 heads, W = 8, 24.9 us instead
// of 22.3: one more waits in a slot that could have been used).
constexpr unsigned DUE_AHEAD = 1;

// ---- a pair's slot; byte offsets.  The last of W record rows lies where the digits and sums of the token were whose record it is ----
struct StepSlot {
  static constexpr int mbar = 0;             // barriers: head block, records; projections taken, decays read (diagonal gate); u is there
  static constexpr int words = 48;           // kt^T q of heads in turn; the next item; the pair's next item in turn
  static constexpr int hdr = 64;             // of a due head: its index; the next head of the slot and its records
  static constexpr int pj = 80;              // [2][8] projections of a group of records
  static constexpr int pk = pj + 64, pq = pk + 4 * STEP_MAX_R;                // projections on the compensators
  static constexpr int head = pq + 4 * STEP_MAX_R;
  int digits, rec, bas, per_record, bytes;
  __host__ __device__ StepSlot(int W, int r, bool diag) {
    const int row = 4 * record_floats(diag);
    digits = head + head_bytes(r);           // planes, then the sums, then the record terms: 1 KB each, as a row of the scalar gate
    rec = digits + row;
    bas = rec + row * (W - 1);               // scalar gate: the records' decays, a copy for each warp and one for the boundary
    per_record = (4 * W + 15) / 16 * 16;
    bytes = bas + (diag ? 0 : 3 * per_record);
  }
};
// what the warps of a CTA share
struct StepShared {
  unsigned turn_items, pool;                 // items handed out in turn, and those drawn
  unsigned due_first, due_mine;              // this CTA's first due item, and how many it has (gridDim apart)
  unsigned due_taken, flushed;               // how many of them a pair has taken, and how many are through their boundary
  unsigned handed_over, at;                  // slots handed over; the one that the boundary's warps have
  unsigned last, through;                    // this CTA was the last to look at win_pos; who is done with the scratch words
  unsigned queue[8];                         // slots handed over
  unsigned first[STEP_PAIRS][2];             // the pairs' first two items
};
template <typename T>
__device__ __forceinline__ T now(const T *x) { return *reinterpret_cast<const volatile T *>(x); }

// Heads are items: those of sequences without a boundary first, then the due ones.
struct StepList {
  const uint16_t *seq;                       // sequences by rank
  const uint8_t *fill;                       // and how many records each holds
  __device__ __forceinline__ HeadIdx locate(unsigned item, unsigned Hv, int &n) const {
    const unsigned rank = item / Hv;
    HeadIdx h;
    h.hv = item - rank * Hv;
    h.b = seq[rank];
    h.bh = h.b * Hv + h.hv;
    n = fill[rank];
    return h;
  }
};
__device__ __forceinline__ void step_wait(uint32_t bar, uint32_t &par) {
  if (!mbar_wait(bar, par) && (threadIdx.x & 31) == 0) atomicOr(&g_device_error, 1);
  par ^= 1u;
  __syncwarp();
}
// (one lane) bring a head block, or the n records of a head, into a slot
__device__ __forceinline__ void step_request_head(const Params &p, const StepSlot &L, uint32_t slot, unsigned bh) {
  const uint32_t bytes = L.digits - StepSlot::head;
  mbar_expect_tx(slot + StepSlot::mbar, bytes);
  bulk_g2s_hint(slot + StepSlot::head, p.heads + bh * (size_t)bytes, bytes, slot + StepSlot::mbar, l2_stream_policy());
}
// The last row of a full window goes where the token's sums are: `last_row` is false as long as those are in use, and
// step_request_last_row follows.
template <bool DIAG>
__device__ __forceinline__ void step_request_last_row(const Params &p, const StepSlot &L, uint32_t slot, unsigned bh) {
  bulk_g2s_hint(slot + L.digits, p.record<float>(bh, p.W - 1, DIAG), sizeof(float) * record_floats(DIAG), slot + StepSlot::mbar + 8, l2_stream_policy());
}
template <bool DIAG>
__device__ __forceinline__ void step_request_records(const Params &p, const StepSlot &L, uint32_t slot, unsigned bh, int n, bool last_row) {
  constexpr uint32_t row = sizeof(float) * record_floats(DIAG);
  const int rows = n < p.W ? n : p.W - 1;
  const uint32_t bar = slot + StepSlot::mbar + 8;
  mbar_expect_tx(bar, row * n);              // with no records the phase completes at once
  if (rows > 0) bulk_g2s_hint(slot + L.rec, p.record<float>(bh, 0, DIAG), row * rows, bar, l2_stream_policy());
  if (n == p.W && last_row) step_request_last_row<DIAG>(p, L, slot, bh);
}
// Gamma_{1:l} of the scalar gate, the chain of decays from the newest record back
__device__ __forceinline__ float step_decay_chain(float alpha, const float *bas, int n) {
  float g = alpha;
#pragma unroll 4
  for (int j = n - 1; j >= 0; j--) g = g * bas[j];
  return g;
}

// ---- stream warp of a pair.  Named barriers: B1 dot -> stream, "the record terms and the next item are there"; B1 + 1 stream -> dot,
// "its sums are out of y" ----
template <int GATE>
__device__ __forceinline__ void step_stream(const Params &p, unsigned char *slot, const StepList q, unsigned item, unsigned item1,
                                            const int B1, const int lane) {
  constexpr bool DIAG = GATE == LQ_GATE_DIAG;
  constexpr int RF = record_floats(DIAG);
  const int W = p.W, r = p.r, c = lane & 15, group = p.heads_v / p.heads_qk;
  const unsigned Hv = p.heads_v;
  const StepSlot L(W, r, DIAG);
  const uint32_t slot_a = smem_addr(slot);
  const uint8_t *block = slot + StepSlot::head;
  int8_t *digits = reinterpret_cast<int8_t *>(slot + L.digits);
  float *y = reinterpret_cast<float *>(slot + L.digits);
  const float *pk = reinterpret_cast<const float *>(slot + StepSlot::pk), *pq = reinterpret_cast<const float *>(slot + StepSlot::pq);
  const float *words = reinterpret_cast<const float *>(slot + StepSlot::words);
  float *bas = reinterpret_cast<float *>(slot + L.bas);
  uint32_t par_head = 0, par_rec = 0, par_comp = 0;
  unsigned bh;
  int n, odd = 0;
  TokenRaw nxt;
  nxt.ba_lo = nxt.ba_hi = 1.0f;
  nxt.alpha = 0;
  {
    const HeadIdx h = q.locate(item, Hv, n);
    bh = h.bh;
    load_token<GATE, true>(p, h, group, lane, 0, nxt);
    if (lane == 0) step_request_head(p, L, slot_a, bh);
  }
  for (;;) {
    float k8[8], q8[8], gam[8];
    widen8_bf16(nxt.k, k8);
    widen8_bf16(nxt.q, q8);
    const uint2 v_raw = nxt.v;
    float gsc = 0.0f;
    if (DIAG) {
      widen8_bf16(nxt.a, gam);
    } else {
      gsc = bf16_bits(nxt.alpha);
      if (lane < W) bas[lane] = nxt.ba_lo;
      if (lane + 32 < W) bas[lane + 32] = nxt.ba_hi;
    }
    unsigned bh1 = NO_ITEM;
    int n1 = 0;
    if (item1 != NO_ITEM) {
      const HeadIdx h = q.locate(item1, Hv, n1);
      bh1 = h.bh;
      load_token<GATE, true>(p, h, group, lane, 0, nxt);
    }
    if (n < W) {
      if (DIAG) {
        step_wait(slot_a + StepSlot::mbar + 8, par_rec);
        const float *rec = reinterpret_cast<const float *>(slot + L.rec) + REC_A + 8 * c;
#pragma unroll 2
        for (int j = n - 1; j >= 0; j--) {
          float aj[8];
          load8(rec + j * RF, aj);
#pragma unroll
          for (int e = 0; e < 8; e++) gam[e] = gam[e] * aj[e];
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(slot_a + StepSlot::mbar + 24);             // this warp is done with the records
      } else {
        __syncwarp();
        gsc = step_decay_chain(gsc, bas, n);
#pragma unroll
        for (int e = 0; e < 8; e++) gam[e] = gsc;
      }
      step_wait(slot_a + StepSlot::mbar, par_head);
      float back_k, back_q;
      digit_planes(reinterpret_cast<const float *>(block + HB_ROW_SMOOTH), gam, k8, q8, digits, lane, back_k, back_q);
      __syncwarp();
      code_sums<4>(reinterpret_cast<const int8_t *>(block + HB_CODES), digits, y, lane);
      __syncwarp();
      float rk[4], rq[4];
      {
        const float4 yk4 = *reinterpret_cast<const float4 *>(y + 4 * lane);
        const float4 yq4 = *reinterpret_cast<const float4 *>(y + D + 4 * lane);
        const float4 s4 = *reinterpret_cast<const float4 *>(block + HB_COL_SCALE + 16 * lane);   // code steps B_j / 127
        rk[0] = s4.x * (yk4.x * back_k); rk[1] = s4.y * (yk4.y * back_k); rk[2] = s4.z * (yk4.z * back_k); rk[3] = s4.w * (yk4.w * back_k);
        rq[0] = s4.x * (yq4.x * back_q); rq[1] = s4.y * (yq4.y * back_q); rq[2] = s4.z * (yq4.z * back_q); rq[3] = s4.w * (yq4.w * back_q);
      }
      named_arrive(B1 + 1);                  // y has been read: the dot warp may put the record terms there
      step_wait(slot_a + StepSlot::mbar + 16, par_comp);                      // the compensator projections are complete
      const uint8_t *cu = block + hb_comp_u(r) + 8 * lane;
#pragma unroll 2
      for (int h = 0; h < r; h++) {
        const uint2 w = *reinterpret_cast<const uint2 *>(cu + 2 * D * h);
        const float2 f01 = __half22float2(*reinterpret_cast<const __half2 *>(&w.x));
        const float2 f23 = __half22float2(*reinterpret_cast<const __half2 *>(&w.y));
        const float uc[4] = {f01.x, f01.y, f23.x, f23.y};
        const float pkh = pk[h], pqh = pq[h];
#pragma unroll
        for (int e = 0; e < 4; e++) { rk[e] = fmaf(uc[e], pkh, rk[e]); rq[e] = fmaf(uc[e], pqh, rq[e]); }
      }
      __syncwarp();
      // nobody reads the head block any more: the slot's next one may land (a due head's slot goes over to the boundary)
      if (lane == 0 && n < W - 1 && bh1 != NO_ITEM) step_request_head(p, L, slot_a, bh1);
      named_wait(B1);
      const float4 tk = *reinterpret_cast<const float4 *>(y + 4 * lane);
      const float4 tq = *reinterpret_cast<const float4 *>(y + D + 4 * lane);
      rk[0] = rk[0] + tk.x; rk[1] = rk[1] + tk.y; rk[2] = rk[2] + tk.z; rk[3] = rk[3] + tk.w;
      rq[0] = rq[0] + tq.x; rq[1] = rq[1] + tq.y; rq[2] = rq[2] + tq.z; rq[3] = rq[3] + tq.w;
      const float ktq = words[odd];
      odd ^= 1;
      const float v4[4] = {__uint_as_float(v_raw.x << 16), __uint_as_float(v_raw.x & 0xFFFF0000u),
                           __uint_as_float(v_raw.y << 16), __uint_as_float(v_raw.y & 0xFFFF0000u)};
      float u[4], o[4];
#pragma unroll
      for (int e = 0; e < 4; e++) { u[e] = p.delta ? v4[e] - rk[e] : v4[e]; o[e] = fmaf(u[e], ktq, rq[e]); }
      *reinterpret_cast<float4 *>(p.o + bh * (size_t)D + 4 * lane) = make_float4(o[0], o[1], o[2], o[3]);
      store4(p.record<float>(bh, n, DIAG) + REC_U + 4 * lane, u[0], u[1], u[2], u[3]);
      if (n == W - 1) {                      // the new record joins the others, as it is stored
        __syncwarp();                        // (the record terms, in the same place, have been read)
        store4(reinterpret_cast<float *>(slot + L.digits) + REC_U + 4 * lane, u[0], u[1], u[2], u[3]);
        __syncwarp();
        if (lane == 0) mbar_arrive(slot_a + StepSlot::mbar + 32);
      } else if (n1 == W) {                  // (the record terms have been read: see step_request_last_row)
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) step_request_last_row<DIAG>(p, L, slot_a, bh1);
      }
    } else {                                 // a window that came in full: no token, on to its boundary
      named_arrive(B1 + 1);
      if (DIAG) step_wait(slot_a + StepSlot::mbar + 8, par_rec);
      step_wait(slot_a + StepSlot::mbar, par_head);
      named_wait(B1);
      if (lane == 0) mbar_arrive(slot_a + StepSlot::mbar + 32);
    }
    const unsigned item2 = now(reinterpret_cast<const unsigned *>(words + 2));
    if (item1 == NO_ITEM) return;
    bh = bh1; n = n1; item1 = item2;
  }
}

// ---- dot warp of a pair: projections and the records' terms, the key side of the new record; it looks for the heads to come, and
// hands a due head's slot over to the boundary's warps ----
template <int GATE>
__device__ __forceinline__ void step_dot(const Params &p, unsigned char *slot, const StepList q, StepShared *sh, unsigned item,
                                         unsigned item1, const int pair_no, const unsigned stride, const uint32_t handed, const int B1,
                                         const int lane) {
  constexpr bool DIAG = GATE == LQ_GATE_DIAG;
  const int W = p.W, r = p.r, c = lane & 15, half = lane >> 4, group = p.heads_v / p.heads_qk;
  const unsigned Hv = p.heads_v;
  const StepSlot L(W, r, DIAG);
  const uint32_t slot_a = smem_addr(slot);
  const uint8_t *block = slot + StepSlot::head;
  const float *rec = reinterpret_cast<const float *>(slot + L.rec);
  float *y = reinterpret_cast<float *>(slot + L.digits), *pj = reinterpret_cast<float *>(slot + StepSlot::pj);
  float *pk = reinterpret_cast<float *>(slot + StepSlot::pk), *pq = reinterpret_cast<float *>(slot + StepSlot::pq);
  unsigned *words = reinterpret_cast<unsigned *>(slot + StepSlot::words);
  float *bas = reinterpret_cast<float *>(slot + L.bas + L.per_record), *dec = reinterpret_cast<float *>(slot + L.bas + 2 * L.per_record);
  uint32_t par_head = 0, par_rec = 0, par_walk = 0, par_u = 0;
  unsigned bh;
  int n, odd = 0;
  TokenRaw nxt;
  nxt.ba_lo = nxt.ba_hi = 1.0f;
  nxt.beta = nxt.alpha = 0;
  {
    const HeadIdx h = q.locate(item, Hv, n);
    bh = h.bh;
    load_token<GATE, true>(p, h, group, lane, 1, nxt);
    if (lane == 0) step_request_records<DIAG>(p, L, slot_a, bh, n, true);
  }
  bool looking = item1 != NO_ITEM;           // there may be more heads than those at hand
  for (;;) {
    // (lane 0) the head after the next one: a due one if the boundary's warps will soon have none before them, else one in turn, else
    // a drawn one; when there are none of those, a due one
    unsigned pick = NO_ITEM, ticket = NO_ITEM;
    if (looking && lane == 0) {
      const unsigned d = now(&sh->due_taken);
      if (d < sh->due_mine && d < now(&sh->flushed) + DUE_AHEAD && atomicCAS(&sh->due_taken, d, d + 1) == d) {
        pick = sh->due_first + d * gridDim.x;
      } else if (words[3] < sh->turn_items) {
        pick = words[3];
        words[3] = pick + stride;
      } else if (sh->pool > 0) {
        ticket = static_cast<unsigned>(atomicAdd(p.work, 1));
      }
    }
    auto settle = [&]() {
      if (lane == 0) {
        if (looking && pick == NO_ITEM) {
          if (ticket < sh->pool) {
            pick = sh->turn_items + ticket;
          } else {
            const unsigned d = atomicAdd(&sh->due_taken, 1u);
            if (d < sh->due_mine) pick = sh->due_first + d * gridDim.x;
          }
        }
        words[2] = pick;
      }
    };
    float2 k2[4], q2[4], g2[4], kt2[4];
    widen8_bf16(nxt.k, k2);
    widen8_bf16(nxt.q, q2);
    const float beta = bf16_bits(nxt.beta), alpha_s = DIAG ? 0.0f : bf16_bits(nxt.alpha);
    const uint4 a_raw = nxt.a;
    if (DIAG) {
      widen8_bf16(nxt.a, g2);
    } else {
      if (lane < W) bas[lane] = nxt.ba_lo;
      if (lane + 32 < W) bas[lane + 32] = nxt.ba_hi;
      __syncwarp();
    }
#pragma unroll
    for (int e = 0; e < 4; e++) kt2[e] = __fmul2_rn(pair(beta), k2[e]);
    unsigned bh1 = NO_ITEM;
    int n1 = 0;
    if (item1 != NO_ITEM) {
      const HeadIdx h = q.locate(item1, Hv, n1);
      bh1 = h.bh;
      load_token<GATE, true>(p, h, group, lane, 1, nxt);
    }
    const bool due = n >= W - 1;
    if (n < W) {
      {
        const float ktq = tree16(block8(kt2, q2));
        if (lane == 0) reinterpret_cast<float *>(words)[odd] = ktq;
        odd ^= 1;
      }
      step_wait(slot_a + StepSlot::mbar + 8, par_rec);
      float2 rk_rec[2] = {{0.0f, 0.0f}, {0.0f, 0.0f}}, rq_rec[2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
      float g1 = alpha_s;
      walk_records<GATE>(rec, 0, bas, pj, n - 1, lane, k2, q2, g2, g1, rk_rec, rq_rec);
      step_wait(slot_a + StepSlot::mbar, par_head);
      if (r > 0) {
        if (!DIAG) {
#pragma unroll
          for (int e = 0; e < 4; e++) g2[e] = pair(g1);       // (Gamma_{1:l}: the walk has come past record 0)
        }
        project_compensators(reinterpret_cast<const uint16_t *>(block + HB_COMP_K), r, g2, k2, q2, pk, pq, lane);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(slot_a + StepSlot::mbar + 16);
      if (DIAG) step_wait(slot_a + StepSlot::mbar + 24, par_walk);           // the stream warp read the records' decays too
      if (lane == 0 && !due && bh1 != NO_ITEM) step_request_records<DIAG>(p, L, slot_a, bh1, n1, false);
      named_wait(B1 + 1);                    // the stream warp has taken its sums out of y
      *reinterpret_cast<float4 *>(y + 4 * lane) = make_float4(rk_rec[0].x, rk_rec[0].y, rk_rec[1].x, rk_rec[1].y);
      *reinterpret_cast<float4 *>(y + D + 4 * lane) = make_float4(rq_rec[0].x, rq_rec[0].y, rq_rec[1].x, rq_rec[1].y);
      settle();
      __syncwarp();
      named_arrive(B1);                      // the record terms are there, and the item
      float *row = p.record<float>(bh, n, DIAG);
      if (half == 0) {
        store8p(row + REC_KT + 8 * c, kt2);
        if (DIAG) {
          float a8[8];
          widen8_bf16(a_raw, a8);
          store8(row + REC_A + 8 * c, a8);
        } else if (lane == 0) {
          p.decays[bh * (size_t)W + n] = alpha_s;
        }
      }
    } else {                                 // a window that came in full
      named_wait(B1 + 1);
      step_wait(slot_a + StepSlot::mbar + 8, par_rec);
      step_wait(slot_a + StepSlot::mbar, par_head);
      settle();
      __syncwarp();
      named_arrive(B1);
    }
    if (due) {
      // the slot goes over to the boundary's warps when u is in the new record's row, which gets its key side, and with the decays
      step_wait(slot_a + StepSlot::mbar + 32, par_u);
      if (n < W && half == 0) {
        float *row = reinterpret_cast<float *>(slot + L.digits);
        store8p(row + REC_KT + 8 * c, kt2);
        if (DIAG) {
          float a8[8];
          widen8_bf16(a_raw, a8);
          store8(row + REC_A + 8 * c, a8);
        }
      }
      if (!DIAG) {
        if (lane < W) dec[lane] = lane < n ? bas[lane] : alpha_s;
        if (lane + 32 < W) dec[lane + 32] = lane + 32 < n ? bas[lane + 32] : alpha_s;
      }
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");          // (written to; a bulk copy lands there next)
      __syncwarp();
      if (lane == 0) {
        unsigned *hdr = reinterpret_cast<unsigned *>(slot + StepSlot::hdr);
        hdr[0] = bh; hdr[1] = bh1; hdr[2] = n1;
        const unsigned k = atomicAdd(&sh->handed_over, 1u);
        sh->queue[k & 7] = pair_no;
        mbar_arrive(handed + 8 * (k & 7));
      }
    }
    const unsigned item2 = __shfl_sync(FULL, pick, 0);
    if (item1 == NO_ITEM) return;
    looking = item2 != NO_ITEM;
    bh = bh1; n = n1; item1 = item2;
  }
}

// Shared memory, byte offsets.  gam is free when Gamma has been applied, a warp's value sides when they have been taken off the
// state: 1 / c and 1 / code step take their places.
template <int RM>
struct StepSmem {
  static constexpr int handed = 0;                           // [8] barriers of the queue of slots handed over
  static constexpr int gam = 64;                             // [128] Gamma_{1:n}, later 1 / c
  static constexpr int gram = gam + 4 * D;
  static constexpr int chol = gram + 4 * RM * RM;
  static constexpr int ub = chol + (RM > 4 ? 4 * (RM * RM + 2 * RM) : 0);      // [8][RM][16]
  static constexpr int invc = ub;                            // [8][16], a warp's in the place of its value sides
  static constexpr int T = ub + (RM > 0 ? 4 * D * RM : 4 * D);
  static constexpr int abs_part = T + 4 * D * RM;            // [8][128]
  static constexpr int Wv = abs_part + 4 * D * 8;            // [r][128] several rounds: S^T q_h
  int seq, fill, slots, slot_bytes, bytes;
  __host__ __device__ StepSmem(int pairs, int batch, int W, int r, bool diag, bool iterate) {
    slot_bytes = StepSlot(W, r, diag).bytes;
    seq = Wv + (iterate ? 4 * D * r : 0);
    fill = seq + (2 * batch + 15) / 16 * 16;
    slots = fill + (batch + 15) / 16 * 16;
    bytes = slots + pairs * slot_bytes;
  }
};

template <int GATE, int RM, bool EXACT, bool ROUNDS>
__global__ void __launch_bounds__(STEP_THREADS, 1) step_kernel(const Params p, const int pairs) {
  constexpr int NW = STEP_WARPS, NT = 32 * NW, U = STEP_MAX_BATCH / NT;
  constexpr bool DIAG = GATE == LQ_GATE_DIAG;
  using Lay = StepSmem<RM>;
  extern __shared__ __align__(128) unsigned char lq_stp[];
  __shared__ StepShared sh;
  __shared__ unsigned counts[NW * U];
  static_assert(NW * U == 64, "two to a lane");
  const int W = p.W, r = EXACT ? RM : RM > 0 ? p.r : 0, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (RM > 0 && r < 1) return;               // (not launched)
  const Lay L(pairs, p.batch, W, p.r, DIAG, RM > 0 && p.n_iter > 1);
  const StepSlot SL(W, p.r, DIAG);
  const unsigned Hv = p.heads_v;
  uint16_t *seq = reinterpret_cast<uint16_t *>(lq_stp + L.seq);
  uint8_t *fill = lq_stp + L.fill;
  const uint32_t handed = smem_addr(lq_stp + Lay::handed);
  if (tid < 8) mbar_init(handed + 8 * tid, 1);
  if (tid >= 32 && tid < 32 + pairs) {
    const uint32_t bar = smem_addr(lq_stp + L.slots + (tid - 32) * L.slot_bytes + StepSlot::mbar);
    for (int e = 0; e < 5; e++) mbar_init(bar + 8 * e, 1);
  }
  if (tid == 0) sh.flushed = sh.handed_over = sh.through = 0;
  __syncthreads();
  grid_dependency_wait();                    // no data in global memory is read or written above this line
  grid_dependents_may_start();               // (their CTAs find no room before these are through)

  // ---- which sequences get a token and no boundary (fill below W - 1), and which are due (W - 1, or W: no token); the others are
  // left alone.  Ranks in the order of (trip, warp, lane), so of their index ----
  int v[U];
  if (warp < NW) {
    uint32_t mn[U], md[U];
#pragma unroll
    for (int u = 0; u < U; u++) v[u] = NT * u + tid < p.batch ? p.win_pos[NT * u + tid] & 0xFFFF : 0xFFFF;
#pragma unroll
    for (int u = 0; u < U; u++) {
      mn[u] = __ballot_sync(FULL, v[u] < W - 1);
      md[u] = __ballot_sync(FULL, v[u] == W - 1 || v[u] == W);
      if (lane == 0) counts[NW * u + warp] = __popc(mn[u]) | __popc(md[u]) << 16;
    }
    boundary_sync<true, NW>();
    const unsigned c0 = counts[lane], c1 = counts[lane + 32];
    unsigned s0 = c0, s1 = c1;
#pragma unroll
    for (int e = 1; e < 32; e <<= 1) {
      const unsigned a = __shfl_up_sync(FULL, s0, e), b = __shfl_up_sync(FULL, s1, e);
      if (lane >= e) { s0 += a; s1 += b; }
    }
    s1 += __shfl_sync(FULL, s0, 31);
    const unsigned all = __shfl_sync(FULL, s1, 31), normal = all & 0xFFFF;
    const uint32_t below = (1u << lane) - 1u;
#pragma unroll
    for (int u = 0; u < U; u++) {
      const unsigned at = __shfl_sync(FULL, u < U / 2 ? s0 - c0 : s1 - c1, (NW * u + warp) & 31);
      int rank = -1;
      if (mn[u] >> lane & 1u) rank = (at & 0xFFFF) + __popc(mn[u] & below);
      if (md[u] >> lane & 1u) rank = normal + (at >> 16) + __popc(md[u] & below);
      if (rank >= 0) { seq[rank] = NT * u + tid; fill[rank] = v[u]; }
    }
    // Items: a pair takes those of sequences without a boundary in turn, the last two rounds by tickets (word 0 of the scratch words
    // counts them), as in the decode kernel; a CTA's due heads go to whichever of its pairs looks for one.  The first pair's first
    // head is a due one, and so are those of pairs that find nothing in turn (all windows due: every slot has one to hand over).
    if (warp == 0 && lane < pairs) {
      const unsigned items = normal * Hv, due = (all >> 16) * Hv, G = gridDim.x * pairs, mine = gridDim.x - 1 - blockIdx.x;
      const unsigned rounds = items / G, in_turn = rounds >= 4 ? (rounds - 2) * G : items;
      const unsigned m = mine < due ? (due - mine + gridDim.x - 1) / gridDim.x : 0;
      unsigned turn = lane * gridDim.x + blockIdx.x, taken = 0;
#pragma unroll
      for (int e = 0; e < 2; e++) {
        const bool wants_due = (e == 0 && lane == 0) || turn >= in_turn;
        const unsigned want = __ballot_sync((1u << pairs) - 1u, wants_due), idx = taken + __popc(want & below);
        unsigned it = NO_ITEM;
        if (wants_due && idx < m) it = items + mine + idx * gridDim.x;
        else if (turn < in_turn) { it = turn; turn += G; }
        sh.first[lane][e] = it;
        taken = min(m, taken + __popc(want));
      }
      reinterpret_cast<unsigned *>(lq_stp + L.slots + lane * L.slot_bytes + StepSlot::words)[3] = turn;
      if (lane == 0) {
        sh.turn_items = in_turn; sh.pool = items - in_turn;
        sh.due_first = items + mine; sh.due_mine = m; sh.due_taken = taken;
      }
    }
  }
  __syncthreads();
  // the last CTA that is through with tickets and arrivals puts the scratch words back to zero
  auto done_with_words = [&]() {
    if (atomicAdd(&sh.through, 1u) == static_cast<unsigned>(pairs) && atomicAdd(p.work + 2, 1) == static_cast<int>(gridDim.x) - 1)
      p.work[0] = p.work[1] = p.work[2] = 0;
  };
  if (warp >= NW) {
    // =========================== tokens ===========================
    const int pair_no = (warp - NW) >> 1, B1 = 1 + 2 * pair_no;              // (the boundary's warps have barrier 15)
    if (pair_no >= pairs) return;
    const StepList q{seq, fill};
    unsigned char *slot = lq_stp + L.slots + pair_no * L.slot_bytes;
    const unsigned item = sh.first[pair_no][0], item1 = sh.first[pair_no][1];
    if (((warp - NW) & 1) == 0) {
      if (item != NO_ITEM) step_stream<GATE>(p, slot, q, item, item1, B1, lane);
    } else {
      if (item != NO_ITEM) step_dot<GATE>(p, slot, q, &sh, item, item1, pair_no, gridDim.x * pairs, handed, B1, lane);
      if (lane == 0) done_with_words();
    }
    return;
  }
  // =========================== boundaries ===========================
  if (tid == 0) {
    __threadfence();
    sh.last = atomicAdd(p.work + 1, 1) == static_cast<int>(gridDim.x) - 1;
    done_with_words();
  }
  boundary_sync<true, NW>();
  if (sh.last) {                             // every CTA has looked: all positions move on
#pragma unroll
    for (int u = 0; u < U; u++)
      if (v[u] <= W) p.win_pos[NT * u + tid] = v[u] >= W - 1 ? 0 : v[u] + 1;
  }
  auto at_bytes = [&](int offset) { return reinterpret_cast<float *>(lq_stp + offset); };
  BoundaryArrays A{nullptr, at_bytes(Lay::gam), nullptr, nullptr, at_bytes(Lay::abs_part), at_bytes(Lay::T), at_bytes(Lay::Wv), at_bytes(Lay::gram),
                   at_bytes(Lay::chol), at_bytes(Lay::ub) + warp * 16 * RM, at_bytes(Lay::gam), at_bytes(Lay::invc) + 16 * (RM > 0 ? RM : 1) * warp};
  const unsigned mine = sh.due_mine;
  for (unsigned k = 0; k < mine; k++) {
    if (tid == 0) {
      const bool there = mbar_wait(handed + 8 * (k & 7), (k >> 3) & 1u);
      if (!there) atomicOr(&g_device_error, 1);
      sh.at = there ? sh.queue[k & 7] : NO_ITEM;
    }
    boundary_sync<true, NW>();               // (and the working arrays of the head before have been read)
    const unsigned which = sh.at;
    if (which == NO_ITEM) return;            // (the pairs' waits for their slots run out in turn)
    unsigned char *slot = lq_stp + L.slots + which * L.slot_bytes;
    const unsigned *hdr = reinterpret_cast<const unsigned *>(slot + StepSlot::hdr);
    A.dec = reinterpret_cast<float *>(slot + SL.bas + 2 * SL.per_record);
    A.part = reinterpret_cast<float *>(slot + StepSlot::head);
    A.newest = slot + SL.digits;
    A.rows = slot + SL.rec;
    boundary_head<GATE, 0, false, RM, false, EXACT, ROUNDS, true, 4, NW>(p, A, slot + StepSlot::head, hdr[0], W, r, r, false, [&] {
      const unsigned next = tid == 224 ? hdr[1] : NO_ITEM;
      if (next != NO_ITEM) {                 // the slot's next head
        step_request_head(p, SL, smem_addr(slot), next);
        step_request_records<DIAG>(p, SL, smem_addr(slot), next, static_cast<int>(hdr[2]), true);
      }
    });
    if (tid == 0) *reinterpret_cast<volatile unsigned *>(&sh.flushed) = k + 1;
  }
}

}  // namespace lq
