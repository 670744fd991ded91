// "Per-window BF16" (the -w baseline of Fig. 3 and Table 2): the window algebra of Sec. 3.2 with the boundary
// state kept as the dense state rounded to bfloat16 once per window - no scale, no smoothing, no compensators.
//
// Between boundaries a head is  S_l = Gamma_{1:l} S0 + sum_j Gamma_{j+1:l} kt_j u_j^T  (Eq. 4) with S0 in bfloat16;
// a token reads it with x = alpha (.) k and x = alpha (.) q exactly like the 8-bit path reads Eq. 7, only the
// boundary-state term is the plain binary32 product S0^T (Gamma x) in the fixed summation order.  The head block
// is S0^T, [d_v][d_k] bfloat16: the eight values a lane fetches with one 16-byte load are one block of the sum.
#pragma once
#include "lq_decode.cuh"

namespace lq {


__device__ __forceinline__ uint16_t *bf16w_state(const Params &p, size_t bh) {
  return reinterpret_cast<uint16_t *>(p.heads + bh * (size_t)BF16W_HEAD_BYTES);
}

// ---------------------------------------------------------------------------------------------
// Boundary: persistent CTAs of 256 threads (8x8 register tiles), each striding over the heads and taking those
// that are due.
// MODE 0: S0 <- bf16(Gamma_{1:n} S0 + sum_j Gamma_{j+1:n} kt_j u_j^T) for the sequences that are due (Eq. 4)
// MODE 1: S0 <- bf16(dense fp32 state)          MODE 2: dense fp32 state <- the sum above, nothing else changes
// Dynamic shared memory: bf16w_boundary_smem(...) bytes: the n rows as stored, then kd, u and Gamma in fp32.
// ---------------------------------------------------------------------------------------------
inline size_t bf16w_boundary_smem(int W, bool diag, bool rec16) {
  return (size_t)W * record_floats(diag) * (rec16 ? 2 : 4) + sizeof(float) * (size_t)(2 * W + 1) * D;
}

template <int GATE, int MODE, bool R16>
__device__ __forceinline__ void bf16w_boundary_head(const Params &p, unsigned char *smem, float *dec_s, const Tile &t,
                                                    size_t bh, int n) {
  using rec_t = typename std::conditional<R16, __half, float>::type;
  constexpr bool DIAG = GATE == LQ_GATE_DIAG;
  constexpr int RF = record_floats(DIAG);
  rec_t *raw_s = reinterpret_cast<rec_t *>(smem);
  float *kd_s = reinterpret_cast<float *>(smem + (size_t)p.W * RF * sizeof(rec_t));
  float *bu_s = kd_s + p.W * D, *gam_s = bu_s + p.W * D;
  const int b = static_cast<int>(bh / p.heads_v);
  float M[8][8];
  uint16_t *S0T = bf16w_state(p, bh);
  if (MODE == 1) {
    const float *S = p.S + bh * (size_t)(D * D);
#pragma unroll
    for (int a = 0; a < 8; a++) load8(S + (8 * t.ty + a) * D + 8 * t.tx, M[a]);
  } else {
    {
      constexpr int PER16 = 16 / sizeof(rec_t);
      const rec_t *rows = p.record<rec_t>(bh, 0, DIAG);       // the n rows are one contiguous piece
      for (int e = t.tid; e < n * (RF / PER16); e += 256) cp_async16(raw_s + PER16 * e, rows + PER16 * e);
      cp_async_commit();
    }
    uint4 wv[8];                                              // column 8tx+bcol, rows 8ty..8ty+7
#pragma unroll
    for (int bcol = 0; bcol < 8; bcol++)
      wv[bcol] = *reinterpret_cast<const uint4 *>(S0T + (8 * t.tx + bcol) * D + 8 * t.ty);
    if (!DIAG && t.tid < n) dec_s[t.tid] = p.decays[bh * (size_t)p.W + t.tid];
    cp_async_wait_all();
    __syncthreads();
    // cumulative decays, newest record first (Appendix B.2): kd_j = Gamma_{j+1:n} kt_j, gam = Gamma_{1:n}
    if (t.tid < D) {
      float gam = 1.0f;
      for (int j = n - 1; j >= 0; j--) {
        kd_s[j * D + t.tid] = gam * static_cast<float>(raw_s[j * RF + REC_KT + t.tid]);
        const float dec = DIAG ? static_cast<float>(raw_s[j * RF + REC_A + t.tid]) : dec_s[j];
        gam = gam * dec;
      }
      gam_s[t.tid] = gam;
    } else {
      const int i = t.tid - D;
      for (int j = 0; j < n; j++) bu_s[j * D + i] = static_cast<float>(raw_s[j * RF + REC_U + i]);
    }
#pragma unroll
    for (int bcol = 0; bcol < 8; bcol++) {
      float2 s2[4];
      widen8_bf16(wv[bcol], s2);
#pragma unroll
      for (int e = 0; e < 4; e++) { M[2 * e][bcol] = s2[e].x; M[2 * e + 1][bcol] = s2[e].y; }
    }
    __syncthreads();
    float gi[8];
    load8(gam_s + 8 * t.ty, gi);
#pragma unroll
    for (int a = 0; a < 8; a++)
#pragma unroll
      for (int bcol = 0; bcol < 8; bcol++) M[a][bcol] = gi[a] * M[a][bcol];
    for (int j = 0; j < n; j++) {                             // oldest record first
      float kj[8], uj[8];
      load8(kd_s + j * D + 8 * t.ty, kj);
      load8(bu_s + j * D + 8 * t.tx, uj);
#pragma unroll
      for (int a = 0; a < 8; a++)
#pragma unroll
        for (int bcol = 0; bcol < 8; bcol++) M[a][bcol] = fmaf(kj[a], uj[bcol], M[a][bcol]);
    }
  }
  if (MODE == 2) {
    float *S = p.S + bh * (size_t)(D * D);
#pragma unroll
    for (int a = 0; a < 8; a++) store8(S + (8 * t.ty + a) * D + 8 * t.tx, M[a]);
  } else {
#pragma unroll
    for (int bcol = 0; bcol < 8; bcol++) {
      uint32_t ws[4];
#pragma unroll
      for (int e = 0; e < 4; e++)
        ws[e] = (uint32_t)to_bf16_bits(M[2 * e][bcol]) | ((uint32_t)to_bf16_bits(M[2 * e + 1][bcol]) << 16);
      *reinterpret_cast<uint4 *>(S0T + (8 * t.tx + bcol) * D + 8 * t.ty) = make_uint4(ws[0], ws[1], ws[2], ws[3]);
    }
    if (MODE == 1 && t.tid == 0) p.win_pos[b] = 0;           // nobody reads win_pos in this mode
  }
}

template <int GATE, int MODE, bool R16>
__global__ void __launch_bounds__(256, 2) bf16w_boundary_kernel(const Params p) {
  extern __shared__ float4 lq_bf16w_smem4[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(lq_bf16w_smem4);
  __shared__ unsigned todo_bh[32];
  __shared__ int todo_n[32], todo_count, any_due;
  __shared__ float dec_s[MAX_W];
  const Tile t;
  const unsigned nh = static_cast<unsigned>(p.batch) * p.heads_v;
  grid_dependency_wait();
  // (as in boundary_kernel: the decode kernel ahead counts its tickets there)
  if (MODE == 0 && p.work != nullptr && blockIdx.x == 0 && t.tid == 0) p.work[0] = 0;
  // Warp 0 puts together the next 32 heads of the CTA: of those that are due (find_due_heads), or every gridDim-th head.
  int count = 32;
  for (unsigned first = blockIdx.x; count == 32; first += 32 * gridDim.x) {
    if (t.warp == 0) {
      unsigned bh_mine = first + t.lane * gridDim.x;
      int n_mine = 0, c, due = 0;
      if (MODE == 0) {
        c = find_due_heads(p, first, gridDim.x, t.lane, bh_mine, n_mine, due);
      } else {
        const bool have = bh_mine < nh;
        if (MODE == 2 && have) n_mine = p.win_pos[bh_mine / p.heads_v] & 0xFFFF;
        c = __popc(__ballot_sync(FULL, have));
      }
      todo_bh[t.lane] = bh_mine;
      todo_n[t.lane] = n_mine > p.W ? p.W : n_mine;
      if (t.lane == 0) { todo_count = c; any_due = due; }
    }
    __syncthreads();
    count = todo_count;
    if (MODE == 0 && count < 32 && any_due > 0 && t.warp == 7) restart_due_windows(p, t.lane);
    for (int k = 0; k < count; k++) {
      bf16w_boundary_head<GATE, MODE, R16>(p, smem, dec_s, t, todo_bh[k], todo_n[k]);
      __syncthreads();                       // this head's use of shared memory is over
    }
    __syncthreads();                         // the list is rewritten by the next round
  }
}

}  // namespace lq
