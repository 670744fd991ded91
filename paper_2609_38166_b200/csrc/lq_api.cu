// C boundary of the library: argument checks, launch configuration, and the kernels that wrap the
// device routines of lq_decode.cuh and lq_boundary.cuh.  Declarations and contracts: include/lq.h.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <tuple>

#include "lq_boundary.cuh"
#include "lq_decode.cuh"
#include "lq_step.cuh"

namespace lq {

// ---------------------------------------------------------------------------------------------
// Baseline: Eq. 1 on a dense state that is read and written in full every token.
// ---------------------------------------------------------------------------------------------
template <int GATE, bool BF16>
__global__ void __launch_bounds__(256, (BF16 || GATE == LQ_GATE_SCALAR) ? 3 : 2) ref_kernel(const Params p) {
  __shared__ __align__(16) float kt_s[D], q_s[D], bv_s[D], a_s[D], col_s[D], part_s[8 * D];
  const Tile t;
  const size_t bh = blockIdx.x;
  const int b = static_cast<int>(bh / p.heads_v), hv = static_cast<int>(bh % p.heads_v);
  float M[8][8];
  if (BF16) {
    const uint16_t *S = p.S16 + bh * (size_t)(D * D);
#pragma unroll
    for (int a = 0; a < 8; a++) {
      const uint4 w = __ldcs(reinterpret_cast<const uint4 *>(S + (8 * t.ty + a) * D + 8 * t.tx));   // streamed: read once
      const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int e = 0; e < 4; e++) {
        M[a][2 * e] = __uint_as_float(ws[e] << 16);
        M[a][2 * e + 1] = __uint_as_float(ws[e] & 0xFFFF0000u);
      }
    }
  } else {
    const float *S = p.S + bh * (size_t)(D * D);
#pragma unroll
    for (int a = 0; a < 8; a++) load8(S + (8 * t.ty + a) * D + 8 * t.tx, M[a]);   // (streaming hints slow this one down)
  }
  if (t.tid < D) {
    const int group = p.heads_v / p.heads_qk;
    const size_t qk_off = ((size_t)b * p.heads_qk + hv / group) * D;
    const float k_i = bf16_bits(p.k[qk_off + t.tid]);
    const float a_i = GATE == LQ_GATE_DIAG ? bf16_bits(p.alpha[bh * D + t.tid]) : bf16_bits(p.alpha[bh]);
    kt_s[t.tid] = bf16_bits(p.beta[bh]) * k_i;
    bv_s[t.tid] = a_i * k_i;
    a_s[t.tid] = a_i;
    q_s[t.tid] = bf16_bits(p.q[qk_off + t.tid]);
  }
  __syncthreads();
  float x[8], pc[8], u[8], o[8], kt[8], ai[8];
  load8(bv_s + 8 * t.ty, x);
  col_blocks(M, x, pc);
  col_tree(pc, part_s, col_s, t, u);                           // S^T (alpha.k)
#pragma unroll
  for (int c = 0; c < 8; c++) {                               // b = 0 (no delta rule): nothing is subtracted
    const float vc = bf16_bits(p.v[bh * D + 8 * t.tx + c]);
    u[c] = p.delta ? vc - u[c] : vc;
  }
  load8(kt_s + 8 * t.ty, kt);
  load8(a_s + 8 * t.ty, ai);
#pragma unroll
  for (int a = 0; a < 8; a++)
#pragma unroll
    for (int c = 0; c < 8; c++) M[a][c] = fmaf(kt[a], u[c], ai[a] * M[a][c]);
  load8(q_s + 8 * t.ty, x);
  col_blocks(M, x, pc);
  col_tree(pc, part_s, col_s, t, o);
  if (t.ty == 0) store8(p.o + bh * D + 8 * t.tx, o);
  if (BF16) {
    uint16_t *S = p.S16 + bh * (size_t)(D * D);
#pragma unroll
    for (int a = 0; a < 8; a++) {
      uint32_t ws[4];
#pragma unroll
      for (int e = 0; e < 4; e++)
        ws[e] = (uint32_t)to_bf16_bits(M[a][2 * e]) | ((uint32_t)to_bf16_bits(M[a][2 * e + 1]) << 16);
      __stcs(reinterpret_cast<uint4 *>(S + (8 * t.ty + a) * D + 8 * t.tx), make_uint4(ws[0], ws[1], ws[2], ws[3]));
    }
  } else {
    float *S = p.S + bh * (size_t)(D * D);
#pragma unroll
    for (int a = 0; a < 8; a++) store8(S + (8 * t.ty + a) * D + 8 * t.tx, M[a]);
  }
}

// ---------------------------------------------------------------------------------------------
// The window representation as separate arrays in the paper's orientation <-> the packed layout of lq_state
// (lq_import_state / lq_export_state): pure data movement, one CTA per head.
// ---------------------------------------------------------------------------------------------
template <bool IMPORT>
__global__ void __launch_bounds__(256) convert_state_kernel(const Params p, const lq_state_arrays a, const int diag) {
  __shared__ __align__(16) int8_t tile[D][D + 16];            // the code matrix on its way through the transposition
  const size_t bh = blockIdx.x;
  const int tid = threadIdx.x, W = p.W, r = p.r;
  const int b = static_cast<int>(bh / p.heads_v), hv = static_cast<int>(bh % p.heads_v);
  int8_t *Z = a.codes + bh * (size_t)(D * D);                 // [d_k][d_v]
  int8_t *ZT = p.codes(bh);                                   // [d_v][d_k]
  const int8_t *src = IMPORT ? Z : ZT;
  int8_t *dst = IMPORT ? ZT : Z;
  for (int e = tid; e < D * D / 16; e += 256) {
    const int row = e >> 3, c16 = e & 7;
    *reinterpret_cast<uint4 *>(&tile[row][16 * c16]) = *reinterpret_cast<const uint4 *>(src + row * D + 16 * c16);
  }
  __syncthreads();
  for (int e = tid; e < D * D / 16; e += 256) {
    const int row = e >> 3, c16 = e & 7;
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      uint32_t x = 0;
#pragma unroll
      for (int j = 0; j < 4; j++) x |= static_cast<uint32_t>(static_cast<uint8_t>(tile[16 * c16 + 4 * q + j][row])) << (8 * j);
      w[q] = x;
    }
    *reinterpret_cast<uint4 *>(dst + row * D + 16 * c16) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  auto move = [&](auto *packed, auto *plain) {
    if (IMPORT) *packed = *plain;
    else *plain = *packed;
  };
  if (tid < D) {
    move(p.col_scale(bh) + tid, a.col_scale + bh * D + tid);
    move(p.row_smooth(bh) + tid, a.row_smooth + bh * D + tid);
  }
  for (int e = tid; e < r * D; e += 256) {
    move(p.comp_k(bh) + e, a.comp_k + bh * (size_t)(r * D) + e);
    move(p.comp_u(bh) + e, a.comp_u + bh * (size_t)(r * D) + e);
  }
  const int RF = record_floats(diag != 0);
  auto move_record = [&](int j, int off, float *plain) {       // one element of record j, fp32 or fp16 in the packed rows
    if (p.rec16) {
      __half *row = p.record<__half>(bh, j, diag != 0);
      if (IMPORT) row[off] = __ushort_as_half(to_f16_bits_sat(*plain));
      else *plain = __half2float(row[off]);
    } else {
      float *row = p.record<float>(bh, j, diag != 0);
      if (IMPORT) row[off] = *plain;
      else *plain = row[off];
    }
  };
  for (int e = tid; e < W * D; e += 256) {
    const int j = e / D, i = e % D;
    move_record(j, REC_KT + i, a.buf_k + (bh * W + j) * (size_t)D + i);
    move_record(j, REC_U + i, a.buf_u + (bh * W + j) * (size_t)D + i);
    if (diag) move_record(j, REC_A + i, a.buf_a + (bh * W + j) * (size_t)D + i);
  }
  if (!diag && tid < W) move(p.decays + bh * (size_t)W + tid, a.buf_a + bh * (size_t)W + tid);
  if (hv == 0 && tid == 0) move(p.win_pos + b, a.win_pos + b);
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
static bool aligned16(const void *ptr) { return (reinterpret_cast<uintptr_t>(ptr) & 15u) == 0; }

static lq_status check_shape(const lq_shape *s) {
  if (!s) return LQ_ERR_NULL;
  if (s->batch < 0 || s->heads_v <= 0 || s->heads_qk <= 0 || s->d_k <= 0 || s->d_v <= 0 || s->W <= 0 || s->r < 0 ||
      s->n_iter < 1 || s->heads_v % s->heads_qk != 0 || (s->gate != LQ_GATE_SCALAR && s->gate != LQ_GATE_DIAG) ||
      (s->delta != 0 && s->delta != 1) || (s->rec16 != 0 && s->rec16 != 1) ||
      (s->state_bf16 != 0 && s->state_bf16 != 1) || (s->state_bf16 && (s->r != 0 || s->smooth != 0)))
    return LQ_ERR_SHAPE;
  if (s->d_k != D || s->d_v != D || s->W > MAX_W || s->r > MAX_R) return LQ_ERR_UNSUPPORTED;
  return LQ_OK;
}

static lq_status check_ptrs(std::initializer_list<const void *> ptrs) {
  for (const void *q : ptrs)
    if (!q) return LQ_ERR_NULL;
  for (const void *q : ptrs)
    if (!aligned16(q)) return LQ_ERR_ALIGN;
  return LQ_OK;
}

// arrays that are only read or written one element at a time need their natural alignment only
static lq_status check_scalar_ptrs(std::initializer_list<const void *> ptrs, unsigned elem_bytes) {
  for (const void *q : ptrs)
    if (!q) return LQ_ERR_NULL;
  for (const void *q : ptrs)
    if (reinterpret_cast<uintptr_t>(q) & (elem_bytes - 1)) return LQ_ERR_ALIGN;
  return LQ_OK;
}

static lq_status check_state(const lq_shape *s, const lq_state *st, bool need_buffers) {
  if (!st) return LQ_ERR_NULL;
  lq_status rc = check_ptrs({st->heads});
  if (rc != LQ_OK) return rc;
  if ((rc = check_scalar_ptrs({st->win_pos}, 4)) != LQ_OK) return rc;
  if (st->work && (reinterpret_cast<uintptr_t>(st->work) & 3u)) return LQ_ERR_ALIGN;
  if (need_buffers) {
    if ((rc = check_ptrs({st->records})) != LQ_OK) return rc;
    if (s->gate == LQ_GATE_SCALAR && (rc = check_scalar_ptrs({st->decays}, 4)) != LQ_OK) return rc;
  }
  return LQ_OK;
}

static Params make_params(const lq_shape *s, const lq_state *st) {
  Params p{};
  p.batch = s->batch; p.heads_v = s->heads_v; p.heads_qk = s->heads_qk; p.W = s->W; p.r = s->r;
  p.n_iter = s->n_iter; p.smooth = s->smooth; p.delta = s->delta; p.rec16 = s->rec16; p.force = 0;
  if (st) {
    p.heads = st->heads; p.records = st->records; p.decays = st->decays; p.win_pos = st->win_pos;
    p.work = st->work;
  }
  return p;
}

static int sm_count() {
  static int cached = 0;
  if (!cached) {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0)
      cached = n;
    else
      return 148;
  }
  return cached;
}

// What a launch needs to ask the runtime only once per (device, kernel): the opt-in to more than 48 KB of shared
// memory and the number of CTAs of a kernel that an SM holds.  Both calls cost a few microseconds of host time,
// which a step of two to ten launches would otherwise pay every token.
static int current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return dev;
}

// (the opt-in is needed once static + dynamic shared memory pass 48 KB; the kernels here hold up to 20 KB static)
static bool smem_opt_in(const void *kernel, size_t smem) {
  if (smem <= 24 * 1024) return true;
  static std::mutex m;
  static std::map<std::pair<int, const void *>, size_t> granted;
  std::lock_guard<std::mutex> lock(m);
  size_t &have = granted[{current_device(), kernel}];
  if (have >= smem) return true;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  have = smem;
  return true;
}

// resident CTAs per SM of `kernel` with this block size and dynamic shared memory (0: the query failed)
static int ctas_per_sm(const void *kernel, int block, size_t smem) {
  static std::mutex m;
  static std::map<std::tuple<int, const void *, int, size_t>, int> known;
  std::lock_guard<std::mutex> lock(m);
  int &per_sm = known[std::make_tuple(current_device(), kernel, block, smem)];
  if (per_sm > 0) return per_sm;
  int v = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kernel, block, smem) != cudaSuccess || v < 1) {
    cudaGetLastError();
    return 0;
  }
  return per_sm = v;
}

// Both of the above for a kernel about to be launched: the opt-in is made, the number of CTAs an SM holds is returned (0: one
// of the calls failed).  A thread remembers its last few answers, so that a step does not take two locks and walk two maps
// per launch.
static int prepare_launch(const void *kernel, int block, size_t smem) {
  struct Known { const void *kernel; size_t smem; int dev, block, per_sm; };
  thread_local Known known[8] = {};
  thread_local unsigned next = 0;
  const int dev = current_device();
  for (const Known &k : known)
    if (k.kernel == kernel && k.smem == smem && k.dev == dev && k.block == block) return k.per_sm;
  if (!smem_opt_in(kernel, smem)) return 0;
  const int per_sm = ctas_per_sm(kernel, block, smem);
  if (per_sm > 0) known[next++ % 8] = Known{kernel, smem, dev, block, per_sm};
  return per_sm;
}

template <typename K, typename P>
static lq_status launch(K kernel, int grid, int block, size_t smem, cudaStream_t stream, const P &p) {
  if (grid <= 0) return LQ_OK;
  if (!smem_opt_in(reinterpret_cast<const void *>(kernel), smem)) return LQ_ERR_CUDA;
  kernel<<<grid, block, smem, stream>>>(p);
  return cudaGetLastError() == cudaSuccess ? LQ_OK : LQ_ERR_CUDA;
}

// Launch that may begin while the kernel before it on the stream is still draining (programmatic dependent
// launch): its CTAs become resident as SM resources free up and sit in griddepcontrol.wait until that kernel
// has completed and its writes are visible.  Only for kernels that execute griddepcontrol.wait before their
// first access to global memory.
template <typename K, typename... Args>
static lq_status launch_dependent(K kernel, int grid, int block, size_t smem, cudaStream_t stream, const Args &...args) {
  if (grid <= 0) return LQ_OK;
  if (prepare_launch(reinterpret_cast<const void *>(kernel), block, smem) < 1) return LQ_ERR_CUDA;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kernel, args...) != cudaSuccess) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  return LQ_OK;
}

// grid <= min(work items, CTAs that fit on the device at once), for kernels that stride over their work
template <typename K>
static lq_status launch_persistent(K kernel, long items, int block, size_t smem, cudaStream_t stream, const Params &p) {
  if (items <= 0) return LQ_OK;
  const int per_sm = prepare_launch(reinterpret_cast<const void *>(kernel), block, smem);
  if (per_sm < 1) return LQ_ERR_CUDA;
  const long resident = (long)per_sm * sm_count();
  // Every CTA takes ceil(items / resident) items at most; the smallest grid with that property leaves no last
  // round in which a fraction of the CTAs works while the others have left (8192 heads: 820 CTAs of 10 heads
  // instead of 888 of which 200 take a tenth).  With scratch words in the state the items of a partial last round
  // go to the CTAs that get there first (decode_slot), and every CTA that fits is launched.
  const long rounds = (items + resident - 1) / resident;
  const long grid = p.work != nullptr ? (items < resident ? items : resident) : (items + rounds - 1) / rounds;
  return launch_dependent(kernel, static_cast<int>(grid), block, smem, stream, p);
}

// persistent two-warp CTAs, each with its own shared-memory slot: as many as are resident at once
template <int GATE, bool R16, bool BF16>
static lq_status launch_decode_t(const lq_shape *s, const Params &p, cudaStream_t stream) {
  const bool diag = GATE == LQ_GATE_DIAG;
  const int whole = DecodeSlot(s->W, s->r, diag, R16, BF16, 0).bytes, ring = DecodeSlot(s->W, s->r, diag, R16, BF16, rec_seg(R16)).bytes;
  // The records of a head at once, or in segments through a smaller slot: in segments where an SM holds no more than three
  // CTAs otherwise.  At 256 x 32 heads, us per step at once / in segments: scalar gate, fp32 records: W = 32 (4 or 5 CTAs)
  // 70.3 / 73.7, W = 40 (3 or 5) 86.5 / 81.3, W = 64 (2 or 5) 129 / 104; fp16 records, W = 64 (4 or 6) 99.1 / 101.7;
  // diagonal gate, fp32: W = 24 (4 or 4) 78.4 / 83.6, W = 32 (3 or 4) 86.8 / 85.6, W = 64 (2 or 4) 224 / 116.
  auto ctas = [](int bytes) { return std::min(6, 228 * 1024 / (bytes + 1024)); };
  const bool longw = s->W - 1 > 2 * rec_seg(R16) && ctas(whole) <= 3 && ctas(ring) > ctas(whole);
  const long nh = (long)s->batch * s->heads_v;
  return longw ? launch_persistent(decode_kernel<GATE, R16, true, BF16>, nh, 64, ring, stream, p)
               : launch_persistent(decode_kernel<GATE, R16, false, BF16>, nh, 64, whole, stream, p);
}
template <bool BF16>
static lq_status launch_decode(const lq_shape *s, const Params &p, cudaStream_t stream) {
  if (s->gate == LQ_GATE_DIAG)
    return s->rec16 ? launch_decode_t<LQ_GATE_DIAG, true, BF16>(s, p, stream) : launch_decode_t<LQ_GATE_DIAG, false, BF16>(s, p, stream);
  return s->rec16 ? launch_decode_t<LQ_GATE_SCALAR, true, BF16>(s, p, stream) : launch_decode_t<LQ_GATE_SCALAR, false, BF16>(s, p, stream);
}

// The boundary kernels are persistent: as many CTAs as are resident at once, each striding over its heads.
template <int GATE, int MODE, bool R16, int RM, bool BF16>
static lq_status launch_boundary_t(const lq_shape *s, const Params &p, cudaStream_t stream, long due) {
  const bool diag = GATE == LQ_GATE_DIAG, iterate = RM > 0 && s->n_iter > 1;
  // Four warps to a state (8 x 16 tiles: a third fewer loads and copies of row values to an FMA) where CTAs have many states in turn and
  // the registers suffice: quantizing with up to four vectors, 2048 states, r = 4 55.3 -> 53.0 us, r = 3 51.5 -> 49.0, r = 4 with two
  // rounds 88.6 -> 84.6.  Not with a state to an SM at most, or one in the last of two rounds: with eight / four warps 64 states 6.5 / 6.8 us,
  // 128 6.7 / 7.1, 160 9.3 / 8.7, 288 9.7 / 9.1, 320 13.8 / 13.8, 384 13.9 / 14.2, 448 16.7 / 15.7, 768 24.2 / 22.7 (r = 4; r = 2 and two rounds alike).
  // Without vectors the memory is the limit for many states: r = 0 416 7.1 / 5.6, 1024 12.2 / 10.9, 1536 23.4 / 23.2, 2048 28.9 / 29.5, 4096 53.0 / 54.9;
  // the BF16 state 416 6.9 / 5.5, 1024 13.2 / 12.7, 2048 32.0 / 32.7.
  // Eight vectors take 98 us with eight warps and 111 with four.  Flushes with four vectors, one round, the scalar
  // gate and fp32 records: figures at boundary_head.  With two rounds 137.2 / 137.7 us a step (512 x 32, W = 24, eight / four warps); 256 x 32,
  // W = 16, in a loop and behind other kernels: diagonal gate 67.3, 69.9 / 67.4, 70.9, fp16 records 58.9, 61.1 / 58.7, 62.2.  One flush by itself is longer with four (32 x 32 heads: 18.1 / 19.1), and so is the
  // search among many sequences: four where all CTAs have one to do and two trips cover the batch.
  constexpr bool QUANTIZE4 = MODE == 1 && RM <= 4, DEQUANTIZE4 = MODE == 2 && RM == 4;
  constexpr bool FLUSH4 = MODE == 0 && RM == 4 && GATE == LQ_GATE_SCALAR && !R16;
  // Dequantizing 8-bit states, more than are resident at once: four warps, and the state is put together in shared memory and leaves by
  // bulk stores, where two CTAs still fit on an SM so (2048 states, W = 16, r = 4: diagonal gate 46.0 -> 43.8 us, scalar gate 47.1 -> 43.9;
  // with eight warps 46.7 and 47.6; 256 states 7.35 / 7.54; the BF16 state 40.4 either way).
  const long nh = (long)s->batch * s->heads_v, sms = sm_count();
  const bool staged_out = DEQUANTIZE4 && nh > 2 * sms &&
                          BoundarySmem<0, 4, false>(MODE, s->W, s->r, diag, R16, BF16, false, 1, true).bytes <= (228 / 2 - 1) * 1024 - 512;
  const bool four = staged_out || (QUANTIZE4 && nh > sms && (RM == 0 ? nh <= 10 * sms : nh <= 2 * sms || nh > 3 * sms)) ||
                    (FLUSH4 && s->r == RM && !iterate && due >= 2 * sms && s->batch <= 2048);
  const int threads = four ? 128 : 256;
  constexpr int RL = MODE == 2 ? 0 : RM;
  auto bytes = [&](int slots, bool staged_out = false) {
    return four ? BoundarySmem<RL, 4, MODE != 2>(MODE, s->W, s->r, diag, R16, BF16, iterate && MODE != 2, slots, staged_out).bytes
                : BoundarySmem<RL, 8, MODE != 2>(MODE, s->W, s->r, diag, R16, BF16, iterate && MODE != 2, slots, staged_out).bytes;
  };
  // A second slot where a head is through in a few microseconds and two CTAs with two slots each still fit on an SM; a head
  // that is requantized leaves its slot early enough for the next one (two slots: 65.3 us against 64.1 at 256 x 32 heads).
  const int slots = (MODE == 2 || (BF16 && MODE == 0)) && !staged_out && bytes(2) <= (228 / 2 - 2) * 1024 ? 2 : 1;
  constexpr bool may_be_exact = (MODE == 0 && (RM == 4 || RM == 8)) || (MODE == 1 && RM == 4);
  const bool exact = may_be_exact && s->r == RM;
  constexpr bool one_round = MODE == 0 && RM == 4;       // (instances for one round)
  auto kernel = boundary_kernel<GATE, MODE, R16, RM, BF16, false, true, false, 8>;
  if (exact) kernel = boundary_kernel<GATE, MODE, R16, RM, BF16, may_be_exact, true, false, 8>;
  if (one_round && exact && !iterate) kernel = boundary_kernel<GATE, MODE, R16, RM, BF16, may_be_exact, !one_round, false, 8>;
  if constexpr (QUANTIZE4 || DEQUANTIZE4 || FLUSH4) {
    if (four) kernel = boundary_kernel<GATE, MODE, R16, RM, BF16, FLUSH4, !FLUSH4, false, 4>;
    if (four && exact) kernel = boundary_kernel<GATE, MODE, R16, RM, BF16, may_be_exact, !FLUSH4, false, 4>;
  }
  // With more than eight compensators two heads on one SM take half as long again as one, and CTAs that leave room for a second
  // one are not placed one to an SM (the first 148 of 296 come to lie on 142 SMs): where windows of every fill would have no
  // more heads due at a time than there are SMs, though all heads at once are more than two to an SM, a CTA asks for more than
  // half of its SM's memory.  64 x 32 heads, W = 16, us per step with one CTA / two to an SM: windows of every fill, r = 9
  // 35.6 / 37.1, r = 12 38.5 / 42.1, r = 16 43.7 / 50.2; all windows due at once (every 16th step), r = 16, on average 37.4 / 31.5.
  const bool alone = RM > 8 && MODE == 0 && due <= sms && nh > 2 * sms;
  const int smem = alone ? std::max(bytes(slots), 116 * 1024) : bytes(slots, staged_out);
  const long resident = prepare_launch(reinterpret_cast<const void *>(kernel), threads, smem) * sms;
  if (resident < 1) return LQ_ERR_CUDA;
  return launch_dependent(kernel, static_cast<int>(nh < resident ? nh : resident), threads, smem, stream, p, slots, staged_out ? 1 : 0);
}

// A whole step of few heads in one launch, a CTA per head: as long as every SM has one head at most (a CTA takes most of an
// SM's registers).  W = 16, r = 4, us per step in a graph as two launches / one: 1 head 6.7 / 5.1, 32 heads 6.7 / 5.2, 128 heads
// 8.3 / 6.9, 148 heads of 37 sequences 13.8 / 12.7, 184 heads 14.5 / 14.5, 280 heads 14.2 / 16.1; 128 heads, diagonal gate,
// W = 64, r = 8: 11.4 / 8.4; called one by one from the host, 1 to 128 heads: 11 / 8.4.  (With the instances for exactly four
// and eight compensators a step of 148 heads takes 12.0 instead of 12.7 us, of 128 heads, W = 8, 10.6 instead of 11.3.)  Two streams
// of 40 to 148 heads each, which then share the GPU less well: 9.6 to 13.4 us for a step of both, 12.4 to 17.8 as two launches each
// (kernels of an earlier build; r = 8 12.1 to 17.3 and 15.9 to 24.2).
static bool one_launch(const lq_shape *s) {
  return (long)s->batch * s->heads_v <= sm_count();
}
template <int GATE, bool R16, int RM, bool BF16>
static lq_status launch_step_t(const lq_shape *s, const Params &p, cudaStream_t stream) {
  const bool diag = GATE == LQ_GATE_DIAG;
  constexpr int NW = 8;
  const int smem = std::max(BoundarySmem<RM, NW>(0, s->W, s->r, diag, R16, BF16, RM > 0 && s->n_iter > 1, 1).bytes,
                            TOKEN_SLOT + DecodeSlot(s->W, s->r, diag, R16, BF16, 0).bytes);
  auto kernel = boundary_kernel<GATE, 0, R16, RM, BF16, false, true, true, NW>;
  if (s->r == RM && (RM == 4 || RM == 8)) kernel = boundary_kernel<GATE, 0, R16, RM, BF16, RM == 4 || RM == 8, true, true, NW>;
  return launch_dependent(kernel, s->batch * s->heads_v, 32 * NW, smem, stream, p, 1, 0);
}
template <int RM, bool BF16>
static lq_status launch_step_gate(const lq_shape *s, const Params &p, cudaStream_t stream) {
  if (s->gate == LQ_GATE_DIAG)
    return s->rec16 ? launch_step_t<LQ_GATE_DIAG, true, RM, BF16>(s, p, stream) : launch_step_t<LQ_GATE_DIAG, false, RM, BF16>(s, p, stream);
  return s->rec16 ? launch_step_t<LQ_GATE_SCALAR, true, RM, BF16>(s, p, stream) : launch_step_t<LQ_GATE_SCALAR, false, RM, BF16>(s, p, stream);
}
static lq_status launch_step(const lq_shape *s, const Params &p, cudaStream_t stream) {
  if (s->state_bf16) return launch_step_gate<0, true>(s, p, stream);
  if (s->r == 0) return launch_step_gate<0, false>(s, p, stream);
  if (s->r <= 4) return launch_step_gate<4, false>(s, p, stream);
  if (s->r <= 8) return launch_step_gate<8, false>(s, p, stream);
  return launch_step_gate<MAX_R, false>(s, p, stream);
}

// A step of many heads in one launch (step_kernel); false where it does not apply.  launch = false: says only whether it does.
// It does with up to one due head to an SM, on average over windows of every fill: such a head is through its boundary while the
// others get their tokens, and the second launch, the wait for the first kernel's last CTA and the search for due heads are saved.  r = 4, us per
// step as two launches / one, in a loop of steps and (in brackets) behind a projection, norms and a softmax, where code and state are fetched anew:
//   scalar gate: 32 x 32 heads, W = 16 17.6 / 16.5 (18.8 / 19.1), W = 8 19.7 / 14.7 (20.9 / 17.1), W = 32 20.5 / 19.4 (20.9 / 23.1);
//     48 x 32, W = 16 19.0 / 19.2 (20.7 / 21.5); 64 x 32, W = 16 25.8 / 22.4 (27.4 / 24.6); 128 x 32, W = 32 43.3 / 31.2 (44.5 / 33.9)
//   diagonal gate: 32 x 32, W = 16 18.3 / 17.7 (19.3 / 21.1); 64 x 32, W = 16 27.6 / 24.5 (29.9 / 27.7); 128 x 32, W = 32 54.6 / 42.2 (56.7 / 44.7)
// Not where every head has a CTA of the decode kernel to itself (six to an SM): 20 x 16 heads, W = 16 14.7 / 14.1 (14.9 / 18.7), diagonal gate
// 14.2 / 14.7 (14.7 / 20.9); 24 x 32 15.7 / 15.9 (16.6 / 18.9).  A boundary of several rounds is more code and longer: from twice as many heads on, or
// where two SMs of three have a due head: a loop of steps gains up to a quarter then, steps behind other kernels lose up to a fifth.
// Two rounds, r = 4, two / one: 32 x 32, W = 8 24.3 / 18.6 (25.8 / 27.3), W = 10 21.1 / 19.0 (24.8 / 27.3), W = 7 24.3 / 23.9 (26.7 / 32.6), r = 8,
// W = 8 35.7 / 27.6 (37.7 / 43.5); 48 x 32, W = 12 26.3 / 21.9 (30.3 / 28.4), W = 15 23.3 / 22.5 (27.0 / 30.4); diagonal gate, 32 x 32, W = 8
// 24.2 / 19.2 (27.5 / 29.1), 48 x 32, W = 12 28.2 / 23.1 (32.0 / 31.6).  With fewer due, 32 x 32,
// W = 16, r = 4, two rounds 20.9 / 20.1 (21.9 / 26.9); 48 x 32 22.2 / 22.8 (22.9 / 26.8); 64 x 32 29.8 / 26.2 (31.4 / 29.8), r = 8 41.2 / 33.8 (42.4 / 45.5);
// 128 x 32, W = 32 47.7 / 34.8 (48.8 / 37.5).
// With more than one due head to an SM they go through their boundaries one after the other, which takes as long as two at a time in a kernel of
// their own behind the tokens: 128 x 32, W = 16 34.9 / 34.7; 256 x 32 60.8 / 63; diagonal gate 38.4 / 39.6 and 67.9 / 73.  With the scalar
// gate and long windows the tokens leave time for all of them (W = 24, 512 x 32: 123.2 / 117.8 (125.4 / 119.2); W = 32, 1024 x 32: 247.7 / 232.0
// (246.8 / 231.8); W = 20: 117 / 118).
// The price of one boundary at a time is paid where all windows fall due in the same step, as those of sequences admitted together do: mean over the
// window and the longest step, two launches / one: 32 x 32, W = 16 12.3 / 11.6, 65 / 72; 64 x 32 18.6 / 20.4, 105 / 131; 128 x 32, W = 32 35.0 / 35.2,
// 256 / 305; 512 x 32, W = 24 119.9 / 124.8, 834 / 1037; 1024 x 32, W = 32 247 / 254, 1911 / 2378; 64 x 32, r = 0 16.1 / 16.5, r = 8 21.8 / 25.2.  Which it is the host does
// not know.  And a CTA fills its SM, so two streams with a state each take turns: a step of both, two launches / one, 32 x 32, W = 16 23.2 / 24.1,
// 64 x 32 33.3 / 40.0 (one state: 25.8 / 22.3), diagonal gate 37.4 / 43.5 (27.7 / 24.4), 128 x 32, W = 32 64.7 / 58.3.
// Three slots to an SM where four do not fit (W = 40, 128 x 32: 48.8 / 42.8); two are too few (W = 64, 256 x 32: 101 / 119).  fp16
// records: no gain (diagonal gate, 64 x 32, r = 3: 26.3 / 26.5), so there are no instances for them.
template <int GATE, int RM, bool EXACT, bool ROUNDS>
static bool launch_merged_t(const lq_shape *s, const Params &p, cudaStream_t stream, lq_status *rc, bool launch) {
  auto bytes = [&](int pairs) { return StepSmem<RM>(pairs, s->batch, s->W, s->r, GATE == LQ_GATE_DIAG, RM > 0 && s->n_iter > 1).bytes; };
  int pairs = STEP_PAIRS;                    // (226 of 227 KB: there are static arrays)
  while (pairs > 0 && bytes(pairs) > 226 * 1024) pairs--;
  if (pairs < STEP_PAIRS - 1) return false;
  const long nh = (long)s->batch * s->heads_v, sms = sm_count();
  if (nh <= 6 * sms || (ROUNDS && nh <= 12 * sms && 3 * nh <= 2 * sms * s->W)) return false;
  if (nh > sms * s->W && !(GATE == LQ_GATE_SCALAR && s->W >= 24 && pairs == STEP_PAIRS)) return false;
  if (launch) *rc = launch_dependent(step_kernel<GATE, RM, EXACT, ROUNDS>, static_cast<int>(sms), STEP_THREADS, bytes(pairs), stream, p, pairs);
  return true;
}
static bool launch_merged(const lq_shape *s, const Params &p, cudaStream_t stream, lq_status *rc, bool launch) {
  if (!p.work || s->batch == 0 || s->batch > STEP_MAX_BATCH || s->r > STEP_MAX_R || s->state_bf16 || s->rec16) return false;
  const bool diag = s->gate == LQ_GATE_DIAG;
  auto by_gate = [&](auto rm, auto exact, auto rounds) {
    return diag ? launch_merged_t<LQ_GATE_DIAG, rm, exact, rounds>(s, p, stream, rc, launch) : launch_merged_t<LQ_GATE_SCALAR, rm, exact, rounds>(s, p, stream, rc, launch);
  };
  constexpr std::integral_constant<int, 0> r0; constexpr std::integral_constant<int, 4> r4; constexpr std::integral_constant<int, 8> r8;
  constexpr std::true_type yes; constexpr std::false_type no;
  if (s->r == 0) return by_gate(r0, no, no);
  if (s->n_iter > 1) return s->r <= 4 ? by_gate(r4, no, yes) : by_gate(r8, no, yes);
  return s->r == 4 ? by_gate(r4, yes, no) : s->r < 4 ? by_gate(r4, no, no) : by_gate(r8, no, no);
}

template <int MODE, int RM, bool BF16>
static lq_status launch_boundary_gate(const lq_shape *s, const Params &p, cudaStream_t stream, long due) {
  if (MODE == 1) return launch_boundary_t<LQ_GATE_SCALAR, MODE, false, RM, BF16>(s, p, stream, due);   // (reads no records)
  constexpr int M_ = MODE == 1 ? 0 : MODE;
  if (s->gate == LQ_GATE_DIAG)
    return s->rec16 ? launch_boundary_t<LQ_GATE_DIAG, M_, true, RM, BF16>(s, p, stream, due) : launch_boundary_t<LQ_GATE_DIAG, M_, false, RM, BF16>(s, p, stream, due);
  return s->rec16 ? launch_boundary_t<LQ_GATE_SCALAR, M_, true, RM, BF16>(s, p, stream, due) : launch_boundary_t<LQ_GATE_SCALAR, M_, false, RM, BF16>(s, p, stream, due);
}

// compiled for r = 0, r <= 4, r <= 8 and any r (the small matrices of the fit live in registers); due: heads that are due at a
// time, as far as the call tells
template <int MODE>
static lq_status launch_boundary(const lq_shape *s, const Params &p, cudaStream_t stream, long due) {
  if (s->batch == 0) return LQ_OK;
  if (s->state_bf16) return launch_boundary_gate<MODE, 0, true>(s, p, stream, due);
  if (s->r == 0) return launch_boundary_gate<MODE, 0, false>(s, p, stream, due);
  if (MODE == 2 || s->r <= 4) return launch_boundary_gate<MODE, 4, false>(s, p, stream, due);
  if (s->r <= 8) return launch_boundary_gate<MODE, MODE == 2 ? 4 : 8, false>(s, p, stream, due);
  return launch_boundary_gate<MODE, MODE == 2 ? 4 : MAX_R, false>(s, p, stream, due);
}

}  // namespace lq

using namespace lq;

extern "C" {

static lq_status decode_step_impl(const lq_shape *shape, const lq_state *state, const uint16_t *q, const uint16_t *k,
                                  const uint16_t *v, const uint16_t *beta, const uint16_t *alpha, float *o,
                                  lq_stream stream, cudaEvent_t between, int part = -1) {
  // part >= 0: the decode kernel only, of sub-batch `part` (each of them counts its tickets in a word of its own)
  lq_status rc = check_shape(shape);
  if (rc != LQ_OK) return rc;
  if ((rc = check_state(shape, state, true)) != LQ_OK) return rc;
  if ((rc = check_ptrs({q, k, v, o})) != LQ_OK) return rc;
  if ((rc = check_scalar_ptrs({beta}, 2)) != LQ_OK) return rc;
  if ((rc = shape->gate == LQ_GATE_DIAG ? check_ptrs({alpha}) : check_scalar_ptrs({alpha}, 2)) != LQ_OK) return rc;
  Params p = make_params(shape, state);
#ifdef LQ_TIMING
  static int generation = 0;
  p.gen = generation++;
#endif
  p.q = q; p.k = k; p.v = v; p.beta = beta; p.alpha = alpha; p.o = o;
  const long nh = (long)shape->batch * shape->heads_v;
  p.overlap = nh >= 2L * sm_count() * shape->W;        // as many boundaries as boundary CTAs, on average
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (!between && part < 0 && one_launch(shape)) return launch_step(shape, p, st);
  if (!between && part < 0 && launch_merged(shape, p, st, &rc, true)) return rc;
  if (part > 0 && p.work) p.work += part;
  rc = shape->state_bf16 ? launch_decode<true>(shape, p, st) : launch_decode<false>(shape, p, st);
  if (rc != LQ_OK) return rc;
  if (between && cudaEventRecord(between, st) != cudaSuccess) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  return part >= 0 ? LQ_OK : launch_boundary<0>(shape, p, st, nh / shape->W);     // sequences whose window just became full
}

lq_status lq_decode_step(const lq_shape *shape, const lq_state *state, const uint16_t *q, const uint16_t *k,
                         const uint16_t *v, const uint16_t *beta, const uint16_t *alpha, float *o, lq_stream stream) {
  return decode_step_impl(shape, state, q, k, v, beta, alpha, o, stream, nullptr);
}

lq_status lq_decode_step_profiled(const lq_shape *shape, const lq_state *state, const uint16_t *q, const uint16_t *k,
                                  const uint16_t *v, const uint16_t *beta, const uint16_t *alpha, float *o,
                                  lq_stream stream, void *event_between) {
  return decode_step_impl(shape, state, q, k, v, beta, alpha, o, stream, static_cast<cudaEvent_t>(event_between));
}

uint64_t lq_head_bytes(const lq_shape *s) {
  if (check_shape(s) != LQ_OK) return 0;
  return s->state_bf16 ? (uint64_t)BF16W_HEAD_BYTES : (uint64_t)head_bytes(s->r);
}

uint64_t lq_record_floats(const lq_shape *s) {
  return check_shape(s) == LQ_OK ? (uint64_t)record_floats(s->gate == LQ_GATE_DIAG) : 0;
}

uint64_t lq_decode_stage_bytes(const lq_shape *s) {
  if (check_shape(s) != LQ_OK) return 0;
  const uint64_t B = s->batch, Hv = s->heads_v, Hqk = s->heads_qk, K = s->d_k, V = s->d_v;
  auto up = [](uint64_t x) { return (x + 255) / 256 * 256; };
  const uint64_t na = s->gate == LQ_GATE_DIAG ? B * Hv * K : B * Hv;
  return 2 * up(2 * B * Hqk * K) + up(2 * B * Hv * V) + up(2 * B * Hv) + up(2 * na) + up(4 * B * Hv * V);
}

}  // extern "C"

// One launch that brings the five input arrays from mapped pinned host memory into the device staging
// buffer (the alternative, five cudaMemcpyAsync calls, costs about 10 us of latency per copy on top of the
// transfer itself).  Every segment is a whole number of 16-byte units; both ends are 16-byte aligned.
namespace {
struct GatherSegs {
  const uint4 *src[5];
  uint4 *dst[5];
  uint32_t units[5];      // 16-byte units per segment
};
__global__ void __launch_bounds__(256) gather_kernel(const GatherSegs g) {
  const uint32_t stride = gridDim.x * blockDim.x;
#pragma unroll
  for (int sgm = 0; sgm < 5; sgm++) {
    const uint4 *__restrict__ src = g.src[sgm];
    uint4 *__restrict__ dst = g.dst[sgm];
    const uint32_t n = g.units[sgm];
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {          // four loads in flight per thread
      const uint4 a = src[i], b = src[i + stride], c = src[i + 2 * stride], d = src[i + 3 * stride];
      dst[i] = a; dst[i + stride] = b; dst[i + 2 * stride] = c; dst[i + 3 * stride] = d;
    }
    for (; i < n; i += stride) dst[i] = src[i];
  }
}

// About five microseconds ahead of a decode kernel, in which the next sub-batch's gather gets its places (see below).  With an empty kernel
// in its place the decode kernel is launched early behind it, and the order is as before.
__global__ void head_start_kernel() {
  const long long t0 = clock64();
  for (int i = 0; i < 4096 && clock64() - t0 < 10000; i++) __nanosleep(100);
}

// The device alias of a pinned, mapped host pointer; null if the memory is not mapped into the device.
template <typename T>
T *device_alias(T *host) {
  void *dev = nullptr;
  if (cudaHostGetDevicePointer(&dev, const_cast<void *>(static_cast<const void *>(host)), 0) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return static_cast<T *>(dev);
}
}  // namespace

extern "C" {

static void host_pipe_break_chain();

static lq_status host_step_impl(const lq_shape *shape, const lq_state *state, const uint16_t *q_h, const uint16_t *k_h,
                                const uint16_t *v_h, const uint16_t *beta_h, const uint16_t *alpha_h, float *o_h,
                                void *stage, lq_stream stream, bool direct_ok) {
  lq_status rc = check_shape(shape);
  if (rc != LQ_OK) return rc;
  if ((rc = check_state(shape, state, true)) != LQ_OK) return rc;     // nothing is enqueued before every argument is checked
  if (!q_h || !k_h || !v_h || !beta_h || !alpha_h || !o_h || !stage) return LQ_ERR_NULL;
  if (!aligned16(stage)) return LQ_ERR_ALIGN;
  const uint64_t B = shape->batch, Hv = shape->heads_v, Hqk = shape->heads_qk, K = shape->d_k, V = shape->d_v;
  auto up = [](uint64_t x) { return (x + 255) / 256 * 256; };
  const uint64_t nqk = 2 * B * Hqk * K, nv = 2 * B * Hv * V, nb = 2 * B * Hv;
  const uint64_t na = 2 * (shape->gate == LQ_GATE_DIAG ? B * Hv * K : B * Hv), no = 4 * B * Hv * V;
  char *base = static_cast<char *>(stage);
  uint16_t *q_d = reinterpret_cast<uint16_t *>(base); base += up(nqk);
  uint16_t *k_d = reinterpret_cast<uint16_t *>(base); base += up(nqk);
  uint16_t *v_d = reinterpret_cast<uint16_t *>(base); base += up(nv);
  uint16_t *b_d = reinterpret_cast<uint16_t *>(base); base += up(nb);
  uint16_t *a_d = reinterpret_cast<uint16_t *>(base); base += up(na);
  float *o_d = reinterpret_cast<float *>(base);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (B == 0) return LQ_OK;
  host_pipe_break_chain();                   // this call writes `stage` in stream order only

  // Fast path, when all six host arrays are pinned, mapped into the device and 16-byte aligned: one gather
  // launch reads the inputs over the bus, and the decode kernel writes o straight into the host array (posted
  // writes that overlap the kernel), so no copy follows the step.
  const uint16_t *src_h[5] = {q_h, k_h, v_h, beta_h, alpha_h};
  uint16_t *dst_d[5] = {q_d, k_d, v_d, b_d, a_d};
  const uint64_t bytes[5] = {nqk, nqk, nv, nb, na};
  GatherSegs g;
  bool mapped = direct_ok && aligned16(o_h) && no < (1ull << 35);
  for (int i = 0; mapped && i < 5; i++) {
    const uint16_t *alias = (aligned16(src_h[i]) && bytes[i] < (1ull << 35)) ? device_alias(src_h[i]) : nullptr;
    mapped = alias != nullptr;
    g.src[i] = reinterpret_cast<const uint4 *>(alias);
    g.dst[i] = reinterpret_cast<uint4 *>(dst_d[i]);
    g.units[i] = static_cast<uint32_t>((bytes[i] + 15) / 16);   // the regions of `stage` are padded to 256 bytes;
  }                                                             // a ragged tail is covered below
  float *o_alias = mapped ? device_alias(o_h) : nullptr;
  // a segment that is not a whole number of 16-byte units would read past the end of the host array
  for (int i = 0; mapped && i < 5; i++) mapped = bytes[i] % 16 == 0;
  if (mapped && o_alias) {
    rc = launch(gather_kernel, 2 * sm_count(), 256, 0, st, g);
    if (rc != LQ_OK) return rc;
    return lq_decode_step(shape, state, q_d, k_d, v_d, b_d, a_d, o_alias, stream);
  }

  if (cudaMemcpyAsync(q_d, q_h, nqk, cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemcpyAsync(k_d, k_h, nqk, cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemcpyAsync(v_d, v_h, nv, cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemcpyAsync(b_d, beta_h, nb, cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemcpyAsync(a_d, alpha_h, na, cudaMemcpyHostToDevice, st) != cudaSuccess) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  rc = lq_decode_step(shape, state, q_d, k_d, v_d, b_d, a_d, o_d, stream);
  if (rc != LQ_OK) return rc;
  if (cudaMemcpyAsync(o_h, o_d, no, cudaMemcpyDeviceToHost, st) != cudaSuccess) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  return LQ_OK;
}

lq_status lq_decode_step_host(const lq_shape *shape, const lq_state *state, const uint16_t *q_h, const uint16_t *k_h,
                              const uint16_t *v_h, const uint16_t *beta_h, const uint16_t *alpha_h, float *o_h,
                              void *stage, lq_stream stream) {
  return host_step_impl(shape, state, q_h, k_h, v_h, beta_h, alpha_h, o_h, stage, stream, true);
}

// ---------------------------------------------------------------------------------------------
// Host-buffer decode step with the copies overlapped with the kernels: the batch is cut into chunks of
// sequences; chunk c+1 is copied in and chunk c-1 copied out while chunk c is computed.  The copies run on two
// streams that the library creates per device on first use; events tie them to the caller's stream, so for the
// caller the call is still one piece of work on `stream`.
// ---------------------------------------------------------------------------------------------
namespace {
constexpr int PIPE_CHUNKS = 2;
static_assert(PIPE_CHUNKS <= LQ_WORK_WORDS, "a ticket counter each");
struct HostPipe {
  bool ready = false;
  cudaStream_t s_in = nullptr, s_out = nullptr;
  cudaEvent_t start = nullptr, out = nullptr, in[PIPE_CHUNKS] = {}, done[PIPE_CHUNKS] = {};
  // The previous pipelined call on this device, if the next one may chain onto it: same staging buffer, stream
  // and staging layout.  done[c] then still marks the moment that call's decode kernel had consumed the inputs
  // of sub-batch c.
  bool chain = false;
  const void *stage = nullptr;
  cudaStream_t stream = nullptr;
  uint64_t layout[5] = {};                   // B, Hv, Hqk, gate, W
};
std::mutex g_pipe_mutex;
HostPipe g_pipes[64];

lq_status host_pipe(HostPipe **out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  HostPipe &hp = g_pipes[dev];
  if (!hp.ready) {
    bool ok = cudaStreamCreateWithFlags(&hp.s_in, cudaStreamNonBlocking) == cudaSuccess &&
              cudaStreamCreateWithFlags(&hp.s_out, cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreateWithFlags(&hp.start, cudaEventDisableTiming) == cudaSuccess &&
              cudaEventCreateWithFlags(&hp.out, cudaEventDisableTiming) == cudaSuccess;
    for (int c = 0; ok && c < PIPE_CHUNKS; c++)
      ok = cudaEventCreateWithFlags(&hp.in[c], cudaEventDisableTiming) == cudaSuccess &&
           cudaEventCreateWithFlags(&hp.done[c], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) {
      cudaGetLastError();
      return LQ_ERR_CUDA;
    }
    hp.ready = true;
  }
  *out = &hp;
  return LQ_OK;
}
}  // namespace

// a later pipelined call must not start reading its inputs early: something else is about to use a staging buffer
static void host_pipe_break_chain() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return;
  }
  std::lock_guard<std::mutex> lock(g_pipe_mutex);
  g_pipes[dev].chain = false;
}

lq_status lq_decode_step_host_pipelined(const lq_shape *shape, const lq_state *state, const uint16_t *q_h,
                                        const uint16_t *k_h, const uint16_t *v_h, const uint16_t *beta_h,
                                        const uint16_t *alpha_h, float *o_h, void *stage, lq_stream stream) {
  lq_status rc = check_shape(shape);
  if (rc != LQ_OK) return rc;
  if (shape->batch < 8 * PIPE_CHUNKS)          // nothing to overlap (breaks a chain of pipelined calls as well)
    return lq_decode_step_host(shape, state, q_h, k_h, v_h, beta_h, alpha_h, o_h, stage, stream);
  if ((rc = check_state(shape, state, true)) != LQ_OK) return rc;
  if (!q_h || !k_h || !v_h || !beta_h || !alpha_h || !o_h || !stage) return LQ_ERR_NULL;
  if (!aligned16(stage)) return LQ_ERR_ALIGN;
  const uint64_t B = shape->batch, Hv = shape->heads_v, Hqk = shape->heads_qk, K = shape->d_k, V = shape->d_v;
  const bool diag = shape->gate == LQ_GATE_DIAG;
  auto up = [](uint64_t x) { return (x + 255) / 256 * 256; };
  const uint64_t eqk = Hqk * K, ev = Hv * V, eb = Hv, ea = diag ? Hv * K : Hv;   // elements per sequence
  char *base = static_cast<char *>(stage);
  uint16_t *q_d = reinterpret_cast<uint16_t *>(base); base += up(2 * B * eqk);
  uint16_t *k_d = reinterpret_cast<uint16_t *>(base); base += up(2 * B * eqk);
  uint16_t *v_d = reinterpret_cast<uint16_t *>(base); base += up(2 * B * ev);
  uint16_t *b_d = reinterpret_cast<uint16_t *>(base); base += up(2 * B * eb);
  uint16_t *a_d = reinterpret_cast<uint16_t *>(base); base += up(2 * B * ea);
  float *o_d = reinterpret_cast<float *>(base);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const uint16_t *src_h[5] = {q_h, k_h, v_h, beta_h, alpha_h};
  uint16_t *dst_d[5] = {q_d, k_d, v_d, b_d, a_d};
  const uint64_t per_seq[5] = {eqk, eqk, ev, eb, ea};

  // every sub-batch starts at a multiple of 8 sequences, which keeps all of its pointers 16-byte aligned and
  // all of its arrays whole numbers of 16-byte units
  const uint64_t per = (B / PIPE_CHUNKS + 7) / 8 * 8;
  uint64_t lo[PIPE_CHUNKS + 1];
  for (int c = 0; c < PIPE_CHUNKS; c++) lo[c] = std::min<uint64_t>(B, c * per);
  lo[PIPE_CHUNKS] = B;

  // Inputs: when the host arrays are pinned, mapped into the device and aligned, one gather launch per
  // sub-batch (a few CTAs, which share the device with the kernels of the sub-batch before); otherwise five
  // copies per sub-batch.
  const uint16_t *src_a[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
  bool mapped = true;
  for (int i = 0; mapped && i < 5; i++) {
    src_a[i] = aligned16(src_h[i]) ? device_alias(src_h[i]) : nullptr;
    mapped = src_a[i] != nullptr && (2 * B * per_seq[i]) % 16 == 0;
  }

  std::lock_guard<std::mutex> lock(g_pipe_mutex);   // the events below are shared by all callers on a device
  HostPipe *hp = nullptr;
  if ((rc = host_pipe(&hp)) != LQ_OK) return rc;
  // Chained onto the previous call (same staging buffer, stream and layout): the inputs of sub-batch c may be
  // brought in as soon as that call's decode kernel of sub-batch c has read its own - next to that call's
  // window-boundary kernels and copies out - instead of after everything on `stream`.
  const uint64_t layout[5] = {B, Hv, Hqk, (uint64_t)shape->gate, (uint64_t)shape->W};
  const bool chained = hp->chain && hp->stage == stage && hp->stream == st &&
                       std::equal(layout, layout + 5, hp->layout);
  hp->chain = false;                         // set again at the end, if everything was enqueued
  // (the copy-out stream needs no tie at the start: all it does waits for a kernel of this call on `stream`)
  bool ok = chained || (cudaEventRecord(hp->start, st) == cudaSuccess &&    // after everything already on `stream`
                        cudaStreamWaitEvent(hp->s_in, hp->start, 0) == cudaSuccess);
  for (int c = 0; ok && c < PIPE_CHUNKS; c++) {
    const uint64_t b0 = lo[c], nb = lo[c + 1] - lo[c];
    if (nb == 0) continue;
    if (chained) ok = cudaStreamWaitEvent(hp->s_in, hp->done[c], 0) == cudaSuccess;   // (the previous call's record)
    if (!ok) break;
    if (mapped) {
      GatherSegs g;
      for (int i = 0; i < 5; i++) {
        g.src[i] = reinterpret_cast<const uint4 *>(src_a[i] + b0 * per_seq[i]);
        g.dst[i] = reinterpret_cast<uint4 *>(dst_d[i] + b0 * per_seq[i]);
        g.units[i] = static_cast<uint32_t>((2 * nb * per_seq[i] + 15) / 16);
      }
      // Sixteen CTAs (262 KB in flight, which the bus does not need more of): each of them keeps a decode CTA of the other
      // sub-batch waiting for its place.  256 x 32 heads: 202 us a call by itself and 151 chained; with 74 CTAs 210 and 158
      // (the decode kernel of half a batch took 43 us instead of 24), with 8 CTAs 222 and 172.  From 16 to 256 sequences of 8 to 64
      // heads and with either gate no other number did better by more than 6 %: 24, 32 and 48 are slower in most by 3 to 20 %.
      ok = launch(gather_kernel, 16, 256, 0, hp->s_in, g) == LQ_OK;
    } else {
      for (int i = 0; ok && i < 5; i++)
        ok = cudaMemcpyAsync(dst_d[i] + b0 * per_seq[i], src_h[i] + b0 * per_seq[i], 2 * nb * per_seq[i],
                             cudaMemcpyHostToDevice, hp->s_in) == cudaSuccess;
    }
    ok = ok && cudaEventRecord(hp->in[c], hp->s_in) == cudaSuccess;
  }
  // Kernels on `stream`, sub-batch after sub-batch.  o of a sub-batch is complete after its decode kernel, so
  // its copy to the host starts there.  The window boundaries come last, in one launch for the whole batch: between the
  // sub-batches they would hold up the second one's decode kernel.
  for (int c = 0; ok && c < PIPE_CHUNKS; c++) {
    const uint64_t b0 = lo[c], nb = lo[c + 1] - lo[c];
    if (nb == 0) continue;
    ok = cudaStreamWaitEvent(st, hp->in[c], 0) == cudaSuccess;
    // The end of a gather lets both go, this sub-batch's decode kernel and the next one's gather, and which of them is first decides how the
    // call goes, and changed with every build of the library: decode CTAs fill every SM, so a gather behind them waits until the first of them
    // leave (20 us), and then shares SMs with the others, whose loads queue up behind its reads over the bus (that decode kernel takes 43 us
    // instead of 28).  So a long gather gets a head start.  us of a call by itself and back to back with those of other states, without (two builds) and
    // with: 256 x 32 heads 216 - 224, 183 - 204 / 201, 183; 180 x 32 179, 144 - 167 / 161, 143; 512 x 32 408, 342 - 396 / 357, 338; diagonal gate 128 x 32
    // 168, 153 / 160, 144, 96 x 32 147, 130 / 136, 118; chained 256 x 32 150 - 165 / 160, 96 x 32 105 - 110 / 99.  Not below 1.25 MB a sub-batch (128 x 32 124, 106 - 113 / 129,
    // 115), not for the BF16 state, whose decode kernel needs the SMs more (199, 184 / 216, 199), and not in long chained calls (512 x 32 302 / 321).
    uint64_t next_bytes = 0;
    for (int i = 0; c + 1 < PIPE_CHUNKS && i < 5; i++) next_bytes += 2 * (lo[c + 2] - lo[c + 1]) * per_seq[i];
    if (ok && mapped && !shape->state_bf16 && next_bytes >= 1250000 && (!chained || next_bytes < 4000000)) {
      head_start_kernel<<<1, 32, 0, st>>>();
      ok = cudaGetLastError() == cudaSuccess;
    }
    if (!ok) break;
    lq_shape sub = *shape;
    sub.batch = static_cast<int>(nb);
    lq_state ss = *state;
    ss.heads += b0 * Hv * (shape->state_bf16 ? (uint64_t)BF16W_HEAD_BYTES : (uint64_t)head_bytes(shape->r));
    ss.records = static_cast<char *>(ss.records) + b0 * Hv * shape->W * record_floats(diag) * (shape->rec16 ? 2 : 4);
    if (ss.decays) ss.decays += b0 * Hv * shape->W;
    ss.win_pos += b0;
    rc = decode_step_impl(&sub, &ss, q_d + b0 * eqk, k_d + b0 * eqk, v_d + b0 * ev, b_d + b0 * eb, a_d + b0 * ea,
                          o_d + b0 * ev, stream, hp->done[c], c);
    if (rc != LQ_OK) break;
    ok = cudaStreamWaitEvent(hp->s_out, hp->done[c], 0) == cudaSuccess &&
         cudaMemcpyAsync(o_h + b0 * ev, o_d + b0 * ev, 4 * nb * ev, cudaMemcpyDeviceToHost, hp->s_out) == cudaSuccess;
  }
  if (ok && rc == LQ_OK) {                   // the windows that became full, of all sub-batches together
    Params p = make_params(shape, state);
    rc = launch_boundary<0>(shape, p, st, (long)shape->batch * shape->heads_v / shape->W);
  }
  // join: whatever was put on the side streams is waited for by `stream`, also after an error above
  // (`stream` has waited for every copy-in of this call already, sub-batch by sub-batch, unless an error cut the
  // loop above short)
  bool joined = cudaEventRecord(hp->out, hp->s_out) == cudaSuccess && cudaStreamWaitEvent(st, hp->out, 0) == cudaSuccess;
  if (rc != LQ_OK || !ok)
    joined = cudaEventRecord(hp->out, hp->s_in) == cudaSuccess && cudaStreamWaitEvent(st, hp->out, 0) == cudaSuccess &&
             joined;
  if (rc != LQ_OK) return rc;
  if (!ok || !joined) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  hp->chain = true;
  hp->stage = stage;
  hp->stream = st;
  std::copy(layout, layout + 5, hp->layout);
  return LQ_OK;
}

// ---------------------------------------------------------------------------------------------
// Host-buffer decode step without a caller-supplied staging buffer: the staging is this array.
// It is a device object of the library: every GPU that loads the library carries it until exit.  In host
// code the name below is only a handle; the device address comes from cudaGetSymbolAddress, looked up once
// per device and cached.
// ---------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_static_stage[LQ_STATIC_STAGE_BYTES];

static lq_status static_stage_address(void **out) {
  constexpr int MAX_DEVICES = 64;
  static std::atomic<void *> cached[MAX_DEVICES];
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  void *ptr = cached[dev].load(std::memory_order_acquire);
  if (!ptr) {                                 // first call on this device (it is the current device)
    if (cudaGetSymbolAddress(&ptr, g_static_stage) != cudaSuccess || !ptr) {
      cudaGetLastError();
      return LQ_ERR_CUDA;
    }
    cached[dev].store(ptr, std::memory_order_release);   // two racing first calls store the same address
  }
  *out = ptr;
  return LQ_OK;
}

lq_status lq_decode_step_host_static(const lq_shape *shape, const lq_state *state, const uint16_t *q_h,
                                     const uint16_t *k_h, const uint16_t *v_h, const uint16_t *beta_h,
                                     const uint16_t *alpha_h, float *o_h, lq_stream stream) {
  lq_status rc = check_shape(shape);
  if (rc != LQ_OK) return rc;
  const uint64_t need = lq_decode_stage_bytes(shape);
  if (need > LQ_STATIC_STAGE_BYTES) return LQ_ERR_TOO_LARGE;
  if ((rc = check_state(shape, state, true)) != LQ_OK) return rc;     // before the clearing below is enqueued
  if (!q_h || !k_h || !v_h || !beta_h || !alpha_h || !o_h) return LQ_ERR_NULL;
  void *stage = nullptr;
  if ((rc = static_stage_address(&stage)) != LQ_OK) return rc;
  if (shape->batch == 0) return LQ_OK;
  // The array still holds the previous call's staging.  The inputs are overwritten in full by this call's
  // copies; the output region is cleared, so that rows no kernel writes (sequences with a full window on
  // entry) do not leak an earlier call's results into o_h.  The output region is the last one in the buffer.
  const uint64_t out_bytes = 4ull * shape->batch * shape->heads_v * shape->d_v;
  unsigned char *out_region = static_cast<unsigned char *>(stage) + (need - (out_bytes + 255) / 256 * 256);
  if (cudaMemsetAsync(out_region, 0, out_bytes, reinterpret_cast<cudaStream_t>(stream)) != cudaSuccess) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  // always through the staging buffer, so that the cleared output region is what reaches o_h for such rows
  return host_step_impl(shape, state, q_h, k_h, v_h, beta_h, alpha_h, o_h, stage, stream, false);
}

lq_status lq_window_flush(const lq_shape *shape, const lq_state *state, int force, lq_stream stream) {
  lq_status rc = check_shape(shape);
  if (rc != LQ_OK) return rc;
  if ((rc = check_state(shape, state, true)) != LQ_OK) return rc;
  Params p = make_params(shape, state);
  p.force = force ? 1 : 0;
  // how many are due: all, forced; else unknown, and taken as too few for what pays with a boundary or more for every CTA (256 x 32
  // heads, the windows of one sequence full: 8.1 us as if all were due, 6.8 so; those of all full: 303 / 314)
  const long nh = (long)shape->batch * shape->heads_v;
  return launch_boundary<0>(shape, p, reinterpret_cast<cudaStream_t>(stream), force ? nh : std::min(nh, 2L * sm_count() - 1));
}

lq_status lq_quantize_state(const lq_shape *shape, const float *S, const lq_state *state, lq_stream stream) {
  lq_status rc = check_shape(shape);
  if (rc != LQ_OK) return rc;
  if ((rc = check_state(shape, state, false)) != LQ_OK) return rc;
  if ((rc = check_ptrs({S})) != LQ_OK) return rc;
  Params p = make_params(shape, state);
  p.S = const_cast<float *>(S);
  return launch_boundary<1>(shape, p, reinterpret_cast<cudaStream_t>(stream), (long)shape->batch * shape->heads_v);
}

lq_status lq_dequantize_state(const lq_shape *shape, const lq_state *state, float *S, lq_stream stream) {
  lq_status rc = check_shape(shape);
  if (rc != LQ_OK) return rc;
  if ((rc = check_state(shape, state, true)) != LQ_OK) return rc;
  if ((rc = check_ptrs({S})) != LQ_OK) return rc;
  Params p = make_params(shape, state);
  p.S = S;
  return launch_boundary<2>(shape, p, reinterpret_cast<cudaStream_t>(stream), (long)shape->batch * shape->heads_v);
}

static lq_status ref_step(const lq_shape *shape, float *S, uint16_t *S16, const uint16_t *q, const uint16_t *k,
                          const uint16_t *v, const uint16_t *beta, const uint16_t *alpha, float *o, lq_stream stream) {
  lq_shape s = *shape;
  s.W = 1; s.r = 0; s.n_iter = 1; s.state_bf16 = 0;      // unused by the baseline
  lq_status rc = check_shape(&s);
  if (rc != LQ_OK) return rc;
  if ((rc = check_ptrs({S ? (const void *)S : (const void *)S16, q, k, v, o})) != LQ_OK) return rc;
  if ((rc = check_scalar_ptrs({beta}, 2)) != LQ_OK) return rc;
  if ((rc = s.gate == LQ_GATE_DIAG ? check_ptrs({alpha}) : check_scalar_ptrs({alpha}, 2)) != LQ_OK) return rc;
  Params p = make_params(&s, nullptr);
  p.S = S; p.S16 = S16; p.q = q; p.k = k; p.v = v; p.beta = beta; p.alpha = alpha; p.o = o;
  const int nh = s.batch * s.heads_v;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const bool diag = s.gate == LQ_GATE_DIAG;
  if (S16) return diag ? launch(ref_kernel<LQ_GATE_DIAG, true>, nh, 256, 0, st, p)
                       : launch(ref_kernel<LQ_GATE_SCALAR, true>, nh, 256, 0, st, p);
  return diag ? launch(ref_kernel<LQ_GATE_DIAG, false>, nh, 256, 0, st, p)
              : launch(ref_kernel<LQ_GATE_SCALAR, false>, nh, 256, 0, st, p);
}

lq_status lq_ref_decode_step_f32(const lq_shape *shape, float *S, const uint16_t *q, const uint16_t *k,
                                 const uint16_t *v, const uint16_t *beta, const uint16_t *alpha, float *o,
                                 lq_stream stream) {
  if (!shape) return LQ_ERR_NULL;
  if (!S) return LQ_ERR_NULL;
  return ref_step(shape, S, nullptr, q, k, v, beta, alpha, o, stream);
}

lq_status lq_ref_decode_step_bf16(const lq_shape *shape, uint16_t *S, const uint16_t *q, const uint16_t *k,
                                  const uint16_t *v, const uint16_t *beta, const uint16_t *alpha, float *o,
                                  lq_stream stream) {
  if (!shape) return LQ_ERR_NULL;
  if (!S) return LQ_ERR_NULL;
  return ref_step(shape, nullptr, S, q, k, v, beta, alpha, o, stream);
}

static lq_status convert_state(const lq_shape *shape, const lq_state_arrays *arr, const lq_state *state, lq_stream stream,
                               bool import) {
  lq_status rc = check_shape(shape);
  if (rc != LQ_OK) return rc;
  if (shape->state_bf16) return LQ_ERR_UNSUPPORTED;
  if ((rc = check_state(shape, state, true)) != LQ_OK) return rc;
  if (!arr) return LQ_ERR_NULL;
  if ((rc = check_ptrs({arr->codes, arr->col_scale, arr->row_smooth, arr->buf_k, arr->buf_u, arr->buf_a})) != LQ_OK) return rc;
  if (shape->r > 0 && (rc = check_ptrs({arr->comp_k, arr->comp_u})) != LQ_OK) return rc;
  if ((rc = check_scalar_ptrs({arr->win_pos}, 4)) != LQ_OK) return rc;
  Params p = make_params(shape, state);
  const int nh = shape->batch * shape->heads_v;
  const int diag = shape->gate == LQ_GATE_DIAG ? 1 : 0;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (nh <= 0) return LQ_OK;
  if (import) convert_state_kernel<true><<<nh, 256, 0, st>>>(p, *arr, diag);
  else convert_state_kernel<false><<<nh, 256, 0, st>>>(p, *arr, diag);
  return cudaGetLastError() == cudaSuccess ? LQ_OK : LQ_ERR_CUDA;
}

lq_status lq_import_state(const lq_shape *shape, const lq_state_arrays *src, const lq_state *dst, lq_stream stream) {
  return convert_state(shape, src, dst, stream, true);
}

lq_status lq_export_state(const lq_shape *shape, const lq_state *src, const lq_state_arrays *dst, lq_stream stream) {
  return convert_state(shape, dst, src, stream, false);
}

lq_status lq_check_device(int *flags) {
  if (!flags) return LQ_ERR_NULL;
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_device_error, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  *flags = v;
  return LQ_OK;
}

lq_status lq_clear_device_flags(void) {
  const int zero = 0;
  if (cudaMemcpyToSymbol(g_device_error, &zero, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return LQ_ERR_CUDA;
  }
  return LQ_OK;
}

uint64_t lq_static_stage_bytes(void) { return LQ_STATIC_STAGE_BYTES; }

}  // extern "C"

// One warp waits, with a limit of a few dozen polls, on a barrier that nothing will ever complete: the wait
// must come back with "gave up", which is reported like in the decode kernel (error flag, bit 3 here).
namespace {
__global__ void bounded_wait_probe_kernel() {
  __shared__ __align__(8) unsigned long long bar;
  const uint32_t b = lq::smem_addr(&bar);
  if (threadIdx.x == 0) lq::mbar_init(b, 1);
  __syncwarp();
  const bool done = lq::mbar_wait<64>(b, 0);
  if (!done && threadIdx.x == 0) atomicOr(&lq::g_device_error, 8);
}
}  // namespace

extern "C" {

lq_status lq_selftest_bounded_wait(lq_stream stream) {
  bounded_wait_probe_kernel<<<1, 32, 0, reinterpret_cast<cudaStream_t>(stream)>>>();
  return cudaGetLastError() == cudaSuccess ? LQ_OK : LQ_ERR_CUDA;
}

#ifdef LQ_TIMING
// development aid: copies the time stamps of the last four steps to host memory (4 x 2 x 6 x 1024 values)
int lq_debug_timeline(unsigned long long *out) {
  return cudaMemcpyFromSymbol(out, g_timeline, sizeof(unsigned long long) * 4 * 2 * 6 * 1024) != cudaSuccess;
}
// development aid: copies the phase counters to host memory and clears them
int lq_debug_phase_cycles(unsigned long long *out) {
  unsigned long long zero[64] = {0};
  if (cudaMemcpyFromSymbol(out, g_phase_cycles, sizeof(zero)) != cudaSuccess) return 1;
  return cudaMemcpyToSymbol(g_phase_cycles, zero, sizeof(zero)) != cudaSuccess;
}
#endif

int lq_step_launches(const lq_shape *shape, const lq_state *state) {
  const int most = lq_decode_launches(shape);
  lq_status rc = LQ_OK;
  return most > 1 && state && launch_merged(shape, make_params(shape, state), nullptr, &rc, false) ? 1 : most;
}

int lq_decode_launches(const lq_shape *shape) { return check_shape(shape) == LQ_OK && shape->batch > 0 ? one_launch(shape) ? 1 : 2 : 0; }

const char *lq_status_string(lq_status status) {
  switch (status) {
    case LQ_OK: return "ok";
    case LQ_ERR_NULL: return "null pointer";
    case LQ_ERR_SHAPE: return "invalid shape";
    case LQ_ERR_ALIGN: return "pointer not 16-byte aligned";
    case LQ_ERR_UNSUPPORTED: return "shape not supported";
    case LQ_ERR_CUDA: return "CUDA runtime error";
    case LQ_ERR_TOO_LARGE: return "request exceeds the built-in scratch buffer";
  }
  return "unknown status";
}

int lq_version(void) { return 7; }

}  // extern "C"
