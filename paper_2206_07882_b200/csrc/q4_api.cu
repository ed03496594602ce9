// C ABI of the library (see include/q4rnnt.h): argument checking on the host, argument
// blocks for the kernels, launch sequencing.  Nothing here waits for the device but q4_poll_status and
// q4_search_plan_destroy, and nothing allocates but a search plan.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include "q4_internal.h"

using namespace q4;

#define Q4_TRY(expr)                               \
  do {                                             \
    cudaError_t e__ = (expr);                      \
    if (e__ != cudaSuccess) return Q4_ERR_CUDA;    \
  } while (0)
#define Q4_CHECK(expr)        \
  do {                        \
    int r__ = (expr);         \
    if (r__ != Q4_OK) return r__; \
  } while (0)

namespace {

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline cudaStream_t S(q4_stream s) { return reinterpret_cast<cudaStream_t>(s); }

int check_act(const q4_act* a) {
  if (!a) return Q4_ERR_NULL;
  if (a->bits != 4 && a->bits != 8) return Q4_ERR_BITS;
  if (!a->is_signed && a->bits != 4) return Q4_ERR_BITS;  // unsigned codes exist at 4 bit only
  if (!a->is_signed && (a->zero_point < 0 || a->zero_point > 15)) return Q4_ERR_DIM;
  if (a->is_signed && a->zero_point != 0) return Q4_ERR_DIM;
  if (!(a->scale > 0.0f) || !(a->inv_scale > 0.0f)) return Q4_ERR_DIM;
  return Q4_OK;
}

int check_mat(const q4_mat* m, int rows, int k_pad_expected) {
  if (!m || !m->q || !m->scale) return Q4_ERR_NULL;
  if (m->bits != 2 && m->bits != 4 && m->bits != 8) return Q4_ERR_BITS;
  if (m->rows <= 0 || m->k <= 0 || m->k_pad < m->k) return Q4_ERR_DIM;
  if (m->k_pad % (m->bits == 2 ? 64 : 32) != 0) return Q4_ERR_ALIGN;   // rows are 16-byte multiples
  if (rows > 0 && m->rows != rows) return Q4_ERR_DIM;
  if (k_pad_expected > 0 && m->k_pad != k_pad_expected) return Q4_ERR_DIM;
  if (!aligned16(m->q) || (reinterpret_cast<uintptr_t>(m->scale) & 3u)) return Q4_ERR_ALIGN;
  return Q4_OK;
}

// Hypothesis rows up to which a search keeps the recurrent sums per state row (see search_keeps_sums).  They take 16 H bytes a
// row and layer through memory instead of a gather and products in the step's longest chain, and the products
// that make them take the SMs from the output heads and the selection when there are many: with 1024, 1024 and 2048 cells,
// 160 frames, labels in half of the iterations, ms with / without: 64 rows 4.06 / 5.05, 256 rows 4.31 / 4.87, 384 rows
// 8.38 / 8.89, 512 rows 9.94 / 9.86, 1024 rows 12.0 / 9.6.  Without the fused output heads (D = 256, up to 2048 labels) the
// heads are launches of their own with tiles for every SM, and the line lies lower: 100 frames, D = 128, 252 rows 4.89 /
// 4.87 with labels all the way and 7.30 / 7.63 in half of the iterations, 384 rows 6.01 / 5.31 and 8.64 / 9.06; 4096 labels,
// 384 rows 10.7 / 9.9 and 12.1 / 11.5.
constexpr int SUMS_MAX_ROWS = 384, SUMS_MAX_ROWS_PLAIN = 256;
constexpr bool fused_heads(int V, int D) { return D == 256 && V <= 2048; }   // 256-wide bottleneck, one cluster per row tile
constexpr int sums_max_rows(int V, int D) { return fused_heads(V, D) ? SUMS_MAX_ROWS : SUMS_MAX_ROWS_PLAIN; }

// Rows that the tensor-core paths can address: a grid has 65535 row tiles, and the gather counts 32-code pieces in 32
// bits (rows of k codes).  More go to the general kernels, which walk any number.
inline bool mma_rows(long long rows, int k) {
  const long long tiles = (rows + 127) / 128;
  return tiles <= 65535 && tiles * 128 * (k / 32) <= INT32_MAX;
}

inline long long row_bytes(int k_pad, int bits) { return (long long)k_pad * bits / 8; }

GemmArgs gemm_args(const void* x, long long x_stride, const int32_t* x_idx, const q4_act& xa, int M,
                   const q4_mat& w, const float* bias, void* out, long long out_stride,
                   const int32_t* out_idx) {
  GemmArgs g;
  memset(&g, 0, sizeof(g));
  g.x.base = static_cast<const uint8_t*>(x);
  g.x.stride = x_stride;
  g.x.idx = x_idx;
  g.x_signed = xa.is_signed;
  g.x_zp = xa.zero_point;
  g.x_bits = xa.bits;
  g.w_bits = w.bits;
  g.M = M;
  g.w = static_cast<const uint8_t*>(w.q);
  g.w_scale = w.scale;
  g.bias = bias;
  g.J = w.rows;
  g.k_pad = w.k_pad;
  g.x_scale = xa.scale;
  g.out = out;
  g.out_stride = out_stride;
  g.out_idx = out_idx;
  return g;
}

}  // namespace

extern "C" {

int q4_version(void) { return 1; }

int q4_timing_set(uint32_t tag_mask, void** start_events, void** stop_events, int32_t* tags_out,
                  int32_t capacity) {
  if (tag_mask != 0 && (!start_events || !stop_events || !tags_out || capacity <= 0)) return Q4_ERR_NULL;
  timing_set(tag_mask, reinterpret_cast<cudaEvent_t*>(start_events),
             reinterpret_cast<cudaEvent_t*>(stop_events), tags_out, tag_mask ? capacity : 0);
  return Q4_OK;
}
int q4_timing_count(void) { return timing_count(); }
int64_t q4_launch_count(void) { return g_launches; }
int64_t q4_quantizer_calls(int32_t reset) {
  const int64_t n = g_quant_calls;
  if (reset) g_quant_calls = 0;
  return n;
}
static int g_select_exact = 0;
static int select_exact_only() { return g_select_exact; }
int q4_beam_select_exact_set(int32_t enabled) {
  const int prev = g_select_exact;
  g_select_exact = enabled ? 1 : 0;
  return prev;
}
int q4_test_wait_expiry_set(int32_t skip_producer, uint32_t wait_limit) {
  test_wait_expiry_set(skip_producer == 2 ? 2 : skip_producer ? 1 : 0, wait_limit);
  return Q4_OK;
}
int q4_encoder_time_slicing_set(int32_t enabled) { return enc_recurrent_sliced_set(enabled ? 1 : 0); }
int q4_encoder_recurrence_plan(int32_t T, int32_t B, int32_t dirs, int32_t H, int32_t w_bits, int32_t hid_bits,
                               int32_t per_sequence_scale, int32_t* out) {
  if (!out) return Q4_ERR_NULL;
  if (T <= 0 || B <= 0 || dirs < 1 || dirs > 2 || H <= 0) return Q4_ERR_DIM;
  const EncRecPlan p = enc_recurrent_plan(T, B, dirs, H, w_bits, hid_bits, true, per_sequence_scale != 0, false, true);
  out[0] = p.kernel;
  out[1] = p.groups_per_cluster;
  out[2] = p.ncl[0];
  out[3] = p.ncl[1];
  out[4] = p.sliced[0];
  out[5] = p.sliced[1];
  out[6] = p.groups;
  out[7] = p.max_clusters;
  for (int j = 0; j < 9; ++j) out[8 + j] = p.win[j];
  return Q4_OK;
}
int q4_dependent_launch_set(int32_t enabled) {
  const int prev = g_dependent_launch;
  g_dependent_launch = enabled ? 1 : 0;
  return prev;
}

int q4_act_symmetric(float alpha, int32_t bits, q4_act* out) {
  if (!out) return Q4_ERR_NULL;
  if (bits != 4 && bits != 8) return Q4_ERR_BITS;
  if (!(alpha > 0.0f)) return Q4_ERR_DIM;
  const volatile float qmax = (float)((1 << (bits - 1)) - 1);
  const volatile float s = alpha / qmax;
  const volatile float inv = 1.0f / s;
  out->scale = s;
  out->inv_scale = inv;
  out->zero_point = 0;
  out->bits = bits;
  out->is_signed = 1;
  return Q4_OK;
}

int q4_act_asymmetric(float lo, float hi, int32_t bits, q4_act* out) {
  if (!out) return Q4_ERR_NULL;
  if (bits != 4) return Q4_ERR_BITS;
  if (!(hi > lo)) return Q4_ERR_DIM;
  const volatile float qmax = (float)((1 << bits) - 1);
  const volatile float s = (hi - lo) / qmax;
  const volatile float inv = 1.0f / s;
  const volatile float zr = -lo / s;
  float z = nearbyintf(zr);
  z = fminf(fmaxf(z, 0.0f), qmax);
  out->scale = s;
  out->inv_scale = inv;
  out->zero_point = (int32_t)z;
  out->bits = bits;
  out->is_signed = 0;
  return Q4_OK;
}

size_t q4_workspace_bytes(int32_t call_id, const int32_t* dims, int32_t ndims) {
  if (!dims) return 0;
  if (call_id == Q4_WS_LSTM_LAYER && ndims >= 4) {
    const size_t T = dims[0], B = dims[1], D = dims[2], H = dims[3];
    const size_t K = ndims >= 5 ? dims[4] : 0;
    size_t n = 256;                                      // status word
    n += align_up(D * T * B * 4 * H * sizeof(int32_t));  // input accumulators
    n += align_up(D * 2 * B * H);                        // recurrent codes, double buffered
    n += align_up(D * B * H * sizeof(float));            // cell state
    if (K > 0) {                                         // int8 operands of the tensor-core GEMM
      n += align_up(T * B * K);
      n += align_up(D * 4 * H * K);
      n += align_up(D * 4 * H * H);                      // resident recurrent weights, int8
      n += 3 * align_up(D * 4 * H * sizeof(float));      // row scales and bias, cell-major
    }
    return n;
  }
  if (call_id == Q4_WS_JOINT && ndims >= 2) {
    const size_t N = dims[0], D = dims[1];
    size_t n = align_up(N * D * sizeof(float)) + align_up(N * D);
    if (ndims >= 3) {   // tensor-core path: status word, int8 copies of the hidden codes and of z
      const size_t Np = (N + 127) / 128 * 128, Hp = dims[2];
      n += 256 + align_up(Np * Hp) + align_up(Np * D);
    }
    return n;
  }
  if (call_id == Q4_WS_LSTM_STEP && ndims >= 3) {   // status word, int8 copies of x and h rows
    const size_t Np = ((size_t)dims[0] + 127) / 128 * 128;
    return 256 + align_up(Np * (size_t)dims[1]) + align_up(Np * (size_t)dims[2]);
  }
  if (call_id == Q4_WS_LINEAR && ndims >= 2) {      // status word, int8 copy of the input rows
    const size_t Np = ((size_t)dims[0] + 127) / 128 * 128;
    return 256 + align_up(Np * (size_t)dims[1]);
  }
  if (call_id == Q4_WS_BEAM && ndims >= 4) {
    const size_t N = (size_t)dims[0] * dims[1], V = dims[2], D = dims[3];
    size_t n = 256 + align_up(N * D) * 3 + align_up(N * V * sizeof(float)) + align_up(N * sizeof(int32_t));
    if (ndims >= 8) {  // int8 operand scratch of the tensor-core path
      const size_t Np = (N + 127) / 128 * 128;
      const size_t E = dims[4], Hp = dims[5], Hs = dims[6], Ht = dims[7];
      const size_t Hmax = Hp > Hs ? (Hp > Ht ? Hp : Ht) : (Hs > Ht ? Hs : Ht);
      n += 3 * align_up(Np * E) + align_up(Np * Hp) + align_up(Np * Hs) + 2 * align_up(Np * Ht);  // gathered x / h operands
      (void)Hmax;
      n += align_up(Np * Hp) + align_up(Np * Hs) + 2 * align_up(Np * Ht); // new cell outputs, int8
      n += 3 * align_up(Np * D);                                         // bottleneck codes, z codes
      if (ndims >= 9 && dims[8] > 0 && N <= (size_t)sums_max_rows((int)V, (int)D)) {   // recurrent sums of every state row
        const size_t R = (size_t)dims[0] * dims[8];
        n += align_up(R * 4 * Hp * sizeof(float)) + align_up(R * 4 * Hs * sizeof(float)) + 2 * align_up(R * 4 * Ht * sizeof(float));
      }
    }
    return n;
  }
  return 0;
}

int q4_poll_status(const int32_t* device_status, q4_stream stream) {
  if (!device_status) return Q4_ERR_NULL;
  int32_t h = 0;
  if (cudaMemcpyAsync(&h, device_status, sizeof(h), cudaMemcpyDeviceToHost, S(stream)) != cudaSuccess)
    return Q4_ERR_CUDA;
  if (cudaStreamSynchronize(S(stream)) != cudaSuccess) return Q4_ERR_CUDA;
  return h == 0 ? Q4_OK : (int)h;
}

int quantize_pack_int4(const void* x, int32_t x_is_fp16, int64_t rows, int32_t k, int32_t k_pad,
                       const q4_act* act, int32_t mode, int32_t n_groups,
                       const float* per_row_scale, void* q_out, float* group_scale_out,
                       q4_stream stream) {
  if (!act) return Q4_ERR_NULL;
  if (rows < 0 || k <= 0 || k_pad < k) return Q4_ERR_DIM;
  if (rows > 0 && (!x || !q_out)) return Q4_ERR_NULL;
  if (k_pad % 32 != 0 || !aligned16(q_out)) return Q4_ERR_ALIGN;
  if (mode < 0 || mode > 2) return Q4_ERR_UNSUPPORTED;
  if (act->bits != 4 && act->bits != 8 && !(act->bits == 2 && mode != 0)) return Q4_ERR_BITS;   // 2 bit: weights
  if (act->bits == 2 && k_pad % 64 != 0) return Q4_ERR_ALIGN;
  q4_act a = *act;
  if (mode == 0) {
    Q4_CHECK(check_act(act));
  } else {
    a.is_signed = 1;
    a.zero_point = 0;
    a.scale = a.inv_scale = 1.0f;
    if (mode == 1 && (!group_scale_out || n_groups <= 0)) return group_scale_out ? Q4_ERR_DIM : Q4_ERR_NULL;
    if (mode == 2 && !per_row_scale) return Q4_ERR_NULL;
  }
  if (rows == 0) return Q4_OK;
  TagScope tag(TAG_QUANT);
  if (mode != 2) ++g_quant_calls;   // an activation tensor (weights are quantized once, off line)
  Q4_TRY(launch_quantize(x, x_is_fp16 != 0, rows, k, k_pad, a, mode, n_groups, per_row_scale,
                         static_cast<uint8_t*>(q_out), group_scale_out, S(stream)));
  return Q4_OK;
}

int q4_linear_forward(const void* xq, const q4_act* x_act, int32_t M, const q4_mat* w,
                      const float* bias, float* out, int32_t* dbg_acc, const void* prepared,
                      void* workspace, size_t workspace_bytes, q4_stream stream) {
  if (!xq || !out) return Q4_ERR_NULL;
  Q4_CHECK(check_act(x_act));
  Q4_CHECK(check_mat(w, 0, 0));
  if (M < 0) return Q4_ERR_DIM;
  if (!aligned16(xq) || !aligned16(out)) return Q4_ERR_ALIGN;
  {
    const int32_t wd[2] = {M, w->k_pad};
    if (prepared && workspace && !dbg_acc && M >= 128 && mma_rows(M, w->k_pad) && aligned16(workspace) && aligned16(prepared) &&
        workspace_bytes >= q4_workspace_bytes(Q4_WS_LINEAR, wd, 2)) {
      // tensor cores: int8 copy of the input rows, then the tiled GEMM on the prepared int8 weights
      cudaStream_t s = S(stream);
      uint8_t* ws = static_cast<uint8_t*>(workspace);
      int32_t* status = reinterpret_cast<int32_t*>(ws);
      int8_t* x8 = reinterpret_cast<int8_t*>(ws + 256);
      const int Mp = (M + 127) / 128 * 128;
      TagScope tag(TAG_LINEAR);
      // the gather clears the status block and may start under the tail of whatever kernel precedes the call
      UnpackJobs uj;
      memset(&uj, 0, sizeof(uj));
      uj.n_rows = M;
      uj.n_rows_pad = Mp;
      uj.zero_tail = 1;
      uj.clear64 = status;
      add_unpack_job(uj, xq, row_bytes(w->k_pad, x_act->bits), nullptr, *x_act, w->k_pad, x8);
      Q4_TRY(launch_unpack_multi(uj, s, true));
      Q4_TRY(launch_mma_gemm(x8, w->k_pad, M, static_cast<const int8_t*>(prepared), w->k_pad, w->rows, w->k_pad,
                             EPI_F32, out, w->rows, nullptr, w->scale, bias, x_act->scale, nullptr, status, nullptr,
                             s, true));   // programmatic dependent of the gather before it
      return Q4_OK;
    }
  }
  GemmArgs g = gemm_args(xq, row_bytes(w->k_pad, x_act->bits), nullptr, *x_act, M, *w, bias, out,
                         w->rows, nullptr);
  g.dbg_acc = dbg_acc;
  TagScope tag(TAG_LINEAR);
  Q4_TRY(launch_gemm(g, EPI_F32, S(stream)));
  return Q4_OK;
}

static int check_lstm(const q4_mat* w_ih, const q4_mat* w_hh, const q4_act* x_act,
                      const q4_act* hid_act, int* H_out) {
  Q4_CHECK(check_act(x_act));
  Q4_CHECK(check_act(hid_act));
  if (!hid_act->is_signed) return Q4_ERR_UNSUPPORTED;
  Q4_CHECK(check_mat(w_ih, 0, 0));
  Q4_CHECK(check_mat(w_hh, 0, 0));
  if (w_ih->rows != w_hh->rows || w_ih->rows % 4 != 0) return Q4_ERR_DIM;
  const int H = w_ih->rows / 4;
  if (w_hh->k != H || w_hh->k_pad != H) return Q4_ERR_DIM;
  if (H % 32 != 0) return Q4_ERR_ALIGN;
  *H_out = H;
  return Q4_OK;
}

static void fill_lstm_weights(LstmArgs& a, const q4_mat& w_ih, const q4_mat& w_hh, const float* bias,
                              const q4_act& x_act, const q4_act& hid_act) {
  a.x_signed = x_act.is_signed;
  a.x_zp = x_act.zero_point;
  a.x_bits = x_act.bits;
  a.wih_bits = w_ih.bits;
  a.whh_bits = w_hh.bits;
  a.kx_pad = w_ih.k_pad;
  a.x_scale = x_act.scale;
  a.w_ih = static_cast<const uint8_t*>(w_ih.q);
  a.s_wih = w_ih.scale;
  a.w_hh = static_cast<const uint8_t*>(w_hh.q);
  a.s_whh = w_hh.scale;
  a.bias = bias;
  a.H = w_ih.rows / 4;
  a.kh_pad = w_hh.k_pad;
  a.hid_act = hid_act;
  a.out_act = hid_act;
}

int qlstm_step(const void* xq, const q4_act* x_act, const int32_t* x_row_idx, const void* hq_in,
               const float* c_in, int32_t N, const q4_mat* w_ih, const q4_mat* w_hh,
               const float* bias, const q4_act* hid_act, void* hq_out, float* c_out,
               float* h_f32_out, int32_t* dbg_acc_ih, int32_t* dbg_acc_hh, const void* prepared,
               void* workspace, size_t workspace_bytes, q4_stream stream) {
  if (!xq || !hq_in || !c_in || !c_out) return Q4_ERR_NULL;
  if (!hq_out && !h_f32_out) return Q4_ERR_NULL;   // Inner placement needs the real-valued output
  int H = 0;
  Q4_CHECK(check_lstm(w_ih, w_hh, x_act, hid_act, &H));
  if (N < 0) return Q4_ERR_DIM;
  if (hq_in == hq_out) return Q4_ERR_UNSUPPORTED;
  if (!aligned16(xq) || !aligned16(hq_in) || !aligned16(hq_out)) return Q4_ERR_ALIGN;
  if (N == 0) return Q4_OK;
  if (hq_out) ++g_quant_calls;   // the one quantizer call at the cell output (Outer placement)
  if (!dbg_acc_ih && !dbg_acc_hh && skinny_lstm_supported(N, H, w_ih->k_pad, w_ih->bits, w_hh->bits, *x_act, *hid_act)) {
    // at most 32 rows of 4-bit codes: the kernel that reads the packed weights once (1024 cells, 16 rows:
    // 4.6 us of device time; two launches on the tensor cores 8.2, the DP4A kernel 24)
    SkinnyLstmArgs k;
    memset(&k, 0, sizeof(k));
    k.N = N;
    k.H = H;
    k.Kx = w_ih->k_pad;
    k.w_ih = static_cast<const uint8_t*>(w_ih->q);
    k.w_hh = static_cast<const uint8_t*>(w_hh->q);
    k.s_wih = w_ih->scale;
    k.s_whh = w_hh->scale;
    k.bias = bias;
    k.x = static_cast<const uint8_t*>(xq);
    k.x_stride = row_bytes(w_ih->k_pad, 4);
    k.x_idx = x_row_idx;
    k.x_signed = x_act->is_signed;
    k.x_zp = x_act->zero_point;
    k.x_scale = x_act->scale;
    k.hid_act = *hid_act;
    k.hq_in = static_cast<const uint8_t*>(hq_in);
    k.c_in = c_in;
    k.hq_out = static_cast<uint8_t*>(hq_out);
    k.c_out = c_out;
    k.h_f32 = h_f32_out;
    TagScope tag(TAG_PRED_LSTM);
    Q4_TRY(launch_skinny_lstm(k, S(stream), true));
    return Q4_OK;
  }
  {
    const int32_t wd[3] = {N, w_ih->k_pad, H};
    if (prepared && workspace && hq_out && H % 128 == 0 && aligned16(workspace) && aligned16(prepared) &&
        mma_rows(N, H > w_ih->k_pad ? H : w_ih->k_pad) &&
        (dbg_acc_ih == nullptr) == (dbg_acc_hh == nullptr) &&
        aligned16(c_in) && aligned16(c_out) && aligned16(h_f32_out) &&   // moved 16 bytes and more at a time
        workspace_bytes >= q4_workspace_bytes(Q4_WS_LSTM_STEP, wd, 3)) {
      // tensor cores, any number of rows (33: 8.4 us of device time, 24.7 on the DP4A kernel): int8 copies of
      // the x rows (gathered) and h rows, then the fused LSTM kernel on the
      // prepared int8 weights (rows 4*cell+gate, scales and bias in the same order)
      cudaStream_t s = S(stream);
      const size_t G = 4 * (size_t)H, Kx = w_ih->k_pad;
      const uint8_t* pb = static_cast<const uint8_t*>(prepared);
      const int8_t* xw8 = reinterpret_cast<const int8_t*>(pb);
      const int8_t* hw8 = xw8 + align_up(G * Kx);
      const float* sc_ih = reinterpret_cast<const float*>(hw8 + align_up(G * H));
      const float* sc_hh = sc_ih + align_up(G * sizeof(float)) / sizeof(float);
      const float* bi = sc_hh + align_up(G * sizeof(float)) / sizeof(float);
      uint8_t* ws = static_cast<uint8_t*>(workspace);
      int32_t* status = reinterpret_cast<int32_t*>(ws);
      const int Np = (N + 127) / 128 * 128;
      int8_t* x8 = reinterpret_cast<int8_t*>(ws + 256);
      int8_t* h8 = x8 + align_up((size_t)Np * Kx);
      TagScope tag(TAG_PRED_LSTM);
      // every kernel of the call is a programmatic dependent of the one before (each waits for its
      // predecessor's completion before it reads anything); the gather clears the status block
      UnpackJobs uj;
      memset(&uj, 0, sizeof(uj));
      uj.n_rows = N;
      uj.n_rows_pad = Np;
      uj.zero_tail = 1;
      uj.clear64 = status;
      add_unpack_job(uj, xq, row_bytes(w_ih->k_pad, x_act->bits), x_row_idx, *x_act, (int)Kx, x8);
      add_unpack_job(uj, hq_in, row_bytes(H, hid_act->bits), nullptr, *hid_act, H, h8);
      Q4_TRY(launch_unpack_multi(uj, s, true));
      MmaLstmArgs a;
      memset(&a, 0, sizeof(a));
      a.N = N;
      a.H = H;
      a.Kx_pad = (int)Kx;
      a.sc_ih = sc_ih;
      a.sc_hh = sc_hh;
      a.bias = bi;
      a.x_scale = x_act->scale;
      a.hid_act = *hid_act;
      a.out_act = *hid_act;
      a.c_in = c_in;
      a.c_out = c_out;
      a.hq_out = static_cast<uint8_t*>(hq_out);
      a.hq_ld = row_bytes(H, hid_act->bits);
      a.h_f32 = h_f32_out;
      a.dbg_ih = dbg_acc_ih;
      a.dbg_hh = dbg_acc_hh;
      a.dbg_ld = 4LL * H;
      a.status = status;
      // programmatic dependent of the gather
      Q4_TRY(launch_mma_lstm(a, x8, (long long)Kx, xw8, (long long)Kx, h8, H, hw8, H, s, true));
      return Q4_OK;
    }
  }
  LstmArgs2 args;
  memset(&args, 0, sizeof(args));
  LstmArgs& a = args.d[0];
  fill_lstm_weights(a, *w_ih, *w_hh, bias, *x_act, *hid_act);
  a.x.base = static_cast<const uint8_t*>(xq);
  a.x.stride = row_bytes(w_ih->k_pad, x_act->bits);
  a.x.idx = x_row_idx;
  a.hin.base = static_cast<const uint8_t*>(hq_in);
  a.hin.stride = row_bytes(H, hid_act->bits);
  a.c_in = c_in;
  a.N = N;
  a.hq_out = static_cast<uint8_t*>(hq_out);
  a.hq_stride = a.hin.stride;
  a.c_out = c_out;
  a.h_f32 = h_f32_out;
  a.dbg_ih = dbg_acc_ih;
  a.dbg_hh = dbg_acc_hh;
  a.dbg_stride = 4LL * H;
  TagScope tag(TAG_PRED_LSTM);
  Q4_TRY(launch_lstm(args, 1, S(stream)));
  return Q4_OK;
}

int qlstm_layer_forward(const void* xq, const q4_act* x_act, const float* x_scale_b, int32_t T,
                        int32_t B, int32_t dirs, const q4_mat* w_ih, const q4_mat* w_hh,
                        const float* const* bias, const q4_act* hid_act, const q4_act* out_act,
                        void* yq, void* hq_n, float* c_n, int32_t* dbg_acc_ih,
                        int32_t* dbg_acc_hh, void* workspace, size_t workspace_bytes,
                        q4_stream stream) {
  if (!xq || !yq || !w_ih || !w_hh || !workspace) return Q4_ERR_NULL;
  if (T <= 0 || B <= 0 || dirs < 1 || dirs > 2) return Q4_ERR_DIM;
  int H = 0;
  for (int d = 0; d < dirs; ++d) {
    int Hd = 0;
    Q4_CHECK(check_lstm(&w_ih[d], &w_hh[d], x_act, hid_act, &Hd));
    if (d == 0) H = Hd;
    if (Hd != H || w_ih[d].k_pad != w_ih[0].k_pad || w_ih[d].bits != w_ih[0].bits) return Q4_ERR_DIM;
  }
  if (!out_act) out_act = hid_act;
  Q4_CHECK(check_act(out_act));
  if (!out_act->is_signed) return Q4_ERR_UNSUPPORTED;
  if (!aligned16(xq) || !aligned16(yq) || !aligned16(workspace)) return Q4_ERR_ALIGN;
  const int32_t dims[5] = {T, B, dirs, H, w_ih[0].k_pad};
  if (workspace_bytes < q4_workspace_bytes(Q4_WS_LSTM_LAYER, dims, 4)) return Q4_ERR_WORKSPACE;
  const long long TB = (long long)T * B;
  // tensor-core input projection when the caller's workspace has room for the int8 operands
  const bool use_mma = TB >= 128 && workspace_bytes >= q4_workspace_bytes(Q4_WS_LSTM_LAYER, dims, 5);

  cudaStream_t s = S(stream);
  const int G = 4 * H;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  int32_t* status = reinterpret_cast<int32_t*>(ws);
  ws += 256;
  int32_t* acc_ih = reinterpret_cast<int32_t*>(ws);
  ws += align_up((size_t)dirs * TB * G * sizeof(int32_t));
  uint8_t* hbuf = ws;  // [dirs][2][B*H bytes]
  ws += align_up((size_t)dirs * 2 * B * H);
  float* cbuf = reinterpret_cast<float*>(ws);  // [dirs][B][H]
  ws += align_up((size_t)dirs * B * H * sizeof(float));
  const int Kx = w_ih[0].k_pad;
  int8_t* x8 = reinterpret_cast<int8_t*>(ws);
  int8_t* w8 = x8 + align_up((size_t)TB * Kx);
  int8_t* whh8 = w8 + align_up((size_t)dirs * G * Kx);
  float* vec_ih = reinterpret_cast<float*>(whh8 + align_up((size_t)dirs * G * H));
  float* vec_hh = vec_ih + align_up((size_t)dirs * G * sizeof(float)) / sizeof(float);
  float* vec_b = vec_hh + align_up((size_t)dirs * G * sizeof(float)) / sizeof(float);
  // persistent recurrence: needs the tensor-core projection (cell-major accumulators)
  const bool persistent = use_mma && enc_recurrent_supported(H, B, dirs);
  const long long hb = row_bytes(H, hid_act->bits);
  const long long yb = row_bytes(dirs * H, out_act->bits);
  const long long xb = row_bytes(w_ih[0].k_pad, x_act->bits);

  // time-parallel input projections for all frames
  if (use_mma) {
    LayerPrep lp;
    memset(&lp, 0, sizeof(lp));
    lp.H = H;
    lp.clear64 = status;
    auto mat = [&](const void* src, int8_t* dst, long long rows, int k_pad, int bits, int is_signed, int zp, int interleave) {
      LayerPrepMat& m = lp.mat[lp.n_mats++];
      m.src = static_cast<const uint8_t*>(src);
      m.dst = dst;
      m.rows = rows;
      m.k_pad = k_pad;
      m.bits = bits;
      m.is_signed = is_signed;
      m.zp = zp;
      m.interleave = interleave;
    };
    auto vec = [&](const float* src, float* dst) {
      lp.vec_src[lp.n_vecs] = src;
      lp.vec_dst[lp.n_vecs++] = dst;
    };
    mat(xq, x8, TB, Kx, x_act->bits, x_act->is_signed, x_act->zero_point, 0);
    for (int d = 0; d < dirs; ++d) {
      mat(w_ih[d].q, w8 + (size_t)d * G * Kx, G, Kx, w_ih[d].bits, 1, 0, persistent ? H : 0);
      if (!persistent) continue;
      mat(w_hh[d].q, whh8 + (size_t)d * G * H, G, H, w_hh[d].bits, 1, 0, H);
      vec(w_ih[d].scale, vec_ih + (size_t)d * G);
      vec(w_hh[d].scale, vec_hh + (size_t)d * G);
      vec(bias ? bias[d] : nullptr, vec_b + (size_t)d * G);
    }
    {
      TagScope tag(TAG_QUANT);
      Q4_TRY(launch_layer_prepare(lp, s, true));
    }
    TagScope tag(TAG_ENC_GEMM);
    Q4_TRY(launch_mma_gemm_i32(x8, (int)TB, w8, G, Kx, dirs, acc_ih, status, s, true));
  } else {
    Q4_TRY(cudaMemsetAsync(status, 0, 256, s));
    for (int d = 0; d < dirs; ++d) {
      TagScope tag(TAG_ENC_GEMM);
      GemmArgs g = gemm_args(xq, xb, nullptr, *x_act, (int)TB, w_ih[d], nullptr,
                             acc_ih + (size_t)d * TB * G, G, nullptr);
      Q4_TRY(launch_gemm(g, EPI_I32, s));
    }
  }
  // per step and direction one quantizer call at the cell output; a second one where the next
  // layer wants the same real value at another precision
  g_quant_calls += (int64_t)T * dirs *
                   ((out_act->bits == hid_act->bits && out_act->scale == hid_act->scale) ? 1 : 2);
  if (persistent) {
    EncRecArgs ra;
    memset(&ra, 0, sizeof(ra));
    ra.T = T;
    ra.B = B;
    ra.H = H;
    ra.dirs = dirs;
    ra.w_bits = w_hh[0].bits;
    ra.status = status;
    ra.x_scale = x_act->scale;
    ra.x_scale_b = x_scale_b;
    ra.hid_act = *hid_act;
    ra.out_act = *out_act;
    ra.yq_ld = yb;
    ra.dbg_ld = (long long)dirs * G;
    // scratch of the time-sliced kernel: counters in the status block (zeroed above), the shared
    // group's state in the buffers the step-by-step path would use
    ra.flags = status + 16;
    for (int d = 0; d < dirs && B >= 8; ++d) {
      ra.hand_h[d] = hbuf + (size_t)d * 2 * B * H;
      ra.hand_c[d] = cbuf + (size_t)d * B * H;
    }
    for (int d = 0; d < dirs; ++d) {
      EncRecDir& D = ra.d[d];
      D.w_hh = whh8 + (size_t)d * G * H;
      D.sc_ih = vec_ih + (size_t)d * G;
      D.sc_hh = vec_hh + (size_t)d * G;
      D.bias = vec_b + (size_t)d * G;
      D.acc_pre = acc_ih + (size_t)d * TB * G;
      D.yq = static_cast<uint8_t*>(yq) + row_bytes(d * H, out_act->bits);
      D.dbg_ih = dbg_acc_ih ? dbg_acc_ih + (size_t)d * G : nullptr;
      D.dbg_hh = dbg_acc_hh ? dbg_acc_hh + (size_t)d * G : nullptr;
      D.hq_n = hq_n ? static_cast<uint8_t*>(hq_n) + (size_t)d * B * hb : nullptr;
      D.c_n = c_n ? c_n + (size_t)d * B * H : nullptr;
    }
    if ((dbg_acc_ih == nullptr) != (dbg_acc_hh == nullptr)) return Q4_ERR_NULL;
    TagScope tag(TAG_ENC_STEP);
    Q4_TRY(launch_enc_recurrent(ra, s));
    return Q4_OK;
  }
  Q4_TRY(cudaMemsetAsync(hbuf, 0, (size_t)dirs * 2 * B * H, s));
  Q4_TRY(cudaMemsetAsync(cbuf, 0, (size_t)dirs * B * H * sizeof(float), s));

  for (int st = 0; st < T; ++st) {
    LstmArgs2 args;
    memset(&args, 0, sizeof(args));
    for (int d = 0; d < dirs; ++d) {
      const int t = d == 0 ? st : T - 1 - st;
      LstmArgs& a = args.d[d];
      fill_lstm_weights(a, w_ih[d], w_hh[d], bias ? bias[d] : nullptr, *x_act, *hid_act);
      a.out_act = *out_act;
      a.x_scale_vec = x_scale_b;
      a.x_scale_mod = B;
      a.acc_pre = acc_ih + ((size_t)d * TB + (size_t)t * B) * G;
      a.acc_pre_stride = G;
      a.hin.base = hbuf + ((size_t)d * 2 + (st & 1)) * B * H;
      a.hin.stride = hb;
      a.c_in = cbuf + (size_t)d * B * H;
      a.N = B;
      a.hq_out = hbuf + ((size_t)d * 2 + ((st + 1) & 1)) * B * H;
      a.hq_stride = hb;
      a.c_out = cbuf + (size_t)d * B * H;
      a.yq_out = static_cast<uint8_t*>(yq) + (size_t)t * B * yb + row_bytes(d * H, out_act->bits);
      a.yq_stride = yb;
      if (dbg_acc_ih) a.dbg_ih = dbg_acc_ih + ((size_t)t * B * dirs + d) * G;
      if (dbg_acc_hh) a.dbg_hh = dbg_acc_hh + ((size_t)t * B * dirs + d) * G;
      a.dbg_stride = (long long)dirs * G;
    }
    TagScope tag(TAG_ENC_STEP);
    Q4_TRY(launch_lstm(args, dirs, s));
  }
  for (int d = 0; d < dirs; ++d) {
    if (hq_n)
      Q4_TRY(cudaMemcpyAsync(static_cast<uint8_t*>(hq_n) + (size_t)d * B * hb,
                             hbuf + ((size_t)d * 2 + (T & 1)) * B * H, (size_t)B * hb,
                             cudaMemcpyDeviceToDevice, s));
    if (c_n)
      Q4_TRY(cudaMemcpyAsync(c_n + (size_t)d * B * H, cbuf + (size_t)d * B * H,
                             (size_t)B * H * sizeof(float), cudaMemcpyDeviceToDevice, s));
  }
  return Q4_OK;
}

int qjoint_logprobs(const float* e, const int32_t* frame_idx, const void* pq, const q4_act* p_act,
                    int32_t N, const q4_mat* w_pred, const float* b_pred, const q4_act* z_act,
                    const q4_mat* w_out, const float* b_out, float* logp, const void* prepared_pred,
                    const void* prepared_out, void* workspace, size_t workspace_bytes, q4_stream stream) {
  if (!e || !frame_idx || !pq || !logp || !workspace) return Q4_ERR_NULL;
  Q4_CHECK(check_act(p_act));
  Q4_CHECK(check_act(z_act));
  Q4_CHECK(check_mat(w_pred, 0, 0));
  Q4_CHECK(check_mat(w_out, 0, 0));
  if (N < 0) return Q4_ERR_DIM;
  const int D = w_pred->rows, V = w_out->rows;
  if (w_out->k != D || w_out->k_pad != D || D % 32 != 0) return Q4_ERR_DIM;
  if (!aligned16(pq) || !aligned16(workspace) || !aligned16(e)) return Q4_ERR_ALIGN;
  const int32_t dims[2] = {N, D};
  if (workspace_bytes < q4_workspace_bytes(Q4_WS_JOINT, dims, 2)) return Q4_ERR_WORKSPACE;
  if (N == 0) return Q4_OK;
  cudaStream_t s = S(stream);
  TagScope tag(TAG_JOINT);
  ++g_quant_calls;   // tanh(e * p)
  const int32_t dims3[3] = {N, D, w_pred->k_pad};
  if (prepared_pred && prepared_out && z_act->is_signed && aligned16(prepared_pred) &&
      aligned16(prepared_out) && mma_rows(N, w_pred->k_pad) && workspace_bytes >= q4_workspace_bytes(Q4_WS_JOINT, dims3, 3)) {
    // tensor cores for any number of rows (a 128-row tile of mostly empty rows included: 16 rows 15.7 us of device time in
    // three launches, 26.9 in the four of the kernels for unprepared weights): int8 copy of the hidden codes; projection GEMM whose epilogue forms
    // tanh(e * p) and quantizes it; output layer with the log-softmax in its epilogue (fused head kernel
    // when D = 256, else GEMM + row log-softmax)
    const int Hp = w_pred->k_pad, Np = (N + 127) / 128 * 128;
    uint8_t* ws = static_cast<uint8_t*>(workspace) + align_up((size_t)N * D * sizeof(float)) + align_up((size_t)N * D);
    int32_t* status = reinterpret_cast<int32_t*>(ws);
    int8_t* p8 = reinterpret_cast<int8_t*>(ws + 256);
    int8_t* z8 = p8 + align_up((size_t)Np * Hp);
    UnpackJobs uj;
    memset(&uj, 0, sizeof(uj));
    uj.n_rows = N;
    uj.n_rows_pad = Np;
    uj.zero_tail = 1;
    uj.clear64 = status;
    add_unpack_job(uj, pq, row_bytes(Hp, p_act->bits), nullptr, *p_act, Hp, p8);
    Q4_TRY(launch_unpack_multi(uj, s, true));
    Q4_TRY(launch_mma_gemm(p8, Hp, N, static_cast<const int8_t*>(prepared_pred), Hp, D, Hp, EPI_JOINTZ, z8, D,
                           nullptr, w_pred->scale, b_pred, p_act->scale, z_act, status, nullptr, s, true, e,
                           frame_idx));   // each kernel of the call is a programmatic dependent of the one before
    if (D == 256 && V <= 2048) {
      LmHeadArgs ja;
      memset(&ja, 0, sizeof(ja));
      ja.N = N;
      ja.H = 0;
      ja.V = V;
      ja.q_scale = z_act->scale;
      ja.sc_out = w_out->scale;
      ja.b_out = b_out;
      ja.lp = logp;
      ja.status = status;
      Q4_TRY(launch_mma_lmhead(ja, z8, D, nullptr, static_cast<const int8_t*>(prepared_out), s, true));
    } else {
      Q4_TRY(launch_mma_gemm(z8, D, N, static_cast<const int8_t*>(prepared_out), D, V, D, EPI_F32, logp, V, nullptr,
                             w_out->scale, b_out, z_act->scale, nullptr, status, nullptr, s));
      Q4_TRY(launch_logsoftmax(logp, logp, N, V, V, nullptr, s));
    }
    return Q4_OK;
  }
  float* p = static_cast<float*>(workspace);
  uint8_t* zq = static_cast<uint8_t*>(workspace) + align_up((size_t)N * D * sizeof(float));
  GemmArgs g1 = gemm_args(pq, row_bytes(w_pred->k_pad, p_act->bits), nullptr, *p_act, N, *w_pred,
                          b_pred, p, D, nullptr);
  Q4_TRY(launch_gemm(g1, EPI_F32, s));
  Q4_TRY(launch_joint_z(e, frame_idx, nullptr, 1, 1, p, nullptr, N, D, *z_act, zq, nullptr, nullptr, s));
  GemmArgs g2 = gemm_args(zq, row_bytes(D, z_act->bits), nullptr, *z_act, N, *w_out, b_out, logp, V,
                          nullptr);
  Q4_TRY(launch_gemm(g2, EPI_F32, s));
  Q4_TRY(launch_logsoftmax(logp, logp, N, V, V, nullptr, s));
  return Q4_OK;
}

int q4_feature_prologue(const float* mel, int32_t B, int32_t T100, int32_t M, void* out_fp16,
                        q4_stream stream) {
  if (!mel || !out_fp16) return Q4_ERR_NULL;
  if (B <= 0 || T100 < 2 || M <= 0) return Q4_ERR_DIM;
  TagScope tag(TAG_MISC);
  Q4_TRY(launch_features(mel, B, T100, M, out_fp16, S(stream)));
  return Q4_OK;
}

// ------------------------------------------------------------------------ prepared weights
namespace {
struct PrepLstm {
  size_t xw, hw, sc_ih, sc_hh, bias;
};
struct PrepPlan {
  PrepLstm lstm[4];   // prediction, source LM, target LM layer 1, target LM layer 2
  size_t lin[6];      // pred_proj, src.bott, src.out, tgt.bott, tgt.out, joint_out
  size_t total;
};
struct TablePlan {
  size_t table[3];    // first layers: de-quantized input sums plus bias of every label (fp32 [V, 4H])
  size_t emb8;        // int8 embedding rows, while the tables are made
  size_t total;
};
// Tables of the first layers' input halves: 16 H bytes a label and network, so a bound on memory (268 MB with 1024, 1024 and
// 2048 cells); a look-up costs the same at any V.  100 frames, ms with / without: 1024 labels, 12 rows 1.41 / 1.92,
// 4096 labels, 12 rows 6.76 / 7.10 and 96 rows 7.38 / 7.54.
constexpr int TABLE_MAX_V = 4096;
bool tables_supported(const q4_model& m) {
  return m.V > 0 && m.V <= TABLE_MAX_V && m.src.n_layers == 1 && m.pred_lstm.w_hh.k_pad % 128 == 0 &&
         m.src.lstm[0].w_hh.k_pad % 128 == 0 && m.tgt.lstm[0].w_hh.k_pad % 128 == 0;
}
const q4_lstm* model_lstm(const q4_model& m, int i) {
  switch (i) {
    case 0: return &m.pred_lstm;
    case 1: return &m.src.lstm[0];
    case 2: return &m.tgt.lstm[0];
    default: return m.tgt.n_layers == 2 ? &m.tgt.lstm[1] : nullptr;
  }
}
const q4_linear* model_linear(const q4_model& m, int i) {
  switch (i) {
    case 0: return &m.pred_proj;
    case 1: return &m.src.bott;
    case 2: return &m.src.out;
    case 3: return &m.tgt.bott;
    case 4: return &m.tgt.out;
    default: return &m.joint_out;
  }
}
PrepPlan plan_prepared(const q4_model& m) {
  PrepPlan p;
  memset(&p, 0, sizeof(p));
  size_t o = 0;
  for (int i = 0; i < 4; ++i) {
    const q4_lstm* L = model_lstm(m, i);
    if (!L) continue;
    const size_t G = L->w_ih.rows;
    p.lstm[i].xw = o;
    o += align_up(G * L->w_ih.k_pad);
    p.lstm[i].hw = o;
    o += align_up(G * L->w_hh.k_pad);
    p.lstm[i].sc_ih = o;
    o += align_up(G * sizeof(float));
    p.lstm[i].sc_hh = o;
    o += align_up(G * sizeof(float));
    p.lstm[i].bias = o;
    o += align_up(G * sizeof(float));
  }
  for (int i = 0; i < 6; ++i) {
    const q4_linear* L = model_linear(m, i);
    p.lin[i] = o;
    o += align_up((size_t)L->w.rows * L->w.k_pad);
  }
  p.total = o;
  return p;
}
TablePlan plan_tables(const q4_model& m) {
  TablePlan p;
  size_t o = 0, ep = 0;
  for (int i = 0; i < 3; ++i) {
    const q4_lstm* L = model_lstm(m, i);
    p.table[i] = o;
    o += align_up((size_t)m.V * L->w_ih.rows * sizeof(float));
    if ((size_t)L->w_ih.k_pad > ep) ep = L->w_ih.k_pad;
  }
  p.emb8 = o;
  p.total = o + align_up((size_t)m.V * ep);
  return p;
}
}  // namespace

size_t q4_prepared_bytes(const q4_model* model) {
  if (!model) return 0;
  return plan_prepared(*model).total;
}

int q4_prepare_model(q4_model* model, void* buffer, size_t bytes, q4_stream stream) {
  if (!model || !buffer) return Q4_ERR_NULL;
  if (!aligned16(buffer)) return Q4_ERR_ALIGN;
  const PrepPlan p = plan_prepared(*model);
  if (bytes < p.total) return Q4_ERR_WORKSPACE;
  cudaStream_t s = S(stream);
  uint8_t* b = static_cast<uint8_t*>(buffer);
  TagScope tag(TAG_MISC);
  for (int i = 0; i < 4; ++i) {
    const q4_lstm* L = model_lstm(*model, i);
    if (!L) continue;
    Q4_CHECK(check_mat(&L->w_ih, 0, 0));
    Q4_CHECK(check_mat(&L->w_hh, 0, 0));
    Q4_TRY(launch_prepare_w(L->w_ih, 1, reinterpret_cast<int8_t*>(b + p.lstm[i].xw), L->w_ih.k_pad, 0, s));
    Q4_TRY(launch_prepare_w(L->w_hh, 1, reinterpret_cast<int8_t*>(b + p.lstm[i].hw), L->w_hh.k_pad, 0, s));
    // de-quantization products of the search (input scale * row scale, hidden scale * row scale)
    const q4_model& mm = *model;
    const float xs = i == 0 ? mm.pred_emb_act.scale : i == 1 ? mm.src.emb_act.scale
                     : i == 2 ? mm.tgt.emb_act.scale : mm.tgt.lstm[0].hid_act.scale;
    Q4_TRY(launch_prepare_vec(L->w_ih.scale, L->w_ih.rows, 1, reinterpret_cast<float*>(b + p.lstm[i].sc_ih), s, xs));
    Q4_TRY(launch_prepare_vec(L->w_hh.scale, L->w_hh.rows, 1, reinterpret_cast<float*>(b + p.lstm[i].sc_hh), s,
                              L->hid_act.scale));
    Q4_TRY(launch_prepare_vec(L->bias, L->w_ih.rows, 1, reinterpret_cast<float*>(b + p.lstm[i].bias), s));
  }
  for (int i = 0; i < 6; ++i) {
    const q4_linear* L = model_linear(*model, i);
    Q4_CHECK(check_mat(&L->w, 0, 0));
    Q4_TRY(launch_prepare_w(L->w, 0, reinterpret_cast<int8_t*>(b + p.lin[i]), L->w.k_pad, 0, s));
  }
  model->prepared = buffer;
  model->tables = nullptr;   // they belong to the preparation before
  return Q4_OK;
}

size_t q4_table_bytes(const q4_model* model, int32_t rows) {
  if (!model || rows <= 0 || rows > sums_max_rows(model->V, model->D) || !tables_supported(*model)) return 0;
  return plan_tables(*model).total;
}
int q4_prepare_tables(q4_model* model, void* buffer, size_t bytes, q4_stream stream) {
  if (!model || !buffer || !model->prepared) return Q4_ERR_NULL;
  if (!tables_supported(*model)) return Q4_ERR_UNSUPPORTED;
  if (reinterpret_cast<uintptr_t>(buffer) & 31u) return Q4_ERR_ALIGN;
  const TablePlan t = plan_tables(*model);
  if (bytes < t.total) return Q4_ERR_WORKSPACE;
  const PrepPlan p = plan_prepared(*model);
  const uint8_t* w = static_cast<const uint8_t*>(model->prepared);
  uint8_t* b = static_cast<uint8_t*>(buffer);
  cudaStream_t s = S(stream);
  TagScope tag(TAG_MISC);
  for (int i = 0; i < 3; ++i) {
    const q4_lstm* L = model_lstm(*model, i);
    const q4_act& act = i == 0 ? model->pred_emb_act : i == 1 ? model->src.emb_act : model->tgt.emb_act;
    const void* emb = i == 0 ? model->pred_emb_q : i == 1 ? model->src.emb_q : model->tgt.emb_q;
    if (!emb) return Q4_ERR_NULL;
    Q4_CHECK(check_act(&act));
    const int Ep = L->w_ih.k_pad, G = L->w_ih.rows;
    int8_t* e8 = reinterpret_cast<int8_t*>(b + t.emb8);
    UnpackJobs uj;
    memset(&uj, 0, sizeof(uj));
    uj.n_rows = uj.n_rows_pad = model->V;
    add_unpack_job(uj, emb, row_bytes(Ep, act.bits), nullptr, act, Ep, e8);
    Q4_TRY(launch_unpack_multi(uj, s, false));
    Q4_TRY(launch_mma_gemm(e8, Ep, model->V, reinterpret_cast<const int8_t*>(w + p.lstm[i].xw), Ep, G, Ep, EPI_F32,
                           b + t.table[i], G, nullptr, reinterpret_cast<const float*>(w + p.lstm[i].sc_ih),
                           reinterpret_cast<const float*>(w + p.lstm[i].bias), 1.0f, nullptr, nullptr, nullptr, s, false));
  }
  model->tables = buffer;
  return Q4_OK;
}

// One-time int8 operands for the tensor-core variants of the step calls.
size_t q4_prepared_lstm_bytes(const q4_mat* w_ih, const q4_mat* w_hh) {
  if (!w_ih || !w_hh) return 0;
  const size_t G = w_ih->rows;
  return align_up(G * w_ih->k_pad) + align_up(G * w_hh->k_pad) + 3 * align_up(G * sizeof(float));
}
int q4_prepare_lstm(const q4_mat* w_ih, const q4_mat* w_hh, const float* bias, void* buffer, size_t bytes,
                    q4_stream stream) {
  if (!buffer) return Q4_ERR_NULL;
  Q4_CHECK(check_mat(w_ih, 0, 0));
  Q4_CHECK(check_mat(w_hh, 0, 0));
  if (w_ih->rows != w_hh->rows || w_ih->rows % 4 != 0) return Q4_ERR_DIM;
  if (!aligned16(buffer)) return Q4_ERR_ALIGN;
  if (bytes < q4_prepared_lstm_bytes(w_ih, w_hh)) return Q4_ERR_WORKSPACE;
  cudaStream_t s = S(stream);
  const size_t G = w_ih->rows;
  uint8_t* b = static_cast<uint8_t*>(buffer);
  int8_t* xw8 = reinterpret_cast<int8_t*>(b);
  int8_t* hw8 = xw8 + align_up(G * w_ih->k_pad);
  float* sc_ih = reinterpret_cast<float*>(hw8 + align_up(G * w_hh->k_pad));
  float* sc_hh = sc_ih + align_up(G * sizeof(float)) / sizeof(float);
  float* bi = sc_hh + align_up(G * sizeof(float)) / sizeof(float);
  TagScope tag(TAG_MISC);
  Q4_TRY(launch_prepare_w(*w_ih, 1, xw8, w_ih->k_pad, 0, s));
  Q4_TRY(launch_prepare_w(*w_hh, 1, hw8, w_hh->k_pad, 0, s));
  Q4_TRY(launch_prepare_vec(w_ih->scale, (int)G, 1, sc_ih, s));
  Q4_TRY(launch_prepare_vec(w_hh->scale, (int)G, 1, sc_hh, s));
  Q4_TRY(launch_prepare_vec(bias, (int)G, 1, bi, s));
  return Q4_OK;
}
size_t q4_prepared_linear_bytes(const q4_mat* w) { return w ? align_up((size_t)w->rows * w->k_pad) : 0; }
int q4_prepare_linear(const q4_mat* w, void* buffer, size_t bytes, q4_stream stream) {
  if (!buffer) return Q4_ERR_NULL;
  Q4_CHECK(check_mat(w, 0, 0));
  if (!aligned16(buffer)) return Q4_ERR_ALIGN;
  if (bytes < q4_prepared_linear_bytes(w)) return Q4_ERR_WORKSPACE;
  TagScope tag(TAG_MISC);
  Q4_TRY(launch_prepare_w(*w, 0, static_cast<int8_t*>(buffer), w->k_pad, 0, S(stream)));
  return Q4_OK;
}

// ------------------------------------------------------------------------ beam search
static int check_state(const q4_beam_state* st, int n_lm_layers) {
  if (!st) return Q4_ERR_NULL;
  const void* req[] = {st->pred_hq, st->pred_c, st->pred_p, st->src_hq, st->src_c, st->src_lp,
                       st->tgt_hq[0], st->tgt_c[0], st->tgt_lp, st->score, st->t, st->u, st->hash,
                       st->prev_hash, st->last_tok, st->row, st->adv_src, st->adv_dst, st->adv_tok,
                       st->bp_parent, st->bp_token, st->bp_score, st->fin_score, st->fin_iter,
                       st->fin_slot, st->fin_n, st->status, st->pend_src, st->pend_dst, st->pend_tok,
                       st->pend_n};
  for (const void* p : req)
    if (!p) return Q4_ERR_NULL;
  if (n_lm_layers > 1 && (!st->tgt_hq[1] || !st->tgt_c[1])) return Q4_ERR_NULL;
  return Q4_OK;
}

int q4_beam_init(q4_beam_state* state, int32_t B, int32_t W, int32_t n_iters, q4_stream stream) {
  Q4_CHECK(check_state(state, 1));
  if (B <= 0 || W <= 0 || W > 16 || n_iters < 0) return Q4_ERR_DIM;
  Q4_TRY(launch_beam_init(*state, B, W, n_iters, S(stream)));
  return Q4_OK;
}

// One network's pending advance for all slots: LSTM layers reading the parent's state row and
// writing the fresh row, then the projection(s).
static int advance_lstm(int tag_id, const q4_lstm& L, const void* x, long long x_stride,
                        const int32_t* x_idx, const q4_act& x_act, void* hq, float* c,
                        const q4_beam_state& st, int N, const int32_t* n_active, cudaStream_t s) {
  TagScope tag(tag_id);
  LstmArgs2 args;
  memset(&args, 0, sizeof(args));
  LstmArgs& a = args.d[0];
  fill_lstm_weights(a, L.w_ih, L.w_hh, L.bias, x_act, L.hid_act);
  const int H = a.H;
  a.x.base = static_cast<const uint8_t*>(x);
  a.x.stride = x_stride;
  a.x.idx = x_idx;
  a.hin.base = static_cast<const uint8_t*>(hq);
  a.hin.stride = row_bytes(H, L.hid_act.bits);
  a.hin.idx = st.adv_src;
  a.c_in = c;
  a.N = N;
  a.hq_out = static_cast<uint8_t*>(hq);
  a.hq_stride = a.hin.stride;
  a.out_idx = st.adv_dst;
  a.c_out = c;
  a.dbg_stride = 4LL * H;
  a.n_active = n_active;
  Q4_TRY(launch_lstm(args, 1, s));
  return Q4_OK;
}

static int check_model_lstm(const q4_lstm& L, const q4_act& x_act) {
  int H = 0;
  return check_lstm(&L.w_ih, &L.w_hh, &x_act, &L.hid_act, &H);
}

constexpr int PLAN_ITERS = 12;   // steps in a search's graph: even (the pending lists alternate), a multiple of the 1, 2, 3 or 4 calls per frame
// Whether a search takes the tensor-core kernels: prepared weights, widths they cover and room for their operands.
static bool search_uses_tensor_cores(const q4_model& m, const q4_beam_state& st, int B, int W, size_t workspace_bytes) {
  const int Hp = m.pred_lstm.w_hh.k_pad, Hs = m.src.lstm[0].w_hh.k_pad, Ht = m.tgt.lstm[0].w_hh.k_pad;
  const int Ep = m.pred_lstm.w_ih.k_pad;
  const int32_t dims8[8] = {B, W, m.V, m.D, Ep, Hp, Hs, Ht};
  return m.prepared != nullptr && m.src.n_layers == 1 && m.src.lstm[0].w_ih.k_pad == Ep && m.tgt.lstm[0].w_ih.k_pad == Ep &&
         Hp % 128 == 0 && Hs % 128 == 0 && Ht % 128 == 0 &&
         aligned16(st.pred_c) && aligned16(st.src_c) && aligned16(st.tgt_c[0]) && aligned16(st.tgt_c[1]) &&
         workspace_bytes >= q4_workspace_bytes(Q4_WS_BEAM, dims8, 8);
}
// In the tensor-core path the first codes block of the workspace is free: there a search keeps when its utterances were frozen.
static int32_t* search_frozen(void* workspace) { return reinterpret_cast<int32_t*>(static_cast<uint8_t*>(workspace) + 256); }

// Whether a whole search takes the kernels that look the first layers' input halves up and keep the sums of the recurrent
// halves per state row: prepared weights, tables and room for the sums, the last two read 32 bytes at a time.
static bool search_keeps_sums(const q4_model& m, const q4_beam_state& st, int B, int W, const void* workspace,
                              size_t workspace_bytes) {
  if (!m.prepared || !m.tables || !tables_supported(m) || !aligned16(m.prepared)) return false;
  if ((reinterpret_cast<uintptr_t>(workspace) | reinterpret_cast<uintptr_t>(m.tables)) & 31u) return false;
  const int RW = st.rows_per_utt > 0 ? st.rows_per_utt : 2 * W;
  const int32_t dims9[9] = {B, W, m.V, m.D, m.pred_lstm.w_ih.k_pad, m.pred_lstm.w_hh.k_pad, m.src.lstm[0].w_hh.k_pad,
                            m.tgt.lstm[0].w_hh.k_pad, RW};
  return B * W <= sums_max_rows(m.V, m.D) && aligned16(st.pred_c) && aligned16(st.src_c) && aligned16(st.tgt_c[0]) && aligned16(st.tgt_c[1]) &&
         workspace_bytes >= q4_workspace_bytes(Q4_WS_BEAM, dims9, 9);
}

// How a step is part of a search.
struct StepMode {
  SearchCall* call;                         // non-null: e, T and u_max come from there, its iteration number is added
  int32_t* frozen;                          // non-null: an utterance without labels to propose is left to launch_search_tail
  const cudaGraphConditionalHandle* loop;   // non-null: the last step of a graph's loop
  bool sums;                                // see search_keeps_sums
  cudaStream_t sums_stream;                 // non-null: a stream for the sums of the recurrent halves, with an event (else
  cudaEvent_t sums_event;                   // they follow the source LM's head)
};
// One step.
static int beam_step(const q4_model* model, q4_beam_state* state, const float* e, int32_t B, int32_t T, int32_t W,
                     int32_t iter, int32_t u_max, float lambda_t, float lambda_s, float rho, int32_t mode,
                     void* workspace, size_t workspace_bytes, q4_stream stream, const StepMode& how) {
  if (!model || !e || !workspace) return Q4_ERR_NULL;
  if (mode < 0 || mode > 2) return Q4_ERR_UNSUPPORTED;
  if (B <= 0 || T <= 0 || W <= 0 || W > 16 || iter < 0 || u_max < 0) return Q4_ERR_DIM;
  const q4_model& m = *model;
  SearchCall* const call = how.call;
  int32_t* const frozen = how.frozen;
  Q4_CHECK(check_state(state, m.tgt.n_layers));
  if (mode != 0) {   // time-synchronous search: candidate set, enough state rows, call number matches
    const q4_beam_state& ts = *state;
    if (!ts.nb_score || !ts.nb_u || !ts.nb_last_tok || !ts.nb_row || !ts.nb_origin || !ts.nb_hash ||
        !ts.nb_prev_hash || !ts.nb_n)
      return Q4_ERR_NULL;
    if (ts.tsd_smax < 0 || ts.tsd_smax > 3 || ts.rows_per_utt < W * (ts.tsd_smax + 1) || ts.rows_per_utt > 64)
      return Q4_ERR_DIM;
    const bool closing = iter % (ts.tsd_smax + 1) == ts.tsd_smax;
    if (closing != (mode == 2) || iter / (ts.tsd_smax + 1) >= T) return Q4_ERR_DIM;
  } else if (state->rows_per_utt != 0 && state->rows_per_utt < 2 * W) {
    return Q4_ERR_DIM;
  }
  const int V = m.V, D = m.D;
  if (V <= 1 || D <= 0 || D % 32 != 0 || m.E <= 0) return Q4_ERR_DIM;
  if (m.src.n_layers < 1 || m.src.n_layers > 2 || m.tgt.n_layers < 1 || m.tgt.n_layers > 2)
    return Q4_ERR_DIM;
  if (!m.pred_emb_q || !m.src.emb_q || !m.tgt.emb_q) return Q4_ERR_NULL;
  Q4_CHECK(check_model_lstm(m.pred_lstm, m.pred_emb_act));
  Q4_CHECK(check_mat(&m.pred_proj.w, D, m.pred_lstm.w_hh.k_pad));
  Q4_CHECK(check_act(&m.z_act));
  Q4_CHECK(check_mat(&m.joint_out.w, V, D));
  const q4_lm* lms[2] = {&m.src, &m.tgt};
  for (const q4_lm* lm : lms) {
    Q4_CHECK(check_model_lstm(lm->lstm[0], lm->emb_act));
    if (lm->n_layers == 2) Q4_CHECK(check_model_lstm(lm->lstm[1], lm->lstm[0].hid_act));
    const q4_lstm& last = lm->lstm[lm->n_layers - 1];
    Q4_CHECK(check_mat(&lm->bott.w, D, last.w_hh.k_pad));
    Q4_CHECK(check_act(&lm->bott_act));
    Q4_CHECK(check_mat(&lm->out.w, V, D));
  }
  if ((size_t)W * V * sizeof(float) > 200 * 1024) return Q4_ERR_UNSUPPORTED;
  const int32_t dims[4] = {B, W, V, D};
  if (workspace_bytes < q4_workspace_bytes(Q4_WS_BEAM, dims, 4)) return Q4_ERR_WORKSPACE;
  if (!aligned16(workspace) || !aligned16(e)) return Q4_ERR_ALIGN;

  cudaStream_t s = S(stream);
  const q4_beam_state& st = *state;
  const int N = B * W;
  // quantizer applications of one iteration: the cell outputs of the advanced networks, the two
  // bottleneck outputs, tanh(e * p)
  g_quant_calls += 1 + 1 + m.tgt.n_layers + 2 + 1;
  int joint_normalized = 0;   // the tensor-core joint kernel leaves log-probabilities, not logits
  // the first call of a frame of the time-synchronous search follows a frame close, which creates
  // no label extension: no network has anything to advance, only the joint runs
  const bool nets = !(mode != 0 && iter > 0 && iter % (state->tsd_smax + 1) == 0);
  uint8_t* ws = static_cast<uint8_t*>(workspace) + 256;   // (the first 256 bytes: SearchCall of q4_beam_search, at 128 a row count)
  uint8_t* zq = ws;
  ws += align_up((size_t)N * D);
  uint8_t* bq_src = ws;
  ws += align_up((size_t)N * D);
  uint8_t* bq_tgt = ws;
  ws += align_up((size_t)N * D);
  float* logits = reinterpret_cast<float*>(ws);
  ws += align_up((size_t)N * V * sizeof(float));
  int32_t* live = reinterpret_cast<int32_t*>(ws);
  ws += align_up((size_t)N * sizeof(int32_t));
  // pending advances of this iteration as the previous selection (or the reset) listed them: up to 128 rows every slot at its
  // own place (those without an advance -1), beyond only the slots that have one
  const int par = iter & 1;
  int32_t* c_src = st.pend_src + (size_t)par * N;
  int32_t* c_dst = st.pend_dst + (size_t)par * N;
  int32_t* c_tok = st.pend_tok + (size_t)par * N;
  const int32_t* n_active = st.pend_n + par;
  q4_beam_state cst = st;   // same state, pending advances in the order of the list
  cst.adv_src = c_src;
  cst.adv_dst = c_dst;
  cst.adv_tok = c_tok;
  // tensor-core path: prepared int8 weights and room for the int8 operand scratch.  It is taken
  // for any number of rows: even 16 rows padded to one 128-row tile finish sooner than on the DP4A
  // kernels (measured 3x on a single utterance), since the time goes to streaming the weights
  const int Hp = m.pred_lstm.w_hh.k_pad, Hs = m.src.lstm[0].w_hh.k_pad, Ht = m.tgt.lstm[0].w_hh.k_pad;
  const int Ep = m.pred_lstm.w_ih.k_pad;
  const bool use_mma = search_uses_tensor_cores(m, st, B, W, workspace_bytes);
  if (use_mma || how.sums) {
    const size_t Np = ((size_t)N + 127) / 128 * 128;
    auto take = [&](size_t bytes) {
      uint8_t* p = ws;
      ws += align_up(bytes);
      return p;
    };
    const int hdim[4] = {Hp, Hs, Ht, Ht};   // prediction, source LM, target LM layers 1 and 2
    int8_t* xa8[3] = {nullptr, nullptr, nullptr};            // embedding rows of the pending symbols
    int8_t* ha8[4] = {nullptr, nullptr, nullptr, nullptr};   // previous cell outputs
    if (!how.sums) {
      for (int i = 0; i < 3; ++i) xa8[i] = reinterpret_cast<int8_t*>(take(Np * Ep));
      for (int i = 0; i < 4; ++i) ha8[i] = reinterpret_cast<int8_t*>(take(Np * (size_t)hdim[i]));
    }
    int8_t* new_h8[4];                                       // new cell outputs
    for (int i = 0; i < 4; ++i) new_h8[i] = reinterpret_cast<int8_t*>(take(Np * (size_t)hdim[i]));
    int8_t* const pred_h8 = new_h8[0];
    int8_t* const src_h8 = new_h8[1];
    int8_t* const tgt_h8[2] = {new_h8[2], new_h8[3]};
    int8_t* bq8[2];
    for (int i = 0; i < 2; ++i) bq8[i] = reinterpret_cast<int8_t*>(take(Np * D));
    int8_t* z8 = reinterpret_cast<int8_t*>(take(Np * D));
    int32_t* const n_work = reinterpret_cast<int32_t*>(static_cast<uint8_t*>(workspace) + 128);
    float* state_sums[4] = {nullptr, nullptr, nullptr, nullptr};
    if (how.sums) {
      const size_t R = (size_t)B * (st.rows_per_utt > 0 ? st.rows_per_utt : 2 * W);
      for (int i = 0; i < 4; ++i) state_sums[i] = reinterpret_cast<float*>(take(R * 4 * (size_t)hdim[i] * sizeof(float)));
    }
    const PrepPlan pp = plan_prepared(m);
    const uint8_t* pb = static_cast<const uint8_t*>(m.prepared);

    // at most 32 hypothesis rows (one utterance): the LSTM steps are bound by reading the weights once,
    // and a weight-streaming kernel reads them as stored (packed 4-bit), the state rows and embedding
    // rows too, so the gathers below are not needed
    const bool skinny = !how.sums &&
        skinny_lstm_supported(N, Hp, Ep, m.pred_lstm.w_ih.bits, m.pred_lstm.w_hh.bits, m.pred_emb_act, m.pred_lstm.hid_act) &&
        skinny_lstm_supported(N, Hs, Ep, m.src.lstm[0].w_ih.bits, m.src.lstm[0].w_hh.bits, m.src.emb_act, m.src.lstm[0].hid_act) &&
        skinny_lstm_supported(N, Ht, Ep, m.tgt.lstm[0].w_ih.bits, m.tgt.lstm[0].w_hh.bits, m.tgt.emb_act, m.tgt.lstm[0].hid_act) &&
        (m.tgt.n_layers == 1 || skinny_lstm_supported(N, Ht, Ht, m.tgt.lstm[1].w_ih.bits, m.tgt.lstm[1].w_hh.bits,
                                                      m.tgt.lstm[0].hid_act, m.tgt.lstm[1].hid_act));
    // all gathers of the iteration in one launch: embedding rows by pending symbol, previous
    // cell-output codes by parent state row, unpacked to int8 operand rows
    if (nets && !skinny && !how.sums) {
      UnpackJobs uj;
      memset(&uj, 0, sizeof(uj));
      add_unpack_job(uj, m.pred_emb_q, row_bytes(Ep, m.pred_emb_act.bits), cst.adv_tok, m.pred_emb_act, Ep, xa8[0]);
      add_unpack_job(uj, m.src.emb_q, row_bytes(Ep, m.src.emb_act.bits), cst.adv_tok, m.src.emb_act, Ep, xa8[1]);
      add_unpack_job(uj, m.tgt.emb_q, row_bytes(Ep, m.tgt.emb_act.bits), cst.adv_tok, m.tgt.emb_act, Ep, xa8[2]);
      add_unpack_job(uj, st.pred_hq, row_bytes(Hp, m.pred_lstm.hid_act.bits), cst.adv_src, m.pred_lstm.hid_act, Hp, ha8[0]);
      add_unpack_job(uj, st.src_hq, row_bytes(Hs, m.src.lstm[0].hid_act.bits), cst.adv_src, m.src.lstm[0].hid_act, Hs, ha8[1]);
      add_unpack_job(uj, st.tgt_hq[0], row_bytes(Ht, m.tgt.lstm[0].hid_act.bits), cst.adv_src, m.tgt.lstm[0].hid_act, Ht, ha8[2]);
      if (m.tgt.n_layers == 2)
        add_unpack_job(uj, st.tgt_hq[1], row_bytes(Ht, m.tgt.lstm[1].hid_act.bits), cst.adv_src, m.tgt.lstm[1].hid_act, Ht, ha8[3]);
      uj.n_rows = N;
      uj.n_rows_pad = (int)Np;
      uj.zero_tail = 0;   // rows beyond the pending advances feed tiles whose results are dropped
      uj.n_active = n_active;
      TagScope tag(TAG_MISC);
      Q4_TRY(launch_unpack_multi(uj, s, true));
    }
    const q4_lstm* const first_layer[3] = {&m.pred_lstm, &m.src.lstm[0], &m.tgt.lstm[0]};
    if (nets && how.sums) {   // the first layers of all networks
      CellJobs cj;
      memset(&cj, 0, sizeof(cj));
      const TablePlan tp = plan_tables(m);
      void* const hq[3] = {st.pred_hq, st.src_hq, st.tgt_hq[0]};
      float* const c[3] = {st.pred_c, st.src_c, st.tgt_c[0]};
      for (int i = 0; i < 3; ++i) {
        CellJob& k = cj.job[i];
        k.table = reinterpret_cast<const float*>(static_cast<const uint8_t*>(m.tables) + tp.table[i]);
        k.sums = state_sums[i];
        k.sc_hh = reinterpret_cast<const float*>(pb + pp.lstm[i].sc_hh);
        k.c = c[i];
        k.hq = static_cast<uint8_t*>(hq[i]);
        k.h8 = new_h8[i];
        k.H = hdim[i];
        k.hid_act = first_layer[i]->hid_act;
      }
      cj.n_jobs = 3;
      cj.N = N;
      cj.src_row = c_src;
      cj.dst_row = c_dst;
      cj.tok = c_tok;
      cj.n_active = n_active;
      cj.n_work = n_work;
      TagScope tag(TAG_CELLS);
      Q4_TRY(launch_search_cells(cj, s, true));
    }
    auto state_products = [&](cudaStream_t s, bool dep, int first, int count) -> int {
      StateProductJobs sj;
      memset(&sj, 0, sizeof(sj));
      for (int i = 0; i < count; ++i) {
        sj.job[i].h8 = new_h8[first + i];
        sj.job[i].w8 = reinterpret_cast<const int8_t*>(pb + pp.lstm[first + i].hw);
        sj.job[i].sums = state_sums[first + i];
        sj.job[i].H = hdim[first + i];
      }
      sj.n_jobs = count;
      sj.N = N;
      sj.dst_row = c_dst;
      sj.n_work = n_work;
      sj.status = st.status;
      TagScope tag(TAG_STATE);
      Q4_TRY(launch_state_products(sj, s, dep));
      return Q4_OK;
    };
    // the three networks are independent until the selection: with two lent streams they run side
    // by side.  The call's own stream carries the target LM's chain (gather -> two layers -> head ->
    // selection as programmatic dependents without an event in between; a fork costs 2 to 4 us, a join 1 to 4), which is
    // the longest of a step that multiplies its first layers: with 1024 rows its launches, each alone, take 114 us, the
    // prediction and joint networks' 109.  In a search that keeps sums the joint network's is longer from 16 rows on: 40 and
    // 33 us with 16 rows, 42 and 34 with 40, 47 and 45 with 128, 48 and 43 with 256.
    // Against the prediction/joint chain there, 150 iterations with labels in most: 16 slots 4.62 -> 4.38 ms, 16 x 16
    // slots 6.64 -> 6.36, time-synchronous 4 x 8 slots 12.8 -> 12.1; with labels in a third: 3.61 -> 3.59, 5.15 ->
    // 5.22, 12.9 -> 12.1
    cudaStream_t sp = s, ss = s, stt = s;
    const bool forked = nets && st.aux_stream[0] && st.aux_stream[1] && st.aux_event[0] && st.aux_event[1] &&
                        st.aux_event[2];
    if (forked) {
      sp = reinterpret_cast<cudaStream_t>(st.aux_stream[0]);
      ss = reinterpret_cast<cudaStream_t>(st.aux_stream[1]);
      cudaEvent_t fork = reinterpret_cast<cudaEvent_t>(st.aux_event[0]);
      Q4_TRY(cudaEventRecord(fork, s));
      Q4_TRY(cudaStreamWaitEvent(sp, fork, 0));
      Q4_TRY(cudaStreamWaitEvent(ss, fork, 0));
      if (how.sums_stream) {
        Q4_TRY(cudaStreamWaitEvent(how.sums_stream, fork, 0));
        Q4_CHECK(state_products(how.sums_stream, false, 0, 3));
      }
    }
    // one LSTM layer of one network for every pending slot
    // `dep`: the previous launch on the same stream is a kernel of this library, so this one may
    // be launched as its programmatic dependent
    auto lstm_mma = [&](cudaStream_t s, bool dep, int tag_id, int li, const q4_lstm& L, const q4_act& x_act,
                        const int8_t* xa, const int8_t* ha, void* hq, float* c, int8_t* h8, int h_first = 0,
                        int trigger_early = 0) -> int {
      TagScope tag(tag_id);
      const int H = L.w_hh.k_pad, Kx = L.w_ih.k_pad;
      if (skinny) {
        // x rows: the embedding table by pending symbol, or (second layer) the first layer's fresh state rows
        const bool second = li == 3;
        SkinnyLstmArgs k;
        memset(&k, 0, sizeof(k));
        k.N = N;
        k.H = H;
        k.Kx = Kx;
        k.w_ih = static_cast<const uint8_t*>(L.w_ih.q);
        k.w_hh = static_cast<const uint8_t*>(L.w_hh.q);
        k.s_wih = L.w_ih.scale;
        k.s_whh = L.w_hh.scale;
        k.bias = L.bias;
        k.x = static_cast<const uint8_t*>(second ? st.tgt_hq[0] : li == 0 ? m.pred_emb_q : li == 1 ? m.src.emb_q : m.tgt.emb_q);
        k.x_stride = row_bytes(Kx, 4);
        k.x_idx = second ? cst.adv_dst : cst.adv_tok;
        k.x_signed = x_act.is_signed;
        k.x_zp = x_act.zero_point;
        k.x_scale = x_act.scale;
        k.hid_act = L.hid_act;
        k.hq_in = static_cast<const uint8_t*>(hq);
        k.c_in = c;
        k.src_row = cst.adv_src;
        k.dst_row = cst.adv_dst;
        k.hq_out = static_cast<uint8_t*>(hq);
        k.c_out = c;
        k.h8_out = h8;
        k.h8_ld = H;
        k.n_active = n_active;
        Q4_TRY(launch_skinny_lstm(k, s, dep));
        return Q4_OK;
      }
      MmaLstmArgs a;
      memset(&a, 0, sizeof(a));
      a.N = N;
      a.H = H;
      a.Kx_pad = Kx;
      a.sc_ih = reinterpret_cast<const float*>(pb + pp.lstm[li].sc_ih);
      a.sc_hh = reinterpret_cast<const float*>(pb + pp.lstm[li].sc_hh);
      a.bias = reinterpret_cast<const float*>(pb + pp.lstm[li].bias);
      a.x_scale = x_act.scale;
      a.hid_act = L.hid_act;
      a.out_act = L.hid_act;
      a.src_row = cst.adv_src;
      a.dst_row = cst.adv_dst;
      a.c_in = c;
      a.c_out = c;
      a.hq_out = static_cast<uint8_t*>(hq);
      a.hq_ld = row_bytes(H, L.hid_act.bits);
      a.h8_out = h8;
      a.h8_ld = H;
      a.status = st.status;
      a.n_active = n_active;
      a.premultiplied = 1;   // q4_prepare_model stored the products
      a.h_first = dep && !how.sums ? h_first : 0;
      a.trigger_early = trigger_early;
      a.hh_pre = how.sums ? state_sums[li] : nullptr;
      Q4_TRY(launch_mma_lstm(a, xa, Kx, reinterpret_cast<const int8_t*>(pb + pp.lstm[li].xw), Kx, ha, H,
                             reinterpret_cast<const int8_t*>(pb + pp.lstm[li].hw), H, s, dep));
      return Q4_OK;
    };
    auto linear_mma = [&](cudaStream_t s, bool dep, int tag_id, int wi, const q4_linear& L, const int8_t* x8,
                          float x_scale, int epi, void* out, long long ldo, const int32_t* out_idx,
                          const q4_act* out_act, const int32_t* rows_active, const int32_t* n_idle = nullptr) -> int {
      TagScope tag(tag_id);
      Q4_TRY(launch_mma_gemm(x8, L.w.k_pad, N, reinterpret_cast<const int8_t*>(pb + pp.lin[wi]), L.w.k_pad,
                             L.w.rows, L.w.k_pad, epi, out, ldo, out_idx, L.w.scale, L.bias, x_scale, out_act,
                             st.status, rows_active, s, dep, nullptr, nullptr, n_idle, B));
      return Q4_OK;
    };

    const int32_t* n_frozen = frozen ? &call->n_frozen : nullptr;   // all utterances frozen: the joint network has nothing to do
    const bool fused_head = fused_heads(V, D);
    // 1a. prediction network, then the joint network for every live slot (stream sp)
    if (nets) {
      if (!how.sums)
        Q4_CHECK(lstm_mma(sp, !forked, TAG_PRED_LSTM, 0, m.pred_lstm, m.pred_emb_act, xa8[0], ha8[0], st.pred_hq,
                          st.pred_c, pred_h8));
      Q4_CHECK(linear_mma(sp, !how.sums || !forked, TAG_PRED_PROJ, 0, m.pred_proj, pred_h8, m.pred_lstm.hid_act.scale, EPI_F32,
                          st.pred_p, D, cst.adv_dst, nullptr, n_active));
    }
    {
      TagScope tag(TAG_JOINT);
      Q4_TRY(launch_joint_z(e, nullptr, st.t, B, W, st.pred_p, st.row, N, D, m.z_act, nullptr, z8, live, sp, true, call,
                            n_frozen ? B : 0));
    }
    // small vocabularies: logits, which the selection normalises in passing (one short kernel instead of a cluster's
    // exchange, and the order of sums of the kernels for few rows)
    const bool joint_head = fused_head && V > 256;
    joint_normalized = joint_head ? 1 : 0;
    if (joint_head) {
      // output layer of the joint network with the log-softmax over the vocabulary in its epilogue
      TagScope tag(TAG_JOINT);
      LmHeadArgs ja;
      memset(&ja, 0, sizeof(ja));
      ja.N = N;
      ja.H = 0;
      ja.V = V;
      ja.q_scale = m.z_act.scale;
      ja.sc_out = m.joint_out.w.scale;
      ja.b_out = m.joint_out.bias;
      ja.lp = logits;
      ja.dst_row = live;
      ja.status = st.status;
      ja.n_idle = n_frozen;
      ja.all_idle = B;
      Q4_TRY(launch_mma_lmhead(ja, z8, D, nullptr, reinterpret_cast<const int8_t*>(pb + pp.lin[5]), sp, true));
    } else {
      Q4_CHECK(linear_mma(sp, true, TAG_JOINT, 5, m.joint_out, z8, m.z_act.scale, EPI_F32, logits, V, live, nullptr,
                          nullptr, n_frozen));
    }
    // 1b. source LM (stream ss) and target LM (stream stt)
    for (int which = 0; which < 2 && nets; ++which) {
      const q4_lm& lm = *lms[which];
      cudaStream_t sl = which == 0 ? ss : stt;
      const q4_lstm& L0 = lm.lstm[0];
      void* hq0 = which == 0 ? st.src_hq : st.tgt_hq[0];
      float* c0 = which == 0 ? st.src_c : st.tgt_c[0];
      int8_t* h8_0 = which == 0 ? src_h8 : tgt_h8[0];
      float* lp = which == 0 ? st.src_lp : st.tgt_lp;
      if (!how.sums)
        Q4_CHECK(lstm_mma(sl, which == 1 || !forked, which == 0 ? TAG_SRC_LSTM : TAG_TGT_L1, which == 0 ? 1 : 2, L0, lm.emb_act,
                          xa8[which + 1], ha8[which + 1], hq0, c0, h8_0, 0, lm.n_layers == 2 ? 1 : 0));
      const int8_t* top8 = h8_0;
      const q4_lstm* last = &L0;
      if (lm.n_layers == 2) {
        const q4_lstm& L1 = lm.lstm[1];
        // layer 2 reads layer 1's output only as its input operand: its recurrent half starts
        // while layer 1 is still in its cell update
        Q4_CHECK(lstm_mma(sl, true, TAG_TGT_L2, 3, L1, L0.hid_act, h8_0, ha8[3], st.tgt_hq[1], st.tgt_c[1],
                          tgt_h8[1], 1, 0));
        top8 = tgt_h8[1];
        last = &L1;
        if (how.sums && forked) Q4_TRY(cudaEventRecord(reinterpret_cast<cudaEvent_t>(st.aux_event[0]), s));
      }
      const bool head_dep = !how.sums || which == 1 || !forked;   // behind an event otherwise
      const int head_tag = which == 0 ? TAG_SRC_HEAD : TAG_TGT_HEAD;
      if (fused_head) {
        // bottleneck, re-quantization, output layer and log-softmax in one kernel
        TagScope tag(head_tag);
        LmHeadArgs ha;
        memset(&ha, 0, sizeof(ha));
        ha.N = N;
        ha.H = last->w_hh.k_pad;
        ha.V = V;
        ha.x_scale = last->hid_act.scale;
        ha.sc_bott = lm.bott.w.scale;
        ha.b_bott = lm.bott.bias;
        ha.bott_act = lm.bott_act;
        ha.q_scale = lm.bott_act.scale;
        ha.sc_out = lm.out.w.scale;
        ha.b_out = lm.out.bias;
        ha.lp = lp;
        ha.dst_row = cst.adv_dst;
        ha.n_active = n_active;
        ha.status = st.status;
        Q4_TRY(launch_mma_lmhead(ha, top8, ha.H, reinterpret_cast<const int8_t*>(pb + pp.lin[which == 0 ? 1 : 3]),
                                 reinterpret_cast<const int8_t*>(pb + pp.lin[which == 0 ? 2 : 4]), sl, head_dep));
      } else {
        Q4_CHECK(linear_mma(sl, head_dep, head_tag, which == 0 ? 1 : 3, lm.bott, top8, last->hid_act.scale, EPI_QUANT8,
                            bq8[which], D, nullptr, &lm.bott_act, n_active));
        Q4_CHECK(linear_mma(sl, true, head_tag, which == 0 ? 2 : 4, lm.out, bq8[which], lm.bott_act.scale, EPI_F32, lp,
                            V, cst.adv_dst, nullptr, n_active));
      }
    }
    if (forked) {
      Q4_TRY(cudaEventRecord(reinterpret_cast<cudaEvent_t>(st.aux_event[1]), sp));
      Q4_TRY(cudaEventRecord(reinterpret_cast<cudaEvent_t>(st.aux_event[2]), ss));
    }
    if (how.sums && nets) {   // sums for the next step, beside the target LM's head and the selection
      cudaStream_t sx = forked && how.sums_stream ? how.sums_stream : ss;
      if (sx == ss) Q4_CHECK(state_products(ss, true, 0, 3));
      if (m.tgt.n_layers == 2) {
        if (forked) Q4_TRY(cudaStreamWaitEvent(sx, reinterpret_cast<cudaEvent_t>(st.aux_event[0]), 0));
        Q4_CHECK(state_products(sx, !forked, 3, 1));
      }
    }
    if (forked) {   // join: the selection waits for both side chains (not for the sums)
      Q4_TRY(cudaStreamWaitEvent(s, reinterpret_cast<cudaEvent_t>(st.aux_event[1]), 0));
      Q4_TRY(cudaStreamWaitEvent(s, reinterpret_cast<cudaEvent_t>(st.aux_event[2]), 0));
    }
    if (!fused_head && nets) {  // log-softmax of both LMs' new rows in one launch
      TagScope tag(TAG_TGT_HEAD);
      Q4_TRY(launch_logsoftmax(st.src_lp, st.src_lp, N, V, V, cst.adv_dst, s, st.tgt_lp, n_active));
    }
  } else {
    // 1. pending advances -------------------------------------------------------------
    if (nets) {  // prediction network: embedding row -> LSTM -> projection to D
      const q4_lstm& L = m.pred_lstm;
      Q4_CHECK(advance_lstm(TAG_PRED_LSTM, L, m.pred_emb_q, row_bytes(L.w_ih.k_pad, m.pred_emb_act.bits), cst.adv_tok,
                            m.pred_emb_act, st.pred_hq, st.pred_c, cst, N, n_active, s));
      GemmArgs g = gemm_args(st.pred_hq, row_bytes(L.w_hh.k_pad, L.hid_act.bits), cst.adv_dst,
                             L.hid_act, N, m.pred_proj.w, m.pred_proj.bias, st.pred_p, D, cst.adv_dst);
      g.n_active = n_active;
      TagScope tag(TAG_PRED_PROJ);
      Q4_TRY(launch_gemm(g, EPI_F32, s));
    }
    for (int which = 0; which < 2 && nets; ++which) {
      const q4_lm& lm = *lms[which];
      void* hq0 = which == 0 ? st.src_hq : st.tgt_hq[0];
      float* c0 = which == 0 ? st.src_c : st.tgt_c[0];
      float* lp = which == 0 ? st.src_lp : st.tgt_lp;
      uint8_t* bq = which == 0 ? bq_src : bq_tgt;
      const q4_lstm& L0 = lm.lstm[0];
      Q4_CHECK(advance_lstm(which == 0 ? TAG_SRC_LSTM : TAG_TGT_L1, L0, lm.emb_q, row_bytes(L0.w_ih.k_pad, lm.emb_act.bits), cst.adv_tok,
                            lm.emb_act, hq0, c0, cst, N, n_active, s));
      const void* top = hq0;
      const q4_lstm* last = &L0;
      if (lm.n_layers == 2) {
        if (which == 0) return Q4_ERR_UNSUPPORTED;  // the state block holds one source-LM layer
        const q4_lstm& L1 = lm.lstm[1];
        Q4_CHECK(advance_lstm(TAG_TGT_L2, L1, hq0, row_bytes(L0.w_hh.k_pad, L0.hid_act.bits), cst.adv_dst,
                              L0.hid_act, st.tgt_hq[1], st.tgt_c[1], cst, N, n_active, s));
        top = st.tgt_hq[1];
        last = &L1;
      }
      GemmArgs gb = gemm_args(top, row_bytes(last->w_hh.k_pad, last->hid_act.bits), cst.adv_dst,
                              last->hid_act, N, lm.bott.w, lm.bott.bias, bq,
                              row_bytes(D, lm.bott_act.bits), nullptr);
      gb.out_act = lm.bott_act;
      gb.n_active = n_active;
      TagScope tag(which == 0 ? TAG_SRC_HEAD : TAG_TGT_HEAD);
      Q4_TRY(launch_gemm(gb, EPI_QUANT, s));
      GemmArgs go = gemm_args(bq, row_bytes(D, lm.bott_act.bits), nullptr, lm.bott_act, N, lm.out.w,
                              lm.out.bias, lp, V, cst.adv_dst);
      go.n_active = n_active;
      Q4_TRY(launch_gemm(go, EPI_F32, s));
      Q4_TRY(launch_logsoftmax(lp, lp, N, V, V, cst.adv_dst, s, nullptr, n_active));
    }

    // 2. joint network for every live slot at its frame -----------------------------------
    TagScope tag_joint(TAG_JOINT);
    Q4_TRY(launch_joint_z(e, nullptr, st.t, B, W, st.pred_p, st.row, N, D, m.z_act, zq, nullptr, live, s, false, call));
    GemmArgs gj = gemm_args(zq, row_bytes(D, m.z_act.bits), live, m.z_act, N, m.joint_out.w,
                            m.joint_out.bias, logits, V, nullptr);
    Q4_TRY(launch_gemm(gj, EPI_F32, s));
  }

  // 3. Eq. 1 proposals, merge, finished list, next beam --------------------------------
  BeamSelArgs sel;
  memset(&sel, 0, sizeof(sel));
  sel.call = call;
  sel.frozen = frozen;
  if (how.loop) {
    sel.loop = *how.loop;
    sel.loop_iters = PLAN_ITERS;
  }
  sel.logits = logits;
  sel.src_lp = st.src_lp;
  sel.tgt_lp = st.tgt_lp;
  sel.st = st;
  sel.B = B;
  sel.T = T;
  sel.W = W;
  sel.V = V;
  sel.iter = iter;
  sel.u_max = u_max;
  sel.lambda_t = lambda_t;
  sel.lambda_s = lambda_s;
  sel.rho = rho;
  sel.exact_only = select_exact_only();
  sel.normalized = joint_normalized;
  sel.mode = mode;
  TagScope tag_sel(TAG_SELECT);
  if (mode != 0)
    Q4_TRY(launch_tsd_select(sel, s, use_mma || how.sums));
  else
    Q4_TRY(launch_beam_select(sel, s, use_mma || how.sums));
  if (how.sums && nets && st.aux_stream[0] && st.aux_stream[1] && st.aux_event[0] && st.aux_event[1] && st.aux_event[2]) {
    // the next step waits for the sums as well
    cudaEvent_t done = how.sums_stream ? how.sums_event : reinterpret_cast<cudaEvent_t>(st.aux_event[2]);
    Q4_TRY(cudaEventRecord(done, how.sums_stream ? how.sums_stream : reinterpret_cast<cudaStream_t>(st.aux_stream[1])));
    Q4_TRY(cudaStreamWaitEvent(s, done, 0));
  }
  return Q4_OK;
}

int dr_fusion_beam_step(const q4_model* model, q4_beam_state* state, const float* e, int32_t B,
                        int32_t T, int32_t W, int32_t iter, int32_t u_max, float lambda_t,
                        float lambda_s, float rho, int32_t mode, void* workspace,
                        size_t workspace_bytes, q4_stream stream) {
  return beam_step(model, state, e, B, T, W, iter, u_max, lambda_t, lambda_s, rho, mode, workspace, workspace_bytes, stream,
                   StepMode());
}

// ------------------------------------------------------------------------ whole search
// A step is 10 short kernels.  With few hypothesis rows they run in less time than the host takes to enqueue them one
// by one (about 45 us a step from Python), and that bounds the search.  A plan therefore holds PLAN_ITERS consecutive
// steps as a CUDA graph.  Its kernels read what changes between searches (frames, length, budget, iteration) from
// the head of the workspace, so one graph serves every search on its state.  228 iterations of one utterance
// (W = 4) with the encoder before them: 8.9 -> 8.1 ms with 4-bit weights, 10.9 -> 9.6 with 8-bit ones (host time 11 -> 1 ms);
// 5 utterances x 8 slots, 360 time-synchronous calls: 12.9 -> 11.9 ms.
namespace {
constexpr int PLAN_MIN_ITERS = 96;   // below, building the graph (1.0 ms of host time, once per kind of search and state) outweighs it
struct SearchKey {                   // everything the graph was built from
  q4_model model;
  q4_beam_state state;
  void* workspace;
  size_t workspace_bytes;
  int32_t B, W, tsd, dependent, exact, loop, sums;
  float lambda_t, lambda_s, rho;
};
// One graph and the search it was built for.  PLAN_GRAPHS of them: a decoder that alternates between a few batch sizes,
// beams or kinds of search, whose states come and go at the same addresses, builds one for each.
constexpr int PLAN_GRAPHS = 4;
struct SearchGraph {
  SearchKey key;
  int64_t launches, quant_calls;     // of the graph
  int64_t last_use;
  cudaEvent_t done;                  // of the last replay
  cudaGraphExec_t exec;
};
struct SearchPlan {
  SearchGraph graph[PLAN_GRAPHS];
  int64_t built, replays, failed;    // graphs made, replays enqueued, attempts to make a graph or a loop that failed
  int32_t test_failure;              // see q4_test_search_loop_failure_set
  int32_t last_iters, last_looped;   // steps of the last search; whether a loop ended them
  int64_t uses;
  // Captured on: the graphs' chains, none of the caller's streams.  side[2] or side[3] take the recurrent sums: up to 128 rows
  // with a lower priority than the rest, so that the launches of the joint network's chain do not queue
  // behind them (8 rows 3.83 -> 3.55 ms); with more rows the next step would wait for them (384 rows 5.1 -> 6.0).  Networks of
  // 1024, 1024 and 2048 cells: 192 tiles of products a row tile, for 148 SMs.
  cudaStream_t stream, side[4];
  cudaEvent_t side_event[4];
};
// While one of these lives, calls of this thread that a capture elsewhere in the process would take for unsafe (streams
// and events made or destroyed, a graph instantiated, an event asked) leave that capture alone: none of them
// concerns it.  A plan may be made, used or dropped while another thread captures.
struct BesideCaptures {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  BesideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~BesideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode); }
};
int step_mode(const SearchKey& k, int iter) {
  const int S1 = k.state.tsd_smax + 1;
  return !k.tsd ? 0 : iter % S1 == S1 - 1 ? 2 : 1;
}
}  // namespace

int q4_search_plan_create(q4_search_plan* out) {
  if (!out) return Q4_ERR_NULL;
  const BesideCaptures guard;
  SearchPlan* p = static_cast<SearchPlan*>(calloc(1, sizeof(SearchPlan)));
  if (!p) return Q4_ERR_CUDA;
  *out = p;
  int low = 0, high = 0;
  bool ok = cudaDeviceGetStreamPriorityRange(&low, &high) == cudaSuccess &&
            cudaStreamCreateWithPriority(&p->stream, cudaStreamNonBlocking, high) == cudaSuccess;
  for (int i = 0; i < PLAN_GRAPHS && ok; ++i)
    ok = cudaEventCreateWithFlags(&p->graph[i].done, cudaEventDisableTiming) == cudaSuccess;
  for (int i = 0; i < 4 && ok; ++i)
    ok = cudaStreamCreateWithPriority(&p->side[i], cudaStreamNonBlocking, i == 2 ? low : high) == cudaSuccess;
  for (int i = 0; i < 4 && ok; ++i) ok = cudaEventCreateWithFlags(&p->side_event[i], cudaEventDisableTiming) == cudaSuccess;
  if (ok) return Q4_OK;
  q4_search_plan_destroy(p);
  *out = nullptr;
  return Q4_ERR_CUDA;
}
int q4_search_plan_destroy(q4_search_plan plan) {
  if (!plan) return Q4_OK;
  const BesideCaptures guard;
  SearchPlan* p = static_cast<SearchPlan*>(plan);
  for (SearchGraph& g : p->graph) {
    if (g.exec) {
      cudaEventSynchronize(g.done);   // a replay of a search may be on its way
      cudaGraphExecDestroy(g.exec);
    }
    if (g.done) cudaEventDestroy(g.done);
  }
  if (p->stream) cudaStreamDestroy(p->stream);
  for (int i = 0; i < 4; ++i)
    if (p->side[i]) cudaStreamDestroy(p->side[i]);
  for (int i = 0; i < 4; ++i)
    if (p->side_event[i]) cudaEventDestroy(p->side_event[i]);
  free(p);
  return Q4_OK;
}

// PLAN_ITERS steps and the call's advance, captured on the plan's stream.  With a loop: the body of a graph's conditional
// node, whose last selection asks for another turn.
static int capture_steps(SearchPlan* p, SearchKey& key, const cudaGraphConditionalHandle* loop) {
  SearchCall* call = static_cast<SearchCall*>(key.workspace);
  // T and u_max (and the frames) only have to pass the argument checks here; the first frame's steps are never in the graph
  for (int it = PLAN_ITERS; it < 2 * PLAN_ITERS; ++it) {
    const StepMode how = {call, loop ? search_frozen(key.workspace) : nullptr, it == 2 * PLAN_ITERS - 1 ? loop : nullptr,
                          key.sums != 0, key.sums && key.state.aux_stream[0] ? p->side[key.B * key.W <= 128 ? 2 : 3] : nullptr,
                          p->side_event[3]};
    Q4_CHECK(beam_step(&key.model, &key.state, static_cast<const float*>(key.workspace), key.B, 1 << 24, key.W, it, 0,
                       key.lambda_t, key.lambda_s, key.rho, step_mode(key, it), key.workspace, key.workspace_bytes, p->stream,
                       how));
  }
  if (!loop) Q4_TRY(launch_search_advance(call, PLAN_ITERS, p->stream));
  return Q4_OK;
}
// A conditional node in `g`, behind nothing, that repeats the steps until every utterance is frozen while *handle is not 0;
// `first`: its value when the graph is launched.  A node that could not be filled stays in the graph (nodes cannot be
// taken out of a graph that is being captured), so there `first` is 0 and launch_search_begin sets the value.
static int add_search_loop(SearchPlan* p, SearchKey& key, cudaGraph_t g, unsigned first, cudaGraphNode_t* node,
                           cudaGraphConditionalHandle* handle) {
  cudaGraphNodeParams np = {};
  np.type = cudaGraphNodeTypeConditional;
  np.conditional.type = cudaGraphCondTypeWhile;
  np.conditional.size = 1;
  if (p->test_failure == 1 ||
      cudaGraphConditionalHandleCreate(&np.conditional.handle, g, first, cudaGraphCondAssignDefault) != cudaSuccess ||
      cudaGraphAddNode(node, g, nullptr, 0, &np) != cudaSuccess || p->test_failure == 2 ||
      cudaStreamBeginCaptureToGraph(p->stream, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                    cudaStreamCaptureModeRelaxed) != cudaSuccess)
    return Q4_ERR_CUDA;
  *handle = np.conditional.handle;
  int r = capture_steps(p, key, handle);
  if (cudaStreamEndCapture(p->stream, nullptr) != cudaSuccess && r == Q4_OK) r = Q4_ERR_CUDA;
  return r;
}

// The graph of a search: the one that was built for the same arguments, else a new one in a free place or in
// place of the one used longest ago whose last replay has ended.  Null (the search then enqueues its steps one by one)
// if there is no such place, for the host does not wait for a replay here, or if the graph cannot be built.
static SearchGraph* plan_graph(SearchPlan* p, const SearchKey& key) {
  SearchGraph* place = nullptr;
  for (SearchGraph& g : p->graph)
    if (g.exec && memcmp(&g.key, &key, sizeof(key)) == 0) {
      g.last_use = ++p->uses;
      return &g;
    }
  for (SearchGraph& g : p->graph)
    if ((!g.exec || cudaEventQuery(g.done) == cudaSuccess) && (!place || g.last_use < place->last_use)) place = &g;
  if (cudaPeekAtLastError() == cudaErrorNotReady) cudaGetLastError();   // an event that is not ready is no error
  if (!place) return nullptr;
  if (place->exec) cudaGraphExecDestroy(place->exec);
  place->exec = nullptr;
  place->last_use = 0;
  memcpy(&place->key, &key, sizeof(key));   // padding included: keys are compared as bytes
  const int64_t l0 = g_launches, q0 = g_quant_calls;
  cudaGraph_t g = nullptr;
  int r;
  if (key.loop) {
    cudaGraphNode_t node;
    cudaGraphConditionalHandle handle;
    r = cudaGraphCreate(&g, 0) == cudaSuccess ? add_search_loop(p, place->key, g, 1, &node, &handle) : Q4_ERR_CUDA;
  } else {
    r = cudaStreamBeginCapture(p->stream, cudaStreamCaptureModeRelaxed) == cudaSuccess ? Q4_OK : Q4_ERR_CUDA;
    if (r == Q4_OK) {
      r = capture_steps(p, place->key, nullptr);
      if (cudaStreamEndCapture(p->stream, &g) != cudaSuccess && r == Q4_OK) r = Q4_ERR_CUDA;
    }
  }
  if (r == Q4_OK && cudaGraphInstantiate(&place->exec, g, cudaGraphInstantiateFlagUseNodePriority) != cudaSuccess) r = Q4_ERR_CUDA;
  if (g) cudaGraphDestroy(g);
  place->launches = g_launches - l0;
  place->quant_calls = g_quant_calls - q0;
  g_launches = l0;
  g_quant_calls = q0;
  ++(r == Q4_OK ? p->built : p->failed);
  if (r != Q4_OK) {
    place->exec = nullptr;
    cudaGetLastError();
    return nullptr;
  }
  place->last_use = ++p->uses;
  return place;
}

int q4_test_search_loop_failure_set(q4_search_plan plan, int32_t where) {
  if (!plan) return Q4_ERR_NULL;
  if (where < 0 || where > 2) return Q4_ERR_UNSUPPORTED;
  static_cast<SearchPlan*>(plan)->test_failure = where;
  return Q4_OK;
}
int q4_search_steps_taken(q4_search_plan plan, const void* workspace, q4_stream stream, int32_t* steps) {
  if (!plan || !workspace || !steps) return Q4_ERR_NULL;
  const SearchPlan* p = static_cast<const SearchPlan*>(plan);
  *steps = p->last_iters;
  if (!p->last_looped) return Q4_OK;
  SearchCall call;
  Q4_TRY(cudaMemcpyAsync(&call, workspace, sizeof(call), cudaMemcpyDeviceToHost, S(stream)));
  Q4_TRY(cudaStreamSynchronize(S(stream)));
  const int taken = call.iter + PLAN_ITERS;   // (the call's number is that of the turn's first step, less PLAN_ITERS)
  if (taken < *steps) *steps = taken;
  return Q4_OK;
}
int q4_search_plan_info(q4_search_plan plan, int64_t* out) {
  if (!plan || !out) return Q4_ERR_NULL;
  const SearchPlan* p = static_cast<const SearchPlan*>(plan);
  out[0] = p->built;
  out[1] = p->replays;
  out[2] = p->failed;
  return Q4_OK;
}

int q4_beam_search(const q4_model* model, q4_beam_state* state, const float* e, int32_t B, int32_t T, int32_t W, int32_t u_max,
                   float lambda_t, float lambda_s, float rho, int32_t time_synchronous, void* workspace,
                   size_t workspace_bytes, q4_search_plan plan, q4_stream stream) {
  if (!model || !state || !workspace) return Q4_ERR_NULL;
  const int S1 = time_synchronous ? state->tsd_smax + 1 : 1, n_iters = time_synchronous ? T * S1 : T + u_max;
  if (n_iters == 0) return Q4_OK;   // no steps: the state stays as q4_beam_init left it
  if (!e) return Q4_ERR_NULL;
  if (T <= 0 || u_max < 0) return Q4_ERR_DIM;
  if (time_synchronous && (state->tsd_smax < 0 || state->tsd_smax > 3)) return Q4_ERR_DIM;
  SearchKey key;
  memset(&key, 0, sizeof(key));
  memcpy(&key.model, model, sizeof(key.model));
  memcpy(&key.state, state, sizeof(key.state));
  key.workspace = workspace;
  key.workspace_bytes = workspace_bytes;
  key.B = B;
  key.W = W;
  key.tsd = time_synchronous != 0;
  key.dependent = g_dependent_launch;
  key.exact = select_exact_only();
  key.lambda_t = lambda_t;
  key.lambda_s = lambda_s;
  key.rho = rho;
  cudaStream_t s = S(stream);
  // The graph's side chains are captured on the plan's own streams: a stream lent by the caller may be in use for other
  // work meanwhile, which would be captured with them.
  SearchPlan* p = static_cast<SearchPlan*>(plan);
  const q4_beam_state& st = key.state;
  const bool lent = st.aux_stream[0] && st.aux_stream[1] && st.aux_event[0] && st.aux_event[1] && st.aux_event[2];
  for (int i = 0; i < 2; ++i) key.state.aux_stream[i] = p && lent ? p->side[i] : nullptr;
  for (int i = 0; i < 3; ++i) key.state.aux_event[i] = p && lent ? p->side_event[i] : nullptr;
  // An alignment-length synchronous search ends its steps when no utterance has labels left to propose; the iterations
  // that are left then are carried out together.
  const bool sums = search_keeps_sums(*model, *state, B, W, workspace, workspace_bytes);
  key.sums = sums;
  key.loop = p && !key.tsd && !key.exact && search_tail_supported(model->V, model->D) && aligned16(state->pred_p) &&
             (sums || search_uses_tensor_cores(*model, *state, B, W, workspace_bytes));
  // step by step: while launches are timed or waits are made to run out (a graph would keep that), in a short search, and
  // without a loop in a stream that is being captured
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (p && (n_iters < PLAN_MIN_ITERS || timing_active() || test_wait_expiry_active() ||
            cudaStreamIsCapturing(s, &cap) != cudaSuccess || (cap != cudaStreamCaptureStatusNone && !key.loop)))
    p = nullptr;
  bool tail = false;
  SearchPlan* const plan_of_call = static_cast<SearchPlan*>(plan);
  for (int it = 0; it < n_iters;) {
    // the first two frames' steps always: the first step's networks start from the reset state, and the kernels set their
    // attributes at their first launch
    if (p && it == 2 * S1) {
      const BesideCaptures guard;          // the first replay of a graph may allocate, too
      SearchCall* call = static_cast<SearchCall*>(workspace);
      int32_t* frozen = key.loop ? search_frozen(workspace) : nullptr;
      const int groups = (n_iters - it) / PLAN_ITERS;
      const int turns = key.loop ? (n_iters - it + PLAN_ITERS - 1) / PLAN_ITERS : groups;
      if (cap != cudaStreamCaptureStatusNone) {   // the loop becomes a node of the caller's graph, if it can be one
        const int64_t l0 = g_launches, q0 = g_quant_calls;
        cudaGraph_t g;
        const cudaGraphNode_t* deps;
        size_t n_deps;
        cudaGraphNode_t node;
        cudaGraphConditionalHandle handle;
        Q4_TRY(cudaStreamGetCaptureInfo_v2(s, &cap, nullptr, &g, &deps, &n_deps));
        if (add_search_loop(p, key, g, 0, &node, &handle) == Q4_OK) {
          g_launches += (g_launches - l0) * (turns - 1);
          g_quant_calls = q0 + (g_quant_calls - q0) / PLAN_ITERS * (n_iters - it);   // every step's, whoever carries it out
          Q4_TRY(launch_search_begin(call, e, T, u_max, it - PLAN_ITERS, frozen, B, s, &handle));
          Q4_TRY(cudaStreamGetCaptureInfo_v2(s, &cap, nullptr, &g, &deps, &n_deps));
          if (n_deps != 1) return Q4_ERR_CUDA;   // the launch above
          const cudaGraphNode_t begin = deps[0];
          Q4_TRY(cudaGraphAddDependencies(g, &begin, &node, 1));
          Q4_TRY(cudaStreamUpdateCaptureDependencies(s, &node, 1, cudaStreamSetCaptureDependencies));
          tail = true;
        } else {
          g_launches = l0;
          g_quant_calls = q0;
          ++p->failed;
          cudaGetLastError();
        }
      } else if (SearchGraph* g = plan_graph(p, key)) {
        Q4_TRY(launch_search_begin(call, e, T, u_max, it - PLAN_ITERS, frozen, B, s));
        for (int i = 0; i < (key.loop ? 1 : groups); ++i) {
          const cudaError_t le = cudaGraphLaunch(g->exec, s);
          if (le != cudaSuccess) {
            cudaEventRecord(g->done, s);   // of the replays before it
            return Q4_ERR_CUDA;
          }
        }
        g_launches += g->launches * turns;
        g_quant_calls += key.loop ? g->quant_calls / PLAN_ITERS * (n_iters - it) : g->quant_calls * groups;
        p->replays += groups;
        Q4_TRY(cudaEventRecord(g->done, s));
        tail = key.loop != 0;
        if (!tail) it += groups * PLAN_ITERS;
      }
      if (tail) break;
      p = nullptr;                         // the rest step by step
      if (it >= n_iters) break;
    }
    Q4_CHECK(beam_step(model, state, e, B, T, W, it, u_max, lambda_t, lambda_s, rho, step_mode(key, it), workspace,
                       workspace_bytes, stream, StepMode{nullptr, nullptr, nullptr, sums, nullptr, nullptr}));
    ++it;
  }
  if (plan_of_call) {
    plan_of_call->last_iters = n_iters;
    plan_of_call->last_looped = tail;
  }
  if (tail) {
    const q4_model& m = *model;
    TailArgs a;
    memset(&a, 0, sizeof(a));
    a.call = static_cast<SearchCall*>(workspace);
    a.frozen = search_frozen(workspace);
    a.st = *state;
    a.B = B;
    a.W = W;
    a.V = m.V;
    a.z_act = m.z_act;
    a.sc_out = m.joint_out.w.scale;
    a.b_out = m.joint_out.bias;
    Q4_TRY(launch_search_tail(a, T, static_cast<const int8_t*>(m.prepared) + plan_prepared(m).lin[5], s));
  }
  return Q4_OK;
}

int q4_traceback(const q4_beam_state* state, int32_t B, int32_t W, int32_t n_iters,
                 int32_t u_max, int32_t* tokens, int32_t* lens, float* scores, q4_stream stream) {
  Q4_CHECK(check_state(state, 1));
  if (!tokens || !lens || !scores) return Q4_ERR_NULL;
  if (B <= 0 || W <= 0 || W > 16 || n_iters < 0 || u_max <= 0) return Q4_ERR_DIM;
  Q4_TRY(launch_traceback(*state, B, W, n_iters, u_max, tokens, lens, scores, S(stream)));
  return Q4_OK;
}

}  // extern "C"
