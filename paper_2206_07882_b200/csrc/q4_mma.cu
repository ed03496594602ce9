// Tensor-core path (sm_100a): TMA-fed tcgen05 kind::i8 GEMMs with int32 accumulators in
// tensor memory.  Activations are the M operand (128 rows per tile), weight rows the N
// operand, both K-major int8 in shared memory under the 128-byte swizzle.
//   k_mma_gemm : D[128 x 32..256] tiles, epilogues: de-quantize+bias / re-quantize / joint element-wise;
//   k_mma_gemm_persistent : the same main loop with the int32 sums stored as they are.
//   k_mma_lstm : D_ih, D_hh[128 x 64 or 128] tiles (16 or 32 cells x 4 gates, gate-interleaved weight
//                rows) with the whole LSTM cell update fused into the epilogue;
//   k_mma_lmhead : bottleneck, re-quantization, output layer and log-softmax of a row tile on a cluster of CTAs.
// Warp roles per CTA: epilogue warps (one TMEM lane quarter each), one producer warp, one MMA issuer warp (an
// elected lane of each issues).  Codes are unpacked to int8 before they meet the tensor cores: rows of a call by
// k_unpack_multi, a layer's input and weights by k_layer_prepare, weights once by k_prepare_w.
#include <string.h>

#include "q4_internal.h"
#include "q4_mma.cuh"

namespace q4 {

constexpr int BM = 128;          // activation rows per tile
constexpr int BK = 128;          // K bytes per pipeline stage (one swizzle row)
template <int BN>
constexpr int GEMM_STAGES = BN >= 128 ? 4 : 6;   // ring depth of the plain GEMM with BN weight rows per tile
constexpr int LSTM_MAX_STAGES = 8;
constexpr int LSTM_RING = 96 * 1024;   // bytes of operand ring per CTA of the LSTM kernel: two CTAs per SM
constexpr int LSTM_SMEM_MAX = LSTM_RING + 10 * 1024;
constexpr int LSTM_EPI_WARPS = 8;

// ------------------------------------------------------------------ operand preparation
__device__ __forceinline__ void unpack_piece32(const uint8_t* p, int k, int bits, bool is_signed, uint32_t zp4, uint4& o0,
                                               uint4& o1) {   // 32 codes of a row -> int8, natural order
  if (bits == 4) {
    const uint4 v = *reinterpret_cast<const uint4*>(p + (k >> 1));
    unpack8_natural(v.x, is_signed, zp4, o0.x, o0.y);
    unpack8_natural(v.y, is_signed, zp4, o0.z, o0.w);
    unpack8_natural(v.z, is_signed, zp4, o1.x, o1.y);
    unpack8_natural(v.w, is_signed, zp4, o1.z, o1.w);
  } else if (bits == 2) {
    const uint2 v = *reinterpret_cast<const uint2*>(p + (k >> 2));
    uint32_t a[4], b[4];
    unpack16x2(v.x, a);
    unpack16x2(v.y, b);
    o0 = make_uint4(a[0], a[1], a[2], a[3]);
    o1 = make_uint4(b[0], b[1], b[2], b[3]);
  } else {
    o0 = *reinterpret_cast<const uint4*>(p + k);
    o1 = *reinterpret_cast<const uint4*>(p + k + 16);
  }
}
// Gather + unpack activation rows to int8, dst[n, k] = code(src[idx[n], k]) - zero_point: several
// jobs in one launch (blockIdx.y selects the job).  The grid is sized for the SMs, not for the
// padded row count: each thread strides over the 32-element pieces of the rows that carry work
// (their number may be known on the device only).
__global__ void __launch_bounds__(256) k_unpack_multi(const __grid_constant__ UnpackJobs jobs) {
  // A dependent successor may set itself up; it reads nothing before this grid has completed but, in a search, the count
  // of rows with work (see tile_without_work), so there the trigger has to follow the wait.
  if (!jobs.n_active) pdl_trigger();
  pdl_wait();      // launched as a programmatic dependent itself: the source rows may be the predecessor's output
  if (jobs.n_active) pdl_trigger();
  if (jobs.clear64 && (blockIdx.x | blockIdx.y) == 0 && threadIdx.x < 64) jobs.clear64[threadIdx.x] = 0;   // the call's status block
  const UnpackJob& j = jobs.job[blockIdx.y];
  const uint32_t per_row = (uint32_t)j.k_pad >> 5;
  int rows = jobs.n_rows_pad;
  if (!jobs.zero_tail) {   // rows without work need not be cleared every time
    rows = jobs.n_rows;
    if (jobs.n_active) rows = min(rows, *jobs.n_active);
  }
  const int n_work = jobs.n_active ? min(jobs.n_rows, *jobs.n_active) : jobs.n_rows;
  const uint32_t zp4 = (uint32_t)j.zp * 0x01010101u;
  const uint32_t total = (uint32_t)rows * per_row;   // checked by the launcher to fit
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int n = (int)(i / per_row), k = (int)(i - (uint32_t)n * per_row) * 32;
    uint4 o0 = make_uint4(0, 0, 0, 0), o1 = o0;
    int r = -1;
    if (n < n_work) r = j.idx ? j.idx[n] : n;
    if (r >= 0) unpack_piece32(j.src + (long long)r * j.src_stride, k, j.bits, j.is_signed != 0, zp4, o0, o1);
    uint4* d = reinterpret_cast<uint4*>(j.dst + (long long)n * j.dst_stride + k);
    d[0] = o0;
    d[1] = o1;
  }
}

cudaError_t launch_unpack_multi(const UnpackJobs& jobs, cudaStream_t s, bool dependent) {
  if (jobs.n_jobs <= 0) return cudaSuccess;
  int kmax = 0;
  for (int i = 0; i < jobs.n_jobs; ++i) kmax = jobs.job[i].k_pad > kmax ? jobs.job[i].k_pad : kmax;
  const long long total = (long long)jobs.n_rows_pad * (kmax >> 5);
  if (total > INT32_MAX) return cudaErrorInvalidValue;
  long long blocks = (total + 255) / 256;
  const long long cap = (6 * sm_count() + jobs.n_jobs - 1) / jobs.n_jobs;   // about six CTAs per SM in all: one or two
                                                                     // pieces per thread at 1024 rows
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  dim3 grid((unsigned)blocks, jobs.n_jobs);
  timing_begin(s);
  cudaError_t e = launch_ex(k_unpack_multi, grid, dim3(256), 0, s, dependent, 1, jobs);
  timing_end(s);
  ++g_launches;
  return e != cudaSuccess ? e : cudaGetLastError();
}
void add_unpack_job(UnpackJobs& u, const void* src, long long src_stride, const int32_t* idx, const q4_act& act, int k_pad,
                    int8_t* dst) {
  UnpackJob& j = u.job[u.n_jobs++];
  j.src = static_cast<const uint8_t*>(src);
  j.src_stride = src_stride;
  j.idx = idx;
  j.bits = act.bits;
  j.is_signed = act.is_signed;
  j.zp = act.zero_point;
  j.k_pad = k_pad;
  j.dst = dst;
  j.dst_stride = k_pad;
}

// Weight preparation: unpack to int8; with `interleave` the 4H rows (gate-major i,f,g,o) are
// reordered to row 4*cell + gate so that one thread of the epilogue owns all gates of a cell.
__global__ void __launch_bounds__(256) k_prepare_w(const uint8_t* src, int bits, int rows, int k_pad,
                                                   int interleave, int8_t* dst, long long dst_stride,
                                                   int col0) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int per_row = k_pad >> 3;
  if (i >= (long long)rows * per_row) return;
  const int r = (int)(i / per_row), k = (int)(i % per_row) * 8;
  int ro = r;
  if (interleave) {
    const int H = rows >> 2;
    ro = 4 * (r % H) + r / H;
  }
  uint2 o;
  if (bits == 4) {
    const uint32_t w = *reinterpret_cast<const uint32_t*>(src + (long long)r * (k_pad >> 1) + (k >> 1));
    uint32_t lo = 0, hi = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int a = (((w >> (4 * e)) & 0xF) ^ 8) - 8, c = (((w >> (4 * (e + 4))) & 0xF) ^ 8) - 8;
      lo |= (uint32_t)(a & 0xFF) << (8 * e);
      hi |= (uint32_t)(c & 0xFF) << (8 * e);
    }
    o = make_uint2(lo, hi);
  } else if (bits == 2) {   // four codes per byte, element i in bits 2i, 2i+1 of the 16-bit group
    const uint32_t w = *reinterpret_cast<const uint16_t*>(src + (long long)r * (k_pad >> 2) + (k >> 2));
    uint32_t lo = 0, hi = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int a = (int)(((w >> (2 * e)) & 3u) ^ 2u) - 2, c = (int)(((w >> (2 * (e + 4))) & 3u) ^ 2u) - 2;
      lo |= (uint32_t)(a & 0xFF) << (8 * e);
      hi |= (uint32_t)(c & 0xFF) << (8 * e);
    }
    o = make_uint2(lo, hi);
  } else {
    o = *reinterpret_cast<const uint2*>(src + (long long)r * k_pad + k);
  }
  *reinterpret_cast<uint2*>(dst + (long long)ro * dst_stride + col0 + k) = o;
}
__global__ void k_prepare_vec(const float* src, int rows, int interleave, float* dst, float mul) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= rows) return;
  int ro = r;
  if (interleave) {
    const int H = rows >> 2;
    ro = 4 * (r % H) + r / H;
  }
  dst[ro] = src ? __fmul_rn(mul, src[r]) : 0.0f;   // mul = 1 leaves the value as it is
}

cudaError_t launch_prepare_w(const q4_mat& w, int interleave, int8_t* dst, long long dst_stride,
                             int col0, cudaStream_t s) {
  const long long total = (long long)w.rows * (w.k_pad >> 3);
  timing_begin(s);
  k_prepare_w<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(static_cast<const uint8_t*>(w.q), w.bits,
                                                              w.rows, w.k_pad, interleave, dst,
                                                              dst_stride, col0);
  timing_end(s);
  ++g_launches;
  return cudaGetLastError();
}
cudaError_t launch_prepare_vec(const float* src, int rows, int interleave, float* dst, cudaStream_t s, float mul) {
  k_prepare_vec<<<(rows + 255) / 256, 256, 0, s>>>(src, rows, interleave, dst, mul);
  ++g_launches;
  return cudaGetLastError();
}

// Everything a layer call prepares, in one launch: int8 copies of the input codes and of all
// directions' weights (rows reordered to 4*cell+gate), row scales and biases in the same order, and
// a cleared status block.  (As separate launches: a memset and 11 kernels of 2 us each per bidirectional layer.)  blockIdx.x walks the jobs' blocks one after the other.
__global__ void __launch_bounds__(256) k_layer_prepare(const __grid_constant__ LayerPrep a) {
  pdl_trigger();
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x < 64 && a.clear64) a.clear64[threadIdx.x] = 0;
  int blk = blockIdx.x, ji = 0;
  while (ji + 1 < a.n_mats && blk >= a.mat[ji].blocks) blk -= a.mat[ji++].blocks;
  const LayerPrepMat& m = a.mat[ji];
  if (blk < m.blocks) {   // a matrix of codes
    const long long i = (long long)blk * 256 + threadIdx.x;
    const int per_row = m.k_pad >> 5;
    if (i >= m.rows * per_row) return;
    const long long r = i / per_row;
    const int k = (int)(i % per_row) * 32;
    uint4 o0, o1;
    unpack_piece32(m.src + r * ((long long)m.k_pad * m.bits / 8), k, m.bits, m.is_signed != 0, (uint32_t)m.zp * 0x01010101u,
                   o0, o1);
    const int H = m.interleave;
    const long long ro = H > 0 ? 4 * (r % H) + r / H : r;
    uint4* d = reinterpret_cast<uint4*>(m.dst + ro * m.k_pad + k);
    d[0] = o0;
    d[1] = o1;
    return;
  }
  // the row vectors: one block per 256 rows of each
  blk -= m.blocks;
  const int per = (4 * a.H + 255) / 256, v = blk / per, r = (blk % per) * 256 + threadIdx.x;
  if (v >= a.n_vecs || r >= 4 * a.H) return;
  a.vec_dst[v][4 * (r % a.H) + r / a.H] = a.vec_src[v] ? a.vec_src[v][r] : 0.0f;
}
cudaError_t launch_layer_prepare(LayerPrep a, cudaStream_t s, bool dependent) {
  long long total = 0;
  for (int i = 0; i < a.n_mats; ++i) {
    const long long b = (a.mat[i].rows * (a.mat[i].k_pad >> 5) + 255) / 256;
    a.mat[i].blocks = (int)b;
    total += b;
  }
  total += (long long)a.n_vecs * ((4 * a.H + 255) / 256);
  timing_begin(s);
  const cudaError_t e = launch_ex(k_layer_prepare, dim3((unsigned)total), dim3(256), 0, s, dependent, 1, a);
  timing_end(s);
  ++g_launches;
  return e != cudaSuccess ? e : cudaGetLastError();
}

// ------------------------------------------------------------------ tensor maps (host)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// int8 matrix [rows, k] with row pitch `pitch` bytes; box = 128 bytes of K x box_rows rows.
bool make_tmap_i8(CUtensorMap* m, const void* base, uint64_t k, uint64_t rows, uint64_t pitch,
                  uint32_t box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  if ((reinterpret_cast<uintptr_t>(base) & 15u) || (pitch & 15u)) return false;
  const cuuint64_t dims[2] = {k, rows};
  const cuuint64_t strides[1] = {pitch};
  const cuuint32_t box[2] = {BK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

__device__ __forceinline__ void flag_timeout(int32_t* status) {
  if (status) atomicExch(status, Q4_ERR_TIMEOUT);
}

// Row tiles without work (n_active: the device's count of rows with work in a search step).  A tile beyond the count
// leaves as its first act, before it has set anything up or waited: in an iteration without labels (two of three in
// speech) that is every tile of seven kernels, and tiles that found out after their set-up cost 150 iterations with few
// labels 1 x 16 slots 3.59 against 3.43 ms, 4 x 8 slots of the paper's model 3.36 against 3.10.
//   The count is the one thing that is read before the kernel's wait.  The selection writes it; the first kernel of
// a step's chains (the gather, the weight-streaming step or a kernel behind an event) triggers its successor only after its own wait
// for the selection, and every later kernel of a chain starts after that.  So the count is in memory when any of these
// kernels starts, and a load that is coherent at device scope cannot meet an older copy of it.  (Nothing else is read on
// its word, so it need not acquire: that would drop the SM's L1 under the kernels beside it.)
//   A grid whose tiles all leave must not complete before its predecessor does, because its successor waits for this
// grid only: one CTA of the first row tile, which leaves only if all do, waits before it leaves.
__device__ __forceinline__ bool tile_without_work(const int32_t* n_active, int m0) {
  if (!n_active) return false;
  if (m0 < ld_coherent(n_active)) return false;
  if (m0 == 0 && blockIdx.x == 0) {
    pdl_trigger();
    pdl_wait();
  }
  return true;
}

// ------------------------------------------------------------------ plain GEMM
struct MmaGemmArgs {
  int M, J, K, epi;
  void* out;
  long long ldo;            // elements (int32 / float) or bytes (codes) between output rows
  const int32_t* out_idx;   // output row of activation row m (nullptr = m, negative = skip)
  const float* w_scale;
  const float* bias;
  float x_scale;
  q4_act out_act;
  int32_t* status;
  const int32_t* n_active;
  const int32_t* n_idle;    // optional: nothing to do once *n_idle >= all_idle
  int32_t all_idle;
  const float* mul_e;       // EPI_JOINTZ: the other factor, row mul_idx[m] of [*, J] fp32
  const int32_t* mul_idx;
  uint32_t wait_limit;      // polls before a wait gives up
  int32_t skip_producer;    // test hook: the producer issues no copy, so the consumer's wait runs out
};

// Test hook (q4_test_wait_expiry_set): the next launches of k_mma_gemm get this limit and flag.
constexpr uint32_t WAIT_LIMIT = 1u << 22;   // polls
static uint32_t g_wait_limit = WAIT_LIMIT, g_ring_wait_limit = WAIT_LIMIT;
static int g_skip_producer = 0;
// mode 1: no copies, short waits in k_mma_gemm; 2: short waits in k_state_products
void test_wait_expiry_set(int mode, uint32_t wait_limit) {
  g_skip_producer = mode == 1;
  g_wait_limit = mode == 1 && wait_limit ? wait_limit : WAIT_LIMIT;
  g_ring_wait_limit = mode == 2 ? wait_limit : WAIT_LIMIT;
}
bool test_wait_expiry_active() { return g_skip_producer != 0 || g_ring_wait_limit != WAIT_LIMIT; }
uint32_t test_ring_wait_limit() { return g_ring_wait_limit; }

template <int GEMM_BN>
__global__ void __launch_bounds__(192, 1)
k_mma_gemm(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b,
           const MmaGemmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  constexpr int A_BYTES = BM * BK, B_BYTES = GEMM_BN * BK, STAGE = A_BYTES + B_BYTES;
  constexpr int NS = GEMM_STAGES<GEMM_BN>;
  __shared__ uint64_t full[NS], empty[NS], acc_full;
  __shared__ uint32_t tmem_base_s;
  __shared__ float s_sc[GEMM_BN], s_bi[GEMM_BN];   // de-quantization constants of this tile's columns
  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * GEMM_BN;   // row tiles slowest: tiles with work are dispatched first
  const int nk = (a.K + BK - 1) / BK;
  const int mm = umma_rows(a.M);
  if (tile_without_work(a.n_active, m0)) return;

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&acc_full, 1);
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == 5) tmem_alloc(&tmem_base_s, GEMM_BN);
  if (warp == 4 && lane == 0) {
    prefetch_tmap(&tma_a);
    prefetch_tmap(&tma_b);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  pdl_wait();   // everything above overlaps the tail of the previous kernel of the stream
  if (a.n_idle && ld_coherent(a.n_idle) >= a.all_idle) {   // the same for every thread of the grid
    pdl_trigger();
  } else if (warp == 4) {
    const uint32_t on = elect_one();
    bool ok = true;
    int s = 0;
    uint32_t ph = 1;
    for (int i = 0; i < nk && ok && !a.skip_producer; ++i) {
      ok = i < NS || mbar_wait_warp(&empty[s], ph, a.wait_limit);   // (a stage that has never been filled is free)
      if (!ok) break;
      mbar_expect_tx(on, &full[s], STAGE);
      tma_load_2d(on, smem + s * STAGE, &tma_a, i * BK, m0, &full[s]);
      tma_load_2d(on, smem + s * STAGE + A_BYTES, &tma_b, i * BK, n0, &full[s]);
      if (++s == NS) {
        s = 0;
        ph ^= 1;
      }
    }
    pdl_trigger();
    if (!ok && lane == 0) flag_timeout(a.status);
  } else if (warp == 5) {
    const uint32_t idesc = umma_idesc_i8(mm, GEMM_BN);
    const uint32_t on = elect_one();
    bool ok = true, ready = mbar_test(&full[0], 0);
    int s = 0;
    uint32_t ph = 0;
    for (int i = 0; i < nk && ok; ++i) {
      ok = mbar_wait_warp_tested(ready, &full[s], ph, a.wait_limit);
      if (!ok) break;
      tc_fence_after();
      const int st = s;
      if (++s == NS) {
        s = 0;
        ph ^= 1;
      }
      ready = mbar_test(&full[s], ph);
      const uint64_t da = umma_desc_sw128(smem_u32(smem + st * STAGE));
      const uint64_t db = umma_desc_sw128(smem_u32(smem + st * STAGE + A_BYTES));
#pragma unroll
      for (int kk = 0; kk < BK / 32; ++kk) umma_i8(on, tmem, da + 2 * kk, db + 2 * kk, idesc, (i | kk) != 0);
      umma_commit(on, &empty[st]);
    }
    if (!ok) {   // recorded before the epilogue is released, so that it stores nothing
      if (lane == 0) flag_timeout(a.status);
      __threadfence();
      __syncwarp();
    }
    umma_commit(on, &acc_full);
    pdl_trigger();
  } else if (warp < 4) {
    for (int c = tid; c < GEMM_BN; c += 128) {   // stage scale * row scale and bias while the MMAs run
      const int j = min(n0 + c, a.J - 1);
      s_sc[c] = __fmul_rn(a.x_scale, __ldg(a.w_scale + j));
      s_bi[c] = a.bias ? __ldg(a.bias + j) : 0.0f;
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    bool ok = mbar_wait(&acc_full, 0, a.wait_limit);
    if (ok && a.status && *reinterpret_cast<volatile int32_t*>(a.status) != 0) ok = false;   // a wait gave up somewhere
    tc_fence_after();
    pdl_trigger();   // the main loop is over: the next kernel may set itself up
    if (!ok && lane == 0) flag_timeout(a.status);
    const int mi = m0 + umma_lane_row(mm, warp, lane);
    int m = -1;
    if (mi < a.M && !(a.n_active && mi >= *a.n_active)) m = a.out_idx ? a.out_idx[mi] : mi;
    const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
    for (int c0 = 0; c0 < GEMM_BN; c0 += 32) {
      int r[32];
      tmem_ld32(taddr + c0, r);
      tmem_ld_wait();
      const int j0 = n0 + c0;
      if (!ok || m < 0 || j0 >= a.J) continue;
      float v[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = __fmaf_rn((float)r[i], s_sc[c0 + i], s_bi[c0 + i]);
      if (a.epi == EPI_JOINTZ) {
        // joint network: z = tanh(e * p) with p the projected value just formed; quantized below.  A row without a
        // frame (negative index) has z = 0, as in k_joint_z
        const int er_idx = a.mul_idx[mi];
        if (er_idx >= 0) {
          const float* er = a.mul_e + (long long)er_idx * a.J + j0;
#pragma unroll
          for (int i = 0; i < 32; i += 4) {
            const float4 ev = *reinterpret_cast<const float4*>(er + i);
            v[i] = tanh_fixed(__fmul_rn(ev.x, v[i]));
            v[i + 1] = tanh_fixed(__fmul_rn(ev.y, v[i + 1]));
            v[i + 2] = tanh_fixed(__fmul_rn(ev.z, v[i + 2]));
            v[i + 3] = tanh_fixed(__fmul_rn(ev.w, v[i + 3]));
          }
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = 0.0f;
        }
      }
      if (a.epi == EPI_F32) {
        float* o = reinterpret_cast<float*>(a.out) + (long long)m * a.ldo + j0;
        if (j0 + 32 <= a.J && (reinterpret_cast<uintptr_t>(o) & 31) == 0) {
#pragma unroll
          for (int i = 0; i < 32; i += 8)
            st_global_v8(o + i, make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]),
                         make_float4(v[i + 4], v[i + 5], v[i + 6], v[i + 7]));
        } else if (j0 + 32 <= a.J && (reinterpret_cast<uintptr_t>(o) & 15) == 0) {
#pragma unroll
          for (int i = 0; i < 32; i += 4) *reinterpret_cast<float4*>(o + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        } else {   // ragged columns, or rows that are no multiple of 16 bytes apart
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (j0 + i < a.J) o[i] = v[i];
        }
      } else {  // EPI_QUANT8 / EPI_JOINTZ (J a multiple of 32)
        const int lo = act_lo(a.out_act), hi = act_hi(a.out_act);
        uint8_t* o = reinterpret_cast<uint8_t*>(a.out) + (long long)m * a.ldo;
        uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < 32; ++i)
          w[i >> 2] |= (uint32_t)((quantize1(v[i], a.out_act.inv_scale, a.out_act.zero_point, lo, hi) -
                                   a.out_act.zero_point) & 0xFF) << (8 * (i & 3));
        *reinterpret_cast<uint4*>(o + j0) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(o + j0 + 16) = make_uint4(w[4], w[5], w[6], w[7]);
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 5) tmem_dealloc(tmem, GEMM_BN);
}

// ------------------------------------------------------------------ persistent GEMM, int32 out
// The encoder input projection is one large GEMM per layer and direction (thousands of tiles)
// whose int32 result (128 KB per tile) costs more time to write than its MMAs take.  One CTA per
// SM walks the tiles t = blockIdx.x, blockIdx.x + gridDim.x, ... (column tile fastest, so the
// CTAs working at the same time share activation rows and all weights in L2), with two
// accumulators in tensor memory: the epilogue warps drain one while the MMAs of the next tile
// fill the other, and the operand ring keeps streaming across tile boundaries.
//
// The directions of a bidirectional layer are planes of one launch: plane p multiplies weight rows
// [p J, (p + 1) J) of the weight map and stores at out + p * plane_out; the column tiles of all planes
// are walked together (tiles_n per plane).
template <int GEMM_BN>
__global__ void __launch_bounds__(192, 1)
k_mma_gemm_persistent(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b,
                      const MmaGemmArgs a, const int tiles_m, const int tiles_n, const int planes,
                      const long long plane_out) {
  constexpr int PG_STAGES = GEMM_STAGES<GEMM_BN>;
  constexpr int TCOLS = 2 * GEMM_BN;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  constexpr int A_BYTES = BM * BK, B_BYTES = GEMM_BN * BK, STAGE = A_BYTES + B_BYTES;
  __shared__ uint64_t full[PG_STAGES], empty[PG_STAGES], acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_base_s;
  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const int nk = (a.K + BK - 1) / BK;
  const int cols = tiles_n * planes, n_tiles = tiles_m * cols;

  if (tid == 0) {
    for (int s = 0; s < PG_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 4);   // one arrival per epilogue warp
    }
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == 5) tmem_alloc(&tmem_base_s, TCOLS);
  if (warp == 4 && lane == 0) {
    prefetch_tmap(&tma_a);
    prefetch_tmap(&tma_b);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  pdl_wait();

  if (warp == 4) {
    // ---- TMA producer: the ring position runs on across tiles
    const uint32_t on = elect_one();
    bool ok = true;
    int s = 0, filled = 0;
    uint32_t ph = 1;
    for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
      const int m0 = (t / cols) * BM, ct = t % cols;
      const int w0 = (ct / tiles_n) * a.J + (ct % tiles_n) * GEMM_BN;   // first weight row of the tile
      for (int i = 0; i < nk; ++i) {
        ok = filled++ < PG_STAGES || mbar_wait_warp(&empty[s], ph);   // (a stage that has never been filled is free)
        if (!ok) break;
        mbar_expect_tx(on, &full[s], STAGE);
        tma_load_2d(on, smem + s * STAGE, &tma_a, i * BK, m0, &full[s]);
        tma_load_2d(on, smem + s * STAGE + A_BYTES, &tma_b, i * BK, w0, &full[s]);
        if (++s == PG_STAGES) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    pdl_trigger();
    if (!ok && lane == 0) flag_timeout(a.status);
  } else if (warp == 5) {
    // ---- MMA issuer: tile `it` of this CTA accumulates into buffer it & 1
    const uint32_t idesc = umma_idesc_i8(BM, GEMM_BN);
    const uint32_t on = elect_one();
    bool ok = true, ready = mbar_test(&full[0], 0);
    int s = 0, it = 0;
    uint32_t ph = 0;
    for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++it) {
      const int buf = it & 1, use = it >> 1;
      if (use >= 1) {   // the epilogue must have read the previous contents of this buffer
        ok = mbar_wait_warp(&acc_empty[buf], (use - 1) & 1);
        if (!ok) break;
        tc_fence_after();
      }
      const uint32_t d = tmem + (uint32_t)(buf * GEMM_BN);
      for (int i = 0; i < nk; ++i) {
        ok = mbar_wait_warp_tested(ready, &full[s], ph);
        if (!ok) break;
        tc_fence_after();
        const int st = s;
        if (++s == PG_STAGES) {
          s = 0;
          ph ^= 1;
        }
        ready = mbar_test(&full[s], ph);
        const uint64_t da = umma_desc_sw128(smem_u32(smem + st * STAGE));
        const uint64_t db = umma_desc_sw128(smem_u32(smem + st * STAGE + A_BYTES));
#pragma unroll
        for (int kk = 0; kk < BK / 32; ++kk) umma_i8(on, d, da + 2 * kk, db + 2 * kk, idesc, (i | kk) != 0);
        umma_commit(on, &empty[st]);
      }
      if (ok) umma_commit(on, &acc_full[buf]);
    }
    pdl_trigger();
    if (!ok && lane == 0) flag_timeout(a.status);
  } else if (warp < 4) {
    // ---- epilogue: warp w drains TMEM lanes [32 w, 32 w + 32) of the finished accumulator
    bool ok = true;
    int it = 0;
    const bool wide = ((reinterpret_cast<uintptr_t>(a.out) | (uintptr_t)(plane_out * 4) | (uintptr_t)(a.ldo * 4)) & 31) == 0;
    for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++it) {
      const int buf = it & 1, use = it >> 1;
      const int m0 = (t / cols) * BM, ct = t % cols, n0 = (ct % tiles_n) * GEMM_BN;
      int32_t* const plane = reinterpret_cast<int32_t*>(a.out) + (ct / tiles_n) * plane_out;
      ok = mbar_wait(&acc_full[buf], use & 1);
      if (!ok) break;
      tc_fence_after();
      const int m = m0 + warp * 32 + lane;
      const uint32_t taddr = tmem + (uint32_t)(buf * GEMM_BN) + ((uint32_t)(warp * 32) << 16);
      // two register sets: the TMEM load of the next 32 columns is in flight while these are stored
      auto store32 = [&](const int (&r)[32], int c0) {
        const int j0 = n0 + c0;
        if (m >= a.M || j0 >= a.J) return;
        int32_t* o = plane + (long long)m * a.ldo + j0;
        if (j0 + 32 <= a.J && wide) {
#pragma unroll
          for (int i = 0; i < 32; i += 8)
            st_global_v8_b32(o + i, r[i], r[i + 1], r[i + 2], r[i + 3], r[i + 4], r[i + 5], r[i + 6], r[i + 7]);
        } else if (j0 + 32 <= a.J) {
#pragma unroll
          for (int i = 0; i < 32; i += 4) *reinterpret_cast<int4*>(o + i) = make_int4(r[i], r[i + 1], r[i + 2], r[i + 3]);
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (j0 + i < a.J) o[i] = r[i];
        }
      };
      int r0[32], r1[32];
      tmem_ld32(taddr, r0);
#pragma unroll 1
      for (int c0 = 0; c0 < GEMM_BN; c0 += 64) {
        tmem_ld_wait();
        tmem_ld32(taddr + c0 + 32, r1);
        store32(r0, c0);
        tmem_ld_wait();
        if (c0 + 64 < GEMM_BN) {
          tmem_ld32(taddr + c0 + 64, r0);
        } else {
          // the accumulator has been read completely: hand it back before the last stores
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[buf]);
        }
        store32(r1, c0 + 32);
      }
    }
    pdl_trigger();
    if (!ok && lane == 0) flag_timeout(a.status);
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 5) tmem_dealloc(tmem, TCOLS);
}

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
      n = 148;
  }
  return n;
}

template <int BN>
static size_t gemm_smem() {
  return (size_t)GEMM_STAGES<BN> * (BM * BK + BN * BK) + 1024;
}
template <int BN>
static cudaError_t gemm_launch(const CUtensorMap& ta, const CUtensorMap& tb, const MmaGemmArgs& a, cudaStream_t s,
                               bool dependent) {
  static bool configured_on[MAX_DEVICES];
  bool& configured = configured_on[device_slot()];
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(k_mma_gemm<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem<BN>());
    if (e != cudaSuccess) return e;
    configured = true;
  }
  return launch_ex(k_mma_gemm<BN>, dim3((a.J + BN - 1) / BN, (a.M + BM - 1) / BM), dim3(192), gemm_smem<BN>(), s, dependent,
                   1, ta, tb, a);
}
template <int BN>
static cudaError_t gemm_persistent_launch(const CUtensorMap& ta, const CUtensorMap& tb, const MmaGemmArgs& a, int planes,
                                          long long plane_out, cudaStream_t s, bool dependent) {
  static bool configured_on[MAX_DEVICES];
  bool& configured = configured_on[device_slot()];
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(k_mma_gemm_persistent<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)gemm_smem<BN>());
    if (e != cudaSuccess) return e;
    configured = true;
  }
  const int tiles_m = (a.M + BM - 1) / BM, tiles_n = (a.J + BN - 1) / BN;
  const long long tiles = (long long)tiles_m * tiles_n * planes;
  const int ctas = tiles < sm_count() ? (int)tiles : sm_count();
  return launch_ex(k_mma_gemm_persistent<BN>, dim3(ctas), dim3(192), gemm_smem<BN>(), s, dependent, 1, ta, tb, a, tiles_m,
                   tiles_n, planes, plane_out);
}
// Weight rows per tile: the widest tile (fewest operand bytes per product) that still gives every SM
// one.  A tile that is alone on its SM is bound by the latency of its own chain (K chunks, then
// an epilogue proportional to its width), so narrower tiles on more SMs end sooner: the projection of 152
// rows of 1280 codes to 256 outputs takes 14.4 us as two 256-wide tiles and 8.4 us as 16 of width 32, the
// input projection of a bidirectional 640-cell layer over 152 rows 2 x 16.7 us as 20 tiles of width 256 per
// direction and 9.5 us as 160 of width 64 in one launch (1903 rows: 2 x 28.9 -> 20.6 us, width 256 in both).
static int gemm_tile_width(int M, int J, int planes, int narrowest) {
  for (int bn = 256; bn > narrowest; bn >>= 1)
    if ((long long)((M + BM - 1) / BM) * ((J + bn - 1) / bn) * planes >= sm_count()) return bn;
  return narrowest;
}

// x8: int8 activations [M, K] (pitch x_pitch), w8: int8 weights [J, K] (pitch w_pitch).
cudaError_t launch_mma_gemm(const int8_t* x8, long long x_pitch, int M, const int8_t* w8,
                            long long w_pitch, int J, int K, int epi, void* out, long long ldo,
                            const int32_t* out_idx, const float* w_scale, const float* bias,
                            float x_scale, const q4_act* out_act, int32_t* status,
                            const int32_t* n_active, cudaStream_t s, bool dependent, const float* mul_e,
                            const int32_t* mul_idx, const int32_t* n_idle, int all_idle) {
  if (M <= 0 || J <= 0) return cudaSuccess;
  if (epi == EPI_JOINTZ && (!mul_e || !mul_idx || J % 32 != 0)) return cudaErrorInvalidValue;
  const int bn = gemm_tile_width(M, J, 1, 32);
  CUtensorMap ta, tb;
  if (!make_tmap_i8(&ta, x8, K, M, x_pitch, BM) || !make_tmap_i8(&tb, w8, K, J, w_pitch, bn))
    return cudaErrorInvalidValue;
  MmaGemmArgs a;
  memset(&a, 0, sizeof(a));
  a.M = M;
  a.J = J;
  a.K = K;
  a.epi = epi;
  a.out = out;
  a.ldo = ldo;
  a.out_idx = out_idx;
  a.w_scale = w_scale;
  a.bias = bias;
  a.x_scale = x_scale;
  if (out_act) a.out_act = *out_act;
  a.status = status;
  a.n_active = n_active;
  a.mul_e = mul_e;
  a.mul_idx = mul_idx;
  a.n_idle = n_idle;
  a.all_idle = all_idle;
  a.wait_limit = g_wait_limit;
  a.skip_producer = g_skip_producer;
  timing_begin(s);
  const cudaError_t le = bn == 256   ? gemm_launch<256>(ta, tb, a, s, dependent)
                         : bn == 128 ? gemm_launch<128>(ta, tb, a, s, dependent)
                         : bn == 64  ? gemm_launch<64>(ta, tb, a, s, dependent)
                                     : gemm_launch<32>(ta, tb, a, s, dependent);
  timing_end(s);
  ++g_launches;
  return le != cudaSuccess ? le : cudaGetLastError();
}

// Input projections of all directions of a layer: x8 int8 [M, K], w8 int8 [planes J, K], out int32
// [planes][M, J]; persistent CTAs whose epilogue overlaps the next tile's MMAs.
cudaError_t launch_mma_gemm_i32(const int8_t* x8, int M, const int8_t* w8, int J, int K, int planes, int32_t* out,
                                int32_t* status, cudaStream_t s, bool dependent) {
  if (M <= 0 || J <= 0) return cudaSuccess;
  const int bn = gemm_tile_width(M, J, planes, 64);
  CUtensorMap ta, tb;
  if (!make_tmap_i8(&ta, x8, K, M, K, BM) || !make_tmap_i8(&tb, w8, K, (uint64_t)J * planes, K, bn))
    return cudaErrorInvalidValue;
  MmaGemmArgs a;
  memset(&a, 0, sizeof(a));
  a.M = M;
  a.J = J;
  a.K = K;
  a.epi = EPI_I32;
  a.out = out;
  a.ldo = J;
  a.status = status;
  const long long plane_out = (long long)M * J;
  timing_begin(s);
  const cudaError_t le = bn == 256   ? gemm_persistent_launch<256>(ta, tb, a, planes, plane_out, s, dependent)
                         : bn == 128 ? gemm_persistent_launch<128>(ta, tb, a, planes, plane_out, s, dependent)
                                     : gemm_persistent_launch<64>(ta, tb, a, planes, plane_out, s, dependent);
  timing_end(s);
  ++g_launches;
  return le != cudaSuccess ? le : cudaGetLastError();
}

// ------------------------------------------------------------------ fused LM head
// One launch per language model (and one for the joint network's output layer) and iteration.
// A cluster of 8 CTAs serves one tile of 128 rows.  Every CTA computes 32 of the 256 bottleneck columns
// (H -> 256, int32 in TMEM), de-quantizes, adds the bias, re-quantizes (asymmetric constants) and sends its
// codes, 32 bytes per row = the operand of one MMA, as one bulk copy to each of the 8 CTAs, counted on an
// mbarrier of the receiver.  Then every CTA multiplies the 256 codes of the rows with its own block of NB
// output-layer rows and keeps its NB logits per row in registers (NB / 4 per thread).  Row maxima and sums
// of the blocks are exchanged through distributed shared memory as well; one cluster barrier later every
// thread knows the row's log-sum-exp and stores log-probabilities: one global write, no separate log-softmax
// pass.  With H = 0 there is no bottleneck: the 256-wide operand rows are read from memory (joint network).
// Bound by the latency of this chain.  (All 256 bottleneck columns in every CTA take 5.0 us of bottleneck sums and 2.8 us
// of re-quantization before the second MMA; codes stored to the peers 8 bytes at a time 5 us with 128 rows.  Dealt out and
// copied as blocks: frame-by-frame search of 5 utterances, 40 rows, 15.95 -> 14.4 ms.)
constexpr int HEAD_D = 256;
constexpr int HEAD_CTAS = 8;                 // = the portable cluster size
constexpr int HEAD_BN1 = HEAD_D / HEAD_CTAS; // bottleneck columns per CTA
constexpr int HEAD_MAX_STAGES = 16;
constexpr int HEAD_RING = 80 * 1024;         // bytes of the operand ring; the output layer's weights, the outgoing codes, then
                                             // the log-probabilities on their way out use the same memory
constexpr int HEAD_EPI_WARPS = 16;           // four warps per TMEM lane quarter
constexpr int HEAD_THREADS = 32 * (HEAD_EPI_WARPS + 2);

__device__ __forceinline__ void cl_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cl_map(uint32_t addr, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
  return remote;
}
__device__ __forceinline__ void cl_store_f32(const float* local, uint32_t rank, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cl_map(smem_u32(local), rank)), "f"(v) : "memory");
}

template <int NB>
__global__ void __cluster_dims__(HEAD_CTAS, 1, 1) __launch_bounds__(HEAD_THREADS, 1)
k_mma_lmhead(const __grid_constant__ CUtensorMap tma_h, const __grid_constant__ CUtensorMap tma_wb,
             const __grid_constant__ CUtensorMap tma_wo, const LmHeadArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  constexpr int B1_BYTES = HEAD_BN1 * BK;
  constexpr int B2_BYTES = NB * BK;            // one K chunk of my block of output-layer rows
  constexpr int CPT = NB / 4;                  // logits per thread
  constexpr int TCOLS = 2 * NB;                // bottleneck sums in columns 0.., logits' sums in columns NB..
  // A stage holds the rows of this launch (a.tile_rows of the tile's 128) and the weight rows.  The MMA always
  // reads 128 operand rows: those beyond tile_rows are whatever follows in the ring, and their sums belong to
  // rows that are not stored.
  const int A_BYTES = a.tile_rows * BK, STAGE = A_BYTES + B1_BYTES, NS = a.n_stages;
  const uint32_t CODE_BYTES = (uint32_t)a.tile_rows * HEAD_BN1;   // a CTA's bottleneck codes
  uint8_t* const ops = smem;                   // bottleneck codes [source CTA][row][32], or two chunks of operand rows
  uint8_t* const ring = smem + 2 * BM * BK;
  __shared__ uint64_t full[HEAD_MAX_STAGES], empty[HEAD_MAX_STAGES], acc1_full, ops_ready, w_full, acc2_full;
  __shared__ uint32_t tmem_base_s;
  __shared__ __align__(16) float s_sc1[HEAD_BN1], s_b1[HEAD_BN1], s_sc2[NB], s_b2[NB];
  __shared__ float part_m[HEAD_CTAS][BM], part_s[HEAD_CTAS][BM];   // filled by every CTA of the cluster
  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const int m0 = blockIdx.y * BM;
  const int nb = blockIdx.x;                    // my blocks of columns = my cluster rank
  const int nk1 = (a.H + BK - 1) / BK;
  const int mm = umma_rows(a.tile_rows);
  if (tile_without_work(a.n_active, m0)) return;   // the whole cluster leaves

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&acc1_full, 1);
    mbar_init(&ops_ready, 1);
    mbar_init(&w_full, 1);
    mbar_init(&acc2_full, 1);
    fence_barrier_init();
    fence_proxy_async();
    if (nk1 > 0) mbar_expect_tx(&ops_ready, HEAD_CTAS * CODE_BYTES);
  }
  if (warp == HEAD_EPI_WARPS + 1) tmem_alloc(&tmem_base_s, TCOLS);
  if (warp == HEAD_EPI_WARPS && lane == 0) {
    prefetch_tmap(&tma_h);
    prefetch_tmap(&tma_wb);
    prefetch_tmap(&tma_wo);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  cl_barrier();   // every CTA of the cluster is running before anyone stores into a peer's shared memory
  pdl_wait();   // everything above (this barrier included) overlaps the tail of the previous kernel of the stream
  const bool idle = a.n_idle && ld_coherent(a.n_idle) >= a.all_idle;   // the same for every thread of the grid
  bool codes_due = false;   // a wait has run out: the peers' codes may still be on their way here

  if (idle) {
    pdl_trigger();
  } else if (warp == HEAD_EPI_WARPS) {
    // ---- TMA producer: bottleneck operands through the ring, then my block of output-layer weights into
    // the ring's memory, which the bottleneck's MMAs have finished reading by then
    const uint32_t on = elect_one();
    bool ok = true;
    int s = 0;
    uint32_t ph = 1;
    for (int i = 0; i < nk1 && ok; ++i) {
      ok = i < NS || mbar_wait_warp(&empty[s], ph);   // (a stage that has never been filled is free)
      if (!ok) break;
      mbar_expect_tx(on, &full[s], STAGE);
      tma_load_2d(on, ring + s * STAGE, &tma_h, i * BK, m0, &full[s]);
      tma_load_2d(on, ring + s * STAGE + A_BYTES, &tma_wb, i * BK, nb * HEAD_BN1, &full[s]);
      if (++s == NS) {
        s = 0;
        ph ^= 1;
      }
    }
    if (ok && nk1 > 0) ok = mbar_wait_warp(&acc1_full, 0);
    if (ok) {
      mbar_expect_tx(on, &w_full, nk1 > 0 ? 2 * B2_BYTES : 2 * (B2_BYTES + A_BYTES));
      for (int kc = 0; kc < 2; ++kc) {
        if (nk1 == 0) tma_load_2d(on, ops + kc * BM * BK, &tma_h, kc * BK, m0, &w_full);
        tma_load_2d(on, ring + kc * B2_BYTES, &tma_wo, kc * BK, nb * NB, &w_full);
      }
    }
    pdl_trigger();
    if (!ok && lane == 0) flag_timeout(a.status);
  } else if (warp == HEAD_EPI_WARPS + 1) {
    // ---- MMA issuer
    const uint32_t idesc1 = umma_idesc_i8(mm, HEAD_BN1), idesc2 = umma_idesc_i8(mm, NB);
    const uint32_t on = elect_one();
    bool ok = true, ready = mbar_test(&full[0], 0);
    int s = 0;
    uint32_t ph = 0;
    for (int i = 0; i < nk1 && ok; ++i) {
      ok = mbar_wait_warp_tested(ready, &full[s], ph);
      if (!ok) break;
      tc_fence_after();
      const int st = s;
      if (++s == NS) {
        s = 0;
        ph ^= 1;
      }
      ready = mbar_test(&full[s], ph);
      const uint64_t da = umma_desc_sw128(smem_u32(ring + st * STAGE));
      const uint64_t db = umma_desc_sw128(smem_u32(ring + st * STAGE + A_BYTES));
#pragma unroll
      for (int kk = 0; kk < BK / 32; ++kk) umma_i8(on, tmem, da + 2 * kk, db + 2 * kk, idesc1, (i | kk) != 0);
      umma_commit(on, &empty[st]);
    }
    umma_commit(on, &acc1_full);
    if (ok) ok = mbar_wait_warp(&w_full, 0);
    if (ok && nk1 > 0) ok = mbar_wait_warp(&ops_ready, 0);
    codes_due = !ok && nk1 > 0;
    tc_fence_after();
#pragma unroll
    for (int j = 0; j < HEAD_D / 32; ++j) {
      const uint64_t da = nk1 > 0 ? umma_desc_sw32(smem_u32(ops + j * BM * HEAD_BN1))
                                  : umma_desc_sw128(smem_u32(ops + (j >> 2) * BM * BK)) + 2 * (j & 3);
      const uint64_t db = umma_desc_sw128(smem_u32(ring + (j >> 2) * B2_BYTES)) + 2 * (j & 3);
      umma_i8(ok ? on : 0u, tmem + NB, da, db, idesc2, j != 0);
    }
    umma_commit(on, &acc2_full);
    pdl_trigger();
    if (!ok && lane == 0) flag_timeout(a.status);
  } else {
    // ---- epilogue: warp = (lane quarter q, column share cs)
    const int q = warp & 3, cs = warp >> 2;
    const int rt = umma_lane_row(mm, q, lane);
    const int n = m0 + rt;
    int dst = -1;
    if (n < a.N && !(a.n_active && n >= *a.n_active)) dst = a.dst_row ? a.dst_row[n] : n;
    const bool busy = __any_sync(0xffffffffu, dst >= 0);   // a warp without a row to store computes nothing
    bool ok = true;
    const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16);
    // de-quantization constants, in the shadow of the operands' way; like all else after the wait
    if (tid < HEAD_BN1 && nk1 > 0) {
      const int c = nb * HEAD_BN1 + tid;
      s_sc1[tid] = __fmul_rn(a.x_scale, __ldg(a.sc_bott + c));
      s_b1[tid] = a.b_bott ? __ldg(a.b_bott + c) : 0.0f;
    }
    for (int c = tid; c < NB; c += 32 * HEAD_EPI_WARPS) {
      const int j = min(nb * NB + c, a.V - 1);
      s_sc2[c] = __fmul_rn(a.q_scale, __ldg(a.sc_out + j));
      s_b2[c] = a.b_out ? __ldg(a.b_out + j) : 0.0f;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * HEAD_EPI_WARPS) : "memory");
    if (nk1 > 0) {
      const int lo = act_lo(a.bott_act), hi = act_hi(a.bott_act), zp = a.bott_act.zero_point;
      ok = mbar_wait(&acc1_full, 0);
      tc_fence_after();
      // codes of my row, columns 32 nb + [8 cs, 8 cs + 8): collected here, then sent as a whole
      uint8_t* const mine = ring + HEAD_RING - BM * HEAD_BN1;   // beyond the output layer's weights
      if (busy) {
        int r[8];
        tmem_ld(taddr + 8 * cs, r);
        tmem_ld_wait();
        uint32_t w[2] = {0, 0};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float x = __fmaf_rn((float)r[i], s_sc1[8 * cs + i], s_b1[8 * cs + i]);
          const int code = quantize1(x, a.bott_act.inv_scale, zp, lo, hi) - zp;
          w[i >> 2] |= (uint32_t)(code & 0xFF) << (8 * (i & 3));
        }
        *reinterpret_cast<uint2*>(mine + rt * HEAD_BN1 + (((cs >> 1) ^ (rt >> 2 & 1)) << 4) + 8 * (cs & 1)) = make_uint2(w[0], w[1]);
      }
      fence_proxy_async();   // read by the copy engine
      tc_fence_before();
      asm volatile("bar.sync 1, %0;" ::"n"(32 * HEAD_EPI_WARPS) : "memory");
      if (warp == 0 && lane < HEAD_CTAS)
        bulk_copy_to_cluster(cl_map(smem_u32(ops + nb * BM * HEAD_BN1), lane), smem_u32(mine), CODE_BYTES,
                             cl_map(smem_u32(&ops_ready), lane));
    }

    // my CPT logits of this block, kept in registers until the row's log-sum-exp is known
    if (ok) ok = mbar_wait(&acc2_full, 0);
    tc_fence_after();
    pdl_trigger();   // both GEMMs are over: the next kernel may set itself up
    float v[CPT];
    float my_m = -INFINITY, lse;
    const int col0 = nb * NB + CPT * cs;       // first vocabulary entry of my share
    if (busy) {
      constexpr int CH = CPT < 32 ? CPT : 32;
#pragma unroll
      for (int ch = 0; ch < CPT / CH; ++ch) {
        const int c0 = CPT * cs + CH * ch;
        int r[CH];
        tmem_ld(taddr + NB + c0, r);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < CH; i += 4) {
          const float4 sc = *reinterpret_cast<const float4*>(s_sc2 + c0 + i);
          const float4 bi = *reinterpret_cast<const float4*>(s_b2 + c0 + i);
          v[CH * ch + i + 0] = __fmaf_rn((float)r[i + 0], sc.x, bi.x);
          v[CH * ch + i + 1] = __fmaf_rn((float)r[i + 1], sc.y, bi.y);
          v[CH * ch + i + 2] = __fmaf_rn((float)r[i + 2], sc.z, bi.z);
          v[CH * ch + i + 3] = __fmaf_rn((float)r[i + 3], sc.w, bi.w);
        }
      }
    }
    // the block's maximum of every row, over the four column shares
    float (*red_m)[BM] = reinterpret_cast<float (*)[BM]>(ring), (*red_s)[BM] = red_m + 4;   // the weights have been read
    // (entries beyond the vocabulary count as -inf; selected, not branched over: a branch around each exponential exposes its
    // latency, 2950 clocks for 32 of them against 450)
    if (busy) {
      const int left = a.V - col0;
#pragma unroll
      for (int i = 0; i < CPT; ++i) {
        if (i >= left) v[i] = -INFINITY;
        my_m = fmaxf(my_m, v[i]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < CPT; ++i) v[i] = 0.0f;
    }
    if (NB == 32) {
      // Vocabularies of at most 256: the sums in the order of k_logsoftmax (one thread per entry, pairwise over
      // lanes, then over warps), so that the kernels for few rows and the tensor-core path give the same bits.
      float (*ex)[33] = reinterpret_cast<float (*)[33]>(ring + 8 * BM * sizeof(float));
      red_m[cs][rt] = my_m;
      asm volatile("bar.sync 1, %0;" ::"n"(32 * HEAD_EPI_WARPS) : "memory");
      if (cs == 0) {
        const float m = fmaxf(fmaxf(red_m[0][rt], red_m[1][rt]), fmaxf(red_m[2][rt], red_m[3][rt]));
#pragma unroll
        for (int r = 0; r < HEAD_CTAS; ++r) cl_store_f32(&part_m[nb][rt], (uint32_t)r, m);
      }
      cl_barrier();
      float m = -INFINITY;
#pragma unroll
      for (int r = 0; r < HEAD_CTAS; ++r) m = fmaxf(m, part_m[r][rt]);
#pragma unroll
      for (int i = 0; i < CPT; ++i) ex[rt][CPT * cs + i] = busy ? expf(v[i] - m) : 0.0f;   // 0 beyond the vocabulary
      asm volatile("bar.sync 1, %0;" ::"n"(32 * HEAD_EPI_WARPS) : "memory");
      if (cs == 0) {
        float t[16];
#pragma unroll
        for (int l = 0; l < 16; ++l) t[l] = ex[rt][l] + ex[rt][l + 16];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
#pragma unroll
          for (int l = 0; l < o; ++l) t[l] += t[l + o];
#pragma unroll
        for (int r = 0; r < HEAD_CTAS; ++r) cl_store_f32(&part_s[nb][rt], (uint32_t)r, t[0]);
      }
      cl_barrier();
      float t[HEAD_CTAS];
#pragma unroll
      for (int r = 0; r < HEAD_CTAS; ++r) t[r] = part_s[r][rt];
#pragma unroll
      for (int o = HEAD_CTAS / 2; o > 0; o >>= 1)
#pragma unroll
        for (int r = 0; r < o; ++r) t[r] += t[r + o];
      lse = m + logf(t[0]);
    } else {
      // exponentials by the hardware base-2 unit: relative error near 1e-6, far inside what the
      // log-sum-exp of a thousand terms needs
      const float my_s = busy ? exp_sum(v, my_m) : 0.0f;
      red_m[cs][rt] = my_m;
      red_s[cs][rt] = my_s;
      asm volatile("bar.sync 1, %0;" ::"n"(32 * HEAD_EPI_WARPS) : "memory");
      if (cs == 0) {   // this CTA's (max, sum) of the row goes to every CTA of the cluster
        const float ms[4] = {red_m[0][rt], red_m[1][rt], red_m[2][rt], red_m[3][rt]};
        const float ss[4] = {red_s[0][rt], red_s[1][rt], red_s[2][rt], red_s[3][rt]};
        const float m = fmaxf(fmaxf(ms[0], ms[1]), fmaxf(ms[2], ms[3]));
        const float ssum = exp_sum(ms, ss, m);
#pragma unroll
        for (int r = 0; r < HEAD_CTAS; ++r) {
          cl_store_f32(&part_m[nb][rt], (uint32_t)r, m);
          cl_store_f32(&part_s[nb][rt], (uint32_t)r, ssum);
        }
      }
      cl_barrier();
      // all partials are fetched at once, then combined in block order
      float pm[HEAD_CTAS], ps[HEAD_CTAS];
#pragma unroll
      for (int r = 0; r < HEAD_CTAS; ++r) {
        pm[r] = part_m[r][rt];
        ps[r] = part_s[r][rt];
      }
      float m = -INFINITY;
#pragma unroll
      for (int r = 0; r < HEAD_CTAS; ++r) m = fmaxf(m, pm[r]);
      lse = m + logf(exp_sum(pm, ps, m));
    }
    // A thread's log-probabilities belong to one row and the rows of a warp's lanes are V floats
    // apart, so storing them directly touches 32 lines per instruction.  A full 128-column block goes
    // through shared memory instead (the operand ring is free: both GEMMs and the copies of the codes are
    // complete) and leaves as whole rows, one 512-byte row per warp-wide store.
    const bool staged = NB == 128 && nb * NB + NB <= a.V && (a.V & 3) == 0 &&
                        (reinterpret_cast<uintptr_t>(a.lp) & 15) == 0;   // uniform per CTA
    if (staged) {
      constexpr int TP = NB + 4;   // row pitch in floats: rows 16-byte aligned, 32 rows spread over the banks
      static_assert(NB != 128 || (BM * TP + BM) * 4 <= HEAD_RING, "log-probabilities fit the ring");
      float* tile = reinterpret_cast<float*>(ring);
      int* tdst = reinterpret_cast<int*>(ring + (size_t)BM * TP * sizeof(float));
      float* trow = tile + rt * TP + CPT * cs;
      if (busy) {
#pragma unroll
        for (int i = 0; i < CPT; i += 4)
          *reinterpret_cast<float4*>(trow + i) = make_float4(v[i] - lse, v[i + 1] - lse, v[i + 2] - lse, v[i + 3] - lse);
      }
      if (cs == 0) tdst[rt] = ok ? dst : -1;
      asm volatile("bar.sync 1, %0;" ::"n"(32 * HEAD_EPI_WARPS) : "memory");
      int d[BM / HEAD_EPI_WARPS];
      float4 t4[BM / HEAD_EPI_WARPS];
#pragma unroll
      for (int j = 0; j < BM / HEAD_EPI_WARPS; ++j) {   // this warp's 8 rows: fetch first, then store
        const int r = warp + j * HEAD_EPI_WARPS;
        d[j] = tdst[r];
        t4[j] = *reinterpret_cast<const float4*>(tile + r * TP + 4 * lane);
      }
#pragma unroll
      for (int j = 0; j < BM / HEAD_EPI_WARPS; ++j)
        if (d[j] >= 0) *reinterpret_cast<float4*>(a.lp + (long long)d[j] * a.V + nb * NB + 4 * lane) = t4[j];
    } else if (dst >= 0 && ok) {
      float* out = a.lp + (long long)dst * a.V + col0;
      const int left = a.V - col0;
      if (left >= CPT && (reinterpret_cast<uintptr_t>(out) & 31) == 0) {
#pragma unroll
        for (int i = 0; i < CPT; i += 8)   // rows of a warp's lanes are V floats apart: few, wide stores
          st_global_v8(out + i, make_float4(v[i] - lse, v[i + 1] - lse, v[i + 2] - lse, v[i + 3] - lse),
                       make_float4(v[i + 4] - lse, v[i + 5] - lse, v[i + 6] - lse, v[i + 7] - lse));
      } else {
#pragma unroll
        for (int i = 0; i < CPT; ++i)
          if (i < left) out[i] = v[i] - lse;
      }
    }
    if (!ok && lane == 0) flag_timeout(a.status);
  }
  __syncwarp();
  if (!idle && warp >= HEAD_EPI_WARPS) {   // the producer and issuer warps join the cluster barrier too
    pdl_trigger();
    cl_barrier();
    if (NB == 32) cl_barrier();
    if (codes_due) mbar_wait_warp(&ops_ready, 0);   // all have been sent by now: nobody leaves while they arrive (bounded)
  }
  tc_fence_before();
  __syncthreads();
  if (warp == HEAD_EPI_WARPS + 1) tmem_dealloc(tmem, TCOLS);
  // no barrier at the exit: every store and copy into a peer's shared memory is issued before the exchange barrier
  // above; stores have arrived with it (release on arrival, acquire on the wait), copies once ops_ready has been waited for
}

template <int NB>
static cudaError_t lmhead_launch(const CUtensorMap& th, const CUtensorMap& tb, const CUtensorMap& to, const LmHeadArgs& a,
                                 cudaStream_t s, bool dependent) {
  static_assert(2 * NB * BK + BM * HEAD_BN1 <= HEAD_RING, "output-layer weights and outgoing codes share the ring's memory");
  const size_t smem = 2 * BM * BK + (size_t)HEAD_RING + 1024;
  static bool configured_on[MAX_DEVICES];
  bool& configured = configured_on[device_slot()];
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(k_mma_lmhead<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  return launch_ex(k_mma_lmhead<NB>, dim3(HEAD_CTAS, (a.N + BM - 1) / BM), dim3(HEAD_THREADS), smem, s, dependent, 1, th, tb,
                   to, a);
}

cudaError_t launch_mma_lmhead(const LmHeadArgs& args, const int8_t* h8, long long h_pitch, const int8_t* wb8,
                              const int8_t* wo8, cudaStream_t s, bool dependent) {
  if (args.N <= 0) return cudaSuccess;
  LmHeadArgs a = args;
  const int rows_pad = (a.N + BM - 1) / BM * BM;
  int nbw = 32;   // output-layer rows per CTA: the narrowest block that covers the vocabulary with 8 CTAs
  while (nbw < 256 && nbw * HEAD_CTAS < a.V) nbw *= 2;
  if (nbw * HEAD_CTAS < a.V) return cudaErrorInvalidValue;
  a.tile_rows = a.N < BM ? (a.N + 7) / 8 * 8 : BM;
  const int stage = (a.tile_rows + HEAD_BN1) * BK;
  a.n_stages = (HEAD_RING - BM * BK) / stage + 1;   // the MMA reads 128 rows from the last stage's start
  if (a.n_stages * stage > HEAD_RING) --a.n_stages;
  if (a.n_stages > HEAD_MAX_STAGES) a.n_stages = HEAD_MAX_STAGES;
  CUtensorMap th, tb, to;
  const int Ka = a.H > 0 ? a.H : HEAD_D;
  if (!make_tmap_i8(&th, h8, Ka, rows_pad, h_pitch, a.tile_rows) || !make_tmap_i8(&to, wo8, HEAD_D, a.V, HEAD_D, nbw))
    return cudaErrorInvalidValue;
  if (a.H > 0) {
    if (!make_tmap_i8(&tb, wb8, a.H, HEAD_D, a.H, HEAD_BN1)) return cudaErrorInvalidValue;
  } else {
    tb = to;   // unused without a bottleneck
  }
  timing_begin(s);
  const cudaError_t e = nbw == 32    ? lmhead_launch<32>(th, tb, to, a, s, dependent)
                        : nbw == 64  ? lmhead_launch<64>(th, tb, to, a, s, dependent)
                        : nbw == 128 ? lmhead_launch<128>(th, tb, to, a, s, dependent)
                                     : lmhead_launch<256>(th, tb, to, a, s, dependent);
  timing_end(s);
  ++g_launches;
  return e != cudaSuccess ? e : cudaGetLastError();
}

// ------------------------------------------------------------------ fused LSTM step
// EXTRAS = false drops the second code (yq_out), the fp32 copy (h_f32) and the accumulator dumps
// from the cell loop: the search needs none of them, and without their branches the four cells
// of a thread are scheduled as one block.
// PREMUL = true: sc_ih / sc_hh already hold (input scale * row scale) and (hidden scale * row
// scale), the products the de-quantization needs (same fp32 multiplication, done once).
// LSTM_BN = weight rows per tile (4 gates of LSTM_BN / 4 cells), see lstm_tile_width.
// HH_MEM = true: the sums of the recurrent half are read from memory (a.hh_pre), the main loop has the input half only.
template <bool EXTRAS, bool PREMUL, int LSTM_BN, bool HH_MEM>
__global__ void __launch_bounds__(32 * (LSTM_EPI_WARPS + 2), 2)
k_mma_lstm(const __grid_constant__ CUtensorMap tma_xa, const __grid_constant__ CUtensorMap tma_xw,
           const __grid_constant__ CUtensorMap tma_ha, const __grid_constant__ CUtensorMap tma_hw,
           const MmaLstmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  // a stage holds the launch's rows of the tile only; the MMA reads 128 (see k_mma_lmhead)
  constexpr int B_BYTES = LSTM_BN * BK;
  const int A_BYTES = a.tile_rows * BK, STAGE = A_BYTES + B_BYTES, NS = a.n_stages;
  constexpr int TCOLS = 2 * LSTM_BN;
  __shared__ uint64_t full[LSTM_MAX_STAGES], empty[LSTM_MAX_STAGES], acc_full;
  __shared__ uint32_t tmem_base_s;
  __shared__ float4 s_cst[3][LSTM_BN / 4];   // input scales, recurrent scales, bias of this tile's cells (4 gates each)
  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * LSTM_BN;   // row tiles slowest: tiles with work are dispatched first
  const int nkx = a.acc_pre ? 0 : (a.Kx_pad + BK - 1) / BK;
  const int nkh = HH_MEM ? 0 : (a.H + BK - 1) / BK;
  const int nk = nkx + nkh;
  const int mm = umma_rows(a.tile_rows);
  if (tile_without_work(a.n_active, m0)) return;

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&acc_full, 1);
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == LSTM_EPI_WARPS + 1) tmem_alloc(&tmem_base_s, TCOLS);
  if (warp == LSTM_EPI_WARPS && lane == 0) {
    prefetch_tmap(&tma_xa);
    prefetch_tmap(&tma_xw);
    if (!HH_MEM) {
      prefetch_tmap(&tma_ha);
      prefetch_tmap(&tma_hw);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  // Everything above overlaps the tail of the previous kernel of the stream.  With h_first only
  // the input operand is that kernel's output: the recurrent half of the K loop runs before the wait, the input half
  // after it.  Its operands are weights and rows that the gather wrote; the kernel between waited for the gather
  // before it triggered, and the tile copies read them from the L2.
  const bool h_first = a.h_first != 0 && nkx > 0;
  if (!h_first) pdl_wait();
  if (a.trigger_early) pdl_trigger();   // the successor has a half it can run beside this kernel
  const int x_first = h_first ? nkh : 0, hh_first = h_first ? 0 : nkx;   // first chunk of each part

  if (warp == LSTM_EPI_WARPS) {
    const uint32_t on = elect_one();
    bool ok = true;
    int s = 0;
    uint32_t ph = 1;
    for (int i = 0; i < nk && ok; ++i) {
      ok = i < NS || mbar_wait_warp(&empty[s], ph);   // (a stage that has never been filled is free)
      if (!ok) break;
      const bool xpart = h_first ? i >= nkh : i < nkx;
      if (h_first && i == x_first) pdl_wait();
      mbar_expect_tx(on, &full[s], STAGE);
      if (xpart) {
        tma_load_2d(on, smem + s * STAGE, &tma_xa, (i - x_first) * BK, m0, &full[s]);
        tma_load_2d(on, smem + s * STAGE + A_BYTES, &tma_xw, (i - x_first) * BK, n0, &full[s]);
      } else {
        tma_load_2d(on, smem + s * STAGE, &tma_ha, (i - hh_first) * BK, m0, &full[s]);
        tma_load_2d(on, smem + s * STAGE + A_BYTES, &tma_hw, (i - hh_first) * BK, n0, &full[s]);
      }
      if (++s == NS) {
        s = 0;
        ph ^= 1;
      }
    }
    pdl_trigger();
    if (!ok && lane == 0) flag_timeout(a.status);
  } else if (warp == LSTM_EPI_WARPS + 1) {
    const uint32_t idesc = umma_idesc_i8(mm, LSTM_BN);
    const uint32_t on = elect_one();
    bool ok = true, ready = mbar_test(&full[0], 0);
    int s = 0;
    uint32_t ph = 0;
    for (int i = 0; i < nk && ok; ++i) {
      ok = mbar_wait_warp_tested(ready, &full[s], ph);
      if (!ok) break;
      tc_fence_after();
      const int st = s;
      if (++s == NS) {
        s = 0;
        ph ^= 1;
      }
      ready = mbar_test(&full[s], ph);
      const uint64_t da = umma_desc_sw128(smem_u32(smem + st * STAGE));
      const uint64_t db = umma_desc_sw128(smem_u32(smem + st * STAGE + A_BYTES));
      const bool xpart = h_first ? i >= nkh : i < nkx;
      const uint32_t d = tmem + (xpart ? 0 : LSTM_BN);
      const int first = xpart ? x_first : hh_first;
#pragma unroll
      for (int kk = 0; kk < BK / 32; ++kk) umma_i8(on, d, da + 2 * kk, db + 2 * kk, idesc, (i != first) || kk != 0);
      umma_commit(on, &empty[st]);
    }
    umma_commit(on, &acc_full);
    pdl_trigger();
    if (!ok && lane == 0) flag_timeout(a.status);
  } else if (warp < LSTM_EPI_WARPS) {
    if (h_first) pdl_wait();   // the row lists and cell states below are read after it, beside the input half
    const int q = warp & 3, hf = warp >> 2;
    const int rt = umma_lane_row(mm, q, lane);   // row within the tile
    const int n = m0 + rt;                   // row of this launch
    int src = -1, dst = -1;
    if (n < a.N && !(a.n_active && n >= *a.n_active)) {
      dst = a.dst_row ? a.dst_row[n] : n;
      src = a.src_row ? a.src_row[n] : n;
    }
    // previous cell states of all my cells: requested before the main loop ends (they belong to
    // rows no kernel of this iteration writes), so that their trip to memory costs the epilogue nothing
    float4 cprev_all[LSTM_BN / 32];
    // 8 or 16 contiguous cells per row: 256-bit accesses when the layout allows it
    const bool wide = (n0 >> 2) + hf * (LSTM_BN / 8) + LSTM_BN / 8 <= a.H && (a.H & 7) == 0 &&
                      ((reinterpret_cast<uintptr_t>(a.c_in) | reinterpret_cast<uintptr_t>(a.c_out)) & 31) == 0;
#pragma unroll
    for (int ch = 0; ch < LSTM_BN / 32; ++ch) cprev_all[ch] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (wide) {
      if (dst >= 0 && src >= 0) {
        const float* cp0 = a.c_in + (long long)src * a.H + (n0 >> 2) + hf * (LSTM_BN / 8);
#pragma unroll
        for (int ch = 0; ch < LSTM_BN / 32; ch += 2) ld_global_v8(cp0 + 4 * ch, cprev_all[ch], cprev_all[ch + 1]);
      }
    } else {
#pragma unroll
      for (int ch = 0; ch < LSTM_BN / 32; ++ch) {
        const int cell0 = (n0 >> 2) + hf * (LSTM_BN / 8) + ch * 4;
        if (dst >= 0 && src >= 0 && cell0 < a.H)
          cprev_all[ch] = *reinterpret_cast<const float4*>(a.c_in + (long long)src * a.H + cell0);
      }
    }
    // de-quantization constants of the tile's 32 cells: weights only (nothing of an earlier kernel),
    // fetched while the main loop runs so that the cell loop reads them from shared memory
    if (tid < 3 * (LSTM_BN / 4)) {
      const int which = tid / (LSTM_BN / 4), cell = (n0 >> 2) + tid % (LSTM_BN / 4);
      const float* src = which == 0 ? a.sc_ih : which == 1 ? a.sc_hh : a.bias;
      s_cst[which][tid % (LSTM_BN / 4)] =
          cell < a.H ? __ldg(reinterpret_cast<const float4*>(src) + cell) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * LSTM_EPI_WARPS) : "memory");
    // Sums of the recurrent half from memory: fetched beside the main loop into the accumulator that its products would fill
    // (a thread reads back what it wrote).  Fetched in the cell loop, one chunk ahead: 9300 clocks instead of 5000 for 256 rows.
    if (HH_MEM) {
      const float* p = a.hh_pre + (long long)max(src, 0) * 4 * a.H + n0 + hf * (LSTM_BN / 2);
      const bool have = dst >= 0 && src >= 0;
#pragma unroll
      for (int ch = 0; ch < LSTM_BN / 32; ++ch) {
        float4 h[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) h[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (have && (n0 >> 2) + hf * (LSTM_BN / 8) + 4 * ch < a.H) {
          ld_global_v8(p + 16 * ch, h[0], h[1]);
          ld_global_v8(p + 16 * ch + 8, h[2], h[3]);
        }
        tmem_st16(tmem + ((uint32_t)(q * 32) << 16) + LSTM_BN + hf * (LSTM_BN / 2) + 16 * ch, h[0], h[1], h[2], h[3]);
      }
      tmem_st_wait();
    }
    const bool ok = mbar_wait(&acc_full, 0);
    tc_fence_after();
    pdl_trigger();   // the main loop is over: the next kernel may set itself up
    if (!ok && lane == 0) flag_timeout(a.status);
    const bool live = ok && dst >= 0;
    const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16);
    const int H = a.H;
    const float sx = (live && a.x_scale_vec) ? a.x_scale_vec[n % a.x_scale_mod] : a.x_scale;
    const float sh = a.hid_act.scale;
    const int hlo = act_lo(a.hid_act), hhi = act_hi(a.hid_act);
    const int ylo = act_lo(a.out_act), yhi = act_hi(a.out_act);
    constexpr int CELLS_PER_HALF = LSTM_BN / 4 / 2;   // 16 or 8
    // Without the extras the codes of all 16 cells of a thread are kept and stored once: the rows
    // of a warp's lanes lie far apart, so every store instruction touches 32 lines, and four small
    // stores per output cost the load/store unit four times as much as one wide one.
    const int cell_first = (n0 >> 2) + hf * CELLS_PER_HALF;
    const bool combine = !EXTRAS && cell_first + CELLS_PER_HALF <= H;
    uint32_t w8[CELLS_PER_HALF / 4];
#pragma unroll
    for (int ch = 0; ch < CELLS_PER_HALF / 4; ++ch) w8[ch] = 0;
    float4 c_even = make_float4(0.f, 0.f, 0.f, 0.f);   // new cell states of the even chunk, stored with the odd one
#pragma unroll
    for (int ch = 0; ch < CELLS_PER_HALF / 4; ++ch) {
      const int ct = hf * CELLS_PER_HALF + ch * 4;     // first cell of the chunk within the tile
      const int cell0 = (n0 >> 2) + ct;
      int ih[16], hh[16];
      if (HH_MEM || nkx > 0) {
        tmem_ld16(taddr + 4 * ct, ih);
      }
      tmem_ld16(taddr + LSTM_BN + 4 * ct, hh);
      tmem_ld_wait();
      float hv[16];   // sums of the recurrent half
#pragma unroll
      for (int c = 0; c < 16; ++c) hv[c] = HH_MEM ? __int_as_float(hh[c]) : (float)hh[c];
      if (!live || cell0 >= H) continue;
      if (!HH_MEM && nkx == 0) {
        const int4* p = reinterpret_cast<const int4*>(a.acc_pre + (long long)n * a.acc_pre_ld + 4 * cell0);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int4 v = p[c];
          ih[4 * c] = v.x;
          ih[4 * c + 1] = v.y;
          ih[4 * c + 2] = v.z;
          ih[4 * c + 3] = v.w;
        }
      }
      const float4 cprev = cprev_all[ch];
      const float cp[4] = {cprev.x, cprev.y, cprev.z, cprev.w};
      float cn[4], hn[4];
      int qh[4], qy[4];
      // pre-activations of the four cells: acc_hh * s_hh + (acc_ih * s_ih + bias), gates (i, f) and (g, o)
      // as pairs on the paired fp32 instructions (the same two roundings per value as the scalar form)
      float pre[4][4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float4 s_ih = s_cst[0][ct + c], s_hh = s_cst[1][ct + c], bb = s_cst[2][ct + c];
        const uint64_t sih0 = PREMUL ? pk2(s_ih.x, s_ih.y) : pk2(__fmul_rn(sx, s_ih.x), __fmul_rn(sx, s_ih.y));
        const uint64_t sih1 = PREMUL ? pk2(s_ih.z, s_ih.w) : pk2(__fmul_rn(sx, s_ih.z), __fmul_rn(sx, s_ih.w));
        const uint64_t shh0 = PREMUL ? pk2(s_hh.x, s_hh.y) : pk2(__fmul_rn(sh, s_hh.x), __fmul_rn(sh, s_hh.y));
        const uint64_t shh1 = PREMUL ? pk2(s_hh.z, s_hh.w) : pk2(__fmul_rn(sh, s_hh.z), __fmul_rn(sh, s_hh.w));
        const uint64_t v0 = fma2(pk2(hv[4 * c + 0], hv[4 * c + 1]), shh0,
                                 fma2(pk2((float)ih[4 * c + 0], (float)ih[4 * c + 1]), sih0, pk2(bb.x, bb.y)));
        const uint64_t v1 = fma2(pk2(hv[4 * c + 2], hv[4 * c + 3]), shh1,
                                 fma2(pk2((float)ih[4 * c + 2], (float)ih[4 * c + 3]), sih1, pk2(bb.z, bb.w)));
        upk2(v0, pre[c][0], pre[c][1]);
        upk2(v1, pre[c][2], pre[c][3]);
      }
#pragma unroll
      for (int c = 0; c < 4; c += 2)   // two cells per call
        cell_fixed2(pre[c][0], pre[c][1], pre[c][2], pre[c][3], cp[c], pre[c + 1][0], pre[c + 1][1], pre[c + 1][2],
                    pre[c + 1][3], cp[c + 1], cn[c], hn[c], cn[c + 1], hn[c + 1]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int cell = cell0 + c;
        qh[c] = quantize1(hn[c], a.hid_act.inv_scale, a.hid_act.zero_point, hlo, hhi);
        qy[c] = EXTRAS ? quantize1(hn[c], a.out_act.inv_scale, a.out_act.zero_point, ylo, yhi) : 0;
        if constexpr (EXTRAS) {
          if (a.dbg_ih) {
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              a.dbg_ih[(long long)n * a.dbg_ld + g * H + cell] = ih[4 * c + g];
              a.dbg_hh[(long long)n * a.dbg_ld + g * H + cell] = hh[4 * c + g];
            }
          }
        }
      }
      if (wide) {
        if (ch & 1)
          st_global_v8(a.c_out + (long long)dst * H + cell0 - 4, c_even, make_float4(cn[0], cn[1], cn[2], cn[3]));
        else
          c_even = make_float4(cn[0], cn[1], cn[2], cn[3]);
      } else {
        *reinterpret_cast<float4*>(a.c_out + (long long)dst * H + cell0) = make_float4(cn[0], cn[1], cn[2], cn[3]);
      }
      if (EXTRAS && a.h_f32) *reinterpret_cast<float4*>(a.h_f32 + (long long)n * H + cell0) = make_float4(hn[0], hn[1], hn[2], hn[3]);
      w8[ch] = (uint32_t)(qh[0] & 0xFF) | ((uint32_t)(qh[1] & 0xFF) << 8) | ((uint32_t)(qh[2] & 0xFF) << 16) |
               ((uint32_t)(qh[3] & 0xFF) << 24);
      if (combine) continue;
      if (a.hq_out) {
        if (a.hid_act.bits == 4)
          *reinterpret_cast<uint16_t*>(a.hq_out + (long long)dst * a.hq_ld + (cell0 >> 1)) =
              (uint16_t)((qh[0] & 0xF) | ((qh[1] & 0xF) << 4) | ((qh[2] & 0xF) << 8) | ((qh[3] & 0xF) << 12));
        else
          *reinterpret_cast<uint32_t*>(a.hq_out + (long long)dst * a.hq_ld + cell0) =
              (uint32_t)(qh[0] & 0xFF) | ((uint32_t)(qh[1] & 0xFF) << 8) | ((uint32_t)(qh[2] & 0xFF) << 16) | ((uint32_t)(qh[3] & 0xFF) << 24);
      }
      if (a.h8_out)
        *reinterpret_cast<uint32_t*>(a.h8_out + (long long)n * a.h8_ld + cell0) =
            (uint32_t)(qh[0] & 0xFF) | ((uint32_t)(qh[1] & 0xFF) << 8) | ((uint32_t)(qh[2] & 0xFF) << 16) | ((uint32_t)(qh[3] & 0xFF) << 24);
      if (EXTRAS && a.yq_out) {
        if (a.out_act.bits == 4)
          *reinterpret_cast<uint16_t*>(a.yq_out + (long long)n * a.yq_ld + (cell0 >> 1)) =
              (uint16_t)((qy[0] & 0xF) | ((qy[1] & 0xF) << 4) | ((qy[2] & 0xF) << 8) | ((qy[3] & 0xF) << 12));
        else
          *reinterpret_cast<uint32_t*>(a.yq_out + (long long)n * a.yq_ld + cell0) =
              (uint32_t)(qy[0] & 0xFF) | ((uint32_t)(qy[1] & 0xFF) << 8) | ((uint32_t)(qy[2] & 0xFF) << 16) | ((uint32_t)(qy[3] & 0xFF) << 24);
      }
    }
    if (combine && live) {
      constexpr int NW = CELLS_PER_HALF / 4;   // words of int8 codes per thread
      static_assert(NW == 4 || NW == 2, "16 or 8 cells");
      auto put8 = [&](uint8_t* o) {
        if (NW == 4)
          *reinterpret_cast<uint4*>(o) = make_uint4(w8[0], w8[1], w8[NW - 2], w8[NW - 1]);
        else
          *reinterpret_cast<uint2*>(o) = make_uint2(w8[0], w8[1]);
      };
      if (a.h8_out) put8(reinterpret_cast<uint8_t*>(a.h8_out) + (long long)n * a.h8_ld + cell_first);
      if (a.hq_out) {
        if (a.hid_act.bits == 4) {
          uint32_t q[NW / 2];   // nibbles, cell order
#pragma unroll
          for (int j = 0; j < NW / 2; ++j) {
            q[j] = 0;
#pragma unroll
            for (int c = 0; c < 4; ++c)
              q[j] |= ((w8[2 * j] >> (8 * c)) & 0xFu) << (4 * c) | ((w8[2 * j + 1] >> (8 * c)) & 0xFu) << (16 + 4 * c);
          }
          uint8_t* o = a.hq_out + (long long)dst * a.hq_ld + (cell_first >> 1);
          if (NW == 4)
            *reinterpret_cast<uint2*>(o) = make_uint2(q[0], q[NW / 2 - 1]);
          else
            *reinterpret_cast<uint32_t*>(o) = q[0];
        } else {
          put8(a.hq_out + (long long)dst * a.hq_ld + cell_first);
        }
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == LSTM_EPI_WARPS + 1) tmem_dealloc(tmem, TCOLS);
}

template <int BN>
static cudaError_t lstm_launch(const MmaLstmArgs& a, const CUtensorMap& txa, const CUtensorMap& txw, const CUtensorMap& tha,
                               const CUtensorMap& thw, size_t smem, cudaStream_t s, bool dependent) {
  static bool configured_on[MAX_DEVICES];
  bool& configured = configured_on[device_slot()];
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(k_mma_lstm<true, false, BN, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, LSTM_SMEM_MAX);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_mma_lstm<false, false, BN, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, LSTM_SMEM_MAX);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_mma_lstm<false, true, BN, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, LSTM_SMEM_MAX);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_mma_lstm<false, true, BN, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, LSTM_SMEM_MAX);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  const dim3 grid((4 * a.H + BN - 1) / BN, (a.N + BM - 1) / BM), block(32 * (LSTM_EPI_WARPS + 2));
  if (a.yq_out || a.h_f32 || a.dbg_ih)
    return launch_ex(k_mma_lstm<true, false, BN, false>, grid, block, smem, s, dependent, 1, txa, txw, tha, thw, a);
  if (a.hh_pre)
    return launch_ex(k_mma_lstm<false, true, BN, true>, grid, block, smem, s, dependent, 1, txa, txw, tha, thw, a);
  if (a.premultiplied)
    return launch_ex(k_mma_lstm<false, true, BN, false>, grid, block, smem, s, dependent, 1, txa, txw, tha, thw, a);
  return launch_ex(k_mma_lstm<false, false, BN, false>, grid, block, smem, s, dependent, 1, txa, txw, tha, thw, a);
}
// Weight rows per tile.  An int8 MMA of 128 operand rows takes 77 clocks with 128 weight rows and 73 with 64
// (the operand rows' way into the tensor core bounds it), so narrower tiles cost nearly twice the tensor time
// in all; they pay only where every tile has an SM of its own, by a deeper ring and half the cell updates
// per CTA: frame-by-frame search of 5 utterances (40 rows) 13.7 -> 12.9 ms, forced scoring of 256 rows 2.36 ->
// 2.25 ms; with 32-wide tiles, and with 64 at two tiles per SM, the target LM's layers waited for the tiles of the
// other networks instead (search of 16 utterances, label iteration 65 -> 70 us).
static int lstm_tile_width(int row_tiles, int H) {
  return row_tiles * ((4 * H + 63) / 64) <= sm_count() ? 64 : 128;
}

// Operands: xa int8 [rows_pad, Kx_pad] (ignored with acc_pre), xw int8 [4H, Kx_pad] interleaved,
// ha int8 [rows_pad, H], hw int8 [4H, H] interleaved.  rows_pad = N rounded up to 128.
cudaError_t launch_mma_lstm(const MmaLstmArgs& a, const int8_t* xa, long long xa_pitch,
                            const int8_t* xw, long long xw_pitch, const int8_t* ha, long long ha_pitch,
                            const int8_t* hw, long long hw_pitch, cudaStream_t s, bool dependent) {
  if (a.N <= 0) return cudaSuccess;
  const int rows_pad = (a.N + BM - 1) / BM * BM;
  const int bn = lstm_tile_width(rows_pad / BM, a.H);
  MmaLstmArgs b = a;
  b.tile_rows = a.N < BM ? (a.N + 7) / 8 * 8 : BM;   // a single row tile fetches no rows beyond the launch's
  const int stage = (b.tile_rows + bn) * BK;
  b.n_stages = LSTM_RING / stage < LSTM_MAX_STAGES ? LSTM_RING / stage : LSTM_MAX_STAGES;
  CUtensorMap txa, txw, tha, thw;
  if (a.hh_pre && (!a.premultiplied || a.acc_pre)) return cudaErrorInvalidValue;
  if (!a.hh_pre &&
      (!make_tmap_i8(&tha, ha, a.H, rows_pad, ha_pitch, b.tile_rows) || !make_tmap_i8(&thw, hw, a.H, 4 * a.H, hw_pitch, bn)))
    return cudaErrorInvalidValue;
  if (a.acc_pre) {
    txa = tha;
    txw = thw;
  } else if (!make_tmap_i8(&txa, xa, a.Kx_pad, rows_pad, xa_pitch, b.tile_rows) ||
             !make_tmap_i8(&txw, xw, a.Kx_pad, 4 * a.H, xw_pitch, bn)) {
    return cudaErrorInvalidValue;
  }
  if (a.hh_pre) {   // not read
    tha = txa;
    thw = txw;
  }
  if (a.premultiplied && (a.yq_out || a.h_f32 || a.dbg_ih || a.x_scale_vec)) return cudaErrorInvalidValue;
  // the MMA reads 128 operand rows from the start of every stage, of the last one too
  const int ring = b.n_stages * stage, last = (b.n_stages - 1) * stage + BM * BK;
  const size_t smem = (size_t)(ring > last ? ring : last) + 1024;
  if (smem > (size_t)LSTM_SMEM_MAX) return cudaErrorInvalidValue;
  timing_begin(s);
  const cudaError_t le = bn == 128 ? lstm_launch<128>(b, txa, txw, tha, thw, smem, s, dependent)
                                   : lstm_launch<64>(b, txa, txw, tha, thw, smem, s, dependent);
  timing_end(s);
  ++g_launches;
  return le != cudaSuccess ? le : cudaGetLastError();
}

}  // namespace q4
