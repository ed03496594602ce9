// Network advances of a whole search without a matrix product in front of the first layers.  Inside one search
//   the input half of a first LSTM layer depends on the label only: its de-quantized sums plus bias are a table, one row
//   per label, made with the prepared weights;
//   the recurrent half depends on the hypothesis that is extended only: its int32 sums are formed right after the
//   hypothesis's state, beside the output heads and the selection, and kept per state row until a label extends it.
// So a step starts with k_search_cells, element-wise over the pending rows, instead of a gather and LSTM products, and the
// second layer multiplies its input half only (k_mma_lstm with sums of the recurrent half in memory).  k_state_products
// forms the sums.  Same integers and the same two roundings per pre-activation as in the step kernels: the same bits.
#include <string.h>

#include "q4_internal.h"
#include "q4_mma.cuh"

namespace q4 {

// One launch for the first layers of all networks (blockIdx.y): a thread owns 4 cells of a pending row, lanes own
// consecutive cells.  Bound by the latency of three dependent reads (row count, row lists, operands) for few rows, by
// 32 bytes of sums per cell for many.
constexpr int CELL_THREADS = 128;
__global__ void __launch_bounds__(CELL_THREADS) k_search_cells(const __grid_constant__ CellJobs a) {
  pdl_wait();
  pdl_trigger();   // after the wait: the kernels behind it read the row count first (see tile_without_work)
  if ((blockIdx.x | blockIdx.y | threadIdx.x) == 0) *a.n_work = min(a.N, *a.n_active);
  const CellJob& j = a.job[blockIdx.y];
  const uint32_t per_row = (uint32_t)j.H >> 2;
  const uint32_t i = blockIdx.x * CELL_THREADS + threadIdx.x;
  const uint32_t n = i / per_row;
  if (n >= (uint32_t)a.N) return;
  const int cell = (int)(i - n * per_row) * 4;
  const int src = a.src_row[n], dst = a.dst_row[n], tok = a.tok[n], n_work = *a.n_active;
  if ((int)n >= n_work || dst < 0) return;
  const int H = j.H;
  float4 x[4], hh[4], cp = make_float4(0.f, 0.f, 0.f, 0.f);
  const float* xp = j.table + (long long)tok * 4 * H + 4 * cell;
  ld_global_v8(xp, x[0], x[1]);
  ld_global_v8(xp + 8, x[2], x[3]);
#pragma unroll
  for (int c = 0; c < 4; ++c) hh[c] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (src >= 0) {
    const float* hp = j.sums + (long long)src * 4 * H + 4 * cell;
    ld_global_v8(hp, hh[0], hh[1]);
    ld_global_v8(hp + 8, hh[2], hh[3]);
    cp = *reinterpret_cast<const float4*>(j.c + (long long)src * H + cell);
  }
  const float cpv[4] = {cp.x, cp.y, cp.z, cp.w};
  float pre[4][4], cn[4], hn[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float4 s = *reinterpret_cast<const float4*>(j.sc_hh + 4 * (cell + c));
    pre[c][0] = __fmaf_rn(hh[c].x, s.x, x[c].x);
    pre[c][1] = __fmaf_rn(hh[c].y, s.y, x[c].y);
    pre[c][2] = __fmaf_rn(hh[c].z, s.z, x[c].z);
    pre[c][3] = __fmaf_rn(hh[c].w, s.w, x[c].w);
  }
#pragma unroll
  for (int c = 0; c < 4; c += 2)
    cell_fixed2(pre[c][0], pre[c][1], pre[c][2], pre[c][3], cpv[c], pre[c + 1][0], pre[c + 1][1], pre[c + 1][2],
                pre[c + 1][3], cpv[c + 1], cn[c], hn[c], cn[c + 1], hn[c + 1]);
  const int lo = act_lo(j.hid_act), hi = act_hi(j.hid_act);
  uint32_t w = 0;
#pragma unroll
  for (int c = 0; c < 4; ++c)
    w |= (uint32_t)(quantize1(hn[c], j.hid_act.inv_scale, j.hid_act.zero_point, lo, hi) & 0xFF) << (8 * c);
  *reinterpret_cast<float4*>(j.c + (long long)dst * H + cell) = make_float4(cn[0], cn[1], cn[2], cn[3]);
  *reinterpret_cast<uint32_t*>(j.h8 + (long long)n * H + cell) = w;
  if (j.hid_act.bits == 4)
    *reinterpret_cast<uint16_t*>(j.hq + (long long)dst * (H >> 1) + (cell >> 1)) =
        (uint16_t)((w & 0xF) | (w >> 8 & 0xF) << 4 | (w >> 16 & 0xF) << 8 | (w >> 24 & 0xF) << 12);
  else
    *reinterpret_cast<uint32_t*>(j.hq + (long long)dst * H + cell) = w;
}
cudaError_t launch_search_cells(const CellJobs& jobs, cudaStream_t s, bool dependent) {
  uint32_t most = 0;
  for (int i = 0; i < jobs.n_jobs; ++i) {
    const uint32_t items = (uint32_t)jobs.N * (uint32_t)(jobs.job[i].H >> 2);
    most = items > most ? items : most;
  }
  timing_begin(s);
  const cudaError_t e = launch_ex(k_search_cells, dim3((most + CELL_THREADS - 1) / CELL_THREADS, jobs.n_jobs), dim3(CELL_THREADS),
                                  0, s, dependent, 1, jobs);
  timing_end(s);
  ++g_launches;
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Recurrent sums of the pending rows' new states: D[128 x 128] tiles of up to three networks in one launch (blockIdx.x
// walks their weight tiles one after the other), int8 operands by TMA, sums converted to float and stored at the rows' state
// rows, columns in 4*cell+gate order.  Nothing waits for it before the next step's cells.  The ring leaves room on the SM for
// the kernels of the longest chain beside it.
constexpr int SP_BM = 128, SP_BN = 128, SP_BK = 128;
constexpr int SP_STAGE_MAX = (SP_BM + SP_BN) * SP_BK, SP_STAGES = 3;
constexpr size_t SP_SMEM = (size_t)SP_STAGES * SP_STAGE_MAX + 1024;
struct StateMaps {
  CUtensorMap a[3], b[3];
};
__global__ void __launch_bounds__(192, 2) k_state_products(const __grid_constant__ StateMaps maps,
                                                           const __grid_constant__ StateProductJobs jobs) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t full[SP_STAGES], empty[SP_STAGES], acc_full;
  __shared__ uint32_t tmem_base_s;
  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const int m0 = blockIdx.y * SP_BM;
  int tile = blockIdx.x, p = 0;
  while (p + 1 < jobs.n_jobs && tile >= jobs.job[p].H / (SP_BN / 4)) tile -= jobs.job[p++].H / (SP_BN / 4);
  const int K = jobs.job[p].H, n0 = tile * SP_BN, nk = K / SP_BK;
  const int A_BYTES = jobs.tile_rows * SP_BK, STAGE = A_BYTES + SP_BN * SP_BK;
  const CUtensorMap* const ta = &maps.a[p];
  const CUtensorMap* const tb = &maps.b[p];

  if (tid == 0) {
    for (int s = 0; s < SP_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&acc_full, 1);
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == 5) tmem_alloc(&tmem_base_s, SP_BN);
  if (warp == 4 && lane == 0) {
    prefetch_tmap(ta);
    prefetch_tmap(tb);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  pdl_wait();
  pdl_trigger();
  const int n_work = *jobs.n_work;
  if (m0 < n_work) {
    if (warp == 4) {
      const uint32_t on = elect_one();
      bool ok = true;
      int s = 0, i = 0;
      uint32_t ph = 1;
      for (; i < nk; ++i) {
        ok = i < SP_STAGES || mbar_wait_warp(&empty[s], ph, jobs.wait_limit);   // (a stage that has never been filled is free)
        if (!ok) break;
        mbar_expect_tx(on, &full[s], STAGE);
        tma_load_2d(on, smem + s * STAGE, ta, i * SP_BK, m0, &full[s]);
        tma_load_2d(on, smem + s * STAGE + A_BYTES, tb, i * SP_BK, n0, &full[s]);
        if (++s == SP_STAGES) {
          s = 0;
          ph ^= 1;
        }
      }
      if (!ok) {
        if (lane == 0) atomicExch(jobs.status, Q4_ERR_TIMEOUT);
        ring_landed(full, SP_STAGES, i);
      }
    } else if (warp == 5) {
      const uint32_t idesc = umma_idesc_i8(umma_rows(jobs.tile_rows), SP_BN);
      const uint32_t on = elect_one();
      bool ok = true, ready = mbar_test(&full[0], 0);
      int s = 0;
      uint32_t ph = 0;
      for (int i = 0; i < nk && ok; ++i) {
        ok = mbar_wait_warp_tested(ready, &full[s], ph, jobs.wait_limit);
        if (!ok) break;
        tc_fence_after();
        const int st = s;
        if (++s == SP_STAGES) {
          s = 0;
          ph ^= 1;
        }
        ready = mbar_test(&full[s], ph);
        const uint64_t da = umma_desc_sw128(smem_u32(smem + st * STAGE));
        const uint64_t db = umma_desc_sw128(smem_u32(smem + st * STAGE + A_BYTES));
#pragma unroll
        for (int kk = 0; kk < SP_BK / 32; ++kk) umma_i8(on, tmem, da + 2 * kk, db + 2 * kk, idesc, (i | kk) != 0);
        umma_commit(on, &empty[st]);
      }
      umma_commit(on, &acc_full);
      if (!ok) {
        if (lane == 0) atomicExch(jobs.status, Q4_ERR_TIMEOUT);
        ring_landed(full, SP_STAGES, nk);
      }
    } else {
      const int n = m0 + umma_lane_row(umma_rows(jobs.tile_rows), warp, lane);
      const int dst = n < n_work ? jobs.dst_row[n] : -1;
      const bool ok = mbar_wait_warp(&acc_full, 0, jobs.wait_limit);
      tc_fence_after();
      if (!ok) {   // tensor memory is not freed before the products that have been issued are done
        if (lane == 0) atomicExch(jobs.status, Q4_ERR_TIMEOUT);
        mbar_wait_warp(&acc_full, 0);
      }
      float* const out = jobs.job[p].sums + (long long)dst * 4 * K + n0;
      const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
      for (int c0 = 0; c0 < SP_BN; c0 += 32) {
        int r[32];
        tmem_ld32(taddr + c0, r);
        tmem_ld_wait();
        if (!ok || dst < 0) continue;
#pragma unroll
        for (int i = 0; i < 32; i += 8)
          st_global_v8(out + c0 + i, make_float4((float)r[i], (float)r[i + 1], (float)r[i + 2], (float)r[i + 3]),
                       make_float4((float)r[i + 4], (float)r[i + 5], (float)r[i + 6], (float)r[i + 7]));
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 5) tmem_dealloc(tmem, SP_BN);
}
cudaError_t launch_state_products(const StateProductJobs& args, cudaStream_t s, bool dependent) {
  StateProductJobs a = args;
  const int rows_pad = (a.N + SP_BM - 1) / SP_BM * SP_BM;
  a.wait_limit = test_ring_wait_limit();
  a.tile_rows = a.N < SP_BM ? (a.N + 7) / 8 * 8 : SP_BM;   // a single row tile fetches no rows beyond the launch's
  StateMaps maps;
  memset(&maps, 0, sizeof(maps));
  int tiles = 0;
  for (int i = 0; i < a.n_jobs; ++i) {
    const int H = a.job[i].H;
    if (H % SP_BK != 0 || !make_tmap_i8(&maps.a[i], a.job[i].h8, H, rows_pad, H, a.tile_rows) ||
        !make_tmap_i8(&maps.b[i], a.job[i].w8, H, 4 * (uint64_t)H, H, SP_BN))
      return cudaErrorInvalidValue;
    tiles += H / (SP_BN / 4);
  }
  static bool configured_on[MAX_DEVICES];
  bool& configured = configured_on[device_slot()];
  if (!configured) {
    const cudaError_t e = cudaFuncSetAttribute(k_state_products, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SP_SMEM);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  timing_begin(s);
  const cudaError_t e = launch_ex(k_state_products, dim3(tiles, rows_pad / SP_BM), dim3(192), SP_SMEM, s, dependent, 1, maps, a);
  timing_end(s);
  ++g_launches;
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace q4
