// The label-free end of an alignment-length synchronous search.  Once no slot of an utterance may emit another label (all
// have spent their budget, or the beam is empty), the rest of its search is known but for the blanks: every slot stays on
// its prediction vector and takes one frame an iteration until the frames end.  So the selection stops at that iteration
// (it "freezes" the utterance), the steps end when all utterances are frozen, and two launches do the rest:
//   k_tail_blank : log P(blank) of every frozen slot at every frame that is left, as one batch of joint-network rows;
//   k_tail_walk  : the remaining iterations of each utterance, one warp each: scores, order, finished list, history.
// The arithmetic is the step kernels' own (tanh(e p) and its codes; sums over the vocabulary in the same order, with the
// heads' functions), so beams and scores are the same bits.  A step costs 12 us (one utterance) to 25 us (64 x 16 slots) of
// dependent launches when nothing is labelled, a joint-network row here about 1 ns.
#include <string.h>

#include "q4_internal.h"
#include "q4_mma.cuh"

namespace q4 {

constexpr int TL_BM = 128;                     // rows (slot, frame) per tile
constexpr int TL_D = 256;                      // width of the joint network
constexpr int TL_WARPS = 16;                   // warps that form codes and read sums; one more copies, one more issues
constexpr int TL_THREADS = 32 * (TL_WARPS + 2);
constexpr int TL_BLOCKS = 8;                   // blocks of the vocabulary, as in the cluster head
constexpr int TL_MAXW = 16;
// Vocabularies of at most 256 entries: logits to shared memory, summed by a warp per row (the selection's row_lse).
constexpr int TL_SMALL_V = 256, TL_PITCH = TL_SMALL_V + 1;

template <int NB, bool SMALL>
struct TailShape {
  static constexpr int STAGE = NB * TL_D;                              // output-layer rows of a block
  static constexpr int NS = SMALL ? 2 : 128 * 1024 / STAGE;
  static constexpr int OPS = TL_BM * TL_D;
  static constexpr int RED = SMALL ? TL_BM * TL_PITCH * 4 : TL_BLOCKS * 4 * TL_BM * 2 * 4;
  static constexpr int CST = (SMALL ? TL_SMALL_V : TL_BLOCKS * NB) * 2 * 4;
  static constexpr size_t SMEM = (size_t)OPS + (size_t)NS * STAGE + RED + CST + 1024;
};

// A persistent CTA per SM walks the tiles g = blockIdx.x, + gridDim.x, ...: tile k of utterance b holds its rows
// [128 k, 128 k + 128), row = frame * W + slot.  16 warps form the codes of tanh(e p) in the operand tile; the copy warp
// streams the output layer's rows block by block from the L2; the MMA warp fills two accumulators in turn, which the 16
// warps read as the head kernel does (row quarter, column share).  Bound by its arithmetic: 32 K tanh and 128 K
// exponentials a tile, about 15 us with V = 1024.
template <int NB, bool SMALL>
__global__ void __launch_bounds__(TL_THREADS, 1) k_tail_blank(const __grid_constant__ CUtensorMap tma_wo,
                                                              const __grid_constant__ TailArgs a) {
  using Z = TailShape<NB, SMALL>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* const ops = smem;
  uint8_t* const ring = ops + Z::OPS;
  float* const red = reinterpret_cast<float*>(ring + Z::NS * Z::STAGE);
  float* const s_sc = reinterpret_cast<float*>(ring + Z::NS * Z::STAGE + Z::RED);
  float* const s_bi = s_sc + Z::CST / 8;
  __shared__ uint64_t full[Z::NS], empty[Z::NS], ops_ready, acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_base_s;
  __shared__ float s_blank[TL_BM];
  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const int W = a.W, V = a.V, B = a.B;
  const int n_blk = (V + NB - 1) / NB;
  const q4_beam_state& st = a.st;

  if (tid == 0) {
    for (int s = 0; s < Z::NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&ops_ready, TL_WARPS);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], TL_WARPS);
    }
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == TL_WARPS + 1) tmem_alloc(&tmem_base_s, 2 * NB);
  if (warp == TL_WARPS && lane == 0) prefetch_tmap(&tma_wo);
  for (int c = tid; c < V; c += TL_THREADS) {
    s_sc[c] = __fmul_rn(a.z_act.scale, a.sc_out[c]);
    s_bi[c] = a.b_out ? a.b_out[c] : 0.0f;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  const int T = a.call->T, n_iters = T + a.call->u_max;
  const int tpu = (T * W + TL_BM - 1) / TL_BM, n_tiles = B * tpu;
  const int32_t* const first = a.frozen;        // iteration an utterance was frozen at (negative: not)
  const int32_t* const left = a.frozen + B;     // frames it has left
  bool ok = true;

  if (warp == TL_WARPS) {
    const uint32_t on = elect_one();
    int s = 0;
    uint32_t ph = 1, issued = 0;
    for (int g = blockIdx.x; g < n_tiles && ok; g += gridDim.x) {
      const int b = g / tpu, k = g - b * tpu;
      if (k * TL_BM >= left[b] * W) continue;
      for (int i = 0; i < n_blk; ++i) {
        ok = mbar_wait_warp(&empty[s], ph);   // passes at once for a stage that has never been filled
        if (!ok) break;
        mbar_expect_tx(on, &full[s], Z::STAGE);
#pragma unroll
        for (int kc = 0; kc < 2; ++kc) tma_load_2d(on, ring + s * Z::STAGE + kc * NB * 128, &tma_wo, kc * 128, i * NB, &full[s]);
        ++issued;
        if (++s == Z::NS) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    if (!ok) {   // nobody leaves while copies are on their way here (bounded)
      const uint32_t n = issued < (uint32_t)Z::NS ? issued : (uint32_t)Z::NS;
      for (uint32_t j = issued - n; j != issued; ++j) mbar_wait_warp(&full[j % Z::NS], (j / Z::NS) & 1);
    }
  } else if (warp == TL_WARPS + 1) {
    const uint32_t idesc = umma_idesc_i8(TL_BM, NB), on = elect_one();
    int s = 0, blk = 0, tile = 0;
    uint32_t ph = 0;
    for (int g = blockIdx.x; g < n_tiles && ok; g += gridDim.x) {
      const int b = g / tpu, k = g - b * tpu;
      if (k * TL_BM >= left[b] * W) continue;
      ok = mbar_wait_warp(&ops_ready, tile & 1);
      if (!ok) break;
      ++tile;
      for (int i = 0; i < n_blk; ++i, ++blk) {
        const int buf = blk & 1, use = blk >> 1;
        if (use >= 1) ok = mbar_wait_warp(&acc_empty[buf], (use - 1) & 1);
        if (ok) ok = mbar_wait_warp(&full[s], ph);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int j = 0; j < TL_D / 32; ++j) {
          const uint64_t da = umma_desc_sw128(smem_u32(ops + (j >> 2) * TL_BM * 128)) + 2 * (j & 3);
          const uint64_t db = umma_desc_sw128(smem_u32(ring + s * Z::STAGE + (j >> 2) * NB * 128)) + 2 * (j & 3);
          umma_i8(on, tmem + buf * NB, da, db, idesc, j != 0);
        }
        umma_commit(on, &empty[s]);
        umma_commit(on, &acc_full[buf]);
        if (++s == Z::NS) {
          s = 0;
          ph ^= 1;
        }
      }
    }
  } else {
    const int q = warp & 3, cs = warp >> 2;
    const int rt = q * 32 + lane;
    const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16);
    const int lo = act_lo(a.z_act), hi = act_hi(a.z_act);
    const float* const e = a.call->e;
    int blk = 0;
    for (int g = blockIdx.x; g < n_tiles; g += gridDim.x) {
      const int b = g / tpu, k = g - b * tpu, rows = left[b] * W;
      if (k * TL_BM >= rows) continue;
      // ---- codes of tanh(e p): a warp's 8 rows, 8 elements per lane
      int my_row = -1, my_t = 0;
      if (lane < TL_BM / TL_WARPS) {
        const int R = k * TL_BM + warp * (TL_BM / TL_WARPS) + lane;
        if (R < rows) {
          const int o = b * W + R % W;
          my_t = st.t[o] + R / W;
          if (my_t < T) my_row = st.row[o];
        }
      }
#pragma unroll 2
      for (int i = 0; i < TL_BM / TL_WARPS; ++i) {
        const int row = __shfl_sync(0xffffffffu, my_row, i), t = __shfl_sync(0xffffffffu, my_t, i);
        uint32_t w[2] = {0, 0};
        if (row >= 0) {
          const float4* ep = reinterpret_cast<const float4*>(e + ((long long)t * B + b) * TL_D + 8 * lane);
          const float4* pp = reinterpret_cast<const float4*>(st.pred_p + (long long)row * TL_D + 8 * lane);
          const float4 e0 = ep[0], e1 = ep[1], p0 = pp[0], p1 = pp[1];
          const float ev[8] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w};
          const float pv[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
          for (int j = 0; j < 8; ++j)
            w[j >> 2] |= (uint32_t)(quantize1(tanh_fixed(__fmul_rn(ev[j], pv[j])), a.z_act.inv_scale, a.z_act.zero_point, lo, hi) &
                                    0xFF) << (8 * (j & 3));
        }
        const int r = warp * (TL_BM / TL_WARPS) + i;
        *reinterpret_cast<uint2*>(ops + (lane >> 4) * TL_BM * 128 + r * 128 + ((((lane & 15) >> 1) ^ (r & 7)) << 4) +
                                  ((lane & 1) << 3)) = make_uint2(w[0], w[1]);
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ops_ready);
      // ---- sums of the blocks
      for (int i = 0; i < n_blk; ++i, ++blk) {
        const int buf = blk & 1;
        if (ok) ok = mbar_wait_warp(&acc_full[buf], (blk >> 1) & 1);   // (after a wait that ran out: no more waits, no stores)
        tc_fence_after();
        constexpr int CPT = NB / 4, CH = CPT < 32 ? CPT : 32;
        float v[CPT];
#pragma unroll
        for (int ch = 0; ch < CPT / CH; ++ch) {
          int r[CH];
          tmem_ld(taddr + buf * NB + CPT * cs + CH * ch, r);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < CH; j += 4) {
            const int c = i * NB + CPT * cs + CH * ch + j;
            const float4 sc = *reinterpret_cast<const float4*>(s_sc + c), bi = *reinterpret_cast<const float4*>(s_bi + c);
            v[CH * ch + j + 0] = __fmaf_rn((float)r[j + 0], sc.x, bi.x);
            v[CH * ch + j + 1] = __fmaf_rn((float)r[j + 1], sc.y, bi.y);
            v[CH * ch + j + 2] = __fmaf_rn((float)r[j + 2], sc.z, bi.z);
            v[CH * ch + j + 3] = __fmaf_rn((float)r[j + 3], sc.w, bi.w);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[buf]);
        const int col0 = i * NB + CPT * cs;
        if (SMALL) {
#pragma unroll
          for (int j = 0; j < CPT; ++j) red[rt * TL_PITCH + col0 + j] = v[j];   // columns beyond V are not read
        } else {
          float my_m = -INFINITY;
#pragma unroll
          for (int j = 0; j < CPT; ++j) {
            if (col0 + j >= V) v[j] = -INFINITY;
            my_m = fmaxf(my_m, v[j]);
          }
          *reinterpret_cast<float2*>(red + ((i * 4 + cs) * TL_BM + rt) * 2) = make_float2(my_m, exp_sum(v, my_m));
          if (i == 0 && cs == 0) s_blank[rt] = v[0];
        }
      }
      asm volatile("bar.sync 1, %0;" ::"n"(32 * TL_WARPS) : "memory");
      // ---- log P(blank) into the history's place of its iteration, where the walk finds it.  (The next tile's sums are
      // written after all 16 warps have handed over its codes, so after what is read here.)
      auto put = [&](int r, float lp) {
        const int R = k * TL_BM + r;
        if (!ok || R >= rows) return;
        const int it = first[b] + R / W;
        if (it < n_iters) st.bp_score[((long long)it * B + b) * W + R % W] = lp;
      };
      if (SMALL) {
#pragma unroll 1
        for (int i = 0; i < TL_BM / TL_WARPS; ++i) {
          const int r = warp * (TL_BM / TL_WARPS) + i;
          const float* x = red + r * TL_PITCH;
          float m = -INFINITY;
          for (int c = lane; c < V; c += 32) m = fmaxf(m, x[c]);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
          float sum = 0.0f;
          for (int c = lane; c < V; c += 32) sum += expf(x[c] - m);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
          if (lane == 0) put(r, x[0] - (m + logf(sum)));
        }
      } else if (cs == 0) {
        float pm[TL_BLOCKS], ps[TL_BLOCKS], m = -INFINITY;
#pragma unroll
        for (int i = 0; i < TL_BLOCKS; ++i) {
          pm[i] = -INFINITY;
          ps[i] = 0.0f;
          if (i < n_blk) {
            float xm[4], xs[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const float2 x = *reinterpret_cast<const float2*>(red + ((i * 4 + c) * TL_BM + rt) * 2);
              xm[c] = x.x;
              xs[c] = x.y;
            }
            pm[i] = fmaxf(fmaxf(xm[0], xm[1]), fmaxf(xm[2], xm[3]));
            ps[i] = exp_sum(xm, xs, pm[i]);
          }
          m = fmaxf(m, pm[i]);
        }
        put(rt, s_blank[rt] - (m + logf(exp_sum(pm, ps, m))));
      }
    }
  }
  if (!ok && lane == 0) atomicExch(st.status, Q4_ERR_TIMEOUT);
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == TL_WARPS + 1) tmem_dealloc(tmem, 2 * NB);
}

// Order-preserving integer of a score (see make_key of the selection; equal scores are ordered by slot).
__device__ __forceinline__ uint32_t score_key(float s) {
  const uint32_t b = __float_as_uint(s);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// One warp per utterance, lane = slot: what the selection does in an iteration without label proposals, once for each
// iteration that is left.  A dependent chain of about 0.15 us an iteration; the blanks' log-probabilities (one 64-byte
// row an iteration) are fetched 8 iterations ahead.
__global__ void __launch_bounds__(32) k_tail_walk(const __grid_constant__ TailArgs a) {
  __shared__ int s_src[TL_MAXW];
  constexpr int AHEAD = 8;
  const int lane = threadIdx.x, b = blockIdx.x, W = a.W, B = a.B;
  const q4_beam_state& st = a.st;
  const float NEG = -INFINITY;
  pdl_wait();
  const int T = a.call->T, n_iters = T + a.call->u_max;
  const int f = a.frozen[b];
  if (f < 0 || f >= n_iters) return;
  const bool mine = lane < W;
  const int o = b * W + (mine ? lane : 0);
  const int row0 = mine ? st.row[o] : -1, u0 = st.u[o], last0 = st.last_tok[o];
  const uint64_t hash0 = st.hash[o], prev0 = st.prev_hash[o];
  float score = st.score[o];
  int t = st.t[o], orig = lane;
  bool alive = row0 >= 0, changed = false;
  int fin_n = st.fin_n[b], fi = 0, fl = 0;
  float fs = NEG;
  bool any_fin = false;
  if (mine && lane < fin_n) {
    fs = st.fin_score[o];
    fi = st.fin_iter[o];
    fl = st.fin_slot[o];
  }
  float next[AHEAD];
  auto fetch = [&](int it0) {
#pragma unroll
    for (int j = 0; j < AHEAD; ++j)
      next[j] = mine && it0 + j < n_iters ? st.bp_score[((long long)(it0 + j) * B + b) * W + lane] : 0.0f;
  };
  fetch(f);
  int it = f;
  while (it < n_iters && __any_sync(0xffffffffu, alive)) {
    float cur[AHEAD];
#pragma unroll
    for (int j = 0; j < AHEAD; ++j) cur[j] = next[j];
    fetch(it + AHEAD);
#pragma unroll
    for (int j = 0; j < AHEAD; ++j) {
      if (it + j >= n_iters) break;
      const float lp = __shfl_sync(0xffffffffu, cur[j], orig);
      float sc = NEG;
      if (alive) sc = (float)((double)score + (double)lp);
      const bool fin = alive && t + 1 == T;   // consumed the last frame: to the finished list, sorted, the W best
      unsigned fm = __ballot_sync(0xffffffffu, fin);
      any_fin = any_fin || fm != 0u;
#pragma unroll 1
      while (fm) {
        const int x = __ffs(fm) - 1;
        fm &= fm - 1;
        const float S = __shfl_sync(0xffffffffu, sc, x);
        const int pos = __popc(__ballot_sync(0xffffffffu, lane < fin_n && !(fs < S)));
        const float fs1 = __shfl_up_sync(0xffffffffu, fs, 1);
        const int fi1 = __shfl_up_sync(0xffffffffu, fi, 1), fl1 = __shfl_up_sync(0xffffffffu, fl, 1);
        if (pos >= W) continue;
        if (lane > pos) {
          fs = fs1;
          fi = fi1;
          fl = fl1;
        } else if (lane == pos) {
          fs = S;
          fi = it + j;
          fl = x;
        }
        fin_n = min(fin_n + 1, W);
      }
      const bool cnd = alive && !fin && sc > NEG;
      const uint32_t key = cnd ? score_key(sc) : 0u;
      int rank = 0;
#pragma unroll
      for (int x = 0; x < TL_MAXW; ++x) {
        const uint32_t kx = __shfl_sync(0xffffffffu, key, x);
        rank += kx > key || (kx == key && x < lane);
      }
      const int nw = __popc(__ballot_sync(0xffffffffu, cnd));
      if (cnd) s_src[rank] = lane;
      __syncwarp();
      const int src = lane < nw ? s_src[lane] : lane;
      __syncwarp();
      const float sc1 = __shfl_sync(0xffffffffu, sc, src);
      const int o1 = __shfl_sync(0xffffffffu, orig, src), t1 = __shfl_sync(0xffffffffu, t, src);
      alive = lane < nw;
      if (alive) {
        score = sc1;
        orig = o1;
        t = t1 + 1;
        changed = true;
      }
      if (mine) {
        const size_t hist = ((size_t)(it + j) * B + b) * W + lane;
        st.bp_parent[hist] = alive ? src : -1;
        st.bp_token[hist] = alive ? 0 : -1;
        st.bp_score[hist] = alive ? score : 0.0f;
      }
    }
    it += AHEAD;
  }
  // nothing is left of the beam: empty iterations
  const long long n = (long long)max(n_iters - it, 0) * W;
  for (long long i = lane; i < n; i += 32) {
    const size_t hist = ((size_t)(it + i / W) * B + b) * W + i % W;
    st.bp_parent[hist] = -1;
    st.bp_token[hist] = -1;
    st.bp_score[hist] = 0.0f;
  }
  // the state as the steps would have left it
  const int u1 = __shfl_sync(0xffffffffu, u0, orig), last1 = __shfl_sync(0xffffffffu, last0, orig);
  const int row1 = __shfl_sync(0xffffffffu, row0, orig);
  const uint64_t hash1 = __shfl_sync(0xffffffffu, hash0, orig), prev1 = __shfl_sync(0xffffffffu, prev0, orig);
  if (mine) {
    if (changed) {
      st.score[o] = score;
      st.t[o] = t;
      st.u[o] = u1;
      st.hash[o] = hash1;
      st.prev_hash[o] = prev1;
      st.last_tok[o] = last1;
    }
    st.row[o] = alive ? row1 : -1;
    st.adv_src[o] = -1;
    st.adv_dst[o] = -1;
    st.adv_tok[o] = -1;
    if (any_fin && lane < fin_n) {
      st.fin_score[o] = fs;
      st.fin_iter[o] = fi;
      st.fin_slot[o] = fl;
    }
  }
  if (any_fin && lane == 0) st.fin_n[b] = fin_n;
}

bool search_tail_supported(int V, int D) { return D == TL_D && V <= TL_BLOCKS * 256; }

template <int NB, bool SMALL>
static cudaError_t tail_blank_launch(const CUtensorMap& to, const TailArgs& a, int ctas, cudaStream_t s) {
  static bool configured_on[MAX_DEVICES];
  bool& configured = configured_on[device_slot()];
  if (!configured) {
    const cudaError_t e = cudaFuncSetAttribute(k_tail_blank<NB, SMALL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)TailShape<NB, SMALL>::SMEM);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  return launch_ex(k_tail_blank<NB, SMALL>, dim3(ctas), dim3(TL_THREADS), TailShape<NB, SMALL>::SMEM, s, false, 1, to, a);
}
cudaError_t launch_search_tail(const TailArgs& a, int T, const int8_t* wo8, cudaStream_t s) {
  const bool small = a.V <= TL_SMALL_V;
  const int nb = small || a.V <= 512 ? 64 : a.V <= 1024 ? 128 : 256;
  CUtensorMap to;
  if (!make_tmap_i8(&to, wo8, TL_D, a.V, TL_D, nb)) return cudaErrorInvalidValue;
  const long long tiles = (long long)a.B * (((long long)T * a.W + TL_BM - 1) / TL_BM);
  if (tiles > INT32_MAX) return cudaErrorInvalidValue;
  const int ctas = tiles < sm_count() ? (int)tiles : sm_count();
  timing_begin(s);
  cudaError_t e = small       ? tail_blank_launch<64, true>(to, a, ctas, s)
                  : nb == 64  ? tail_blank_launch<64, false>(to, a, ctas, s)
                  : nb == 128 ? tail_blank_launch<128, false>(to, a, ctas, s)
                              : tail_blank_launch<256, false>(to, a, ctas, s);
  timing_end(s);
  ++g_launches;
  if (e != cudaSuccess) return e;
  e = launch_ex(k_tail_walk, dim3(a.B), dim3(32), 0, s, false, 1, a);
  ++g_launches;
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace q4
