// Beam bookkeeping kernels: per-utterance log-softmax of the joint logits, the
// density-ratio score of Eq. 1 for every proposal, merging of equal label strings,
// the finished list, selection of the W best, state-row allocation and back-pointers.
// One CTA per utterance; nothing here leaves the GPU (the paper ran hypothesis sorting
// on the host CPU, Section 4.1).
#include <math.h>

#include "q4_internal.h"

namespace q4 {

constexpr int SEL_NT = 512;
constexpr int MAXW = 16;
constexpr uint64_t HASH0 = 0x243F6A8885A308D3ull;  // hash of the empty label string

__device__ __forceinline__ uint64_t hash_mix(uint64_t h, uint32_t k) {
  uint64_t z = h ^ (0x9E3779B97F4A7C15ull * (uint64_t)(k + 1u));
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Order-preserving key: larger score first, then smaller proposal index
// (index = parent slot * V + token, so parent ascending then token ascending).
__device__ __forceinline__ uint64_t make_key(float s, uint32_t idx) {
  uint32_t b = __float_as_uint(s);
  b = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
  return ((uint64_t)b << 32) | (uint64_t)(~idx);
}
__device__ __forceinline__ float key_score(uint64_t key) {
  uint32_t b = (uint32_t)(key >> 32);
  b = (b & 0x80000000u) ? (b & 0x7FFFFFFFu) : ~b;
  return __uint_as_float(b);
}
__device__ __forceinline__ uint64_t u64max(uint64_t a, uint64_t b) { return a > b ? a : b; }
// A selection is a chain of short phases on 16 warps of one SM per utterance, each bound by a memory or barrier
// latency: rows of the three tables 3.0 us (196 KB into one SM), state 1.3 to 2.2, list 1.2, ranking 1, merge
// .5 to 1, bookkeeping 1.2 (64 utterances, label iteration: 9.9 us after its wait; 12.6 before).  Every
// instruction runs a few times at most and other kernels have used the instruction caches in between, so
// code size counts: 41 KB instead of 108 KB with every pass over the proposals in registers and unrolled loops.
// ---- proposals of one slot, by one warp.  A label's score is (float)(S + rho + inc) in double, where inc =
// log P(k) + lambda_t log P_tgt(k) - lambda_s log P_src(k) in fp32 (magnitude of tens) and S is the slot's
// running score: within a slot the score grows with inc, so proposals are compared by inc and only the few
// that matter are scored (conversions to and from double run at an eighth of the fp32 rate: scoring all
// 16 x 1024 proposals cost 1 us of the selection).
// MODE 2: V <= 1024, a multiple of 4, 16-byte aligned rows: element i of a lane is k = 128 (i / 4) + 4 lane +
// i % 4; MODE 1: V <= 1024: k = lane + 32 i; the 32 values of a lane stay in registers.  MODE 0: any V, by loops
// over shared memory.
template <int MODE>
__device__ __forceinline__ int slot_elem(int i, int lane) {
  return MODE == 2 ? 128 * (i >> 2) + 4 * lane + (i & 3) : lane + 32 * i;
}
template <int MODE, int N>
__device__ __forceinline__ void load_elems(const float* p, int i0, int V, int lane, float beyond, float (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; i += MODE == 2 ? 4 : 1) {
    const int k = slot_elem<MODE>(i0 + i, lane);
    if (MODE == 2) {
      const float4 q = k < V ? *reinterpret_cast<const float4*>(p + k) : make_float4(beyond, beyond, beyond, beyond);
      v[i] = q.x;
      v[i + 1] = q.y;
      v[i + 2] = q.z;
      v[i + 3] = q.w;
    } else {
      v[i] = k < V ? p[k] : beyond;
    }
  }
}
// log(sum(exp)) of a row of logits in memory, by a warp
__device__ __forceinline__ float row_lse(const float* x, int V, int lane) {
  float m = -INFINITY;
#pragma unroll 8
  for (int k = lane; k < V; k += 32) m = fmaxf(m, x[k]);
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float sum = 0.0f;
#pragma unroll 4
  for (int k = lane; k < V; k += 32) sum += expf(x[k] - m);
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return m + logf(sum);
}
__device__ __forceinline__ float label_inc(const BeamSelArgs& a, float lp, float s, float t) {
  return __fmaf_rn(a.lambda_t, t, __fmaf_rn(-a.lambda_s, s, lp));
}
// The increments of a slot's labels, from the joint's row (v: loaded already in MODE 1 and 2), into inc[]
// (shared memory) and v; returns the lane's best one, elements with a bit in `skip` left out.
template <int MODE>
__device__ __forceinline__ float slot_increments(const BeamSelArgs& a, float (&v)[32], const float* x, const float* ls,
                                                 const float* lt, float lse, uint32_t skip, float* inc, int lane) {
  const int V = a.V;
  float best = -INFINITY;
  if (MODE == 0) {
#pragma unroll 4
    for (int k = lane; k < V; k += 32) {
      const float w = label_inc(a, x[k] - lse, ls[k], lt[k]);
      inc[k] = w;
      if (k > 0) best = fmaxf(best, w);   // (no bound is taken from it)
    }
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h) {   // two round trips to memory
      float sv[16], tv[16];
      load_elems<MODE>(ls, 16 * h, V, lane, 0.0f, sv);
      load_elems<MODE>(lt, 16 * h, V, lane, 0.0f, tv);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[16 * h + i] = label_inc(a, v[16 * h + i] - lse, sv[i], tv[i]);
    }
#pragma unroll
    for (int i = 0; i < 32; i += MODE == 2 ? 4 : 1) {
      const int k = slot_elem<MODE>(i, lane);
      if (k < V) {
        if (MODE == 2)
          *reinterpret_cast<float4*>(inc + k) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        else
          inc[k] = v[i];
      }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (!((skip >> i) & 1u)) best = fmaxf(best, v[i]);   // -inf beyond the row
  }
  return best;
}
__device__ __forceinline__ float label_score(double s_rho, float inc) { return (float)(s_rho + (double)inc); }

// A lower bound of the W-th best label proposal: the proposals are split into 16 disjoint groups (by lane
// modulo 16); each group's best is a distinct proposal, so at least 16 >= W proposals reach the smallest of
// the 16 group maxima.  An empty group gives -inf: everything valid passes.
__device__ __forceinline__ float label_bound(const float (*gmax)[16], int lane) {   // rows of slots that are not there hold -inf
  float g = -INFINITY;
#pragma unroll
  for (int w = 0; w < SEL_NT / 32; w += 2) g = fmaxf(g, gmax[w + (lane >> 4)][lane & 15]);
  g = fmaxf(g, __shfl_xor_sync(0xffffffffu, g, 16));
#pragma unroll 1
  for (int o = 8; o > 0; o >>= 1) g = fminf(g, __shfl_xor_sync(0xffffffffu, g, o));
  return g;
}
__device__ __forceinline__ void list_add(uint64_t* list, int* list_n, int cap, float score, uint32_t idx) {
  const int p = atomicAdd(list_n, 1);
  if (p < cap) list[p] = make_key(score, idx);
}
// The labels of a slot with a score of at least `bound` go to the list (entries beyond `cap` are only counted).
template <int MODE>
__device__ __forceinline__ void collect_labels(const float (&v)[32], uint32_t skip, const float* inc, double s_rho, float bound,
                                               int V, uint32_t off, uint64_t* list, int* list_n, int cap, int lane) {
  // (float)(s_rho + inc) >= bound implies inc >= bound - s_rho - (half a rounding step of bound)
  const float thr = __double2float_rd((double)bound - s_rho - 2.4e-7 * fabs((double)bound) - 1e-30);
  uint32_t hit = 0;
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (v[i] >= thr) hit |= 1u << i;
  hit &= ~skip;
#pragma unroll 1
  while (hit) {
    const int i = __ffs(hit) - 1;
    hit &= hit - 1;
    const int k = slot_elem<MODE>(i, lane);
    if (k >= V) continue;   // without a bound (a group is empty) -inf passes the comparison
    const float sc = label_score(s_rho, inc[k]);
    if (sc >= bound && sc > -INFINITY) list_add(list, list_n, cap, sc, off + (uint32_t)k);
  }
}

// The list by the exact threshold: (1) every thread's best proposal ("head") among its strided share of its
// slots; (2) the W-th best head, found bit by bit with block-wide counts, is a lower bound of the W-th
// best proposal, and only the threads owning the W best heads can hold anything at or above it; (3) those
// go to the list.  blank: the slots' blank scores (null: blanks are no proposals here).
__device__ __forceinline__ void collect_exact(const float* cand, const int* s_row, const int* s_lab, const float* s_score, float rho,
                                              const float* blank, int W, int V, uint64_t* list, int* list_n, int cap, int warp,
                                              int lane) {
  uint64_t head = 0, th = 0;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    if (pass == 0 || (head != 0ull && head >= th)) {
#pragma unroll 1
      for (int w = warp; w < W; w += SEL_NT / 32) {
        if (s_row[w] < 0) continue;
        const double s_rho = (double)s_score[w] + (double)rho;
#pragma unroll 2
        for (int k = lane; k < (s_lab[w] ? V : 1); k += 32) {
          if (k == 0 && !blank) continue;
          const float x = k == 0 ? blank[w] : label_score(s_rho, cand[(size_t)w * V + k]);
          if (!(x > -INFINITY)) continue;
          const uint64_t key = make_key(x, (uint32_t)w * (uint32_t)V + (uint32_t)k);
          if (pass == 0) {
            head = u64max(head, key);
          } else if (key >= th) {
            const int p = atomicAdd(list_n, 1);
            if (p < cap) list[p] = key;
          }
        }
      }
    }
    if (pass == 1) break;
    // score bits first (32 counts); the index bits matter only if equal scores straddle the bound
#pragma unroll 1
    for (int bit = 63; bit >= 0; --bit) {
      if (bit == 31 && __syncthreads_count(head >= th) <= W) break;
      const uint64_t c = th | (1ull << bit);
      if (__syncthreads_count(head >= c) >= W) th = c;
    }
    // th = the W-th best head (0 if there are fewer than W heads: then everything valid passes)
  }
  __syncthreads();
}

// rank of every list entry by counting; the W best are the winners
__device__ __forceinline__ void rank_list(const uint64_t* list, int ln, int W, int* win_idx, float* win_score, int tid) {
#pragma unroll 1
  for (int i = tid; i < ln; i += SEL_NT) {
    const uint64_t mine = list[i];
    int rank = 0;
#pragma unroll 8
    for (int j = 0; j < ln; ++j) rank += list[j] > mine;
    if (rank < W) {
      win_idx[rank] = (int)(~(uint32_t)mine);
      win_score[rank] = key_score(mine);
    }
  }
}
// entries of the short list; smaller vocabularies have as many proposals near the bound as large ones
__host__ __device__ constexpr int sel_list_cap(int V) { return 16 * ((V + 31) / 32) > 512 ? 16 * ((V + 31) / 32) : 512; }

// End of the last step of a graph's loop, by one thread of each utterance after all that it does: the last one
// advances the call and asks for another turn.  (As a kernel of its own 2 us a turn.)  Every utterance is frozen by
// iteration T + u_max, since no hypothesis lives beyond it, so the second condition never ends a loop; it bounds it.
__device__ __forceinline__ void loop_step_end(const BeamSelArgs& a, int iter, int last) {
  __threadfence();
  if (atomicAdd(&a.call->arrived, 1) != a.B - 1) return;
  __threadfence();
  a.call->arrived = 0;
  a.call->iter += a.loop_iters;   // (everyone has read it)
  cudaGraphSetConditional(a.loop, ld_coherent(&a.call->n_frozen) < a.B && iter + 1 < last ? 1u : 0u);
}

template <int MODE>
__global__ void __launch_bounds__(SEL_NT, 1) k_beam_select(const __grid_constant__ BeamSelArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int W = a.W, V = a.V;
  float* cand = reinterpret_cast<float*>(smem_raw);                         // [W * V] increments of the labels
  uint64_t* list = reinterpret_cast<uint64_t*>(smem_raw + ((size_t)W * V * sizeof(float) + 15) / 16 * 16);       // survivors of the filter
  __shared__ float s_score[MAXW];
  __shared__ int s_t[MAXW], s_u[MAXW], s_row[MAXW], s_last[MAXW];
  __shared__ uint64_t s_hash[MAXW], s_prev[MAXW];
  __shared__ int list_n, s_lab[MAXW];   // s_lab: the slot proposes labels
  __shared__ float s_blank[MAXW];       // scores of the blank proposals
  __shared__ int win_idx[MAXW];
  __shared__ float win_score[MAXW];
  __shared__ float s_gmax[SEL_NT / 32][16];   // per warp: best label proposal of lanes g and g + 16

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x;
  const int base = b * W;
  const q4_beam_state& st = a.st;
  const float NEG = -INFINITY;
  const int N = a.B * W;
  const bool normalized = a.normalized != 0;   // `logits` holds log-probabilities already

  pdl_wait();
  // a replayed search: its length, budget and iteration are in memory
  int T = a.T, u_max = a.u_max, iter = a.iter;
  if (a.call) {
    T = a.call->T;
    u_max = a.call->u_max;
    iter += a.call->iter;
  }
  // what the proposals of slot `warp` read does not wait for the block: the joint's row at once, the language
  // models' rows as soon as the slot's state row is known
  const float* const x = a.logits + (size_t)(base + warp) * V;
  float v[32];
  int my_row = -1, my_u = 0;
  float my_score = 0.0f;
  if (warp < W) {
    my_row = st.row[base + warp];
    my_u = st.u[base + warp];
    my_score = st.score[base + warp];
    if (MODE > 0) load_elems<MODE>(x, 0, V, lane, NEG, v);
  }
  if (tid < W) {
    const int o = base + tid;
    const int row = st.row[o], u = st.u[o];
    s_score[tid] = st.score[o];
    s_t[tid] = st.t[o];
    s_last[tid] = st.last_tok[o];
    s_hash[tid] = st.hash[o];
    s_prev[tid] = st.prev_hash[o];
    s_row[tid] = row;
    s_u[tid] = u;
    s_lab[tid] = row >= 0 && u < u_max;
  }
  if (tid == 0) {
    list_n = 0;
    // the list of pending advances consumed by this iteration is free again
    if (b == 0) st.pend_n[iter & 1] = 0;
  }
  if (lane < 16) s_gmax[warp][lane] = NEG;
  const bool any_labels = __syncthreads_or(my_row >= 0 && my_u < u_max) != 0;
  if (a.frozen && !any_labels) {   // this utterance's remaining iterations are carried out together (q4_tail.cu)
    pdl_trigger();
    if (warp == 0 && a.frozen[b] < 0) {
      int left = lane < W && s_row[lane] >= 0 ? T - s_t[lane] : 0;
      left = max(__reduce_max_sync(0xffffffffu, left), 0);
      if (lane == 0) {
        a.frozen[b] = iter;
        a.frozen[a.B + b] = left;
        atomicAdd(&a.call->n_frozen, 1);
      }
    }
    if (a.loop_iters && tid == 0) loop_step_end(a, iter, T + u_max);
    return;
  }

  // ---- no slot of this utterance may emit a label (all at their label budget, or empty): the only
  // proposals are the blanks of the live slots, at most W of them, no two of which can describe the
  // same string.  One warp, lane = slot: the same score arithmetic, the same finished list and the
  // same order (score descending, then slot) as the general path below, without its passes over V.
  const int cap = sel_list_cap(V);
  const bool blank_only = !a.exact_only && normalized && !any_labels;
  if (blank_only) {
    if (warp == 0) {
      const int w = lane;
      const bool alive = w < W && s_row[w] >= 0;
      float sc = NEG;
      if (alive) sc = (float)((double)s_score[w] + (double)a.logits[(size_t)(base + w) * V]);
      const bool fin = alive && s_t[w] + 1 == T;   // consumed the last frame: goes to the finished list
      if (__any_sync(0xffffffffu, fin)) {
        if (w < W) win_score[w] = sc;                // staging only; overwritten by the ranking below
        __syncwarp();
        if (lane == 0) {
          float* fs = st.fin_score + base;
          int* fi = st.fin_iter + base;
          int* fl = st.fin_slot + base;
          int n = st.fin_n[b];
#pragma unroll 1
          for (int x = 0; x < W; ++x) {
            if (s_row[x] < 0 || s_t[x] + 1 != T) continue;
            const float S = win_score[x];
            int pos = n;
#pragma unroll 1
            while (pos > 0 && fs[pos - 1] < S) --pos;
            if (pos >= W) continue;
            const int last = min(n, W - 1);
#pragma unroll 1
            for (int i = last; i > pos; --i) {
              fs[i] = fs[i - 1];
              fi[i] = fi[i - 1];
              fl[i] = fl[i - 1];
            }
            fs[pos] = S;
            fi[pos] = iter;
            fl[pos] = x;
            n = min(n + 1, W);
          }
          st.fin_n[b] = n;
        }
        __syncwarp();
      }
      const bool cnd = alive && !fin && sc > NEG;
      const uint64_t key = cnd ? make_key(sc, (uint32_t)w * (uint32_t)V) : 0ull;
      int rank = 0;
#pragma unroll 1
      for (int x = 0; x < W; ++x) rank += __shfl_sync(0xffffffffu, key, x) > key;
      if (cnd) {
        win_idx[rank] = w * V;
        win_score[rank] = sc;
      }
      const int n_c = __popc(__ballot_sync(0xffffffffu, cnd));
      if (lane == 0) list_n = n_c;
    }
    __syncthreads();
  } else {
  // ---- proposals: one warp per slot
  const bool fast = MODE > 0 && !a.exact_only;   // a lower bound of the W-th best from group maxima
  const bool my_labels = my_row >= 0 && my_u < u_max;
  const double s_rho = (double)my_score + (double)a.rho;
  // elements that do not count for the bound and are not collected: element 0 (blank), and labels that the merge
  // below folds into another slot's blank (lane w1 tests slot w1, the few hits are handed round the warp)
  uint32_t skip = lane == 0 ? 1u : 0u;
  if (my_row >= 0) {
    const float lse = normalized ? 0.0f : row_lse(x, V, lane);
    if (lane == 0) s_blank[warp] = (float)((double)my_score + (double)((MODE > 0 ? v[0] : x[0]) - lse));
    if (my_labels) {
      if (MODE > 0) {
        const bool hit = lane < W && s_row[lane] >= 0 && s_u[lane] == my_u + 1 && s_prev[lane] == s_hash[warp];
        const int tok = hit ? s_last[lane] : 0;
        unsigned hits = __ballot_sync(0xffffffffu, hit);
#pragma unroll 1
        while (hits) {
          const int src = __ffs(hits) - 1;
          hits &= hits - 1;
          const int t = __shfl_sync(0xffffffffu, tok, src);
          if (MODE == 2 ? (t >> 2 & 31) == lane : (t & 31) == lane) skip |= 1u << (MODE == 2 ? (t >> 7) * 4 + (t & 3) : t >> 5);
        }
      }
      float best = slot_increments<MODE>(a, v, x, a.src_lp + (size_t)my_row * V, a.tgt_lp + (size_t)my_row * V, lse, skip,
                                         cand + (size_t)warp * V, lane);
      best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, 16));
      if (lane < 16) s_gmax[warp][lane] = label_score(s_rho, best);
    }
  }
  __syncthreads();

  // ---- merge: label proposal (w2, k) describing the same string as the blank proposal of w
  if (tid < W * W) {
    const int w = tid / W, w2 = tid % W;
    if (s_row[w] >= 0 && s_lab[w2] && s_u[w] == s_u[w2] + 1 && s_prev[w] == s_hash[w2]) {
      const int k = s_last[w];
      const double p = (double)s_blank[w];
      const double q = (double)label_score((double)s_score[w2] + (double)a.rho, cand[(size_t)w2 * V + k]);
      s_blank[w] = (float)(fmax(p, q) + log1p(exp(-fabs(p - q))));
      cand[(size_t)w2 * V + k] = NEG;
    }
  }
  const float bound = fast ? label_bound(s_gmax, lane) : NEG;
  __syncthreads();

  // ---- finished hypotheses: blank proposals that consume the last frame
  const bool any_fin = __any_sync(0xffffffffu, lane < W && s_row[lane] >= 0 && s_t[lane] + 1 == T);
  if (any_fin) {   // uniform for the block
    if (tid == 0) {
      float* fs = st.fin_score + base;
      int* fi = st.fin_iter + base;
      int* fl = st.fin_slot + base;
      int n = st.fin_n[b];
#pragma unroll 1
      for (int w = 0; w < W; ++w) {
        if (s_row[w] < 0 || s_t[w] + 1 != T) continue;
        const float S = s_blank[w];
        s_blank[w] = NEG;
        int pos = n;
#pragma unroll 1
        while (pos > 0 && fs[pos - 1] < S) --pos;
        if (pos >= W) continue;
        const int last = min(n, W - 1);
#pragma unroll 1
        for (int i = last; i > pos; --i) {
          fs[i] = fs[i - 1];
          fi[i] = fi[i - 1];
          fl[i] = fl[i - 1];
        }
        fs[pos] = S;
        fi[pos] = iter;
        fl[pos] = w;
        n = min(n + 1, W);
      }
      st.fin_n[b] = n;
    }
    __syncthreads();
  }

  // ---- the W best remaining proposals
  bool exact = !fast;
  if (fast) {
    if (my_row >= 0) {
      const uint32_t off = (uint32_t)warp * (uint32_t)V;
      if (lane == 0 && s_blank[warp] >= bound && s_blank[warp] > NEG) list_add(list, &list_n, cap, s_blank[warp], off);
      if (my_labels) collect_labels<MODE>(v, skip, cand + (size_t)warp * V, s_rho, bound, V, off, list, &list_n, cap, lane);
    }
    __syncthreads();
    exact = list_n > cap;     // the bound was too loose for the list: take the exact threshold instead
    if (exact) {
      __syncthreads();
      if (tid == 0) list_n = 0;
      __syncthreads();
    }
  }
  if (exact) collect_exact(cand, s_row, s_lab, s_score, a.rho, s_blank, W, V, list, &list_n, cap, warp, lane);
  rank_list(list, min(list_n, cap), W, win_idx, win_score, tid);
  }
  __syncthreads();
  pdl_trigger();   // only the bookkeeping is left: the next kernel of the stream may set itself up

  if (warp == 0) {
    const int n_win = min(min(list_n, cap), W);

    // ---- next beam, state rows, back-pointers, pending advances: lane s writes slot s
    const int nw = n_win;
    const int row0 = b * (st.rows_per_utt > 0 ? st.rows_per_utt : 2 * W);
    const uint32_t used = __reduce_or_sync(0xffffffffu, lane < W && s_row[lane] >= 0 ? 1u << (s_row[lane] - row0) : 0u);
    const uint32_t free_mask = ~used & (W >= 16 ? 0xFFFFFFFFu : ((1u << (2 * W)) - 1u));
    const int s = lane;
    int idx = 0, w = 0, k = 0;
    bool is_label = false;
    if (s < nw) {
      idx = win_idx[s];
      w = idx / V;
      k = idx % V;
      is_label = k != 0;
    }
    const unsigned lab = __ballot_sync(0xffffffffu, is_label);
    // reserve a range of the next iteration's pending list for this utterance's label extensions
    int pbase = 0;
    if (lane == 0 && lab != 0u) pbase = atomicAdd(st.pend_n + ((iter + 1) & 1), __popc(lab));
    pbase = __shfl_sync(0xffffffffu, pbase, 0);
    const size_t poff = (size_t)((iter + 1) & 1) * N;
    if (s < W) {
      const int o = base + s;
      const size_t hist = ((size_t)iter * a.B + b) * W + s;
      if (s < nw) {
        st.score[o] = win_score[s];
        if (!is_label) {
          st.t[o] = s_t[w] + 1;
          st.u[o] = s_u[w];
          st.hash[o] = s_hash[w];
          st.prev_hash[o] = s_prev[w];
          st.last_tok[o] = s_last[w];
          st.row[o] = s_row[w];
          st.adv_src[o] = -1;
          st.adv_dst[o] = -1;
          st.adv_tok[o] = -1;
        } else {
          // the j-th label extension (in slot order) takes the j-th state row not used by the
          // beam that is being replaced
          const int j = __popc(lab & ((1u << s) - 1u));
          uint32_t rest = free_mask;
#pragma unroll 1
          for (int i = 0; i < j; ++i) rest &= rest - 1;
          const int f = __ffs(rest) - 1;
          st.t[o] = s_t[w];
          st.u[o] = s_u[w] + 1;
          st.hash[o] = hash_mix(s_hash[w], (uint32_t)k);
          st.prev_hash[o] = s_hash[w];
          st.last_tok[o] = k;
          st.row[o] = row0 + f;
          st.adv_src[o] = s_row[w];
          st.adv_dst[o] = row0 + f;
          st.adv_tok[o] = k;
          st.pend_src[poff + pbase + j] = s_row[w];
          st.pend_dst[poff + pbase + j] = row0 + f;
          st.pend_tok[poff + pbase + j] = k;
        }
        st.bp_parent[hist] = w;
        st.bp_token[hist] = k;
        st.bp_score[hist] = win_score[s];
      } else {
        st.row[o] = -1;
        st.adv_src[o] = -1;
        st.adv_dst[o] = -1;
        st.adv_tok[o] = -1;
        st.bp_parent[hist] = -1;
        st.bp_token[hist] = -1;
        st.bp_score[hist] = 0.0f;
      }
    }
    if (a.loop_iters && lane == 0) loop_step_end(a, iter, T + u_max);
  }
}

// rows of the three log-probability tables can be read 16 bytes at a time
static int sel_mode(const BeamSelArgs& a) {
  if (a.V > 1024) return 0;
  const bool wide = a.V % 4 == 0 && ((reinterpret_cast<uintptr_t>(a.logits) | reinterpret_cast<uintptr_t>(a.src_lp) |
                                      reinterpret_cast<uintptr_t>(a.tgt_lp)) & 15) == 0;
  return wide ? 2 : 1;
}
static size_t sel_smem(const BeamSelArgs& a) {
  return ((size_t)a.W * a.V * sizeof(float) + 15) / 16 * 16 + (size_t)sel_list_cap(a.V) * sizeof(uint64_t);
}
template <int MODE>
static cudaError_t beam_select_launch(const BeamSelArgs& a, cudaStream_t s, bool dependent) {
  const size_t smem = sel_smem(a);
  static size_t configured_on[MAX_DEVICES];
  size_t& configured = configured_on[device_slot()];
  if (smem > configured) {
    cudaError_t e = cudaFuncSetAttribute(k_beam_select<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    configured = smem;
  }
  return launch_ex(k_beam_select<MODE>, dim3(a.B), dim3(SEL_NT), smem, s, dependent, 1, a);
}
cudaError_t launch_beam_select(const BeamSelArgs& a, cudaStream_t s, bool dependent) {
  const int mode = sel_mode(a);
  timing_begin(s);
  const cudaError_t le = mode == 2   ? beam_select_launch<2>(a, s, dependent)
                         : mode == 1 ? beam_select_launch<1>(a, s, dependent)
                                     : beam_select_launch<0>(a, s, dependent);
  timing_end(s);
  ++g_launches;
  return le != cudaSuccess ? le : cudaGetLastError();
}

// ------------------------------------------------------------------ time-synchronous search
// One call of the time-synchronous search for one utterance per CTA (the networks and the joint
// have already run for the hypotheses of the current set A, all at frame t).  Every live slot's
// blank proposal joins the candidate set of the next frame (global arrays nb_*, at most
// W (S+1) entries, equal label strings merged by log-addition in insertion order).  In an inner
// call (mode 1) the W best label proposals (score, parent slot, token) become the next set A at
// the same frame: fresh state rows, pending network advances, back-pointers, exactly like label
// extensions of the alignment-length synchronous search.  In the frame-closing call (mode 2) no
// label is proposed and the W best candidates (score, insertion order) open frame t + 1.
constexpr int TSD_MAXC = 64;
template <int MODE>
__global__ void __launch_bounds__(SEL_NT, 1) k_tsd_select(const __grid_constant__ BeamSelArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int W = a.W, V = a.V;
  float* cand = reinterpret_cast<float*>(smem_raw);                         // [W * V] increments of the labels
  uint64_t* list = reinterpret_cast<uint64_t*>(smem_raw + ((size_t)W * V * sizeof(float) + 15) / 16 * 16);
  __shared__ float s_score[MAXW], s_blank[MAXW];
  __shared__ int s_u[MAXW], s_row[MAXW], s_last[MAXW];
  __shared__ uint64_t s_hash[MAXW], s_prev[MAXW];
  __shared__ int list_n, s_lab[MAXW];
  __shared__ int win_idx[MAXW];
  __shared__ float win_score[MAXW];
  __shared__ float c_score[TSD_MAXC];
  __shared__ int c_u[TSD_MAXC], c_last[TSD_MAXC], c_row[TSD_MAXC], c_org[TSD_MAXC], c_n;
  __shared__ uint64_t c_hash[TSD_MAXC], c_prev[TSD_MAXC];
  __shared__ float s_gmax[SEL_NT / 32][16];   // per warp: best label proposal of lanes g and g + 16

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x;
  const int base = b * W;
  const q4_beam_state& st = a.st;
  const float NEG = -INFINITY;
  const int N = a.B * W;
  const int S = st.tsd_smax;
  const int CB = W * (S + 1);
  const bool inner = a.mode == 1;
  const int RW = st.rows_per_utt;
  const bool fast = inner && MODE > 0 && !a.exact_only;   // as in k_beam_select

  pdl_wait();
  // a replayed search: its length, budget and iteration are in memory
  int T = a.T, u_max = a.u_max, iter = a.iter;
  if (a.call) {
    T = a.call->T;
    u_max = a.call->u_max;
    iter += a.call->iter;
  }
  const int step = iter % (S + 1), frame = iter / (S + 1);
  const float* const x = a.logits + (size_t)(base + warp) * V;
  float v[32];
  int my_row = -1, my_u = 0;
  float my_score = 0.0f;
  if (warp < W) {
    my_row = st.row[base + warp];
    my_u = st.u[base + warp];
    my_score = st.score[base + warp];
    if (MODE > 0 && inner) load_elems<MODE>(x, 0, V, lane, NEG, v);
  }
  if (tid < W) {
    const int o = base + tid;
    s_row[tid] = st.row[o];
    s_score[tid] = st.score[o];
    s_u[tid] = st.u[o];
    s_last[tid] = st.last_tok[o];
    s_hash[tid] = st.hash[o];
    s_prev[tid] = st.prev_hash[o];
    s_lab[tid] = inner && s_row[tid] >= 0 && s_u[tid] < u_max;   // a frame close proposes blanks only
  }
  const int cn0 = st.nb_n[b];
#pragma unroll 1
  for (int j = tid; j < cn0; j += SEL_NT) {
    const size_t o = (size_t)b * CB + j;
    c_score[j] = st.nb_score[o];
    c_u[j] = st.nb_u[o];
    c_last[j] = st.nb_last_tok[o];
    c_row[j] = st.nb_row[o];
    c_org[j] = st.nb_origin[o];
    c_hash[j] = st.nb_hash[o];
    c_prev[j] = st.nb_prev_hash[o];
  }
  if (tid == 0) {
    list_n = 0;
    c_n = cn0;
    if (b == 0) st.pend_n[iter & 1] = 0;   // the list consumed by this call is free again
  }
  if (lane < 16) s_gmax[warp][lane] = NEG;
  __syncthreads();

  // ---- proposals: one warp per slot
  const bool my_labels = inner && my_row >= 0 && my_u < u_max;
  const double s_rho = (double)my_score + (double)a.rho;
  const uint32_t skip = lane == 0 ? 1u : 0u;   // element 0 is the blank
  if (warp < W && my_row < 0 && lane == 0) s_blank[warp] = NEG;
  if (my_row >= 0) {
    const float lse = a.normalized ? 0.0f : row_lse(x, V, lane);
    if (lane == 0) s_blank[warp] = (float)((double)my_score + (double)(x[0] - lse));
    if (my_labels) {
      float best = slot_increments<MODE>(a, v, x, a.src_lp + (size_t)my_row * V, a.tgt_lp + (size_t)my_row * V, lse, skip,
                                         cand + (size_t)warp * V, lane);
      best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, 16));
      if (lane < 16) s_gmax[warp][lane] = label_score(s_rho, best);
    }
  }
  __syncthreads();

  // ---- blanks join the candidate set, in slot order (warp 0; lanes search, lane 0 updates)
  if (warp == 0) {
#pragma unroll 1
    for (int w = 0; w < W; ++w) {
      if (s_row[w] < 0) continue;             // uniform
      const int n = c_n;
      const uint64_t h = s_hash[w];
      int found = -1;
#pragma unroll 1
      for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + lane;
        const unsigned m = __ballot_sync(0xffffffffu, j < n && c_hash[j] == h);
        if (m) {
          found = j0 + __ffs(m) - 1;
          break;
        }
      }
      if (lane == 0) {
        if (found >= 0) {
          const double x = (double)c_score[found], y = (double)s_blank[w];
          c_score[found] = (float)(fmax(x, y) + log1p(exp(-fabs(x - y))));
        } else if (n < TSD_MAXC && n < CB) {
          c_score[n] = s_blank[w];
          c_u[n] = s_u[w];
          c_last[n] = s_last[w];
          c_row[n] = s_row[w];
          c_org[n] = (step << 8) | w;
          c_hash[n] = h;
          c_prev[n] = s_prev[w];
          c_n = n + 1;
        }
      }
      __syncwarp();
    }
  }
  const float bound = fast ? label_bound(s_gmax, lane) : NEG;
  __syncthreads();

  if (inner) {
    const int cap = sel_list_cap(V);
    bool exact = !fast;
    if (fast) {
      if (my_labels)
        collect_labels<MODE>(v, skip, cand + (size_t)warp * V, s_rho, bound, V, (uint32_t)warp * (uint32_t)V, list, &list_n, cap, lane);
      __syncthreads();
      exact = list_n > cap;
      if (exact) {
        __syncthreads();
        if (tid == 0) list_n = 0;
        __syncthreads();
      }
    }
    if (exact) collect_exact(cand, s_row, s_lab, s_score, a.rho, nullptr, W, V, list, &list_n, cap, warp, lane);
    rank_list(list, min(list_n, cap), W, win_idx, win_score, tid);
    __syncthreads();
    pdl_trigger();
    if (warp == 0) {
      const int nw = min(min(list_n, cap), W);
      const int row0 = b * RW;
      // rows in use: those of the current set and those the candidates refer to
      uint64_t used = 0;
#pragma unroll 1
      for (int w = 0; w < W; ++w)
        if (s_row[w] >= 0) used |= 1ull << (s_row[w] - row0);
#pragma unroll 1
      for (int j = 0; j < c_n; ++j) used |= 1ull << (c_row[j] - row0);
      const uint64_t all = RW >= 64 ? ~0ull : ((1ull << RW) - 1ull);
      uint64_t free_mask = ~used & all;
      const int s = lane;
      // the j-th winner takes the j-th free row
      int f = -1;
      {
        uint64_t m = free_mask;
#pragma unroll 1
        for (int j = 0; j <= s && j < nw; ++j) {
          f = m ? __ffsll((long long)m) - 1 : -1;
          m &= m - 1;
        }
      }
      int pbase = 0;
      if (lane == 0 && nw > 0) pbase = atomicAdd(st.pend_n + ((iter + 1) & 1), nw);
      pbase = __shfl_sync(0xffffffffu, pbase, 0);
      const size_t poff = (size_t)((iter + 1) & 1) * N;
      if (s < W) {
        const int o = base + s;
        const size_t hist = ((size_t)iter * a.B + b) * W + s;
        if (s < nw && f >= 0) {
          const int idx = win_idx[s];
          const int w = idx / V, k = idx % V;
          st.score[o] = win_score[s];
          st.t[o] = frame;
          st.u[o] = s_u[w] + 1;
          st.hash[o] = hash_mix(s_hash[w], (uint32_t)k);
          st.prev_hash[o] = s_hash[w];
          st.last_tok[o] = k;
          st.row[o] = row0 + f;
          st.adv_src[o] = s_row[w];
          st.adv_dst[o] = row0 + f;
          st.adv_tok[o] = k;
          st.pend_src[poff + pbase + s] = s_row[w];
          st.pend_dst[poff + pbase + s] = row0 + f;
          st.pend_tok[poff + pbase + s] = k;
          st.bp_parent[hist] = w;
          st.bp_token[hist] = k;
          st.bp_score[hist] = win_score[s];
        } else {
          st.row[o] = -1;
          st.adv_src[o] = -1;
          st.adv_dst[o] = -1;
          st.adv_tok[o] = -1;
          st.bp_parent[hist] = -1;
          st.bp_token[hist] = 0;
          st.bp_score[hist] = 0.0f;
        }
      }
    }
    // the candidate set goes back to memory
#pragma unroll 1
    for (int j = tid; j < c_n; j += SEL_NT) {
      const size_t o = (size_t)b * CB + j;
      st.nb_score[o] = c_score[j];
      st.nb_u[o] = c_u[j];
      st.nb_last_tok[o] = c_last[j];
      st.nb_row[o] = c_row[j];
      st.nb_origin[o] = c_org[j];
      st.nb_hash[o] = c_hash[j];
      st.nb_prev_hash[o] = c_prev[j];
    }
    if (tid == 0) st.nb_n[b] = c_n;
  } else {
    // ---- frame close: the W best candidates (score descending, then insertion order)
    pdl_trigger();
    const int n = c_n;
    const int nw = min(n, W);
    if (tid < n) {
      const float mine = c_score[tid];
      int rank = 0;
#pragma unroll 1
      for (int j = 0; j < n; ++j) rank += (c_score[j] > mine) || (c_score[j] == mine && j < tid);
      if (rank < W) {
        const int o = base + rank;
        const size_t hist = ((size_t)iter * a.B + b) * W + rank;
        st.score[o] = mine;
        st.t[o] = frame + 1;
        st.u[o] = c_u[tid];
        st.hash[o] = c_hash[tid];
        st.prev_hash[o] = c_prev[tid];
        st.last_tok[o] = c_last[tid];
        st.row[o] = c_row[tid];
        st.adv_src[o] = -1;
        st.adv_dst[o] = -1;
        st.adv_tok[o] = -1;
        st.bp_parent[hist] = c_org[tid] & 0xFF;
        st.bp_token[hist] = -1 - (c_org[tid] >> 8);
        st.bp_score[hist] = mine;
        if (frame + 1 == T) {
          st.fin_score[base + rank] = mine;
          st.fin_iter[base + rank] = iter + 1;
          st.fin_slot[base + rank] = rank;
        }
      }
    }
    if (tid >= nw && tid < W) {
      const int o = base + tid;
      const size_t hist = ((size_t)iter * a.B + b) * W + tid;
      st.row[o] = -1;
      st.adv_src[o] = -1;
      st.adv_dst[o] = -1;
      st.adv_tok[o] = -1;
      st.bp_parent[hist] = -1;
      st.bp_token[hist] = 0;
      st.bp_score[hist] = 0.0f;
    }
    if (tid == 0) {
      st.nb_n[b] = 0;
      if (frame + 1 == T) st.fin_n[b] = nw;
    }
  }
}

template <int MODE>
static cudaError_t tsd_select_launch(const BeamSelArgs& a, cudaStream_t s, bool dependent) {
  const size_t smem = sel_smem(a);
  static size_t configured_on[MAX_DEVICES];
  size_t& configured = configured_on[device_slot()];
  if (smem > configured) {
    cudaError_t e = cudaFuncSetAttribute(k_tsd_select<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    configured = smem;
  }
  return launch_ex(k_tsd_select<MODE>, dim3(a.B), dim3(SEL_NT), smem, s, dependent, 1, a);
}
cudaError_t launch_tsd_select(const BeamSelArgs& a, cudaStream_t s, bool dependent) {
  const int mode = sel_mode(a);
  timing_begin(s);
  const cudaError_t le = mode == 2   ? tsd_select_launch<2>(a, s, dependent)
                         : mode == 1 ? tsd_select_launch<1>(a, s, dependent)
                                     : tsd_select_launch<0>(a, s, dependent);
  timing_end(s);
  ++g_launches;
  return le != cudaSuccess ? le : cudaGetLastError();
}

// Trace-back of the time-synchronous search: a frame-closing call points at the call of the same
// frame whose blank created the entry; an inner call points at its parent slot of the call before.
__global__ void k_traceback_tsd(q4_beam_state st, int B, int W, int n_iters, int u_max, int32_t* tokens,
                                int32_t* lens, float* scores) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const int S1 = st.tsd_smax + 1;
  int j = -1, s = -1;
  float sc = 0.0f;
  if (st.fin_n[b] > 0) {
    sc = st.fin_score[b * W];
    j = st.fin_iter[b * W] - 1;
    s = st.fin_slot[b * W];
  } else if (n_iters > 0 && st.row[b * W] >= 0) {
    sc = st.score[b * W];
    j = n_iters - 1;
    s = 0;
  }
  int32_t* out = tokens + (size_t)b * u_max;
  int len = 0;
  while (j >= 0 && s >= 0) {
    const size_t h = ((size_t)j * B + b) * W + s;
    const int k = st.bp_token[h];
    const int par = st.bp_parent[h];
    if (j % S1 == S1 - 1) {         // frame close: jump to the set the blank was proposed from
      j = j - (S1 - 1) + (-1 - k) - 1;
    } else {
      if (k > 0 && len < u_max) out[len++] = k;
      --j;
    }
    s = par;
  }
  for (int i = 0; i < len / 2; ++i) {
    const int32_t tmp = out[i];
    out[i] = out[len - 1 - i];
    out[len - 1 - i] = tmp;
  }
  for (int i = len; i < u_max; ++i) out[i] = 0;
  lens[b] = len;
  scores[b] = sc;
}

__global__ void k_beam_init(q4_beam_state st, int B, int W) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o == 0) st.status[0] = 0;
  if (o >= B * W) return;
  const int b = o / W, s = o % W;
  const bool root = s == 0;
  st.score[o] = 0.0f;
  st.t[o] = 0;
  st.u[o] = 0;
  st.hash[o] = HASH0;
  st.prev_hash[o] = 0;
  st.last_tok[o] = 0;
  const int RW = st.rows_per_utt > 0 ? st.rows_per_utt : 2 * W;
  st.row[o] = root ? b * RW : -1;
  st.adv_src[o] = -1;                      // zero state
  st.adv_dst[o] = root ? b * RW : -1;
  st.adv_tok[o] = root ? 0 : -1;           // start symbol
  st.fin_score[o] = -INFINITY;
  st.fin_iter[o] = 0;
  st.fin_slot[o] = 0;
  if (s == 0) {
    st.fin_n[b] = 0;
    st.pend_src[b] = -1;               // pending list of iteration 0: every utterance's root,
    st.pend_dst[b] = b * RW;           // fed the start symbol from the zero state
    if (st.nb_n) st.nb_n[b] = 0;
    st.pend_tok[b] = 0;
  }
  if (o == 0) {
    st.pend_n[0] = B;
    st.pend_n[1] = 0;
  }
}

__global__ void k_search_begin(SearchCall* call, const float* e, int T, int u_max, int iter, int32_t* frozen, int B) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (frozen && i < B) frozen[i] = -1;
  if (i != 0) return;
  call->e = e;
  call->T = T;
  call->u_max = u_max;
  call->iter = iter;
  call->n_frozen = 0;
  call->arrived = 0;
}
__global__ void k_search_advance(SearchCall* call, int iters) { call->iter += iters; }
cudaError_t launch_search_begin(SearchCall* call, const float* e, int T, int u_max, int iter, int32_t* frozen, int B,
                                cudaStream_t s) {
  k_search_begin<<<frozen ? (B + 127) / 128 : 1, 128, 0, s>>>(call, e, T, u_max, iter, frozen, B);
  ++g_launches;
  return cudaGetLastError();
}
cudaError_t launch_search_advance(SearchCall* call, int iters, cudaStream_t s) {
  k_search_advance<<<1, 1, 0, s>>>(call, iters);
  ++g_launches;
  return cudaGetLastError();
}
cudaError_t launch_beam_init(const q4_beam_state& st, int B, int W, int n_iters, cudaStream_t s) {
  (void)n_iters;
  k_beam_init<<<(B * W + 255) / 256, 256, 0, s>>>(st, B, W);
  ++g_launches;
  return cudaGetLastError();
}

// One warp per utterance.  The walk from the winning slot back to the root is a chain of
// dependent look-ups; to keep it off the memory latency, the warp first copies the back-pointer
// rows of 32 consecutive iterations into shared memory (one iteration per lane, all W slots),
// then lane 0 follows the chain there.
constexpr int TB_WARPS = 4;
__global__ void __launch_bounds__(32 * TB_WARPS) k_traceback(q4_beam_state st, int B, int W, int n_iters, int u_max,
                                                             int32_t* tokens, int32_t* lens, float* scores) {
  __shared__ int s_par[TB_WARPS][32][MAXW], s_tok[TB_WARPS][32][MAXW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * TB_WARPS + warp;
  if (b >= B) return;
  int j, s;
  float sc;
  if (st.fin_n[b] > 0) {
    sc = st.fin_score[b * W];
    j = st.fin_iter[b * W] - 1;
    s = st.fin_slot[b * W];
  } else if (n_iters > 0 && st.row[b * W] >= 0) {
    sc = st.score[b * W];
    j = n_iters - 1;
    s = 0;
  } else {
    sc = 0.0f;
    j = -1;
    s = -1;
  }
  int32_t* out = tokens + (size_t)b * u_max;
  int len = 0;
  while (j >= 0 && s >= 0) {   // uniform across the warp
    const int jl = j - lane;
    if (jl >= 0) {
      const size_t h = ((size_t)jl * B + b) * W;
      for (int i = 0; i < W; ++i) {
        s_par[warp][lane][i] = st.bp_parent[h + i];
        s_tok[warp][lane][i] = st.bp_token[h + i];
      }
    }
    __syncwarp();
    if (lane == 0) {
      for (int l = 0; l < 32 && j >= 0 && s >= 0; ++l, --j) {
        const int k = s_tok[warp][l][s];
        if (k > 0 && len < u_max) out[len++] = k;
        s = s_par[warp][l][s];
      }
    }
    j = __shfl_sync(0xffffffffu, j, 0);
    s = __shfl_sync(0xffffffffu, s, 0);
    __syncwarp();
  }
  if (lane == 0) {
    for (int i = 0; i < len / 2; ++i) {
      const int32_t tmp = out[i];
      out[i] = out[len - 1 - i];
      out[len - 1 - i] = tmp;
    }
    for (int i = len; i < u_max; ++i) out[i] = 0;
    lens[b] = len;
    scores[b] = sc;
  }
}

cudaError_t launch_traceback(const q4_beam_state& st, int B, int W, int n_iters, int u_max,
                             int32_t* tokens, int32_t* lens, float* scores, cudaStream_t s) {
  if (st.nb_score)   // the state of a time-synchronous search
    k_traceback_tsd<<<(B + 63) / 64, 64, 0, s>>>(st, B, W, n_iters, u_max, tokens, lens, scores);
  else
    k_traceback<<<(B + TB_WARPS - 1) / TB_WARPS, 32 * TB_WARPS, 0, s>>>(st, B, W, n_iters, u_max, tokens, lens, scores);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace q4
