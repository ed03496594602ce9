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
// A selection is a chain of short phases on 17 warps of one SM per utterance, each bound by a memory or barrier latency
// (state and joint rows, rows of the language models, bound, list, ranking, bookkeeping).  What shortens it:
//   kernel arguments are touched before the wait (a cold line of them costs 300 to 700 clocks);
//   the rows of both language models are requested together, as soon as a slot's state row is known;
//   merges (double precision) and the candidate set of the time-synchronous search run on a warp of their own meanwhile;
//   the bound is the W-th best of 32 group maxima: some 25 proposals pass it (55 the smallest of 16), and each is scored
//   by a thread of its own;
//   the closing stores are split over three warps.
// Clocks of a selection after its wait, label iteration: 64 x 16 slots, V = 1024: 26400 before; 8 x 16 slots, V = 46: 16500.
constexpr int SEL_WARPS = SEL_NT / 32;   // one warp per slot
constexpr int SEL_THREADS = SEL_NT + 32; // and one for merges
template <typename T>
__device__ __forceinline__ void touch_arguments(const T& a) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(&a);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(T) / 4); i += 16) asm volatile("" ::"r"(w[i]));
}
// ---- proposals of one slot, by one warp.  A label's score is (float)(S + rho + inc) in double, where inc =
// log P(k) + lambda_t log P_tgt(k) - lambda_s log P_src(k) in fp32 (magnitude of tens) and S is the slot's
// running score: within a slot the score grows with inc, so proposals are compared by inc and only the few
// that matter are scored (conversions to and from double run at an eighth of the fp32 rate: scoring all
// 16 x 1024 proposals cost 1 us of the selection).
// MODE 2: NE elements per lane, V <= 32 NE, a multiple of 4, 16-byte aligned rows: element i of a lane is
// k = 128 (i / 4) + 4 lane + i % 4; MODE 1: k = lane + 32 i; a lane's values stay in registers.  MODE 0: any V, by loops
// over shared memory.
template <int MODE>
__device__ __forceinline__ int slot_elem(int i, int lane) {
  return MODE == 2 ? 128 * (i >> 2) + 4 * lane + (i & 3) : lane + 32 * i;
}
template <int MODE, int NE>
__device__ __forceinline__ uint32_t slot_valid(int V, int lane) {   // the elements of a lane that the row has
  const int n = MODE == 2 ? 4 * max((V - 4 * lane + 127) / 128, 0) : max((V - lane + 31) / 32, 0);
  return n >= 32 ? 0xFFFFFFFFu : (1u << n) - 1u;
}
template <int MODE, int NE>
__device__ __forceinline__ void load_elems(const float* p, int V, int lane, float beyond, float (&v)[NE]) {
#pragma unroll
  for (int i = 0; i < NE; i += MODE == 2 ? 4 : 1) {
    const int k = slot_elem<MODE>(i, lane);
    if (MODE == 2) {
      const float4 q = k < V ? *reinterpret_cast<const float4*>(p + k) : make_float4(beyond, beyond, beyond, beyond);
      v[i] = q.x;
      v[i + 1 < NE ? i + 1 : i] = q.y;
      v[i + 2 < NE ? i + 2 : i] = q.z;
      v[i + 3 < NE ? i + 3 : i] = q.w;
    } else {
      v[i] = k < V ? p[k] : beyond;
    }
  }
}
template <int MODE, int NE>
__device__ __forceinline__ void store_elems(float* p, int V, int lane, const float (&v)[NE]) {
#pragma unroll
  for (int i = 0; i < NE; i += MODE == 2 ? 4 : 1) {
    const int k = slot_elem<MODE>(i, lane);
    if (k >= V) continue;
    if (MODE == 2)
      *reinterpret_cast<float4*>(p + k) = make_float4(v[i], v[i + 1 < NE ? i + 1 : i], v[i + 2 < NE ? i + 2 : i], v[i + 3 < NE ? i + 3 : i]);
    else
      p[k] = v[i];
  }
}
// MODE 2: a joint row on its way to shared memory without registers, which the rows of both language models take
template <int NE>
__device__ __forceinline__ void copy_row(float* dst, const float* src, int V, int lane) {
#pragma unroll
  for (int i = 0; i < NE; i += 4) {
    const int k = slot_elem<2>(i, lane);
    if (k < V)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + k)), "l"(src + k)
                   : "memory");
  }
}
// where a warp reads its slot's joint row: the copy on its way to shared memory (waits for it), else the row itself
template <bool COPIED>
__device__ __forceinline__ const float* logits_row(const float* copy, const float* row) {
  if (!COPIED) return row;
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
  return copy;
}
// log(sum(exp)) of a row of logits, by a warp: in registers (MODE 1, -inf beyond the row) or in memory.  The same sums in
// the same order: a lane's elements 32 apart, then pairwise over the lanes.
template <int MODE, int NE>
__device__ __forceinline__ float row_lse(const float (&v)[NE], const float* x, int V, int lane) {
  float m = -INFINITY, sum = 0.0f;
  if (MODE == 1) {
#pragma unroll
    for (int i = 0; i < NE; ++i) m = fmaxf(m, v[i]);
  } else {
#pragma unroll 8
    for (int k = lane; k < V; k += 32) m = fmaxf(m, x[k]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (MODE == 1) {
#pragma unroll
    for (int i = 0; i < NE; ++i) sum += expf(v[i] - m);
  } else {
#pragma unroll 4
    for (int k = lane; k < V; k += 32) sum += expf(x[k] - m);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return m + logf(sum);
}
__device__ __forceinline__ float label_inc(const BeamSelArgs& a, float lp, float s, float t) {
  return __fmaf_rn(a.lambda_t, t, __fmaf_rn(-a.lambda_s, s, lp));
}
__device__ __forceinline__ float label_score(double s_rho, float inc) { return (float)(s_rho + (double)inc); }
// order-preserving integer of a score
__device__ __forceinline__ uint32_t ordered(float s) {
  const uint32_t b = __float_as_uint(s);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float from_ordered(uint32_t b) { return __uint_as_float((b & 0x80000000u) ? (b & 0x7FFFFFFFu) : ~b); }

// A lower bound of the W-th best label proposal: the proposals are split into 32 disjoint groups (by lane); each group's
// best is a distinct proposal, so the W-th best of the 32 bests is one.  Groups without a proposal count as -inf.  Two of
// the 32 per warp: one that fewer than W exceed lowers *bound, which so ends as the W-th best (all warps, then a barrier).
__device__ __forceinline__ void label_bound(const uint32_t (*gmax)[32], uint32_t* bound, int W, int warp, int lane) {
  uint32_t g = 0;
#pragma unroll
  for (int w = 0; w < SEL_WARPS; ++w) g = max(g, gmax[w][lane]);
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const uint32_t gx = __shfl_sync(0xffffffffu, g, 2 * warp + j);
    if (__popc(__ballot_sync(0xffffffffu, g > gx)) < W && lane == 0) atomicMin(bound, gx);
  }
}
// The labels of a slot whose score may reach `bound` go to the list as slot << 16 | label (entries beyond `cap` are only
// counted), to be scored by a thread each.  s_up: the slot's score plus rho, rounded up.
template <int MODE, int NE>
__device__ __forceinline__ void collect_labels(const float (&v)[NE], uint32_t use, float s_up, float bound, int slot,
                                               uint32_t* list, int* list_n, int cap, int lane) {
  // (float)(s_rho + inc) >= bound implies inc >= bound - s_rho - (half a rounding step of bound); the difference is off by
  // less than 1.2e-7 of the larger operand
  const float thr = __fsub_rd(__fsub_rd(bound, s_up), __fmaf_ru(5e-7f, fmaxf(fabsf(bound), fabsf(s_up)), 1e-30f));
  uint32_t hit = 0;
#pragma unroll
  for (int i = 0; i < NE; ++i) hit |= v[i] >= thr ? 1u << i : 0u;
  hit &= use;
  if (hit == 0u) return;
  int p = atomicAdd(list_n, __popc(hit));
#pragma unroll 1
  while (hit) {
    const int i = __ffs(hit) - 1;
    hit &= hit - 1;
    if (p < cap) list[p] = (uint32_t)slot << 16 | (uint32_t)slot_elem<MODE>(i, lane);
    ++p;
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

// rank of a list entry by counting; the W best are the winners (win slots were set to -1)
__device__ __forceinline__ int list_rank(const uint64_t* list, int ln, uint64_t mine) {
  int rank = 0;
#pragma unroll 8
  for (int j = 0; j < ln; ++j) rank += list[j] > mine;
  return rank;
}
// Entries of the short list: what the exact threshold can leave (W heads, each with a strided share of its slot's labels);
// smaller vocabularies have as many proposals near the bound as large ones.  By W, so that the list and its entries (12
// bytes) leave room for every W x V that a step takes (200 KB of increments): with 16 shares for every W a beam of 8 took
// 6016 labels, a beam of 1 22848 instead of 51200.
__host__ __device__ constexpr int sel_list_cap(int W, int V) { return W * ((V + 31) / 32) > 512 ? W * ((V + 31) / 32) : 512; }

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

// The closing stores of a selection by three warps: next beam (warp 0, lane s writes slot s), history (warp 1) and pending
// advances (warp 2).  A label extension takes a fresh state row: the j-th one (in slot order) the j-th row not in use.
// Up to 128 rows a step's networks have one row tile, so entries of the pending list keep their slot's place (no row: -1)
// and its length is N; beyond, utterances reserve ranges with an atomic (1000 clocks at the end of the chain).
struct SelWinners {
  int slot[MAXW], tok[MAXW];
  float score[MAXW];
};
struct SelSlots {
  float score[MAXW], blank[MAXW];   // running scores, scores of the blank proposals
  int t[MAXW], u[MAXW], row[MAXW], last[MAXW];
  int lab[MAXW];                    // the slot proposes labels
  uint64_t hash[MAXW], prev[MAXW];
  float lse[MAXW];                  // of its joint row (0 if that is normalised)
};
// The winners of a list of proposals (see collect_labels), one thread each: the score, its rank among the list's keys.
// All threads; ends behind a barrier.
__device__ __forceinline__ void rank_proposals(const BeamSelArgs& a, const SelSlots& slots, const float* cand, const uint32_t* entry,
                                               uint64_t* list, int ln, SelWinners& win, int tid) {
  uint64_t key = 0;
  uint32_t e = 0;
  float sc = 0.0f;
  if (tid < ln) {
    e = entry[tid];
    const int slot = (int)(e >> 16), k = (int)(e & 0xFFFFu);
    sc = k == 0 ? slots.blank[slot] : label_score((double)slots.score[slot] + (double)a.rho, cand[(size_t)slot * a.V + k]);
    if (sc > -INFINITY) key = make_key(sc, (uint32_t)slot * (uint32_t)a.V + (uint32_t)k);
    list[tid] = key;
  }
  __syncthreads();
  if (key != 0ull) {
    const int rank = list_rank(list, ln, key);
    if (rank < a.W) {
      win.slot[rank] = (int)(e >> 16);
      win.tok[rank] = (int)(e & 0xFFFFu);
      win.score[rank] = sc;
    }
  }
  __syncthreads();
}
// The winners of a list of keys.
__device__ __forceinline__ void rank_keys(const uint64_t* list, int ln, int W, int V, SelWinners& win, int tid) {
#pragma unroll 1
  for (int i = tid; i < ln; i += SEL_THREADS) {
    const uint64_t mine = list[i];
    const int rank = list_rank(list, ln, mine);
    if (rank >= W) continue;
    const uint32_t idx = ~(uint32_t)mine;
    win.slot[rank] = (int)(idx / (uint32_t)V);
    win.tok[rank] = (int)(idx % (uint32_t)V);
    win.score[rank] = key_score(mine);
  }
  __syncthreads();
}
__device__ __forceinline__ void write_pending(const q4_beam_state& st, int N, int W, int b, int iter, int s, bool is_label, int src,
                                              int dst, int tok, int lane) {
  const unsigned lab = __ballot_sync(0xffffffffu, is_label);
  const size_t list = (size_t)((iter + 1) & 1) * N;
  int32_t* const count = st.pend_n + ((iter + 1) & 1);
  size_t at = list + (size_t)b * W + s;
  if (N <= 128) {
    if (lane == 0 && lab != 0u) *count = N;   // every utterance with labels writes the same value
    if (s >= W) return;
    if (!is_label) src = dst = tok = -1;
  } else {
    int base = 0;
    if (lane == 0 && lab != 0u) base = atomicAdd(count, __popc(lab));
    at = list + __shfl_sync(0xffffffffu, base, 0) + __popc(lab & ((1u << s) - 1u));
    if (!is_label) return;
  }
  st.pend_src[at] = src;
  st.pend_dst[at] = dst;
  st.pend_tok[at] = tok;
}
// Rows free for label extensions, in order, into rows[] (one warp).
__device__ __forceinline__ void list_free_rows(uint64_t free_mask, int* rows, int lane) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int p = lane + 32 * h;
    if ((free_mask >> p) & 1ull) rows[__popcll(free_mask & ((1ull << p) - 1ull))] = p;
  }
  __syncwarp();
}

template <int MODE, int NE, bool LOGITS = false>
__global__ void __launch_bounds__(SEL_THREADS, 1) k_beam_select(const __grid_constant__ BeamSelArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int W = a.W, V = a.V;
  const int cap = sel_list_cap(W, V);
  uint64_t* list = reinterpret_cast<uint64_t*>(smem_raw);                   // keys of the proposals that pass the bound
  uint32_t* entry = reinterpret_cast<uint32_t*>(list + cap);
  float* cand = reinterpret_cast<float*>(entry + cap);                      // [W * V] increments of the labels
  __shared__ SelSlots s_slot;
  __shared__ SelWinners win;
  __shared__ int list_n;
  __shared__ uint32_t s_gmax[SEL_WARPS][32];   // per warp and lane: best label proposal
  __shared__ uint32_t s_bound;
  __shared__ int s_free[3][64];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x;
  const int base = b * W;
  const q4_beam_state& st = a.st;
  const float NEG = -INFINITY;
  const int N = a.B * W;
  const bool normalized = a.normalized != 0;   // `logits` holds log-probabilities already

  touch_arguments(a);
  if (tid < W) win.slot[tid] = -1;
  if (tid == 0) {
    list_n = 0;
    s_bound = 0xFFFFFFFFu;
  }
  if (warp < SEL_WARPS) s_gmax[warp][lane] = ordered(NEG);
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
  const bool mine = warp < W;
  const float* const x = a.logits + (size_t)(base + warp) * V;
  float v[NE], sv[NE], tv[NE];
  int my_row = -1, my_u = 0;
  float my_score = 0.0f, x0 = 0.0f;   // x0: the blank's entry (lane 0)
  if (mine) {
    my_row = st.row[base + warp];
    my_u = st.u[base + warp];
    my_score = st.score[base + warp];
    if (MODE == 1) load_elems<MODE>(x, V, lane, NEG, v);
    if (MODE == 2) copy_row<NE>(cand + (size_t)warp * V, x, V, lane);
    if (MODE != 1) x0 = x[0];
  }
  if (warp == SEL_WARPS && lane < W) {   // the slots' other values
    const int o = base + lane;
    const int row = st.row[o], u = st.u[o];
    s_slot.score[lane] = st.score[o];
    s_slot.t[lane] = st.t[o];
    s_slot.last[lane] = st.last_tok[o];
    s_slot.hash[lane] = st.hash[o];
    s_slot.prev[lane] = st.prev_hash[o];
    s_slot.row[lane] = row;
    s_slot.u[lane] = u;
    s_slot.lab[lane] = row >= 0 && u < u_max;
    // the list of pending advances consumed by this iteration is free again
    if (b == 0 && lane == 0) st.pend_n[iter & 1] = 0;
  }
  const bool my_labels = my_row >= 0 && my_u < u_max;
  const float* const ls = a.src_lp + (size_t)max(my_row, 0) * V;
  const float* const lt = a.tgt_lp + (size_t)max(my_row, 0) * V;
  if (MODE > 0 && my_labels) {
    load_elems<MODE>(ls, V, lane, 0.0f, sv);
    load_elems<MODE>(lt, V, lane, 0.0f, tv);
  }
  float lse = 0.0f;
  if (my_row >= 0) {
    if (!normalized) lse = row_lse<MODE>(v, logits_row<LOGITS>(cand + (size_t)warp * V, x), V, lane);
    if (lane == 0) {
      s_slot.lse[warp] = lse;
      s_slot.blank[warp] = (float)((double)my_score + (double)((MODE == 1 ? v[0] : x0) - lse));
    }
  }
  const bool any_labels = __syncthreads_or(my_labels) != 0;
  if (a.frozen && !any_labels) {   // this utterance's remaining iterations are carried out together (q4_tail.cu)
    pdl_trigger();
    if (MODE == 2) asm volatile("cp.async.wait_all;" ::: "memory");
    if (N <= 128 && tid < W) st.pend_dst[(size_t)((iter + 1) & 1) * N + base + tid] = -1;   // its place in the list, see write_pending
    if (warp == 0 && a.frozen[b] < 0) {
      int left = lane < W && s_slot.row[lane] >= 0 ? T - s_slot.t[lane] : 0;
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

  // ---- increments of the labels (one warp per slot); element 0 (blank) and labels that describe another slot's string
  // (its blank takes them in, below) do not count: lane w1 tests slot w1, the few hits are handed round the warp
  // a lower bound of the W-th best from group maxima (without labels there are blanks only, at most W)
  const bool fast = (MODE > 0 || !any_labels) && !a.exact_only;
  const double s_rho = (double)my_score + (double)a.rho;
  const float s_up = __double2float_ru(s_rho);
  uint32_t use = MODE > 0 ? slot_valid<MODE, NE>(V, lane) & ~(lane == 0 ? 1u : 0u) : 0u;
  if (my_labels) {
    const bool folds = lane < W && s_slot.row[lane] >= 0 && s_slot.u[lane] == my_u + 1 && s_slot.prev[lane] == s_slot.hash[warp];
    const int tok = folds ? s_slot.last[lane] : 0;
    unsigned hits = __ballot_sync(0xffffffffu, folds);
    if (MODE == 0) {
#pragma unroll 4
      for (int k = lane; k < V; k += 32) cand[(size_t)warp * V + k] = label_inc(a, x[k] - lse, ls[k], lt[k]);
      __syncwarp();
      if (folds) cand[(size_t)warp * V + tok] = NEG;
    } else {
#pragma unroll 1
      while (hits) {
        const int src = __ffs(hits) - 1;
        hits &= hits - 1;
        const int t = __shfl_sync(0xffffffffu, tok, src);
        if (MODE == 2 ? (t >> 2 & 31) == lane : (t & 31) == lane) use &= ~(1u << (MODE == 2 ? (t >> 7) * 4 + (t & 3) : t >> 5));
      }
      if (MODE == 2) {
        asm volatile("cp.async.wait_all;" ::: "memory");   // a lane reads what it has copied
        load_elems<MODE>(cand + (size_t)warp * V, V, lane, NEG, v);
      }
      float best = NEG;
#pragma unroll
      for (int i = 0; i < NE; ++i) {
        v[i] = label_inc(a, v[i] - lse, sv[i], tv[i]);
        best = fmaxf(best, (use >> i) & 1u ? v[i] : NEG);
      }
      store_elems<MODE>(cand + (size_t)warp * V, V, lane, v);
      s_gmax[warp][lane] = ordered(label_score(s_rho, best));
    }
  }
  if (MODE == 2) asm volatile("cp.async.wait_all;" ::: "memory");   // of slots without labels
  // ---- merge, by a warp of its own: lane w adds the label proposal (w2, k) that describes the string of its blank (at
  // most one: the slots' strings differ).  All are found first: the double-precision part takes over 1000 clocks a time.
  if (warp == SEL_WARPS) {
    int from = -1;
    if (lane < W && s_slot.row[lane] >= 0) {
      const int u = s_slot.u[lane] - 1;
      const uint64_t prev = s_slot.prev[lane];
#pragma unroll 8
      for (int w2 = 0; w2 < W; ++w2)
        if (s_slot.lab[w2] && s_slot.u[w2] == u && s_slot.hash[w2] == prev) from = w2;
    }
    if (from >= 0) {
      const int k = s_slot.last[lane];
      const size_t row = (size_t)s_slot.row[from] * V + k;
      const float inc = label_inc(a, a.logits[(size_t)(base + from) * V + k] - s_slot.lse[from], a.src_lp[row], a.tgt_lp[row]);
      const double p = (double)s_slot.blank[lane];
      const double q = (double)label_score((double)s_slot.score[from] + (double)a.rho, inc);
      s_slot.blank[lane] = (float)(fmax(p, q) + log1p(exp(-fabs(p - q))));
    }
  }
  // ---- finished hypotheses, by the same warp: blank proposals that consume the last frame
  if (warp == SEL_WARPS) {
    const bool fin = lane < W && s_slot.row[lane] >= 0 && s_slot.t[lane] + 1 == T;
    __syncwarp();
    if (__any_sync(0xffffffffu, fin) && lane == 0) {
      float* fs = st.fin_score + base;
      int* fi = st.fin_iter + base;
      int* fl = st.fin_slot + base;
      int n = st.fin_n[b];
#pragma unroll 1
      for (int w = 0; w < W; ++w) {
        if (s_slot.row[w] < 0 || s_slot.t[w] + 1 != T) continue;
        const float S = s_slot.blank[w];
        s_slot.blank[w] = NEG;
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
    __syncwarp();
  }

  // ---- the W best remaining proposals: labels that pass the bound (the warp of the blanks is not waited for before the
  // list), blanks all of them
  bool exact = !fast;
  if (fast) {
    if (warp < SEL_WARPS) {
      asm volatile("bar.sync 1, %0;" ::"n"(SEL_NT) : "memory");
      label_bound(s_gmax, &s_bound, W, warp, lane);
      asm volatile("bar.sync 1, %0;" ::"n"(SEL_NT) : "memory");
      if (MODE > 0 && my_labels) collect_labels<MODE>(v, use, s_up, from_ordered(s_bound), warp, entry, &list_n, cap, lane);
    } else if (lane < W && s_slot.row[lane] >= 0 && s_slot.blank[lane] > NEG) {
      const int p = atomicAdd(&list_n, 1);
      if (p < cap) entry[p] = (uint32_t)lane << 16;
    }
    __syncthreads();
    exact = list_n > cap;     // the bound was too loose for the list: take the exact threshold instead
  }
  if (exact) {
    __syncthreads();
    if (tid == 0) list_n = 0;
    if (MODE > 0 && my_labels) {   // labels that another slot's blank has taken in
#pragma unroll 1
      for (uint32_t gone = slot_valid<MODE, NE>(V, lane) & ~use; gone; gone &= gone - 1)
        cand[(size_t)warp * V + slot_elem<MODE>(__ffs(gone) - 1, lane)] = NEG;
    }
    __syncthreads();
    collect_exact(cand, s_slot.row, s_slot.lab, s_slot.score, a.rho, s_slot.blank, W, V, list, &list_n, cap, warp, lane);
    rank_keys(list, min(list_n, cap), W, V, win, tid);
  } else {
    rank_proposals(a, s_slot, cand, entry, list, list_n, win, tid);
  }
  pdl_trigger();   // only the bookkeeping is left: the next kernel of the stream may set itself up

  // ---- next beam, history, pending advances
  if (warp < 3) {
    const int s = lane, o = base + s;
    const int w = s < W ? win.slot[s] : -1;
    const bool live = w >= 0;
    const int k = live ? win.tok[s] : 0;
    const bool is_label = live && k != 0;
    if (warp == 1) {
      if (s < W) {
        const size_t hist = ((size_t)iter * a.B + b) * W + s;
        st.bp_parent[hist] = live ? w : -1;
        st.bp_token[hist] = live ? k : -1;
        st.bp_score[hist] = live ? win.score[s] : 0.0f;
      }
    } else {
      const int row0 = b * (st.rows_per_utt > 0 ? st.rows_per_utt : 2 * W);
      const uint32_t used = __reduce_or_sync(0xffffffffu, lane < W && s_slot.row[lane] >= 0 ? 1u << (s_slot.row[lane] - row0) : 0u);
      list_free_rows(~used & (W >= 16 ? 0xFFFFFFFFu : (1u << (2 * W)) - 1u), s_free[warp], lane);
      const unsigned lab = __ballot_sync(0xffffffffu, is_label);
      const int dst = is_label ? row0 + s_free[warp][__popc(lab & ((1u << s) - 1u))] : -1;
      const int src = is_label ? s_slot.row[w] : -1;
      if (warp == 2) {
        write_pending(st, N, W, b, iter, s, is_label, src, dst, k, lane);
      } else if (s < W) {
        if (live) {
          st.score[o] = win.score[s];
          st.t[o] = s_slot.t[w] + (is_label ? 0 : 1);
          st.u[o] = s_slot.u[w] + (is_label ? 1 : 0);
          st.hash[o] = is_label ? hash_mix(s_slot.hash[w], (uint32_t)k) : s_slot.hash[w];
          st.prev_hash[o] = is_label ? s_slot.hash[w] : s_slot.prev[w];
          st.last_tok[o] = is_label ? k : s_slot.last[w];
        }
        st.row[o] = is_label ? dst : live ? s_slot.row[w] : -1;
        st.adv_src[o] = src;
        st.adv_dst[o] = dst;
        st.adv_tok[o] = is_label ? k : -1;
      }
      if (warp == 0 && a.loop_iters && lane == 0) loop_step_end(a, iter, T + u_max);
    }
  }
}

// Which form of the kernels takes a vocabulary: registers hold up to 1024 labels of a slot, and rows are read 16 bytes at
// a time where those of all three tables can be.  A selection with joint rows that are not normalised, summed 32 elements
// apart in the shared copy / in registers that were read 4 bytes at a time: 8 x 16 slots of 1024 labels 13.9 / 17.9 us,
// 24 x 16 of 512 12.9 / 15.8, 64 x 16 of 1000 14.2 / 16.4.  A kernel of its own: without LOGITS the sums in the
// kernel of the normalised rows cost a search of 16 x 16 slots 0.8 %.
enum { SEL_ANY, SEL_64, SEL_256, SEL_1024, SEL_WIDE, SEL_WIDE_LOGITS };
static int sel_form(const BeamSelArgs& a) {
  if (a.V > 1024) return SEL_ANY;
  if (a.V <= 64) return SEL_64;
  if (a.V <= 256) return SEL_256;
  const bool wide = a.V % 4 == 0 && ((reinterpret_cast<uintptr_t>(a.logits) | reinterpret_cast<uintptr_t>(a.src_lp) |
                                      reinterpret_cast<uintptr_t>(a.tgt_lp)) & 15) == 0;
  return !wide ? SEL_1024 : a.normalized ? SEL_WIDE : SEL_WIDE_LOGITS;
}
static size_t sel_smem(const BeamSelArgs& a) {
  return (size_t)sel_list_cap(a.W, a.V) * (sizeof(uint64_t) + sizeof(uint32_t)) + (size_t)a.W * a.V * sizeof(float);
}
static cudaError_t sel_launch(void (*kern)(const BeamSelArgs), size_t (&configured_on)[MAX_DEVICES], const BeamSelArgs& a,
                              cudaStream_t s, bool dependent) {
  const size_t smem = sel_smem(a);
  size_t& configured = configured_on[device_slot()];
  if (smem > configured) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    configured = smem;
  }
  return launch_ex(kern, dim3(a.B), dim3(SEL_THREADS), smem, s, dependent, 1, a);
}
cudaError_t launch_beam_select(const BeamSelArgs& a, cudaStream_t s, bool dependent) {
  static size_t configured[6][MAX_DEVICES];
  static void (*const kern[6])(const BeamSelArgs) = {k_beam_select<0, 1>, k_beam_select<1, 2>, k_beam_select<1, 8>,
                                                     k_beam_select<1, 32>, k_beam_select<2, 32>, k_beam_select<2, 32, true>};
  const int form = sel_form(a);
  timing_begin(s);
  const cudaError_t le = sel_launch(kern[form], configured[form], a, s, dependent);
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
template <int MODE, int NE, bool LOGITS = false>
__global__ void __launch_bounds__(SEL_THREADS, 1) k_tsd_select(const __grid_constant__ BeamSelArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int W = a.W, V = a.V;
  const int cap = sel_list_cap(W, V);
  uint64_t* list = reinterpret_cast<uint64_t*>(smem_raw);                   // keys of the proposals that pass the bound
  uint32_t* entry = reinterpret_cast<uint32_t*>(list + cap);
  float* cand = reinterpret_cast<float*>(entry + cap);                      // [W * V] increments of the labels
  __shared__ SelSlots s_slot;
  __shared__ SelWinners win;
  __shared__ int list_n;
  __shared__ float c_score[TSD_MAXC];
  __shared__ int c_u[TSD_MAXC], c_last[TSD_MAXC], c_row[TSD_MAXC], c_org[TSD_MAXC], c_n;
  __shared__ uint64_t c_hash[TSD_MAXC], c_prev[TSD_MAXC];
  __shared__ uint32_t s_gmax[SEL_WARPS][32];   // per warp and lane: best label proposal
  __shared__ uint32_t s_bound;
  __shared__ int s_free[3][64];

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

  touch_arguments(a);
  if (tid < W) win.slot[tid] = -1;
  if (tid == 0) {
    list_n = 0;
    s_bound = 0xFFFFFFFFu;
  }
  if (warp < SEL_WARPS) s_gmax[warp][lane] = ordered(NEG);
  pdl_wait();
  // a replayed search: its length, budget and iteration are in memory
  int T = a.T, u_max = a.u_max, iter = a.iter;
  if (a.call) {
    T = a.call->T;
    u_max = a.call->u_max;
    iter += a.call->iter;
  }
  const int step = iter % (S + 1), frame = iter / (S + 1);
  const bool mine = warp < W;
  const float* const x = a.logits + (size_t)(base + warp) * V;
  float v[NE], sv[NE], tv[NE];
  int my_row = -1, my_u = 0;
  float my_score = 0.0f, x0 = 0.0f;   // x0: the blank's entry (lane 0)
  if (mine) {
    my_row = st.row[base + warp];
    my_u = st.u[base + warp];
    my_score = st.score[base + warp];
    if (MODE == 1) load_elems<MODE>(x, V, lane, NEG, v);
    if (MODE == 2) copy_row<NE>(cand + (size_t)warp * V, x, V, lane);
    if (MODE != 1) x0 = x[0];
  }
  if (warp == SEL_WARPS) {
    if (lane < W) {
      const int o = base + lane;
      s_slot.row[lane] = st.row[o];
      s_slot.score[lane] = st.score[o];
      s_slot.u[lane] = st.u[o];
      s_slot.last[lane] = st.last_tok[o];
      s_slot.hash[lane] = st.hash[o];
      s_slot.prev[lane] = st.prev_hash[o];
      s_slot.lab[lane] = inner && s_slot.row[lane] >= 0 && s_slot.u[lane] < u_max;   // a frame close proposes blanks only
      if (b == 0 && lane == 0) st.pend_n[iter & 1] = 0;   // the list consumed by this call is free again
    }
    const int cn0 = st.nb_n[b];
    if (lane == 0) c_n = cn0;
#pragma unroll 1
    for (int j = lane; j < cn0; j += 32) {
      const size_t o = (size_t)b * CB + j;
      c_score[j] = st.nb_score[o];
      c_u[j] = st.nb_u[o];
      c_last[j] = st.nb_last_tok[o];
      c_row[j] = st.nb_row[o];
      c_org[j] = st.nb_origin[o];
      c_hash[j] = st.nb_hash[o];
      c_prev[j] = st.nb_prev_hash[o];
    }
  }
  const bool my_labels = inner && my_row >= 0 && my_u < u_max;
  const float* const ls = a.src_lp + (size_t)max(my_row, 0) * V;
  const float* const lt = a.tgt_lp + (size_t)max(my_row, 0) * V;
  if (MODE > 0 && my_labels) {
    load_elems<MODE>(ls, V, lane, 0.0f, sv);
    load_elems<MODE>(lt, V, lane, 0.0f, tv);
  }
  float lse = 0.0f;
  if (my_row >= 0) {
    if (!a.normalized) lse = row_lse<MODE>(v, logits_row<LOGITS>(cand + (size_t)warp * V, x), V, lane);
    if (lane == 0) s_slot.lse[warp] = lse;
    if (lane == 0) s_slot.blank[warp] = (float)((double)my_score + (double)((MODE == 1 ? v[0] : x0) - lse));
  }
  __syncthreads();

  // ---- increments of the labels: one warp per slot, element 0 (blank) does not count
  const double s_rho = (double)my_score + (double)a.rho;
  const float s_up = __double2float_ru(s_rho);
  const uint32_t use = MODE > 0 ? slot_valid<MODE, NE>(V, lane) & ~(lane == 0 ? 1u : 0u) : 0u;
  if (my_labels) {
    if (MODE == 0) {
#pragma unroll 4
      for (int k = lane; k < V; k += 32) cand[(size_t)warp * V + k] = label_inc(a, x[k] - lse, ls[k], lt[k]);
    } else {
      if (MODE == 2) {
        asm volatile("cp.async.wait_all;" ::: "memory");   // a lane reads what it has copied
        load_elems<MODE>(cand + (size_t)warp * V, V, lane, NEG, v);
      }
      float best = NEG;
#pragma unroll
      for (int i = 0; i < NE; ++i) {
        v[i] = label_inc(a, v[i] - lse, sv[i], tv[i]);
        best = fmaxf(best, (use >> i) & 1u ? v[i] : NEG);
      }
      store_elems<MODE>(cand + (size_t)warp * V, V, lane, v);
      s_gmax[warp][lane] = ordered(label_score(s_rho, best));
    }
  }
  if (MODE == 2) asm volatile("cp.async.wait_all;" ::: "memory");   // of slots without labels
  // ---- blanks join the candidate set, in slot order, by a warp of its own (lanes search, lane 0 updates)
  if (warp == SEL_WARPS) {
#pragma unroll 1
    for (int w = 0; w < W; ++w) {
      if (s_slot.row[w] < 0) continue;        // uniform
      const int n = c_n;
      const uint64_t h = s_slot.hash[w];
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
          const double x = (double)c_score[found], y = (double)s_slot.blank[w];
          c_score[found] = (float)(fmax(x, y) + log1p(exp(-fabs(x - y))));
        } else if (n < TSD_MAXC && n < CB) {
          c_score[n] = s_slot.blank[w];
          c_u[n] = s_slot.u[w];
          c_last[n] = s_slot.last[w];
          c_row[n] = s_slot.row[w];
          c_org[n] = (step << 8) | w;
          c_hash[n] = h;
          c_prev[n] = s_slot.prev[w];
          c_n = n + 1;
        }
      }
      __syncwarp();
    }
  }
  if (inner) {
    bool exact = !fast;
    if (fast) {
      // (the warp with the candidate set is not waited for here)
      if (warp < SEL_WARPS) {
        asm volatile("bar.sync 1, %0;" ::"n"(SEL_NT) : "memory");
        label_bound(s_gmax, &s_bound, W, warp, lane);
        asm volatile("bar.sync 1, %0;" ::"n"(SEL_NT) : "memory");
        if (my_labels) collect_labels<MODE>(v, use, s_up, from_ordered(s_bound), warp, entry, &list_n, cap, lane);
      }
      __syncthreads();
      exact = list_n > cap;
    }
    if (exact) {
      __syncthreads();
      if (tid == 0) list_n = 0;
      __syncthreads();
      collect_exact(cand, s_slot.row, s_slot.lab, s_slot.score, a.rho, nullptr, W, V, list, &list_n, cap, warp, lane);
      rank_keys(list, min(list_n, cap), W, V, win, tid);
    } else {
      rank_proposals(a, s_slot, cand, entry, list, list_n, win, tid);
    }
    pdl_trigger();
    if (warp < 3) {
      const int s = lane, o = base + s;
      const int w = s < W ? win.slot[s] : -1;
      const int k = w >= 0 ? win.tok[s] : 0;
      // rows in use: those of the current set and those the candidates refer to
      const int row0 = b * RW;
      uint64_t used = lane < W && s_slot.row[lane] >= 0 ? 1ull << (s_slot.row[lane] - row0) : 0ull;
      for (int j = lane; j < c_n; j += 32) used |= 1ull << (c_row[j] - row0);
      used = (uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(used >> 32)) << 32 | __reduce_or_sync(0xffffffffu, (uint32_t)used);
      const uint64_t free_mask = ~used & (RW >= 64 ? ~0ull : (1ull << RW) - 1ull);
      list_free_rows(free_mask, s_free[warp], lane);
      // the j-th winner takes the j-th free row
      const bool live = w >= 0 && s < __popcll(free_mask);
      const int dst = live ? row0 + s_free[warp][s] : -1;
      const int src = live ? s_slot.row[w] : -1;
      if (warp == 1) {
        if (s < W) {
          const size_t hist = ((size_t)iter * a.B + b) * W + s;
          st.bp_parent[hist] = live ? w : -1;
          st.bp_token[hist] = k;
          st.bp_score[hist] = live ? win.score[s] : 0.0f;
        }
      } else if (warp == 2) {
        write_pending(st, N, W, b, iter, s, live, src, dst, k, lane);
      } else if (s < W) {
        if (live) {
          st.score[o] = win.score[s];
          st.t[o] = frame;
          st.u[o] = s_slot.u[w] + 1;
          st.hash[o] = hash_mix(s_slot.hash[w], (uint32_t)k);
          st.prev_hash[o] = s_slot.hash[w];
          st.last_tok[o] = k;
        }
        st.row[o] = dst;
        st.adv_src[o] = src;
        st.adv_dst[o] = dst;
        st.adv_tok[o] = live ? k : -1;
      }
    }
    // the candidate set goes back to memory
#pragma unroll 1
    for (int j = tid; j < c_n; j += SEL_THREADS) {
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
    __syncthreads();
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

cudaError_t launch_tsd_select(const BeamSelArgs& a, cudaStream_t s, bool dependent) {
  static size_t configured[6][MAX_DEVICES];
  static void (*const kern[6])(const BeamSelArgs) = {k_tsd_select<0, 1>, k_tsd_select<1, 2>, k_tsd_select<1, 8>,
                                                     k_tsd_select<1, 32>, k_tsd_select<2, 32>, k_tsd_select<2, 32, true>};
  const int form = sel_form(a);
  timing_begin(s);
  const cudaError_t le = sel_launch(kern[form], configured[form], a, s, dependent);
  timing_end(s);
  ++g_launches;
  return le != cudaSuccess ? le : cudaGetLastError();
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

__global__ void k_search_begin(SearchCall* call, const float* e, int T, int u_max, int iter, int32_t* frozen, int B, int has_loop,
                               cudaGraphConditionalHandle loop) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (frozen && i < B) frozen[i] = -1;
  if (i != 0) return;
  if (has_loop) cudaGraphSetConditional(loop, 1);
  call->e = e;
  call->T = T;
  call->u_max = u_max;
  call->iter = iter;
  call->n_frozen = 0;
  call->arrived = 0;
}
__global__ void k_search_advance(SearchCall* call, int iters) { call->iter += iters; }
cudaError_t launch_search_begin(SearchCall* call, const float* e, int T, int u_max, int iter, int32_t* frozen, int B,
                                cudaStream_t s, const cudaGraphConditionalHandle* loop) {
  k_search_begin<<<frozen ? (B + 127) / 128 : 1, 128, 0, s>>>(call, e, T, u_max, iter, frozen, B, loop != nullptr,
                                                              loop ? *loop : cudaGraphConditionalHandle());
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

// One CTA per utterance.  The walk from the winning slot back to the root is a chain of dependent look-ups; to keep it off
// the memory latency, the back-pointers of TB_ITERS consecutive iterations are copied into shared memory (one iteration per
// thread, the next block's while the present one is walked), then thread 0 follows the chain there, 40 clocks an iteration.
// 750 iterations: 168 us with 32 iterations per round trip, the strings written as they are found.
//   TSD: a frame-closing call of the time-synchronous search points at the call of the same frame whose blank created the
// entry; an inner call points at its parent slot of the call before.
constexpr int TB_ITERS = 128;
template <bool TSD>
__global__ void __launch_bounds__(TB_ITERS) k_traceback(q4_beam_state st, int B, int W, int n_iters, int u_max, int32_t* tokens,
                                                        int32_t* lens, float* scores) {
  __shared__ int s_par[TB_ITERS][MAXW + 1], s_tok[TB_ITERS][MAXW + 1];
  __shared__ int s_out[TB_ITERS];            // labels of the block, last one first
  __shared__ int s_n, s_slot, s_iter;
  const int S1 = TSD ? st.tsd_smax + 1 : 1;
  const int tid = threadIdx.x, b = blockIdx.x;
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
  int par[MAXW], tok[MAXW];
  auto fetch = [&](int top) {
    const int it = top - tid;
    const size_t h = ((size_t)max(it, 0) * B + b) * W;
#pragma unroll
    for (int i = 0; i < MAXW; ++i)
      if (i < W && it >= 0) {
        par[i] = st.bp_parent[h + i];
        tok[i] = st.bp_token[h + i];
      }
  };
  if (j >= 0) fetch(j);
  for (int top = j; j >= 0 && s >= 0; top -= TB_ITERS) {   // uniform across the block; iterations [top - TB_ITERS + 1, top]
#pragma unroll
    for (int i = 0; i < MAXW; ++i)
      if (i < W) {
        s_par[tid][i] = par[i];
        s_tok[tid][i] = tok[i];
      }
    __syncthreads();
    if (top >= TB_ITERS) fetch(top - TB_ITERS);
    if (tid == 0) {
      int n = 0;
      while (j > top - TB_ITERS && j >= 0 && s >= 0) {
        const int k = s_tok[top - j][s], p = s_par[top - j][s];
        if (TSD && j % S1 == S1 - 1) {   // frame close: to the set the blank was proposed from
          j = j - (S1 - 1) + (-1 - k) - 1;
        } else {
          if (k > 0) s_out[n++] = k;
          --j;
        }
        s = p;
      }
      s_n = n;
      s_slot = s;
      s_iter = j;
    }
    __syncthreads();
    const int n = min(s_n, u_max - len);
    if (tid < n) out[len + tid] = s_out[tid];
    len += n;
    s = s_slot;
    j = s_iter;
    __syncthreads();
  }
  // the string was found from its end (no more than u_max labels, the last ones of the walk dropped)
  for (int i = tid; i < len / 2; i += TB_ITERS) {
    const int32_t a = out[i];
    out[i] = out[len - 1 - i];
    out[len - 1 - i] = a;
  }
  for (int i = len + tid; i < u_max; i += TB_ITERS) out[i] = 0;
  if (tid == 0) {
    lens[b] = len;
    scores[b] = sc;
  }
}

cudaError_t launch_traceback(const q4_beam_state& st, int B, int W, int n_iters, int u_max,
                             int32_t* tokens, int32_t* lens, float* scores, cudaStream_t s) {
  if (st.nb_score)   // the state of a time-synchronous search
    k_traceback<true><<<B, TB_ITERS, 0, s>>>(st, B, W, n_iters, u_max, tokens, lens, scores);
  else
    k_traceback<false><<<B, TB_ITERS, 0, s>>>(st, B, W, n_iters, u_max, tokens, lens, scores);
  ++g_launches;
  return cudaGetLastError();
}

}  // namespace q4
