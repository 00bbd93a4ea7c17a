// CUDA kernels of the mask path (sm_100a): advance, plan and sweep of the mask fill, gather
// and the logits masking.  Integer work only: no tensor cores are involved anywhere.
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/fmt.h"
#include "chart_step.cuh"
#include "sweep_warp.cuh"
#include "kernels.h"

namespace fmt {

// ===================================================================================== helpers


__device__ __forceinline__ uint32_t* private_buf(const StateDev& S, uint32_t row, uint32_t which) {
  return S.arena + ((size_t)row * 3u + which) * S.chart_words;
}

// Look the finished chart `ch` up in the state cache, inserting it if it is new and there is room.
// Returns (uniformly) the cache id and the word offset of the cached copy, or id -1 when the
// chart is not in the cache and could not be added.  Wait-free: concurrent inserts of equal
// charts meet in the same hash slot and the loser adopts the winner's entry.
__device__ int32_t intern_chart(const StateDev& S, const uint32_t* ch, uint64_t& off_out) {
  const uint32_t lane = lane_id();
  off_out = 0;
  if (!S.cache_on) return -1;
  const uint32_t words = ch[CH_WORDS];
  const uint32_t hlo = ch[CH_HASH_LO];
  uint32_t slot = hlo & S.ht_mask;
  int32_t my_id = -1;
  uint64_t my_off = 0;
  const uint32_t taken = lane == 0 ? ld_acquire(&S.counters[CNT_N_STATES]) : 0u;  // (asked for together with the first probe)
  for (uint32_t probe = 0; probe < 512; ++probe) {
    uint32_t v = 0;
    if (lane == 0) v = ld_acquire(&S.ht[slot]);
    v = __shfl_sync(FULL, v, 0);
    if (v == 0) {
      if (my_id < 0) {
        unsigned long long off = 0;
        int32_t id = -1;
        if (lane == 0) {
          if (taken < S.max_states) {
            const unsigned long long need = (words + 31u) & ~31u;
            const uint32_t got = atomicAdd(&S.counters[CNT_N_STATES], 1u);
            off = atomicAdd(reinterpret_cast<unsigned long long*>(S.counters + CNT_POOL_LO), need);
            if (got < S.max_states && off + need <= S.pool_words) id = (int32_t)got;
          }
        }
        id = __shfl_sync(FULL, id, 0);
        off = __shfl_sync(FULL, off, 0);
        if (id < 0) {  // the cache is full: tell the host, which empties it before the next advance
          if (lane == 0 && S.full_flag) *reinterpret_cast<volatile uint32_t*>(S.full_flag) = 1u;
          return -1;
        }
        uint32_t* dst = S.arena + S.pool_base + off;
        for (uint32_t i = lane; i < words; i += 32) dst[i] = ch[i];
        if (lane == 0) {
          S.st_off[id] = S.pool_base + off;
          S.st_mask[id] = -1;
        }
        __syncwarp();
        __threadfence();
        my_id = id;
        my_off = S.pool_base + off;
      }
      uint32_t old = 0;
      if (lane == 0) old = atomicCAS(&S.ht[slot], 0u, (uint32_t)my_id + 1u);
      old = __shfl_sync(FULL, old, 0);
      if (old == 0) {
        off_out = my_off;
        return my_id;
      }
      v = old;  // somebody else took the slot meanwhile: compare with theirs
    }
    const uint32_t sid = v - 1u;
    if (sid >= S.max_states) return -1;
    const uint64_t poff = ld_cg64(&S.st_off[sid]);
    const uint32_t* other = S.arena + poff;
    bool same = (__ldcg(other + CH_WORDS) == words) && (__ldcg(other + CH_HASH_LO) == hlo);
    if (same)
      for (uint32_t i = lane; i < words; i += 32)
        if (__ldcg(other + i) != ch[i]) same = false;
    same = __all_sync(FULL, same);
    if (same) {
      if (lane == 0 && S.st_ref) S.st_ref[sid] = 1;  // (found again)
      off_out = poff;
      return (int32_t)sid;
    }
    slot = (slot + 1u) & S.ht_mask;
  }
  return -1;
}

// ===================================================================================== transition cache
//
// What advancing the chart with cache id `sid` by `tok` leads to, if that is known: the next chart's
// cache id, TR_REJECT, or TR_UNSET (not known).  For one lane: other blocks of the launch enter pairs meanwhile, and lanes that
// looked for themselves could see different answers.
__device__ __forceinline__ uint32_t tr_slot(const StateDev& S, unsigned long long key) {
  return (mix32((uint32_t)key) ^ mix32((uint32_t)(key >> 32) * 0x9E3779B9u)) & S.tr_mask;
}
__device__ int32_t tr_lookup(const StateDev& S, int32_t sid, uint32_t tok) {
  const unsigned long long key = ((unsigned long long)((uint32_t)sid + 1u) << 32) | tok;
  uint32_t slot = tr_slot(S, key);
  for (uint32_t probe = 0; probe < 32; ++probe) {
    // Both are under way at once.  The value is acquired: what it names (the chart's offset) was written by another block, of this
    // launch perhaps, before the value was.  (One that is not there yet, behind a key that is: the pair counts as unknown.)
    const unsigned long long k = __ldcg(S.tr_key + slot);
    const int32_t v = (int32_t)ld_acquire(reinterpret_cast<const uint32_t*>(S.tr_val + slot));
    if (k == 0ull) return TR_UNSET;
    if (k == key) return (v >= 0 || v == TR_REJECT) ? v : TR_UNSET;
    slot = (slot + 1u) & S.tr_mask;
  }
  return TR_UNSET;
}
// Remember the outcome (one lane).  The first to claim a slot for the key writes the value; a full
// neighbourhood simply leaves the pair unrecorded.
__device__ void tr_insert(const StateDev& S, int32_t sid, uint32_t tok, int32_t val) {
  const unsigned long long key = ((unsigned long long)((uint32_t)sid + 1u) << 32) | tok;
  uint32_t slot = tr_slot(S, key);
  for (uint32_t probe = 0; probe < 32; ++probe) {
    const unsigned long long k = atomicCAS(S.tr_key + slot, 0ull, key);
    if (k == 0ull) {
      asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(S.tr_val + slot), "r"(val) : "memory");
      return;
    }
    if (k == key) return;
    slot = (slot + 1u) & S.tr_mask;
  }
}

// ===================================================================================== start chart

__global__ void __launch_bounds__(32) init_kernel(GrammarDev G, StateDev S, int32_t* result) {
  extern __shared__ uint32_t smem[];
  AdvScratch s = adv_scratch(smem);
  hset_clear_all(s.w.hset, s.w.hset_mask);
  uint32_t* dst = S.arena + S.init_off;
  int r = chart_init(G, s, dst, S.chart_words);
  if (lane_id() == 0) *result = r;
}

// one warp: put the start chart into the cache and record its id
__global__ void __launch_bounds__(32) intern_init_kernel(StateDev S, int32_t* init_state) {
  uint64_t off;
  int32_t id = intern_chart(S, S.arena + S.init_off, off);
  if (lane_id() == 0) *init_state = id;
}

// rows[i] (or rows 0..n-1) go back to the start chart
__global__ void reset_kernel(const __grid_constant__ StateDev S, const uint32_t* rows, uint32_t n, const int32_t* init_state) {
  before_me();
  uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t row = rows ? rows[i] : i;
  if (row >= S.B) return;
  S.row_chart[row] = S.init_off;
  S.row_buf[row] = 255;
  S.row_state[row] = *init_state;
  S.row_flags[row] = 0;
  S.row_mask[row] = MASK_ZERO;
}

// ===================================================================================== advance

constexpr int ADV_WARPS = 4;

// A block of rows that advance gets its tables into shared memory before the kernel before it in the stream is through, behind its
// back (they do not change), and clears its scratch.  A row's steps are a chain of short look-ups, and 850 cycles each where
// an automaton's table is read from L2; the tables' way into shared memory took another 3,000 at the start.  Where the
// last calls were answered by the transition cache alone it is left until a row takes a step (64 warm rows of a schema with 90 KB
// of automata: 11.4 us a decoding step with the tables copied in vain, 10.8 without).
__device__ __forceinline__ uint32_t* advance_table_space(const StateDev& S, uint32_t* smem) { return smem + S.adv_rows * ADV_WARP_WORDS; }
template <bool HOT, bool DFA>
__device__ __forceinline__ void advance_copy_tables(const GrammarDev& G, const StateDev& S, uint32_t* smem) {
  uint32_t* dst = advance_table_space(S, smem);
  auto copy = [&](const uint32_t* src, uint32_t words) {  // (multiples of 16 bytes)
    for (uint32_t i = threadIdx.x * 4u; i < words; i += ADV_WARPS * 128u)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + i)), "l"(src + i) : "memory");
    dst += words;
  };
  if (HOT) copy(G.hot_block, G.hot_words + (S.adv_pred ? G.pred_words : 0u));
  if (DFA) copy(G.dfa_block, G.dfa_words);
}
__device__ __forceinline__ AdvScratch advance_scratch(const StateDev& S, uint32_t* smem) {
  const uint32_t warp = threadIdx.x >> 5;
  const AdvScratch s = adv_scratch(smem + (size_t)min(warp, S.adv_rows - 1u) * ADV_WARP_WORDS);
  if (warp < S.adv_rows) {
    hset_clear_all(s.w.hset, s.w.hset_mask);
    for (uint32_t i = lane_id(); i < ADV_NT_WORDS; i += 32) s.w.nt[i] = 0u;
  }
  return s;
}
// ... and the grammar as it is to be read from then on.
template <bool HOT, bool DFA>
__device__ __forceinline__ GrammarDev advance_tables(const GrammarDev& Gg, const StateDev& S, uint32_t* smem) {
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const uint32_t* at = advance_table_space(S, smem);
  GrammarDev G = Gg;
  if (HOT) G = with_hot_tables(Gg, at), at += Gg.hot_words + (S.adv_pred ? Gg.pred_words : 0u);
  if (!HOT || !S.adv_pred) G.pred = nullptr;
  if (DFA) {
    G.dfa_done = reinterpret_cast<const uint16_t*>(at + (reinterpret_cast<const uint32_t*>(Gg.dfa_done) - Gg.dfa_block));
    G.dfa_trans = reinterpret_cast<const uint16_t*>(at);
  }
  return G;
}

template <bool HOT, bool DFA>
__global__ void __launch_bounds__(ADV_WARPS * 32, 1) advance_kernel(const __grid_constant__ GrammarDev Gg,
                                                                    const __grid_constant__ StateDev S, const int32_t* tokens,
                                                                    int32_t* status) {
  extern __shared__ __align__(16) uint32_t smem[];
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  const uint32_t row = warp < S.adv_rows ? blockIdx.x * S.adv_rows + warp : 0xFFFFFFFFu;
  __shared__ uint32_t early_s;  // (the kernel before may be writing the word: one reading of it holds for the block)
  if (threadIdx.x == 0) early_s = S.adv_no - *reinterpret_cast<volatile const uint32_t*>(S.counters + CNT_ADV_STEPPED) <= 8u ? 1u : 0u;
  __syncthreads();
  const bool early = early_s != 0u;
  if (early) advance_copy_tables<HOT, DFA>(Gg, S, smem);
  AdvScratch s = advance_scratch(S, smem);
  before_me();
  const int32_t tok = row < S.B ? tokens[row] : -1;
  uint32_t flags = 0, b0 = 0, b1 = 0, own_byte = 0, held = 0;
  ChartAhead ahead;
  int32_t sid = -1;
  const uint32_t* cur = nullptr;
  auto finish = [&](int32_t st) {
    if (status && lane == 0) status[row] = st;
  };
  // What can be said without an Earley step; true: it takes one.  (Everything is asked for before anything is looked at: a row
  // that is answered by the transition cache is three reads one after the other.)
  auto first_look = [&]() -> bool {
    if (row >= S.B) return false;
    flags = S.row_flags[row];
    sid = S.cache_on ? S.row_state[row] : -1;
    cur = S.arena + S.row_chart[row];
    held = S.row_buf[row];
    if (tok == -1) return finish(FMT_OK), false;
    if (flags & ROW_FINISHED) return finish(FMT_ERR_FINISHED), false;
    if (tok < 0 || (uint32_t)tok >= Gg.V) return finish(FMT_ERR_INVALID_ARG), false;
    if (flags & ROW_BROKEN) return finish(FMT_ERR_CAPACITY), false;
    b0 = __ldg(&Gg.vocab_off[tok]), b1 = __ldg(&Gg.vocab_off[tok + 1]);
    ahead = read_ahead(cur);  // (under way while it is looked up whether they are needed)
    // has this chart been advanced by this token before?  (Section 5.2: the state cache)
    int32_t known = TR_UNSET;
    if (lane == 0 && sid >= 0 && tok != Gg.eos) known = tr_lookup(S, sid, (uint32_t)tok);
    known = __shfl_sync(FULL, known, 0);
    if (tok == Gg.eos) {
      if (!(cur[CH_FLAGS] & CHART_ACCEPTING)) return finish(FMT_ERR_TOKEN_REJECTED), false;
      if (lane == 0) S.row_flags[row] = flags | ROW_FINISHED;
      return finish(FMT_OK), false;
    }
    if (b1 == b0 || known == TR_REJECT) return finish(FMT_ERR_TOKEN_REJECTED), false;
    if (known < 0 || (uint32_t)known >= S.max_states) {
      if (lane < b1 - b0) own_byte = __ldg(&Gg.vocab_bytes[b0 + lane]);
      return true;
    }
    if (lane == 0) {
      S.row_state[row] = known;
      S.st_ref[known] = 1;
      S.row_chart[row] = ld_cg64(&S.st_off[known]);
      S.row_buf[row] = 255;
      stat_add(S, CNT_STAT_ADV, 1u);
      stat_add(S, CNT_STAT_ADV_HIT, 1u);
    }
    return finish(FMT_OK), false;
  };
  const bool steps = first_look();
  if (early) {
    if (steps && lane == 0) S.counters[CNT_ADV_STEPPED] = S.adv_no;
  } else {
    if (!__syncthreads_or(steps)) return;
    if (threadIdx.x == 0) S.counters[CNT_ADV_STEPPED] = S.adv_no;
    advance_copy_tables<HOT, DFA>(Gg, S, smem);
  }
  // the pair is entered now, its value when it is known: the answer comes while the steps are made
  unsigned long long tr_there = 1ull;
  uint32_t tr_at = 0;
  const unsigned long long tr_pair = ((unsigned long long)((uint32_t)sid + 1u) << 32) | (uint32_t)tok;
  if (steps && sid >= 0) {
    tr_at = tr_slot(S, tr_pair);
    if (lane == 0) tr_there = atomicCAS(S.tr_key + tr_at, 0ull, tr_pair);
  }
  const GrammarDev G = advance_tables<HOT, DFA>(Gg, S, smem);
  if (!steps) return;
  auto remember = [&](int32_t val) {  // (one lane)
    if (tr_there == 0ull) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(S.tr_val + tr_at), "r"(val) : "memory");
    else if (tr_there != tr_pair) tr_insert(S, sid, (uint32_t)tok, val);
  };
  // a private buffer that does not hold the current chart
  const uint32_t final_buf = (held == 0) ? 1u : 0u;
  uint32_t* dst = private_buf(S, row, final_buf);
  uint32_t* const sm_arena = s.w.cur;
  const bool staged = stage_chart(s, cur, ahead);
  const uint32_t* const src = staged ? s.stage : cur;
  const uint32_t src_words = src[CH_WORDS];
  int r;
  if (HOT && staged) r = token_steps(G, s, s.stage, own_byte, b1 - b0, dst, S.chart_words, sm_arena, ADV_CUR_CAP, nullptr);
  else r = token_step(G, s, src, own_byte, b1 - b0, dst, S.chart_words, sm_arena, ADV_CUR_CAP);
  if (r == -2) {  // the token's sets outgrew shared memory: use the row's third private buffer as the arena
    uint32_t* big = private_buf(S, row, 2);
    uint32_t cap = 32;
    while (cap * 2u <= S.chart_words) cap *= 2u;
    hset_clear_all(s.w.hset, s.w.hset_mask);
    for (uint32_t i = lane; i < ADV_NT_WORDS; i += 32) s.w.nt[i] = 0u;
    __syncwarp();
    r = (held == 2) ? -1 : token_step(G, s, src, own_byte, b1 - b0, dst, S.chart_words, big, cap);
  }
  if (r == 0) {
    if (sid >= 0 && lane == 0) remember(TR_REJECT);
    return finish(FMT_ERR_TOKEN_REJECTED);
  }
  if (r < 0) {
    if (lane == 0) {
      S.row_flags[row] = flags | ROW_BROKEN;
      atomicExch(&S.counters[CNT_ERR], 1u);
      stat_add(S, CNT_STAT_CAPERR, 1u);
    }
    return finish(FMT_ERR_CAPACITY);
  }
  const uint32_t* const made = s.out;
  const uint32_t made_words = made[CH_WORDS];
  if (lane == 0) {
    stat_add(S, CNT_STAT_ADV, 1u);
    stat_max(S, CNT_STAT_ITEMS_MAX, made[CH_ITEMS]);
    stat_max(S, CNT_STAT_SETS_MAX, made[CH_SETS]);
    stat_add(S, CNT_STAT_ADV_WORDS, src_words + made_words);
  }
  uint64_t off;
  int32_t id = intern_chart(S, made, off);
  if (id < 0 && made != dst)  // it stays the row's own
    for (uint32_t i = lane; i < made_words; i += 32) dst[i] = made[i];
  if (lane == 0) {
    if (sid >= 0 && id >= 0) remember(id);
    S.row_state[row] = id;
    if (id >= 0) {
      S.row_chart[row] = off;
      S.row_buf[row] = 255;
    } else {
      S.row_chart[row] = (uint64_t)(dst - S.arena);
      S.row_buf[row] = (uint8_t)final_buf;
    }
  }
  finish(FMT_OK);
}

// ===================================================================================== forced bytes
//
// Per row, the run of bytes that every continuation of the row's text must begin with (the keys and
// punctuation a JSON schema fixes, Section 5.1's JSON-Schema task): as long as the text is not a
// sentence and the last Earley set can scan exactly one byte, that byte is taken and the chart is
// stepped over it.  Nothing of the row changes: the sets made on the way live in the warp's scratch.
template <bool HOT, bool DFA>
__global__ void __launch_bounds__(ADV_WARPS * 32, 1) forced_kernel(const __grid_constant__ GrammarDev Gg,
                                                                   const __grid_constant__ StateDev S, uint8_t* bytes_out,
                                                                   size_t stride, uint32_t* len_out, uint32_t max_len) {
  extern __shared__ __align__(16) uint32_t smem[];
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  const uint32_t row = warp < S.adv_rows ? blockIdx.x * S.adv_rows + warp : 0xFFFFFFFFu;
  advance_copy_tables<HOT, DFA>(Gg, S, smem);
  AdvScratch s = advance_scratch(S, smem);
  before_me();
  const GrammarDev G = advance_tables<HOT, DFA>(Gg, S, smem);
  if (row >= S.B) return;
  int n = 0;
  if (!(S.row_flags[row] & (ROW_FINISHED | ROW_BROKEN)) && max_len > 0) {
    const uint32_t* cur = S.arena + S.row_chart[row];
    uint8_t* const out = bytes_out + (size_t)row * stride;
    const bool staged = stage_chart(s, cur, read_ahead(cur));
    if (HOT && staged) n = token_steps(G, s, s.stage, 0u, min(max_len, MAX_TOKEN_BYTES), nullptr, 0u, s.w.cur, ADV_CUR_CAP, out);
    else n = token_step(G, s, staged ? s.stage : cur, 0u, min(max_len, MAX_TOKEN_BYTES), nullptr, 0u, s.w.cur, ADV_CUR_CAP, out);
    if (n < 0) n = 0;
  }
  if (lane == 0) len_out[row] = (uint32_t)n;
}

// ===================================================================================== fill: plan

// One block decides, row by row, where each mask comes from: the state cache, another row of
// this call with the same chart, or a fresh computation (a "job").  (For the sweeps; the automaton's fill decides by itself.)
__global__ void __launch_bounds__(1024) plan_kernel(const __grid_constant__ GrammarDev G, const __grid_constant__ StateDev S) {
  before_me();
  __shared__ uint32_t n_jobs, n_rows, n_cached, n_shared;
  auto clear = [&](uint32_t* counters) {  // barrier and level counters: there may be fewer threads than counters
    for (uint32_t i = CNT_BAR + threadIdx.x; i < CNT_HASH_GEN; i += blockDim.x) counters[i] = 0u;
    for (uint32_t i = CNT_LEVEL_TAKEN + threadIdx.x; i <= CNT_LAST_LEVEL; i += blockDim.x) counters[i] = 0u;
  };
  clear(S.counters);
  if (threadIdx.x == 0) {
    S.counters[CNT_N_FJOBS] = 0u;
    S.counters[CNT_AUTO_ITEMS] = 0u;
    n_jobs = n_cached = n_shared = 0u;
    n_rows = S.counters[CNT_N_MASK_ROWS];
  }
  if (S.rt.on) {  // the root sweep of this fill starts from clean counters, too
    clear(S.rt.counters);
    if (threadIdx.x == 0) S.rt.counters[CNT_N_JOBS] = 0u, S.rt.counters[CNT_AUTO_ITEMS] = 0u;
  }
  __syncthreads();
  for (uint32_t row = threadIdx.x; row < S.B; row += blockDim.x) {
    const uint32_t flags = S.row_flags[row];
    const int32_t sid = S.row_state[row];
    S.row_job[row] = 0u;
    if (flags & ROW_BROKEN) {
      S.row_mask[row] = MASK_ZERO;
      continue;
    }
    if (flags & ROW_FINISHED) {
      S.row_mask[row] = MASK_EOS_ONLY;
      continue;
    }
    int32_t mrow = (int32_t)row;
    if (sid >= 0) {
      const int32_t old = atomicCAS(&S.st_mask[sid], -1, -2 - (int32_t)row);
      if (old >= 0) {  // cached
        S.st_ref[sid] = 1;  // (used again: it outlives the next emptying of the cache)
        S.row_mask[row] = old;
        atomicAdd(&n_cached, 1u);
        continue;
      }
      if (old <= -2) {  // another row of this call computes it
        S.row_mask[row] = MASK_ALIAS0 - (-2 - old);
        atomicAdd(&n_shared, 1u);
        continue;
      }
      // this row computes it, into a cache row if one is left
      const uint32_t got = atomicAdd(&n_rows, 1u);
      if (got < S.max_mask_rows) mrow = (int32_t)(S.mrow_base + got);
      else if (S.full_flag) *reinterpret_cast<volatile uint32_t*>(S.full_flag) = 1u;  // no mask row left to cache it in
    }
    S.row_mask[row] = mrow;
    S.row_job[row] = 1u;
    S.jobs[atomicAdd(&n_jobs, 1u)] = row;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    S.counters[CNT_N_JOBS] = n_jobs;
    S.counters[CNT_N_MASK_ROWS] = min(n_rows, max(S.max_mask_rows, S.counters[CNT_N_MASK_ROWS]));
    stat_add(S, CNT_STAT_FILLS, S.B);
    if (n_cached) stat_add(S, CNT_STAT_CACHED, n_cached);
    if (n_shared) stat_add(S, CNT_STAT_SHARED, n_shared);
    if (n_jobs) stat_add(S, CNT_STAT_COMPUTED, n_jobs);
  }
}

// ===================================================================================== fill: sweep
//
// For every job (a row whose mask must be computed) and every trie node the sweep answers "is the
// Earley set reached by this node's bytes non-empty?".  Sets are hash-consed per job (AutoDev): a
// transition (set, byte class) is computed once, by whichever warp needs it first, with the
// warp-cooperative scan / complete / predict of earley_device.cuh; everybody else reads it from
// the set's record.  The trie is processed one depth at a time by the whole grid, one THREAD per
// (job, node): st[node] = transition(st[parent], byte).  Reads of parent, byte and writes of st
// are coalesced because nodes are numbered breadth first.  The depths are not separated by grid
// barriers: a CTA reports the end of its part of a depth's pass, its warps then serve the queued
// transitions (tickets) while the other CTAs finish, and go on to the next depth once all have
// reported; a node whose parent's transition is still being computed waits for that transition
// alone.  The kernel is launched cooperatively so that all CTAs are resident, and every wait is a
// poll with an iteration limit that flags an error instead of hanging.

// (phase 0 of the sweep) what later phases need to know about job j, in one 16-byte record
__device__ __forceinline__ void make_job_info(const StateDev& S, uint32_t j) {
  const uint32_t row = S.jobs[j];
  const uint64_t off = S.row_chart[row];
  const uint32_t* chart = S.arena + off;
  const uint32_t acc = (chart[CH_FLAGS] & CHART_ACCEPTING) ? 0x80000000u : 0u;
  S.au.job_info[j] = make_uint4((uint32_t)off, (uint32_t)(off >> 32), chart[CH_SETS], row | acc);
}

__device__ __forceinline__ JobCtx job_ctx(const StateDev& S, uint32_t j) {
  const AutoDev& A = S.au;
  const uint4 ji = __ldcg(A.job_info + j);
  JobCtx J;
  J.row = ji.w & 0x7FFFFFFFu;
  J.accepting = (ji.w >> 31) != 0u;
  const uint32_t* chart = S.arena + (((uint64_t)ji.y << 32) | ji.x);
  J.m = ji.z;
  J.base_off = chart + CH_HDR;
  J.base_items = chart + CH_HDR + J.m + 1;
  J.recs = A.recs + (size_t)j * A.cap * A.rec_words;
  J.hash = A.hash + (size_t)j * (A.hash_mask + 1);
  J.n_states = A.n_states + j;
  J.cap = min(A.cap, (ORIGIN_SELF - 1u > J.m) ? ORIGIN_SELF - 1u - J.m : 0u);
  if (S.ctx_mode) J.cap = min(J.cap, ORIGIN_SELF - 16u - RBASE);  // a root's sets are named RBASE + id later on
  J.st = A.st + (size_t)j * A.st_stride;
  return J;
}

// What the Earley set at `node` is, given that its mark says "pending": the transition it waited
// for has been computed meanwhile.  `parent_state` is the (final) state of its parent.
__device__ __forceinline__ uint32_t settled(const GrammarDev& G, const AutoDev& A, const JobCtx& J, uint32_t parent_state,
                                            uint32_t byte) {
  const uint32_t* slot = J.recs + (size_t)parent_state * A.rec_words + AR_TRANS + G.eq_of_byte[byte];
  return ld_acquire(slot);  // (the set it names was written before the transition was published)
}

constexpr uint32_t SWEEP_PER_LANE = 4;  // trie nodes per lane and pass iteration (independent loads in flight)

__global__ void __launch_bounds__(SWEEP_WARPS * 32, 1) sweep_kernel(GrammarDev Gg, StateDev S) {
  const uint32_t n_jobs = S.counters[CNT_N_JOBS];
  if (n_jobs == 0) return;  // every CTA sees the same count: nobody is left at a barrier
  extern __shared__ __align__(16) uint32_t smem[];
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  const AutoDev& A = S.au;
  const uint32_t ntw = (2u * Gg.Nw + 7u) & ~7u;
  const uint32_t warp_words = SWEEP_CUR + SWEEP_HSET + ntw + W_CTRS + 8;
  uint32_t* mine = smem + (size_t)warp * warp_words;
  uint32_t* sm_cur = mine;
  uint32_t* sm_hset = sm_cur + SWEEP_CUR;
  uint32_t* nt = sm_hset + SWEEP_HSET;
  uint32_t* ctr = nt + ntw;
  uint32_t* tmp8 = ctr + W_CTRS;
  // ---- the small grammar tables every Earley step reads go to shared memory when they fit
  GrammarDev G = Gg;
  if (A.tables_in_smem) G = stage_hot_tables(Gg, smem + (size_t)SWEEP_WARPS * warp_words);
  uint32_t* big = S.big_scratch + ((size_t)blockIdx.x * SWEEP_WARPS + warp) * ((size_t)S.big_arena_items + S.big_hset_slots);
  const uint32_t gw = blockIdx.x * SWEEP_WARPS + warp, GW = gridDim.x * SWEEP_WARPS;
  uint32_t bar_phase = 0, pass_phase = 0;

  hset_clear_all(sm_hset, SWEEP_HSET - 1);
  for (uint32_t i = lane; i < ntw; i += 32) nt[i] = 0u;
  __syncthreads();

  // ---- the automata start with one state each: the base chart's last set
  for (uint32_t j = blockIdx.x; j < n_jobs; j += gridDim.x) {
    uint32_t* rec0 = A.recs + (size_t)j * A.cap * A.rec_words;
    for (uint32_t i = threadIdx.x; i < A.rec_words; i += blockDim.x)
      if (i < AR_SCAN || i >= AR_SCAN + 8) rec0[i] = (i >= AR_TRANS) ? T_UNKNOWN : 0u;
    if (threadIdx.x == 0) A.n_states[j] = 1u;
    if (warp == 0) {
      if (lane == 0) make_job_info(S, j);
      __syncwarp();
      __threadfence_block();
      JobCtx J = job_ctx(S, j);
      scannable_bytes(G, J.base_items + J.base_off[J.m - 1], J.base_off[J.m] - J.base_off[J.m - 1], tmp8);
      if (lane < 8) rec0[AR_SCAN + lane] = tmp8[lane];
    }
  }
  if (!grid_barrier(S, bar_phase)) return;

  SweepWarp sw{G, S};
  sw.gen = S.gen & 0xFFFFu;  // (a slot of the per-job hashes written under another generation counts as empty)
  sw.w.nt = nt;
  sw.w.ctr = ctr;
  sw.tmp8 = tmp8;
  sw.w.cur = sm_cur;
  sw.w.cur_cap = SWEEP_CUR;
  sw.w.hset = sm_hset;
  sw.w.hset_mask = SWEEP_HSET - 1;
  bool big_mode = false;

  uint32_t last_level = 0;
  uint32_t expect_req = n_jobs * Gg.n_eq;  // transitions likely to be queued at the next depth (depth 1: every byte class of every job)
  for (uint32_t L = 1; L <= G.depth; ++L) {
    const uint32_t lo = __ldg(&G.lvl_off[L]), hi = __ldg(&G.lvl_off[L + 1]);
    constexpr uint32_t CH = 32 * SWEEP_PER_LANE;
    const uint32_t nL = hi - lo, cpj = (nL + CH - 1) / CH;
    const uint32_t chunks = n_jobs * cpj;
    // ---- the pass: one thread per (job, node).  Known transitions are final; an unknown one is
    // claimed by the first thread that meets it, which queues it for the compute phase below, and
    // the node is marked pending.  A pending PARENT (marked at the previous depth, computed since)
    // is settled on the way; pending leaves are settled when the mask words are formed.
    bool any_alive = false;
    // a queued transition carries the fill's generation and the depth, so that whoever takes it can tell when it has landed
    const unsigned long long req_tag = ((unsigned long long)sw.gen << 48) | ((unsigned long long)L << 24);
    // the queue has two halves, used by odd and even depths in turn: a depth's transitions may still be
    // in the making while the next depth queues its own
    const uint32_t req_half = A.req_cap / 2u, req_base = (L & 1u) * req_half;
    for (uint32_t c = gw; c < chunks; c += GW) {
      const uint32_t j = c / cpj;
      const uint32_t first = lo + (c % cpj) * CH + lane;
      const JobCtx J = job_ctx(S, j);
      uint32_t node[SWEEP_PER_LANE], byte[SWEEP_PER_LANE], par[SWEEP_PER_LANE], ps[SWEEP_PER_LANE];
#pragma unroll
      for (uint32_t u = 0; u < SWEEP_PER_LANE; ++u) {
        node[u] = first + 32u * u;
        const bool v = node[u] < hi;
        byte[u] = v ? __ldg(&G.node_byte[node[u]]) : 0u;
        par[u] = (v && L > 1) ? __ldg(&G.parent[node[u]]) : 0u;
      }
#pragma unroll
      for (uint32_t u = 0; u < SWEEP_PER_LANE; ++u)
        ps[u] = (node[u] < hi) ? ((L == 1) ? 0u : (uint32_t)__ldcg(J.st + par[u])) : (uint32_t)ST_DEAD;  // written by other SMs: bypass L1
#pragma unroll
      for (uint32_t u = 0; u < SWEEP_PER_LANE; ++u) {
        if (node[u] >= hi) continue;
        uint32_t p_state = ps[u];
        if (p_state == ST_PENDING) {  // settle the parent first
          const uint32_t gp_state = (L == 2) ? 0u : (uint32_t)__ldcg(J.st + __ldg(&G.parent[par[u]]));
          uint32_t t2 = settled(G, A, J, gp_state, __ldg(&G.node_byte[par[u]]));
          // the transition was queued at the previous depth; the warp that drew it may still be at it
          for (uint32_t spin = 0; t2 == T_PENDING && spin < poll_limit(S, 21); ++spin) {
            __nanosleep(40);
            t2 = settled(G, A, J, gp_state, __ldg(&G.node_byte[par[u]]));
          }
          if (t2 == T_UNKNOWN || t2 == T_PENDING) {  // the wait ran out: give the row up rather than guess
            diag(S, DIAG_WAIT_VALUE);
            if (!(atomicOr(&S.row_flags[J.row], ROW_BROKEN) & ROW_BROKEN)) stat_add(S, CNT_STAT_CAPERR, 1u);
            atomicExch(&S.counters[CNT_ERR], 1u);
            p_state = ST_DEAD;
          } else {
            p_state = (t2 == T_DEAD) ? (uint32_t)ST_DEAD : (t2 == T_CTX) ? (uint32_t)ST_CTX : t2;
          }
          J.st[par[u]] = (uint16_t)p_state;
        }
        uint32_t t = T_DEAD;
        if (p_state != ST_DEAD && p_state != ST_CTX) {  // (what lies below a context-dependent node is not this sweep's business)
          // records are written by other SMs while the sweep runs: read them past L1.  A record is complete
          // before its id appears anywhere (the writer fences, then publishes the transition that names it).
          const uint32_t* rec = J.recs + (size_t)p_state * A.rec_words;
          // one 256-bit test rejects most bytes without touching the transition table
          if ((__ldcg(rec + AR_SCAN + (byte[u] >> 5)) >> (byte[u] & 31u)) & 1u) {
            uint32_t* slot = J.recs + (size_t)p_state * A.rec_words + AR_TRANS + G.eq_of_byte[byte[u]];
            t = __ldcg(slot);  // (a final value is final; anything else is read again, in order)
            if (t == T_UNKNOWN || t == T_PENDING) t = ld_acquire(slot);
            if (t == T_UNKNOWN) {
              t = atomicCAS(slot, T_UNKNOWN, T_PENDING);
              if (t == T_UNKNOWN) {  // ours to queue
                const uint32_t at = atomicAdd(&S.counters[CNT_LEVEL_REQ + L], 1u);
                if (at < req_half) {
                  A.req[req_base + at] = req_tag | ((unsigned long long)j << 32) | ((unsigned long long)p_state << 8) | byte[u];
                  t = T_PENDING;
                } else {
                  // the depth's queue is full: nobody will compute this transition.  Settle it here so that
                  // nobody waits for it: the root sweep calls it context-dependent (always a safe answer),
                  // a row's own sweep gives the row up.
                  t = S.ctx_mode ? T_CTX : T_DEAD;
                  diag(S, DIAG_QUEUE_FULL);
                  if (!S.ctx_mode) {
                    if (!(atomicOr(&S.row_flags[J.row], ROW_BROKEN) & ROW_BROKEN)) stat_add(S, CNT_STAT_CAPERR, 1u);
                    atomicExch(&S.counters[CNT_ERR], 1u);
                  }
                  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(slot), "r"(t) : "memory");
                }
              }
            }
          }
        }
        J.st[node[u]] = (t == T_PENDING) ? ST_PENDING : (t == T_DEAD) ? ST_DEAD : (t == T_CTX) ? ST_CTX : (uint16_t)t;
        any_alive |= (t != T_DEAD && t != T_CTX);
      }
    }
    __syncwarp();
    if (__any_sync(FULL, any_alive) && lane == 0) atomicOr(&S.counters[CNT_LEVEL_ALIVE + L], 1u);
    // ---- this CTA's part of the pass is done.  The queued transitions are computed WHILE the other
    // CTAs finish theirs: every warp draws a ticket and serves the transition with that number as
    // soon as it has been queued; a ticket beyond the last transition queued, once all CTAs are
    // done with the pass, is void.  One transition per warp at a time, all warps of the grid in parallel.
    if (!pass_arrive(S, pass_phase)) return;
    const uint32_t all_passed = pass_phase * gridDim.x;
    // When few transitions are being queued (as many as at the depth before, roughly), eight warps of
    // every CTA stand by for tickets and the others simply wait for them at the CTA's barrier below:
    // thousands of warps polling the same counters slow down the few that work.  A heavy fill
    // needs all hands.
    const uint32_t takers = (expect_req > 4u * gridDim.x) ? (uint32_t)SWEEP_WARPS : 8u;
    bool have_ticket = false, gave_up = false;
    uint32_t ticket = 0;
    for (uint32_t polls = 0; warp < takers;) {
      if (!have_ticket) {
        if (lane == 0) ticket = atomicAdd(&S.counters[CNT_LEVEL_TAKEN + L], 1u);
        ticket = __shfl_sync(FULL, ticket, 0);
        have_ticket = true;
      }
      uint32_t passed = 0, queued = 0;
      if (lane == 0) {  // in this order: once all have passed, the number queued is final
        passed = ld_acquire(&S.counters[CNT_PASS_DONE]) >= all_passed ? 1u : 0u;
        queued = min(ld_acquire(&S.counters[CNT_LEVEL_REQ + L]), req_half);
      }
      passed = __shfl_sync(FULL, passed, 0);
      queued = __shfl_sync(FULL, queued, 0);
      if (ticket >= queued) {
        if (passed) break;
        if (++polls > poll_limit(S, 21)) {
          gave_up = true;
          if (lane == 0) diag(S, DIAG_WAIT_QUEUE);
        }
        if ((polls & 63u) == 0u && lane == 0 && ld_acquire(&S.counters[CNT_BAR_ERR])) gave_up = true;
        gave_up = __any_sync(FULL, gave_up);
        if (gave_up) break;
        __nanosleep(polls < 16u ? 40 : 200);  // thousands of warps read the same two counters: back off
        continue;
      }
      polls = 0;
      unsigned long long rq = 0;
      if (lane == 0) {  // the entry is written right after its number was drawn: wait for it to land
        for (uint32_t spin = 0; spin < poll_limit(S, 22); ++spin) {
          rq = ld_acquire64(A.req + req_base + ticket);  // (a volatile access: a plain load may be hoisted out of the loop)
          if ((rq >> 48) == sw.gen && ((rq >> 24) & 0xFFu) == L) break;
          rq = 0;
        }
      }
      rq = __shfl_sync(FULL, rq, 0);
      have_ticket = false;
      if (rq == 0) {
        if (lane == 0) diag(S, DIAG_WAIT_QUEUE);
        gave_up = true;
        break;
      }
      const uint32_t j = (uint32_t)(rq >> 32) & 0xFFFFu, p_state = (uint32_t)(rq >> 8) & 0xFFFFu, pb = (uint32_t)rq & 0xFFu;
      const JobCtx J = job_ctx(S, j);
      uint32_t r = sw.compute(J, p_state, pb, !big_mode);
      if (r == T_FAIL && !big_mode) {  // a set outgrew the shared-memory scratch: use the large area from now on
        big_mode = true;
        hset_clear_all(sw.w.hset, sw.w.hset_mask);
        clear_nt(G, sw.w);
        sw.w.cur = big;
        sw.w.cur_cap = S.big_arena_items;
        sw.w.hset = big + S.big_arena_items;
        sw.w.hset_mask = S.big_hset_slots - 1;
        if (lane == 0) stat_add(S, CNT_STAT_BIG, 1u);
        r = sw.compute(J, p_state, pb, false);
      }
      if (r == T_FAIL) {  // a capacity was exceeded: the row's mask cannot be trusted
        hset_clear_all(sw.w.hset, sw.w.hset_mask);
        clear_nt(G, sw.w);
        if (lane == 0) {
          diag(S, DIAG_SET_SCRATCH);
          uint32_t* slot = J.recs + (size_t)p_state * A.rec_words + AR_TRANS + G.eq_of_byte[pb];
          if (S.ctx_mode) {  // the root sweep leaves what it cannot hold to the rows' own walks
            atomicExch(slot, T_CTX);
          } else {
            if (!(atomicOr(&S.row_flags[J.row], ROW_BROKEN) & ROW_BROKEN)) stat_add(S, CNT_STAT_CAPERR, 1u);
            atomicExch(&S.counters[CNT_ERR], 1u);
            atomicExch(slot, T_DEAD);  // lets the sweep go on
          }
        }
      }
    }
    if (gave_up && lane == 0) atomicExch(&S.counters[CNT_BAR_ERR], 1u);  // cannot happen short of a fault elsewhere
    // all CTAs have passed this depth: how it went is read once per CTA, so that all its warps agree
    // (The next depth's pass starts at once: a node whose parent waits for a transition that is still
    // being computed waits for that one transition, see above.)
    __shared__ uint32_t lvl_s[3];
    __syncthreads();
    if (threadIdx.x == 0) {
      lvl_s[0] = ld_acquire(&S.counters[CNT_LEVEL_ALIVE + L]);
      lvl_s[1] = ld_acquire(&S.counters[CNT_BAR_ERR]);
      lvl_s[2] = ld_acquire(&S.counters[CNT_LEVEL_REQ + L]);
    }
    __syncthreads();
    const bool alive = lvl_s[0] != 0u;
    if (lvl_s[1]) return;
    expect_req = lvl_s[2];
    last_level = L;
    if (!alive) break;  // nothing survives this depth in any job
  }
  // All CTAs have passed the last depth.  Transitions queued there may still be in the making: a
  // leaf that waits for one waits for it below, so no barrier is needed here either.
  {
    uint32_t abandoned = 0;
    if (lane == 0) abandoned = ld_acquire(&S.counters[CNT_BAR_ERR]);
    if (__shfl_sync(FULL, abandoned, 0) != 0u) return;  // the rows are marked broken when the masks are published
  }
  if (big_mode) hset_clear_all(sw.w.hset, sw.w.hset_mask);
  if (lane == 0 && (sw.n_computed | sw.n_created)) {
    stat_add(S, CNT_STAT_TRANS, sw.n_computed);
    stat_add(S, CNT_STAT_LOCAL, sw.n_created);
    stat_add64(S, CNT_STAT_STEP_CYCLES, sw.cycles);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) S.counters[CNT_LAST_LEVEL] = last_level;

  // ---- mask words: 32 tokens per warp pass, one ballot per word (token t is valid iff the node
  // where its bytes end was reached alive; EOS iff the chart is accepting)
  const uint32_t Wm = G.Wm;
  constexpr uint32_t MW = 6;  // mask words per warp and iteration: their loads are in flight together
  // nodes are numbered breadth first: a node was visited iff it comes before the first node of depth last_level + 1
  const uint32_t visited_end = __ldg(&G.lvl_off[last_level + 1]);
  for (uint32_t c0 = gw; c0 < n_jobs * Wm; c0 += MW * GW) {
    uint32_t node[MW], s_[MW], dst[MW];
    bool valid[MW], eos_ok[MW];
#pragma unroll
    for (uint32_t u = 0; u < MW; ++u) {
      const uint32_t c = c0 + u * GW;
      valid[u] = c < n_jobs * Wm;
      const uint32_t tok = (c % Wm) * 32 + lane;
      node[u] = (valid[u] && tok < G.V) ? __ldg(&G.tok_node[tok]) : 0xFFFFFFFEu;
      // where the word goes (needed last, asked for first: one lane, off the chain of the loads below)
      dst[u] = (valid[u] && lane == 0) ? (uint32_t)S.row_mask[__ldcg(A.job_info + c / Wm).w & 0x7FFFFFFFu] : 0u;
    }
#pragma unroll
    for (uint32_t u = 0; u < MW; ++u) {
      const uint32_t c = c0 + u * GW;
      s_[u] = ST_DEAD;
      eos_ok[u] = false;
      if (node[u] == 0xFFFFFFFFu) {  // a token without bytes: only EOS can be valid
        const uint32_t tok = (c % Wm) * 32 + lane;
        eos_ok[u] = ((int32_t)tok == G.eos) && !S.ctx_mode && job_ctx(S, c / Wm).accepting;
      } else if (node[u] < visited_end) {
        s_[u] = __ldcg(A.st + (size_t)(c / Wm) * A.st_stride + node[u]);
      }
    }
#pragma unroll
    for (uint32_t u = 0; u < MW; ++u) {
      if (!valid[u]) continue;  // (uniform)
      const uint32_t c = c0 + u * GW;
      const uint32_t j = c / Wm, wd = c % Wm;
      uint32_t s = s_[u];
      if (__any_sync(FULL, s == ST_PENDING)) {  // leaves that waited for a transition: their parents are final by now
        const JobCtx J = job_ctx(S, j);
        if (s == ST_PENDING) {
          const uint32_t p = __ldg(&G.parent[node[u]]);
          const uint32_t p_state = (p == 0) ? 0u : (uint32_t)__ldcg(J.st + p);
          uint32_t t2 = (p_state == ST_DEAD || p_state == ST_CTX || p_state == ST_PENDING) ? T_DEAD : settled(G, A, J, p_state, __ldg(&G.node_byte[node[u]]));
          for (uint32_t spin = 0; t2 == T_PENDING && spin < poll_limit(S, 21); ++spin) {  // some warp is still at it
            __nanosleep(40);
            t2 = settled(G, A, J, p_state, __ldg(&G.node_byte[node[u]]));
          }
          if (t2 == T_UNKNOWN || t2 == T_PENDING || p_state == ST_PENDING) {
            diag(S, DIAG_WAIT_VALUE);
            if (!(atomicOr(&S.row_flags[J.row], ROW_BROKEN) & ROW_BROKEN)) stat_add(S, CNT_STAT_CAPERR, 1u);
            s = ST_DEAD;
          } else {
            s = (t2 == T_DEAD) ? (uint32_t)ST_DEAD : (t2 == T_CTX) ? (uint32_t)ST_CTX : t2;
          }
          if (S.ctx_mode) J.st[node[u]] = (uint16_t)s;  // the frontier is collected from st afterwards
        }
      }
      const uint32_t word = __ballot_sync(FULL, (s != ST_DEAD && s != ST_CTX) || eos_ok[u]);
      if (lane == 0) S.mask_rows[(size_t)dst[u] * Wm + wd] = word;
    }
  }
}

// The mask row of a row after a fill.  A fill that was given up (a bounded wait ran out) hands out all-zero masks, never a guess;
// the rows themselves are fine and the next fill computes them afresh.
__device__ __forceinline__ int32_t resolve_mask_row(const StateDev& S, uint32_t row) {
  int32_t r = S.row_mask[row];
  const bool aborted = S.counters[CNT_BAR_ERR] != 0u;
  if ((S.row_flags[row] & ROW_BROKEN) || (aborted && S.row_job[row])) return MASK_ZERO;
  if (r <= MASK_ALIAS0) {  // the mask another row of this call computed: not to be used if that row broke
    const uint32_t other = (uint32_t)(MASK_ALIAS0 - r);
    if (aborted || (S.row_flags[other] & ROW_BROKEN)) return MASK_ZERO;
    r = S.row_mask[other];
  }
  return r;
}
// (one thread per row, in the kernel that reads the masks) A mask computed in this call becomes the cache's, or its claim is
// released: when the row had no cache row, or broke, or the fill was given up.
__device__ __forceinline__ void publish_row(const StateDev& S, uint32_t row) {
  if (!S.row_job[row]) return;
  const bool aborted = S.counters[CNT_BAR_ERR] != 0u;
  const int32_t sid = S.row_state[row], mrow = S.row_mask[row];
  if (sid >= 0) S.st_mask[sid] = (!(S.row_flags[row] & ROW_BROKEN) && !aborted && mrow >= (int32_t)S.B) ? mrow : -1;
  if (aborted && !S.af.on && row == S.jobs[0]) stat_add(S, CNT_STAT_ABORTS, 1u);
}
// (one thread of that kernel) The automaton's fill counts from zero again, and the rows that it gives up have the whole item pool.
__device__ __forceinline__ void fill_is_through(const StateDev& S) {
  if (!S.af.on) return;
  S.counters[CNT_AF_TICKET] = S.counters[CNT_AF_GIVEN] = S.counters[CNT_AF_GIVEN_TAKEN] = S.counters[CNT_AUTO_ITEMS] = 0u;
  atomicAdd(&S.counters[CNT_AF_NO], 1u);  // (nothing waits for it)
}

// mask_out[row][w] for every row
__global__ void gather_kernel(const __grid_constant__ GrammarDev G, const __grid_constant__ StateDev S, uint32_t* out,
                              size_t stride_words) {
  before_me();
  const uint32_t row = blockIdx.y;
  if (blockIdx.x == 0 && threadIdx.x == 0) publish_row(S, row);
  if (blockIdx.x == 0 && row == 0u && threadIdx.x == 32) fill_is_through(S);
  const int32_t r = resolve_mask_row(S, row);
  const uint32_t* src = (r >= 0) ? S.mask_rows + (size_t)r * G.Wm : nullptr;
  uint32_t* dst = out + (size_t)row * stride_words;
  for (size_t i = blockIdx.x * blockDim.x + threadIdx.x; i < stride_words; i += (size_t)gridDim.x * blockDim.x) {
    uint32_t v = 0;
    if (i < G.Wm) {
      if (src) v = src[i];
      else if (r == MASK_EOS_ONLY && G.eos >= 0 && i == ((uint32_t)G.eos >> 5)) v = 1u << ((uint32_t)G.eos & 31u);
    }
    dst[i] = v;
  }
}

// logits[t] = -inf where bit t is 0, for one row.  A row is taken in units of 32 bytes (16 bf16 or 8 fp32 logits), which begin
// at the first 32-byte boundary of the row, wherever in the mask that is: the unit's bits are cut out of two mask words.  Units that
// are all valid are not touched, units that are all invalid are stored without being read.  What is left is bound by
// DRAM, so a thread asks for the mask words of all its units, then for all their logits, before it stores anything.
// 256 rows of 128,256 bf16 logits, four of ten rows half valid (95 MB to move): 22.5 us a launch; one group of 16 bytes after the
// other took 27.9.  Rows that do not begin on 16 bytes were written logit by logit: 48 rows of 50,001, 22 -> 5.2 us.
constexpr uint32_t APPLY_UNITS = 2;  // units per thread (1, 2, 3, 4: 22.5, 22.5, 24.5, 26.5 us for the launch above)
struct Unit {
  uint32_t v[8];
};
__device__ __forceinline__ Unit load_unit(const void* p) {
  Unit u;
  asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(u.v[0]), "=r"(u.v[1]), "=r"(u.v[2]), "=r"(u.v[3]), "=r"(u.v[4]), "=r"(u.v[5]), "=r"(u.v[6]), "=r"(u.v[7])
               : "l"(p));
  return u;
}
__device__ __forceinline__ void store_unit(void* p, const Unit& u) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(u.v[0]), "r"(u.v[1]), "r"(u.v[2]),
               "r"(u.v[3]), "r"(u.v[4]), "r"(u.v[5]), "r"(u.v[6]), "r"(u.v[7])
               : "memory");
}

template <typename T>
__device__ __forceinline__ void apply_row(const uint32_t* mask_row, int32_t special, int32_t eos, T* logits, uint32_t V,
                                          uint32_t* mask_out) {
  constexpr uint32_t PER = 32u / sizeof(T), ALL = (1u << PER) - 1u;  // logits of a unit
  const uint32_t nthreads = gridDim.x * blockDim.x;
  const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t words = (V + 31) / 32;
  const T neg = sizeof(T) == 2 ? (T)0xFF80u : (T)0xFF800000u;
  auto word_at = [&](uint32_t wd) -> uint32_t {
    if (mask_row) return __ldg(&mask_row[wd]);
    return (special == MASK_EOS_ONLY && eos >= 0 && wd == ((uint32_t)eos >> 5)) ? 1u << ((uint32_t)eos & 31u) : 0u;
  };
  if (mask_out)
    for (uint32_t wd = tid; wd < words; wd += nthreads) mask_out[wd] = word_at(wd);
  const uint32_t head = min(V, (uint32_t)((0u - reinterpret_cast<uintptr_t>(logits)) & 31u) / (uint32_t)sizeof(T));
  const uint32_t units = (V - head) / PER;
  for (uint32_t base = tid; base < units; base += APPLY_UNITS * nthreads) {
    uint32_t bits[APPLY_UNITS];
#pragma unroll
    for (uint32_t u = 0; u < APPLY_UNITS; ++u) {
      const uint32_t t = head + (base + u * nthreads) * PER, sh = t & 31u;
      bits[u] = ALL;
      if (base + u * nthreads < units) {
        const uint32_t lo = word_at(t >> 5), hi = sh + PER > 32u ? word_at((t >> 5) + 1u) : 0u;  // (the unit ends before V: the word is there)
        bits[u] = __funnelshift_r(lo, hi, sh) & ALL;
      }
    }
    Unit x[APPLY_UNITS];
#pragma unroll
    for (uint32_t u = 0; u < APPLY_UNITS; ++u)
      if (bits[u] != 0u && bits[u] != ALL) x[u] = load_unit(logits + head + (size_t)(base + u * nthreads) * PER);
#pragma unroll
    for (uint32_t u = 0; u < APPLY_UNITS; ++u) {
      if (bits[u] == ALL) continue;
#pragma unroll
      for (uint32_t i = 0; i < 8u; ++i) {
        if (sizeof(T) == 2) {
          const uint32_t keep = ((bits[u] >> (2u * i)) & 1u ? 0x0000FFFFu : 0u) | ((bits[u] >> (2u * i + 1u)) & 1u ? 0xFFFF0000u : 0u);
          x[u].v[i] = bits[u] == 0u ? 0xFF80FF80u : (x[u].v[i] & keep) | (0xFF80FF80u & ~keep);
        } else {
          x[u].v[i] = (bits[u] >> i) & 1u ? x[u].v[i] : 0xFF800000u;
        }
      }
      store_unit(logits + head + (size_t)(base + u * nthreads) * PER, x[u]);
    }
  }
  const uint32_t tail = head + units * PER;  // the logits before the first unit and after the last
  if (tid < head + (V - tail)) {
    const uint32_t t = tid < head ? tid : tail + (tid - head);
    if (!((word_at(t >> 5) >> (t & 31u)) & 1u)) logits[t] = neg;
  }
}

template <typename T>
__global__ void apply_kernel(const uint32_t* mask, size_t stride_words, T* logits, uint32_t V, size_t row_stride) {
  before_me();
  const uint32_t row = blockIdx.y;
  apply_row<T>(mask + (size_t)row * stride_words, 0, -1, logits + (size_t)row * row_stride, V, nullptr);
}

template <typename T>
__global__ void gather_apply_kernel(const __grid_constant__ GrammarDev G, const __grid_constant__ StateDev S, T* logits,
                                    size_t row_stride, uint32_t* mask_out, size_t stride_words) {
  before_me();
  const uint32_t row = blockIdx.y;
  if (blockIdx.x == 0 && threadIdx.x == 0) publish_row(S, row);
  if (blockIdx.x == 0 && row == 0u && threadIdx.x == 32) fill_is_through(S);
  const int32_t r = resolve_mask_row(S, row);
  const uint32_t* src = (r >= 0) ? S.mask_rows + (size_t)r * G.Wm : nullptr;
  uint32_t* mo = mask_out ? mask_out + (size_t)row * stride_words : nullptr;
  apply_row<T>(src, r, G.eos, logits + (size_t)row * row_stride, G.V, mo);
  if (mo)  // padding words beyond ceil(V/32)
    for (size_t i = G.Wm + blockIdx.x * blockDim.x + threadIdx.x; i < stride_words; i += (size_t)gridDim.x * blockDim.x)
      mo[i] = 0u;
}

// ===================================================================================== cache clear, query

// Step 1 of a cache clear: rows whose chart lives in the pool copy it to private buffer 0.
__global__ void evacuate_kernel(StateDev S) {
  const uint32_t row = blockIdx.x;
  if (row >= S.B) return;
  const uint64_t off = S.row_chart[row];
  __syncthreads();
  if (off >= S.pool_lo) {
    const uint32_t* src = S.arena + off;
    uint32_t* dst = private_buf(S, row, 0);
    const uint32_t words = src[CH_WORDS];
    for (uint32_t i = threadIdx.x; i < words; i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    if (threadIdx.x == 0) {
      S.row_chart[row] = (uint64_t)(dst - S.arena);
      S.row_buf[row] = 0;
    }
  }
  if (threadIdx.x == 0) S.row_state[row] = -1;
}
// Step 3: the start chart (block B) and every row's chart go back into the now empty cache.
__global__ void __launch_bounds__(32) reintern_kernel(StateDev S, int32_t* init_state) {
  const uint32_t row = blockIdx.x;
  uint64_t off;
  if (row == S.B) {
    int32_t id = intern_chart(S, S.arena + S.init_off, off);
    if (lane_id() == 0) *init_state = id;
    return;
  }
  if (S.row_chart[row] == S.init_off) return;  // fixed up by the caller's second pass
  const uint32_t* ch = S.arena + S.row_chart[row];
  int32_t id = intern_chart(S, ch, off);
  if (lane_id() == 0 && id >= 0) {
    S.row_state[row] = id;
    S.row_chart[row] = off;
    S.row_buf[row] = 255;
  }
}
// Step 4: rows still at the start chart take the start chart's new id.
__global__ void fix_init_rows_kernel(StateDev S, const int32_t* init_state) {
  const uint32_t row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row < S.B && S.row_chart[row] == S.init_off) S.row_state[row] = *init_state;
}

// Emptying the cache with survivors (see fmt_state_create's cache_keep_when_full): `Old` is the cache as it
// was - its charts, mask rows and tables are still intact in the other half of the storage -, S the emptied
// one.  Every entry of Old that was found again after it was made is entered into S, with its mask row.
__global__ void __launch_bounds__(32) survivors_kernel(GrammarDev G, StateDev Old, StateDev S, const uint32_t* old_count) {
  const uint32_t id = blockIdx.x * gridDim.y + blockIdx.y;
  if (id >= min(*old_count, Old.max_states) || !Old.st_ref[id]) return;
  const uint32_t lane = lane_id();
  uint64_t off;
  const int32_t nid = intern_chart(S, Old.arena + Old.st_off[id], off);
  if (nid < 0) return;  // no room: it goes after all
  const int32_t orow = Old.st_mask[id];
  if (orow < (int32_t)Old.B) return;  // no mask was kept for it
  uint32_t nrow = 0;
  if (lane == 0) {
    nrow = 0xFFFFFFFFu;
    if (S.st_mask[nid] == -1 && ld_acquire(&S.counters[CNT_N_MASK_ROWS]) < S.max_mask_rows) {
      const uint32_t got = atomicAdd(&S.counters[CNT_N_MASK_ROWS], 1u);
      if (got < S.max_mask_rows) nrow = S.mrow_base + got;
    }
  }
  nrow = __shfl_sync(FULL, nrow, 0);
  if (nrow == 0xFFFFFFFFu) return;
  const uint32_t* src = Old.mask_rows + (size_t)orow * G.Wm;
  uint32_t* dst = S.mask_rows + (size_t)nrow * G.Wm;
  for (uint32_t i = lane; i < G.Wm; i += 32) dst[i] = src[i];
  __syncwarp();
  if (lane == 0) S.st_mask[nid] = (int32_t)nrow;
}

__global__ void query_kernel(StateDev S, uint8_t* accepting, uint8_t* finished, uint32_t* n_sets, uint32_t* n_items,
                             int32_t* state_id) {
  const uint32_t row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= S.B) return;
  const uint32_t* ch = S.arena + S.row_chart[row];
  accepting[row] = (ch[CH_FLAGS] & CHART_ACCEPTING) ? 1 : 0;
  finished[row] = (S.row_flags[row] & ROW_FINISHED) ? 1 : ((S.row_flags[row] & ROW_BROKEN) ? 2 : 0);
  n_sets[row] = ch[CH_SETS];
  n_items[row] = ch[CH_ITEMS];
  state_id[row] = S.row_state[row];
}

// ===================================================================================== launchers

constexpr size_t ADV_SMEM_LIMIT = 226 * 1024, ADV_SMEM_SM = 228 * 1024;  // dynamic shared memory of a block, shared memory of an SM

static inline cudaError_t opt_in_smem(const void* fn, size_t bytes) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

static size_t adv_smem_bytes(const GrammarDev& G, const StateDev& S) {
  const uint32_t tables = G.hot_words * 4u <= HOT_TABLE_BYTES ? G.hot_words + (S.adv_pred ? G.pred_words : 0u) : 0u;
  return ((size_t)S.adv_rows * ADV_WARP_WORDS + tables + (S.adv_dfa ? G.dfa_words : 0u)) * 4;
}
// One row to a block as long as all rows run at once: a block then has room for its grammar's automata (JSON 6 KB, a schema of
// twelve members 60 KB).  Else two or four, with the automata if they fit.
void advance_layout(const GrammarDev& G, uint32_t rows, uint32_t sms, StateDev& S) {
  for (S.adv_rows = 1;; S.adv_rows *= 2) {
    S.adv_pred = 0;
    S.adv_dfa = G.dfa_words && G.hot_words * 4u <= HOT_TABLE_BYTES ? 1u : 0u;
    if (S.adv_dfa && adv_smem_bytes(G, S) > ADV_SMEM_LIMIT) S.adv_dfa = 0;
    S.adv_pred = 1u;
    if (adv_smem_bytes(G, S) > ADV_SMEM_LIMIT) S.adv_pred = 0;
    const uint64_t blocks = (uint64_t)sms * (ADV_SMEM_SM / (adv_smem_bytes(G, S) + 1024));
    if (S.adv_rows == (uint32_t)ADV_WARPS || blocks * S.adv_rows >= rows) return;
  }
}
static_assert(ADV_WARPS * ADV_WARP_WORDS * 4 + HOT_TABLE_BYTES <= ADV_SMEM_LIMIT, "a block of so many rows fits without automata");
static size_t init_smem_bytes() { return (size_t)ADV_WARP_WORDS * 4; }
// Dynamic shared memory of the sweep for a grammar: per-warp scratch plus, if they fit the
// budget, the item-info / byte-class / byte-class-number tables.
constexpr uint32_t SWEEP_SMEM_LIMIT = 224 * 1024;  // what the sweep kernels opt in to
void sweep_layout(const GrammarDev& G, uint32_t* smem_bytes, uint32_t* tables_in_smem) {
  const uint32_t ntw = (2u * G.Nw + 7u) & ~7u;
  const uint32_t warp_words = SWEEP_CUR + SWEEP_HSET + ntw + W_CTRS + 8;
  uint32_t bytes = SWEEP_WARPS * warp_words * 4u;
  const uint32_t tab = G.hot_words * 4u;
  *tables_in_smem = (tab <= HOT_TABLE_BYTES && bytes + tab <= SWEEP_SMEM_LIMIT) ? 1u : 0u;
  if (*tables_in_smem) bytes += tab;
  *smem_bytes = bytes;
}
int sweep_warps() { return SWEEP_WARPS; }

cudaError_t configure_kernels() {
  cudaError_t e;
  if ((e = opt_in_smem((const void*)init_kernel, init_smem_bytes())) != cudaSuccess) return e;
  const void* const advancing[] = {(const void*)advance_kernel<false, false>, (const void*)advance_kernel<true, false>, (const void*)advance_kernel<true, true>,
                                   (const void*)forced_kernel<false, false>, (const void*)forced_kernel<true, false>, (const void*)forced_kernel<true, true>};
  for (const void* f : advancing)
    if ((e = opt_in_smem(f, ADV_SMEM_LIMIT)) != cudaSuccess) return e;
  if ((e = opt_in_smem((const void*)sweep_kernel, SWEEP_SMEM_LIMIT)) != cudaSuccess) return e;
  if ((e = configure_automaton_fill()) != cudaSuccess) return e;
  return configure_walk_kernels();
}

cudaError_t sweep_blocks_per_sm(int* out, uint32_t smem_bytes) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, sweep_kernel, SWEEP_WARPS * 32, smem_bytes);
}

void launch_init(const GrammarDev& G, const StateDev& S, int32_t* result_dev, cudaStream_t st) {
  init_kernel<<<1, 32, init_smem_bytes(), st>>>(G, S, result_dev);
}
void launch_intern_init(const StateDev& S, int32_t* init_state_dev, cudaStream_t st) {
  intern_init_kernel<<<1, 32, 0, st>>>(S, init_state_dev);
}
void launch_reset(const StateDev& S, const uint32_t* rows_dev, uint32_t n, const int32_t* init_state_dev, cudaStream_t st) {
  if (n == 0) return;
  launch_overlapped(reset_kernel, dim3((n + 127) / 128), dim3(128), 0, st, S, rows_dev, n, init_state_dev);
}
void launch_forced(const GrammarDev& G, const StateDev& S, uint8_t* bytes_out, size_t stride, uint32_t* len_out,
                   uint32_t max_len, cudaStream_t st) {
  const auto kernel = G.hot_words * 4u > HOT_TABLE_BYTES ? forced_kernel<false, false> : S.adv_dfa ? forced_kernel<true, true> : forced_kernel<true, false>;
  launch_overlapped(kernel, dim3((S.B + S.adv_rows - 1) / S.adv_rows), dim3(ADV_WARPS * 32), adv_smem_bytes(G, S), st, G, S, bytes_out,
                    stride, len_out, max_len);
}
void launch_advance(const GrammarDev& G, const StateDev& S, const int32_t* tokens, int32_t* status, cudaStream_t st) {
  const auto kernel = G.hot_words * 4u > HOT_TABLE_BYTES ? advance_kernel<false, false> : S.adv_dfa ? advance_kernel<true, true> : advance_kernel<true, false>;
  launch_overlapped(kernel, dim3((S.B + S.adv_rows - 1) / S.adv_rows), dim3(ADV_WARPS * 32), adv_smem_bytes(G, S), st, G, S, tokens, status);
}
static void launch_sweep_coop(const GrammarDev& G, const StateDev& S, int grid, cudaStream_t st) {
  GrammarDev g = G;
  StateDev s = S;
  void* args[] = {&g, &s};
  cudaLaunchCooperativeKernel((const void*)sweep_kernel, dim3((unsigned)grid), dim3(SWEEP_WARPS * 32), args,
                              S.au.smem_bytes, st);
}
void launch_plan(const GrammarDev& G, const StateDev& S, cudaStream_t st) {
  launch_overlapped(plan_kernel, dim3(1), dim3(std::min<uint32_t>(1024u, std::max<uint32_t>(64u, (S.B + 31u) / 32u * 32u))), 0, st, G, S);
}
// the sweep alone, for jobs the caller has already listed (used by the allocation-free entry point)
void launch_sweep(const GrammarDev& G, const StateDev& S, int grid, cudaStream_t st) { launch_sweep_coop(G, S, grid, st); }
void launch_gather(const GrammarDev& G, const StateDev& S, uint32_t* out, size_t stride_words, cudaStream_t st) {
  dim3 grid((unsigned)std::min<size_t>((stride_words + 255) / 256, 64), S.B);
  launch_overlapped(gather_kernel, grid, dim3(256), 0, st, G, S, out, stride_words);
}
static dim3 apply_grid(uint32_t V, int dtype, uint32_t batch) {
  const uint32_t units = V / (dtype == FMT_BF16 ? 16u : 8u) + 1u;
  return dim3((units + 256u * APPLY_UNITS - 1u) / (256u * APPLY_UNITS), batch);
}
void launch_apply(const uint32_t* mask, size_t stride_words, void* logits, int dtype, uint32_t batch, uint32_t V,
                  size_t row_stride, cudaStream_t st) {
  if (batch == 0 || V == 0) return;
  const dim3 grid = apply_grid(V, dtype, batch);
  if (dtype == FMT_BF16) launch_overlapped(apply_kernel<uint16_t>, grid, dim3(256), 0, st, mask, stride_words, (uint16_t*)logits, V, row_stride);
  else launch_overlapped(apply_kernel<uint32_t>, grid, dim3(256), 0, st, mask, stride_words, (uint32_t*)logits, V, row_stride);
}
void launch_gather_apply(const GrammarDev& G, const StateDev& S, void* logits, int dtype, size_t row_stride,
                         uint32_t* mask_out, size_t stride_words, cudaStream_t st) {
  const dim3 grid = apply_grid(G.V, dtype, S.B);
  if (dtype == FMT_BF16)
    launch_overlapped(gather_apply_kernel<uint16_t>, grid, dim3(256), 0, st, G, S, (uint16_t*)logits, row_stride, mask_out, stride_words);
  else
    launch_overlapped(gather_apply_kernel<uint32_t>, grid, dim3(256), 0, st, G, S, (uint32_t*)logits, row_stride, mask_out, stride_words);
}
void launch_evacuate(const StateDev& S, cudaStream_t st) { evacuate_kernel<<<S.B, 128, 0, st>>>(S); }
void launch_reintern(const StateDev& S, int32_t* init_state_dev, cudaStream_t st) {
  reintern_kernel<<<S.B + 1, 32, 0, st>>>(S, init_state_dev);
  fix_init_rows_kernel<<<(S.B + 127) / 128, 128, 0, st>>>(S, init_state_dev);
}
void launch_survivors(const GrammarDev& G, const StateDev& Old, const StateDev& S, const uint32_t* old_count, cudaStream_t st) {
  const uint32_t n = Old.max_states;
  dim3 grid((n + 255) / 256, 256);
  survivors_kernel<<<grid, 32, 0, st>>>(G, Old, S, old_count);
}
void launch_query(const StateDev& S, uint8_t* a, uint8_t* f, uint32_t* ns, uint32_t* ni, int32_t* sid, cudaStream_t st) {
  query_kernel<<<(S.B + 127) / 128, 128, 0, st>>>(S, a, f, ns, ni, sid);
}

}  // namespace fmt
