// One row's mask by Earley steps, by one thread block: the way out for a row that the fill by the grammar's automaton gives up
// (automaton_fill.cu).  The same walk as the grid's sweep (kernels.cu: hash-consed sets, one thread per trie node, a depth at a time), with
// the block's barriers between pass and steps in the place of queues and tickets, so that it waits for nobody.
#pragma once
#include "sweep_warp.cuh"

namespace fmt {

constexpr uint32_t BS_NREQ = 0, BS_ALIVE = 1, BS_AGAIN = 2, BS_FAILED = 3, BS_HDR = 8;
constexpr uint32_t BS_PER_THREAD = 4;  // trie nodes of a thread, their loads under way together
__host__ __device__ constexpr uint32_t block_sweep_words(uint32_t warps, uint32_t Nw) {
  return BS_HDR + warps * (SWEEP_CUR + SWEEP_HSET + ((2u * Nw + 7u) & ~7u) + W_CTRS + 8u);
}

// The row's mask row is written (all of it, whatever the fill has set in it before it gave the row up).  `slot`: whose tables (S.au) are used.
// False: a capacity was exceeded.  By all threads of a block; smem: block_sweep_words, 16-byte aligned.
__device__ __noinline__ bool sweep_row_by_block(const GrammarDev& G, const StateDev& S, uint32_t row, uint32_t slot, uint32_t* smem) {
  const AutoDev& A = S.au;
  const uint32_t tid = threadIdx.x, threads = blockDim.x, warp = tid >> 5, warps = threads >> 5, lane = lane_id();
  const uint32_t ntw = (2u * G.Nw + 7u) & ~7u;
  uint32_t* const sh = smem;
  uint32_t* const mine = smem + BS_HDR + warp * (SWEEP_CUR + SWEEP_HSET + ntw + W_CTRS + 8u);
  JobCtx J;
  {
    const uint32_t* chart = S.arena + S.row_chart[row];
    J.row = row;
    J.accepting = (chart[CH_FLAGS] & CHART_ACCEPTING) != 0u;
    J.m = chart[CH_SETS];
    J.base_off = chart + CH_HDR;
    J.base_items = chart + CH_HDR + J.m + 1u;
    J.recs = A.recs + (size_t)slot * A.cap * A.rec_words;
    J.hash = A.hash + (size_t)slot * (A.hash_mask + 1u);
    J.n_states = A.n_states + slot;
    J.cap = min(A.cap, (ORIGIN_SELF - 1u > J.m) ? ORIGIN_SELF - 1u - J.m : 0u);
    J.st = A.st + (size_t)slot * A.st_stride;
  }
  uint32_t* const req = reinterpret_cast<uint32_t*>(A.req) + (size_t)slot * A.req_cap;  // set << 8 | byte
  SweepWarp sw{G, S};
  sw.gen = 1u;  // (the hash is cleared for every row)
  sw.w.cur = mine, sw.w.cur_cap = SWEEP_CUR;
  sw.w.hset = mine + SWEEP_CUR, sw.w.hset_mask = SWEEP_HSET - 1u;
  sw.w.nt = sw.w.hset + SWEEP_HSET;
  sw.w.ctr = sw.w.nt + ntw;
  sw.tmp8 = sw.w.ctr + W_CTRS;
  uint32_t* const big = S.big_scratch + ((size_t)slot * warps + warp) * ((size_t)S.big_arena_items + S.big_hset_slots);
  bool big_mode = false;

  __syncthreads();
  hset_clear_all(sw.w.hset, sw.w.hset_mask);
  for (uint32_t i = lane; i < ntw; i += 32) sw.w.nt[i] = 0u;
  for (uint32_t i = tid; i <= A.hash_mask; i += threads) J.hash[i] = 0u;
  for (uint32_t i = tid; i < A.rec_words; i += threads)
    if (i < AR_SCAN || i >= AR_SCAN + 8u) J.recs[i] = i >= AR_TRANS ? T_UNKNOWN : 0u;
  if (tid == 0) *J.n_states = 1u, sh[BS_FAILED] = 0u;
  if (warp == 0) {  // set 0: the chart's last one
    scannable_bytes(G, J.base_items + J.base_off[J.m - 1u], J.base_off[J.m] - J.base_off[J.m - 1u], sw.tmp8);
    if (lane < 8u) J.recs[AR_SCAN + lane] = sw.tmp8[lane];
  }
  __threadfence();

  auto transition = [&](uint32_t p, uint32_t byte) { return J.recs + (size_t)p * A.rec_words + AR_TRANS + G.eq_of_byte[byte]; };
  auto mark = [](uint32_t t) { return t == T_PENDING ? (uint32_t)ST_PENDING : t == T_DEAD ? (uint32_t)ST_DEAD : t; };
  // the set at `node`, whose mark says that its transition was yet to be computed (it has been since)
  auto settle = [&](uint32_t node) -> uint32_t {
    const uint32_t p = __ldg(&G.parent[node]);
    const uint32_t s = mark(__ldcg(transition(p == 0u ? 0u : (uint32_t)__ldcg(J.st + p), __ldg(&G.node_byte[node]))));
    J.st[node] = (uint16_t)s;
    return s;
  };
  uint32_t last_level = 0;
  for (uint32_t L = 1; L <= G.depth; ++L) {
    const uint32_t lo = __ldg(&G.lvl_off[L]), hi = __ldg(&G.lvl_off[L + 1]);
    bool alive = false;
    for (bool again = true; again;) {  // (again: the queue was too short for all transitions of the depth)
      __syncthreads();
      if (tid == 0) sh[BS_NREQ] = sh[BS_ALIVE] = sh[BS_AGAIN] = 0u;
      __syncthreads();
      alive = false;
      for (uint32_t first = lo + tid; first < hi; first += BS_PER_THREAD * threads) {
        uint32_t byte[BS_PER_THREAD], ps[BS_PER_THREAD];
#pragma unroll
        for (uint32_t u = 0; u < BS_PER_THREAD; ++u) {
          const uint32_t node = first + u * threads;
          byte[u] = node < hi ? __ldg(&G.node_byte[node]) : 0u;
          ps[u] = node >= hi ? (uint32_t)ST_DEAD : L == 1u ? 0u : (uint32_t)__ldcg(J.st + __ldg(&G.parent[node]));
        }
#pragma unroll
        for (uint32_t u = 0; u < BS_PER_THREAD; ++u) {
          const uint32_t node = first + u * threads;
          if (node >= hi) continue;
          if (ps[u] == ST_PENDING) ps[u] = settle(__ldg(&G.parent[node]));
          uint32_t t = T_DEAD;
          if (ps[u] != ST_DEAD && ((__ldcg(J.recs + (size_t)ps[u] * A.rec_words + AR_SCAN + (byte[u] >> 5)) >> (byte[u] & 31u)) & 1u)) {
            uint32_t* slot_t = transition(ps[u], byte[u]);
            t = __ldcg(slot_t);
            if (t == T_UNKNOWN && (t = atomicCAS(slot_t, T_UNKNOWN, T_PENDING)) == T_UNKNOWN) {
              const uint32_t at = atomicAdd(&sh[BS_NREQ], 1u);
              t = T_PENDING;
              if (at < A.req_cap) req[at] = ps[u] << 8 | byte[u];
              else atomicExch(slot_t, T_UNKNOWN), sh[BS_AGAIN] = 1u;
            }
          }
          J.st[node] = (uint16_t)mark(t);
          alive |= t != T_DEAD;
        }
      }
      alive = __any_sync(FULL, alive);
      if (alive && lane == 0) sh[BS_ALIVE] = 1u;
      __syncthreads();
      const uint32_t n = min(sh[BS_NREQ], A.req_cap);
      again = sh[BS_AGAIN] != 0u, alive = sh[BS_ALIVE] != 0u;
      for (uint32_t q = warp; q < n; q += warps) {
        const uint32_t p = __ldcg(req + q) >> 8, byte = __ldcg(req + q) & 0xFFu;
        uint32_t r = sw.compute(J, p, byte, !big_mode);
        if (r == T_FAIL && !big_mode) {  // a set outgrew the scratch in shared memory: the large area from now on
          big_mode = true;
          sw.w.cur = big, sw.w.cur_cap = S.big_arena_items;
          sw.w.hset = big + S.big_arena_items, sw.w.hset_mask = S.big_hset_slots - 1u;
          clear_nt(G, sw.w);
          hset_clear_all(sw.w.hset, sw.w.hset_mask);
          if (lane == 0) stat_add(S, CNT_STAT_BIG, 1u);
          r = sw.compute(J, p, byte, false);
        }
        if (r == T_FAIL) {
          hset_clear_all(sw.w.hset, sw.w.hset_mask);
          clear_nt(G, sw.w);
          if (lane == 0) sh[BS_FAILED] = 1u, atomicExch(transition(p, byte), T_DEAD);
        }
      }
    }
    last_level = L;
    if (!alive) break;  // (the same for all threads)
  }
  __syncthreads();
  if (lane == 0 && sw.n_computed) {
    stat_add(S, CNT_STAT_TRANS, sw.n_computed);
    stat_add(S, CNT_STAT_LOCAL, sw.n_created);
  }
  // ---- mask words, as in the grid's sweep
  const uint32_t visited_end = __ldg(&G.lvl_off[last_level + 1u]);
  uint32_t* const mask = S.mask_rows + (size_t)S.row_mask[row] * G.Wm;
  for (uint32_t wd = warp; wd < G.Wm; wd += warps) {
    const uint32_t tok = wd * 32u + lane;
    const uint32_t node = tok < G.V ? __ldg(&G.tok_node[tok]) : 0xFFFFFFFEu;
    bool valid = false;
    if (node == 0xFFFFFFFFu) {
      valid = (int32_t)tok == G.eos && J.accepting;
    } else if (node < visited_end) {
      uint32_t s = __ldcg(J.st + node);
      if (s == ST_PENDING) s = settle(node);
      valid = s != ST_DEAD;
    }
    const uint32_t word = __ballot_sync(FULL, valid);
    if (lane == 0) mask[wd] = word;
  }
  __syncthreads();
  const bool ok = sh[BS_FAILED] == 0u;
  __syncthreads();
  return ok;
}

}  // namespace fmt
