// The fill of a row's mask by the grammar automaton (grammar_automaton.cpp; Sections 3.3, 4.1, 4.3 of the paper).
//
// A thread block, or a cluster of them, takes one row.  The kernel items of the chart's last set are grouped by dotted rule;
// every group starts a THREAD at the root of the vocabulary trie: a code of the automaton and a CONTEXT, the set of
// origins its items were begun in.  A trie node's children are reached by one table look-up each.  Where the automaton says that a
// rule begun in the chart ends, the thread's context is EXPANDED: the items that waited in its origins, completed upwards (Section
// 3.2's Complete), start threads of their own at that node.  A context is expanded once per row.  A token is valid iff some
// thread is alive at the node where its bytes end.
//
// What bounds it: at the sizes measured, latency - rounds of "take threads from the stack, look their children up, push
// what is alive", each two dependent reads in L2 and three block barriers, about as many rounds as the longest token has bytes.
// Nothing waits for another block and no Earley set is built.
// Measured on a B200, the fill alone, against the sweep of the whole grid by Earley steps (kernels.cu) before:
//   8 rows of JSON, 32,000 tokens               239 -> 95 us    (where about half of the rows are computed)
//   64 rows of a JSON schema, 128,256 tokens    263 -> 60 us
//   128 rows of SQL, 152,064 tokens             667 -> 279 us
//   37 rows of JSON, 50,001 tokens              362 -> 129 us
//   256 rows of ambiguous JSON, 128,256 tokens  3.51 -> 2.68 ms
// The sweep stays for grammars without an automaton and for the cache of context-independent entries.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "sweep_warp.cuh"

namespace fmt {
namespace cg = cooperative_groups;

constexpr int AF_WARPS = 8, AF_THREADS = AF_WARPS * 32;
constexpr uint32_t AF_BATCH = 1024;       // threads taken from the stack per round
constexpr uint32_t AF_SEEN = 1024;        // recently started threads (a lossy table: repeats only cost time)
constexpr uint32_t AF_STAGE = 2048;       // a chart up to this many words is read from shared memory
constexpr uint32_t AF_BUF = 1024;         // items of an expansion in shared memory (larger ones: global memory)
constexpr uint32_t AF_WORK = 512, AF_HSET = 1024;
constexpr uint32_t AF_MASK_SMEM = 6144;   // mask rows up to this many words are collected in shared memory
// stack entries that are not threads, told by their code
constexpr uint32_t AF_SPAWN = 0xFFFFFFFDu;   // the expansion of a context at a node (first child, children)
constexpr uint32_t AF_EXITS = 0xFFFFFFFCu;   // the same at a list of nodes (where in ga_wide_exit, count)
constexpr uint32_t AF_EXIT_PIECE = 1024;     // nodes of such a list taken at once
constexpr uint32_t AF_TOKENS = 0xFFFFFFFBu;  // tokens to mark (where in ga_tok, count)
constexpr uint32_t CTX_NEW = 0xFFFFFFFFu;

enum : uint32_t { AC_TOP = 0, AC_FAIL = 1, AC_NCTX = 2, AC_POOL = 3, AC_NWORK = 4, AC_NBUF = 5, AC_OVER = 6, AC_WSUM = 8,
                  AC_NWIDE = 16, AC_WIDE = 20, AC_WORDS = 84 };

// A block's contexts, in global memory that only this block uses.
struct Contexts {
  const AutoFillDev& A;
  uint2* org;       // [ctx_cap] origins: offset into pool, count
  uint2* exp;       // [ctx_cap] expansion: offset into pool, count (CTX_NEW: not made yet); pairs (code, rule << 16 | context)
  uint32_t* lhs;    // [ctx_cap] the non-terminal whose rule is open
  uint32_t* hash;   // [hash_mask + 1] context + 1, 0 = empty
  uint32_t* pool;
  uint32_t *big_work, *big_hset, *big_buf;
  __device__ __forceinline__ explicit Contexts(const AutoFillDev& a, uint32_t block) : A(a) {
    uint32_t* p = a.scratch + (size_t)block * a.scratch_words;
    org = reinterpret_cast<uint2*>(p), p += 2 * a.ctx_cap;
    exp = reinterpret_cast<uint2*>(p), p += 2 * a.ctx_cap;
    lhs = p, p += a.ctx_cap;
    hash = p, p += 2 * a.ctx_cap;
    pool = p, p += a.pool_cap;
    big_work = p, p += a.big_cap / 4;
    big_hset = p, p += a.big_cap / 2;
    big_buf = p;
  }
};

// The row's chart as an expansion reads it.
struct AfChart {
  const uint32_t* off;
  const uint32_t* items;
  uint32_t m;
};

// ---- the parts one warp does: contexts and their expansions

// The context (lhs, list[0..n) & 0xFFFF) (ascending): its number, or CTX_NEW when there is no room.
__device__ uint32_t intern_context(const Contexts& C, uint32_t* ctl, uint32_t lhs, const uint32_t* list, uint32_t n) {
  const uint32_t lane = lane_id();
  uint32_t h = 0;
  for (uint32_t i = lane; i < n; i += 32) h += mix32((list[i] & 0xFFFFu) + 1u);
  h = mix32(__reduce_add_sync(FULL, h) + lhs * 0x9E3779B9u + n);
  const uint32_t mask = 2u * C.A.ctx_cap - 1u;
  uint32_t slot = h & mask;
  for (;;) {
    const uint32_t v = C.hash[slot];
    if (v == 0u) break;
    const uint2 o = C.org[v - 1u];
    bool same = o.y == n && C.lhs[v - 1u] == lhs;
    if (same)
      for (uint32_t i = lane; i < n; i += 32) same = same && C.pool[o.x + i] == (list[i] & 0xFFFFu);
    if (__all_sync(FULL, same)) return v - 1u;
    slot = (slot + 1u) & mask;
  }
  const uint32_t id = ctl[AC_NCTX], at = ctl[AC_POOL];
  if (id >= C.A.ctx_cap || n > C.A.pool_cap - at) return CTX_NEW;
  for (uint32_t i = lane; i < n; i += 32) C.pool[at + i] = list[i] & 0xFFFFu;
  __syncwarp();
  if (lane == 0) {
    C.org[id] = make_uint2(at, n);
    C.exp[id] = make_uint2(0u, CTX_NEW);
    C.lhs[id] = lhs;
    C.hash[slot] = id + 1u;
    ctl[AC_NCTX] = id + 1u;
    ctl[AC_POOL] = at + n;
  }
  __syncwarp();
  return id;
}

// buf[0..n), values rule << 16 | origin in any order, room for the next power of two: sorted, grouped by rule, as the expansion
// list (offset, count) in the pool.  False when there is no room.
__device__ bool group_items(const GrammarDev& G, const Contexts& C, uint32_t* ctl, uint32_t* buf, uint32_t n, uint2& out) {
  const uint32_t lane = lane_id();
  sort_items(buf, n, 1u << 30);
  uint32_t k = 0;  // repeats go
  for (uint32_t base = 0; base < n; base += 32) {
    const uint32_t i = base + lane;
    const uint32_t v = i < n ? buf[i] : 0u;
    const bool keep = i < n && (i == 0u || buf[i - 1u] != v);
    const uint32_t b = __ballot_sync(FULL, keep);
    __syncwarp();
    if (keep) buf[k + __popc(b & ((1u << lane) - 1u))] = v;  // (never beyond what has been read: i - 1 of the next piece is i's own value or earlier)
    k += __popc(b);
    __syncwarp();
  }
  uint32_t groups = 0;
  for (uint32_t base = 0; base < k; base += 32) {
    const uint32_t i = base + lane;
    groups += __popc(__ballot_sync(FULL, i < k && (i == 0u || (buf[i - 1u] >> 16) != (buf[i] >> 16))));
  }
  const uint32_t at = (ctl[AC_POOL] + 1u) & ~1u;
  __syncwarp();
  if (at + 2u * groups > C.A.pool_cap) return false;
  if (lane == 0) ctl[AC_POOL] = at + 2u * groups;
  __syncwarp();
  uint32_t g = 0;
  for (uint32_t i = 0; i < k;) {
    const uint32_t d = buf[i] >> 16;
    uint32_t e = i + 1u;
    for (;;) {  // the end of the group
      const uint32_t b = __ballot_sync(FULL, e + lane >= k || (buf[e + lane] >> 16) != d);
      if (b) {
        e += (uint32_t)__ffs(b) - 1u;
        break;
      }
      e += 32u;
    }
    const uint32_t code = __ldg(&G.ga_root[d]);
    if (code != GA_DEAD) {
      const uint32_t c = intern_context(C, ctl, __ldg(&G.lhs[d]), buf + i, e - i);
      if (c == CTX_NEW) return false;
      if (lane == 0) reinterpret_cast<uint2*>(C.pool)[at / 2u + g] = make_uint2(code, d << 16 | c);
      ++g;
    }
    i = e;
  }
  __syncwarp();
  out = make_uint2(at, g);
  return true;
}

// Complete upwards from the origins of context c: what waits there, with the dot moved.
__device__ bool expand_into(const GrammarDev& G, const Contexts& C, const AfChart& J, uint32_t c, uint32_t* ctl, uint32_t* work,
                            uint32_t work_cap, uint32_t* hset, uint32_t hset_mask, uint32_t* buf, uint32_t buf_cap) {
  const uint32_t lane = lane_id();
  __syncwarp();
  if (lane == 0) ctl[AC_NWORK] = 0u, ctl[AC_NBUF] = 0u, ctl[AC_OVER] = 0u;
  __syncwarp();
  auto need = [&](uint32_t a, uint32_t o) {  // "a, begun in set o, is complete"
    const uint32_t key = a << 16 | o;
    const int r = hset_insert(hset, hset_mask, key);
    if (r == 0) return;
    const uint32_t at = r < 0 ? work_cap : atomicAdd(&ctl[AC_NWORK], 1u);
    if (at < work_cap) work[at] = key;
    else ctl[AC_OVER] = 1u;
  };
  const uint2 org = C.org[c];
  const uint32_t lhs = C.lhs[c];
  for (uint32_t i = lane; i < org.y; i += 32) need(lhs, C.pool[org.x + i]);
  for (uint32_t head = 0;; ++head) {
    __syncwarp();
    const uint32_t n = ctl[AC_NWORK], over = ctl[AC_OVER];
    __syncwarp();
    if (over) return false;
    if (head >= n) break;
    const uint32_t a = work[head] >> 16, o = work[head] & 0xFFFFu;
    const uint32_t lo = J.off[o], hi = J.off[o + 1u];
    for (uint32_t k = lo + lane; k < hi; k += 32) {
      const uint32_t it = J.items[k], inf = __ldg(&G.info[it & 0xFFFFu]);
      if ((inf >> INFO_KIND_SHIFT) != KIND_NT || (inf & INFO_ARG_MASK) != a) continue;
      const uint32_t x = (it & 0xFFFFu) + 1u, ix = __ldg(&G.info[x]);
      const uint32_t skip = (ix >> INFO_SKIP_SHIFT) & INFO_SKIP_MASK;
      if ((ix >> INFO_KIND_SHIFT) != KIND_END) {
        const uint32_t at = atomicAdd(&ctl[AC_NBUF], 1u);
        if (at < buf_cap) buf[at] = x << 16 | (it >> 16);
        else ctl[AC_OVER] = 1u;
      }
      const uint32_t ie = skip ? __ldg(&G.info[x + skip]) : ix;
      if ((ie >> INFO_KIND_SHIFT) == KIND_END) need(ie & INFO_ARG_MASK, it >> 16);
    }
  }
  return true;
}

__device__ bool expand_context(const GrammarDev& G, const Contexts& C, const AfChart& J, uint32_t c, uint32_t* ctl, uint32_t* work,
                               uint32_t* hset, uint32_t* buf) {
  const uint32_t lane = lane_id();
  uint32_t* b = buf;
  bool ok = expand_into(G, C, J, c, ctl, work, AF_WORK, hset, AF_HSET - 1u, buf, AF_BUF);
  hset_clear_all(hset, AF_HSET - 1u);
  if (!ok) {  // too large for shared memory
    b = C.big_buf;
    hset_clear_all(C.big_hset, C.A.big_cap / 2u - 1u);
    ok = expand_into(G, C, J, c, ctl, C.big_work, C.A.big_cap / 4u, C.big_hset, C.A.big_cap / 2u - 1u, C.big_buf, C.A.big_cap);
  }
  uint2 list;
  ok = ok && group_items(G, C, ctl, b, ctl[AC_NBUF], list);
  __syncwarp();
  if (lane == 0) C.exp[c] = ok ? list : make_uint2(0u, 0u);
  __syncwarp();
  return ok;
}

// Where `code` leads on byte class e.
__device__ __forceinline__ uint32_t ga_next(const GrammarDev& G, uint32_t code, uint32_t e) {
  if (!(code & GA_ITEM)) return __ldg(&G.ga_trans[(size_t)code * G.n_eq + e]);
  const uint32_t org = (code >> 14) & 0xFFFFu;
  const uint32_t t = __ldg(&G.dfa_trans[(size_t)(code & 0x3FFFu) * G.n_eq + e]);
  if (t == 0xFFFFu || !(t & 0xC000u)) return GA_DEAD;
  if (!(t & 0x8000u)) return GA_ITEM | (org << 14) | (t & 0x3FFFu);
  if (org == 0u) return GA_EXIT | ((t & 0x4000u) ? (GA_ITEM | (t & 0x3FFFu)) : GA_NONE);
  const uint32_t key = org << 16 | t;
  for (uint32_t s = ga_hash(key) & G.ga_acc_mask;; s = (s + 1u) & G.ga_acc_mask) {
    const uint2 kv = __ldg(reinterpret_cast<const uint2*>(G.ga_acc) + s);
    if (kv.x == key) return kv.y;
    if (kv.x == 0u) return GA_UNKNOWN;
  }
}

__global__ void __launch_bounds__(AF_THREADS) automaton_fill_kernel(const __grid_constant__ GrammarDev G,
                                                                    const __grid_constant__ StateDev S) {
  const uint32_t n_jobs = S.counters[CNT_N_JOBS];
  if (n_jobs == 0u) return;  // (every block sees the same count)
  extern __shared__ __align__(16) uint32_t smem[];
  const AutoFillDev& A = S.af;
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
  uint4* cur = reinterpret_cast<uint4*>(smem);
  unsigned long long* seen = reinterpret_cast<unsigned long long*>(cur + AF_BATCH);
  uint32_t* pre = reinterpret_cast<uint32_t*>(seen + AF_SEEN);  // [AF_BATCH + 1]
  uint32_t* ctl = pre + AF_BATCH + 4;
  uint32_t* stage = ctl + AC_WORDS;
  uint32_t* buf = stage + AF_STAGE;
  uint32_t* work = buf + AF_BUF;
  uint32_t* hset = work + AF_WORK;
  uint32_t* mask_sm = hset + AF_HSET;
  const bool in_smem = G.Wm <= AF_MASK_SMEM;
  uint4* stack = A.stack + (size_t)blockIdx.x * A.stack_cap;
  const Contexts C(A, blockIdx.x);
  const cg::cluster_group cluster = cg::this_cluster();
  const uint32_t parts = cluster.num_blocks(), part = cluster.block_rank();
  for (uint32_t i = tid; i < AF_HSET; i += AF_THREADS) hset[i] = EMPTY_SLOT;
  uint32_t looked_up = 0, contexts = 0;

  for (uint32_t j = blockIdx.x / parts; j < n_jobs; j += gridDim.x / parts) {
    const uint32_t row = S.jobs[j];
    const uint32_t* chart = S.arena + S.row_chart[row];
    AfChart J;
    J.m = chart[CH_SETS];
    const uint32_t chart_words = chart[CH_WORDS];
    const bool accepting = (chart[CH_FLAGS] & CHART_ACCEPTING) != 0u;
    J.off = chart + CH_HDR;
    if (chart_words <= AF_STAGE) {
      for (uint32_t i = CH_HDR + tid; i < chart_words; i += AF_THREADS) stage[i] = chart[i];
      J.off = stage + CH_HDR;
    }
    J.items = J.off + J.m + 1u;
    uint32_t* const out = S.mask_rows + (size_t)S.row_mask[row] * G.Wm;
    uint32_t* const mask = in_smem ? mask_sm : out;  // (clusters only with masks in shared memory)
    for (uint32_t i = tid; i < G.Wm; i += AF_THREADS) mask[i] = 0u;
    for (uint32_t i = tid; i < AF_SEEN; i += AF_THREADS) seen[i] = 0ull;
    for (uint32_t i = tid; i < 2u * A.ctx_cap; i += AF_THREADS) C.hash[i] = 0u;
    if (tid < AC_WORDS) ctl[tid] = 0u;
    __syncthreads();
    if (warp == 0) {  // the kernel of the chart's last set starts the first threads
      const uint32_t lo = J.off[J.m - 1u], hi = J.off[J.m], self = J.m - 1u;
      uint32_t* b = hi - lo <= AF_BUF ? buf : C.big_buf;
      uint32_t n = 0;
      if (hi - lo <= A.big_cap) {
        for (uint32_t base = lo; base < hi; base += 32) {
          const uint32_t k = base + lane;
          const uint32_t it = k < hi ? J.items[k] : 0u;
          bool take = k < hi && ((it >> 16) != self || (it & 0xFFFFu) == ITEM_START);
          if (take && k > lo && J.items[k - 1u] == it - 1u && (it & 0xFFFFu) != 0u) {  // the item before it skips to it
            const uint32_t d = (it & 0xFFFFu) - 1u;
            take = !((__ldg(&G.info[d]) & INFO_NULLABLE) && __ldg(&G.ga_root[d]) != GA_DEAD);
          }
          const uint32_t bal = __ballot_sync(FULL, take);
          if (take) b[n + __popc(bal & ((1u << lane) - 1u))] = (it << 16) | (it >> 16);
          n += __popc(bal);
        }
        __syncwarp();
      }
      uint2 list = make_uint2(0u, 0u);
      const bool ok = hi - lo <= A.big_cap && group_items(G, C, ctl, b, n, list) && list.y <= A.stack_cap;
      const uint4 root = __ldg(reinterpret_cast<const uint4*>(G.ga_node));
      uint32_t top = 0;
      if (ok)
        for (uint32_t base = 0; base < list.y; base += 32) {
          const uint32_t i = base + lane;
          const uint2 x = i < list.y ? reinterpret_cast<const uint2*>(C.pool)[list.x / 2u + i] : make_uint2(0u, 0u);
          const uint32_t wide = i < list.y ? __ldg(&G.ga_wide[x.y >> 16]) : GA_DEAD;
          uint4 en = make_uint4(root.x, root.y >> 8, x.x, x.y & 0xFFFFu);
          if (wide != GA_DEAD) {  // most of the vocabulary follows from this item alone
            const uint4 r = __ldg(reinterpret_cast<const uint4*>(G.ga_wide_rec) + wide);
            en = make_uint4(r.y, r.z, AF_EXITS, en.w);
            const uint32_t at = atomicAdd(&ctl[AC_NWIDE], 1u);
            if (at < AC_WORDS - AC_WIDE) ctl[AC_WIDE + at] = r.x;
            else ctl[AC_FAIL] = 1u + DIAG_SET_SCRATCH;
          }
          const bool take = i < list.y && en.y != 0u;
          const uint32_t bal = __ballot_sync(FULL, take);
          if (take) stack[top + __popc(bal & ((1u << lane) - 1u))] = en;
          top += __popc(bal);
        }
      if (lane == 0) {
        ctl[AC_TOP] = top;
        if (!ok) ctl[AC_FAIL] = 1u + DIAG_SET_SCRATCH;
      }
    }
    __syncthreads();
    for (uint32_t k = 0, nw = min(ctl[AC_NWIDE], AC_WORDS - AC_WIDE); k < nw; ++k) {
      const uint32_t* row_of = G.ga_wide_mask + (size_t)ctl[AC_WIDE + k] * G.Wm;
      for (uint32_t i = part * AF_THREADS + tid; i < G.Wm; i += parts * AF_THREADS) mask[i] |= __ldg(row_of + i);
    }
    __syncthreads();

    for (;;) {  // ---- rounds
      const uint32_t top = ctl[AC_TOP];
      if (top == 0u || ctl[AC_FAIL]) break;
      // (a crowded stack is taken in smaller pieces, which keeps it from growing: depth first)
      const uint32_t room = A.stack_cap - top;
      const uint32_t n = min(top, max(1u, min(AF_BATCH, room / 16u)));
      bool missing = false;
      uint4 mine[AF_BATCH / AF_THREADS];
#pragma unroll
      for (uint32_t u = 0; u < AF_BATCH / AF_THREADS; ++u) {
        const uint32_t i = tid * (AF_BATCH / AF_THREADS) + u;
        if (i < n) {
          mine[u] = stack[top - n + i];
          cur[i] = mine[u];
          if (mine[u].z == AF_SPAWN || mine[u].z == AF_EXITS) missing |= C.exp[mine[u].w].y == CTX_NEW;
        }
      }
      const bool expand = __syncthreads_or(missing) != 0;
      if (tid == 0) ctl[AC_TOP] = top - n;
      if (expand) {
        if (warp == 0)
          for (uint32_t base = 0; base < n; base += 32) {
            const uint32_t i = base + lane;
            const uint32_t c = i < n && (cur[i].z == AF_SPAWN || cur[i].z == AF_EXITS) ? cur[i].w : 0xFFFFFFFFu;
            uint32_t todo = __ballot_sync(FULL, c != 0xFFFFFFFFu && C.exp[c].y == CTX_NEW);
            while (todo) {
              const uint32_t x = __shfl_sync(FULL, c, __ffs(todo) - 1);
              if (!expand_context(G, C, J, x, ctl, work, hset, buf) && lane == 0) ctl[AC_FAIL] = 1u + DIAG_SET_TABLE;
              todo &= ~__ballot_sync(FULL, c == x);
            }
          }
        __syncthreads();
      }
      // the items of work: a thread's children, an expansion's elements (at least one each, so that all starts differ)
      uint32_t w[AF_BATCH / AF_THREADS], sum = 0;
#pragma unroll
      for (uint32_t u = 0; u < AF_BATCH / AF_THREADS; ++u) {
        const uint32_t i = tid * (AF_BATCH / AF_THREADS) + u;
        w[u] = i >= n ? 0u
               : mine[u].z == AF_SPAWN ? max(1u, C.exp[mine[u].w].y)
               : mine[u].z == AF_EXITS ? min(mine[u].y, AF_EXIT_PIECE) * max(1u, C.exp[mine[u].w].y) : mine[u].y;
        sum += w[u];
      }
      uint32_t incl = sum;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL, incl, d);
        if ((int)lane >= d) incl += t;
      }
      if (lane == 31u) ctl[AC_WSUM + warp] = incl;
      __syncthreads();
      uint32_t before = incl - sum, total = 0;
#pragma unroll
      for (uint32_t k = 0; k < AF_WARPS; ++k) {
        const uint32_t s = ctl[AC_WSUM + k];
        if (k < warp) before += s;
        total += s;
      }
#pragma unroll
      for (uint32_t u = 0; u < AF_BATCH / AF_THREADS; ++u) {
        const uint32_t i = tid * (AF_BATCH / AF_THREADS) + u;
        if (i <= n) pre[i] = before;  // (pre[n] = the total)
        before += w[u];
      }
      if (n == AF_BATCH && tid == 0) pre[n] = total;
      looked_up += total;
      __syncthreads();
      for (uint32_t base = warp * 32u; base < total; base += AF_THREADS) {
        // the entry that item `base` belongs to (all lanes the same search), then each lane's own
        uint32_t lo = 0, hi = n;
        while (hi - lo > 1u) {
          const uint32_t mid = (lo + hi) >> 1;
          if (pre[mid] <= base) lo = mid;
          else hi = mid;
        }
        const uint32_t nb = lo + 1u + lane <= n ? pre[lo + 1u + lane] - base : 32u;
        const uint32_t starts = __reduce_or_sync(FULL, nb < 32u ? 1u << nb : 0u);
        const uint32_t i = base + lane;
        const uint32_t e = lo + __popc(starts & (0xFFFFFFFFu >> (31u - lane)));
        // what the item pushes: `a` (a thread that goes on, or tokens), `b` and `c` (threads that start here)
        bool has_a = false, has_b = false, has_c = false;
        uint4 a, b, c;
        auto start = [&](uint32_t first, uint32_t rule, uint32_t ctx) {  // false: it was started here a moment ago
          const unsigned long long key = (unsigned long long)first << 32 | rule << 16 | ctx;
          return atomicExch(&seen[(mix32(first ^ (rule * 0x9E3779B1u)) + ctx) & (AF_SEEN - 1u)], key) != key;
        };
        if (i < total) {
          const uint4 en = cur[e];
          const uint32_t k = i - pre[e];
          if (en.z < AF_TOKENS) {
            const uint32_t child = en.x + k;
            // a cluster's blocks share the nodes of depth 2, and with them what lies below
            if (parts == 1u || child < G.ga_lvl2 || child >= G.ga_lvl3 || child % parts == part) {
              const uint4 nd = __ldg(reinterpret_cast<const uint4*>(G.ga_node) + child);
              const uint32_t t = ga_next(G, en.z, nd.y & 0xFFu);
              if (t == GA_UNKNOWN) ctl[AC_FAIL] = 1u + DIAG_ROOT_FAILED;  // (cannot happen: the automaton covers the vocabulary)
              else if (t != GA_DEAD) {
                const uint32_t kids = nd.y >> 8;
                if (nd.w == 1u) atomicOr(&mask[nd.z >> 5], 1u << (nd.z & 31u));
                else if (nd.w > 1u) has_c = true, c = make_uint4(nd.z, nd.w, AF_TOKENS, 0u);
                if (kids) {
                  if ((t & ~GA_EXIT) != GA_NONE) has_a = true, a = make_uint4(nd.x, kids, t & ~GA_EXIT, en.w);
                  if (t & GA_EXIT) {
                    const uint2 x = C.exp[en.w];
                    if (x.y == 1u) {
                      const uint2 el = reinterpret_cast<const uint2*>(C.pool)[x.x / 2u];
                      has_b = start(nd.x, el.y >> 16, el.y & 0xFFFFu);
                      b = make_uint4(nd.x, kids, el.x, el.y & 0xFFFFu);
                    } else if (x.y) {
                      has_b = start(nd.x, 0xFFFFu, en.w);
                      b = make_uint4(nd.x, kids, AF_SPAWN, en.w);
                    }
                  }
                }
              }
            }
          } else if (en.z == AF_TOKENS) {
            const uint32_t tok = __ldg(&G.ga_tok[en.x + k]);
            atomicOr(&mask[tok >> 5], 1u << (tok & 31u));
          } else {
            const uint2 x = C.exp[en.w];
            if (x.y) {
              uint2 nd = make_uint2(en.x, en.y);
              uint32_t q = k;
              bool ours = true;
              if (en.z == AF_EXITS) {
                if (k == 0u && en.y > AF_EXIT_PIECE)  // the rest of the list
                  has_a = true, a = make_uint4(en.x + AF_EXIT_PIECE, en.y - AF_EXIT_PIECE, AF_EXITS, en.w);
                nd = __ldg(reinterpret_cast<const uint2*>(G.ga_wide_exit) + en.x + k / x.y);
                q = k % x.y;
                // (a cluster's blocks all start the threads of nodes of depth 1 and deal out the others)
                ours = parts == 1u || (nd.x >= G.ga_lvl2 && nd.x < G.ga_lvl3) || (k / x.y) % parts == part;
              }
              if (ours) {
                const uint2 el = reinterpret_cast<const uint2*>(C.pool)[x.x / 2u + q];
                has_b = start(nd.x, el.y >> 16, el.y & 0xFFFFu);
                b = make_uint4(nd.x, nd.y, el.x, el.y & 0xFFFFu);
              }
            }
          }
        }
        __syncwarp();
        const uint32_t ba = __ballot_sync(FULL, has_a), bb = __ballot_sync(FULL, has_b), bc = __ballot_sync(FULL, has_c);
        if (ba | bb | bc) {
          const uint32_t lt = (1u << lane) - 1u, count = __popc(ba) + __popc(bb) + __popc(bc);
          uint32_t at = 0;
          if (lane == 0) at = atomicAdd(&ctl[AC_TOP], count);
          at = __shfl_sync(FULL, at, 0);
          if (at + count > A.stack_cap) {
            ctl[AC_FAIL] = 1u + DIAG_QUEUE_FULL;
          } else {
            if (has_a) stack[at + __popc(ba & lt)] = a;
            at += __popc(ba);
            if (has_b) stack[at + __popc(bb & lt)] = b;
            at += __popc(bb);
            if (has_c) stack[at + __popc(bc & lt)] = c;
          }
        }
      }
      __syncthreads();
    }
    // ---- the mask row
    __syncthreads();
    const uint32_t fail = ctl[AC_FAIL];
    contexts += ctl[AC_NCTX];
    if (fail && tid == 0) {  // a capacity was exceeded: the row's mask cannot be trusted
      diag(S, fail - 1u);
      if (!(atomicOr(&S.row_flags[row], ROW_BROKEN) & ROW_BROKEN)) stat_add(S, CNT_STAT_CAPERR, 1u);
      atomicExch(&S.counters[CNT_ERR], 1u);
    }
    if (tid == 0 && accepting && G.eos >= 0) atomicOr(&mask[(uint32_t)G.eos >> 5], 1u << ((uint32_t)G.eos & 31u));
    if (parts > 1u) {
      cluster.sync();
      for (uint32_t i = part * AF_THREADS + tid; i < G.Wm; i += parts * AF_THREADS) {
        uint32_t v = 0;
        for (uint32_t p = 0; p < parts; ++p) v |= *cluster.map_shared_rank(mask_sm + i, p);
        out[i] = v;
      }
      cluster.sync();
    } else if (in_smem) {
      __syncthreads();
      for (uint32_t i = tid; i < G.Wm; i += AF_THREADS) out[i] = mask_sm[i];
    }
    __syncthreads();
  }
  if (tid == 0 && contexts) {
    stat_add(S, CNT_STAT_TRANS, looked_up);
    stat_add(S, CNT_STAT_LOCAL, contexts);
  }
}

// ===================================================================================== launchers

static uint32_t fill_smem_bytes(const GrammarDev& G) {
  return AF_BATCH * 16u + AF_SEEN * 8u + (AF_BATCH + 4u + AC_WORDS + AF_STAGE + AF_BUF + AF_WORK + AF_HSET + (G.Wm <= AF_MASK_SMEM ? G.Wm : 0u)) * 4u;
}

void automaton_fill_layout(const GrammarDev& G, uint32_t rows, uint32_t max_blocks, AutoFillDev& A) {
  A.smem_bytes = fill_smem_bytes(G);
  A.scratch_words = 7u * A.ctx_cap + A.pool_cap + A.big_cap / 4u + A.big_cap / 2u + A.big_cap;
  // few rows: a cluster of blocks takes one, so that the chip is filled; many: one block each
  A.parts = 1;
  while (A.parts < 8u && G.Wm <= AF_MASK_SMEM && (uint64_t)rows * A.parts * 2u <= max_blocks) A.parts *= 2u;
  A.grid = std::min(rows, std::max(1u, max_blocks / A.parts)) * A.parts;
}

cudaError_t configure_automaton_fill() {
  return cudaFuncSetAttribute((const void*)automaton_fill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
}

void launch_automaton_fill(const GrammarDev& G, const StateDev& S, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(S.af.grid);
  cfg.blockDim = dim3(AF_THREADS);
  cfg.dynamicSmemBytes = S.af.smem_bytes;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = S.af.parts, at[0].val.clusterDim.y = 1, at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, automaton_fill_kernel, G, S);
}

}  // namespace fmt
