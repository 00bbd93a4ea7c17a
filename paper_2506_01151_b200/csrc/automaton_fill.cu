// The fill of rows' masks by what the grammar automaton tabulates (grammar_automaton.cpp; Sections 3.3, 4.1, 4.3 of the paper).
//
// A thread block takes a row.  The kernel items of the chart's last set are grouped by dotted rule; each group has a CONTEXT, the set
// of origins its items were begun in, and the record of what follows from the item (its start): the tokens that are valid whatever
// the chart holds, and edges for the places inside tokens where the item's rule ends.  There the chart is asked: the context is
// EXPANDED, once per row, into the items that waited in its origins, completed upwards (Section 3.2's Complete), grouped
// in the same way.  An edge whose item is among them sets its own tokens, and its edges go on with that group's context.  A
// round takes all edges that are known, looks their items up in the contexts' expansions, and lists the edges of those that are found.
//
// What bounds it: latency - a few rounds (as many as rules end one after the other inside a token), each a read of edges in L2, and
// between them the expansions, which one warp makes.  Following edges replaced a walk of the trie over byte classes by table look-ups, a
// byte a round (the same automaton, tabulated less far).  Fills on a B200 before and now, us: 37 rows of JSON, 50,001 tokens 139 -> 65;
// 256 rows of ambiguous JSON, 128,256 tokens 1,010 -> 795; 24 charts of JSON without allocations 123 -> 72; 12 decoding steps of 128
// rows of SQL, 152,064 tokens 4,930 -> 2,460, 16 of 64 rows of a JSON schema 2,440 -> 1,690.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "block_sweep.cuh"
#include "sweep_warp.cuh"

namespace fmt {

constexpr int AF_WARPS = 8, AF_THREADS = AF_WARPS * 32;
constexpr uint32_t AF_BATCH = 512;        // entries (lists of edges with a context) of a round,
constexpr uint32_t AF_EDGES = 32768;      // edges of a round,
constexpr uint32_t AF_CHUNK = 4096;       // and of an entry
constexpr uint32_t AF_LISTS = 512, AF_TOKENS = 32768;  // lists of tokens that are written when a round's edges are through, and tokens in them
constexpr uint32_t AF_TIGHT = 2048;       // free places of a block's stack, its reserve not counted, below which entries are taken one at a time,
constexpr uint32_t AF_TIGHT_EDGES = 32;   // so many edges of them
constexpr uint32_t AF_SLICE = 1024;       // items of a last set whose starts are taken together
constexpr uint32_t AF_SEEN = 512;         // recently listed edges (a lossy table: repeats only cost time)
constexpr uint32_t AF_STAGE = 1024;       // a chart up to this many words is read from shared memory
constexpr uint32_t AF_CTX = 64, AF_CTX_HASH = 128, AF_POOL = 2048;  // contexts in shared memory, words of their lists
constexpr uint32_t AF_BUF = 512, AF_WORK = 256, AF_HSET = 512;      // an expansion in shared memory (larger ones: global memory)
constexpr uint32_t AF_KCYCLES = 1u << 14;      // a share of a row that takes longer (2^24 cycles, 8.5 ms) is given up for a sweep by Earley steps
// AC_FAIL: 0, 1 + the capacity that was exceeded, or
constexpr uint32_t AF_GIVEN_UP = 0xFFFFFFFFu;  // a wait ran out: the fill is given up, the row itself is fine
constexpr uint32_t AF_GONE = 0xFFFFFFFEu;      // another block has given the row up
constexpr uint32_t AF_LATE = 0xFFFFFFFDu;      // the share takes too long
constexpr uint32_t CTX_NEW = 0xFFFFFFFFu;

enum : uint32_t {
  AC_OVF = 0, AC_GTOP = 1, AC_FAIL = 2, AC_NCTX = 3, AC_POOL = 4, AC_NWORK = 5, AC_NBUF = 6, AC_OVER = 7, AC_SPILLED = 8, AC_JOB = 9,
  AC_NWIDE = 10, AC_LIST = 11, AC_LIST_END = 12, AC_LOOKED = 13, AC_BEGAN = 14, AC_SLOT = 15,
  AC_EDGES = 16,   // [2] counters of the entries (see Deal)
  AC_TOKENS = 24,  // [2] and of the lists of tokens
  AC_PEEK = 32, AC_FULL = 36, AC_WORDS = 40
};
static_assert(AC_WORDS % 4 == 0 && AC_WORDS <= AF_THREADS, "what follows in shared memory is cleared in 16-byte pieces; a thread clears a word");

// Lists whose elements are dealt out to the lanes: places and elements are counted by one atomic operation, so that the places are in
// the order of the elements.
struct Deal {
  uint32_t* count;   // 64 bits: places << 32 | elements; then the first place and the first element that found no room
  uint2* what;       // [cap] where the list begins, and what it comes with
  uint32_t* pre;     // [cap] its first element's number
  uint16_t* owner;   // [things / 32] the place of the list to which the element 32 * i belongs
  uint32_t cap, things;
};
__device__ __forceinline__ uint32_t dealt_lists(const Deal& D) { return min(D.count[1], D.count[2]); }
__device__ __forceinline__ uint32_t dealt_things(const Deal& D) { return min(D.count[0], D.count[3]); }
__device__ __forceinline__ void deal_clear(const Deal& D) {
  D.count[0] = D.count[1] = 0u;
  D.count[2] = D.count[3] = 0xFFFFFFFFu;
}
// By all lanes of a warp: the lists of the lanes with `yes`.  False: there is no room for the lane's.
__device__ __forceinline__ bool deal(const Deal& D, bool yes, uint32_t n, uint2 what) {
  const uint32_t lane = lane_id(), b = __ballot_sync(FULL, yes);
  if (b == 0u) return true;
  uint32_t incl = yes ? n : 0u;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t t = __shfl_up_sync(FULL, incl, d);
    if ((int)lane >= d) incl += t;
  }
  unsigned long long base = 0;
  if (lane == 31u) base = atomicAdd(reinterpret_cast<unsigned long long*>(D.count), (unsigned long long)__popc(b) << 32 | incl);
  const uint32_t slot = __shfl_sync(FULL, (uint32_t)(base >> 32), 31) + __popc(b & ((1u << lane) - 1u));
  const uint32_t before = __shfl_sync(FULL, (uint32_t)base, 31) + incl - (yes ? n : 0u);
  const bool fits = slot < D.cap && before + n <= D.things, longer = n > 128u;
  if (yes && fits) {
    D.what[slot] = what;
    D.pre[slot] = before;
    if (!longer)
      for (uint32_t p = (before + 31u) / 32u; p * 32u < before + n; ++p) D.owner[p] = (uint16_t)slot;
  } else if (yes) {
    atomicMin(&D.count[2], slot);
    atomicMin(&D.count[3], before);
  }
  for (uint32_t m = __ballot_sync(FULL, yes && fits && longer); m; m &= m - 1u) {
    const int src = __ffs(m) - 1;
    const uint32_t from = __shfl_sync(FULL, before, src), until = from + __shfl_sync(FULL, n, src), s = __shfl_sync(FULL, slot, src);
    for (uint32_t p = (from + 31u) / 32u + lane; p * 32u < until; p += 32u) D.owner[p] = (uint16_t)s;
  }
  return fits || !yes;
}
// The list to which element base + lane of n lists belongs (base a multiple of 32).
__device__ __forceinline__ uint32_t whose(const Deal& D, uint32_t n, uint32_t base) {
  const uint32_t lane = lane_id(), lo = D.owner[base / 32u];
  const uint32_t nb = lo + 1u + lane < n ? D.pre[lo + 1u + lane] - base : 32u;  // where the lists after it begin
  const uint32_t starts = __reduce_or_sync(FULL, nb < 32u ? 1u << nb : 0u);
  return lo + __popc(starts & (0xFFFFFFFFu >> (31u - lane)));
}

// The contexts of the row a block works on: in shared memory, or, when they outgrow it, in global memory of the block's own.
struct Contexts {
  uint2* org;       // [cap] origins: offset into pool, count
  uint2* exp;       // [cap] expansion: offset into pool, count (CTX_NEW: not made yet); rule << 16 | context, ascending
  uint32_t* lhs;    // [cap] the non-terminal whose rule is open
  uint32_t* hash;   // [hash_mask + 1] context + 1, 0 = empty
  uint32_t* pool;
  uint32_t cap, hash_mask, pool_cap;
};
// Four words of global memory (16-byte aligned, read past L1) on their way into shared memory.
__device__ __forceinline__ void peek(uint32_t* to, const uint32_t* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from) : "memory");
}
__device__ __forceinline__ uint32_t vload(const uint32_t* p) { return *reinterpret_cast<const volatile uint32_t*>(p); }
__device__ __forceinline__ Contexts global_contexts(const AutoFillDev& A) {
  uint32_t* p = A.scratch + (size_t)blockIdx.x * A.scratch_words;
  Contexts C;
  C.org = reinterpret_cast<uint2*>(p), p += 2 * A.ctx_cap;
  C.exp = reinterpret_cast<uint2*>(p), p += 2 * A.ctx_cap;
  C.lhs = p, p += A.ctx_cap;
  C.hash = p, p += 2 * A.ctx_cap;
  C.pool = p;
  C.cap = A.ctx_cap, C.hash_mask = 2u * A.ctx_cap - 1u, C.pool_cap = A.pool_cap;
  return C;
}
// (what follows them in the block's scratch)
__device__ __forceinline__ uint32_t* big_area(const AutoFillDev& A) {
  return A.scratch + (size_t)blockIdx.x * A.scratch_words + 7u * A.ctx_cap + A.pool_cap;
}

struct AfChart {
  const uint32_t* off;
  const uint32_t* items;
  uint32_t m;
};

// ---- the parts one warp does: contexts and their expansions

__device__ __forceinline__ uint32_t context_hash(uint32_t lhs, const uint32_t* list, uint32_t n) {
  uint32_t h = 0;
  for (uint32_t i = lane_id(); i < n; i += 32) h += mix32((list[i] & 0xFFFFu) + 1u);
  return mix32(__reduce_add_sync(FULL, h) + lhs * 0x9E3779B9u + n);
}

// The context (lhs, list[0..n) & 0xFFFF) (ascending): its number, or CTX_NEW when there is no room.
__device__ uint32_t intern_context(const Contexts& C, uint32_t* ctl, uint32_t lhs, const uint32_t* list, uint32_t n) {
  const uint32_t lane = lane_id();
  uint32_t slot = context_hash(lhs, list, n) & C.hash_mask;
  for (;;) {
    const uint32_t v = C.hash[slot];
    if (v == 0u) break;
    const uint2 o = C.org[v - 1u];
    bool same = o.y == n && C.lhs[v - 1u] == lhs;
    if (same)
      for (uint32_t i = lane; i < n; i += 32) same = same && C.pool[o.x + i] == (list[i] & 0xFFFFu);
    if (__all_sync(FULL, same)) return v - 1u;
    slot = (slot + 1u) & C.hash_mask;
  }
  const uint32_t id = ctl[AC_NCTX], at = ctl[AC_POOL];
  __syncwarp();
  if (id >= C.cap || n > C.pool_cap - at) return CTX_NEW;
  for (uint32_t i = lane; i < n; i += 32) C.pool[at + i] = list[i] & 0xFFFFu;
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

// The contexts leave shared memory.
__device__ void spill_contexts(Contexts& C, uint32_t* ctl, const AutoFillDev& A) {
  const uint32_t lane = lane_id(), n = ctl[AC_NCTX], words = ctl[AC_POOL];
  const Contexts D = global_contexts(A);
  for (uint32_t i = lane; i < n; i += 32) D.org[i] = C.org[i], D.exp[i] = C.exp[i], D.lhs[i] = C.lhs[i];
  for (uint32_t i = lane; i < words; i += 32) D.pool[i] = C.pool[i];
  for (uint32_t i = lane; i <= D.hash_mask; i += 32) D.hash[i] = 0u;
  __syncwarp();
  for (uint32_t c = 0; c < n; ++c) {
    const uint2 o = D.org[c];
    uint32_t slot = context_hash(D.lhs[c], D.pool + o.x, o.y) & D.hash_mask;
    if (lane == 0) {
      while (D.hash[slot]) slot = (slot + 1u) & D.hash_mask;
      D.hash[slot] = c + 1u;
    }
    __syncwarp();
  }
  C = D;
  if (lane == 0) ctl[AC_SPILLED] = 1u;
  __syncwarp();
}

// The contexts (lhs, {origin}) of the lanes with `valid`, all looked up at once: each lane's number, or CTX_NEW for all of them when there
// is no room.  (Nearly all contexts have one origin.  One after the other, each with its own chain of look-ups, those of a union of 60
// variants took 2.4 ms a fill of 4 rows, see below.)
__device__ uint32_t intern_singles(const Contexts& C, uint32_t* ctl, bool valid, uint32_t lhs, uint32_t origin) {
  const uint32_t lane = lane_id();
  const uint32_t peers = __match_any_sync(FULL, valid ? lhs << 16 | origin : 0xFFFFFFFFu);
  const int leader = __ffs(peers) - 1;
  const uint32_t home = mix32(mix32(origin + 1u) + lhs * 0x9E3779B9u + 1u) & C.hash_mask;  // (as context_hash has it)
  uint32_t id = CTX_NEW;
  if (valid && (int)lane == leader)
    for (uint32_t slot = home; id == CTX_NEW; slot = (slot + 1u) & C.hash_mask) {
      const uint32_t v = C.hash[slot];
      if (v == 0u) break;
      const uint2 o = C.org[v - 1u];
      if (o.y == 1u && C.lhs[v - 1u] == lhs && C.pool[o.x] == origin) id = v - 1u;
    }
  const bool fresh = valid && (int)lane == leader && id == CTX_NEW;
  const uint32_t b = __ballot_sync(FULL, fresh), n = __popc(b), first = ctl[AC_NCTX], at = ctl[AC_POOL];
  __syncwarp();
  if (first + n > C.cap || n > C.pool_cap - at) return CTX_NEW;
  if (fresh) {
    const uint32_t r = __popc(b & ((1u << lane) - 1u));
    id = first + r;
    C.pool[at + r] = origin;
    C.org[id] = make_uint2(at + r, 1u);
    C.exp[id] = make_uint2(0u, CTX_NEW);
    C.lhs[id] = lhs;
    for (uint32_t slot = home; atomicCAS(&C.hash[slot], 0u, id + 1u) != 0u;) slot = (slot + 1u) & C.hash_mask;
  }
  if (lane == 0) ctl[AC_NCTX] = first + n, ctl[AC_POOL] = at + n;
  __syncwarp();
  return __shfl_sync(FULL, id, leader);
}

// buf[0..n), room for the next power of two: sorted, without repeats.  How many are left, and how many rules they are of.
__device__ uint32_t sort_unique(uint32_t* buf, uint32_t n, uint32_t& groups) {
  const uint32_t lane = lane_id();
  sort_items(buf, n, 1u << 30);
  uint32_t k = 0;
  groups = 0;
  for (uint32_t base = 0, last = 0xFFFFFFFFu; base < n; base += 32) {
    const uint32_t i = base + lane;
    const uint32_t v = i < n ? buf[i] : 0xFFFFFFFFu;
    uint32_t p = __shfl_up_sync(FULL, v, 1);
    if (lane == 0) p = last;
    last = __shfl_sync(FULL, v, 31);
    const uint32_t b = __ballot_sync(FULL, i < n && v != p);
    groups += __popc(__ballot_sync(FULL, i < n && (v >> 16) != (p >> 16)));  // (no rule has the number 0xFFFF)
    __syncwarp();
    if (i < n && v != p) buf[k + __popc(b & ((1u << lane) - 1u))] = v;
    k += __popc(b);
  }
  __syncwarp();
  return k;
}

// buf[0..n), values rule << 16 | origin in any order, room for the next power of two: sorted, grouped by rule, as the expansion
// list (offset, count) in the pool.  False when there is no room.
__device__ bool group_items(const GrammarDev& G, const Contexts& C, uint32_t* ctl, uint32_t* buf, uint32_t n, uint2& out) {
  const uint32_t lane = lane_id();
  uint32_t groups;
  const uint32_t k = sort_unique(buf, n, groups);
  const uint32_t at = ctl[AC_POOL];
  __syncwarp();
  if (at + groups > C.pool_cap) return false;
  if (lane == 0) ctl[AC_POOL] = at + groups;
  __syncwarp();
  uint32_t g = 0;
  for (uint32_t i = 0; i < k;) {
    {  // rules with one item each, up to 32 of them together
      const uint32_t x = i + lane < k ? buf[i + lane] : 0xFFFFFFFFu, y = i + lane + 1u < k ? buf[i + lane + 1u] >> 16 : 0xFFFFu;
      const uint32_t before = __shfl_up_sync(FULL, x >> 16, 1);
      const uint32_t other = __ballot_sync(FULL, i + lane >= k || y == x >> 16 || (lane && before == x >> 16));
      const uint32_t run = other ? (uint32_t)__ffs(other) - 1u : 32u;
      if (run) {
        const bool v = lane < run;
        const uint32_t c = intern_singles(C, ctl, v, v ? __ldg(&G.ga_item[2u * (x >> 16)]) & 0xFFFFu : 0u, x & 0xFFFFu);
        if (__any_sync(FULL, v && c == CTX_NEW)) return false;
        if (v) C.pool[at + g + lane] = (x & 0xFFFF0000u) | c;
        g += run;
        i += run;
        continue;
      }
    }
    const uint32_t d = buf[i] >> 16;
    uint32_t e = i + 1u;
    for (;;) {  // the end of the group
      const uint32_t b = __ballot_sync(FULL, e + lane >= k || (buf[min(e + lane, k - 1u)] >> 16) != d);
      if (b) {
        e += (uint32_t)__ffs(b) - 1u;
        break;
      }
      e += 32u;
    }
    const uint32_t c = intern_context(C, ctl, __ldg(&G.ga_item[2u * d]) & 0xFFFFu, buf + i, e - i);
    if (c == CTX_NEW) return false;
    if (lane == 0) C.pool[at + g] = d << 16 | c;
    ++g;
    i = e;
  }
  __syncwarp();
  out = make_uint2(at, g);
  return true;
}

// The same for at most 32 different items that sit one to a lane (lane l < n: item l).
__device__ __forceinline__ bool group_lanes(const GrammarDev& G, const Contexts& C, uint32_t* ctl, uint32_t item, uint32_t n, uint2& out) {
  const uint32_t lane = lane_id(), at = ctl[AC_POOL];
  if (lane >= n) item = 0xFFFFFFFFu;
  if (n > 1u) {
#pragma unroll
    for (uint32_t k = 2; k <= 32; k <<= 1)
#pragma unroll
      for (uint32_t j = k >> 1; j > 0; j >>= 1) {
        const uint32_t other = __shfl_xor_sync(FULL, item, j);
        item = (((lane & k) == 0) == ((lane & j) == 0)) ? min(item, other) : max(item, other);
      }
  }
  const uint32_t d = item >> 16, before = __shfl_up_sync(FULL, d, 1);
  const bool leads = lane < n && (lane == 0u || before != d);
  const uint32_t lb = __ballot_sync(FULL, leads), groups = __popc(lb);
  if (at + groups + n > C.pool_cap) return false;
  __syncwarp();
  if (lane == 0) ctl[AC_POOL] = at + groups;
  __syncwarp();
  const uint32_t after = lane == 31u ? 0u : lb >> (lane + 1u), size = after ? (uint32_t)__ffs(after) : n - lane;  // (of the group of a lane that leads)
  const uint32_t lhs = leads ? __ldg(&G.ga_item[2u * d]) & 0xFFFFu : 0u;
  uint32_t ctx = CTX_NEW;
  if (__any_sync(FULL, leads && size == 1u)) {
    ctx = intern_singles(C, ctl, leads && size == 1u, lhs, item & 0xFFFFu);
    if (__any_sync(FULL, leads && size == 1u && ctx == CTX_NEW)) return false;
  }
  for (uint32_t m = __ballot_sync(FULL, leads && size > 1u); m; m &= m - 1u) {
    const uint32_t first = (uint32_t)__ffs(m) - 1u, k = __shfl_sync(FULL, size, first);
    const uint32_t top = ctl[AC_POOL];  // its origins, ascending, at the pool's top (which grows only if the context is new)
    if (top + k > C.pool_cap) return false;
    if (lane >= first && lane < first + k) C.pool[top + lane - first] = item & 0xFFFFu;
    __syncwarp();
    const uint32_t c = intern_context(C, ctl, __shfl_sync(FULL, lhs, first), C.pool + top, k);
    if (c == CTX_NEW) return false;
    if (lane == first) ctx = c;
  }
  if (leads) C.pool[at + __popc(lb & ((1u << lane) - 1u))] = d << 16 | ctx;
  __syncwarp();
  out = make_uint2(at, groups);
  return true;
}

// Complete upwards from the origins of context c: what waits there, with the dot moved.
__device__ bool expand_into(const GrammarDev& G, const Contexts& C, const AfChart& J, uint32_t c, uint32_t* ctl, uint32_t* work,
                            uint32_t work_cap, uint32_t* hset, uint32_t hset_mask, uint32_t* buf, uint32_t buf_cap) {
  const uint32_t lane = lane_id();
  __syncwarp();
  uint32_t nbuf = 0;
  if (lane == 0) ctl[AC_NWORK] = 0u, ctl[AC_OVER] = 0u;
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
    for (uint32_t base = lo; base < hi; base += 32) {
      const uint32_t k = base + lane;
      const uint32_t it = k < hi ? J.items[k] : 0u;
      const uint2 rec = __ldg(reinterpret_cast<const uint2*>(G.ga_item) + (it & 0xFFFFu));
      const bool match = k < hi && (rec.x >> 16) == a, on = match && (rec.y & GA_GOES_ON);
      const uint32_t b = __ballot_sync(FULL, on);
      if (nbuf + __popc(b) > buf_cap) {  // an item comes once for every set that it waits in: the repeats go
        uint32_t groups;
        __syncwarp();
        nbuf = sort_unique(buf, nbuf, groups);
        if (nbuf > buf_cap / 2u) return false;
      }
      if (on) buf[nbuf + __popc(b & ((1u << lane) - 1u))] = ((it & 0xFFFFu) + 1u) << 16 | (it >> 16);
      nbuf += __popc(b);
      if (match && (rec.y & 0xFFFFu) != 0xFFFFu) need(rec.y & 0xFFFFu, it >> 16);
    }
  }
  if (lane == 0) ctl[AC_NBUF] = nbuf;
  __syncwarp();
  return true;
}

// The same with everything in the warp's lanes: one context of at most 32 origins, at most 32 completions and 32 items.  Nearly all
// expansions are of this kind (one origin, two or three completions, one item); the general form takes some four times as many
// instructions.  False: it does not fit (nothing has changed but the pool's top).
__device__ bool expand_small(const GrammarDev& G, const Contexts& C, const AfChart& J, uint32_t c, uint32_t* ctl) {
  const uint32_t lane = lane_id();
  const uint2 org = C.org[c];
  if (org.y > 32u) return false;
  uint32_t work = lane < org.y ? C.lhs[c] << 16 | C.pool[org.x + lane] : 0u, nw = org.y;  // lane l: completion l
  uint32_t item = 0u, ni = 0u;                                                           // lane l: item l
  for (uint32_t head = 0; head < nw; ++head) {
    const uint32_t key = __shfl_sync(FULL, work, head);
    const uint32_t a = key >> 16, o = key & 0xFFFFu;
    const uint32_t lo = J.off[o], hi = J.off[o + 1u];
    for (uint32_t base = lo; base < hi; base += 32) {
      const uint32_t k = base + lane;
      const uint32_t it = k < hi ? J.items[k] : 0u;
      const uint2 rec = __ldg(reinterpret_cast<const uint2*>(G.ga_item) + (it & 0xFFFFu));
      const bool match = k < hi && (rec.x >> 16) == a;
      uint32_t on = __ballot_sync(FULL, match && (rec.y & GA_GOES_ON));
      if (on) {
        const uint32_t x = ((it & 0xFFFFu) + 1u) << 16 | (it >> 16);
        if (ni + __popc(on) > 32u) return false;
        for (; on; on &= on - 1u) {
          const uint32_t v = __shfl_sync(FULL, x, __ffs(on) - 1);
          if (__ballot_sync(FULL, lane < ni && item == v)) continue;
          if (lane == ni) item = v;
          ++ni;
        }
      }
      for (uint32_t up = __ballot_sync(FULL, match && (rec.y & 0xFFFFu) != 0xFFFFu); up; up &= up - 1u) {
        const uint32_t v = __shfl_sync(FULL, (rec.y & 0xFFFFu) << 16 | (it >> 16), __ffs(up) - 1);
        if (__ballot_sync(FULL, lane < nw && work == v)) continue;
        if (nw == 32u) return false;
        if (lane == nw) work = v;
        ++nw;
      }
    }
  }
  if (ctl[AC_NCTX] + ni > C.cap) return false;
  uint2 list;
  if (!group_lanes(G, C, ctl, item, ni, list)) return false;
  if (lane == 0) C.exp[c] = list;
  __syncwarp();
  return true;
}

__device__ __noinline__ bool expand_context(const GrammarDev& G, const AutoFillDev& A, Contexts& C, const AfChart& J, uint32_t c,
                                            uint32_t* ctl, uint32_t* work, uint32_t* hset, uint32_t* buf) {
  const uint32_t lane = lane_id();
  if (expand_small(G, C, J, c, ctl)) return true;
  for (;;) {
    uint32_t* b = buf;
    bool ok = expand_into(G, C, J, c, ctl, work, AF_WORK, hset, AF_HSET - 1u, buf, AF_BUF);
    hset_clear_all(hset, AF_HSET - 1u);
    if (!ok) {  // too large for shared memory
      uint32_t* big_work = big_area(A);
      uint32_t* big_hset = big_work + A.big_cap / 4u;
      b = big_hset + A.big_cap / 2u;
      hset_clear_all(big_hset, A.big_cap / 2u - 1u);
      ok = expand_into(G, C, J, c, ctl, big_work, A.big_cap / 4u, big_hset, A.big_cap / 2u - 1u, b, A.big_cap);
    }
    uint2 list = make_uint2(0u, 0u);
    const bool fits = ok && group_items(G, C, ctl, b, ctl[AC_NBUF], list);
    if (ok && !fits && !ctl[AC_SPILLED]) {
      spill_contexts(C, ctl, A);
      continue;
    }
    __syncwarp();
    if (lane == 0) C.exp[c] = list;
    __syncwarp();
    return fits;
  }
}

// Tokens at .. at + cnt of each lane's list, dealt out to the lanes two by two.
__device__ __forceinline__ void set_tokens(const GrammarDev& G, uint32_t* mask, uint32_t at, uint32_t cnt) {
  const uint32_t lane = lane_id();
  uint32_t incl = cnt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t t = __shfl_up_sync(FULL, incl, d);
    if ((int)lane >= d) incl += t;
  }
  const uint32_t total = __shfl_sync(FULL, incl, 31), excl = incl - cnt, from = at - excl;
  for (uint32_t base = 0; base < total; base += 64) {
    uint32_t tok[2];
#pragma unroll
    for (uint32_t u = 0; u < 2; ++u) {
      const uint32_t first = base + u * 32u;
      uint32_t e = 0;  // the last lane that begins at or before it
#pragma unroll
      for (uint32_t d = 16; d; d >>= 1)
        if (__shfl_sync(FULL, excl, e + d) <= first + lane) e += d;
      const uint32_t f = __shfl_sync(FULL, from, e);
      tok[u] = first + lane < total ? __ldg(&G.ga_tok[f + first + lane]) : 0xFFFFFFFFu;
    }
#pragma unroll
    for (uint32_t u = 0; u < 2; ++u)
      if (tok[u] != 0xFFFFFFFFu) atomicOr(&mask[tok[u] >> 5], 1u << (tok[u] & 31u));
  }
}

__global__ void __launch_bounds__(AF_THREADS, 4) automaton_fill_kernel(const __grid_constant__ GrammarDev G,
                                                                       const __grid_constant__ StateDev S) {
  before_me();
  const uint32_t n_jobs = S.counters[CNT_N_JOBS];
  const AutoFillDev& A = S.af;
  const uint32_t parts = A.parts;  // (a power of two)
  if (blockIdx.x >= n_jobs * parts) return;
  extern __shared__ __align__(16) uint32_t smem[];
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id(), lt = (1u << lane) - 1u;
  uint2* const entries = reinterpret_cast<uint2*>(smem);  // [2][AF_BATCH], in turn: first edge, context
  uint2* const lists = entries + 2 * AF_BATCH;            // [AF_LISTS] where in ga_tok
  unsigned long long* const seen = reinterpret_cast<unsigned long long*>(lists + AF_LISTS);
  Contexts C0;
  C0.org = reinterpret_cast<uint2*>(seen + AF_SEEN);
  C0.exp = C0.org + AF_CTX;
  C0.lhs = reinterpret_cast<uint32_t*>(C0.exp + AF_CTX);
  C0.pool = C0.lhs + AF_CTX;
  C0.hash = C0.pool + AF_POOL;
  C0.cap = AF_CTX, C0.hash_mask = AF_CTX_HASH - 1u, C0.pool_cap = AF_POOL;
  uint32_t* const pre = C0.hash + AF_CTX_HASH;  // [2][AF_BATCH], [AF_LISTS]
  uint32_t* const ctl = pre + 2 * AF_BATCH + AF_LISTS;
  uint32_t* const wide = ctl + AC_WORDS;        // [AF_THREADS] rows of ga_mask
  uint32_t* const stage = wide + AF_THREADS;
  uint32_t* const buf = stage + AF_STAGE;
  uint32_t* const work = buf + AF_BUF;
  uint32_t* const hset = work + AF_WORK;
  uint16_t* const owner = reinterpret_cast<uint16_t*>(hset + AF_HSET);
  uint4* const stack = A.stack + (size_t)blockIdx.x * A.stack_cap;  // entries that found no room: first edge, edges, context
  auto edge_deal = [&](uint32_t side) {
    return Deal{ctl + AC_EDGES + 4u * side, entries + side * AF_BATCH, pre + side * AF_BATCH, owner + side * (AF_EDGES / 32u), AF_BATCH, AF_EDGES};
  };
  auto token_deal = [&](uint32_t side) {
    return Deal{ctl + AC_TOKENS + 4u * side, lists, pre + 2u * AF_BATCH, owner + 2u * (AF_EDGES / 32u), AF_LISTS, AF_TOKENS};
  };
  for (uint32_t i = tid; i < AF_HSET; i += AF_THREADS) hset[i] = EMPTY_SLOT;
  uint32_t looked_up = 0, contexts = 0;
  bool gave_up = false;

  uint32_t ticket = blockIdx.x;
  if (parts > 1u) {  // (drawn by blocks that run: nobody ever waits for a block that has not started)
    if (tid == 0) ctl[AC_JOB] = atomicAdd(&S.counters[CNT_AF_TICKET], 1u);
    __syncthreads();
    ticket = ctl[AC_JOB];
    __syncthreads();
  }
  for (;;) {
    // ---- (a share of) a row
    const uint32_t j = ticket / parts, part = ticket & (parts - 1u);
    if (j >= n_jobs) break;
    const uint32_t row = S.jobs[j];
    const uint32_t* chart = S.arena + S.row_chart[row];
    uint32_t* const mask = S.mask_rows + (size_t)S.row_mask[row] * G.Wm;
    AfChart J;
    const uint32_t ahead = tid < A.ahead ? chart[tid] : 0u;  // (asked for together with the header)
    J.m = chart[CH_SETS];
    const uint32_t chart_words = chart[CH_WORDS];
    const bool accepting = (chart[CH_FLAGS] & CHART_ACCEPTING) != 0u;
    J.off = chart + CH_HDR;
    if (chart_words <= AF_STAGE) {
      if (tid < A.ahead) stage[tid] = ahead;
      for (uint32_t i = A.ahead + tid; i < chart_words; i += AF_THREADS) stage[i] = chart[i];
      J.off = stage + CH_HDR;
    }
    J.items = J.off + J.m + 1u;
    auto eos_word = [&](uint32_t i) -> uint32_t { return (accepting && G.eos >= 0 && i == (uint32_t)G.eos >> 5) ? 1u << ((uint32_t)G.eos & 31u) : 0u; };
    if (parts > 1u && part == 0u) {  // the mask is cleared first: the other blocks of the row wait for that
      for (uint32_t i = tid; i < G.Wm; i += AF_THREADS) mask[i] = eos_word(i);
      __threadfence();
    }
    for (uint32_t i = tid; i < AF_SEEN; i += AF_THREADS) seen[i] = 0ull;
    if (tid < AC_WORDS) ctl[tid] = 0u;
    if (tid < AF_CTX_HASH) C0.hash[tid] = 0u;
    __syncthreads();
    if (warp == 0) {  // the kernel of the chart's last set
      if (lane < 4u) deal_clear(lane < 2u ? edge_deal(lane) : token_deal(lane - 2u));
      const uint32_t lo = J.off[J.m - 1u], hi = J.off[J.m], self = J.m - 1u;
      uint32_t* b = hi - lo <= AF_BUF ? buf : big_area(A) + A.big_cap / 4u + A.big_cap / 2u;
      uint32_t n = 0, mine = 0;
      bool ok = hi - lo <= A.big_cap;
      if (ok)
        for (uint32_t base = lo; base < hi; base += 32) {
          const uint32_t k = base + lane;
          const uint32_t it = k < hi ? J.items[k] : 0u;
          bool take = k < hi && ((it >> 16) != self || (it & 0xFFFFu) == ITEM_START);
          if (take) take = (__ldg(&G.ga_item[2u * (it & 0xFFFFu) + 1u]) & GA_ALIVE) != 0u;
          if (take && k > lo && (it & 0xFFFFu) != 0u && J.items[k - 1u] == it - 1u)  // the item before it skips to it
            take = !(__ldg(&G.ga_item[2u * ((it & 0xFFFFu) - 1u) + 1u]) & GA_SKIPS);
          const uint32_t bal = __ballot_sync(FULL, take);
          if (take) b[n + __popc(bal & lt)] = (it << 16) | (it >> 16);
          n += __popc(bal);
        }
      __syncwarp();
      uint2 list = make_uint2(0u, 0u);
      Contexts C = C0;
      if (lane < n) mine = b[lane];
      bool grouped = n <= 32u && group_lanes(G, C, ctl, mine, n, list);
      if (!grouped && ok && !(ok = group_items(G, C, ctl, b, n, list))) {
        spill_contexts(C, ctl, A);
        ok = group_items(G, C, ctl, b, n, list);  // (sorted and without repeats already)
      }
      if (lane == 0) {
        ctl[AC_LIST] = list.x, ctl[AC_LIST_END] = list.y;
        if (!ok) ctl[AC_FAIL] = 1u + DIAG_SET_SCRATCH;
      }
    } else if (tid == AF_THREADS - 1) {
      ctl[AC_BEGAN] = (uint32_t)(clock64() >> 10);
      if (parts > 1u && part == 0u) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(A.row_begun + j), "r"(S.gen) : "memory");
      if (part)  // the block that began with the row clears the mask
        for (uint32_t polls = 0; ld_acquire(A.row_begun + j) != S.gen; ++polls) {
          if (polls > poll_limit(S, 22)) {
            diag(S, DIAG_WAIT_GRID);
            atomicExch(&S.counters[CNT_BAR_ERR], 1u);
            ctl[AC_FAIL] = AF_GIVEN_UP;
            break;
          }
          if (polls) __nanosleep(64);
        }
    }
    __syncthreads();

    bool spilled = false;
    // the expansion of a context (offset into pool, count), and its elements
    auto expansion = [&](uint32_t c) -> uint2 { return spilled ? global_contexts(A).exp[c] : C0.exp[c]; };
    auto element = [&](uint32_t at) -> uint32_t { return spilled ? global_contexts(A).pool[at] : C0.pool[at]; };
    // false: these edges were listed with this context a moment ago
    auto fresh = [&](uint32_t edge, uint32_t ctx) -> bool {
      const uint32_t slot = (edge * 0x9E3779B1u ^ ctx * 0x85EBCA6Bu) >> 23;
      static_assert(AF_SEEN == 512, "the slot is the upper nine bits");
      const unsigned long long key = (unsigned long long)(edge + 1u) << 32 | ctx;
      volatile unsigned long long* p = seen + slot;
      const bool yes = *p != key;
      *p = key;
      return yes;
    };
    auto expand_all = [&](const Deal& D, uint32_t entries_of) {  // (by warp 0) the contexts of these entries
      Contexts C = ctl[AC_SPILLED] ? global_contexts(A) : C0;
      for (uint32_t base = 0; base < entries_of; base += 32) {
        const uint32_t c = base + lane < entries_of ? D.what[base + lane].y : CTX_NEW;
        for (uint32_t todo = __ballot_sync(FULL, c != CTX_NEW && C.exp[c].y == CTX_NEW); todo;) {
          const uint32_t x = __shfl_sync(FULL, c, __ffs(todo) - 1);
          if (!expand_context(G, A, C, J, x, ctl, work, hset, buf) && lane == 0) ctl[AC_FAIL] = 1u + DIAG_SET_TABLE;
          todo &= ~__ballot_sync(FULL, c == x);
        }
      }
    };
    uint32_t list_at = 0;  // items of the last set whose starts have been taken
    bool begun = false;
    for (uint32_t side = 0;; side ^= 1u) {  // ---- rounds
      const Deal E = edge_deal(side), N = edge_deal(side ^ 1u), T = token_deal(side);
      uint32_t n = dealt_lists(E), total = dealt_things(E), gtop = ctl[AC_GTOP];
      const uint32_t list_end = ctl[AC_LIST_END];
      if (ctl[AC_FAIL] || (n + gtop == 0u && begun && list_at == list_end)) break;
      spilled = ctl[AC_SPILLED] != 0u;
      if (parts > 1u && tid == AF_THREADS - 1) peek(ctl + AC_PEEK, A.row_gone + (j & ~3u));  // (looked at when the round ends)
      auto overflow = [&](uint32_t edge, uint32_t cnt, uint32_t ctx) {
        const uint32_t p = atomicAdd(&ctl[AC_OVF], 1u);
        if (gtop + p < A.stack_cap) stack[gtop + p] = make_uint4(edge, cnt, ctx, 0u);
        else ctl[AC_FULL] = 1u;  // (cannot happen, see below)
      };
      auto list_edges = [&](bool yes, uint32_t edge, uint32_t cnt, uint32_t ctx) {  // (by all lanes of a warp)
        const bool fits = deal(N, yes, min(cnt, AF_CHUNK), make_uint2(edge, ctx));
        if (yes && !fits) overflow(edge, cnt, ctx);
        else if (yes && cnt > AF_CHUNK) overflow(edge + AF_CHUNK, cnt - AF_CHUNK, ctx);
      };
      auto list_tokens = [&](uint32_t at, uint32_t cnt) {
        const bool fits = deal(T, cnt != 0u, cnt, make_uint2(at, 0u));
        if (__any_sync(FULL, !fits)) set_tokens(G, mask, at, fits ? 0u : cnt);
      };
      if (n + gtop == 0u) {
        // ---- the starts of the last set's items; blocks that share a row share their tokens and edges
        const uint32_t from = list_at, until = min(list_end, from + AF_SLICE);
        list_at = until, begun = true;
        for (uint32_t base = from; base == from || base < until; base += AF_THREADS) {
          const uint32_t i = base + tid;
          const uint32_t x = i < until ? element(ctl[AC_LIST] + i) : 0u;
          uint4 r = i < until ? __ldg(reinterpret_cast<const uint4*>(G.ga_start) + (x >> 16)) : make_uint4(0u, 0u, 0u, 0u);
          if (r.y == GA_MASK) wide[atomicAdd(&ctl[AC_NWIDE], 1u)] = r.x, r.y = 0u;
          __syncthreads();
          // what is valid from the items with masks, four words of a thread under way at once
          const uint32_t nw = ctl[AC_NWIDE], step = parts * AF_THREADS;
          if (tid == 0) looked_up += nw * (G.Wm / parts);
          if (nw || base == 0u)
            for (uint32_t i4 = part * AF_THREADS + tid; i4 < G.Wm; i4 += 4u * step) {
              uint32_t v[4];
#pragma unroll
              for (uint32_t u = 0; u < 4; ++u) v[u] = 0u;
              for (uint32_t k = 0; k < nw; ++k) {
                const uint32_t* src = G.ga_mask + (size_t)wide[k] * G.Wm;
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) v[u] |= i4 + u * step < G.Wm ? __ldg(src + i4 + u * step) : 0u;
              }
#pragma unroll
              for (uint32_t u = 0; u < 4; ++u) {
                if (i4 + u * step >= G.Wm) continue;
                if (parts == 1u && base == 0u) mask[i4 + u * step] = v[u] | eos_word(i4 + u * step);
                else if (v[u]) atomicOr(&mask[i4 + u * step], v[u]);
              }
            }
          __syncthreads();
          if (tid == 0) ctl[AC_NWIDE] = 0u;
          if (r.y == 1u && part == 0u) atomicOr(&mask[r.x >> 5], 1u << (r.x & 31u));
          const uint32_t t0 = r.y > 1u ? (uint32_t)((uint64_t)r.y * part / parts) : 0u, t1 = r.y > 1u ? (uint32_t)((uint64_t)r.y * (part + 1u) / parts) : 0u;
          const uint32_t e0 = (uint32_t)((uint64_t)r.w * part / parts), e1 = (uint32_t)((uint64_t)r.w * (part + 1u) / parts);
          list_tokens(r.x + t0, t1 - t0);
          list_edges(e1 > e0, r.z + e0, e1 - e0, x & 0xFFFFu);
          looked_up += t1 - t0 + (r.y == 1u ? 1u : 0u);
          __syncthreads();
        }
      } else {
        // The stack cannot run over: a round takes no more edges than there are places above the reserve, and lists what follows from
        // one of them at most once.  On a crowded stack one entry is taken at a time, from the top, and a few of its edges: depth first
        // the stack grows along one path of the trie.
        const uint32_t places = A.stack_cap - min(gtop + A.reserve, A.stack_cap);
        if (places < AF_TIGHT) {
          for (uint32_t i = tid; i < n; i += AF_THREADS) {
            const uint2 w = E.what[i];
            stack[gtop + i] = make_uint4(w.x, (i + 1u < n ? E.pre[i + 1u] : total) - E.pre[i], w.y, 0u);
          }
          __syncthreads();
          gtop += n - 1u;
          const uint4 v = stack[gtop];
          total = min(v.y, AF_TIGHT_EDGES), n = 1u;
          __syncthreads();
          if (tid == 0) {
            E.what[0] = make_uint2(v.x, v.z), E.pre[0] = 0u, E.owner[0] = 0u;
            if (v.y > total) stack[gtop] = make_uint4(v.x + total, v.y - total, v.z, 0u);
          }
          if (v.y > total) ++gtop;
          __syncthreads();
          if (warp == 0) expand_all(E, 1u);
          __syncthreads();
          spilled = ctl[AC_SPILLED] != 0u;
        } else if (places < total) {
          for (uint32_t i = tid; i < n; i += AF_THREADS) {
            const uint2 w = E.what[i];
            const uint32_t first = E.pre[i], end = i + 1u < n ? E.pre[i + 1u] : total;
            if (end > places) overflow(w.x + (max(first, places) - first), end - max(first, places), w.y);
          }
          total = places;
        }
        // ---- the edges
        if (tid == 0) looked_up += total;
        for (uint32_t base = warp * 32u; base < total; base += AF_THREADS) {
          const uint32_t e = whose(E, n, base);
          uint4 g = make_uint4(0u, 0u, 0u, 0u);
          uint32_t to = CTX_NEW;
          if (base + lane < total) {
            const uint2 w = E.what[e];
            g = __ldg(reinterpret_cast<const uint4*>(G.ga_edge) + w.x + (base + lane - E.pre[e]));
            const uint2 x = expansion(w.y);
            uint32_t lo = 0, hi = x.y;
            while (lo < hi) {
              const uint32_t mid = (lo + hi) >> 1;
              if ((element(x.x + mid) >> 16) < (g.x >> 16)) lo = mid + 1u;
              else hi = mid;
            }
            const uint32_t el = lo < x.y ? element(x.x + lo) : 0xFFFFFFFFu;
            if ((el >> 16) == (g.x >> 16) && lo < x.y) to = el & 0xFFFFu;
          }
          const uint32_t cnt = to != CTX_NEW ? g.x & 0xFFFFu : 0u;
          looked_up += cnt;
          if (cnt == 1u) atomicOr(&mask[g.y >> 5], 1u << (g.y & 31u));
          __syncwarp();
          list_tokens(g.y, cnt > 1u ? cnt : 0u);
          list_edges(to != CTX_NEW && g.w && fresh(g.z, to), g.z, g.w, to);
        }
      }
      __syncthreads();
      if (warp == 0) {
        // ---- entries from the stack, as far as there is room, and the expansions that the next round needs
        gtop += ctl[AC_OVF];
        __syncwarp();
        if (lane == 0) ctl[AC_OVF] = 0u, deal_clear(E);
        if (lane == 1u) deal_clear(token_deal(side ^ 1u));
        __syncwarp();
        while (gtop && A.stack_cap - min(gtop + A.reserve, A.stack_cap) >= AF_TIGHT && N.count[1] < AF_BATCH / 2u && N.count[0] < AF_EDGES / 2u) {
          const uint32_t take = min(gtop, 32u);
          const uint4 v = lane < take ? stack[gtop - 1u - lane] : make_uint4(0u, 0u, 0u, 0u);
          __syncwarp();
          gtop -= take;
          list_edges(lane < take, v.x, v.y, v.z);
          __syncwarp();
          gtop += ctl[AC_OVF];
          __syncwarp();
          if (lane == 0) ctl[AC_OVF] = 0u;
          __syncwarp();
        }
        if (lane == 0) {
          ctl[AC_GTOP] = gtop;
          if (ctl[AC_FULL]) ctl[AC_FAIL] = 1u + DIAG_QUEUE_FULL;
        }
        expand_all(N, dealt_lists(N));
      } else {
        // ---- tokens, meanwhile
        const uint32_t nt = dealt_lists(T), tt = dealt_things(T);
        for (uint32_t base = (warp - 1u) * 32u; base < tt; base += 4u * (AF_THREADS - 32u)) {
          uint32_t tok[4];
#pragma unroll
          for (uint32_t u = 0; u < 4; ++u) {
            const uint32_t at = base + u * (AF_THREADS - 32u);
            tok[u] = 0xFFFFFFFFu;
            if (at >= tt) continue;
            const uint32_t e = whose(T, nt, at);
            if (at + lane < tt) tok[u] = __ldg(&G.ga_tok[T.what[e].x + (at + lane - T.pre[e])]);
          }
#pragma unroll
          for (uint32_t u = 0; u < 4; ++u)
            if (tok[u] != 0xFFFFFFFFu) atomicOr(&mask[tok[u] >> 5], 1u << (tok[u] & 31u));
        }
        if (tid == AF_THREADS - 1) {
          asm volatile("cp.async.wait_all;" ::: "memory");
          const bool gone = parts > 1u && ctl[AC_PEEK + (j & 3u)] == S.gen, late = (uint32_t)(clock64() >> 10) - ctl[AC_BEGAN] > AF_KCYCLES;
          if ((gone || late) && !ctl[AC_FAIL]) ctl[AC_FAIL] = gone ? AF_GONE : AF_LATE;
        }
      }
      __syncthreads();
    }
    contexts += ctl[AC_NCTX];
    if (ctl[AC_FAIL] && ctl[AC_FAIL] != AF_GONE && ctl[AC_FAIL] != AF_GIVEN_UP) {  // too many contexts, or too long a time: the row is left to a sweep by Earley steps
      gave_up = true;
      if (tid == 0) {
        if (ctl[AC_FAIL] != AF_LATE) diag(S, ctl[AC_FAIL] - 1u);
        if (atomicExch(A.row_gone + j, S.gen) != S.gen)  // (its other blocks stop when they see that)
          *reinterpret_cast<volatile uint32_t*>(A.given + atomicAdd(&S.counters[CNT_AF_GIVEN], 1u)) = S.gen << 16 | j;
      }
    }
    // ---- the next row
    __threadfence();
    if (gridDim.x >= n_jobs * parts) break;
    __syncthreads();
    if (tid == 0) ctl[AC_JOB] = gridDim.x + atomicAdd(&S.counters[CNT_AF_TICKET], 1u);
    __syncthreads();
    ticket = ctl[AC_JOB];
    __syncthreads();
  }
  looked_up = __reduce_add_sync(FULL, looked_up);
  __syncthreads();
  if (lane == 0 && looked_up) atomicAdd(&ctl[AC_LOOKED], looked_up);
  __syncthreads();
  if (tid == 0) {
    stat_add(S, CNT_STAT_TRANS, ctl[AC_LOOKED]);
    stat_add(S, CNT_STAT_LOCAL, contexts);
  }
  // ---- rows that were given up, swept by the blocks that gave them up when they have no row left.  Only blocks that look for tables
  // wait, and who has tables waits for nobody.
  while (gave_up) {
    __syncthreads();
    if (tid == 0) {
      uint32_t at = vload(&S.counters[CNT_AF_GIVEN_TAKEN]), got = 0xFFFFFFFFu, slot = 0xFFFFFFFFu;
      while (at < ld_acquire(&S.counters[CNT_AF_GIVEN])) {
        const uint32_t was = atomicCAS(&S.counters[CNT_AF_GIVEN_TAKEN], at, at + 1u);
        if (was == at) {
          got = at;
          break;
        }
        at = was;
      }
      if (got != 0xFFFFFFFFu) {
        uint32_t k = blockIdx.x % A.sweep_slots, v = 0u;
        for (uint32_t polls = 0; slot == 0xFFFFFFFFu; ++polls, k = (k + 1u) % A.sweep_slots) {
          if ((v >> 16) != S.gen) v = vload(A.given + got);  // (written right after its number was drawn)
          if ((v >> 16) == S.gen && atomicCAS(A.sweep_lock + k, 0u, 1u) == 0u) slot = k;
          else if (ld_acquire(&S.counters[CNT_BAR_ERR])) break;
          else if (polls > poll_limit(S, 22)) {
            diag(S, DIAG_WAIT_VALUE);
            atomicExch(&S.counters[CNT_BAR_ERR], 1u);
            break;
          } else {
            __nanosleep(400);
          }
        }
        ctl[AC_SLOT] = v & 0xFFFFu;
        __threadfence();
      }
      ctl[AC_JOB] = slot;
    }
    __syncthreads();
    const uint32_t slot = ctl[AC_JOB], row = slot == 0xFFFFFFFFu ? 0u : S.jobs[ctl[AC_SLOT]];
    __syncthreads();
    if (slot == 0xFFFFFFFFu) break;
    // (copies: if the parameters themselves were passed by reference, the rounds above would read them anew each time they are used; 12
    // steps of 128 rows of SQL 5.42 ms, with copies 5.22)
    const GrammarDev g = G;
    const StateDev s = S;
    const bool ok = sweep_row_by_block(g, s, row, slot, smem);
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      atomicExch(A.sweep_lock + slot, 0u);
      stat_add(S, CNT_STAT_SWEPT, 1u);
      if (!ok) {  // a capacity was exceeded there, too: the row's mask cannot be trusted
        diag(S, DIAG_SET_SCRATCH);
        if (!(atomicOr(&S.row_flags[row], ROW_BROKEN) & ROW_BROKEN)) stat_add(S, CNT_STAT_CAPERR, 1u);
        atomicExch(&S.counters[CNT_ERR], 1u);
      }
    }
  }
}

// ===================================================================================== launchers

constexpr uint32_t AF_SMEM = (2 * AF_BATCH + AF_LISTS + AF_SEEN) * 8 + (5 * AF_CTX + AF_POOL + AF_CTX_HASH + 2 * AF_BATCH + AF_LISTS + AC_WORDS + AF_THREADS + AF_STAGE + AF_BUF + AF_WORK + AF_HSET) * 4 +
                             (2 * AF_EDGES + AF_TOKENS) / 32 * 2;
constexpr uint32_t AF_SWEEP_SMEM = block_sweep_words(AF_WARPS, MAX_NONTERMINALS / 32u) * 4u;  // a row that is given up is swept in the same shared memory
constexpr uint32_t AF_SMEM_ASKED = AF_SMEM > AF_SWEEP_SMEM ? AF_SMEM : AF_SWEEP_SMEM;

// Places of a block's stack that only its depth-first rounds use - what is left of an entry and what its edges start, along the longest
// path of the trie - and the entries of a round that are put back.
uint32_t automaton_fill_reserve() { return (MAX_TOKEN_BYTES + 2u) * (2u * AF_TIGHT_EDGES + 2u) + 3u * AF_BATCH; }
uint32_t automaton_fill_warps() { return AF_WARPS; }
uint32_t automaton_fill_least_stack() { return automaton_fill_reserve() + AF_TIGHT + AF_SLICE; }

void automaton_fill_layout(const GrammarDev& G, uint32_t rows, uint32_t max_blocks, AutoFillDev& A) {
  A.reserve = automaton_fill_reserve();
  A.scratch_words = 7u * A.ctx_cap + A.pool_cap + A.big_cap / 4u + A.big_cap / 2u + A.big_cap;
  // few rows: several blocks take one, so that the chip is filled (a small trie gives the others nothing to do)
  A.parts = 1;
  while (A.parts < 8u && (uint64_t)rows * A.parts * 2u <= max_blocks && A.parts * 2048u <= G.T) A.parts *= 2u;
  A.grid = (uint32_t)std::min<uint64_t>(max_blocks, (uint64_t)rows * A.parts);
}

cudaError_t configure_automaton_fill() {
  return cudaFuncSetAttribute((const void*)automaton_fill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AF_SMEM_ASKED);
}

void launch_automaton_fill(const GrammarDev& G, const StateDev& S, cudaStream_t st) {
  launch_overlapped(automaton_fill_kernel, dim3(S.af.grid), dim3(AF_THREADS), AF_SMEM_ASKED, st, G, S);
}

}  // namespace fmt
