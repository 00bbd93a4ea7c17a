// The fill of rows' masks by what the grammar automaton tabulates (grammar_automaton.cpp; Sections 3.3, 4.1, 4.3 of the paper).
//
// A thread block takes a row.  The kernel items of the chart's last set are grouped by dotted rule; each group has a CONTEXT, the set
// of origins its items were begun in, and the record of what follows from the item (its start): the tokens that are valid whatever
// the chart holds, and edges for the places inside tokens where the item's rule ends.  There the chart is asked: the context is
// EXPANDED, once per row, into the items that waited in its origins, completed upwards (Section 3.2's Complete), grouped
// in the same way.  An edge whose item is among them sets its own tokens, and its edges go on with that group's context.  A
// round takes all edges that are known, looks their items up in the contexts' expansions, and lists the edges of those that are found.
//
// A block decides by itself where its row's mask comes from (the state cache, another row of the call, or from here): a kernel that listed
// the rows to be filled took longer than most of the rows do.
//
// What bounds it: latency, 35,000 cycles for a row of JSON.  About 2,500 until the chart is there, 5,000 for the contexts of its items, 5,000 for
// the starts and their masks, and a few rounds (as many as rules end one after the other inside a token) of 2,500 to 3,500 each: a
// read of edges, a search, the sums that deal lists out to the lanes, and two barriers.  Fills on a B200 by a walk of the trie over byte
// classes, a byte a round; by edges with eight blocks to a row, each with its own contexts; and now, us (the last: 254 to 282 on one B200 and
// another):
//   37 rows of JSON, 50,001 tokens                      139     65     33
//   24 charts of JSON, 32,000 tokens, no allocations    123     71     39
//   256 rows of ambiguous JSON, 128,256 tokens        1,010    790    265
// and with all that goes with it, 12 decoding steps of 128 rows of SQL, 152,064 tokens, 4.93, 2.33 and 2.10 ms, 16 of 64 rows of a JSON
// schema, 128,256 tokens, 2.44, 1.52 and 1.37 ms, 24 of 8 rows of JSON 3.58, 2.14 and 1.62 ms.
// Slower than by the walk of the trie, where up to eight blocks shared a row: text of braces whose every byte ends a rule (20,000
// lists of an edge or two go through a block's rounds), 1 and 4 rows 268 and 196 us then, 286 now; 64 and 256 rows 306 and 689 then, 290 and 313.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "block_sweep.cuh"
#include "sweep_warp.cuh"

namespace fmt {

constexpr int AF_WARPS = 8, AF_THREADS = AF_WARPS * 32;
constexpr uint32_t AF_BATCH = 512;        // entries (lists of edges with a context) of a round,
constexpr uint32_t AF_EDGES = 32768;      // edges of a round,
constexpr uint32_t AF_CHUNK = 1024;       // and of an entry
constexpr uint32_t AF_LISTS = 512, AF_TOKENS = 32768;  // lists of tokens that are written when a round's edges are through, and tokens in them
constexpr uint32_t AF_TIGHT = 2048;       // free places of a block's stack, its reserve not counted, below which entries are taken one at a time,
constexpr uint32_t AF_TIGHT_EDGES = 32;   // so many edges of them
constexpr uint32_t AF_SLICE = 1024;       // items of a last set whose starts are taken together
// Recently listed edges with their contexts (a lossy table: repeats only cost time).  256 rows of ambiguous JSON: 670 us a fill with 512
// of them, 330 with 4,096, 52,000 and 25,000 edges for the rows that take longest.
constexpr uint32_t AF_SEEN_BITS = 13, AF_SEEN = 1u << AF_SEEN_BITS;
constexpr uint32_t AF_STAGE = 768;        // a chart up to this many words is read from shared memory, with its items' records
constexpr uint32_t AF_ITEMS = AF_THREADS - 32;  // items of a chart whose contexts are made and expanded beforehand, an item to a thread
constexpr uint32_t AF_NODE = 24, AF_NODES = 1344;  // items of such an expansion, and of all of them, at most
constexpr uint32_t AF_QUEUE = 13;         // completions that such an expansion makes at most
constexpr uint32_t AF_SCAN = 256, AF_LANES = 4;  // items that a lane looks at to expand a context by itself, and contexts from which on lanes do
constexpr uint32_t AF_CTX = AF_ITEMS + 96, AF_CTX_HASH = 1024, AF_POOL = 3072;  // contexts in shared memory, words of their lists
constexpr uint32_t AF_BUF = 512, AF_WORK = 256, AF_HSET = 512;      // an expansion in shared memory (larger ones: global memory)
constexpr uint32_t AF_KCYCLES = 1u << 14;      // a row that takes longer (2^24 cycles, 8.5 ms) is given up for a sweep by Earley steps
// AC_FAIL: 0, 1 + the capacity that was exceeded, or
constexpr uint32_t AF_GIVEN_UP = 0xFFFFFFFFu;  // more rounds than a bounded wait has polls: the fill is given up, the row itself is fine
constexpr uint32_t AF_LATE = 0xFFFFFFFDu;      // the row takes too long
constexpr uint32_t CTX_NEW = 0xFFFFFFFFu;
constexpr uint32_t AF_FOUND = 1u << 31;        // an entry whose edges are all of one item, with that item's context

enum : uint32_t {
  AC_OVF = 0, AC_LATER = 1, AC_FAIL = 2, AC_NCTX = 3, AC_POOL = 4, AC_NWORK = 5, AC_NBUF = 6, AC_OVER = 7, AC_SPILLED = 8, AC_WANT = 9,
  AC_NWIDE = 10, AC_LIST = 11, AC_LIST_END = 12, AC_LOOKED = 13, AC_BEGAN = 14, AC_SLOT = 15,
  AC_EDGES = 16,   // [2] counters of the entries (see Deal)
  AC_TOKENS = 24,  // [2] and of the lists of tokens
  AC_FULL = 32, AC_CLEARED = 33, AC_ROW = 33, AC_MASK = 34,
  AC_CROWDED = 35, AC_CUT = 36,  // rounds of all the block's rows: those that took one entry at a time, and those that put edges back
  AC_ONE_BY_ONE = 37,            // the row's contexts are not for lanes
  AC_WORDS = 40
};
static_assert(AC_WORDS % 4 == 0 && AC_WORDS <= AF_THREADS, "what follows in shared memory is cleared in 16-byte pieces; a thread clears a word");

// Lists whose elements are dealt out to the lanes: places and elements are counted by one atomic operation, so that the places are in
// the order of the elements.
struct Deal {
  uint32_t* count;   // places << DEAL_SHIFT | elements; then the first place and the first element that found no room
  uint2* what;       // [cap] where the list begins, and what it comes with
  uint32_t* pre;     // [cap] its first element's number
  uint16_t* owner;   // [things / 32] the place of the list to which the element 32 * i belongs
  uint32_t cap, things;
};
// (a warp that finds the places taken counts nothing: 32 lists of each of eight warps go beyond at most)
constexpr uint32_t DEAL_SHIFT = 21, DEAL_THINGS = (1u << DEAL_SHIFT) - 1u;
static_assert(AF_BATCH + AF_THREADS < 1u << (32 - DEAL_SHIFT) && AF_LISTS + AF_THREADS < 1u << (32 - DEAL_SHIFT), "places of a deal");
static_assert(AF_EDGES + AF_THREADS * AF_CHUNK <= DEAL_THINGS && AF_TOKENS + AF_THREADS * GA_EDGE_TOKENS <= DEAL_THINGS, "elements of a deal");
__device__ __forceinline__ uint32_t dealt_lists(const Deal& D) { return min(D.count[0] >> DEAL_SHIFT, D.count[1]); }
__device__ __forceinline__ uint32_t dealt_things(const Deal& D) { return min(D.count[0] & DEAL_THINGS, D.count[2]); }
__device__ __forceinline__ void deal_clear(const Deal& D) {
  D.count[0] = 0u;
  D.count[1] = D.count[2] = 0xFFFFFFFFu;
}
// By one lane: places for `lists` lists with `things` elements in all, or 0xFFFFFFFF.
__device__ __forceinline__ uint32_t deal_take(const Deal& D, uint32_t lists, uint32_t things) {
  const uint32_t now = *reinterpret_cast<volatile uint32_t*>(D.count);
  return now >> DEAL_SHIFT < D.cap && (now & DEAL_THINGS) < D.things ? atomicAdd(D.count, lists << DEAL_SHIFT | things) : 0xFFFFFFFFu;
}
// By all lanes of a warp: the list of a lane with `yes`, its place and first element.  False: there is no room for it.
__device__ __forceinline__ bool deal_put(const Deal& D, bool yes, uint32_t slot, uint32_t before, uint32_t n, uint2 what) {
  const bool fits = slot < D.cap && before + n <= D.things, longer = n > 128u;
  if (yes && fits) {
    D.what[slot] = what;
    D.pre[slot] = before;
    if (!longer)
#pragma unroll 1
      for (uint32_t p = (before + 31u) / 32u; p * 32u < before + n; ++p) D.owner[p] = (uint16_t)slot;
  } else if (yes) {
    atomicMin(&D.count[1], slot);
    atomicMin(&D.count[2], before);
  }
#pragma unroll 1
  for (uint32_t m = __ballot_sync(FULL, yes && fits && longer); m; m &= m - 1u) {
    const int src = __ffs(m) - 1;
    const uint32_t from = __shfl_sync(FULL, before, src), until = from + __shfl_sync(FULL, n, src), s = __shfl_sync(FULL, slot, src);
#pragma unroll 1
    for (uint32_t p = (from + 31u) / 32u + lane_id(); p * 32u < until; p += 32u) D.owner[p] = (uint16_t)s;
  }
  return fits;
}
// By all lanes of a warp: the lanes' lists of nt tokens (at most GA_EDGE_TOKENS) and of ne edges (at most AF_CHUNK), 0 if a lane has none, go
// to T and N.  Returns 1 if there is no room for a lane's tokens, 2 if there is none for its edges.
__device__ __forceinline__ uint32_t deal_both(const Deal& T, const Deal& N, uint32_t nt, uint32_t tokens, uint32_t ne, uint2 edges) {
  const uint32_t lane = lane_id(), lt = (1u << lane) - 1u, bt = __ballot_sync(FULL, nt != 0u), be = __ballot_sync(FULL, ne != 0u);
  if ((bt | be) == 0u) return 0u;
  static_assert(32u * GA_EDGE_TOKENS < 65536u && 32u * AF_CHUNK < 65536u, "two sums in a word");
  uint32_t incl = ne << 16 | nt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t t = __shfl_up_sync(FULL, incl, d);
    if ((int)lane >= d) incl += t;
  }
  uint32_t base_t = 0xFFFFFFFFu, base_e = 0xFFFFFFFFu;
  if (lane == 31u && bt) base_t = deal_take(T, __popc(bt), incl & 0xFFFFu);
  if (lane == 31u && be) base_e = deal_take(N, __popc(be), incl >> 16);
  uint32_t none = 0u;
  if (bt) {
    base_t = __shfl_sync(FULL, base_t, 31);
    const bool ok = base_t != 0xFFFFFFFFu && deal_put(T, nt != 0u, (base_t >> DEAL_SHIFT) + __popc(bt & lt), (base_t & DEAL_THINGS) + (incl & 0xFFFFu) - nt, nt, make_uint2(tokens, 0u));
    if (nt && !ok) none |= 1u;
  }
  if (be) {
    base_e = __shfl_sync(FULL, base_e, 31);
    const bool ok = base_e != 0xFFFFFFFFu && deal_put(N, ne != 0u, (base_e >> DEAL_SHIFT) + __popc(be & lt), (base_e & DEAL_THINGS) + (incl >> 16) - ne, ne, edges);
    if (ne && !ok) none |= 2u;
  }
  return none;
}
// The list to which element base + lane of n lists belongs (base a multiple of 32).
__device__ __forceinline__ uint32_t whose(const Deal& D, uint32_t n, uint32_t base) {
  const uint32_t lane = lane_id(), lo = D.owner[base / 32u];
  const uint32_t nb = lo + 1u + lane < n ? D.pre[lo + 1u + lane] - base : 32u;  // where the lists after it begin
  const uint32_t starts = __reduce_or_sync(FULL, nb < 32u ? 1u << nb : 0u);
  return lo + __popc(starts & (0xFFFFFFFFu >> (31u - lane)));
}

// Shared memory, in words.
enum : uint32_t {
  SM_ENTRIES = 0,                                // [2][AF_BATCH] uint2, in turn: first edge, context
  SM_LISTS = SM_ENTRIES + 4 * AF_BATCH,          // [AF_LISTS] uint2: where in ga_tok
  SM_SEEN = SM_LISTS + 2 * AF_LISTS,             // [AF_SEEN]
  SM_RECS = SM_SEEN + AF_SEEN,               // [AF_STAGE] uint2: ga_item of the chart's items
  SM_ORG = SM_RECS + 2 * AF_STAGE,               // contexts (see Contexts)
  SM_EXP = SM_ORG + 2 * AF_CTX,
  SM_LHS = SM_EXP + 2 * AF_CTX,
  SM_POOL = SM_LHS + AF_CTX,
  SM_HASH = SM_POOL + AF_POOL,
  SM_PRE = SM_HASH + AF_CTX_HASH,                // [2][AF_BATCH], [AF_LISTS]
  SM_CTL = SM_PRE + 2 * AF_BATCH + AF_LISTS,
  SM_LINK = SM_CTL + AC_WORDS,                   // [AF_THREADS] per item of the chart: see enter_items
  SM_REP = SM_LINK + AF_THREADS,                 // [AF_THREADS] 16 bits: the context of its rule and origin
  SM_WIDE = SM_REP + AF_THREADS / 2,             // [AF_THREADS] rows of ga_mask
  SM_STAGE = SM_WIDE + AF_THREADS,               // [AF_STAGE] the chart
  SM_BUF = SM_STAGE + AF_STAGE,                  // expansions that do not fit a warp's lanes
  SM_WORK = SM_BUF + AF_BUF,
  SM_HSET = SM_WORK + AF_WORK,
  SM_OWNER = SM_HSET + AF_HSET,                  // 16 bits each: [2][AF_EDGES / 32], [AF_TOKENS / 32]
  SM_WORDS = SM_OWNER + (2 * AF_EDGES + AF_TOKENS) / 64
};
extern __shared__ __align__(16) uint32_t smem[];
// All warps but the first.
__device__ __forceinline__ void others_meet() { asm volatile("bar.sync 1, %0;" ::"n"(AF_THREADS - 32) : "memory"); }

// The contexts of the row a block works on: in shared memory, or, when they outgrow it, in global memory of the block's own.
struct Contexts {
  uint2* org;       // [cap] origins: offset into pool, count
  uint2* exp;       // [cap] expansion: offset into pool, count (CTX_NEW: not made yet); rule << 16 | context, ascending if there are more than AF_NODE
  uint32_t* lhs;    // [cap] the non-terminal whose rule is open
  uint32_t* hash;   // [hash_mask + 1] context + 1, 0 = empty
  uint32_t* pool;
  uint32_t cap, hash_mask, pool_cap;
};
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
__device__ __forceinline__ Contexts shared_contexts() {
  Contexts C;
  C.org = reinterpret_cast<uint2*>(smem + SM_ORG), C.exp = reinterpret_cast<uint2*>(smem + SM_EXP);
  C.lhs = smem + SM_LHS, C.hash = smem + SM_HASH, C.pool = smem + SM_POOL;
  C.cap = AF_CTX, C.hash_mask = AF_CTX_HASH - 1u, C.pool_cap = AF_POOL;
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
  #pragma unroll 1
  for (uint32_t i = lane_id(); i < n; i += 32) h += mix32((list[i] & 0xFFFFu) + 1u);
  return mix32(__reduce_add_sync(FULL, h) + lhs * 0x9E3779B9u + n);
}

// The context (lhs, list[0..n) & 0xFFFF) (ascending): its number, or CTX_NEW when there is no room.
__device__ uint32_t intern_context(const Contexts& C, uint32_t* ctl, uint32_t lhs, const uint32_t* list, uint32_t n) {
  const uint32_t lane = lane_id();
  uint32_t slot = context_hash(lhs, list, n) & C.hash_mask;
  #pragma unroll 1
  for (;;) {
    const uint32_t v = C.hash[slot];
    if (v == 0u) break;
    const uint2 o = C.org[v - 1u];
    bool same = o.y == n && C.lhs[v - 1u] == lhs;
    if (same)
      #pragma unroll 1
      for (uint32_t i = lane; i < n; i += 32) same = same && C.pool[o.x + i] == (list[i] & 0xFFFFu);
    if (__all_sync(FULL, same)) return v - 1u;
    slot = (slot + 1u) & C.hash_mask;
  }
  const uint32_t id = ctl[AC_NCTX], at = ctl[AC_POOL];
  __syncwarp();
  if (id >= C.cap || n > C.pool_cap - at) return CTX_NEW;
  #pragma unroll 1
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
__device__ __noinline__ void spill_contexts(Contexts& C, uint32_t* ctl, const AutoFillDev& A) {
  const uint32_t lane = lane_id(), n = ctl[AC_NCTX], words = ctl[AC_POOL];
  const Contexts D = global_contexts(A);
  #pragma unroll 1
  for (uint32_t i = lane; i < n; i += 32) D.org[i] = C.org[i], D.exp[i] = C.exp[i], D.lhs[i] = C.lhs[i];
  #pragma unroll 1
  for (uint32_t i = lane; i < words; i += 32) D.pool[i] = C.pool[i];
  #pragma unroll 1
  for (uint32_t i = lane; i <= D.hash_mask; i += 32) D.hash[i] = 0u;
  __syncwarp();
  #pragma unroll 1
  for (uint32_t c = lane; c < n; c += 32) {  // (none is compared: a repeat, of a chart of few items, does as well)
    const uint2 o = D.org[c];
    uint32_t h = 0;
    #pragma unroll 1
    for (uint32_t i = 0; i < o.y; ++i) h += mix32(D.pool[o.x + i] + 1u);
    #pragma unroll 1
    for (uint32_t slot = mix32(h + D.lhs[c] * 0x9E3779B9u + o.y) & D.hash_mask; atomicCAS(&D.hash[slot], 0u, c + 1u) != 0u;) slot = (slot + 1u) & D.hash_mask;  // (as context_hash has it)
  }
  __syncwarp();
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
    #pragma unroll 1
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
    #pragma unroll 1
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
  #pragma unroll 1
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
__device__ __noinline__ bool group_items(const GrammarDev& G, const Contexts& C, uint32_t* ctl, uint32_t* buf, uint32_t n, uint2& out) {
  const uint32_t lane = lane_id();
  uint32_t groups;
  const uint32_t k = sort_unique(buf, n, groups);
  const uint32_t at = ctl[AC_POOL];
  __syncwarp();
  if (at + groups > C.pool_cap) return false;
  if (lane == 0) ctl[AC_POOL] = at + groups;
  __syncwarp();
  uint32_t g = 0;
  #pragma unroll 1
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
    #pragma unroll 1
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
__device__ __forceinline__ bool group_lanes(const uint32_t* ga_item, const Contexts& C, uint32_t* ctl, uint32_t item, uint32_t n, uint2& out) {
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
  const uint32_t lhs = leads ? __ldg(&ga_item[2u * d]) & 0xFFFFu : 0u;
  uint32_t ctx = CTX_NEW;
  if (__any_sync(FULL, leads && size == 1u)) {
    ctx = intern_singles(C, ctl, leads && size == 1u, lhs, item & 0xFFFFu);
    if (__any_sync(FULL, leads && size == 1u && ctx == CTX_NEW)) return false;
  }
  #pragma unroll 1
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

__device__ __noinline__ bool group_shared(const uint32_t* ga_item, uint32_t item, uint32_t n, uint2& out) {
  return group_lanes(ga_item, shared_contexts(), smem + SM_CTL, item, n, out);
}

// Complete upwards from the origins of context c: what waits there, with the dot moved.
__device__ __noinline__ bool expand_into(const GrammarDev& G, const Contexts& C, const AfChart& J, uint32_t c, uint32_t* ctl, uint32_t* work,
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
  #pragma unroll 1
  for (uint32_t i = lane; i < org.y; i += 32) need(lhs, C.pool[org.x + i]);
  #pragma unroll 1
  for (uint32_t head = 0;; ++head) {
    __syncwarp();
    const uint32_t n = ctl[AC_NWORK], over = ctl[AC_OVER];
    __syncwarp();
    if (over) return false;
    if (head >= n) break;
    const uint32_t a = work[head] >> 16, o = work[head] & 0xFFFFu;
    const uint32_t lo = J.off[o], hi = J.off[o + 1u];
    #pragma unroll 1
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

// The same with everything in the warp's lanes and the chart and the contexts in shared memory: one context of at most 32 origins, at most
// 32 completions and 32 items.  The general form takes some four times as many
// instructions.  False: it does not fit (nothing has changed but the pool's top).  (Not inlined, as the code of a fill is run
// once or twice, and what is fetched for it takes longer than what is executed.)
__device__ __noinline__ bool expand_shared(const uint32_t* ga_item, uint32_t m, uint32_t c) {
  const uint32_t *off = smem + SM_STAGE + CH_HDR, *items = off + m + 1u;
  const uint2* recs = reinterpret_cast<const uint2*>(smem + SM_RECS);
  uint32_t* const ctl = smem + SM_CTL;
  const Contexts C = shared_contexts();
  const uint32_t lane = lane_id();
  const uint2 org = C.org[c];
  if (org.y > 32u) return false;
  uint32_t work = lane < org.y ? C.lhs[c] << 16 | C.pool[org.x + lane] : 0u, nw = org.y;  // lane l: completion l
  uint32_t item = 0u, ni = 0u;                                                           // lane l: item l
  #pragma unroll 1
  for (uint32_t head = 0; head < nw; ++head) {
    const uint32_t key = __shfl_sync(FULL, work, head);
    const uint32_t a = key >> 16, o = key & 0xFFFFu;
    const uint32_t lo = off[o], hi = off[o + 1u];
    #pragma unroll 1
    for (uint32_t base = lo; base < hi; base += 32) {
      const uint32_t k = base + lane;
      const uint32_t it = k < hi ? items[k] : 0u;
      const uint2 rec = k < hi ? recs[k] : make_uint2(0xFFFF0000u, 0xFFFFu);
      const bool match = (rec.x >> 16) == a;
      uint32_t on = __ballot_sync(FULL, match && (rec.y & GA_GOES_ON)), up = __ballot_sync(FULL, match && (rec.y & 0xFFFFu) != 0xFFFFu);
      if (ni + __popc(on) > 32u) return false;
      const uint32_t x = ((it & 0xFFFFu) + 1u) << 16 | (it >> 16), y = (rec.y << 16) | (it >> 16);
      #pragma unroll 1
      for (; on; on &= on - 1u) {
        const uint32_t v = __shfl_sync(FULL, x, __ffs(on) - 1);
        if (__ballot_sync(FULL, lane < ni && item == v)) continue;
        if (lane == ni) item = v;
        ++ni;
      }
      #pragma unroll 1
      for (; up; up &= up - 1u) {
        const uint32_t v = __shfl_sync(FULL, y, __ffs(up) - 1);
        if (__ballot_sync(FULL, lane < nw && work == v)) continue;
        if (nw == 32u) return false;
        if (lane == nw) work = v;
        ++nw;
      }
    }
  }
  uint2 list = make_uint2(0u, 0u);
  if (ni) {
    if (ctl[AC_NCTX] + ni > C.cap) return false;
    if (!group_shared(ga_item, item, ni, list)) return false;
  }
  if (lane == 0) C.exp[c] = list;
  __syncwarp();
  return true;
}

// Contexts of one origin, a lane for each (CTX_NEW: none): the lanes look through the sets that their completions lead to, then the warp enters
// what each has found.  Those that have more than AF_NODE items or AF_QUEUE completions, or items of one rule begun in several
// sets, and those for which there is no room stay as they were.  One after the other, by the whole warp, the contexts of 64 charts
// of 20 kinds of brackets, 20 deep (some 800 items, 240 contexts), took 1,500 us a fill, now 820; below four at a time the warp is as fast.
__device__ __noinline__ void expand_by_lanes(const uint32_t* ga_item, const Contexts& C, const AfChart& J, bool staged, uint32_t* ctl, uint32_t c) {
  const uint32_t lane = lane_id();
  const uint2* recs = reinterpret_cast<const uint2*>(smem + SM_RECS);
  uint32_t* const found = smem + SM_BUF;  // [AF_NODE][32] rule << 16 | origin
  static_assert(32u * AF_NODE <= AF_BUF + AF_WORK, "what the lanes have found");
  uint32_t queue[AF_QUEUE], nq = 0, cnt = 0, left = AF_SCAN;  // what has been completed, non-terminal << 16 | origin
  bool fits = c != CTX_NEW;
  if (fits) queue[nq++] = C.lhs[c] << 16 | C.pool[C.org[c].x];
#pragma unroll 1
  for (uint32_t head = 0; fits && head < nq; ++head) {
    const uint32_t a = queue[head] >> 16, o = queue[head] & 0xFFFFu, lo = J.off[o], hi = J.off[o + 1u];
    fits = hi - lo <= left;
    left -= hi - lo;
#pragma unroll 1
    for (uint32_t j = lo; fits && j < hi; ++j) {
      const uint32_t it = J.items[j];
      const uint2 rec = staged ? recs[j] : __ldg(reinterpret_cast<const uint2*>(ga_item) + (it & 0xFFFFu));
      if (rec.x >> 16 != a) continue;
      if (rec.y & GA_GOES_ON) {
        const uint32_t v = ((it & 0xFFFFu) + 1u) << 16 | it >> 16;
        uint32_t same = 0xFFFFFFFFu;
#pragma unroll 1
        for (uint32_t x = 0; x < cnt; ++x) {
          const uint32_t u = found[32u * x + lane];
          if (u >> 16 == v >> 16) same = u;
        }
        if (same != 0xFFFFFFFFu) fits = same == v;
        else if (cnt == AF_NODE) fits = false;
        else found[32u * cnt++ + lane] = v;
      }
      if ((rec.y & 0xFFFFu) != 0xFFFFu) {
        const uint32_t up = rec.y << 16 | it >> 16;
        uint32_t x = 0;
#pragma unroll 1
        while (x < nq && queue[x] != up) ++x;
        if (x == AF_QUEUE) fits = false;
        else if (x == nq) queue[nq++] = up;
      }
    }
  }
  __syncwarp();
  uint32_t m = __ballot_sync(FULL, fits);
  if (m == 0u && lane == 0) ctl[AC_ONE_BY_ONE] = 1u;  // (what one of them lacks others will: lists of a hundred rules, sets of hundreds of items)
#pragma unroll 1
  for (; m; m &= m - 1u) {
    const uint32_t src = (uint32_t)__ffs(m) - 1u, n = __shfl_sync(FULL, cnt, src), x = lane < n ? found[32u * lane + src] : 0u;
    const uint32_t to = intern_singles(C, ctl, lane < n, lane < n ? __ldg(&ga_item[2u * (x >> 16)]) & 0xFFFFu : 0u, x & 0xFFFFu);
    const uint32_t at = ctl[AC_POOL];
    if (__any_sync(FULL, lane < n && to == CTX_NEW) || n > C.pool_cap - at) break;
    if (lane < n) C.pool[at + lane] = (x & 0xFFFF0000u) | to;
    if (lane == src) C.exp[c] = make_uint2(at, n);
    __syncwarp();
    if (lane == 0) ctl[AC_POOL] = at + n;
    __syncwarp();
  }
  __syncwarp();
}

// ---- contexts of one origin that a chart of few items can ask for, all at once
//
// Such a context is the rule and the origin of some item of the chart, and is known by the number of the first such item.  A thread
// for each item enters its context and finds the items that wait for it (links), then expands it by following links.  One
// after the other, as they are asked for, by a warp, the thirteen contexts of a row of JSON took 60,000 of its 100,000 cycles.
constexpr uint32_t NO_ITEM = 0xFFFFu;
// (before: recs are there, and the hash is empty; after: contexts 0 .. n - 1)
__device__ __forceinline__ void enter_items(uint32_t m, uint32_t k) {
  const uint32_t *off = smem + SM_STAGE + CH_HDR, *items = off + m + 1u;
  const uint2* recs = reinterpret_cast<const uint2*>(smem + SM_RECS);
  const Contexts C = shared_contexts();
  const uint32_t lhs = recs[k].x & 0xFFFFu, nt = recs[k].x >> 16, o = items[k] >> 16;
  C.pool[k] = o, C.org[k] = make_uint2(k, 1u), C.lhs[k] = lhs, C.exp[k] = make_uint2(0u, CTX_NEW);
  uint32_t rep = k;
  #pragma unroll 1
  for (uint32_t slot = mix32(mix32(o + 1u) + lhs * 0x9E3779B9u + 1u) & C.hash_mask;; slot = (slot + 1u) & C.hash_mask) {  // (as context_hash has it)
    const uint32_t v = atomicCAS(&C.hash[slot], 0u, k + 1u);
    if (v == 0u) break;
    if ((recs[v - 1u].x & 0xFFFFu) == lhs && items[v - 1u] >> 16 == o) {
      rep = v - 1u;
      break;
    }
  }
  reinterpret_cast<uint16_t*>(smem + SM_REP)[k] = (uint16_t)rep;
  // the first item of set o that waits for its rule's non-terminal, and the next item of its own set that waits for the same as it does
  uint32_t first = NO_ITEM, next = NO_ITEM, lo = 0, hi = m;
  #pragma unroll 1
  for (uint32_t i = off[o], end = off[o + 1u]; i < end; ++i)
    if (recs[i].x >> 16 == lhs) {
      first = i;
      break;
    }
  if (nt != 0xFFFFu) {
    #pragma unroll 1
    while (hi - lo > 1u) {
      const uint32_t mid = (lo + hi) >> 1;
      if (off[mid] <= k) lo = mid;
      else hi = mid;
    }
    #pragma unroll 1
    for (uint32_t i = k + 1u, end = off[hi]; i < end; ++i)
      if (recs[i].x >> 16 == nt) {
        next = i;
        break;
      }
  }
  smem[SM_LINK + k] = next << 16 | first;
}
// (after all have been entered; at most `most` items in pool[n + most * k ..]; contexts that need more, or items of one rule begun in
// several sets, are left to be expanded by a warp when they are asked for)
__device__ __forceinline__ void expand_items(uint32_t m, uint32_t n, uint32_t most, uint32_t k) {
  const uint32_t* items = smem + SM_STAGE + CH_HDR + m + 1u;
  const uint2* recs = reinterpret_cast<const uint2*>(smem + SM_RECS);
  const uint16_t* reps = reinterpret_cast<const uint16_t*>(smem + SM_REP);
  uint16_t* const queue = reinterpret_cast<uint16_t*>(smem + SM_OWNER) + AF_QUEUE * k;  // what has been completed (the place is not used yet)
  static_assert(AF_QUEUE * AF_ITEMS <= (2 * AF_EDGES + AF_TOKENS) / 32, "the queues' place");
  const Contexts C = shared_contexts();
  if (reps[k] != k) return;
  uint32_t* const list = C.pool + n + most * k;
  uint32_t nq = 1, cnt = 0;
  queue[0] = (uint16_t)k;
#pragma unroll 1
  for (uint32_t head = 0; head < nq; ++head) {
#pragma unroll 1
    for (uint32_t j = smem[SM_LINK + queue[head]] & 0xFFFFu; j != NO_ITEM; j = smem[SM_LINK + j] >> 16) {
      const uint32_t flags = recs[j].y, to = reps[j];
      if (flags & GA_GOES_ON) {
        const uint32_t v = ((items[j] & 0xFFFFu) + 1u) << 16 | to;
        uint32_t same = 0xFFFFFFFFu;
#pragma unroll 4
        for (uint32_t i = 0; i < cnt; ++i) {
          const uint32_t u = list[i];
          if (u >> 16 == v >> 16) same = u;
        }
        if (same == 0xFFFFFFFFu) {
          if (cnt == most) return;
          list[cnt++] = v;
        } else if (same != v) {
          return;  // begun in another set, too
        }
      }
      if ((flags & 0xFFFFu) != 0xFFFFu) {
        uint32_t i = 0;
#pragma unroll 1
        while (i < nq && queue[i] != to) ++i;
        if (i == nq) {
          if (nq == AF_QUEUE) return;
          queue[nq++] = (uint16_t)to;
        }
      }
    }
  }
  C.exp[k] = make_uint2(n + most * k, cnt);
}

// More items of a last set than a warp's lanes hold.  False: their contexts do not fit shared memory (buf is in order then).
__device__ __noinline__ bool group_many(const GrammarDev& G, uint32_t* ctl, uint32_t* buf, uint32_t n, uint2& out) {
  return group_items(G, shared_contexts(), ctl, buf, n, out);
}
// The same when that was so.  Nobody else may be at the contexts: they are copied.
__device__ __noinline__ bool group_spilled(const GrammarDev& G, const AutoFillDev& A, uint32_t* ctl, uint32_t* buf, uint32_t n, uint2& out) {
  Contexts C = shared_contexts();
  spill_contexts(C, ctl, A);
  return group_items(G, C, ctl, buf, n, out);
}

// Wherever the chart and the contexts are, and however large the expansion is.
__device__ __noinline__ bool expand_context(const GrammarDev& G, const AutoFillDev& A, Contexts& C, const AfChart& J, uint32_t c,
                                            uint32_t* ctl, uint32_t* work, uint32_t* hset, uint32_t* buf) {
  const uint32_t lane = lane_id();
  #pragma unroll 1
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

// Tokens at .. at + cnt of each lane's list, dealt out to the lanes four by four.
__device__ __forceinline__ void set_tokens(const GrammarDev& G, uint32_t* mask, uint32_t at, uint32_t cnt) {
  const uint32_t lane = lane_id();
  uint32_t incl = cnt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t t = __shfl_up_sync(FULL, incl, d);
    if ((int)lane >= d) incl += t;
  }
  const uint32_t total = __shfl_sync(FULL, incl, 31), excl = incl - cnt, from = at - excl;
  #pragma unroll 1
  for (uint32_t base = 0; base < total; base += 128) {
    uint32_t tok[4];
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) {
      const uint32_t first = base + u * 32u;
      uint32_t e = 0;  // the last lane that begins at or before it
#pragma unroll
      for (uint32_t d = 16; d; d >>= 1)
        if (__shfl_sync(FULL, excl, e + d) <= first + lane) e += d;
      const uint32_t f = __shfl_sync(FULL, from, e);
      tok[u] = first + lane < total ? __ldg(&G.ga_tok[f + first + lane]) : 0xFFFFFFFFu;
    }
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u)
      if (tok[u] != 0xFFFFFFFFu) atomicOr(&mask[tok[u] >> 5], 1u << (tok[u] & 31u));
  }
}

__global__ void __launch_bounds__(AF_THREADS, 2) automaton_fill_kernel(const __grid_constant__ GrammarDev G,
                                                                       const __grid_constant__ StateDev S) {
  before_me();
  const AutoFillDev& A = S.af;
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id(), lt = (1u << lane) - 1u;
  uint2* const entries = reinterpret_cast<uint2*>(smem + SM_ENTRIES);
  uint2* const lists = reinterpret_cast<uint2*>(smem + SM_LISTS);
  uint32_t* const seen = smem + SM_SEEN;
  const Contexts C0 = shared_contexts();
  uint32_t* const pre = smem + SM_PRE;
  uint32_t* const ctl = smem + SM_CTL;
  uint32_t* const wide = smem + SM_WIDE;
  uint32_t* const stage = smem + SM_STAGE;
  uint32_t* const buf = smem + SM_BUF;
  uint32_t* const work = smem + SM_WORK;
  uint32_t* const hset = smem + SM_HSET;
  uint16_t* const owner = reinterpret_cast<uint16_t*>(smem + SM_OWNER);
  uint4* const stack = A.stack + (size_t)blockIdx.x * A.stack_cap;  // entries that found no room: first edge, edges, context
  auto edge_deal = [&](uint32_t side) {
    return Deal{ctl + AC_EDGES + 4u * side, entries + side * AF_BATCH, pre + side * AF_BATCH, owner + side * (AF_EDGES / 32u), AF_BATCH, AF_EDGES};
  };
  auto token_deal = [&](uint32_t side) {
    return Deal{ctl + AC_TOKENS + 4u * side, lists, pre + 2u * AF_BATCH, owner + 2u * (AF_EDGES / 32u), AF_LISTS, AF_TOKENS};
  };
  // where the kernel of a last set of so many items is put together
  auto kernel_items = [&](uint32_t items) -> uint32_t* { return items <= AF_BUF ? buf : big_area(A) + A.big_cap / 4u + A.big_cap / 2u; };
  uint32_t looked_up = 0, contexts = 0;
  bool gave_up = false, filled = false;
  auto fill_tag = [&]() -> uint32_t { return S.counters[CNT_AF_NO] << 1 | 1u; };  // what this fill's blocks leave when one of them gives up
  if (blockIdx.x == 0 && tid == 0) stat_add(S, CNT_STAT_FILLS, S.B);
  #pragma unroll 1
  for (uint32_t row = blockIdx.x; row < S.B;) {
    // ---- where the row's mask comes from: the state cache, another row of this call with the same chart, or from here
    const uint32_t flags = S.row_flags[row];
    if (!S.row_state && (flags & ROW_BROKEN)) break;  // (a chart that did not pass its check; such calls have a block for each)
    const uint32_t* chart = S.arena + S.row_chart[row];
    const int32_t sid = S.row_state ? S.row_state[row] : -1;
    const uint32_t taken = tid == 0 && S.cache_on ? vload(&S.counters[CNT_N_MASK_ROWS]) : 0u;
    const uint32_t ahead = tid < A.ahead ? chart[tid] : 0u;  // (asked for together with the header)
    AfChart J;
    J.m = chart[CH_SETS];
    const uint32_t chart_words = chart[CH_WORDS], chart_flags = chart[CH_FLAGS];
    if (tid == 0) {
      int32_t from = (int32_t)row;
      bool here = false;
      if (flags & ROW_BROKEN) {
        from = MASK_ZERO;
      } else if (flags & ROW_FINISHED) {
        from = MASK_EOS_ONLY;
      } else {
        const int32_t old = sid >= 0 ? atomicCAS(&S.st_mask[sid], -1, -2 - (int32_t)row) : -1;
        here = old == -1;
        if (old >= 0) {
          S.st_ref[sid] = 1;  // (used again: it outlives the next emptying of the cache)
          from = old;
          stat_add(S, CNT_STAT_CACHED, 1u);
        } else if (old <= -2) {
          from = MASK_ALIAS0 - (-2 - old);
          stat_add(S, CNT_STAT_SHARED, 1u);
        }
      }
      if (!here) S.row_mask[row] = from;
      if (S.row_job) S.row_job[row] = here ? 1u : 0u;
      ctl[AC_ROW] = here ? 1u : 0u;
    }
    __syncthreads();
    if (ctl[AC_ROW]) {
      const bool accepting = (chart_flags & CHART_ACCEPTING) != 0u, staged = chart_words <= AF_STAGE;
      if (tid < AC_CLEARED) ctl[tid] = 0u;
      J.off = chart + CH_HDR;
      if (staged) {
        if (tid < A.ahead) stage[tid] = ahead;
#pragma unroll 1
        for (uint32_t i = A.ahead + tid; i < chart_words; i += AF_THREADS) stage[i] = chart[i];
        J.off = stage + CH_HDR;
      }
      J.items = J.off + J.m + 1u;
      #pragma unroll 1
      for (uint32_t i = tid; i < AF_SEEN / 4u; i += AF_THREADS) reinterpret_cast<uint4*>(seen)[i] = make_uint4(EMPTY_SLOT, EMPTY_SLOT, EMPTY_SLOT, EMPTY_SLOT);
      #pragma unroll 1
      for (uint32_t i = tid; i < AF_CTX_HASH; i += AF_THREADS) C0.hash[i] = 0u;
      if (!filled)
        #pragma unroll 1
        for (uint32_t i = tid; i < AF_HSET; i += AF_THREADS) hset[i] = EMPTY_SLOT;
      if (!filled && tid == 0) ctl[AC_CROWDED] = ctl[AC_CUT] = 0u;
      filled = true;
      __syncthreads();
      const uint32_t n_items = J.off[J.m];
      const bool few = staged && n_items <= AF_ITEMS;  // (a chart can have no item: a finite grammar's text, read to its end)
      const uint32_t most = min(AF_NODE, AF_NODES / max(n_items, 1u)), own_item = lane * (AF_WARPS - 1u) + warp - 1u;  // (neighbouring items to different warps)
      uint2* const recs = reinterpret_cast<uint2*>(smem + SM_RECS);
      if (tid == 0) {  // a row for the mask, of the cache if one is left
        int32_t mrow = (int32_t)row;
        if (sid >= 0) {
          const uint32_t got = taken < S.max_mask_rows ? atomicAdd(&S.counters[CNT_N_MASK_ROWS], 1u) : S.max_mask_rows;
          if (got < S.max_mask_rows) mrow = (int32_t)(S.mrow_base + got);
          else if (S.full_flag) *reinterpret_cast<volatile uint32_t*>(S.full_flag) = 1u;  // no mask row left to cache it in
        }
        S.row_mask[row] = mrow;
        ctl[AC_MASK] = (uint32_t)mrow;
        stat_add(S, CNT_STAT_COMPUTED, 1u);
      }
      if (warp == 0) {
        if (lane < 4u) deal_clear(lane < 2u ? edge_deal(lane) : token_deal(lane - 2u));
        if (lane == 30u) ctl[AC_ONE_BY_ONE] = 0u;
        if (few && lane == 31u) ctl[AC_NCTX] = n_items, ctl[AC_POOL] = n_items * (1u + most);
      } else if (staged) {  // what the expansions need to know about the chart's items
#pragma unroll 1
        for (uint32_t k = tid - 32u; k < n_items; k += AF_THREADS - 32u) recs[k] = __ldg(reinterpret_cast<const uint2*>(G.ga_item) + (J.items[k] & 0xFFFFu));
        if (few) {
          others_meet();
          if (own_item < n_items) enter_items(J.m, own_item);
        }
      }
      __syncthreads();
      if (warp == 0) {  // the kernel of the chart's last set
        const uint32_t lo = J.off[J.m - 1u], hi = J.off[J.m], self = J.m - 1u;
        uint32_t* const b = kernel_items(hi - lo);
        uint32_t n = 0;
        bool ok = hi - lo <= A.big_cap;
        if (ok)
#pragma unroll 1
          for (uint32_t base = lo; base < hi; base += 32) {
            const uint32_t k = base + lane;
            const uint32_t it = k < hi ? J.items[k] : 0u, d = it & 0xFFFFu;
            bool take = k < hi && ((it >> 16) != self || d == ITEM_START);
            const bool after = take && k > lo && d != 0u && J.items[k - 1u] == it - 1u;
            uint32_t own = 0u, before = 0u;
            if (take) own = staged ? recs[k].y : __ldg(&G.ga_item[2u * d + 1u]);
            if (after) before = staged ? recs[k - 1u].y : __ldg(&G.ga_item[2u * d - 1u]);
            take = take && (own & GA_ALIVE) && !(before & GA_SKIPS);  // (an item that the one before it skips to comes with that)
            const uint32_t bal = __ballot_sync(FULL, take);
            if (take) b[n + __popc(bal & lt)] = (it << 16) | (it >> 16);
            n += __popc(bal);
          }
        __syncwarp();
        uint2 list = make_uint2(0u, 0u);
        const bool later = ok && (n > 32u || !group_shared(G.ga_item, lane < n ? b[lane] : 0xFFFFFFFFu, n, list)) && !group_many(G, ctl, b, n, list);
        if (lane == 0) {
          ctl[AC_LIST] = list.x, ctl[AC_LIST_END] = list.y;
          if (later) ctl[AC_LATER] = n;
          if (!ok) ctl[AC_FAIL] = 1u + DIAG_SET_SCRATCH;
        }
      } else {
        if (few && own_item < n_items) expand_items(J.m, n_items, most, own_item);
        if (tid == AF_THREADS - 1) ctl[AC_BEGAN] = (uint32_t)(clock64() >> 10);
      }
      __syncthreads();
      if (ctl[AC_LATER]) {  // (contexts leave shared memory when the other warps have made theirs)
        if (warp == 0) {
          uint2 list = make_uint2(0u, 0u);
          const bool ok = group_spilled(G, A, ctl, kernel_items(J.off[J.m] - J.off[J.m - 1u]), ctl[AC_LATER], list);
          if (lane == 0) {
            ctl[AC_LIST] = list.x, ctl[AC_LIST_END] = list.y;
            if (!ok) ctl[AC_FAIL] = 1u + DIAG_SET_SCRATCH;
          }
        }
        __syncthreads();
      }

      uint32_t* const mask = S.mask_rows + (size_t)ctl[AC_MASK] * G.Wm;
      bool spilled = false;
      // the expansion of a context (offset into pool, count), and its elements
      auto expansion = [&](uint32_t c) -> uint2 { return spilled ? global_contexts(A).exp[c] : C0.exp[c]; };
      auto element = [&](uint32_t at) -> uint32_t { return spilled ? global_contexts(A).pool[at] : C0.pool[at]; };
      // False: these edges were listed with this context a moment ago.  (Where they begin, 24 bits, and the context, 12 bits, are mixed one
      // to one: the slot and what it holds are all 36 of them.)
      auto fresh = [&](uint32_t edge, uint32_t ctx) -> bool {
        unsigned long long x = (unsigned long long)edge << 12 | ctx;
        x = (x ^ x >> 19) * 0x9E3779B97F4A7C15ull & 0xFFFFFFFFFull;
        volatile uint32_t* p = seen + (uint32_t)(x >> (36u - AF_SEEN_BITS));
        const uint32_t rest = (uint32_t)x & ((1u << (36u - AF_SEEN_BITS)) - 1u);
        const bool yes = *p != rest;
        *p = rest;
        return yes;
      };
      uint32_t list_at = 0, gtop = 0, rounds = 0;  // items of the last set whose starts have been taken, entries on the stack
      bool begun = false;
#pragma unroll 1
      for (uint32_t side = 0;; side ^= 1u) {  // ---- rounds
        const Deal E = edge_deal(side), N = edge_deal(side ^ 1u), T = token_deal(side);
        const uint32_t n = dealt_lists(E), all = dealt_things(E), list_end = ctl[AC_LIST_END];
        if (ctl[AC_FAIL] || (n == 0u && begun && list_at == list_end)) break;
        spilled = ctl[AC_SPILLED] != 0u;
        auto overflow = [&](uint32_t edge, uint32_t cnt, uint32_t ctx) {
          const uint32_t p = atomicAdd(&ctl[AC_OVF], 1u);
          if (gtop + p < A.stack_cap) stack[gtop + p] = make_uint4(edge, cnt, ctx, 0u);
          else ctl[AC_FULL] = 1u;  // (cannot happen, see below)
        };
        // (by all lanes of a warp) tokens to be written, and edges with their context (flagged AF_FOUND if they are all of one item)
        auto list = [&](uint32_t tokens, uint32_t nt, bool yes, uint32_t edge, uint32_t cnt, uint32_t ctx) {
          const uint32_t none = deal_both(T, N, nt, tokens, yes ? min(cnt, AF_CHUNK) : 0u, make_uint2(edge, ctx));
          if (yes) {
            if (none & 2u) overflow(edge, cnt, ctx);
            else if (cnt > AF_CHUNK) overflow(edge + AF_CHUNK, cnt - AF_CHUNK, ctx);
            if (!(none & 2u)) {
              asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const uint4*>(G.ga_edge) + edge));
              if (!(ctx & AF_FOUND) && expansion(ctx).y == CTX_NEW) ctl[AC_WANT] = 1u;
            }
          }
          if (__any_sync(FULL, none & 1u)) set_tokens(G, mask, tokens, none & 1u ? nt : 0u);
        };
        if (n == 0u) {
          // ---- the starts of the last set's items
          const uint32_t until = min(list_end, list_at + AF_SLICE);
#pragma unroll 1
          for (uint32_t base = list_at; base == list_at || base < until; base += AF_THREADS) {
            const uint32_t i = base + tid;
            const uint32_t x = i < until ? element(ctl[AC_LIST] + i) : 0u;
            uint4 r = i < until ? __ldg(reinterpret_cast<const uint4*>(G.ga_start) + (x >> 16)) : make_uint4(0u, 0u, 0u, 0u);
            if (r.y == GA_MASK) wide[atomicAdd(&ctl[AC_NWIDE], 1u)] = r.x, r.y = 0u;
            __syncthreads();
            // what is valid from the items with masks, 16 words of a thread under way at once
            const uint32_t nw = ctl[AC_NWIDE];
            if (tid == 0) looked_up += nw * G.Wm;
            if (nw || base == 0u)
#pragma unroll 1
              for (uint32_t at = 4u * tid; at < G.Wm; at += 16u * AF_THREADS) {
                uint4 v[4];
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) v[u] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
                for (uint32_t k = 0; k < nw; ++k) {
                  const uint32_t* src = G.ga_mask + (size_t)wide[k] * G.ga_mask_words + at;
#pragma unroll
                  for (uint32_t u = 0; u < 4; ++u)
                    if (at + 4u * u * AF_THREADS < G.Wm) {
                      const uint4 y = __ldg(reinterpret_cast<const uint4*>(src + 4u * u * AF_THREADS));
                      v[u].x |= y.x, v[u].y |= y.y, v[u].z |= y.z, v[u].w |= y.w;
                    }
                }
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) {
                  const uint32_t first = at + 4u * u * AF_THREADS, words[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                  for (uint32_t q = 0; q < 4; ++q) {
                    const uint32_t i4 = first + q;
                    if (i4 >= G.Wm) continue;
                    if (base == 0u) mask[i4] = words[q] | ((accepting && G.eos >= 0 && i4 == (uint32_t)G.eos >> 5) ? 1u << ((uint32_t)G.eos & 31u) : 0u);
                    else if (words[q]) atomicOr(&mask[i4], words[q]);
                  }
                }
              }
            __syncthreads();
            if (tid == 0) ctl[AC_NWIDE] = 0u;
            if (r.y == 1u) atomicOr(&mask[r.x >> 5], 1u << (r.x & 31u));
            looked_up += r.y;
            list(r.x, r.y > 1u ? r.y : 0u, r.w != 0u, r.z, r.w, x & 0xFFFFu);
            if (base + AF_THREADS < until) __syncthreads();
          }
          list_at = until, begun = true;
        } else {
          // The stack cannot run over: a round takes no more edges than there are places above the reserve, and lists what follows from
          // one of them at most once.  On a crowded stack one entry is taken at a time, from the top, and a few of its edges: depth
          // first the stack grows along one path of the trie.
          const uint32_t room = max(A.stack_cap - min(gtop + A.reserve, A.stack_cap), AF_TIGHT_EDGES), total = min(all, room);
          if (total < all)
            #pragma unroll 1
            for (uint32_t i = tid; i < n; i += AF_THREADS) {
              const uint2 w = E.what[i];
              const uint32_t from = E.pre[i], end = i + 1u < n ? E.pre[i + 1u] : all;
              if (end > total) overflow(w.x + (max(from, total) - from), end - max(from, total), w.y);
            }
          // ---- the edges; those of a warp's next 32 are under way while these are looked at
          if (tid == 0) {
            looked_up += total;
            if (total < all) ++ctl[AC_CUT];
          }
          auto edge_of = [&](uint32_t base, uint2& w) -> uint4 {
            const uint32_t e = whose(E, n, base);
            if (base + lane >= total) return make_uint4(0u, 0u, 0u, 0u);
            w = E.what[e];
            return __ldg(reinterpret_cast<const uint4*>(G.ga_edge) + w.x + (base + lane - E.pre[e]));
          };
          uint2 w = make_uint2(0u, 0u);
          uint32_t base = warp * 32u;
          uint4 g = make_uint4(0u, 0u, 0u, 0u);
          if (base < total) g = edge_of(base, w);
#pragma unroll 1
          while (base < total) {
            const uint32_t after = base + AF_THREADS;
            uint2 w_after = make_uint2(0u, 0u);
            uint4 g_after = make_uint4(0u, 0u, 0u, 0u);
            if (after < total) g_after = edge_of(after, w_after);
            uint32_t to = CTX_NEW;
            if (base + lane < total) {
              to = w.y & ~AF_FOUND;
              if (!(w.y & AF_FOUND)) {
                const uint2 x = expansion(to);
                const uint32_t d = g.x >> 16;
                uint32_t lo = 0;
                to = CTX_NEW;
                if (x.y <= AF_NODE) {  // (in any order)
#pragma unroll 1
                  for (; lo < x.y; lo += 4u) {
                    uint32_t el[4];
#pragma unroll
                    for (uint32_t u = 0; u < 4; ++u) el[u] = lo + u < x.y ? element(x.x + lo + u) : 0xFFFFFFFFu;
#pragma unroll
                    for (uint32_t u = 0; u < 4; ++u)
                      if (lo + u < x.y && el[u] >> 16 == d) to = el[u] & 0xFFFFu;
                  }
                } else {
                  uint32_t hi = x.y;
#pragma unroll 1
                  while (lo < hi) {
                    const uint32_t mid = (lo + hi) >> 1;
                    if ((element(x.x + mid) >> 16) < d) lo = mid + 1u;
                    else hi = mid;
                  }
                  const uint32_t el = lo < x.y ? element(x.x + lo) : 0u;
                  if (lo < x.y && el >> 16 == d) to = el & 0xFFFFu;
                }
              }
            }
            const bool hit = to != CTX_NEW, group = (g.x & 0xFFFFu) == GA_GROUP;
            if (__any_sync(FULL, hit)) {
              const uint32_t cnt = hit && !group ? g.x & 0xFFFFu : 0u;
              looked_up += cnt;
              if (cnt == 1u) atomicOr(&mask[g.y >> 5], 1u << (g.y & 31u));
              __syncwarp();
              list(g.y, cnt > 1u ? cnt : 0u, hit && g.w && fresh(g.z, to), g.z, g.w, group ? to | AF_FOUND : to);
            }
            base = after, g = g_after, w = w_after;
          }
        }
        __syncthreads();
        gtop += ctl[AC_OVF];
        if (gtop) {
          // ---- entries from the stack, as far as there is room
          const uint32_t k = dealt_lists(N), t = dealt_things(N);
          const bool tight = gtop + A.reserve + AF_TIGHT > A.stack_cap;
          __syncthreads();
          if (tid == 0) {
            ctl[AC_OVF] = 0u;
            if (tight) ++ctl[AC_CROWDED];
          }
          if (tight) {
            #pragma unroll 1
            for (uint32_t i = tid; i < k; i += AF_THREADS) stack[gtop + i] = make_uint4(N.what[i].x, (i + 1u < k ? N.pre[i + 1u] : t) - N.pre[i], N.what[i].y, 0u);
            gtop += k;
            __syncthreads();
            if (tid == 0) deal_clear(N);
          }
          const uint32_t take = tight ? 1u : k < AF_BATCH / 2u && t < AF_EDGES / 2u ? min(gtop, AF_BATCH / 2u) : 0u;
          const uint4 v = tid < take ? stack[gtop - 1u - tid] : make_uint4(0u, 0u, 0u, 0u);
          const uint32_t now = tight ? min(v.y, AF_TIGHT_EDGES) : v.y;
          static_assert(AF_BATCH / 2u <= AF_THREADS, "an entry to a thread");
          const bool part = __syncthreads_or(now < v.y);
          gtop -= take;
          if (part) {
            if (tid == 0) stack[gtop] = make_uint4(v.x + now, v.y - now, v.z, 0u);
            ++gtop;
          }
          list(0u, 0u, tid < take, v.x, now, v.z);
          __syncthreads();
          gtop += ctl[AC_OVF];
          __syncthreads();
        }
        if (tid == 0) {
          ctl[AC_OVF] = 0u;
          deal_clear(E), deal_clear(token_deal(side ^ 1u));
          if (ctl[AC_FULL]) ctl[AC_FAIL] = 1u + DIAG_QUEUE_FULL;
          if (++rounds > poll_limit(S, 22)) {
            diag(S, DIAG_WAIT_QUEUE);
            if (atomicExch(&S.counters[CNT_BAR_ERR], fill_tag()) != fill_tag()) stat_add(S, CNT_STAT_ABORTS, 1u);
            ctl[AC_FAIL] = AF_GIVEN_UP;
          }
        }
        if (warp == 0 && ctl[AC_WANT]) {
          // ---- expansions that the next round needs
          const uint32_t k = dealt_lists(N);
          Contexts C = spilled ? global_contexts(A) : C0;
          __syncwarp();
          if (lane == 0) ctl[AC_WANT] = 0u;
#pragma unroll 1
          for (uint32_t base = 0; base < k; base += 32) {
            const uint32_t c = base + lane < k ? N.what[base + lane].y : AF_FOUND;
            const uint32_t many = __ballot_sync(FULL, !(c & AF_FOUND) && C.exp[c & ~AF_FOUND].y == CTX_NEW);
            if (__popc(many) >= AF_LANES && !ctl[AC_ONE_BY_ONE]) {
              const bool first = (uint32_t)__ffs(__match_any_sync(FULL, c)) == lane + 1u, mine = (many >> lane & 1u) && first && C.org[c & ~AF_FOUND].y == 1u;
              if (__popc(__ballot_sync(FULL, mine)) >= AF_LANES) expand_by_lanes(G.ga_item, C, J, staged, ctl, mine ? c : CTX_NEW);
            }
#pragma unroll 1
            for (uint32_t todo = __ballot_sync(FULL, !(c & AF_FOUND) && C.exp[c & ~AF_FOUND].y == CTX_NEW); todo;) {
              const uint32_t x = __shfl_sync(FULL, c, __ffs(todo) - 1);
              const bool ok = staged && !ctl[AC_SPILLED] && expand_shared(G.ga_item, J.m, x);
              if (!ok && !expand_context(G, A, C, J, x, ctl, work, hset, buf) && lane == 0) ctl[AC_FAIL] = 1u + DIAG_SET_TABLE;
              todo &= ~__ballot_sync(FULL, c == x);
            }
          }
        }
        if (warp) {
          // ---- tokens, meanwhile
          const uint32_t nt = dealt_lists(T), tt = dealt_things(T);
#pragma unroll 1
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
          if (tid == AF_THREADS - 1 && (uint32_t)(clock64() >> 10) - ctl[AC_BEGAN] > AF_KCYCLES && !ctl[AC_FAIL]) ctl[AC_FAIL] = AF_LATE;
        }
        __syncthreads();
      }
      contexts += ctl[AC_NCTX];
      if (ctl[AC_FAIL] && ctl[AC_FAIL] != AF_GIVEN_UP) {  // too many contexts, or too long a time: the row is left to a sweep by Earley steps
        gave_up = true;
        __threadfence();
        if (tid == 0) {
          if (ctl[AC_FAIL] != AF_LATE) diag(S, ctl[AC_FAIL] - 1u);
          *reinterpret_cast<volatile unsigned long long*>(A.given + atomicAdd(&S.counters[CNT_AF_GIVEN], 1u)) = (unsigned long long)fill_tag() << 32 | row;
        }
      }
    }
    // ---- the next row
    if (S.B <= gridDim.x) break;
    __syncthreads();
    if (tid == 0) ctl[AC_ROW] = gridDim.x + atomicAdd(&S.counters[CNT_AF_TICKET], 1u);
    __syncthreads();
    row = ctl[AC_ROW];
    __syncthreads();
  }
  if (blockIdx.x == 0 && tid == AF_THREADS - 1) {  // an earlier fill's mark goes (a block of this one that gives up sets this one's)
    const uint32_t mark = vload(&S.counters[CNT_BAR_ERR]);
    if (mark && mark != fill_tag()) atomicCAS(&S.counters[CNT_BAR_ERR], mark, 0u);
  }
  if (!filled) return;
  looked_up = __reduce_add_sync(FULL, looked_up);
  __syncthreads();
  if (tid == 0) ctl[AC_LOOKED] = 0u;
  __syncthreads();
  if (lane == 0 && looked_up) atomicAdd(&ctl[AC_LOOKED], looked_up);
  __syncthreads();
  if (tid == 0) {
    stat_add(S, CNT_STAT_TRANS, ctl[AC_LOOKED]);
    stat_add(S, CNT_STAT_LOCAL, contexts);
    if (ctl[AC_CROWDED]) stat_add(S, CNT_STAT_CROWDED, ctl[AC_CROWDED]);
    if (ctl[AC_CUT]) stat_add(S, CNT_STAT_CUT, ctl[AC_CUT]);
  }
  // ---- rows that were given up, swept by the blocks that gave them up when they have no row left.  Only blocks that look for tables
  // wait, and who has tables waits for nobody.
  #pragma unroll 1
  while (gave_up) {
    __syncthreads();
    if (tid == 0) {
      uint32_t at = vload(&S.counters[CNT_AF_GIVEN_TAKEN]), got = 0xFFFFFFFFu, slot = 0xFFFFFFFFu;
      #pragma unroll 1
      while (at < ld_acquire(&S.counters[CNT_AF_GIVEN])) {
        const uint32_t was = atomicCAS(&S.counters[CNT_AF_GIVEN_TAKEN], at, at + 1u);
        if (was == at) {
          got = at;
          break;
        }
        at = was;
      }
      if (got != 0xFFFFFFFFu) {
        uint32_t k = blockIdx.x % A.sweep_slots;
        unsigned long long v = 0u;
        #pragma unroll 1
        for (uint32_t polls = 0; slot == 0xFFFFFFFFu; ++polls, k = (k + 1u) % A.sweep_slots) {
          if (v >> 32 != fill_tag()) v = *reinterpret_cast<const volatile unsigned long long*>(A.given + got);  // (written right after its number was drawn)
          if (v >> 32 == fill_tag() && atomicCAS(A.sweep_lock + k, 0u, 1u) == 0u) slot = k;
          else if (ld_acquire(&S.counters[CNT_BAR_ERR]) == fill_tag()) break;
          else if (polls > poll_limit(S, 22)) {
            diag(S, DIAG_WAIT_VALUE);
            if (atomicExch(&S.counters[CNT_BAR_ERR], fill_tag()) != fill_tag()) stat_add(S, CNT_STAT_ABORTS, 1u);
            break;
          } else {
            __nanosleep(400);
          }
        }
        ctl[AC_SLOT] = (uint32_t)v;
        __threadfence();
      }
      ctl[AC_ROW] = slot;
    }
    __syncthreads();
    const uint32_t slot = ctl[AC_ROW], row = ctl[AC_SLOT];
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

constexpr uint32_t AF_SMEM = SM_WORDS * 4u;
static_assert(SM_CTL % 4 == 0 && SM_HSET % 4 == 0 && SM_SEEN % 4 == 0 && SM_RECS % 2 == 0 && SM_ORG % 2 == 0, "what is read and cleared in 16- and 8-byte pieces");
constexpr uint32_t AF_SWEEP_SMEM = block_sweep_words(AF_WARPS, MAX_NONTERMINALS / 32u) * 4u;  // a row that is given up is swept in the same shared memory
constexpr uint32_t AF_SMEM_ASKED = AF_SMEM > AF_SWEEP_SMEM ? AF_SMEM : AF_SWEEP_SMEM;

// Places of a block's stack that only its depth-first rounds use, along the longest path of the trie - for every byte the edges to the
// groups of a long list, then a group's, each edge's list and the rest of that, and what is left of both entries - and the entries of a
// round that are put back.
uint32_t automaton_fill_reserve() { return (MAX_TOKEN_BYTES + 2u) * (3u * AF_TIGHT_EDGES + 2u) + 3u * AF_BATCH; }
static_assert(GA_EDGE_GROUP <= AF_CHUNK && AF_TIGHT_EDGES * AF_CHUNK <= AF_EDGES, "a group is one entry, and a depth-first round's lists find room");
uint32_t automaton_fill_warps() { return AF_WARPS; }
uint32_t automaton_fill_least_stack() { return automaton_fill_reserve() + AF_TIGHT + AF_SLICE; }

void automaton_fill_layout(uint32_t rows, uint32_t max_blocks, AutoFillDev& A) {
  A.reserve = automaton_fill_reserve();
  A.scratch_words = 7u * A.ctx_cap + A.pool_cap + A.big_cap / 4u + A.big_cap / 2u + A.big_cap;
  A.grid = std::min(max_blocks, rows);
}

cudaError_t configure_automaton_fill() {
  return cudaFuncSetAttribute((const void*)automaton_fill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AF_SMEM_ASKED);
}

void launch_automaton_fill(const GrammarDev& G, const StateDev& S, cudaStream_t st) {
  launch_overlapped(automaton_fill_kernel, dim3(S.af.grid), dim3(AF_THREADS), AF_SMEM_ASKED, st, G, S);
}

}  // namespace fmt
