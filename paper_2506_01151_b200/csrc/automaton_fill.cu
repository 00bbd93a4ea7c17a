// The fill of rows' masks by the grammar automaton (grammar_automaton.cpp; Sections 3.3, 4.1, 4.3 of the paper).
//
// A thread block takes a row.  The kernel items of the chart's last set are grouped by dotted rule; every group starts a
// THREAD at the root of the vocabulary trie: a code of the automaton and a CONTEXT, the set of origins its items were begun in.  A
// trie node's children are reached by one table look-up each.  Where the automaton says that a rule begun in the chart ends, the
// thread's context is EXPANDED: the items that waited in its origins, completed upwards (Section 3.2's Complete), start
// threads of their own at that node.  A context is expanded once per row.  A token is valid iff some thread is alive at the
// node where its bytes end; its bit is set in the row's mask in global memory at once.
//
// What bounds it: at the sizes measured, latency - rounds of "take threads, look their children up, push what is alive", each
// two or three dependent reads in L2 and four block barriers, about as many rounds as the longest token has bytes.  Hence
// the threads, the contexts and the chart sit in shared memory (with a way out to global memory), and three blocks
// share an SM (58 KB each).  The grid has four for each all the same: a row's blocks are a power of two, and with three 128 rows of SQL
// got two blocks each in the place of four.  Rows differ by a factor of a hundred in work (measured: 800 to 290,000 look-ups), so blocks that have no row left wait
// for work, and a block with many threads hands parts of them out, with its contexts.
// Measured on a B200, the fill alone, against the sweep of the whole grid by Earley steps (kernels.cu) before:
//   8 rows of JSON, 32,000 tokens               239 -> 94 us    (where about half of the rows are computed)
//   64 rows of a JSON schema, 128,256 tokens    263 -> 77 us
//   128 rows of SQL, 152,064 tokens             667 -> 231 us
//   37 rows of JSON, 50,001 tokens              362 -> 126 us
//   256 rows of ambiguous JSON, 128,256 tokens  3.51 -> 0.93 ms (2.65 ms when no work is handed on)
// Blocks of an SM, us (timed call by call) for those 37 rows of JSON, those 256 ambiguous rows and 12 decoding steps of the SQL rows: three resident of four
// asked for 150, 1,076 and 5,437; four resident, with half the specials 176, 1,372 and 6,055; three of three asked for 153, 1,223 and 7,454;
// three of four with 80 registers a thread 153, 1,107 and 5,340.
// The sweep stays for grammars without an automaton and for the cache of context-independent entries.  A row that outgrows the
// contexts' storage, or takes far longer than rows do, is swept by Earley steps within the call (block_sweep.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "block_sweep.cuh"
#include "sweep_warp.cuh"

namespace fmt {

constexpr int AF_WARPS = 8, AF_THREADS = AF_WARPS * 32;
constexpr uint32_t AF_BATCH = 512;        // threads of a round
constexpr uint32_t AF_PER = AF_BATCH / AF_THREADS;
constexpr uint32_t AF_SPEC = AF_THREADS;  // expansions to be made at the start of a round
constexpr uint32_t AF_EXITS = 60;         // lists of nodes at which expansions are to be made (from wide items)
constexpr uint32_t AF_TIGHT = 6144;       // free places of a block's stack, its reserve not counted, below which entries are taken one at a time
constexpr uint32_t AF_LIST_STARTS = 64;   // expansions of more elements are started from a list's nodes by specials
constexpr uint32_t AF_SEEN = 512;         // recently started threads (a lossy table: repeats only cost time)
constexpr uint32_t AF_STAGE = 1024;       // a chart up to this many words is read from shared memory
constexpr uint32_t AF_CTX = 64, AF_CTX_HASH = 128, AF_POOL = 2048;  // contexts in shared memory, words of their lists
constexpr uint32_t AF_BUF = 512, AF_WORK = 256, AF_HSET = 512;      // an expansion in shared memory (larger ones: global memory)
constexpr uint32_t AF_OWNER = AF_BATCH * 8;  // pieces of 32 children a round can hold (a node has at most 256)
constexpr uint32_t AF_HEAVY = 16384;      // after so many look-ups for a row, or for a unit of work,
constexpr uint32_t AF_SHARE = 384;        // a block with so many threads gives some to blocks that wait,
constexpr uint32_t AF_MAX_UNITS = 7;      // to so many at once, 128 threads at the least to each
// code of a special: to start the threads of a context's expansion at a node (first child, children, AF_SPAWN, elements that have been
// started << 16 | context)
constexpr uint32_t AF_SPAWN = 0xFFFFFFFDu;
constexpr uint32_t AF_KCYCLES = 1u << 14;      // a share of a row that takes longer (2^24 cycles, 8.5 ms) is given up for a sweep by Earley steps
// AC_FAIL: 0, 1 + the capacity that was exceeded, or
constexpr uint32_t AF_GIVEN_UP = 0xFFFFFFFFu;  // a wait ran out: the fill is given up, the row itself is fine
constexpr uint32_t AF_GONE = 0xFFFFFFFEu;      // another block has given the row up
constexpr uint32_t AF_LATE = 0xFFFFFFFDu;      // the share takes too long
constexpr uint32_t CTX_NEW = 0xFFFFFFFFu;

enum : uint32_t {
  AC_NEXT = 0, AC_SPEC = 1, AC_OVF = 2, AC_GTOP = 3, AC_FAIL = 4, AC_NCTX = 5, AC_POOL = 6, AC_NWORK = 7, AC_WSUM = 8, AC_NBUF = 16, AC_OVER = 17,
  AC_SPILLED = 18, AC_WAITING = 19, AC_BASE = 20, AC_JOB = 21, AC_NWIDE = 22, AC_POPPED = 24, AC_NEXITS = 25, AC_LIST = 26,
  AC_LIST_AT = 27, AC_LIST_END = 28, AC_POPPED_SPEC = 29, AC_BEGAN = 30,
  AC_PEEK = 32, AC_WIDE = 40, AC_WORDS = (AC_WIDE + AF_EXITS + 3) & ~3u
};
static_assert(AC_WORDS % 4 == 0 && AC_WORDS <= AF_THREADS, "what follows in shared memory is cleared in 16-byte pieces; a thread clears a word");

// A unit of work handed out: AU_HDR words, then the giver's contexts, lists and the threads.
enum : uint32_t { AU_ROWJOB = 0, AU_N = 1, AU_NCTX = 2, AU_POOL = 3, AU_PART = 4, AU_HDR = 8 };
constexpr uint32_t AU_ENTRIES = AF_BATCH / 2 + 4;
constexpr uint32_t AU_WORDS = AU_HDR + 5 * AF_CTX + AF_POOL + 4 * AU_ENTRIES;
static_assert(AU_WORDS % 4 == 0 && (AU_HDR + 5 * AF_CTX + AF_POOL) % 4 == 0, "the threads of a unit are 16-byte records");

// The contexts of the row a block works on: in shared memory, or, when they outgrow it, in global memory of the block's own.
struct Contexts {
  uint2* org;       // [cap] origins: offset into pool, count
  uint2* exp;       // [cap] expansion: offset into pool, count (CTX_NEW: not made yet); pairs (code, rule << 16 | context)
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
  const uint32_t at = (ctl[AC_POOL] + 1u) & ~1u;
  __syncwarp();
  if (at + 2u * groups > C.pool_cap) return false;
  if (lane == 0) ctl[AC_POOL] = at + 2u * groups;
  __syncwarp();
  uint32_t g = 0;
  for (uint32_t i = 0; i < k;) {
    {  // rules with one item each, up to 32 of them together
      const uint32_t x = i + lane < k ? buf[i + lane] : 0xFFFFFFFFu, y = i + lane + 1u < k ? buf[i + lane + 1u] >> 16 : 0xFFFFu;
      const uint32_t before = __shfl_up_sync(FULL, x >> 16, 1);
      const uint32_t other = __ballot_sync(FULL, i + lane >= k || y == x >> 16 || (lane && before == x >> 16));
      const uint32_t run = other ? (uint32_t)__ffs(other) - 1u : 32u;
      if (run) {
        const uint4 rec = lane < run ? __ldg(reinterpret_cast<const uint4*>(G.ga_item) + (x >> 16)) : make_uint4(GA_DEAD, 0u, 0u, 0u);
        const bool v = lane < run && rec.x != GA_DEAD;
        const uint32_t alive = __ballot_sync(FULL, v);
        const uint32_t c = intern_singles(C, ctl, v, rec.y & 0xFFFFu, x & 0xFFFFu);
        if (__any_sync(FULL, v && c == CTX_NEW)) return false;
        if (v) reinterpret_cast<uint2*>(C.pool)[at / 2u + g + __popc(alive & ((1u << lane) - 1u))] = make_uint2(rec.x, (x & 0xFFFF0000u) | c);
        g += __popc(alive);
        i += run;
        continue;
      }
    }
    const uint32_t d = buf[i] >> 16;
    const uint4 rec = __ldg(reinterpret_cast<const uint4*>(G.ga_item) + d);
    uint32_t e = i + 1u;
    for (;;) {  // the end of the group
      const uint32_t b = __ballot_sync(FULL, e + lane >= k || (buf[min(e + lane, k - 1u)] >> 16) != d);
      if (b) {
        e += (uint32_t)__ffs(b) - 1u;
        break;
      }
      e += 32u;
    }
    if (rec.x != GA_DEAD) {
      const uint32_t c = intern_context(C, ctl, rec.y & 0xFFFFu, buf + i, e - i);
      if (c == CTX_NEW) return false;
      if (lane == 0) reinterpret_cast<uint2*>(C.pool)[at / 2u + g] = make_uint2(rec.x, d << 16 | c);
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
      const uint4 rec = __ldg(reinterpret_cast<const uint4*>(G.ga_item) + (it & 0xFFFFu));
      const bool match = k < hi && (rec.y >> 16) == a, on = match && (rec.w & GA_GOES_ON);
      const uint32_t b = __ballot_sync(FULL, on);
      if (nbuf + __popc(b) > buf_cap) {  // an item comes once for every set that it waits in: the repeats go
        uint32_t groups;
        __syncwarp();
        nbuf = sort_unique(buf, nbuf, groups);
        if (nbuf > buf_cap / 2u) return false;
      }
      if (on) buf[nbuf + __popc(b & ((1u << lane) - 1u))] = ((it & 0xFFFFu) + 1u) << 16 | (it >> 16);
      nbuf += __popc(b);
      if (match && (rec.w & 0xFFFFu) != 0xFFFFu) need(rec.w & 0xFFFFu, it >> 16);
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
      const uint4 rec = __ldg(reinterpret_cast<const uint4*>(G.ga_item) + (it & 0xFFFFu));
      const bool match = k < hi && (rec.y >> 16) == a;
      uint32_t on = __ballot_sync(FULL, match && (rec.w & GA_GOES_ON));
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
      for (uint32_t up = __ballot_sync(FULL, match && (rec.w & 0xFFFFu) != 0xFFFFu); up; up &= up - 1u) {
        const uint32_t v = __shfl_sync(FULL, (rec.w & 0xFFFFu) << 16 | (it >> 16), __ffs(up) - 1);
        if (__ballot_sync(FULL, lane < nw && work == v)) continue;
        if (nw == 32u) return false;
        if (lane == nw) work = v;
        ++nw;
      }
    }
  }
  // by rule: one context for each
  uint32_t at = (ctl[AC_POOL] + 1u) & ~1u, g = 0;
  if (at + 2u * ni + 64u > C.pool_cap || ctl[AC_NCTX] + ni > C.cap) return false;
  __syncwarp();
  if (lane == 0) ctl[AC_POOL] = at + 2u * ni;
  __syncwarp();
  uint32_t left = ni == 32u ? FULL : (1u << ni) - 1u;
  {  // rules with one item
    const bool mine = (left >> lane) & 1u;
    const uint32_t same = __match_any_sync(FULL, mine ? item >> 16 : 0x10000u + lane);
    const bool single = mine && same == 1u << lane;
    const uint4 rec = single ? __ldg(reinterpret_cast<const uint4*>(G.ga_item) + (item >> 16)) : make_uint4(GA_DEAD, 0u, 0u, 0u);
    const bool v = single && rec.x != GA_DEAD;
    const uint32_t alive = __ballot_sync(FULL, v);
    left &= ~__ballot_sync(FULL, single);
    if (alive) {
      const uint32_t ctx = intern_singles(C, ctl, v, rec.y & 0xFFFFu, item & 0xFFFFu);
      if (__any_sync(FULL, v && ctx == CTX_NEW)) return false;
      if (v) reinterpret_cast<uint2*>(C.pool)[at / 2u + __popc(alive & ((1u << lane) - 1u))] = make_uint2(rec.x, (item & 0xFFFF0000u) | ctx);
      g = __popc(alive);
    }
  }
  while (left) {
    const uint32_t d = __shfl_sync(FULL, item >> 16, __ffs(left) - 1);
    const bool in = ((left >> lane) & 1u) && (item >> 16) == d;
    const uint32_t members = __ballot_sync(FULL, in), n = __popc(members);
    left &= ~members;
    const uint4 rec = __ldg(reinterpret_cast<const uint4*>(G.ga_item) + d);
    if (rec.x == GA_DEAD) continue;
    // its origins, ascending, at the pool's top (which grows only if the context is new)
    const uint32_t top = ctl[AC_POOL];
    if (top + n > C.pool_cap) return false;
    uint32_t rank = 0;
    if (n > 1u)
      for (uint32_t m = members; m; m &= m - 1u) rank += __shfl_sync(FULL, item, __ffs(m) - 1) < item ? 1u : 0u;
    if (in) C.pool[top + rank] = item & 0xFFFFu;
    __syncwarp();
    const uint32_t ctx = intern_context(C, ctl, rec.y & 0xFFFFu, C.pool + top, n);
    if (ctx == CTX_NEW) return false;
    if (lane == 0) reinterpret_cast<uint2*>(C.pool)[at / 2u + g] = make_uint2(rec.x, d << 16 | ctx);
    ++g;
  }
  __syncwarp();
  if (lane == 0) C.exp[c] = make_uint2(at, g);
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

// Nodes at which several tokens end (byte strings that the grammar cannot tell apart): tokens at .. at + cnt of each lane, dealt out to
// the lanes two by two.  (Node by node, each waited for its own read of ga_tok: 3,000 of the 7,000 cycles of a round.  64 rows of a
// JSON schema decode 16 steps in 2.46 ms instead of 2.57, 37 rows of JSON are filled in 126 us instead of 132.)
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
  if (n_jobs == 0u) return;  // (every block sees the same count)
  extern __shared__ __align__(16) uint32_t smem[];
  const AutoFillDev& A = S.af;
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id(), lt = (1u << lane) - 1u;
  uint4* const entries = reinterpret_cast<uint4*>(smem);               // [2][AF_BATCH], in turn
  uint4* const specials = entries + 2 * AF_BATCH;                      // [2][AF_SPEC], in turn
  uint4* const exits = specials + 2 * AF_SPEC;                         // [AF_EXITS] where in ga_wide_exit, count, -, context
  unsigned long long* const seen = reinterpret_cast<unsigned long long*>(exits + AF_EXITS);
  Contexts C0;
  C0.org = reinterpret_cast<uint2*>(seen + AF_SEEN);
  C0.exp = C0.org + AF_CTX;
  C0.lhs = reinterpret_cast<uint32_t*>(C0.exp + AF_CTX);
  C0.pool = C0.lhs + AF_CTX;
  C0.hash = C0.pool + AF_POOL;
  C0.cap = AF_CTX, C0.hash_mask = AF_CTX_HASH - 1u, C0.pool_cap = AF_POOL;
  uint32_t* const pre = C0.hash + AF_CTX_HASH;  // [AF_BATCH + 1]
  uint32_t* const ctl = pre + AF_BATCH + 4;
  uint32_t* const stage = ctl + AC_WORDS;
  uint32_t* const buf = stage + AF_STAGE;
  uint32_t* const work = buf + AF_BUF;
  uint32_t* const hset = work + AF_WORK;
  uint16_t* const owner = reinterpret_cast<uint16_t*>(hset + AF_HSET);  // [AF_OWNER] the thread to whom the first child of a piece belongs
  uint4* const stack = A.stack + (size_t)blockIdx.x * A.stack_cap;  // threads that found no room in `entries`
  for (uint32_t i = tid; i < AF_HSET; i += AF_THREADS) hset[i] = EMPTY_SLOT;
  uint32_t looked_up = 0, contexts = 0;
  // (expansions look items up one after the other: what fits is brought near at once)
  for (uint32_t i = tid * 8u; i < min(G.D, 8u * AF_THREADS); i += 8u * AF_THREADS) {
    uint32_t v;
    asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(G.ga_item + 4u * i));
    (void)v;
  }
  bool rows_left = true;
  const uint32_t parts = A.parts;  // (a power of two)

  for (;;) {
    // ---- (a share of) a row, or, when there is none left, a unit of work that another block gives
    // (they are taken by blocks that run: nobody ever waits for a block that has not started)
    __syncthreads();
    if (tid == 0) ctl[AC_JOB] = rows_left ? atomicAdd(&S.counters[CNT_AF_TICKET], 1u) : 0xFFFFFFFFu;
    __syncthreads();
    uint32_t j = ctl[AC_JOB] / parts, part = ctl[AC_JOB] & (parts - 1u);
    uint32_t* unit = nullptr;
    rows_left = j < n_jobs;
    if (j >= n_jobs) {
      __syncthreads();
      if (tid == 0) {
        const uint32_t ticket = atomicAdd(&S.counters[CNT_AF_TAKEN], 1u);
        uint32_t got = 0;
        if (ticket < A.unit_cap) {
          for (uint32_t polls = 0;; ++polls) {
            if (ld_acquire(&A.unit_flag[ticket]) == S.gen) {
              got = 1u;
              break;
            }
            if (ld_acquire(&S.counters[CNT_AF_ACTIVE]) == 0u || ld_acquire(&S.counters[CNT_BAR_ERR])) break;  // all is done
            if (polls > poll_limit(S, 22)) {
              diag(S, DIAG_WAIT_QUEUE);
              atomicExch(&S.counters[CNT_BAR_ERR], 1u);  // the fill is given up: its rows get all-zero masks
              break;
            }
            __nanosleep(400);
          }
        }
        ctl[AC_JOB] = got ? ticket : 0xFFFFFFFFu;
        ctl[AC_BASE] = vload(&S.counters[CNT_AF_GIVEN]);
      }
      __syncthreads();
      const uint32_t u = ctl[AC_JOB];
      if (u == 0xFFFFFFFFu) break;
      unit = A.units + (size_t)u * AU_WORDS;
      j = __ldcg(unit + AU_ROWJOB), part = __ldcg(unit + AU_PART);
    }
    const uint32_t row = S.jobs[j];
    const uint32_t* chart = S.arena + S.row_chart[row];
    uint32_t* const mask = S.mask_rows + (size_t)S.row_mask[row] * G.Wm;
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
    const bool begins = !unit && part == 0u;
    auto eos_word = [&](uint32_t i) -> uint32_t { return (accepting && G.eos >= 0 && i == (uint32_t)G.eos >> 5) ? 1u << ((uint32_t)G.eos & 31u) : 0u; };
    if (begins && parts > 1u) {  // the mask is cleared first: the other blocks of the row wait for that
      for (uint32_t i = tid; i < G.Wm; i += AF_THREADS) mask[i] = eos_word(i);
      __threadfence();
    }
    __syncthreads();
    if (begins && parts > 1u && tid == AF_THREADS - 1)
      asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(A.unit_flag + A.unit_cap + j), "r"(S.gen) : "memory");
    for (uint32_t i = tid; i < AF_SEEN; i += AF_THREADS) seen[i] = 0ull;
    if (tid < AC_WORDS) ctl[tid] = 0u;
    if (tid < AF_CTX_HASH) C0.hash[tid] = 0u;
    uint32_t side = 0;  // the threads of this round are entries[side]
    __syncthreads();
    if (unit) {
      const uint32_t n = __ldcg(unit + AU_N), nc = __ldcg(unit + AU_NCTX), np = __ldcg(unit + AU_POOL);
      const uint32_t* src = unit + AU_HDR;
      uint32_t* dst = reinterpret_cast<uint32_t*>(C0.org);  // org, exp, lhs and pool follow one another here and there
      for (uint32_t i = tid; i < 5u * AF_CTX + np; i += AF_THREADS) dst[i] = __ldcg(src + i);
      const uint4* th = reinterpret_cast<const uint4*>(unit + AU_HDR + 5 * AF_CTX + AF_POOL);
      for (uint32_t i = tid; i < n; i += AF_THREADS) entries[i] = __ldcg(th + i);
      __syncthreads();
      if (warp == 0) {
        for (uint32_t c = 0; c < nc; ++c) {
          const uint2 o = C0.org[c];
          uint32_t slot = context_hash(C0.lhs[c], C0.pool + o.x, o.y) & (AF_CTX_HASH - 1u);
          while (C0.hash[slot]) slot = (slot + 1u) & (AF_CTX_HASH - 1u);
          __syncwarp();
          if (lane == 0) C0.hash[slot] = c + 1u;
          __syncwarp();
        }
        if (lane == 0) ctl[AC_NEXT] = n, ctl[AC_NCTX] = nc, ctl[AC_POOL] = np;
      }
    } else if (warp == 0) {  // the kernel of the chart's last set starts the first threads
      const uint32_t lo = J.off[J.m - 1u], hi = J.off[J.m], self = J.m - 1u;
      uint32_t* b = hi - lo <= AF_BUF ? buf : big_area(A) + A.big_cap / 4u + A.big_cap / 2u;
      uint32_t n = 0;
      bool ok = hi - lo <= A.big_cap;
      if (ok)
        for (uint32_t base = lo; base < hi; base += 32) {
          const uint32_t k = base + lane;
          const uint32_t it = k < hi ? J.items[k] : 0u;
          bool take = k < hi && ((it >> 16) != self || (it & 0xFFFFu) == ITEM_START);
          if (take && k > lo && (it & 0xFFFFu) != 0u && J.items[k - 1u] == it - 1u)  // the item before it skips to it
            take = !(__ldg(&G.ga_item[4u * ((it & 0xFFFFu) - 1u) + 3u]) & GA_SKIPS);
          const uint32_t bal = __ballot_sync(FULL, take);
          if (take) b[n + __popc(bal & ((1u << lane) - 1u))] = (it << 16) | (it >> 16);
          n += __popc(bal);
        }
      __syncwarp();
      uint2 list = make_uint2(0u, 0u);
      Contexts C = C0;
      if (ok && !(ok = group_items(G, C, ctl, b, n, list))) {
        spill_contexts(C, ctl, A);
        ok = group_items(G, C, ctl, b, n, list);  // (sorted and without repeats already)
      }
      const uint4 root = __ldg(reinterpret_cast<const uint4*>(G.ga_node));
      uint32_t top = 0;
      for (uint32_t base = 0; base < list.y; base += 32) {
        const uint32_t i = base + lane;
        const uint2 x = i < list.y ? reinterpret_cast<const uint2*>(C.pool)[list.x / 2u + i] : make_uint2(0u, 0u);
        const uint32_t wide = i < list.y ? __ldg(&G.ga_item[4u * (x.y >> 16) + 2u]) : GA_DEAD;
        uint4 en = make_uint4(root.x, root.y >> 8, x.x, x.y & 0xFFFFu);
        bool take = i < list.y && en.y != 0u;
        if (wide != GA_DEAD) {  // most of the vocabulary follows from this item alone
          const uint4 r = __ldg(reinterpret_cast<const uint4*>(G.ga_wide_rec) + wide);
          const uint32_t at = atomicAdd(&ctl[AC_NWIDE], 1u);
          if (at < AF_EXITS) {  // (those that find no room start threads like any other)
            ctl[AC_WIDE + at] = r.x;
            if (r.z) exits[atomicAdd(&ctl[AC_NEXITS], 1u)] = make_uint4(r.y, r.z, 0u, en.w);
            take = false;
          }
        }
        const uint32_t bal = __ballot_sync(FULL, take);
        const uint32_t at = top + __popc(bal & ((1u << lane) - 1u));
        if (take && at < AF_BATCH) entries[at] = en;
        else if (take) reinterpret_cast<uint2*>(C.pool)[list.x / 2u + at - AF_BATCH] = x;  // they wait in the list, closed up
        top += __popc(bal);
      }
      if (lane == 0) {
        ctl[AC_NEXT] = min(top, AF_BATCH);
        ctl[AC_LIST] = list.x, ctl[AC_LIST_END] = top > AF_BATCH ? top - AF_BATCH : 0u;
        if (!ok) ctl[AC_FAIL] = 1u + DIAG_SET_SCRATCH;
      }
    }
    __syncthreads();
    if (!unit) {
      if (part && tid == 0)  // the block that began with the row clears the mask
        for (uint32_t polls = 0; ld_acquire(A.unit_flag + A.unit_cap + j) != S.gen; ++polls) {
          if (polls > poll_limit(S, 22)) {
            diag(S, DIAG_WAIT_GRID);
            atomicExch(&S.counters[CNT_BAR_ERR], 1u);
            ctl[AC_FAIL] = AF_GIVEN_UP;
            break;
          }
          if (polls) __nanosleep(64);
        }
      __syncthreads();
      // what follows from wide items, four words of a thread under way at once; a row's blocks share them (one dependent read
      // after the other, by the block that began, they took 15,000 of the 150,000 cycles of a row of a JSON schema)
      const uint32_t nw = min(ctl[AC_NWIDE], AF_EXITS), step = parts * AF_THREADS;
      if (parts == 1u) {
        for (uint32_t i = tid; i < G.Wm; i += 4u * AF_THREADS) {
          uint32_t v[4];
#pragma unroll
          for (uint32_t u = 0; u < 4; ++u) v[u] = eos_word(i + u * AF_THREADS);
          for (uint32_t k = 0; k < nw; ++k) {
            const uint32_t* src = G.ga_wide_mask + (size_t)ctl[AC_WIDE + k] * G.Wm;
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) v[u] |= i + u * AF_THREADS < G.Wm ? __ldg(src + i + u * AF_THREADS) : 0u;
          }
#pragma unroll
          for (uint32_t u = 0; u < 4; ++u)
            if (i + u * AF_THREADS < G.Wm) mask[i + u * AF_THREADS] = v[u];
        }
      }
      for (uint32_t k = 0; parts > 1u && k < nw; ++k) {
        const uint32_t* src = G.ga_wide_mask + (size_t)ctl[AC_WIDE + k] * G.Wm;
        for (uint32_t i = part * AF_THREADS + tid; i < G.Wm; i += 4u * step) {
          uint32_t v[4];
#pragma unroll
          for (uint32_t u = 0; u < 4; ++u) v[u] = i + u * step < G.Wm ? __ldg(src + i + u * step) : 0u;
#pragma unroll
          for (uint32_t u = 0; u < 4; ++u)
            if (v[u]) atomicOr(&mask[i + u * step], v[u]);
        }
      }
    }
    const uint32_t looked_up_before = looked_up;
    if (tid == AF_THREADS - 1) ctl[AC_BEGAN] = (uint32_t)(clock64() >> 10);

    bool spilled = false;
    // the expansion of a context (offset into pool, count), and its elements
    auto expansion = [&](uint32_t c) -> uint2 { return spilled ? global_contexts(A).exp[c] : C0.exp[c]; };
    auto element = [&](uint32_t off, uint32_t k) -> uint2 {
      return spilled ? reinterpret_cast<const uint2*>(global_contexts(A).pool)[off / 2u + k] : reinterpret_cast<const uint2*>(C0.pool)[off / 2u + k];
    };
    // false: this thread was started here a moment ago
    auto start = [&](uint32_t first, uint32_t rule_ctx) -> bool {
      const uint32_t slot = (first * 0x9E3779B1u ^ rule_ctx * 0x85EBCA6Bu) >> 23;
      static_assert(AF_SEEN == 512, "the slot is the upper nine bits");
      const unsigned long long key = (unsigned long long)first << 32 | rule_ctx;
      volatile unsigned long long* p = seen + slot;
      const bool fresh = *p != key;
      *p = key;
      return fresh;
    };
    for (;;) {  // ---- rounds
      uint32_t n = min(ctl[AC_NEXT], AF_BATCH), ns = min(ctl[AC_SPEC], AF_SPEC), gtop = ctl[AC_GTOP], nx = ctl[AC_NEXITS];
      const uint32_t first_at = ctl[AC_LIST_AT], first_left = ctl[AC_LIST_END] - first_at;  // items of the last set that have not started
      if (ctl[AC_FAIL] || n + ns + gtop + nx + first_left == 0u) break;
      spilled = ctl[AC_SPILLED] != 0u;
      const uint32_t waiting = ctl[AC_WAITING];
      __syncthreads();
      uint4* const cur = entries + side * AF_BATCH;
      uint4* const nxt = entries + (side ^ 1u) * AF_BATCH;
      uint4* const spec = specials + side * AF_SPEC;
      uint4* const spec_nxt = specials + (side ^ 1u) * AF_SPEC;
      if (tid == 0) ctl[AC_NEXT] = 0u, ctl[AC_SPEC] = 0u, ctl[AC_OVF] = 0u;
      if (tid == AF_THREADS - 1) {  // (looked at when the round ends; nobody waits for them until then)
        peek(ctl + AC_PEEK, S.counters + CNT_AF_TICKET);
        peek(ctl + AC_PEEK + 4u, A.row_gone + (j & ~3u));
      }
      // The stack cannot run over.  A round pushes at most the threads that its specials and its list start and two entries for each
      // child it looks up, and takes no more than fits above the reserve.  On a crowded stack one entry is taken at a time, from the top:
      // depth first the stack grows by two entries a child along one path of the trie (A.reserve, which has room for `cur` and `spec`, too).
      const bool tight = A.stack_cap - gtop < A.reserve + AF_TIGHT, pops = !tight && gtop && n < AF_BATCH && ns < AF_SPEC;
      if (tight) {
        for (uint32_t i = tid; i < n; i += AF_THREADS) stack[gtop + i] = cur[i];
        for (uint32_t i = tid; i < ns; i += AF_THREADS) stack[gtop + n + i] = spec[i];
        gtop += n + ns;
        __syncthreads();
        const uint4 v = stack[--gtop];
        ns = v.z == AF_SPAWN ? 1u : 0u, n = 1u - ns, nx = 0u;
        if (tid == 0) (ns ? spec : cur)[0] = v;
      } else if (pops) {
        const uint32_t take = min(min(AF_BATCH - n, AF_SPEC - ns), gtop);
        static_assert(AF_SPEC <= AF_THREADS, "one entry to a thread");
        gtop -= take;
        const uint4 v = tid < take ? stack[gtop + tid] : make_uint4(0u, 0u, 0u, 0u);
        const bool is_spec = tid < take && v.z == AF_SPAWN, is_thread = tid < take && v.z != AF_SPAWN;
        const uint32_t bt = __ballot_sync(FULL, is_thread), bs = __ballot_sync(FULL, is_spec);
        uint32_t at = 0, at_spec = 0;
        if (lane == 0 && bt) at = atomicAdd(&ctl[AC_POPPED], __popc(bt));
        if (lane == 0 && bs) at_spec = atomicAdd(&ctl[AC_POPPED_SPEC], __popc(bs));
        at = __shfl_sync(FULL, at, 0), at_spec = __shfl_sync(FULL, at_spec, 0);
        if (is_thread) cur[n + at + __popc(bt & lt)] = v;
        if (is_spec) spec[ns + at_spec + __popc(bs & lt)] = v;
      } else if (n < AF_BATCH && first_left) {
        const uint32_t take = min(AF_BATCH - n, first_left);
        const uint4 root = __ldg(reinterpret_cast<const uint4*>(G.ga_node));
        for (uint32_t i = tid; i < take; i += AF_THREADS) {
          const uint2 x = element(ctl[AC_LIST], first_at + i);
          cur[n + i] = make_uint4(root.x, root.y >> 8, x.x, x.y & 0xFFFFu);
        }
        if (tid == 0) ctl[AC_LIST_AT] = first_at + take;
        n += take;
      }
      __syncthreads();
      if (pops) n += ctl[AC_POPPED], ns += ctl[AC_POPPED_SPEC];
      const uint32_t places = tight ? 0u : A.stack_cap - A.reserve - gtop;  // (at least AF_TIGHT)
      auto overflow = [&](const uint4& v) {
        const uint32_t p = atomicAdd(&ctl[AC_OVF], 1u);
        if (gtop + p < A.stack_cap) stack[gtop + p] = v;
        else ctl[AC_FAIL] = 1u + DIAG_QUEUE_FULL;  // (cannot happen, see above)
      };
      if (ns + nx) {
        // ---- expansions: contexts that have none yet, then the threads they start, in this very round as far as there is room
        const bool list = nx != 0u && n < AF_BATCH / 2u;  // a list of nodes waits its turn
        const uint4 ex = list ? exits[nx - 1u] : make_uint4(0u, 0u, 0u, 0u);
        const uint4 en = tid < ns ? spec[tid] : make_uint4(0u, 0u, 0u, 0u);
        const uint32_t en_ctx = en.w & 0xFFFFu;
        if (__syncthreads_or((tid < ns && expansion(en_ctx).y == CTX_NEW) || (list && tid == 0 && expansion(ex.w).y == CTX_NEW))) {
          if (warp == 0) {
            Contexts C = spilled ? global_contexts(A) : C0;
            for (uint32_t base = 0; base <= ns; base += 32) {  // (the list's comes last)
              const uint32_t i = base + lane;
              const uint32_t c = i < ns ? spec[i].w & 0xFFFFu : i == ns && list ? ex.w : CTX_NEW;
              for (uint32_t todo = __ballot_sync(FULL, c != CTX_NEW && C.exp[c].y == CTX_NEW); todo;) {
                const uint32_t x = __shfl_sync(FULL, c, __ffs(todo) - 1);
                if (!expand_context(G, A, C, J, x, ctl, work, hset, buf) && lane == 0) ctl[AC_FAIL] = 1u + DIAG_SET_TABLE;
                todo &= ~__ballot_sync(FULL, c == x);
              }
            }
          }
          __syncthreads();
          spilled = ctl[AC_SPILLED] != 0u;
        }
        if (tid == 0) ctl[AC_NBUF] = n;
        __syncthreads();
        auto begin = [&](bool yes, uint32_t first, uint32_t kids, const uint2& el) {  // (by all lanes of a warp)
          yes = yes && start(first, el.y);
          const uint32_t bal = __ballot_sync(FULL, yes);
          if (bal == 0u) return;
          uint32_t at = 0;
          if (lane == 0) at = atomicAdd(&ctl[AC_NBUF], __popc(bal));
          at = __shfl_sync(FULL, at, 0) + __popc(bal & ((1u << lane) - 1u));
          const uint4 v = make_uint4(first, kids, el.x, el.y & 0xFFFFu);
          if (yes && at < AF_BATCH) cur[at] = v;
          else if (yes) overflow(v);
        };
        if (warp * 32u < ns) {
          // (all of its elements as a rule; what might not fit the stack is left for another round)
          const uint2 spawns = tid < ns ? expansion(en_ctx) : make_uint2(0u, 0u);
          const uint32_t from = en.w >> 16, count = min(spawns.y - min(from, spawns.y), tight ? 1u : max(1u, places / (2u * ns)));
          const uint32_t most_of = __reduce_max_sync(FULL, count);
          if (from + count < spawns.y) overflow(make_uint4(en.x, en.y, AF_SPAWN, (from + count) << 16 | en_ctx));
          for (uint32_t q = 0; q < most_of; ++q) begin(q < count, en.x, en.y, q < count ? element(spawns.x, from + q) : make_uint2(0u, 0u));
        }
        if (list) {
          const uint2 x = expansion(ex.w);
          const uint32_t nodes = x.y ? min(ex.y, max(parts * (AF_BATCH / 2u / x.y), 32u)) : ex.y;  // (at most 2048 threads)
          const bool by_specials = x.y > AF_LIST_STARTS;
          if (x.y)
            for (uint32_t base = warp * 32u; base < nodes; base += AF_THREADS) {
              bool v = base + lane < nodes;
              const uint2 nd = v ? __ldg(reinterpret_cast<const uint2*>(G.ga_wide_exit) + ex.x + base + lane) : make_uint2(0u, 0u);
              // (blocks that share a row all start the threads of nodes of depth 1, and deal out the others)
              if (parts > 1u && (nd.x < G.ga_lvl2 || nd.x >= G.ga_lvl3)) v = v && ((base + lane) & (parts - 1u)) == part;
              if (by_specials) {
                v = v && start(nd.x, 0xFFFF0000u | ex.w);
                const uint4 b = make_uint4(nd.x, nd.y, AF_SPAWN, ex.w);
                const uint32_t p = v ? atomicAdd(&ctl[AC_SPEC], 1u) : 0u;
                if (v && p < AF_SPEC) spec_nxt[p] = b;
                else if (v) overflow(b);
                continue;
              }
              for (uint32_t q = 0; q < x.y; ++q) begin(v, nd.x, nd.y, element(x.x, q));
            }
          __syncthreads();
          if (tid == 0) {
            if (nodes == ex.y) ctl[AC_NEXITS] = nx - 1u;
            else exits[nx - 1u] = make_uint4(ex.x + nodes, ex.y - nodes, 0u, ex.w);
          }
        }
        __syncthreads();
        n = min(ctl[AC_NBUF], AF_BATCH);
      }
      if (waiting && n >= AF_SHARE && looked_up - looked_up_before >= AF_HEAVY && !spilled) {
        // ---- other blocks wait: entry i stays here when i is a multiple of units + 1, else it goes to unit i % (units + 1) - 1
        const uint32_t units = min(min(waiting, n / 128u - 1u), AF_MAX_UNITS);
        if (tid == 0) {
          const uint32_t at = atomicAdd(&S.counters[CNT_AF_POSTED], units);
          const uint32_t fit = at >= A.unit_cap ? 0u : min(units, A.unit_cap - at);
          if (fit == units) atomicAdd(&S.counters[CNT_AF_ACTIVE], units);
          ctl[AC_BASE] = fit == units ? at : 0xFFFFFFFFu;  // (near the end of the units' storage nothing is given any more)
        }
        __syncthreads();
        const uint32_t at = ctl[AC_BASE];
        if (at != 0xFFFFFFFFu) {
          const uint32_t nc = ctl[AC_NCTX], np = ctl[AC_POOL];
          const uint32_t* src = reinterpret_cast<const uint32_t*>(C0.org);
          for (uint32_t u = 0; u < units; ++u) {
            uint32_t* dst = A.units + (size_t)(at + u) * AU_WORDS;
            for (uint32_t i = tid; i < 5u * AF_CTX + np; i += AF_THREADS) dst[AU_HDR + i] = src[i];
            if (tid == 0) dst[AU_ROWJOB] = j, dst[AU_N] = (n + units - 1u - u) / (units + 1u), dst[AU_NCTX] = nc, dst[AU_POOL] = np, dst[AU_PART] = part;
          }
          uint4 keep[AF_PER];
#pragma unroll
          for (uint32_t k = 0; k < AF_PER; ++k) {
            const uint32_t i = k * AF_THREADS + tid;
            if (i < n) {
              keep[k] = cur[i];
              const uint32_t to = i % (units + 1u);
              if (to)
                reinterpret_cast<uint4*>(A.units + (size_t)(at + to - 1u) * AU_WORDS + AU_HDR + 5 * AF_CTX + AF_POOL)[i / (units + 1u)] = keep[k];
            }
          }
          __threadfence();
          __syncthreads();
          if (tid < units) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(A.unit_flag + at + tid), "r"(S.gen) : "memory");
#pragma unroll
          for (uint32_t k = 0; k < AF_PER; ++k) {
            const uint32_t i = k * AF_THREADS + tid;
            if (i < n && i % (units + 1u) == 0u) cur[i / (units + 1u)] = keep[k];
          }
          n = (n + units) / (units + 1u);
          __syncthreads();
        }
      }
      // ---- the threads' children, 32 to a piece
      uint32_t w[AF_PER], sum = 0;
#pragma unroll
      for (uint32_t u = 0; u < AF_PER; ++u) {
        const uint32_t i = tid * AF_PER + u;
        w[u] = i < n ? cur[i].y : 0u;
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
      for (uint32_t u = 0; u < AF_PER; ++u) {
        const uint32_t i = tid * AF_PER + u;
        if (i <= n) pre[i] = before;  // (pre[n] = the total)
        for (uint32_t piece = (before + 31u) / 32u; piece * 32u < before + w[u]; ++piece) owner[piece] = (uint16_t)i;
        before += w[u];
      }
      if (n == AF_BATCH && tid == 0) pre[n] = total;
      const uint32_t pushed = ctl[AC_OVF];
      __syncthreads();
      if (!tight && 2u * total > places - pushed) {  // more children than can be pushed: the last threads wait
        uint32_t fit = 0;
#pragma unroll
        for (uint32_t u = 0; u < AF_PER; ++u) {
          const uint32_t i = u * AF_THREADS + tid;
          fit += __syncthreads_count(i < n && 2u * pre[i + 1u] <= places - pushed);
        }
        for (uint32_t i = fit + tid; i < n; i += AF_THREADS) overflow(cur[i]);
        n = fit, total = pre[n];
        __syncthreads();
      }
      looked_up += total;
      for (uint32_t base = warp * 32u; base < total; base += AF_THREADS) {
        const uint32_t lo = owner[base / 32u];
        const uint32_t nb = lo + 1u + lane <= n ? pre[lo + 1u + lane] - base : 32u;  // where the threads after it begin
        const uint32_t starts = __reduce_or_sync(FULL, nb < 32u ? 1u << nb : 0u);
        const uint32_t e = lo + __popc(starts & (0xFFFFFFFFu >> (31u - lane)));
        bool goes_on = false, starts_one = false, special = false;
        uint4 a, b;
        uint4 nd = make_uint4(0u, 0u, 0u, 0u);
        uint32_t many = 0;
        uint4 en = make_uint4(0u, 0u, 0u, 0u);
        uint32_t child = 0;
        bool ours = base + lane < total;
        if (ours) {
          en = cur[e];
          child = en.x + (base + lane - pre[e]);
          // blocks that share a row share the nodes of depth 2, and with them what lies below
          if (parts > 1u && child >= G.ga_lvl2 && child < G.ga_lvl3) ours = (child & (parts - 1u)) == part;
        }
        if (ours) {
          nd = __ldg(reinterpret_cast<const uint4*>(G.ga_node) + child);
          const uint32_t t = ga_next(G, en.z, nd.y & 0xFFu);
          if (t < GA_UNKNOWN) {
            if (nd.w == 1u) atomicOr(&mask[nd.z >> 5], 1u << (nd.z & 31u));
            else many = nd.w;
            const uint32_t kids = nd.y >> 8;
            if (kids) {
              goes_on = (t & ~GA_EXIT) != GA_NONE;
              a = make_uint4(nd.x, kids, t & ~GA_EXIT, en.w);
              if (t & GA_EXIT) {
                const uint2 x = expansion(en.w);
                if (x.y) {
                  const uint2 el = x.y == 1u ? element(x.x, 0u) : make_uint2(AF_SPAWN, 0xFFFF0000u | en.w);
                  starts_one = start(nd.x, el.y);
                  special = starts_one && x.y != 1u;
                  b = make_uint4(nd.x, kids, el.x, el.y & 0xFFFFu);
                }
              }
            }
          } else if (t == GA_UNKNOWN) {
            ctl[AC_FAIL] = 1u + DIAG_ROOT_FAILED;  // (cannot happen: the automaton covers the vocabulary)
          }
        }
        __syncwarp();
        if (__any_sync(FULL, many != 0u)) set_tokens(G, mask, nd.z, many);
        const uint32_t ba = __ballot_sync(FULL, goes_on), bb = __ballot_sync(FULL, starts_one && !special);
        if (ba | bb) {
          uint32_t at = 0;
          if (lane == 0) at = atomicAdd(&ctl[AC_NEXT], __popc(ba) + __popc(bb));
          at = __shfl_sync(FULL, at, 0);
          if (goes_on) {
            const uint32_t p = at + __popc(ba & lt);
            if (p < AF_BATCH) nxt[p] = a;
            else overflow(a);
          }
          if (starts_one && !special) {
            const uint32_t p = at + __popc(ba) + __popc(bb & lt);
            if (p < AF_BATCH) nxt[p] = b;
            else overflow(b);
          }
        }
        if (special) {
          const uint32_t p = atomicAdd(&ctl[AC_SPEC], 1u);
          if (p < AF_SPEC) spec_nxt[p] = b;
          else overflow(b);
        }
      }
      side ^= 1u;
      __syncthreads();
      if (tid == 0) {
        ctl[AC_GTOP] = gtop + ctl[AC_OVF];
        if (pops) ctl[AC_POPPED] = ctl[AC_POPPED_SPEC] = 0u;
      }
      if (tid == AF_THREADS - 1) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        const uint32_t t = ctl[AC_PEEK + CNT_AF_TAKEN - CNT_AF_TICKET], p = ctl[AC_PEEK + CNT_AF_POSTED - CNT_AF_TICKET];
        const bool gone = ctl[AC_PEEK + 4u + (j & 3u)] == S.gen, late = (uint32_t)(clock64() >> 10) - ctl[AC_BEGAN] > AF_KCYCLES;
        ctl[AC_WAITING] = t > p ? t - p : 0u;
        if ((gone || late) && !ctl[AC_FAIL]) ctl[AC_FAIL] = gone ? AF_GONE : AF_LATE;
      }
      __syncthreads();
    }
    contexts += ctl[AC_NCTX];
    if (tid == 0 && ctl[AC_FAIL] && ctl[AC_FAIL] < AF_GONE) {  // too many contexts, or too long a time: the row is left to a sweep by Earley steps
      if (ctl[AC_FAIL] != AF_LATE) diag(S, ctl[AC_FAIL] - 1u);
      if (atomicExch(A.row_gone + j, S.gen) != S.gen)  // (its other blocks stop when they see that)
        *reinterpret_cast<volatile uint32_t*>(A.given + atomicAdd(&S.counters[CNT_AF_GIVEN], 1u)) = S.gen << 16 | j;
    }
    // ---- the next row
    __threadfence();
    __syncthreads();
    if (tid == 0) atomicSub(&S.counters[CNT_AF_ACTIVE], 1u);
  }
  if (tid == 0 && looked_up) {
    stat_add(S, CNT_STAT_TRANS, looked_up);
    stat_add(S, CNT_STAT_LOCAL, contexts);
  }
  // ---- rows that were given up, swept by blocks that have nothing else to do any more: who gives one up comes here later itself.  Only
  // blocks that look for tables wait, and who has tables waits for nobody.
  for (bool given = ctl[AC_BASE] != 0u; given;) {
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
        ctl[AC_BASE] = v & 0xFFFFu;
        __threadfence();
      }
      ctl[AC_JOB] = slot;
    }
    __syncthreads();
    const uint32_t slot = ctl[AC_JOB], row = slot == 0xFFFFFFFFu ? 0u : S.jobs[ctl[AC_BASE]];
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

constexpr uint32_t AF_SMEM = (2 * AF_BATCH + 2 * AF_SPEC + AF_EXITS) * 16 + AF_SEEN * 8 + AF_OWNER * 2 + (5 * AF_CTX + AF_POOL + AF_CTX_HASH + AF_BATCH + 4 + AC_WORDS + AF_STAGE + AF_BUF + AF_WORK + AF_HSET) * 4;
static_assert(block_sweep_words(AF_WARPS, MAX_NONTERMINALS / 32u) * 4u <= AF_SMEM, "a row that is given up is swept in the same shared memory");

// Places of a block's stack that only its depth-first rounds use: two for each child along the longest path of the trie and one for
// what is left of a special at each of its nodes, and what a round may hold or has put back when the last places above are taken.
uint32_t automaton_fill_reserve(const GrammarDev& G) {
  return 2u * G.ga_path + MAX_TOKEN_BYTES + 1u + 2u * (AF_BATCH + AF_SPEC) + 32u;
}
uint32_t automaton_fill_warps() { return AF_WARPS; }
uint32_t automaton_fill_least_stack(const GrammarDev& G) { return automaton_fill_reserve(G) + AF_TIGHT; }

void automaton_fill_layout(const GrammarDev& G, uint32_t rows, uint32_t max_blocks, AutoFillDev& A) {
  A.reserve = automaton_fill_reserve(G);
  A.scratch_words = 7u * A.ctx_cap + A.pool_cap + A.big_cap / 4u + A.big_cap / 2u + A.big_cap;
  A.unit_words = AU_WORDS;
  // few rows: several blocks take one, so that the chip is filled (a small trie gives the others nothing to do)
  A.parts = 1;
  while (A.parts < 8u && (uint64_t)rows * A.parts * 2u <= max_blocks && A.parts * 2048u <= G.T) A.parts *= 2u;
  A.grid = (uint32_t)std::min<uint64_t>(max_blocks, (uint64_t)rows * std::max(A.parts, 1u + G.T / 16384u));
}

cudaError_t configure_automaton_fill() {
  return cudaFuncSetAttribute((const void*)automaton_fill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AF_SMEM);
}

void launch_automaton_fill(const GrammarDev& G, const StateDev& S, cudaStream_t st) {
  launch_overlapped(automaton_fill_kernel, dim3(S.af.grid), dim3(AF_THREADS), AF_SMEM, st, G, S);
}

}  // namespace fmt
