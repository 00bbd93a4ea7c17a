// One token on a whole pruned chart, by one warp (used when a sequence advances).  Per byte:
//   Scan -> Complete (fixpoint) -> Predict; after the token's last byte: Compact (Section 4.2.3),
// which leaves exactly the chart that compacting after every byte would leave (an item needed at
// the end was needed at every step before), at a fraction of the work,
// and the state cache: the pruned chart, densely renumbered, is the cache key (Section 5.2: token
// sequences that differ may still end in one and the same pruned chart, and then share an entry).
//
// Compact keeps, besides the unfinished items of the new last set, exactly the items a later
// Complete can still read: an item (Y -> mu . A nu, o') of an earlier set o stays iff a kept item
// with left-hand side A and origin o exists (Figure 3: sets not on a reference chain of the last
// set's items are removed; completed items go once their set is done).
//
// What bounds it: the chain of instructions of one warp, some 5,000 for a token of four bytes of JSON, 8 to 10 cycles each.  The loops here
// and in earley_device.cuh are not unrolled and each helper stands in the steps once: the kernel's code came to 400 KB, of which a
// step touches every part a few times, and a quarter of its time went into fetching it (now 210 KB, a twentieth).  With that, runs
// of single items taken in one go, predicted items copied from lists, and the new chart built in shared memory: 400 advances of 32 rows of
// ambiguous JSON 28.2 -> 25.7 ms, 24 decoding steps of 8 rows of JSON 2.43 -> 2.25 ms, 16 of 64 rows of a JSON schema 1.72 -> 1.57 ms.
#pragma once
#include "earley_device.cuh"

namespace fmt {

constexpr uint32_t ADV_CUR_CAP = 2048;     // items of the sets a token adds to a chart (shared-memory arena)
constexpr uint32_t ADV_HSET = 2048;        // hash slots (power of two)
constexpr uint32_t ADV_MAX_ITEMS = 65536;  // items of a chart the live bitmap can describe
constexpr uint32_t ADV_PAIRS = 1024;       // (set, non-terminal) needs of one Compact
constexpr uint32_t ADV_MAX_SETS = 2048;
constexpr uint32_t ADV_NT_WORDS = 256;     // 2 * Nw, Nw <= 128
constexpr uint32_t ADV_STAGE = 2048;       // a source chart up to this many words is read from shared memory
constexpr uint32_t ADV_OUT = 1024;         // a new chart that cannot have more words is built in shared memory (the upper half of the bitmap)
constexpr uint32_t ADV_WARP_WORDS =
    ADV_CUR_CAP + ADV_HSET + ADV_MAX_ITEMS / 32 + ADV_PAIRS + ADV_MAX_SETS + ADV_NT_WORDS + W_CTRS + ADV_STAGE;

struct AdvScratch {
  WarpCtx w;
  uint32_t* live;   // [ADV_MAX_ITEMS/32] bitmap over the source chart's items
  uint32_t* pairs;  // [ADV_PAIRS]
  uint32_t* sets;   // [ADV_MAX_SETS] per-set live count, then new index
  uint32_t* stage;  // [ADV_STAGE]
  uint32_t* out;    // where the new chart is: in shared memory, if it is small, or where the caller asked for it
};

__device__ __forceinline__ AdvScratch adv_scratch(uint32_t* base) {
  AdvScratch s;
  s.w.cur = base;
  s.w.cur_cap = ADV_CUR_CAP;
  s.w.hset = base + ADV_CUR_CAP;
  s.w.hset_mask = ADV_HSET - 1;
  s.live = s.w.hset + ADV_HSET;
  s.pairs = s.live + ADV_MAX_ITEMS / 32;
  s.sets = s.pairs + ADV_PAIRS;
  s.w.nt = s.sets + ADV_MAX_SETS;
  s.w.ctr = s.w.nt + ADV_NT_WORDS;
  s.stage = s.w.ctr + W_CTRS;
  return s;
}

struct ChartView {
  const uint32_t* off;  // set_off
  const uint32_t* items;
  __device__ __forceinline__ void operator()(uint32_t o, const uint32_t*& p, uint32_t& n) const {
    uint32_t a = off[o], b = off[o + 1];
    p = items + a;
    n = b - a;
  }
  __device__ __forceinline__ uint32_t fix(uint32_t item, uint32_t) const { return item; }
};

__device__ __forceinline__ void push_need(const AdvScratch& s, uint32_t o, uint32_t A) {
  uint32_t key = (o << 16) | A;
  int r = hset_insert(s.w.hset, s.w.hset_mask, key);
  if (r == 0) return;  // already asked for
  // r < 0 (hash full): ask again anyway, a repeated need only costs time
  uint32_t idx = atomicAdd(&s.w.ctr[W_NPAIRS], 1u);
  if (idx < ADV_PAIRS) s.pairs[idx] = key;
  else s.w.ctr[W_OVERFLOW] = 1u;
}

// The chart hash is a sum over (word index, value) pairs, so it can be accumulated while the
// words are written, in any order and by any lane.  Two independent 32-bit sums.
struct HashAcc {
  uint32_t h1 = 0, h2 = 0;
  __device__ __forceinline__ void add(uint32_t i, uint32_t v) {
    h1 += mix32(v ^ (i * 0x9E3779B1u));
    h2 += mix32((v + 0x632BE5ABu) ^ (i * 0x85EBCA77u));
  }
};
__device__ __forceinline__ void put(uint32_t* ch, HashAcc& h, uint32_t i, uint32_t v) {
  ch[i] = v;
  h.add(i, v);
}

// Write the last set (cur[0..n), unsorted, completed items already removed) and finish the header.
// dst already holds set_off[0..m_new) and the kept items of the earlier sets (`kept` of them), all
// accounted for in `h`.
__device__ __forceinline__ int finish_chart(const AdvScratch& s, uint32_t* dst, uint32_t dst_cap, uint32_t m_new,
                                            uint32_t kept, uint32_t n, bool accepting, HashAcc h) {
  const uint32_t lane = lane_id();
  uint32_t words = CH_HDR + (m_new + 2) + kept + n;
  if (words > dst_cap || kept + n >= ADV_MAX_ITEMS) return -1;
  sort_items(s.w.cur, n, 1u << 30);
  const uint32_t items_at = CH_HDR + (m_new + 2);
  #pragma unroll 1
  for (uint32_t i = lane; i < n; i += 32) put(dst, h, items_at + kept + i, s.w.cur[i]);
  if (lane == 0) {
    put(dst, h, CH_SETS, m_new + 1);
    put(dst, h, CH_ITEMS, kept + n);
    put(dst, h, CH_FLAGS, accepting ? CHART_ACCEPTING : 0u);
    put(dst, h, CH_WORDS, words);
    put(dst, h, 6, 0u);
    put(dst, h, 7, 0u);
    put(dst, h, CH_HDR + m_new, kept);          // first item of the last set
    put(dst, h, CH_HDR + m_new + 1, kept + n);  // end
  }
  #pragma unroll 1
  for (int d = 16; d > 0; d >>= 1) {
    h.h1 += __shfl_xor_sync(FULL, h.h1, d);
    h.h2 += __shfl_xor_sync(FULL, h.h2, d);
  }
  if (lane == 0) {
    dst[CH_HASH_LO] = h.h1;
    dst[CH_HASH_HI] = h.h2;
  }
  __syncwarp();
  return 1;
}

// The start chart: S[0] = closure of ($ -> . start, 0).
__device__ int chart_init(const GrammarDev& G, const AdvScratch& s, uint32_t* dst, uint32_t dst_cap) {
  const uint32_t lane = lane_id();
  if (lane < W_CTRS) s.w.ctr[lane] = 0u;
  clear_nt(G, s.w);
  if (lane == 0) add_item(G, s.w, ITEM_START);
  __syncwarp();
  ChartView none{nullptr, nullptr};
  complete_fixpoint(G, s.w, none, 0u, 0u);  // only collects post-dot non-terminals and the accept flag
  uint32_t hashed = min(s.w.ctr[W_NCUR], s.w.cur_cap);
  bool accepting = s.w.ctr[W_ACCEPT] != 0u;
  hset_clear_items(s.w, hashed);
  predict_into_cur(G, s.w, 0u);
  if (s.w.ctr[W_OVERFLOW]) {
    hset_clear_all(s.w.hset, s.w.hset_mask);
    clear_nt(G, s.w);
    return -1;
  }
  uint32_t n = drop_completed(G, s.w, min(s.w.ctr[W_NCUR], s.w.cur_cap));
  return finish_chart(s, dst, dst_cap, 0u, 0u, n, accepting, HashAcc{});
}

// Where set o of "source chart + the token's sets so far" lives.  Sets 0..m-1 are the source
// chart's, set m-1+L is the token's L-th.
struct TokenView {
  const uint32_t* soff;
  const uint32_t* sitems;
  uint32_t m;
  const uint32_t* arena;
  const uint32_t* lvl_off;  // [MAX_TOKEN_BYTES + 2] first item of each level in the arena
  __device__ __forceinline__ void operator()(uint32_t o, const uint32_t*& p, uint32_t& n) const {
    if (o < m) {
      uint32_t a = soff[o], b = soff[o + 1];
      p = sitems + a;
      n = b - a;
    } else {
      const uint32_t L = o - (m - 1);
      p = arena + lvl_off[L];
      n = lvl_off[L + 1] - lvl_off[L];
    }
  }
  __device__ __forceinline__ uint32_t fix(uint32_t item, uint32_t) const { return item; }
  // position of item k of set o in the live bitmap (source items first, then the arena)
  __device__ __forceinline__ uint32_t bit_base(uint32_t o, uint32_t n_items) const {
    return (o < m) ? soff[o] : n_items + lvl_off[o - (m - 1)];
  }
};

// Scan and Complete (Section 3.2) for sets that outgrow a warp's lanes - an ambiguous grammar's, of a hundred items and more
// out of as many origins.  What is in the set, and which (non-terminal, origin) have been completed, are bits in
// shared memory, and the waiting items of all sets that a wave of completions asks are dealt out to the lanes together:
// 58,000 cycles a byte in an ambiguous segment of sixty letters with a hash and one set asked after the other, now 15,000.  Returns the number of items in
// s.w.cur, GEN_FULL when they outgrow it; the bits must fit (gen_fits).
constexpr uint32_t GEN_FULL = 0xffffffffu;
__device__ __forceinline__ bool gen_fits(const GrammarDev& G, uint32_t index) {
  return G.D * (index + 1u) <= ADV_HSET * 32u && G.N * (index + 1u) <= ADV_PAIRS * 32u;
}
__device__ uint32_t gen_scan_complete(const GrammarDev& G, const AdvScratch& s, const TokenView& view, const uint32_t* set,
                                      uint32_t len, uint32_t byte, uint32_t index) {
  const uint32_t lane = lane_id(), lt = (1u << lane) - 1u, row = index + 1u;
  uint32_t* const in_set = s.w.hset;   // [D][row] bits
  uint32_t* const done = s.pairs;      // [N][row] bits
  const uint32_t set_words = (G.D * row + 31u) / 32u, done_words = (G.N * row + 31u) / 32u;
  __syncwarp();
  #pragma unroll 1
  for (uint32_t i = lane; i < set_words; i += 32) in_set[i] = 0u;
  #pragma unroll 1
  for (uint32_t i = lane; i < done_words; i += 32) done[i] = 0u;
  __syncwarp();
  uint32_t n = 0;
  auto add = [&](bool v, uint32_t key) {  // by all lanes; the items reached over nullable non-terminals come along
    const uint32_t more = v ? (G.info[key & 0xFFFFu] >> INFO_SKIP_SHIFT) & INFO_SKIP_MASK : 0u;
    #pragma unroll 1
    for (uint32_t j = 0;; ++j) {
      bool fresh = false;
      if (v && j <= more) {
        const uint32_t at = ((key & 0xFFFFu) + j) * row + (key >> 16), bit = 1u << (at & 31u);
        fresh = !(in_set[at >> 5] & bit) && !(atomicOr(&in_set[at >> 5], bit) & bit);
      }
      const uint32_t b = __ballot_sync(FULL, fresh);
      if (fresh && n + __popc(b & lt) < s.w.cur_cap) s.w.cur[n + __popc(b & lt)] = key + j;
      n += __popc(b);
      if (!__any_sync(FULL, v && j < more)) break;
    }
  };
  #pragma unroll 1
  for (uint32_t base = 0; base < len; base += 32) {
    const bool v = base + lane < len;
    const uint32_t it = v ? set[base + lane] : 0u;
    const Scanned sc = scan_item(G, it, v ? G.info[it & 0xFFFFu] : (KIND_NT << INFO_KIND_SHIFT), byte);
    if (__any_sync(FULL, sc.has_a)) add(sc.has_a, sc.a);
    if (__any_sync(FULL, sc.has_b)) add(sc.has_b, sc.b);
  }
  uint2* const ask = reinterpret_cast<uint2*>(s.live);  // per completion of a wave: where its set's items begin
  uint32_t* const want = s.live + 64;                   // its non-terminal and origin
  uint32_t* const from = s.live + 96;                   // its first place among the items dealt out
  #pragma unroll 1
  for (uint32_t head = 0; head < min(n, s.w.cur_cap);) {
    __syncwarp();
    const bool have = head + lane < n && head + lane < s.w.cur_cap;
    const uint32_t until = n;
    const uint32_t it = have ? s.w.cur[head + lane] : 0u;
    const uint32_t inf = have ? G.info[it & 0xFFFFu] : 0u, kind = inf >> INFO_KIND_SHIFT, a = inf & INFO_ARG_MASK;
    if (have && kind == KIND_NT) atomicOr(&s.w.nt[a >> 5], 1u << (a & 31u));
    if (have && kind == KIND_END && (it & 0xFFFFu) == ITEM_ACCEPT) s.w.ctr[W_ACCEPT] = 1u;
    bool asks = have && kind == KIND_END && (it >> 16) != index && (it & 0xFFFFu) != ITEM_ACCEPT;
    if (asks) {
      const uint32_t at = a * row + (it >> 16), bit = 1u << (at & 31u);
      asks = !(atomicOr(&done[at >> 5], bit) & bit);
    }
    const uint32_t* sp = nullptr;
    uint32_t sl = 0;
    if (asks) view(it >> 16, sp, sl);
    asks = sl != 0u;
    uint32_t incl = sl;
    #pragma unroll 1
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t t = __shfl_up_sync(FULL, incl, d);
      if ((int)lane >= d) incl += t;
    }
    const uint32_t total = __shfl_sync(FULL, incl, 31), ab = __ballot_sync(FULL, asks), r = __popc(ab & lt);
    if (asks) {
      ask[r] = make_uint2((uint32_t)(uintptr_t)sp, (uint32_t)((uintptr_t)sp >> 32));
      want[r] = a;
      from[r] = incl - sl;
    }
    __syncwarp();
    const uint32_t my_start = lane < (uint32_t)__popc(ab) ? from[lane] : 0xFFFFFFFFu;
    #pragma unroll 1
    for (uint32_t base = 0; base < total; base += 32) {
      const uint32_t before = __popc(__ballot_sync(FULL, my_start <= base));  // completions that begin up to here
      const uint32_t starts = __reduce_or_sync(FULL, my_start > base && my_start - base < 32u ? 1u << (my_start - base) : 0u);
      const uint32_t q = before - 1u + __popc(starts & (0xFFFFFFFFu >> (31u - lane)));
      bool match = false;
      uint32_t wi = 0;
      if (base + lane < total) {
        const uint2 p = ask[q];
        const uint32_t* items = reinterpret_cast<const uint32_t*>((uintptr_t)p.x | ((uintptr_t)p.y << 32));
        wi = items[base + lane - from[q]];
        const uint32_t winf = G.info[wi & 0xFFFFu];
        match = (winf >> INFO_KIND_SHIFT) == KIND_NT && (winf & INFO_ARG_MASK) == want[q];
      }
      if (__any_sync(FULL, match)) add(match, wi + 1u);
    }
    head = min(head + 32u, until);  // (items added by this wave begin at `until`)
  }
  __syncwarp();
  #pragma unroll 1
  for (uint32_t i = lane; i < set_words; i += 32) in_set[i] = EMPTY_SLOT;
  __syncwarp();
  return n <= s.w.cur_cap ? n : GEN_FULL;
}

// All bytes of one token.  Returns 1 (dst holds the new chart), 0 (some byte cannot follow: dst
// is garbage), -1 (a capacity limit was hit) or -2 (the arena for the token's sets is too small:
// the caller may retry with a larger one).  src and dst must not overlap.  `arena` (arena_cap
// items, a power of two if the last set is to be sorted in place) holds the token's sets.  Lane l brings the token's byte l.  s.out says
// where the new chart is: at dst, or in shared memory.
//
// With `forced_out` set, the bytes are not given but found: as long as the text so far is not a sentence and
// exactly one byte can follow, that byte is taken (and written to forced_out); `len` is then the longest run
// looked for, nothing is compacted or written to dst, and the return value is the length of the run.
__device__ __forceinline__ int token_steps(const GrammarDev& G, AdvScratch& s, const uint32_t* src, uint32_t own_byte, uint32_t len,
                                           uint32_t* dst, uint32_t dst_cap, uint32_t* arena, uint32_t arena_cap, uint8_t* forced_out) {
  const uint32_t lane = lane_id();
  const uint32_t m = src[CH_SETS];
  const uint32_t n_items = src[CH_ITEMS];
  if (m == 0 || m + len + MAX_TOKEN_BYTES + 4 > ADV_MAX_SETS || n_items > ADV_MAX_ITEMS || len > MAX_TOKEN_BYTES)
    return forced_out ? 0 : -1;
  static_assert(MAX_TOKEN_BYTES <= 32, "a token's bytes sit one to a lane");
  uint32_t* lvl_off = s.sets + ADV_MAX_SETS - (MAX_TOKEN_BYTES + 2);  // the tail of `sets` is free until Compact ends
  TokenView view{src + CH_HDR, src + CH_HDR + m + 1, m, arena, lvl_off};
  const uint32_t* soff = view.soff;
  const uint32_t* sitems = view.sitems;
  if (lane == 0) lvl_off[0] = 0, lvl_off[1] = 0;
  __syncwarp();
  // ---- per byte: Scan, Complete, Predict; the new set is appended to the arena
  uint32_t top = 0;
  bool accepting = forced_out != nullptr && (src[CH_FLAGS] & CHART_ACCEPTING) != 0u;
  const uint32_t* prev = sitems + soff[m - 1];
  uint32_t prev_len = soff[m] - soff[m - 1];
  #pragma unroll 1
  for (uint32_t L = 1; L <= len; ++L) {
    if (top + 64 > arena_cap) return forced_out ? (int)(L - 1) : -2;
    uint32_t byte;
    if (forced_out) {  // is the next byte forced?
      if (accepting) return (int)(L - 1);  // the text may end here
      scannable_bytes(G, prev, prev_len, s.pairs);
      uint32_t wd = lane < 8 ? s.pairs[lane] : 0u;
      uint32_t cnt = __popc(wd);
      #pragma unroll 1
      for (int dd = 16; dd > 0; dd >>= 1) cnt += __shfl_xor_sync(FULL, cnt, dd);
      if (cnt != 1u) return (int)(L - 1);
      const uint32_t has = __ballot_sync(FULL, wd != 0u);
      const int src_lane = __ffs(has) - 1;
      byte = (uint32_t)src_lane * 32u + (uint32_t)(__ffs(__shfl_sync(FULL, wd, src_lane)) - 1);
      __syncwarp();
    } else {
      byte = __shfl_sync(FULL, own_byte, L - 1);
    }
    s.w.cur = arena + top;
    s.w.cur_cap = arena_cap - top;
    __syncwarp();
    if (lane < W_CTRS) s.w.ctr[lane] = 0u;
    __syncwarp();
    if (prev_len == 1u && !forced_out) {
      // One item inside a literal or an automaton that moves on and completes nothing: the new set is that one item, and
      // there is nothing to predict (inside strings and names: half of the steps and more).  Nothing begins in the sets on the
      // way, so nobody asks for them: they are left empty.
      uint32_t it = prev[0], moves = 0;
#pragma unroll 1
      for (;;) {
        const uint32_t inf = G.info[it & 0xFFFFu], kind = inf >> INFO_KIND_SHIFT;
        uint32_t to = 0;
        if (kind == KIND_DFA) {
          const uint32_t t = G.dfa_trans[(size_t)(inf & INFO_ARG_MASK) * G.n_eq + G.eq_of_byte[byte]];
          if (t != 0xFFFFu && (t & 0xC000u) == 0x4000u) to = (it & 0xFFFF0000u) | (G.dfa_first + (t & 0x3FFFu));
        } else if (kind == KIND_TERM && class_has(G, inf & INFO_ARG_MASK, byte)) {
          const uint32_t next = G.info[(it & 0xFFFFu) + 1u] >> INFO_KIND_SHIFT;
          if (next == KIND_TERM || next == KIND_DFA) to = it + 1u;
        }
        if (!to) break;
        it = to, ++moves;
        if (lane == 0) lvl_off[L + 1] = top;
        if (++L > len) break;
        byte = __shfl_sync(FULL, own_byte, L - 1);
      }
      if (moves) {
        prev = arena + top;
        __syncwarp();
        if (lane == 0) arena[top] = it, lvl_off[L] = top + 1u;
        ++top;
        accepting = false;
        __syncwarp();
        if (L > len) break;
        s.w.cur = arena + top;
        s.w.cur_cap = arena_cap - top;
        if (top + 64 > arena_cap) return -2;
      }
    }
    const uint32_t index = m - 1 + L;
    uint32_t n;
    // sets of up to 32 scanned and completed items (nearly all) are built in lanes; what comes from a set of more than 32 items
    // seldom is one (trying it all the same cost an advance of 32 ambiguous rows 90 us, not trying 80) ...
    uint32_t mine;
    const uint32_t ns = (prev_len <= (gen_fits(G, index) ? 32u : 96u)) ? small_scan_complete(G, s.w, view, prev, prev_len, byte, index,
                                                                                                   [](uint32_t it) { return it; }, mine, accepting)
                                                                       : SMALL_OVERFLOW;
    if (ns == 0) return forced_out ? (int)(L - 1) : 0;
    if (ns != SMALL_OVERFLOW) {
      n = small_drop_completed(G, s.w, ns, mine);
    } else {
      if (gen_fits(G, index)) {  // ... larger ones with a bit for every item there can be
        n = gen_scan_complete(G, s, view, prev, prev_len, byte, index);
        if (n == GEN_FULL) {
          clear_nt(G, s.w);
          return forced_out ? (int)(L - 1) : -2;
        }
        if (n == 0) return forced_out ? (int)(L - 1) : 0;
      } else {  // ... and where that is too many, with the uniqueness hash
        n = scan_into_cur(G, s.w, prev, prev_len, byte);
        if (s.w.ctr[W_OVERFLOW]) {
          hset_clear_all(s.w.hset, s.w.hset_mask);
          return forced_out ? (int)(L - 1) : -2;
        }
        if (n == 0) return forced_out ? (int)(L - 1) : 0;
        complete_fixpoint(G, s.w, view, index, 0u);
        n = min(s.w.ctr[W_NCUR], s.w.cur_cap);
        if (s.w.ctr[W_OVERFLOW]) {
          hset_clear_all(s.w.hset, s.w.hset_mask);
          clear_nt(G, s.w);
          return forced_out ? (int)(L - 1) : -2;
        }
        hset_clear_items(s.w, n);
      }
      accepting = s.w.ctr[W_ACCEPT] != 0u;
      n = drop_completed(G, s.w, n);
    }
    n = predict_set<true>(G, s.w, n, index);
    if (n == PREDICT_FULL) return forced_out ? (int)(L - 1) : -2;
    prev = arena + top;
    prev_len = n;
    top += n;
    if (lane == 0) lvl_off[L + 1] = top;
    if (forced_out && lane == 0) forced_out[L - 1] = (uint8_t)byte;  // (the step went through: the byte counts)
    __syncwarp();
  }
  if (forced_out) return (int)len;
  // ---- Compact once: which items of the earlier sets can a later Complete still read?
  const uint32_t last = m - 1 + len;           // index of the last set
  const uint32_t last_at = lvl_off[len];       // its first item in the arena
  const uint32_t n_last = top - last_at;
  const uint32_t n_bits = n_items + last_at;   // source items, then the token's earlier sets
  if (n_bits > ADV_MAX_ITEMS) return -1;
  #pragma unroll 1
  for (uint32_t i = lane; i < (n_bits + 31) / 32; i += 32) s.live[i] = 0u;
  __syncwarp();
  // ---- the needs, "somebody may complete a non-terminal begun in this set".  An item begun in a set lies in that set or
  // in a later one, so one pass over the sets from the last to the first finds them all: per set a bit for every non-terminal.
  // An item whose non-terminal pulls an asked one in by prediction is waited for, too, which settles the items begun in the set itself.  One
  // pass over a set's items per set: with a list of (set, non-terminal) pairs served one after the other Compact
  // took 31,000 cycles for a JSON chart of 12 sets and 280,000 for an ambiguous one of 60, now 8,500 and 90,000.
  const uint32_t M = last;  // earlier sets: 0..last-1
  if (M * G.Nw <= ADV_HSET) {
    uint32_t* need = s.w.hset;  // [M][Nw]
    const uint32_t Nw = G.Nw;
    #pragma unroll 1
    for (uint32_t i = lane; i < M * Nw; i += 32) need[i] = 0u;
    #pragma unroll 1
    for (uint32_t k = lane; k < M; k += 32) s.sets[k] = 0u;
    __syncwarp();
    // Where no item of the source chart's sets after set o begins before o, everything before o is held by o's items alone, and as the
    // source chart is pruned, all of it is needed if they all are: the way down a deep nesting ends at the first such set.
    uint32_t earliest = 0xFFFFFFFFu, looked_at = n_items;  // (each lane: over some of the items from looked_at on)
    const bool narrow = M <= 32u;        // (then the sets that have been asked are a word)
    uint32_t first_asked = 0xFFFFFFFFu;  // (each lane: the earliest set it has asked, or all of them)
    uint32_t asked_sets = 0u;
    if (narrow) first_asked = 0u;
    auto ask = [&](uint32_t o, uint32_t A) {
      first_asked = narrow ? first_asked | 1u << o : min(first_asked, o);
      atomicOr(&need[o * Nw + (A >> 5)], 1u << (A & 31u));
    };
    #pragma unroll 1
    for (uint32_t i = lane; i < n_last; i += 32) {
      const uint32_t it = arena[last_at + i];
      if ((it >> 16) < last) ask(it >> 16, G.lhs[it & 0xFFFFu]);
    }
    #pragma unroll 1
    for (uint32_t end = M; end;) {  // sets 0 .. end-1 are left: the last of them that is asked for
      __syncwarp();
      uint32_t o;
      bool sole;  // nothing before it has been asked yet
      if (narrow) {
        asked_sets |= __reduce_or_sync(FULL, first_asked);
        const uint32_t left = asked_sets & (0xFFFFFFFFu >> (32u - end));
        if (left == 0u) break;
        o = 31u - __clz(left);
        sole = left == 1u << o;
      } else {
        const uint32_t k = end - 1u - lane;  // (wraps around for lanes beyond set 0)
        bool asked = false;
        if (k < end)
#pragma unroll 1
          for (uint32_t w = 0; w < Nw; ++w) asked = asked || need[k * Nw + w] != 0u;
        const uint32_t bal = __ballot_sync(FULL, asked);
        if (bal == 0u) {
          end -= min(end, 32u);
          continue;
        }
        o = end - (uint32_t)__ffs(bal);
        sole = __reduce_min_sync(FULL, first_asked) == o;
      }
      end = o;
      const uint32_t* sp;
      uint32_t sl;
      view(o, sp, sl);
      const uint32_t first_bit = view.bit_base(o, n_items);
      uint32_t live = 0;
      #pragma unroll 1
      for (uint32_t base = 0; base < sl; base += 32) {
        const uint32_t it = base + lane < sl ? sp[base + lane] : 0u;
        const uint32_t inf = G.info[it & 0xFFFFu], A = inf & INFO_ARG_MASK;
        bool keep = false;
        if (base + lane < sl && (inf >> INFO_KIND_SHIFT) == KIND_NT)
          #pragma unroll 1
          for (uint32_t w = 0; w < Nw; ++w) keep = keep || (need[o * Nw + w] & G.nt_closure[A * Nw + w]);
        const uint32_t kb = __ballot_sync(FULL, keep);
        if (kb == 0u) continue;
        live += __popc(kb);
        if (keep && (it >> 16) != o) ask(it >> 16, G.lhs[it & 0xFFFFu]);
        const uint32_t at = first_bit + base, sh = at & 31u;
        if (lane == 0) s.live[at >> 5] |= kb << sh;
        if (lane == 1 && sh && (kb >> (32u - sh))) s.live[(at >> 5) + 1u] |= kb >> (32u - sh);
        __syncwarp();
      }
      if (lane == 0) s.sets[o] = live;
      bool rest = false;
      if (sole && live == sl && o < m) {
        const uint32_t from = soff[o + 1u];
#pragma unroll 1
        for (uint32_t i = from + lane; i < looked_at; i += 32) earliest = min(earliest, sitems[i] >> 16);
        looked_at = from;
        rest = __reduce_min_sync(FULL, earliest) >= o;
      }
      if (rest) {  // it stays as it is
        const uint32_t bits = soff[o];
        __syncwarp();
        #pragma unroll 1
        for (uint32_t k = lane; k < o; k += 32) s.sets[k] = soff[k + 1] - soff[k];
        #pragma unroll 1
        for (uint32_t i = lane; i < (bits + 31u) / 32u; i += 32) s.live[i] |= (i + 1u) * 32u <= bits ? FULL : (1u << (bits & 31u)) - 1u;
        break;
      }
    }
    __syncwarp();
    #pragma unroll 1
    for (uint32_t i = lane; i < M * Nw; i += 32) need[i] = EMPTY_SLOT;
    __syncwarp();
  } else {
    #pragma unroll 1
    for (uint32_t i = lane; i < n_last; i += 32) {
      uint32_t it = arena[last_at + i];
      if ((it >> 16) < last) push_need(s, it >> 16, G.lhs[it & 0xFFFFu]);
    }
    // needs are served a wave at a time: a need whose set is short is served by its own lane, the
    // needs of long sets (alternations of many literals predicted at once) by the whole warp in turn
    constexpr uint32_t NEED_SHORT = 8;
    #pragma unroll 1
    for (uint32_t head = 0;;) {
      __syncwarp();
      const uint32_t np = min(s.w.ctr[W_NPAIRS], ADV_PAIRS);
      __syncwarp();
      if (head >= np) break;
      const uint32_t mine = head + lane;
      uint32_t o = 0, A = 0, sl = 0, base = 0;
      const uint32_t* sp = nullptr;
      if (mine < np) {
        const uint32_t key = s.pairs[mine];
        o = key >> 16, A = key & 0xFFFFu;
        view(o, sp, sl);
        base = view.bit_base(o, n_items);
      }
      auto serve = [&](const uint32_t* set, uint32_t k, uint32_t bit_base, uint32_t want) {
        const uint32_t wi = set[k];
        const uint32_t inf = G.info[wi & 0xFFFFu];
        if ((inf >> INFO_KIND_SHIFT) == KIND_NT && (inf & INFO_ARG_MASK) == want) {
          const uint32_t pos = bit_base + k;
          const uint32_t bit = 1u << (pos & 31u);
          const uint32_t old = atomicOr(&s.live[pos >> 5], bit);
          if (!(old & bit)) push_need(s, wi >> 16, G.lhs[wi & 0xFFFFu]);
        }
      };
      if (sl <= NEED_SHORT)
        #pragma unroll 1
        for (uint32_t k = 0; k < sl; ++k) serve(sp, k, base, A);
      uint32_t longs = __ballot_sync(FULL, sl > NEED_SHORT);
      #pragma unroll 1
      while (longs) {
        const int src = __ffs(longs) - 1;
        longs &= longs - 1;
        const uint32_t so = __shfl_sync(FULL, o, src), sA = __shfl_sync(FULL, A, src);
        const uint32_t* lp;
        uint32_t ll;
        view(so, lp, ll);
        const uint32_t lbase = view.bit_base(so, n_items);
        #pragma unroll 1
        for (uint32_t k = lane; k < ll; k += 32) serve(lp, k, lbase, sA);
      }
      head = min(head + 32u, np);
    }
    const uint32_t n_pairs = min(s.w.ctr[W_NPAIRS], ADV_PAIRS);
    __syncwarp();
    if (n_pairs * 8u > s.w.hset_mask) {
      hset_clear_all(s.w.hset, s.w.hset_mask);  // the hash held (set, non-terminal) pairs
    } else {
      #pragma unroll 1
      for (uint32_t i = lane; i < n_pairs; i += 32) {
        const uint32_t key = s.pairs[i];
        uint32_t hh = mix32(key) & s.w.hset_mask;
        #pragma unroll 1
        for (uint32_t probe = 0; probe <= s.w.hset_mask; ++probe) {
          if (s.w.hset[hh] == key) {
            s.w.hset[hh] = EMPTY_SLOT;
            break;
          }
          hh = (hh + 1) & s.w.hset_mask;
        }
      }
      __syncwarp();
    }
    if (s.w.ctr[W_OVERFLOW]) {
      hset_clear_all(s.w.hset, s.w.hset_mask);
      clear_nt(G, s.w);
      return -1;
    }
    // ---- live items per earlier set, new set numbers, new offsets
    #pragma unroll 1
    for (uint32_t k = lane; k < M; k += 32) {
      const uint32_t* sp;
      uint32_t sl;
      view(k, sp, sl);
      const uint32_t base = view.bit_base(k, n_items);
      uint32_t c = 0;
      #pragma unroll 1
      for (uint32_t i = 0; i < sl; ++i) c += (s.live[(base + i) >> 5] >> ((base + i) & 31u)) & 1u;
      s.sets[k] = c;
    }
    __syncwarp();
  }
  if (CH_HDR + (M + 2u) + n_bits + n_last <= ADV_OUT && n_bits <= 16384u) dst = s.live + ADV_MAX_ITEMS / 64u;
  static_assert(ADV_MAX_ITEMS / 64u >= ADV_OUT, "the upper half of the bitmap has room for a small chart");
  s.out = dst;
  HashAcc h;
  uint32_t m_new = 0, kept = 0;
  #pragma unroll 1
  for (uint32_t base = 0; base < M; base += 32) {
    uint32_t k = base + lane;
    uint32_t c = (k < M) ? s.sets[k] : 0u;
    uint32_t keep = __ballot_sync(FULL, c > 0);
    uint32_t my_new = m_new + __popc(keep & ((1u << lane) - 1u));
    uint32_t incl = c;  // inclusive prefix sum of the counts within the wave
    #pragma unroll 1
    for (int d = 1; d < 32; d <<= 1) {
      uint32_t t = __shfl_up_sync(FULL, incl, d);
      if ((int)lane >= d) incl += t;
    }
    __syncwarp();
    if (k < M) {
      if (c > 0) {
        if (CH_HDR + my_new < dst_cap) put(dst, h, CH_HDR + my_new, kept + incl - c);
        s.sets[k] = my_new;
      } else {
        s.sets[k] = 0xffffffffu;
      }
    }
    kept += __shfl_sync(FULL, incl, 31);
    m_new += __popc(keep);
  }
  __syncwarp();
  if (CH_HDR + (m_new + 2) + kept + n_last + 64 > dst_cap) return -1;
  // ---- copy the live items (source chart first, then the token's earlier sets), origins renumbered
  const uint32_t items_at = CH_HDR + (m_new + 2);
  uint32_t bad = 0;
  uint32_t out = 0;
  #pragma unroll 1
  for (uint32_t base = 0; base < n_bits; base += 32) {
    uint32_t i = base + lane;
    bool lv = (i < n_bits) && ((s.live[i >> 5] >> (i & 31u)) & 1u);
    uint32_t bal = __ballot_sync(FULL, lv);
    if (lv) {
      uint32_t it = (i < n_items) ? sitems[i] : arena[i - n_items];
      uint32_t no = s.sets[it >> 16];
      if (no == 0xffffffffu) bad = 1;
      const uint32_t at = items_at + out + __popc(bal & ((1u << lane) - 1u)), v = (no << 16) | (it & 0xFFFFu);
      if (i < n_items) put(dst, h, at, v);  // the source chart's sets are sorted and stay so
      else dst[at] = v;                     // the token's own sets are in the order they were built: sorted below
    }
    out += __popc(bal);
  }
  // ---- the kept items of the token's earlier sets, ascending like every other set: the chart is
  // the cache key, and the same bytes fed as other tokens must give the same words
  __syncwarp();
  #pragma unroll 1
  for (uint32_t L = 1; L < len; ++L) {
    const uint32_t nw = s.sets[m - 1 + L];
    if (nw == 0xffffffffu) continue;  // (uniform)
    const uint32_t a = dst[CH_HDR + nw], b = (nw + 1 < m_new) ? dst[CH_HDR + nw + 1] : kept;
    uint32_t* set = dst + items_at + a;
    const uint32_t ns = b - a;
    if (ns <= 1) {
    } else if (ns <= 32) {
      sort_items(set, ns, 32);
    } else {  // rare: by rank, through the part of the arena whose sets have been copied out by now
      #pragma unroll 1
      for (uint32_t i = lane; i < ns; i += 32) arena[i] = set[i];
      __syncwarp();
      #pragma unroll 1
      for (uint32_t i = lane; i < ns; i += 32) {
        const uint32_t x = arena[i];
        uint32_t rank = 0;
        #pragma unroll 1
        for (uint32_t k = 0; k < ns; ++k) rank += arena[k] < x ? 1u : 0u;
        set[rank] = x;  // (the items of a set are distinct)
      }
      __syncwarp();
    }
    #pragma unroll 1
    for (uint32_t i = lane; i < ns; i += 32) h.add(items_at + a + i, set[i]);
  }
  // ---- the last set: renumber origins (its own index becomes m_new), move it to the front of the
  // arena region it occupies so that it can be sorted in place
  #pragma unroll 1
  for (uint32_t i = lane; i < n_last; i += 32) {
    uint32_t it = arena[last_at + i];
    uint32_t o = it >> 16;
    uint32_t no = (o == last) ? m_new : s.sets[o];
    if (no == 0xffffffffu) bad = 1;
    arena[last_at + i] = (no << 16) | (it & 0xFFFFu);
  }
  bad = __any_sync(FULL, bad);
  __syncwarp();
  if (bad) return -1;
  uint32_t P = 32;
  #pragma unroll 1
  while (P < n_last) P <<= 1;
  if (last_at + P > arena_cap) return -2;  // the sort pads the set to a power of two
  s.w.cur = arena + last_at;
  return finish_chart(s, dst, dst_cap, m_new, kept, n_last, accepting, h);
}

// A chart that is not too large comes into shared memory.  Its first words are read with its header: nearly all charts are no longer, and
// the arena goes on so far behind its last chart.
struct ChartAhead {
  uint32_t w[ADV_AHEAD / 32];
};
__device__ __forceinline__ ChartAhead read_ahead(const uint32_t* src) {
  ChartAhead a;
#pragma unroll
  for (uint32_t k = 0; k < ADV_AHEAD / 32; ++k) a.w[k] = src[k * 32u + lane_id()];
  return a;
}
__device__ __forceinline__ bool stage_chart(const AdvScratch& s, const uint32_t* src, const ChartAhead& a) {
  const uint32_t lane = lane_id();
  const uint32_t words = __shfl_sync(FULL, a.w[0], CH_WORDS);
  if (words > ADV_STAGE) return false;
#pragma unroll
  for (uint32_t k = 0; k < ADV_AHEAD / 32; ++k) s.stage[k * 32u + lane] = a.w[k];
#pragma unroll 1
  for (uint32_t i = ADV_AHEAD + lane; i < words; i += 32) s.stage[i] = src[i];
  __syncwarp();
  return true;
}

// The same steps, wherever the tables, the chart and the arena are.  (Where all of them are in shared memory the steps are
// compiled into the kernel, with 32-bit addresses throughout: a step is a chain of some hundred instructions of one warp.)
__device__ __noinline__ int token_steps_anywhere(const GrammarDev& G, AdvScratch& s, const uint32_t* src, uint32_t own_byte, uint32_t len,
                                                 uint32_t* dst, uint32_t dst_cap, uint32_t* arena, uint32_t arena_cap, uint8_t* forced_out) {
  return token_steps(G, s, src, own_byte, len, dst, dst_cap, arena, arena_cap, forced_out);
}
__device__ __forceinline__ int token_step(const GrammarDev& G, AdvScratch& s, const uint32_t* src, uint32_t own_byte, uint32_t len,
                                          uint32_t* dst, uint32_t dst_cap, uint32_t* arena, uint32_t arena_cap, uint8_t* forced_out = nullptr) {
  const GrammarDev g = G;  // (copies: what a call takes by reference is kept in memory)
  AdvScratch t = s;
  const int r = token_steps_anywhere(g, t, src, own_byte, len, dst, dst_cap, arena, arena_cap, forced_out);
  s.out = t.out;
  return r;
}

}  // namespace fmt
