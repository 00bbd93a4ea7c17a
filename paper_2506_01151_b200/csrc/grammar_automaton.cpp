// The grammar automaton: what a token's bytes do to ONE unfinished Earley item, worked out at compile time.
//
// Earley's steps are linear in the kernel of a set (its scanned and completed items): the sets reached from a kernel
// by some bytes are the unions of what is reached from its items taken one by one.  From one item (d, o) - dotted rule d,
// begun in set o - everything that happens inside a token depends on d alone, except where the rule of d is completed
// and o has to be asked who waited for it.  So the sets reached from {(d, here)} along byte strings, with the origin o left
// open, can be hash-consed and their transitions tabulated once for a grammar and a vocabulary (Section 4.3 of the paper
// keeps a context-independent part of the masks in the same spirit).
//
// Which transitions are needed follows from the vocabulary: the trie is walked once with the codes of all items that a
// kernel can hold, and where a rule of non-terminal A ends inside a token the walk goes on, from that node, with every item that
// completing A can yield in any chart of the grammar.
//
// What the fill gets (automaton_fill.cu) is no trie any more.  A START is an item at a trie node: an item of a chart's kernel at the root,
// or one that completing a rule inside a token yields, at the node where the rule ends.  Its TOKENS are those below the node that end before
// the item's own rule has: they are valid whatever the chart holds.  Where the rule ends with bytes still to come, the chart is
// asked, and for every item that it can answer there is an EDGE to the start of that item at that node.  So a fill follows edges, one
// for each rule that ends inside a token, and not the trie byte by byte.
#include <algorithm>
#include <array>
#include <cstring>
#include <unordered_map>
#include <utility>

#include "host_tables.h"

namespace fmt {
namespace {

using u32 = uint32_t;
using u64 = uint64_t;

// limits; a grammar beyond them has no automaton and its fills run the Earley steps themselves
constexpr u32 GA_MAX_SETS = 1u << 18;
constexpr u64 GA_MAX_TRANS = 32u << 20;   // table entries (4 bytes each)
// Look-ups of the walk over the trie, items scanned and every eighth comparison for a new transition: a quarter of a second at most (10 to
// 15 ns each: HTML with 90 tags, 44 million 0.69 s; JSON, SQL and JSON schemas over 128 K tokens have 0.5 to 4 million, 0.04 to 0.2 s).
constexpr u64 GA_MAX_WORK = 16u << 20;
// The same for the starts, every eighth token of theirs and GA_LINK_WORK for each edge, which takes as long as that: three quarters of a
// second at most.  Those of JSON, SQL, JSON schemas and tagged unions over 128 K tokens take 0.3 to 1.6 times as many look-ups as that
// walk and have up to 200,000 edges; words of letters whose every byte may end a word, 12,000 of 32 bytes, have 6.6 million and took
// 1.65 s while only look-ups counted.
constexpr u64 GA_MAX_START_WORK = 48u << 20;
constexpr u64 GA_LINK_WORK = 16;
constexpr size_t GA_MAX_WORDS = 64u << 20;  // of masks, tokens and edges
constexpr size_t GA_MASK_TOKENS = 1024;   // a kernel's item from which so many tokens follow has a mask in the place of a list
constexpr size_t GA_LONG_LIST = 64;       // edges of a start from which on it has one for each item and the others behind it
constexpr size_t GA_MAX_ITEMS = 1024;     // items of one set, predicted ones included: alternations of thousands of literals
                                          // would be scanned again for every set that predicts them

// Where the chart has to be asked at many places a fill by the automaton can be the slower one: each exit has an edge for every item that
// completing the rule yields, and a block follows those of its row where the whole grid sweeps the trie.  Two counts over the walk tell such
// grammars; they go without.  Fills of 4 and of 64 rows of 128,256 tokens (SQL 152,064, braces 60,000) on a B200, us, by edges / by the sweep:
//                                       4 rows           64 rows
//   JSON                              40 /    276       40 /    614
//   ambiguous JSON                   396 /  1,342      405 /  4,255
//   SQL                               45 /    326       45 /    966
//   text of one kind of character     44 /    111       45 /    303
//   two like texts                    45 /    203       46 /    466
//   a union of 20 variants            63 /    154       64 /    378     (starts a node 1.7)
//   braces                           286 /    163      290 /    375
//   those without, with both limits lifted:
//   a union of 40, of 60             110, 143 / 172    111, 147 / 404   (60: 5.1)
//   a union of 100, of 180           218, 367 / 181    221, 375 / 411, 435
//   HTML with 2 tags, with 20        455, 1,260 / 146  465, 1,275 / 397, 420  (exits at 0.75 of the nodes)
//   XML                           13,100 /  1,018   18,000 /  1,504     (0.75)
// HTML and XML are on the right side of the line, unions of a hundred variants gain in large batches and lose in small ones, and
// those of 40 and 60 would be faster by edges: the line was drawn for fills that walked the trie, and a higher one for them has not
// been looked for.  The texts of one kind have few nodes (GA_EXITS).
constexpr u32 GA_EXIT_SHARE = 4;          // no automaton if more than one in so many nodes has an exit
constexpr u32 GA_EXITS = 1024;            // (and more than so many nodes: a small trie is walked in no time)
constexpr u32 GA_STARTS = 2;              // nor if there are more starts than so many a node
constexpr u64 GA_STARTS_FREE = 64u << 10; // and so many

struct VecHash {
  size_t operator()(const std::vector<u64>& v) const {
    u64 h = 0x9E3779B97F4A7C15ull;
    for (u64 x : v) {
      h = (h ^ x) * 0xD6E8FEB86659FD93ull;
      h ^= h >> 32;
    }
    return (size_t)h;
  }
};

class Builder {
 public:
  explicit Builder(HostTables& h) : h_(h), n_eq_(h.n_eq) {
    for (int b = 255; b >= 0; --b) rep_[h.eq_of_byte[b]] = (uint8_t)b;
  }

  bool run() {
    roots();
    class_trie();
    follow();
    std::vector<u32> first;
    for (u32 d = 0; d < h_.D; ++d)
      if (root_[d] != GA_DEAD) first.push_back(root_[d]);
    dedupe(first, 0);
    arena_ = first;
    if (!too_big_) walk(0, 0, arena_.size());
    if (too_big_) return false;
    starts();
    return !too_big_;
  }

 private:
  struct Set {
    std::vector<u64> kernel;                  // origin << 32 | dotted rule; origin 0 = open, u + 1 = set u
    std::vector<u64> scan;                    // kernel and predicted items before a terminal or inside an automaton
    std::vector<std::pair<u32, u64>> wait;    // post-dot non-terminal -> the item with the dot moved over it
    u32 lhs = 0;                              // whose rule the open origin belongs to
    bool expanded = false;
  };

  HostTables& h_;
  const u32 n_eq_;
  std::vector<u32> root_;                     // [D] code of the kernel {(d, open)}
  // the vocabulary trie over byte classes, breadth first: [nodes][4] first child, children << 8 | byte class, the token (or where in tok_
  // they begin), tokens
  std::vector<u32> node_, tok_;
  uint8_t rep_[256];
  std::vector<Set> sets_;
  std::unordered_map<std::vector<u64>, u32, VecHash> ids_;
  std::vector<u32> trans_;
  std::unordered_map<u32, u32> accept_;
  std::vector<u64> cur_;
  std::vector<u32> arena_;
  std::vector<std::vector<u32>> follow_;      // per non-terminal: the items that completing it can yield,
  std::vector<std::vector<u32>> codes_;       // and their codes
  u64 work_ = 0, begun_ = 0, exit_nodes_ = 0;
  bool too_big_ = false;

  const u32* node(u32 n) const { return &node_[(size_t)n * 4]; }
  u32 kind(u32 d) const { return h_.info[d] >> INFO_KIND_SHIFT; }
  u32 arg(u32 d) const { return h_.info[d] & INFO_ARG_MASK; }

  u32 lhs_of(u32 code) const {
    if (!(code & GA_ITEM)) return sets_[code].lhs;
    const u32 org = (code >> 14) & 0xFFFFu;
    return org ? sets_[org - 1].lhs : h_.lhs[h_.dfa_first + (code & 0x3FFFu)];
  }

  // The code of the set with this kernel (ascending).  A kernel of one item inside an automaton is its own code.
  u32 intern(std::vector<u64>& k) {
    if (k.empty()) return GA_NONE;
    const u64 org = k[0] >> 32;
    if (k.size() == 1 && kind((u32)k[0]) == KIND_DFA && org < 0xFFFFu)
      return GA_ITEM | (u32)(org << 14) | arg((u32)k[0]);
    const auto it = ids_.find(k);
    if (it != ids_.end()) return it->second;
    const u32 id = (u32)sets_.size();
    if (id + 1 >= GA_MAX_SETS || (u64)(id + 1) * n_eq_ > GA_MAX_TRANS) {
      too_big_ = true;
      return GA_NONE;
    }
    ids_.emplace(k, id);
    sets_.emplace_back();
    sets_[id].kernel = k;
    sets_[id].lhs = org ? sets_[org - 1].lhs : h_.lhs[(u32)k[0]];
    trans_.resize((size_t)(id + 1) * n_eq_, GA_UNKNOWN);
    return id;
  }

  void expand(u32 s) {
    if (sets_[s].expanded) return;
    Set& set = sets_[s];
    set.expanded = true;
    std::vector<u32> nts(h_.Nw, 0u);
    auto put = [&](u64 it) {
      const u32 d = (u32)it;
      if (kind(d) == KIND_NT) set.wait.push_back({arg(d), it + 1});
      else if (kind(d) != KIND_END) set.scan.push_back(it);
    };
    for (u64 it : set.kernel) {
      put(it);
      if (kind((u32)it) == KIND_NT)
        for (u32 w = 0; w < h_.Nw; ++w) nts[w] |= h_.nt_closure[(size_t)arg((u32)it) * h_.Nw + w];
    }
    for (u32 w = 0; w < h_.Nw; ++w)
      for (u32 bits = nts[w]; bits; bits &= bits - 1) {
        const u32 z = w * 32 + (u32)__builtin_ctz(bits);
        for (u32 k = h_.direct_off[z]; k < h_.direct_off[z + 1]; ++k) put((u64)(s + 1) << 32 | h_.direct_items[k]);
      }
    std::sort(set.wait.begin(), set.wait.end());
    work_ += set.scan.size() + set.wait.size();
    if (set.scan.size() + set.wait.size() > GA_MAX_ITEMS) too_big_ = true;
  }

  void add(u64 it) {
    work_ += cur_.size() / 8u;
    for (u32 j = 0; j <= h_.skip[(u32)it]; ++j)
      if (std::find(cur_.begin(), cur_.end(), it + j) == cur_.end()) cur_.push_back(it + j);
  }

  // Complete (Section 3.2) over cur_, then the set's code; GA_EXIT when the open origin has to be asked.
  u32 complete() {
    if (cur_.empty()) return GA_DEAD;
    bool exits = false;
    std::vector<u64> k;
    for (size_t i = 0; i < cur_.size() && !too_big_; ++i) {
      const u64 it = cur_[i];
      if (kind((u32)it) != KIND_END) {
        k.push_back(it);
        continue;
      }
      const u32 org = (u32)(it >> 32);
      if (org == 0) {
        exits = true;
        continue;
      }
      expand(org - 1);
      const auto& w = sets_[org - 1].wait;
      for (auto lo = std::lower_bound(w.begin(), w.end(), std::make_pair(arg((u32)it), (u64)0)); lo != w.end() && lo->first == arg((u32)it); ++lo)
        add(lo->second);
    }
    std::sort(k.begin(), k.end());
    return intern(k) | (exits ? GA_EXIT : 0u);
  }

  u32 next(u32 code, u32 e) {
    ++work_;
    if (code & GA_ITEM) {
      const u32 org = (code >> 14) & 0xFFFFu, g = code & 0x3FFFu;
      const u32 t = h_.dfa_trans[(size_t)g * n_eq_ + e];
      if (t == 0xFFFFu || !(t & 0xC000u)) return GA_DEAD;
      if (!(t & 0x8000u)) return GA_ITEM | (org << 14) | (t & 0x3FFFu);
      if (org == 0) return GA_EXIT | ((t & 0x4000u) ? (GA_ITEM | (t & 0x3FFFu)) : GA_NONE);
      const u32 key = org << 16 | t;
      const auto it = accept_.find(key);
      if (it != accept_.end()) return it->second;
      cur_.clear();
      if (t & 0x4000u) cur_.push_back((u64)org << 32 | (h_.dfa_first + (t & 0x3FFFu)));
      cur_.push_back((u64)org << 32 | h_.dfa_done[t & 0x3FFFu]);
      const u32 r = complete();
      accept_.emplace(key, r);
      return r;
    }
    const size_t slot = (size_t)code * n_eq_ + e;
    if (trans_[slot] != GA_UNKNOWN) return trans_[slot];
    expand(code);
    cur_.clear();
    work_ += sets_[code].scan.size();
    const u32 b = rep_[e];
    for (u64 it : sets_[code].scan) {
      const u32 d = (u32)it, a = arg(d);
      if (kind(d) == KIND_TERM) {
        if ((h_.class_bits[(size_t)a * 8 + (b >> 5)] >> (b & 31)) & 1u) add(it + 1);
      } else {
        const u32 t = h_.dfa_trans[(size_t)a * n_eq_ + e];
        if (t == 0xFFFFu) continue;
        if (t & 0x4000u) add((it & ~0xFFFFFFFFull) | (h_.dfa_first + (t & 0x3FFFu)));
        if (t & 0x8000u) add((it & ~0xFFFFFFFFull) | h_.dfa_done[a]);
      }
    }
    const u32 r = complete();
    trans_[slot] = r;
    return r;
  }

  // root_[d]: the code of the kernel {(d, open)}, nullable non-terminals skipped, for every item a kernel can hold
  void roots() {
    root_.assign(h_.D, GA_DEAD);
    for (u32 d = 0; d < h_.D && !too_big_; ++d) {
      if (kind(d) == KIND_END) continue;
      if (kind(d) == KIND_DFA) {
        root_[d] = GA_ITEM | arg(d);
        continue;
      }
      const bool begins_rule = d != ITEM_START && (kind(d - 1) == KIND_END || d == 0);
      if (begins_rule) continue;
      std::vector<u64> k;
      for (u32 j = 0; j <= h_.skip[d]; ++j)
        if (kind(d + j) != KIND_END) k.push_back(d + j);
      root_[d] = intern(k);
    }
  }

  // follow_[A]: what completing A yields, whoever waits for it
  void follow() {
    const u32 N = h_.N;
    std::vector<std::vector<u32>> up(N);  // A -> non-terminals completed with it (its rule may end right after A)
    std::vector<std::vector<u32>> own(N);
    for (u32 d = 0; d < h_.D; ++d) {
      if (kind(d) != KIND_NT) continue;
      const u32 a = arg(d), skip = h_.skip[d + 1];
      if (kind(d + 1) != KIND_END) own[a].push_back(d + 1);
      if (kind(d + 1 + skip) == KIND_END) up[a].push_back(h_.lhs[d]);
    }
    follow_.assign(N, {}), codes_.assign(N, {});
    for (u32 a = 0; a < N; ++a) {
      std::vector<char> seen(N, 0);
      std::vector<u32> work{a};
      seen[a] = 1;
      while (!work.empty()) {
        const u32 x = work.back();
        work.pop_back();
        follow_[a].insert(follow_[a].end(), own[x].begin(), own[x].end());
        for (u32 y : up[x])
          if (!seen[y]) seen[y] = 1, work.push_back(y);
      }
      dedupe(follow_[a], 0);
      for (u32 d : follow_[a]) codes_[a].push_back(root_[d]);
      dedupe(codes_[a], 0);
    }
  }

  static void dedupe(std::vector<u32>& v, size_t from) {
    std::sort(v.begin() + from, v.end());
    v.erase(std::unique(v.begin() + from, v.end()), v.end());
  }

  // The vocabulary trie over byte classes: bytes that no terminal tells apart share a node.  Nodes are numbered breadth
  // first, so the children of a node are consecutive; the tokens that end at a node are listed together.
  void class_trie() {
    std::vector<u32> node(h_.T, 0);  // byte trie -> preliminary number
    size_t cap = 1024;
    while (cap < (size_t)h_.T * 2) cap <<= 1;
    std::vector<u64> key(cap, 0);
    std::vector<u32> val(cap), child(1, 0), sibling(1, 0);
    std::vector<uint8_t> eq(1, 0);
    for (u32 v = 1; v < h_.T; ++v) {
      const u32 p = node[h_.parent[v]], e = h_.eq_of_byte[h_.node_byte[v]];
      const u64 k = ((u64)p << 8 | e) + 1;
      size_t s = (size_t)(k * 0x9E3779B97F4A7C15ull >> 32) & (cap - 1);
      while (key[s] && key[s] != k) s = (s + 1) & (cap - 1);
      if (!key[s]) {
        key[s] = k, val[s] = (u32)eq.size();
        eq.push_back((uint8_t)e), child.push_back(0), sibling.push_back(child[p]);
        child[p] = val[s];
      }
      node[v] = val[s];
    }
    const u32 n = (u32)eq.size();
    std::vector<u32> order(1, 0), number(n, 0);
    order.reserve(n);
    node_.assign((size_t)n * 4, 0u);
    for (u32 i = 0; i < (u32)order.size(); ++i) {
      u32* r = &node_[(size_t)i * 4];
      r[0] = (u32)order.size();
      u32 kids = 0;
      for (u32 c = child[order[i]]; c; c = sibling[c], ++kids) number[c] = (u32)order.size(), order.push_back(c);
      r[1] = kids << 8 | eq[order[i]];
    }
    std::vector<u32> count(n + 1, 0);  // tokens by node
    for (u32 v = 0; v < h_.T; ++v) count[number[node[v]] + 1] += h_.tok_off[v + 1] - h_.tok_off[v];
    for (u32 i = 0; i < n; ++i) count[i + 1] += count[i];
    tok_.assign(std::max<u32>(count[n], 1), 0);
    std::vector<u32> at(count.begin(), count.end() - 1);
    for (u32 v = 0; v < h_.T; ++v)
      for (u32 k = h_.tok_off[v]; k < h_.tok_off[v + 1]; ++k) tok_[at[number[node[v]]]++] = h_.tok_ids[k];
    for (u32 i = 0; i < n; ++i) {  // a single token is named in the node itself
      u32* r = &node_[(size_t)i * 4];
      r[3] = count[i + 1] - count[i];
      r[2] = r[3] == 1 ? tok_[count[i]] : count[i];
    }
  }

  // All children of trie node v with the codes arena_[lo, hi) at v.
  void walk(u32 v, size_t lo, size_t hi) {
    const u32 first = node(v)[0], end = first + (node(v)[1] >> 8);
    for (u32 c = first; c < end && !too_big_; ++c) {
      const size_t base = arena_.size();
      const u32 e = node(c)[1] & 0xFFu, kids = node(c)[1] >> 8;
      bool asks = false;
      for (size_t i = lo; i < hi && work_ <= GA_MAX_WORK; ++i) {
        const u32 code = arena_[i], r = next(code, e);
        if (r == GA_DEAD || kids == 0) continue;
        if ((r & ~GA_EXIT) != GA_NONE) arena_.push_back(r & ~GA_EXIT);
        if (r & GA_EXIT) {
          const auto& f = codes_[lhs_of(code)];
          arena_.insert(arena_.end(), f.begin(), f.end());
          asks = true, begun_ += f.size();
        }
      }
      if (asks) ++exit_nodes_;
      const u64 nodes = node_.size() / 4;
      if (exit_nodes_ > GA_EXITS && exit_nodes_ * GA_EXIT_SHARE > nodes) too_big_ = true;
      if (begun_ > GA_STARTS * nodes + GA_STARTS_FREE) too_big_ = true;
      if (work_ > GA_MAX_WORK) too_big_ = true;
      dedupe(arena_, base);
      if (arena_.size() > base) walk(c, base, arena_.size());
      arena_.resize(base);
    }
  }

  struct Start {
    u32 node, code;
    u32 tok = 0, n_tok = 0;    // in h_.ga_tok; the token itself if it is one
    u32 link = 0, n_link = 0;  // in links: the starts that it has edges to, if anything follows from them
    u32 edge = 0, n_edge = 0;  // in h_.ga_edge
  };

  // Is any child of node v reached from there?
  bool goes_on(u32 v, u32 code) {
    const u32 first = node(v)[0], end = first + (node(v)[1] >> 8);
    for (u32 c = first; c < end; ++c)
      if (next(code, node(c)[1] & 0xFFu) != GA_DEAD) return true;
    return false;
  }

  // The starts with their tokens and edges, from the kernels' items on, and the items' records.
  void starts() {
    work_ = 0;
    std::vector<Start> st;
    std::vector<std::pair<u32, u32>> links, walked;  // (item, start); (node, code)
    std::vector<u32> exits, toks, hash(1u << 12, 0u);  // hash: start + 1
    h_.ga_tok.clear(), h_.ga_edge.clear(), h_.ga_mask.clear();
    auto slot_of = [&](u32 v, u32 code) {
      size_t s = (size_t)((((u64)v << 32 | code) + 1) * 0x9E3779B97F4A7C15ull >> 32) & (hash.size() - 1);
      while (hash[s] && (st[hash[s] - 1].node != v || st[hash[s] - 1].code != code)) s = (s + 1) & (hash.size() - 1);
      return s;
    };
    auto start = [&](u32 v, u32 code) -> u32 {
      const size_t s = slot_of(v, code);
      if (hash[s]) return hash[s] - 1;
      st.push_back({v, code});
      hash[s] = (u32)st.size();
      if (st.size() * 2 > hash.size()) {
        hash.assign(hash.size() * 4, 0u);
        for (u32 i = 0; i < st.size(); ++i) hash[slot_of(st[i].node, st[i].code)] = i + 1;
      }
      return (u32)st.size() - 1;
    };
    std::vector<u32> root_start(h_.D, GA_DEAD), mask_of;
    for (u32 d = 0; d < h_.D; ++d)
      if (root_[d] != GA_DEAD) root_start[d] = start(0, root_[d]);
    const u32 roots = (u32)st.size();
    mask_of.assign(roots, GA_DEAD);
    for (u32 i = 0; i < (u32)st.size(); ++i) {
      if (work_ > GA_MAX_START_WORK || h_.ga_tok.size() + h_.ga_mask.size() + 4 * links.size() > GA_MAX_WORDS) too_big_ = true;
      if (too_big_) return;
      walked.assign(1, {st[i].node, st[i].code});
      exits.clear(), toks.clear();
      while (!walked.empty()) {
        const auto [v, code] = walked.back();
        walked.pop_back();
        const u32 first = node(v)[0], end = first + (node(v)[1] >> 8);
        for (u32 c = first; c < end; ++c) {
          const u32 r = next(code, node(c)[1] & 0xFFu);
          if (r == GA_DEAD) continue;
          if (node(c)[3] == 1) toks.push_back(node(c)[2]);
          else toks.insert(toks.end(), tok_.begin() + node(c)[2], tok_.begin() + node(c)[2] + node(c)[3]);
          if ((node(c)[1] >> 8) == 0u) continue;
          if ((r & ~GA_EXIT) != GA_NONE) walked.push_back({c, r & ~GA_EXIT});
          if (r & GA_EXIT) exits.push_back(c);
        }
      }
      st[i].n_tok = (u32)toks.size();
      work_ += toks.size() / 8u;
      if (i < roots && toks.size() >= GA_MASK_TOKENS) {
        const u32 words = (h_.Wm + 3u) & ~3u;
        mask_of[i] = (u32)(h_.ga_mask.size() / words);
        h_.ga_mask.resize(h_.ga_mask.size() + words, 0u);
        u32* m = &h_.ga_mask[(size_t)mask_of[i] * words];
        for (u32 t : toks) m[t >> 5] |= 1u << (t & 31);
      } else if (toks.size() == 1) {
        st[i].tok = toks[0];
      } else {
        st[i].tok = (u32)h_.ga_tok.size();
        h_.ga_tok.insert(h_.ga_tok.end(), toks.begin(), toks.end());
      }
      std::sort(exits.begin(), exits.end());
      const auto& f = follow_[lhs_of(st[i].code)];
      st[i].link = (u32)links.size();
      for (u32 c : exits)
        for (u32 d : f)
          if (root_[d] != GA_DEAD && goes_on(c, root_[d])) links.push_back({d, start(c, root_[d])}), work_ += GA_LINK_WORK;
      st[i].n_link = (u32)links.size() - st[i].link;
    }
    // edges: deeper nodes have larger numbers, so what a start's edges lead to is there before it
    std::vector<u32> order(st.size());
    for (u32 i = 0; i < (u32)st.size(); ++i) order[i] = i;
    std::sort(order.begin(), order.end(), [&](u32 a, u32 b) { return st[a].node > st[b].node; });
    std::vector<char> reached(h_.D, 0);
    using Edge = std::array<u32, 4>;
    std::vector<Edge> out;
    for (u32 i : order) {
      out.clear();
      for (u32 k = st[i].link; k < st[i].link + st[i].n_link; ++k) {
        const u32 d = links[k].first;
        const Start& to = st[links[k].second];
        if (to.n_tok == 0 && to.n_edge == 0) continue;
        reached[d] = 1;
        u32 n = std::min(to.n_tok, GA_EDGE_TOKENS);
        out.push_back({d << 16 | n, to.tok, to.edge, to.n_edge});
        for (u32 at = n; at < to.n_tok; at += n) {
          n = std::min(to.n_tok - at, GA_EDGE_TOKENS);
          out.push_back({d << 16 | n, n == 1 ? h_.ga_tok[to.tok + at] : to.tok + at, 0u, 0u});
        }
      }
      if (out.size() > GA_LONG_LIST) {  // those of one item together, behind an edge to all of them
        std::stable_sort(out.begin(), out.end(), [](const Edge& a, const Edge& b) { return a[0] >> 16 < b[0] >> 16; });
        std::vector<Edge> heads;
        for (size_t k = 0, e; k < out.size(); k = e) {
          for (e = k; e < out.size() && e - k < GA_EDGE_GROUP && out[e][0] >> 16 == out[k][0] >> 16;) ++e;
          if (e == k + 1) heads.push_back(out[k]);
          else heads.push_back({(out[k][0] & 0xFFFF0000u) | GA_GROUP, 0u, (u32)(h_.ga_edge.size() / 4), (u32)(e - k)});
          if (e > k + 1)
            for (size_t x = k; x < e; ++x) h_.ga_edge.insert(h_.ga_edge.end(), out[x].begin(), out[x].end());
        }
        out.swap(heads);
      }
      st[i].edge = (u32)(h_.ga_edge.size() / 4);
      for (const Edge& x : out) h_.ga_edge.insert(h_.ga_edge.end(), x.begin(), x.end());
      st[i].n_edge = (u32)(h_.ga_edge.size() / 4) - st[i].edge;
      if (h_.ga_tok.size() + h_.ga_mask.size() + h_.ga_edge.size() > GA_MAX_WORDS) {
        too_big_ = true;
        return;
      }
    }
    h_.ga_start.assign((size_t)h_.D * 4, 0u);
    h_.ga_item.assign((size_t)h_.D * 2, 0u);
    for (u32 d = 0; d < h_.D; ++d) {
      u32* r = &h_.ga_item[(size_t)d * 2];
      r[0] = h_.lhs[d] | 0xFFFF0000u;
      r[1] = 0xFFFFu;
      if (root_start[d] != GA_DEAD) {
        const Start& s = st[root_start[d]];
        const u32 mask = mask_of[root_start[d]];
        u32* q = &h_.ga_start[(size_t)d * 4];
        q[0] = mask != GA_DEAD ? mask : s.tok, q[1] = mask != GA_DEAD ? GA_MASK : s.n_tok;
        q[2] = s.edge, q[3] = s.n_edge;
        if (s.n_tok || s.n_edge) r[1] |= GA_ALIVE;
      }
      if (kind(d) != KIND_NT) continue;
      r[0] = h_.lhs[d] | arg(d) << 16;
      const u32 skip = h_.skip[d + 1];
      if (kind(d + 1 + skip) == KIND_END) r[1] = (r[1] & ~0xFFFFu) | h_.lhs[d];
      if (reached[d + 1]) r[1] |= GA_GOES_ON;
      if ((h_.info[d] & INFO_NULLABLE) && root_[d] != GA_DEAD) r[1] |= GA_SKIPS;
    }
  }
};

}  // namespace

void build_grammar_automaton(HostTables& h) {
  h.ga_on = false;
  if (h.D > 65535 || h.T >= (1u << 24)) return;
  Builder b(h);
  h.ga_on = b.run();
  if (!h.ga_on) h.ga_tok.clear(), h.ga_edge.clear(), h.ga_mask.clear();
}

}  // namespace fmt
