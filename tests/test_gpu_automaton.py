"""The fill by the grammar's automaton (fmt_compile tabulates what a token does to one Earley item) at the sizes where it
takes another path: rows per thread block, large vocabularies, many tokens at one trie node, long expansions, and grammars
without an automaton.  Masks are exact: they are compared with the oracle's bit by bit."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


def _run(text, start, vocab, prefixes, batch=None, check=None, **options):
    """Rows with these prefixes (taken in turn up to `batch`); the masks of the rows `check` against the oracle's."""
    import torch

    import paper_2506_01151_b200 as fmt

    eos = len(vocab) - 1
    g = fmt.Grammar(text, start, vocab, eos)
    batch = batch or len(prefixes)
    st = fmt.State(g, batch, cache=False, **options)
    longest = max(len(p) for p in prefixes)
    for i in range(longest):
        t = [prefixes[b % len(prefixes)][i] if i < len(prefixes[b % len(prefixes)]) else -1 for b in range(batch)]
        st.advance(torch.tensor(t, dtype=torch.int32, device="cuda"))
    mask = torch.full((batch, g.mask_words), -1, dtype=torch.int32, device="cuda")
    st.fill_mask(mask)
    got = mask.cpu().numpy().view(np.uint32)
    og, ov = oracle.Grammar(text, start), oracle.Vocab(vocab, eos)
    want = []
    for p in prefixes:
        s = oracle.Sequence_(og)
        assert s.advance(bytes(p)) or not p
        want.append(s.mask(ov))
    for b in range(batch) if check is None else check:
        assert np.array_equal(got[b], want[b % len(want)]), b
    stats = dict(st.stats(), counters=st.counters())
    assert stats["capacity_errors"] == 0 and stats["fills_aborted"] == 0
    return stats


JSON_PREFIXES = [list(x) for x in (b"", b'{"a": "x', b"[1, 2", b'{"k": tr', b"[[[", b'[{"a":[1.5e', b'{"a\\', b'["b", nul', b" ", b'{"q":{"r":[] ')]


@pytest.mark.parametrize("batch", [1, 2, 19, 37, 74, 75, 148, 297, 700])
def test_rows_of_every_share_of_the_grid(batch):
    """A block takes a row, or several rows in turn where there are more of them than blocks."""
    w = workloads.build(2, V=3000, batch=1, steps=1)
    _run(w.ebnf, w.start, w.vocab, JSON_PREFIXES, batch=batch)


@pytest.mark.parametrize("size", [258, 6144 * 32, 6144 * 32 + 1])
def test_many_tokens_at_a_node(size):
    """Thousands of tokens end at one node of the trie over byte classes (words no terminal tells apart), duplicates among them, in
    vocabularies up to 196,609 tokens."""
    rng = np.random.default_rng(3)
    letters = b"ghijkmopqvwxyzGHIJ"
    vocab = [bytes([b]) for b in range(256)]
    while len(vocab) < size - 1:
        n = int(rng.integers(1, 7))
        vocab.append(bytes(letters[i] for i in rng.integers(0, len(letters), n)) + (b'"' if rng.random() < 0.1 else b""))
    w = workloads.build(2, V=300, batch=1, steps=1)
    _run(w.ebnf, w.start, vocab + [b""], JSON_PREFIXES, batch=12)


@pytest.mark.parametrize("n", [1, 2, 31, 32])
def test_tokens_up_to_the_longest(n):
    vocab = [bytes([b]) for b in range(256)] + [b"["] * 2 + [b"[" * n, b"]" * n, (b"[]," * 11)[:n], b'"' + b"a" * (n - 1), b"a" * (n - 1) + b'"', b""]
    w = workloads.build(2, V=300, batch=1, steps=1)
    prefixes = [b"", b"[" * 5, b"[" * 40, b'["', b"[[1"]
    _run(w.ebnf, w.start, vocab, [list(p) for p in prefixes])


@pytest.mark.parametrize("n", [4, 60, 150])
def test_contexts_of_many_origins(n):
    """In an ambiguous grammar the rules that may end inside a token were begun in as many sets as there are letters; from some
    fifty on an expansion leaves shared memory."""
    text = 's ::= "<" e ">"\ne ::= e e | e "+" e | "(" e ")" | "a" | "b"'
    vocab = [bytes([b]) for b in range(256)] + [b"ab", b"a+b", b"a>", b"b)", b")+", b"ab+a(b)a>", b"+a>", b">a", b"(((a", b""]
    rng = np.random.default_rng(n)
    prefix = b"<" + bytes(b"ab"[i] for i in rng.integers(0, 2, n))
    _run(text, "s", vocab, [list(prefix), list(prefix + b"("), list(b"<(" + prefix[1:] + b")+")], chart_words=1 << 20)


def test_left_recursion_nullables_and_shared_prefixes():
    text = ('s ::= x\nx ::= x y | x z | ""\ny ::= w "a" w | "(" x ")"\nz ::= w "a" w | w "b" x "b"\nw ::= n n\nn ::= "_" | ""')
    vocab = [bytes([b]) for b in range(256)] + [b"aa", b"_a", b"a_a_", b"(a", b")a)", b"bab", b"__", b"_" * 5, b"((__a", b""]
    _run(text, "s", vocab, [list(p) for p in (b"", b"a", b"a_", b"(a_", b"bab", b"((b_", b"baaaab(a)")])


def _union(variants):
    """A union told apart by what follows a member that all variants begin with: as many items in the set, each followed by a string."""
    text = "s ::= " + " | ".join("t%d" % i for i in range(variants)) + "\n"
    text += "".join('t%d ::= "{\\"id\\":" str ",\\"k%d\\":" val "}"\n' % (i, i) for i in range(variants))
    return text + 'str ::= "\\"" [^"\\\\]* "\\""\nval ::= str | "[" val "]"\n'


@pytest.mark.parametrize("variants", [59, 60, 61, 100, 180])
@pytest.mark.parametrize("batch", [1, 4, 75, 300])
def test_more_wide_items_than_there_is_room_for(variants, batch):
    """A union's last set has an item of every variant, each with a mask of its own or a list of tokens: 59 to 180 of them are joined."""
    rng = np.random.default_rng(variants)
    some = np.frombuffer(b"0123456789kid[]{}:,", np.uint8)
    vocab = workloads.build(2, V=32000, batch=1, steps=1).vocab[:-1] + sorted({bytes(some[rng.integers(0, 19, 6)]) for _ in range(70000)}) + [b""]
    prefixes = [list(p) for p in (b'{"id":', b'{"id":"x', b'{"id":"x","k1', b'{"id":"y","k%d":[[' % (variants - 1))]
    s = _run(_union(variants), "s", vocab, prefixes, batch=batch, check=range(min(batch, 4)))
    assert batch == 1 or s["walk_transitions"] > 1000 * batch  # (look-ups: the rows were not swept)


@pytest.mark.parametrize("n", [511, 512, 513, 600, 1000])
@pytest.mark.parametrize("batch", [1, 5, 300])
def test_more_items_than_a_round_takes(n, batch):
    """After the byte that all literals of an alternation begin with, the last set has an item for each: their starts are taken 256 at a time."""
    rng = np.random.default_rng(n)
    names = _words(rng, n, 15, "k")
    text = 's ::= "[" v ("," v)* "]"\nv ::= "\\"" name "\\"" | "[" v "]"\nname ::= ' + " | ".join('"%s"' % x for x in names)
    vocab = [bytes([b]) for b in range(256)] + [x[1:9].encode() for x in names[::3]] + [(x[1:] + '","').encode() for x in names[1::3]] + [b"k" + x[1:3].encode() for x in names[2::3]] + [b""]
    prefixes = [list(p) for p in (b'["k', b'["' + names[5].encode() + b'","k', b'["' + names[1][:9].encode(), b'["')]
    s = _run(text, "s", vocab, prefixes, batch=batch, check=range(min(batch, 4)))
    assert s["walk_states"] < 200 * batch  # (the automaton's contexts, not Earley sets)


def _braces():
    """Text whose every byte ends a rule, at any depth of braces; each byte a class of its own.  Three quarters of the vocabulary
    are no text (a vocabulary in which rules end nearly everywhere is swept by Earley steps)."""
    kw = " | ".join('"\\x%02x!"' % b for b in range(33, 256) if chr(b) not in "{}")
    text = 'doc ::= piece*\npiece ::= char | "{" doc "}" | "}}" kw\nchar ::= [^{}\\x80-\\xff]\nkw ::= "!" | ' + kw + "\n"
    rng = np.random.default_rng(11)
    vocab, seen = [bytes([b]) for b in range(256)], set()
    while len(vocab) < 60000:
        n = 2 + int(rng.integers(0, 5))
        t = bytes(rng.integers(32, 126, n).astype(np.uint8)) if len(vocab) % 4 == 0 else bytes(rng.integers(128, 256, n).astype(np.uint8))
        if rng.random() < 0.2:
            t += b"}" * int(rng.integers(1, 4))
        if t not in seen:
            seen.add(t)
            vocab.append(t)
    return text, vocab + [b""]


@pytest.mark.parametrize("batch", [1, 64, 149, 300])
def test_text_whose_every_byte_ends_a_rule(batch):
    """Twenty thousand places at which the chart is asked: a row has its mask, however many rows share the grid."""
    text, vocab = _braces()
    s = _run(text, "doc", vocab, [list(p) for p in (b"x {a{b{c", b"{" * 30, b"a{}b{{", b"")], batch=batch, check=range(min(batch, 4)))
    assert s["walk_transitions"] > 20000 * batch  # (look-ups)


CNT_CROWDED, CNT_CUT = 198, 200  # (device_tables.h)


@pytest.mark.parametrize("batch", [1, 150, 300])
def test_rounds_that_push_more_than_the_stack_holds(batch):
    """A token of text for every two bytes it can begin with: each of 48,000 edges lists a further one, all at once, and a block's stack
    has 32,768 places.  Rounds put back what may not find room, and take one entry at a time while little is left."""
    kw = " | ".join('"\\x%02x!"' % b for b in range(256) if chr(b) not in "{}")
    text = 'doc ::= piece*\npiece ::= char | "{" doc "}" | "}}" kw\nchar ::= [^{}\\x00-\\x20]\nkw ::= "!" | ' + kw + "\n"
    rng = np.random.default_rng(12)
    chars = np.array([b for b in range(33, 256) if chr(b) not in "{}"], np.uint8)
    vocab = [bytes([b]) for b in range(256)]
    vocab += [bytes([a, b]) + bytes(chars[rng.integers(0, len(chars), 2 if rng.random() < 0.9 else 6)]) for a in chars for b in chars]
    vocab += sorted({bytes(rng.integers(0, 33, 7).astype(np.uint8)) for _ in range(80000)}) + [b""]  # (no text: see _braces)
    s = _run(text, "doc", vocab, [list(p) for p in (b"x{a{b", b"")], batch=batch, check=range(min(batch, 2)))
    assert s["rows_swept_again"] == 0 and s["walk_transitions"] > 80000 * batch
    assert s["counters"][CNT_CROWDED] > 500 * batch and s["counters"][CNT_CUT] >= batch / 2  # (the second row has no braces to end)


def _endings(n):
    """Brackets of n kinds, told apart after they close: every level of the text is completed to n kinds, n contexts a level.  Nearly
    all of the vocabulary are words that are no text (where the chart is asked at most of the trie, grammars have no automaton)."""
    kinds = [chr(97 + i) if i < 20 else "z%c%c" % (97 + i // 26, 97 + i % 26) for i in range(n)]
    text = "s ::= t\nt ::= \"x\" | " + " | ".join("t%d" % i for i in range(n)) + "\n"
    text += "".join('t%d ::= "(" t ")" "%s"\n' % (i, k) for i, k in enumerate(kinds))
    rng = np.random.default_rng(n)
    chains = [b"".join(b")" + kinds[int(i)].encode() for i in rng.integers(0, n if k % 2 else min(n, 20), 16))[:32] for k in range(60)]
    vocab = [bytes([b]) for b in range(256)] + [b"x" + c[:3 * k + 1] for k, c in enumerate(chains[:10])] + chains + [b")(", b"(("]
    letters = np.frombuffer(b"abcdefghijklmnopqrstuvwxyz", np.uint8)
    return text, vocab + sorted({bytes(letters[rng.integers(0, 26, 6)]) for _ in range(100000)}) + [b""]


@pytest.mark.parametrize("n, batch", [(20, 3), (100, 3), (340, 1), (340, 9), (340, 80)])
def test_rows_that_outgrow_the_storage_of_contexts(n, batch):
    """Contexts begin in shared memory (320) and go on in storage of the block's own (1,024).  A row that needs more is swept by
    Earley steps in the same call, by a block that has no row left; the rows beside it are not touched by that."""
    text, vocab = _endings(n)
    prefixes = [list(p) for p in (b"(" * 20, b"(" * 20 + b"x", b"(" * 20 + b"x)a", b"((x)a")]
    s = _run(text, "s", vocab, prefixes, batch=batch, check=range(min(batch, 4)))
    assert s["rows_swept_again"] <= batch and (n == 20 or s["rows_swept_again"] > 0)


@pytest.mark.parametrize("kinds, depth", [(2, 60), (3, 60), (4, 60), (5, 40), (23, 12), (24, 12), (25, 12), (20, 24), (64, 5), (65, 5), (130, 4)])
def test_contexts_asked_for_many_at_once(kinds, depth):
    """A closing bracket asks for a context of every kind.  Charts of more items than threads: from four contexts on lanes expand them,
    up to 24 items each, having looked at 256 (two sets of two items a kind); the others are left to the warp."""
    text, vocab = _endings(kinds)
    s = _run(text, "s", vocab, [list(p) for p in (b"(" * depth, b"(" * depth + b"x", b"(" * depth + b"x)a", b"((x)a")])
    assert s["rows_swept_again"] == 0


def test_rows_given_up_in_one_fill_after_the_other():
    """The Earley sets of rows that are given up come from one pool (64 Mi words, some 50,000 a row here): every fill begins with all of
    it, however many rows were swept before."""
    import torch

    import paper_2506_01151_b200 as fmt

    text, vocab = _endings(340)
    prefixes = [b"(" * 20, b"(" * 20 + b"x", b"(" * 20 + b"x)a"]
    g, batch = fmt.Grammar(text, "s", vocab, len(vocab) - 1), 255
    st = fmt.State(g, batch, cache=False)
    for i in range(max(map(len, prefixes))):
        t = [prefixes[b % 3][i] if i < len(prefixes[b % 3]) else -1 for b in range(batch)]
        st.advance(torch.tensor(t, dtype=torch.int32, device="cuda"))
    og, ov = oracle.Grammar(text, "s"), oracle.Vocab(vocab, len(vocab) - 1)
    want = []
    for p in prefixes:
        s = oracle.Sequence_(og)
        assert s.advance(p)
        want.append(s.mask(ov))
    want = np.tile(np.stack(want), (batch // 3, 1))
    mask = torch.zeros((batch, g.mask_words), dtype=torch.int32, device="cuda")
    for _ in range(9):
        st.fill_mask(mask)
        assert np.array_equal(mask.cpu().numpy().view(np.uint32), want)
    s = st.stats()
    assert s["capacity_errors"] == 0 and s["rows_swept_again"] > 1500


@pytest.mark.parametrize("text, start, prefixes", [
    ('content ::= node*\nnode ::= char | entity | "<p>" content "</p>" | "<b>" content "</b>"\nchar ::= [^<&]\nentity ::= "&" [a-z]+ ";"\n', "content",
     [b"<p>some <b>bold", b"text &am", b"", b"<p><b>x</"]),
    ('doc ::= el\nel ::= "<" name ">" (el | text)* "</" name ">"\ntext ::= [^<&]+\nname ::= [a-zA-Z] [a-zA-Z0-9-]*\n', "doc",
     [b"<a><b>some words of text", b"<a", b"<a><b>x</b>yz", b"<a>x</"])])
@pytest.mark.parametrize("batch", [1, 64, 300])
def test_text_whose_rules_end_everywhere(text, start, prefixes, batch):
    """Grammars whose chart is asked at most nodes of the trie have no automaton: their rows are swept, a few steps each."""
    w = workloads.build(2, V=20000, batch=1, steps=1)
    s = _run(text, start, w.vocab, [list(p) for p in prefixes], batch=batch, check=range(min(batch, 4)))
    assert s["walk_transitions"] < 2000 * batch and s["rows_swept_again"] == 0


def _compile_seconds(text, start, vocab, eos):
    """Processor time of the automaton's tables (and of the upload)."""
    import time

    import paper_2506_01151_b200 as fmt

    took = []
    for host_only in (True, True, False):  # (the first call builds or loads the library)
        t = time.process_time()
        fmt.Grammar(text, start, vocab, eos, host_only=host_only)
        took.append(time.process_time() - t)
    return took[2] - took[1]


def test_compiling_takes_a_bounded_time():
    """The walk over the trie takes a quarter of a second at most, whether the grammar gets the tables or not (300 kinds of elements around
    text, refused in the walk)."""
    w = workloads.build(2, V=128256, batch=1, steps=1)
    tags = _words(np.random.default_rng(1), 300, 4)
    text = "content ::= node*\nnode ::= char | entity | " + " | ".join('"<%s>" content "</%s>"' % (x, x) for x in tags)
    text += '\nchar ::= [^<&]\nentity ::= "&" [a-z]+ ";"\n'
    took = _compile_seconds(text, "content", w.vocab, w.eos)
    assert took < 0.7, took


def test_starts_and_edges_take_a_bounded_time():
    """Words of letters whose every byte may end a word, one after the other: 24,000 tokens of 32 bytes would have 13 million edges.  The walk
    and the starts' allowance, a second together, and the trie of 3 million nodes."""
    rng = np.random.default_rng(1)
    kw = " | ".join('"%s!"' % c for c in "abcdefghijklmnopqrstuvwxyz0123456789")
    text = 's ::= "(" p ")"\np ::= (w | "(" p ")" | "=" kw)*\nkw ::= %s\nw ::= [a-z]+ "0"?\n' % kw
    letters, others = np.frombuffer(b"abcdefghijklmnopqrstuvwxyz", np.uint8), np.frombuffer(b"0123456789!", np.uint8)
    vocab = [bytes([b]) for b in range(256)] + [bytes(letters[rng.integers(0, 26, 32)]) for _ in range(24000)]
    vocab += [b"!" + bytes(others[rng.integers(0, 11, 31)]) for _ in range(88800)] + [b""]  # (no text: see _braces)
    took = _compile_seconds(text, "s", vocab, len(vocab) - 1)
    assert took < 2.0, took  # (3.3 s while only look-ups counted, 0.95 now)


def test_grammar_without_an_automaton():
    """Alternations of more than a thousand literals have none: their rows are swept by Earley steps."""
    names = sorted({"k%06d" % (i * 7919 % 999983) for i in range(1200)})
    text = 's ::= "[" name ( "," name )* "]"\nname ::= ' + " | ".join('"%s"' % x for x in names)
    vocab = [bytes([b]) for b in range(256)] + [b"[k", b"k0", b"k1", names[5].encode(), (names[3] + ",").encode(), b""]
    s = _run(text, "s", vocab, [list(b"[k"), list(b"[" + names[9].encode()), list(b"")])
    assert s["walk_states"] > 0


def test_no_automaton_for_states_that_ask_for_earley_steps():
    """sweep_states limits the Earley sets of a sweep: a state that sets it runs the steps, and gives the same masks."""
    w = workloads.build(2, V=3000, batch=1, steps=1)
    a = _run(w.ebnf, w.start, w.vocab, JSON_PREFIXES)
    b = _run(w.ebnf, w.start, w.vocab, JSON_PREFIXES, sweep_states=4096)
    assert a["walk_states"] < b["walk_states"]


@pytest.mark.parametrize("batch", [1, 3, 65])
@pytest.mark.parametrize("options", [dict(sweep_states=4096), dict(roots=True)])
def test_sweeps_in_a_row_with_the_longest_tokens(batch, options):
    """Every fill starts from clean counters at every depth of the trie, however few rows (and so threads that clear them) there
    are: sweeps one after the other, each with steps to be made at depth 32."""
    import torch

    import paper_2506_01151_b200 as fmt

    w = workloads.build(2, V=300, batch=1, steps=1)
    vocab = [bytes([b]) for b in range(256)] + [b'"' + b"a" * 30 + b'"', b"[" * 32, b"[]," * 10 + b"[]", b"]" * 32, b""]
    g, og, ov = fmt.Grammar(w.ebnf, w.start, vocab, len(vocab) - 1), oracle.Grammar(w.ebnf, w.start), oracle.Vocab(vocab, len(vocab) - 1)
    st, seq = fmt.State(g, batch, cache=False, **options), oracle.Sequence_(og)
    mask = torch.zeros((batch, g.mask_words), dtype=torch.int32, device="cuda")
    for token in [ord("["), ord("["), 257, ord('"'), ord("x")]:
        st.advance(torch.full((batch,), token, dtype=torch.int32, device="cuda"))
        assert seq.advance(vocab[token])
        st.fill_mask(mask)
        got = mask.cpu().numpy().view(np.uint32)
        assert all(np.array_equal(row, seq.mask(ov)) for row in got), token
    assert st.stats()["fills_aborted"] == 0 and st.stats()["capacity_errors"] == 0


def _feed(text, start, data, options, dfa=True):
    """The chart words after feeding the bytes one by one, and in one token where they are at most 32."""
    import torch

    import paper_2506_01151_b200 as fmt

    pieces = [data[i:i + 32] for i in range(0, len(data), 32)]
    vocab = [bytes([b]) for b in range(256)] + pieces + [b""]
    g = fmt.Grammar(text, start, vocab, len(vocab) - 1, dfa=dfa)
    st = fmt.State(g, 2, **options)
    status = torch.zeros(2, dtype=torch.int32, device="cuda")
    for i in range(len(data)):
        whole = 256 + i // 32 if i % 32 == 0 else -1
        st.advance(torch.tensor([data[i], whole], dtype=torch.int32, device="cuda"), status)
        assert status.tolist() == [fmt.FMT_OK, fmt.FMT_OK], (i, data[:i + 1])
    q = st.query()
    return st.chart_words(0), st.chart_words(1), q


@pytest.mark.parametrize("nests", [1, 31, 32, 33, 70])
@pytest.mark.parametrize("dfa", [True, False])
def test_compact_down_a_deep_nesting(nests, dfa):
    """Compact stops at a set that holds everything before it: charts around multiples of 32 sets, the same words whether it ran
    after every byte or once per 32 bytes, every set still referenced."""
    w = workloads.build(2, V=300, batch=1, steps=1)
    data = b"".join(b'[1, {"k":' if i % 3 == 0 else b"[" for i in range(nests)) + b'"x'
    a, b, _ = _feed(w.ebnf, w.start, data, {}, dfa)
    assert a.tolist() == b.tolist()
    closing = data + b'"' + b"".join(b"}]" if i % 3 == 0 else b"]" for i in reversed(range(nests)))
    a, b, q = _feed(w.ebnf, w.start, closing, {}, dfa)
    assert a.tolist() == b.tolist() and q["accepting"].tolist() == [1, 1]


@pytest.mark.parametrize("letters", [8, 30, 33, 64, 200])
def test_sets_with_a_bit_for_every_item(letters):
    """Earley sets that outgrow a warp's lanes: around 32 items, and beyond what the bits hold (the hash takes over)."""
    text = 's ::= "<" e ">"\ne ::= e e | e n "+" n e | "(" e ")" | "a" | "b"\nn ::= "!" | ""'
    data = b"<" + b"".join(b"a" if i % 5 else b"(b+a)" for i in range(letters))
    a, b, _ = _feed(text, "s", data, dict(chart_words=1 << 18), True)
    assert a.tolist() == b.tolist()
    og = oracle.Grammar(text, "s")
    s = oracle.Sequence_(og, pruned=True)
    assert s.advance(data)
    assert int(a[0]) == s.num_sets and int(a[1]) == s.total_items


@pytest.mark.parametrize("n", [31, 32, 33, 64, 130, 300])
def test_compact_with_many_non_terminals(n):
    """What Compact keeps, with the non-terminals in one and in several words: chains of prediction and left recursion among them."""
    text = "s ::= n0 | s \",\" n1\n"
    text += "".join('n%d ::= n%d | "(" n%d ")" "%c" | n%d "+" "x"\n' % (i, i + 1, i * 7 % (n - 2), 97 + i % 26, i) for i in range(n - 2))
    text += 'n%d ::= "x" | "[" s "]"' % (n - 2)
    data = b"x,((x+x"
    for dfa in (True, False):
        a, b, _ = _feed(text, "s", data, {}, dfa)
        assert a.tolist() == b.tolist()
        seq = oracle.Sequence_(oracle.Grammar(text, "s"), pruned=True)
        assert seq.advance(data)
        assert int(a[0]) == seq.num_sets and int(a[1]) == seq.total_items


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("V", [1, 7, 8, 15, 16, 17, 31, 33, 63, 64, 65, 4095, 4097, 16 * 512 + 3])
def test_masking_rows_that_begin_anywhere(dtype, V):
    """Rows are masked in units of 32 bytes from their first 32-byte boundary on: every place in a unit a row can begin, vocabularies
    around whole units, units that are all valid, all invalid and mixed, and nothing written beside the row."""
    import torch

    import paper_2506_01151_b200 as fmt

    rng = np.random.default_rng(V)
    kind, bits = (np.uint16, 16) if dtype == "bf16" else (np.uint32, 32)
    stride, batch = V + 5, 9
    keep = rng.random((batch, V)) < np.array([0.0, 1.0, 0.5, 0.9, 0.05, 0.5, 0.5, 0.5, 0.5])[:, None]
    words = (V + 31) // 32
    mask = np.zeros((batch, words * 32), np.uint8)
    mask[:, :V] = keep
    mask = np.packbits(mask, axis=1, bitorder="little").view(np.uint32)
    for shift in range(0, 32 * 8 // bits, 3 if V > 100 else 1):
        logits = rng.integers(0, 1 << bits, size=shift + batch * stride, dtype=np.uint64).astype(kind)
        want = logits.copy()
        rows = want[shift:].reshape(batch, stride)
        rows[:, :V][~keep] = 0xFF80 if dtype == "bf16" else 0xFF800000
        on_gpu = torch.from_numpy(logits.view(np.int16 if bits == 16 else np.int32)).cuda()
        m = torch.from_numpy(np.ascontiguousarray(mask).view(np.int32)).cuda()
        fmt.apply_mask(m, on_gpu.data_ptr() + shift * bits // 8, fmt.BF16 if dtype == "bf16" else fmt.FP32, batch, V, row_stride=stride)
        assert np.array_equal(on_gpu.cpu().numpy().view(kind), want), shift


def test_transitions_met_by_several_blocks_of_a_launch():
    """Rows at one chart take one token, from caches that know nothing: some rows of a launch find what others of it have entered a
    moment before.  All of them end up at the same chart, the one a single row reaches."""
    import torch

    import paper_2506_01151_b200 as fmt

    w = workloads.build(2, V=300, batch=1, steps=1)
    g = fmt.Grammar(w.ebnf, w.start, w.vocab, w.eos)
    batch = 3000
    many, one = fmt.State(g, batch, chart_words=1 << 12), fmt.State(g, 1, cache=False)
    status = torch.zeros(batch, dtype=torch.int32, device="cuda")
    for _ in range(20):
        many.cache_clear()
        many.reset()
        one.reset()
        for b in b'{"a": [1, {"k": tr':
            many.advance(torch.full((batch,), b, dtype=torch.int32, device="cuda"), status)
            one.advance(torch.full((1,), b, dtype=torch.int32, device="cuda"))
            assert not status.any()
        q, want = many.query(), one.query()
        assert len(set(q["state_id"].tolist())) == 1 and (q["n_items"] == want["n_items"][0]).all() and (q["n_sets"] == want["n_sets"][0]).all()
        assert many.chart_words(batch - 1).tolist() == one.chart_words(0).tolist()
    s = many.stats()
    assert s["capacity_errors"] == 0 and 0 < s["advances_cached"] < s["steps_advanced"]


def _words(rng, n, length, first=""):
    got = set()
    while len(got) < n:
        got.add(first + "".join(chr(97 + int(c)) for c in rng.integers(0, 26, length)))
    return sorted(got)


@pytest.mark.parametrize("batch", [1, 3, 149, 700])
@pytest.mark.parametrize("tables", ["all in shared memory", "automata in global memory", "all in global memory"])
def test_advance_wherever_the_tables_are(tables, batch):
    """Rows advance one, two or four to a block, by how many there are and by how large the grammar's tables are: the same charts
    as one row's fed byte by byte, and as many sets and items as the oracle's."""
    import torch

    import paper_2506_01151_b200 as fmt

    rng = np.random.default_rng(7)
    if tables == "all in shared memory":
        names, text = _words(rng, 12, 4), 's ::= "(" s ")" | s "+" s | name\nname ::= %s'
    elif tables == "automata in global memory":
        names = [w for d in range(12) for w in _words(rng, 70, 6, str(d))]
        text = 's ::= "(" s ")" | s "+" s | ' + " | ".join("w%d" % d for d in range(12)) + "\n"
        text += "\n".join('w%d ::= %s' % (d, " | ".join('"%s"' % x for x in names[70 * d:70 * d + 70])) for d in range(12)) + "\nunused ::= %s"
    else:
        names, text = _words(rng, 700, 7), 's ::= "(" s ")" | s "+" s | name\nname ::= %s'
    text = text % " | ".join('"%s"' % x for x in names)
    data = ("((%s+%s)+%s" % (names[0], names[-1], names[len(names) // 2])).encode()
    tokens = [data[:2], data[2:7], data[7:13], data[13:]]
    vocab = [bytes([b]) for b in range(256)] + tokens + [b""]
    g = fmt.Grammar(text, "s", vocab, len(vocab) - 1, dfa=tables != "all in global memory")
    one, many = fmt.State(g, 1), fmt.State(g, batch, max_states=4096, chart_words=1 << 14, pool_words=1 << 22, max_mask_rows=8)
    status, statuses = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(batch, dtype=torch.int32, device="cuda")
    for b in data:
        one.advance(torch.tensor([b], dtype=torch.int32, device="cuda"), status)
        assert status.tolist() == [fmt.FMT_OK]
    for i in range(len(tokens)):
        many.advance(torch.full((batch,), 256 + i, dtype=torch.int32, device="cuda"), statuses)
        assert not statuses.any()
    want = one.chart_words(0).tolist()
    for row in {0, batch // 2, batch - 1}:
        assert many.chart_words(row).tolist() == want
    seq = oracle.Sequence_(oracle.Grammar(text, "s"), pruned=True)
    assert seq.advance(data)
    if tables == "all in global memory":  # (automata have items of their own)
        assert want[1] == seq.total_items
    assert want[0] == seq.num_sets


@pytest.mark.parametrize("n", [64, 65, 1024, 1025, 2047, 2048, 5000])
def test_lists_of_edges_and_of_tokens(n):
    """Where strings end inside n tokens, one kernel item has n edges (grouped by item from 65 on, behind several edges from 1,025 on),
    and where one string ends and the next begins inside n more, an edge has n tokens (several edges from 2,048 on, and more lists of
    tokens in a round than there is room for)."""
    w = workloads.build(2, V=300, batch=1, steps=1)
    words = [bytes([97 + i // 676, 97 + i // 26 % 26, 97 + i % 26]) for i in range(n)]
    vocab = [bytes([b]) for b in range(256)] + [x + b'",' for x in words] + [b'","' + x for x in words] + [x + b'":[]' for x in words[::2]] + [x + b'"]' for x in words[::3]] + [b""]
    _run(w.ebnf, w.start, vocab, [list(p) for p in (b'["x', b'{"k":"x', b'{"', b'[["x"', b'[')])


@pytest.mark.parametrize("depth", [20, 56, 73, 74, 75, 76, 112, 150, 190, 260])
def test_charts_around_an_item_to_a_thread(depth):
    """The contexts of a chart of up to 224 items are made by a thread for each; larger ones, and charts of more than 768 words, have
    them made as they are asked for."""
    vocab = [bytes([b]) for b in range(256)] + [b"]" * k for k in range(2, 33)] + [b"]}", b'],"', b"}]", b"1]", b"]]}", b'"]]', b"1,[[", b"]," * 8, b""]
    w = workloads.build(2, V=300, batch=1, steps=1)
    _run(w.ebnf, w.start, vocab, [list(p) for p in (b"[" * depth, b"[1," * depth + b'"', b'{"a":[' * (depth // 2) + b"1")])


@pytest.mark.parametrize("n", [2, 12, 29, 31, 33, 70])
@pytest.mark.parametrize("dfa", [True, False])
def test_chains_completed_in_one_set(n, dfa):
    """What is completed with a completed item in the set where both began: chains of n rules of one symbol, with something nullable
    behind it, in sets below and above 32 items."""
    text = "s ::= n0 | s \",\" n0\n" + "".join('n%d ::= n%d z | n%d "+" n%d\n' % (i, i + 1, i, i + 1) for i in range(n))
    text += 'n%d ::= "x" | "(" s ")"\nz ::= "!" | ""' % n
    data = b"x,(x+x!,(x)),x"
    a, b, _ = _feed(text, "s", data, dict(chart_words=1 << 16), dfa)
    assert a.tolist() == b.tolist()
    seq = oracle.Sequence_(oracle.Grammar(text, "s"), pruned=True)
    assert seq.advance(data)
    assert int(a[0]) == seq.num_sets
    if not dfa:  # (automata have items of their own)
        assert int(a[1]) == seq.total_items


def test_a_captured_fill_that_gave_up_starts_afresh():
    """A fill whose rounds run out hands out empty masks, and the next one is a fill like any, also where both are replays of one
    captured call: "[[[[[[" with tokens of closing brackets takes a round for each, a string without tokens that end it takes one."""
    import torch

    import paper_2506_01151_b200 as fmt

    w = workloads.build(2, V=300, batch=1, steps=1)
    vocab = [bytes([b]) for b in range(256)] + [b"]" * k for k in range(2, 7)] + [b"xy", b""]
    g = fmt.Grammar(w.ebnf, w.start, vocab, len(vocab) - 1)
    st = fmt.State(g, 2, cache=False, wait_limit_log2=1)
    seq, ov = oracle.Sequence_(oracle.Grammar(w.ebnf, w.start)), oracle.Vocab(vocab, len(vocab) - 1)
    mask = torch.full((2, g.mask_words), -1, dtype=torch.int32, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        st.fill_mask(mask, stream=torch.cuda.current_stream().cuda_stream)

    def feed(data):
        for b in data:
            st.advance(torch.full((2,), b, dtype=torch.int32, device="cuda"))
        assert seq.advance(data)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        return mask.cpu().numpy().view(np.uint32)

    assert not feed(b"[[[[[[").any() and st.stats()["fills_aborted"] == 1
    for data in (b'"x', b"y"):
        got = feed(data)
        assert np.array_equal(got[0], seq.mask(ov)) and np.array_equal(got[1], seq.mask(ov))
    assert not feed(b'",[[').any()
    assert st.stats()["fills_aborted"] == 2 and st.stats()["capacity_errors"] == 0


def test_captured_fills_with_rows_given_up():
    """Rows that a replayed fill gives up are swept, those of this replay and not of the one before."""
    import torch

    import paper_2506_01151_b200 as fmt

    text, vocab = _endings(340)
    g, og, ov = fmt.Grammar(text, "s", vocab, len(vocab) - 1), oracle.Grammar(text, "s"), oracle.Vocab(vocab, len(vocab) - 1)
    st = fmt.State(g, 24, cache=False)
    mask = torch.full((24, g.mask_words), -1, dtype=torch.int32, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        st.fill_mask(mask, stream=torch.cuda.current_stream().cuda_stream)
    deep, flat = b"(" * 20, b"((x)"
    for replay in range(3):
        texts = [deep + b"x" * (b % 2) if (b + replay) % 3 else flat for b in range(24)]
        st.reset()
        for i in range(max(map(len, texts))):
            st.advance(torch.tensor([t[i] if i < len(t) else -1 for t in texts], dtype=torch.int32, device="cuda"))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        got, want = mask.cpu().numpy().view(np.uint32), {}
        for t in set(texts):
            s = oracle.Sequence_(og)
            assert s.advance(t)
            want[t] = s.mask(ov)
        for b in range(24):
            assert np.array_equal(got[b], want[texts[b]]), (replay, b)
    s = st.stats()
    assert s["rows_swept_again"] >= 3 * 12 and s["capacity_errors"] == 0 and s["fills_aborted"] == 0


def test_text_read_to_its_end():
    """Nothing is left in the chart of a finite text that has been read to its end: EOS alone is valid."""
    text = 's ::= "[" t "]" | "(" t ")"\nt ::= "ab" | "[" "x" "]"'
    vocab = [bytes([b]) for b in range(256)] + [b"ab]", b"[x]", b"[x])", b"]]", b""]
    _run(text, "s", vocab, [list(p) for p in (b"[ab]", b"([x])", b"[ab", b"(")])


@pytest.mark.parametrize("pairs", [98, 101, 102, 104])
def test_contexts_that_leave_shared_memory_with_the_last_set(pairs):
    """The items of the chart have contexts of their own; those of the last set's kernel, each begun in two of fifteen sets, come on
    top, and from 102 pairs on all of them together are more than the 320 that shared memory holds."""
    letters = b"abcdefghijklmno"
    two = [(a, b) for a in range(15) for b in range(a + 1, 15)][:pairs]
    end = lambda k: "%c%c" % (65 + k // 26, 65 + k % 26)
    text = "s ::= p m \"!\"\np ::= [a-o]*\nm ::= " + " | ".join('x%d "%s"' % (k, end(k)) for k in range(pairs)) + ' | "(" m ")"\n'
    text += "".join('x%d ::= "%sz" | "%sz"\n' % (k, letters[a:].decode(), letters[b:].decode()) for k, (a, b) in enumerate(two))
    vocab = [bytes([b]) for b in range(256)] + [(end(k) + ("!" if k % 2 else "?")).encode() for k in range(pairs)] + [b""]
    s = _run(text, "s", vocab, [list(letters + b"z")])
    assert s["rows_swept_again"] == 0 and (s["walk_states"] > 320) == (pairs >= 102)
