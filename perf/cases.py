"""What this library is used for, as cases that can be timed: decoding loops, single mask fills, prefix replays, logits
masking, allocation-free fills and jump-ahead, over the grammars, vocabularies and batches that the tests and the
benchmark use and the sizes around them.

A case's kind says which public calls one pass makes:
  decode   a batch of documents from empty caches: caches emptied, rows reset, each row's text so far replayed, then per
           decoding step State.advance with the chosen tokens and State.fill_and_apply on that step's logits
  steady   the same with the caches kept, as a server has them after a while (most charts have been met before)
  fill     State.fill_mask for rows in the middle of their documents, on a state without the state cache, so that every
           row's mask is computed
  prefill  State.advance over a long text (a request taken up again), then the mask of where it ends
  apply    apply_mask on the logits of several positions with masks that are there already
  noalloc  fill_mask_noalloc for charts held in device memory
  forced   State.forced_bytes: the bytes every continuation must begin with
"""
import functools
import json
import math
import random

import numpy as np
import torch

import paper_2506_01151_b200 as fmt

# ------------------------------------------------------------------------------------------------ grammars

_ARITH = r"""
expr   ::= expr [+\-] term | term
term   ::= term [*/] factor | factor
factor ::= "(" expr ")" | number
number ::= [0-9]+
"""

_JSON = r"""
json     ::= ws value ws
value    ::= object | array | string | number | "true" | "false" | "null" @EXTRA@
object   ::= "{" ws "}" | "{" members "}"
members  ::= pair | members "," pair
pair     ::= ws string ws ":" ws value ws
array    ::= "[" ws "]" | "[" elements "]"
elements ::= element | elements "," element
element  ::= ws value ws
ws       ::= [ \t\n\r]*
string   ::= "\"" char* "\""
char     ::= [\x20-\x21\x23-\x5b\x5d-\x7f] | "\\" escape | utf8
escape   ::= ["\\/bfnrt] | "u" hex hex hex hex
hex      ::= [0-9a-fA-F]
utf8     ::= [\xc2-\xdf] cont
           | "\xe0" [\xa0-\xbf] cont | [\xe1-\xec\xee-\xef] cont cont | "\xed" [\x80-\x9f] cont
           | "\xf0" [\x90-\xbf] cont cont | [\xf1-\xf3] cont cont cont | "\xf4" [\x80-\x8f] cont cont
cont     ::= [\x80-\xbf]
number   ::= "-"? ( "0" | [1-9] [0-9]* ) ( "." [0-9]+ )? ( [eE] [+\-]? [0-9]+ )?
"""

# the ambiguous, nullable-heavy value alternative of the long-context workload
_AMBIGUOUS = r"""
amb  ::= W E W
E    ::= E E | E O3 "+" O3 E | "(" W E W ")" | "a" | "b"
W    ::= N0 | O4
O1   ::= "!"?
O2   ::= O1 O1
O3   ::= O2 | "" | O1 O2
O4   ::= O3 O3 | O1
""" + "".join('N%d ::= N%d N%d | ""\n' % (i, i + 1, i + 2) for i in range(10)) + 'N10 ::= "_" | ""\nN11 ::= "~" | ""\n'

_SQL = r"""
query      ::= select_stmt ";"?
select_stmt ::= "SELECT " distinct? select_list " FROM " table_ref join* where? group? order? limit?
distinct   ::= "DISTINCT "
select_list ::= "*" | select_item ( "," sp select_item )*
select_item ::= expr alias?
alias      ::= " AS " colname
table_ref  ::= tabname tab_alias?
tab_alias  ::= " " tabalias
join       ::= join_kind "JOIN " table_ref " ON " cond
join_kind  ::= " " | " LEFT " | " INNER " | " RIGHT "
where      ::= " WHERE " cond
group      ::= " GROUP BY " colref ( "," sp colref )* having?
having     ::= " HAVING " cond
order      ::= " ORDER BY " order_item ( "," sp order_item )*
order_item ::= colref ( " ASC" | " DESC" )?
limit      ::= " LIMIT " uint
cond       ::= cond " OR " cond_and | cond_and
cond_and   ::= cond_and " AND " cond_not | cond_not
cond_not   ::= "NOT " cond_not | pred
pred       ::= expr cmp expr | expr " IS NULL" | expr " IS NOT NULL" | expr " IN (" expr_list ")"
             | expr " BETWEEN " expr " AND " expr | expr " LIKE " sqlstring | "(" cond ")"
cmp        ::= " = " | " <> " | " < " | " > " | " <= " | " >= "
expr_list  ::= expr ( "," sp expr )*
expr       ::= expr " + " term | expr " - " term | term
term       ::= term " * " factor | term " / " factor | factor
factor     ::= colref | number | sqlstring | func "(" func_arg ")" | "(" expr ")" | "-" factor
func       ::= "COUNT" | "SUM" | "AVG" | "MIN" | "MAX"
func_arg   ::= "*" | expr | "DISTINCT " expr
colref     ::= colname | tabname "." colname | tabalias "." colname
tabalias   ::= [a-z] [0-9]
sqlstring  ::= "'" sqlchar* "'"
sqlchar    ::= [\x20-\x26\x28-\x7e] | "''"
number     ::= uint ( "." [0-9]+ )?
uint       ::= [0-9]+
sp         ::= " "?
"""


def _name(rng, lo, hi):
    return "".join(rng.choice("aeiou" if i % 2 else "bcdfghjklmnprstvwz") for i in range(rng.randint(lo, hi)))


def _names(rng, n, lo, hi, prefix=""):
    got = set()
    while len(got) < n:
        got.add(prefix + _name(rng, lo, hi))
    return sorted(got)


@functools.lru_cache(maxsize=None)
def _sql_names():
    rng = random.Random(41)
    return _names(rng, 60, 3, 8, "t_"), _names(rng, 140, 3, 9)


@functools.lru_cache(maxsize=None)
def _schema():
    """Twelve required and optional typed members, enums, nested objects and an array of objects."""
    rng = random.Random(31)

    def node(kind, depth):
        if kind == "enum":
            return {"enum": _names(rng, rng.randint(3, 10), 3, 9)}
        if kind == "object":
            return members(rng.randint(2, 4), depth + 1)
        if kind == "array":
            return {"type": "array", "items": members(rng.randint(2, 4), depth + 1)}
        return {"type": kind}

    def members(n, depth):
        kinds = ["string", "number", "integer", "boolean", "enum"] + (["object", "array", "enum", "string"] if depth < 3 else [])
        names = _names(rng, n, 3, 10)
        rng.shuffle(names)
        wanted = ["object" if depth == 1 and i == 3 else "array" if depth == 1 and i == 7 else rng.choice(kinds) for i in range(n)]
        props = {name: node(kind, depth) for name, kind in zip(names, wanted)}
        return {"type": "object", "properties": props, "required": [x for i, x in enumerate(names) if i == 0 or rng.random() < 0.6]}

    return members(12, 1)


# ------------------------------------------------------------------------------------------------ documents

_CHARS = "abcdefghijklmnopqrstuvwxyzABCDEFGHIJKLMNOPQRSTUVWXYZ0123456789"


def _ws(rng, p=0.3):
    return rng.choice((" ", " ", "\n", "\n  ", "\t")) if rng.random() < p else ""


def _count(rng, mean, most):
    return min(most, int(rng.expovariate(1.0 / mean)))


def _string(rng, mean=6.0):
    out = []
    for _ in range(_count(rng, mean, 40)):
        r = rng.random()
        out.append(rng.choice(_CHARS) if r < 0.8 else rng.choice(" _-.,:;!?/()") if r < 0.9 else chr(rng.randint(0xA0, 0x7FF)) if r < 0.93
                   else chr(rng.randint(0x3041, 0x9FA0)) if r < 0.95 else "\\" + rng.choice('"\\/bfnrt') if r < 0.99 else "\\u%04x" % rng.randint(0, 0xFFFF))
    return '"' + "".join(out) + '"'


def _number(rng, whole=False):
    out = ("-" if rng.random() < 0.2 else "") + ("0" if rng.random() < 0.15 else str(rng.randint(1, 9)) + "".join(rng.choice("0123456789") for _ in range(_count(rng, 1.5, 8))))
    if not whole and rng.random() < 0.3:
        out += "." + str(rng.randint(0, 9999))
    return out + ("e%d" % rng.randint(-9, 9) if not whole and rng.random() < 0.1 else "")


def _expression(rng, budget, depth=0):
    """A sentence of `E` of the ambiguous grammar, of at most about `budget` bytes."""
    r = rng.random()
    if budget <= 2 or depth > 6 or r < 0.2:
        return rng.choice("ab")
    if r < 0.4 and budget > 8:
        return "(" + _expression(rng, budget - 2, depth + 1) + ")"
    left = _expression(rng, budget // 2, depth + 1)
    plus = "" if r < 0.8 else "!" * rng.randint(0, 2) + "+"
    return left + plus + _expression(rng, budget - len(left) - len(plus), depth + 1)


def _ambiguous(rng):
    return "<" + rng.choice(("", "", "_", "~", "!")) + _expression(rng, rng.randint(4, 60)) + rng.choice(("", "", "!!", "_")) + ">"


def _value(rng, depth, most, extra):
    r = rng.random()
    if extra and r < 0.18:
        return _ambiguous(rng)
    r = rng.random() if depth < most else 0.5 + rng.random() / 2
    if r < 0.3:
        return "{" + (",".join(_pair(rng, depth + 1, most, extra) for _ in range(rng.randint(0, 4))) or _ws(rng)) + "}"
    if r < 0.5:
        return "[" + (",".join(_ws(rng) + _value(rng, depth + 1, most, extra) + _ws(rng, 0.1) for _ in range(rng.randint(0, 4))) or _ws(rng)) + "]"
    return _string(rng) if r < 0.7 else _number(rng) if r < 0.85 else rng.choice(("true", "false", "null"))


def _pair(rng, depth, most, extra):
    return _ws(rng) + _string(rng, 4.0) + _ws(rng, 0.1) + ":" + _ws(rng, 0.5) + _value(rng, depth, most, extra) + _ws(rng, 0.1)


def _deep(rng, depth):
    """A spine of nested arrays and objects with an ambiguous value at its end."""
    if depth == 0:
        return _ambiguous(rng)
    if rng.random() < 0.5:
        return "[" + _deep(rng, depth - 1) + "," + _value(rng, 9, 9, True) + "]"
    return "{" + _string(rng, 3.0) + ":" + _deep(rng, depth - 1) + "}"


def _json_doc(rng, size, extra=False):
    parts = []
    while sum(map(len, parts)) < size:
        parts.append(_string(rng, 4.0) + ":" + _deep(rng, rng.randint(8, 30)) if extra and rng.random() < 0.15 else _pair(rng, 1, 6, extra))
    return "{" + ",".join(parts) + "}"


def _instance(rng, node):
    if "enum" in node:
        return '"' + rng.choice(node["enum"]) + '"'
    kind = node["type"]
    if kind == "object":
        took = [k for k in node["properties"] if k in node["required"] or rng.random() < 0.6]
        return "{" + _ws(rng) + ("," + _ws(rng, 0.5)).join('"%s":%s%s' % (k, _ws(rng, 0.5), _instance(rng, node["properties"][k])) for k in took) + "}"
    if kind == "array":
        return "[" + ",".join(_ws(rng) + _instance(rng, node["items"]) for _ in range(rng.randint(0, 3))) + "]"
    return _string(rng, 8.0) if kind == "string" else rng.choice(("true", "false")) if kind == "boolean" else _number(rng, kind == "integer")


def _sql_doc(rng):
    tabs, cols = _sql_names()

    def factor(d):
        r = rng.random()
        if r < 0.5:
            return rng.choice(cols) if r < 0.25 else rng.choice(tabs) + "." + rng.choice(cols) if r < 0.4 else "%s%d.%s" % (rng.choice("abcdxyz"), rng.randint(0, 9), rng.choice(cols))
        if r < 0.8 or d > 2:
            return str(rng.randint(0, 99999)) if r < 0.65 else "'" + "".join(rng.choice(_CHARS + " ") for _ in range(_count(rng, 5.0, 16))) + "'"
        return rng.choice(("COUNT", "SUM", "AVG", "MIN", "MAX")) + "(" + expr(d + 1) + ")" if r < 0.9 else "(" + expr(d + 1) + ")"

    def expr(d=0):
        return rng.choice((" + ", " - ", " * ", " / ")).join(factor(d) for _ in range(1 + (rng.random() < 0.3)))

    def pred():
        r = rng.random()
        if r < 0.5:
            return expr() + rng.choice((" = ", " <> ", " < ", " > ", " <= ", " >= ")) + expr()
        return expr() + (" IS NOT NULL" if r < 0.6 else " IN (" + ", ".join(expr(2) for _ in range(3)) + ")" if r < 0.8 else " BETWEEN " + expr() + " AND " + expr())

    def cond():
        return rng.choice((" AND ", " OR ")).join(pred() for _ in range(rng.randint(1, 3)))

    out = "SELECT " + ", ".join(expr() for _ in range(rng.randint(1, 4))) + " FROM " + rng.choice(tabs) + " a1"
    for _ in range(rng.randint(0, 2)):
        out += rng.choice((" ", " LEFT ", " INNER ")) + "JOIN " + rng.choice(tabs) + " b2 ON " + cond()
    out += " WHERE " + cond() if rng.random() < 0.7 else ""
    out += " GROUP BY " + rng.choice(cols) if rng.random() < 0.3 else ""
    return out + (" ORDER BY " + rng.choice(cols) + " DESC" if rng.random() < 0.4 else "")


def _arith_doc(rng, depth=0):
    terms = ["(" + _arith_doc(rng, depth + 1) + ")" if depth < 4 and rng.random() < 0.3 else str(rng.randint(0, 99999)) for _ in range(rng.randint(1, 5) if depth else 24)]
    return "".join(t + rng.choice("+-*/") for t in terms[:-1]) + terms[-1]


def _document(grammar, rng, size):
    doc = {"arith": lambda: _arith_doc(rng), "json": lambda: _json_doc(rng, size), "stress": lambda: _json_doc(rng, size, True),
           "schema": lambda: _instance(rng, _schema()), "sql": lambda: _sql_doc(rng)}[grammar]()
    return doc.encode("utf-8")


# ------------------------------------------------------------------------------------------------ vocabularies

_MAX_TOKEN = 16


def _vocabulary(grammar, size):
    """256 single bytes, distinct tokens of 2 to 16 bytes (mean about 4; most of them substrings of documents, the rest
    words), and as the last one the end of the sequence, which has no bytes."""
    rng = random.Random("vocabulary " + grammar)
    corpus = b"\n".join(_document(grammar, rng, 1500) for _ in range(300 if grammar in ("arith", "schema", "sql") else 120))
    vocab = [bytes([b]) for b in range(256)]
    seen = set(vocab)
    tries = 0
    while len(vocab) < size - 1:
        tries += 1
        n = min(_MAX_TOKEN, 2 + int(rng.expovariate(0.42)) + (tries > 8 * size) * rng.randint(0, 6))
        if rng.random() < 0.6:
            at = rng.randrange(len(corpus) - n)
            token = corpus[at:at + n]
        elif rng.random() < 0.9:
            token = ((" " if rng.random() < 0.4 else "") + "".join(rng.choices(_CHARS, k=n)))[:n].encode()
        else:
            token = "".join(chr(rng.randint(0xA0, 0x7FF)) for _ in range(n // 2)).encode("utf-8")
        if token not in seen:
            seen.add(token)
            vocab.append(token)
    return vocab + [b""]


@functools.lru_cache(maxsize=6)
def _compiled(grammar, size):
    """The compiled grammar, which a server keeps for as long as it runs, its tokens, and each token's id."""
    vocab = _vocabulary(grammar, size)
    if grammar == "schema":
        g = fmt.Grammar.from_json_schema(json.dumps(_schema()), vocab, size - 1)
    else:
        tabs, cols = _sql_names()
        text, start = {
            "arith": (_ARITH, "expr"), "json": (_JSON.replace("@EXTRA@", ""), "json"),
            "stress": (_JSON.replace("@EXTRA@", '| "<" amb ">"') + _AMBIGUOUS, "json"),
            "sql": (_SQL + "tabname ::= %s\ncolname ::= %s\n" % tuple(" | ".join('"%s"' % x for x in names) for names in (tabs, cols)), "query"),
        }[grammar]
        g = fmt.Grammar(text, start, vocab, size - 1)
    return g, vocab, {t: i for i, t in enumerate(vocab) if t}


def _encode(ids, data):
    """Greedy longest match."""
    out, at = [], 0
    while at < len(data):
        n = _MAX_TOKEN
        while data[at:at + n] not in ids:
            n = min(n, len(data) - at) - 1
        out.append(ids[data[at:at + n]])
        at += len(data[at:at + n])
    return out


def _streams(case, rng):
    """Per row a document, cut after up to case["context"] tokens: the text so far, and then `steps` tokens to decode: the
    document's rest, the end of the sequence, and further documents from their start (the row is reset before one).
    Long documents are dealt out to several rows, which cut them at different places."""
    grammar, batch, context, steps = case["grammar"], case["batch"], case["context"], case.get("steps", 0)
    _, vocab, ids = _compiled(grammar, case["vocab"])
    eos = len(vocab) - 1
    size = 200 + 4 * (context + steps)
    pool = [_encode(ids, _document(grammar, rng, size)) for _ in range(min(batch + 4, max(12, 150000 // size)))]
    prefix = np.full((max(context, 1), batch), -1, np.int32)
    tokens = np.full((steps, batch), -1, np.int32)
    resets = [[] for _ in range(steps)]
    for b in range(batch):
        doc = pool[b % len(pool)]
        cut = min(rng.randint(context // 4, context) if b else context, len(doc))
        prefix[:cut, b] = doc[:cut]
        queue = doc[cut:] + [eos]
        for s in range(steps):
            if not queue:
                queue = rng.choice(pool) + [eos]
                resets[s].append(b)
            tokens[s, b] = queue.pop(0)
    return prefix, tokens, resets


# ------------------------------------------------------------------------------------------------ the cases


def listed():
    return [
        # one decoding step of one sequence in a small vocabulary, every answer in the caches: call and launch latency
        {"name": "steady-arith-512-b1", "kind": "steady", "grammar": "arith", "vocab": 512, "batch": 1, "context": 0, "steps": 1, "logits": "bf16"},
        # a few interactive sessions writing JSON that nobody has written before
        {"name": "decode-json-32k-b8", "kind": "decode", "grammar": "json", "vocab": 32000, "batch": 8, "context": 32, "steps": 24, "logits": "bf16"},
        # structured output under a JSON schema, a batch job's start
        {"name": "decode-schema-128k-b64", "kind": "decode", "grammar": "schema", "vocab": 128256, "batch": 64, "context": 48, "steps": 16, "logits": "bf16"},
        # the same service once it is warm; a model whose logits are in 32 bits
        {"name": "steady-schema-128k-b64", "kind": "steady", "grammar": "schema", "vocab": 128256, "batch": 64, "context": 16, "steps": 16, "logits": "fp32"},
        # a large batch of semantic parsing: long alternations of names
        {"name": "decode-sql-152k-b128", "kind": "decode", "grammar": "sql", "vocab": 152064, "batch": 128, "context": 32, "steps": 12, "logits": "bf16"},
        # an ordinary fill at an odd vocabulary and an odd batch
        {"name": "fill-json-50001-b37", "kind": "fill", "grammar": "json", "vocab": 50001, "batch": 37, "context": 150},
        # the heaviest fill: deep nesting and ambiguous segments, thousands of bytes into the documents
        {"name": "fill-stress-128k-b256", "kind": "fill", "grammar": "stress", "vocab": 128256, "batch": 256, "context": 800},
        # long requests that are taken up again
        {"name": "prefill-stress-128k-b32", "kind": "prefill", "grammar": "stress", "vocab": 128256, "batch": 32, "context": 400},
        # masks that came from elsewhere (another process, the host), applied to the logits of a few drafted positions
        {"name": "apply-bf16-128k-b256", "kind": "apply", "vocab": 128256, "batch": 256, "steps": 4, "logits": "bf16"},
        # the same where rows do not begin on 16-byte boundaries
        {"name": "apply-bf16-50001-b48", "kind": "apply", "vocab": 50001, "batch": 48, "steps": 4, "logits": "bf16"},
        # a plug-in that may not allocate device memory
        {"name": "noalloc-json-32k-n24", "kind": "noalloc", "grammar": "json", "vocab": 32000, "batch": 24, "context": 150},
        # jump-ahead over the keys and the punctuation that a schema fixes
        {"name": "forced-schema-128k-b64", "kind": "forced", "grammar": "schema", "vocab": 128256, "batch": 64, "context": 48},
    ]


def _spread(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# per kind: the grammars with their largest vocabulary, batch, context and number of steps.  (Kinds that return masks or
# bytes alone begin at a few rows: one row's answer is often the same for two texts.)
_RANGES = {
    "decode": [("arith", 8192, 32, 16, 16), ("json", 65536, 64, 32, 16), ("schema", 128256, 64, 48, 16), ("sql", 152064, 128, 32, 12)],
    "steady": [("arith", 8192, 32, 16, 16), ("json", 65536, 64, 32, 16), ("schema", 128256, 64, 48, 16), ("sql", 152064, 96, 32, 8)],
    "fill": [("arith", 8192, 64, 16, 0), ("json", 128256, 128, 400, 0), ("schema", 128256, 128, 48, 0), ("sql", 152064, 128, 48, 0), ("stress", 128256, 192, 600, 0)],
    "prefill": [("json", 128256, 64, 400, 0), ("schema", 128256, 64, 48, 0), ("sql", 152064, 64, 48, 0), ("stress", 128256, 32, 350, 0)],
    "noalloc": [("json", 32000, 24, 150, 0), ("schema", 32000, 24, 48, 0)],
    "forced": [("schema", 128256, 128, 48, 0)],
}


def draw(rng):
    kind = rng.choice(("decode", "decode", "steady", "fill", "fill", "prefill", "apply", "apply", "noalloc", "forced"))
    if kind == "apply":
        return {"kind": kind, "vocab": _spread(rng, 512, 152064), "batch": _spread(rng, 1, 128), "steps": rng.randint(2, 4), "logits": rng.choice(("bf16", "fp32"))}
    grammar, vocab, batch, context, steps = rng.choice(_RANGES[kind])
    case = {"kind": kind, "grammar": grammar, "vocab": _spread(rng, 512, vocab), "batch": _spread(rng, 1 if steps else 12, batch), "context": _spread(rng, 8, context)}
    if steps:
        case.update(steps=_spread(rng, 1, steps), logits=rng.choice(("bf16", "fp32")))
    return case


# ------------------------------------------------------------------------------------------------ preparing and running


def _mask_words(case):
    return (case["vocab"] + 31) // 32


def _logits(case, seed, steps):
    """Fresh logits for every step, about as wide as a model's."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dtype = torch.bfloat16 if case["logits"] == "bf16" else torch.float32
    out = torch.empty((steps, case["batch"], case["vocab"]), dtype=dtype, device="cuda")
    for s in range(steps):
        out[s] = torch.randn((case["batch"], case["vocab"]), generator=gen, device="cuda").mul_(2.0)
    return out


def _masks(case, seed):
    """Masks as grammars give them: most rows allow few tokens, the others (inside a string) most of them."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = random.Random(seed)
    words = _mask_words(case)
    shares = torch.tensor([rng.uniform(0.0005, 0.03) if rng.random() < 0.6 else rng.uniform(0.4, 0.9) for _ in range(case["batch"])], device="cuda")
    bits = torch.rand((case["batch"], words * 32), generator=gen, device="cuda") < shares[:, None]
    bits[:, case["vocab"]:] = False
    weights = (1 << torch.arange(32, dtype=torch.int64, device="cuda"))
    return (bits.view(case["batch"], words, 32) * weights).sum(dim=2).to(torch.int32)


def _advanced(case, prefix, **options):
    """A state whose rows have taken their texts so far."""
    g = _compiled(case["grammar"], case["vocab"])[0]
    state = fmt.State(g, case["batch"], **options)
    status = torch.zeros(case["batch"], dtype=torch.int32, device="cuda")
    on_gpu = torch.from_numpy(prefix).cuda()
    for p in range(on_gpu.shape[0]):
        state.advance(on_gpu[p], status)
    return state


def prepare(case, seed):
    kind, batch = case["kind"], case["batch"]
    rng = random.Random("%s %d" % (json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True), seed))
    s = {"kind": kind, "batch": batch, "vocab": case["vocab"], "stream": torch.cuda.current_stream().cuda_stream}
    if "logits" in case:
        s["dtype"] = fmt.BF16 if case["logits"] == "bf16" else fmt.FP32
        s["logits"] = _logits(case, seed, case.get("steps", 1))
    if kind == "apply":
        s["masks"] = [_masks(case, seed + 1000003 * k) for k in range(case["steps"])]
        return s
    prefix, tokens, resets = _streams(case, rng)
    if kind in ("decode", "steady", "prefill"):
        s["state"] = fmt.State(_compiled(case["grammar"], case["vocab"])[0], batch)
        s["prefix"] = list(torch.from_numpy(prefix).cuda()) if case["context"] else []
        s["tokens"] = list(torch.from_numpy(tokens).cuda())
        s["resets"] = [torch.tensor(r, dtype=torch.int32, device="cuda") if r else None for r in resets]
        s["status"] = torch.zeros((len(s["prefix"]) + len(s["tokens"]), batch), dtype=torch.int32, device="cuda")
    if kind in ("prefill", "fill", "noalloc"):
        s["mask"] = torch.zeros((batch, _mask_words(case)), dtype=torch.int32, device="cuda")
    if kind == "fill":
        s["state"] = _advanced(case, prefix, cache=False)
    if kind == "forced":
        s["state"] = _advanced(case, prefix)
        s["bytes"] = torch.zeros((batch, 32), dtype=torch.uint8, device="cuda")
        s["length"] = torch.zeros(batch, dtype=torch.int32, device="cuda")
    if kind == "noalloc":
        state = _advanced(case, prefix)
        charts = [state.chart_words(b) for b in range(batch)]
        s["grammar"] = _compiled(case["grammar"], case["vocab"])[0]
        s["offsets"] = np.concatenate([[0], np.cumsum([len(c) for c in charts])]).astype(np.uint64)
        s["charts"] = torch.from_numpy(np.concatenate(charts).view(np.int32)).cuda()
        s["status"] = torch.zeros(batch, dtype=torch.int32, device="cuda")
    return s


def run(s):
    kind, stream = s["kind"], s["stream"]
    if kind == "apply":
        for mask, logits in zip(s["masks"], s["logits"]):
            fmt.apply_mask(mask, logits, s["dtype"], s["batch"], s["vocab"], stream=stream)
        return s["logits"]
    if kind == "fill":
        s["state"].fill_mask(s["mask"], stream=stream)
        return s["mask"]
    if kind == "forced":
        s["state"].forced_bytes(s["bytes"], s["length"], stream=stream)
        return {"bytes": s["bytes"], "length": s["length"]}
    if kind == "noalloc":
        fmt.fill_mask_noalloc(s["grammar"], s["charts"], s["offsets"], s["mask"], s["status"], stream=stream)
        return {"mask": s["mask"], "status": s["status"]}
    state, status = s["state"], s["status"]
    if kind != "steady":
        state.cache_clear(stream=stream)
    state.reset(stream=stream)
    at = 0
    for tokens in s["prefix"]:
        state.advance(tokens, status[at], stream=stream)
        at += 1
    if kind == "prefill":
        state.fill_mask(s["mask"], stream=stream)
        return {"status": status, "mask": s["mask"]}
    for i, tokens in enumerate(s["tokens"]):
        if s["resets"][i] is not None:
            state.reset(s["resets"][i], stream=stream)
        state.advance(tokens, status[at], stream=stream)
        state.fill_and_apply(s["logits"][i], s["dtype"], stream=stream)
        at += 1
    return {"status": status, "logits": s["logits"]}


def work(case):
    """The bytes of one pass: per decoding step or fill the vocabulary once (about 8 bytes a token: its bytes, where it
    begins, where it ends in the trie) and the mask words written, the logits read and written where they are masked,
    and a small chart per row read and written wherever rows advance.  There is no arithmetic to count."""
    kind, batch, vocab = case["kind"], case["batch"], case["vocab"]
    chart = 512 * batch
    mask = 4 * _mask_words(case) * batch
    logits = 2 * (2 if case.get("logits") == "bf16" else 4) * batch * vocab
    if kind == "apply":
        return {"bytes": case["steps"] * (mask + logits), "flops": 0}
    if kind == "forced":
        return {"bytes": chart + 36 * batch, "flops": 0}
    if kind in ("fill", "noalloc"):
        return {"bytes": 8 * vocab + chart + mask, "flops": 0}
    if kind == "prefill":
        return {"bytes": case["context"] * 2 * chart + 8 * vocab + mask, "flops": 0}
    return {"bytes": case["context"] * 2 * chart + case["steps"] * (8 * vocab + 2 * chart + mask + logits), "flops": 0}


def tolerance(case):
    """Masks are sets of tokens and masked logits keep their bits: there is nothing to round."""
    return "exact"
