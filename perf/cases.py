"""Measured cases: the calls that a grammar-constrained decoding loop makes.

Each case is one pass through the public binding (``paper_2607_11951_gb300.grid``)
as a serving program makes it: it keeps the compiled grammar, the vocabulary and
the specialized tables (``Spec``) for its lifetime, has parser configurations
for a batch of requests in hand, and calls the library once per decoding step
(or once per request, for the prompt and for a fresh schema).

Kinds of pass (``case["kind"]``):

  step        one decoding step: ``grid_advance_masks`` feeds each row's sampled
              token, computes the next masks and fills the logits (fp32, bf16 or
              none), optionally through a mask cache
  masks       ``grid_masks`` of a batch of configurations (masks without logits)
  prefill     a request's start: ``grid_configs_reset``, ``grid_advance`` over
              every token of the prompt, ``grid_masks`` for the first step
  specialize  a fresh schema: ``grid_specialize``, ``grid_configs_create`` and
              the masks of the empty output, from a compiled grammar
  apply       ``grid_apply_mask``: the -inf fill of logits by finished masks
  span        jump-forward: the sampled token fed (``grid_advance``), then
              ``grid_forced_span``
  reserve     ``grid_reserve``: the cheapest completion of every row, with the
              budget trigger
  audit       a decoding step with the audit chain on: ``grid_audit_append`` of
              the step's record, then ``grid_advance_masks``

Inputs are synthetic: the repository's SQL and expression grammars, snake_case
schemas, BPE-like vocabularies of a fixed random pool, and configurations that
random statements leave when they are cut after a number of tokens.
"""
import functools
import math
import os
import random

import numpy as np
import torch

from paper_2607_11951_gb300 import grid as G

MAX_V = 151_936  # the largest vocabulary of the repository's configurations
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


# ---------------------------------------------------------------------------
# cases
def listed():
    return [
        # the smallest call: one request, a six-terminal grammar, 512 tokens;
        # launches and dependent loads are all of it
        dict(name="step_expr_b1", kind="step", grammar="expr", role="all", tables=0, cols=0, V=512, B=1, n=30, depth=4,
             dtype="f32", cache=False),
        # one interactive request against a 152k vocabulary, bf16 logits
        dict(name="step_sql_b1_bf16", kind="step", grammar="sql", role="select", tables=200, cols=30, V=151_936, B=1,
             n=400, depth=2, dtype="bf16", cache=False),
        # the benchmark's step: a batch of 32 requests, fp32 logits
        dict(name="step_sql_b32_f32", kind="step", grammar="sql", role="select", tables=200, cols=30, V=151_936, B=32,
             n=2000, depth=2, dtype="f32", cache=False),
        # the largest serving batch, a catalog of 50,000 identifiers, bf16 logits
        dict(name="step_sql_b256_bf16", kind="step", grammar="sql", role="select", tables=1000, cols=50, V=151_936,
             B=256, n=2000, depth=2, dtype="bf16", cache=False),
        # a ragged batch and a vocabulary with one added token: rows of fp32
        # logits that start off the sector boundaries
        dict(name="step_sql_b27_ragged", kind="step", grammar="sql", role="admin", tables=20, cols=10, V=32_001, B=27,
             n=200, depth=2, dtype="f32", cache=False),
        # long generations of deeply nested statements, masks only
        dict(name="masks_deep_b32", kind="masks", grammar="sql", role="admin", tables=200, cols=30, V=128_256, B=32,
             n=16_000, depth=64, cache=False),
        # prompts (or outputs being resumed) fed in one call
        dict(name="prefill_b32", kind="prefill", grammar="sql", role="admin", tables=200, cols=30, V=128_256, B=32,
             n=2000, depth=8),
        # a schema seen for the first time, up to the first mask
        dict(name="specialize_cold", kind="specialize", grammar="sql", role="select", tables=1000, cols=50, V=151_936,
             B=8),
        # masks made elsewhere (or earlier) applied to a large batch's logits
        dict(name="apply_b256_bf16", kind="apply", V=151_936, B=256, dtype="bf16"),
        # jump-forward after each sampled token
        dict(name="span_b32", kind="span", grammar="sql", role="admin", tables=20, cols=10, V=32_000, B=32, n=200,
             depth=2, max_span=8),
        # the termination reserve, asked for every row of the batch
        dict(name="reserve_b32", kind="reserve", grammar="sql", role="select", tables=200, cols=30, V=151_936, B=32,
             n=2000, depth=8, cap=256),
        # the audited decoding step
        dict(name="audit_b32", kind="audit", grammar="sql", role="select", tables=200, cols=30, V=151_936, B=32, n=500,
             depth=2),
    ]


def _spread(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["masks", "masks", "prefill", "specialize", "apply", "span", "reserve", "audit"])
    B = _spread(rng, 1, 256 if kind in ("step", "masks", "apply") else 32)
    V = _spread(rng, 2_000, MAX_V)
    if kind == "apply":
        return dict(kind=kind, V=V, B=B, dtype=rng.choice(["f32", "bf16"]) if B <= 128 else "bf16")
    tables = _spread(rng, 5, 1000)
    case = dict(kind=kind, grammar="sql", role=rng.choice(["select", "admin"]), tables=tables, cols=rng.randint(5, 50),
                V=V, B=B)
    if kind == "specialize":
        case["B"] = _spread(rng, 1, 8)
        return case
    if kind in ("step", "masks") and rng.random() < 0.1:
        case.update(grammar="expr", role="all", tables=0, cols=0, V=_spread(rng, 128, 2_000))
    case["n"] = _spread(rng, 20, 2000)
    case["depth"] = rng.randint(0, 64 if kind == "masks" else 8)
    if kind in ("step", "masks"):
        case["cache"] = rng.random() < 0.2
    if kind == "step":
        case["dtype"] = "bf16" if B > 128 else rng.choice(["f32", "bf16", "none"])
    if kind == "span":
        # a vocabulary of whole blank-led words leaves some positions one token
        case["words"] = rng.random() < 0.5
        case["V"] = len(vocabulary("sql", 0, (tables, case["cols"]))[0]) if case["words"] else _spread(rng, 2_000, 32_000)
        case["max_span"] = rng.randint(1, 8)
    if kind == "reserve":
        case["cap"] = _spread(rng, 64, 256)
    return case


# ---------------------------------------------------------------------------
# grammar, schema, vocabulary
@functools.lru_cache(maxsize=None)
def grammar_text(name):
    with open(os.path.join("workloads", "grammars", name + ".grid")) as f:
        return f.read()


ROLES = {"all": None, "admin": ["dml"], "select": []}
KEYWORDS = "select distinct from where inner left join on group by having order asc desc limit and or not in exists " \
           "is null like true false count sum avg min max insert into values update set delete".split()
ONSETS = "b c d f g h j k l m n p r s t v w z ch sh th br cr dr gr pr st tr pl kl sp qu".split()
VOWELS = "a e i o u ai ea io ou ee oa".split()
CODAS = ["", "", "", "n", "r", "s", "t", "l", "m", "x", "nd", "st", "rk", "ng"]
PUNCT = "(),;.*=<>!+-/%'"
EXPR_ALPHABET = "abcdefghijklmnopqrstuvwxyz0123456789+*() "


@functools.lru_cache(maxsize=None)
def syllables():
    rng = random.Random(7)
    out = {}
    while len(out) < 320:
        out[rng.choice(ONSETS) + rng.choice(VOWELS) + rng.choice(CODAS)] = None
    return list(out)


def schema(tables, cols, seed):
    """Distinct snake_case names: (table names, column names), no name in both.
    Catalogs repeat column names over their tables, very large ones less."""
    rng = random.Random(seed)
    syl = syllables()
    seen = set(KEYWORDS)

    def names(count, most):
        out = []
        while len(out) < count:
            name = "_".join(rng.choice(syl) + (rng.choice(syl) if rng.random() < 0.3 else "")
                            for _ in range(rng.randint(1, most)))
            if rng.random() < 0.05:
                name += str(rng.randint(1, 9))
            if name not in seen:
                seen.add(name)
                out.append(name)
        return out

    words = tables * cols if tables * cols >= 40_000 else max(cols, tables * cols // 2)
    return names(tables, 2), names(words, 3)


@functools.lru_cache(maxsize=None)
def token_pool():
    """Distinct byte strings of 2 to 16 bytes, P(length) ~ 1 / length, in
    random order: identifier pieces, keyword fragments, digits, punctuation,
    blanks, unrelated text and windows over several lexemes."""
    rng = random.Random(11)
    syl = syllables()
    lengths = list(range(2, 17))
    weights = [x ** -1.1 for x in lengths]
    kinds = ["syl", "junk", "kw", "digit", "punct", "ws", "multi"]
    shares = [0.46, 0.2, 0.1, 0.06, 0.09, 0.03, 0.09]
    tables, cols = schema(50, 12, 12)
    text = "".join(Sentences(rng, tables, cols).statement(4, 0, "select") for _ in range(1500))
    printable = "".join(map(chr, range(33, 127)))
    out, seen = [], set()
    while len(out) < MAX_V:
        for kind, L in zip(rng.choices(kinds, shares, k=4096), rng.choices(lengths, weights, k=4096)):
            lead = " " if rng.random() < 0.45 else ""
            if kind == "syl":
                s = lead
                while len(s) < L:
                    s += rng.choice(syl) + ("_" if rng.random() < 0.15 else "")
            elif kind == "kw":
                s = lead + rng.choice(KEYWORDS)
                if rng.random() < 0.5:
                    s = s[rng.randrange(len(s)):]
                while len(s) < L:
                    s += " " + rng.choice(KEYWORDS)
            elif kind == "digit":
                s = lead + "".join(rng.choices("0123456789", k=L))
            elif kind == "punct":
                s = "".join(rng.choices(PUNCT + "    ", k=L))
            elif kind == "ws":
                s = " " * L if rng.random() < 0.5 else "\n" + " " * (L - 1)
            elif kind == "junk":
                s = "".join(rng.choices(printable, k=L))
                if rng.random() < 0.3:
                    s = "".join(chr(128 + ord(x)) for x in s)
            else:
                a = rng.randrange(len(text) - L)
                s = text[a:a + L]
            b = s[:L].encode("latin-1")
            if b not in seen:
                seen.add(b)
                out.append(b)
    return out[:MAX_V]


@functools.lru_cache(maxsize=None)
def vocabulary(grammar, V, words=None):
    """(tokens, eos, specials): every single byte of the alphabet, the rest of
    the pool's first strings, a few aliases, specials and EOS last.  `words`: a
    schema (tables, cols) whose names, the keywords and the punctuation are the
    only spellings, each with a leading blank."""
    if grammar == "expr":
        rng = random.Random(V)
        toks = list(dict.fromkeys(EXPR_ALPHABET))
        seen = set(toks)
        while len(toks) < V - 1:
            s = "".join(rng.choices(EXPR_ALPHABET, k=rng.randint(2, 4)))
            if s not in seen:
                seen.add(s)
                toks.append(s)
        return [t.encode() for t in toks] + [b"<eos>"], V - 1, []
    if words:
        tables, cols = schema(*words, 1)
        toks = [" " + w for w in KEYWORDS + tables + cols]
        toks += [" " + x for x in PUNCT + "0123456789"] + list("(),;.0123456789") + [" <=", " >=", " <>", " 'a'"]
        toks = [t.encode() for t in toks]
        return toks + [b"<eos>"], len(toks), []
    toks = [bytes([b]) for b in range(256)]
    aliases = V // 1000
    toks += token_pool()[:V - len(toks) - 3 - aliases]
    toks += toks[300:300 + aliases]
    specials = [len(toks), len(toks) + 1]
    return toks + [b"<|special_0|>", b"<|special_1|>", b"<|endoftext|>"], V - 1, specials


class Sentences:
    """Random statements as lists of text segments; each segment is a run of
    whole lexemes that starts with a blank."""

    def __init__(self, rng, tables, cols):
        self.rng, self.tables, self.cols = rng, tables, cols

    def column(self):
        c = self.rng.choice(self.cols)
        return c if self.rng.random() < 0.8 else self.rng.choice(self.tables) + "." + c

    def value(self):
        r = self.rng.random()
        if r < 0.5:
            return self.column()
        if r < 0.75:
            return str(self.rng.randrange(100_000)) if r < 0.7 else "%.2f" % (self.rng.random() * 100)
        if r < 0.85:
            return "'" + "".join(self.rng.choices("abcdefgh ijk", k=self.rng.randrange(8))) + "'"
        if r < 0.95:
            f = self.rng.choice(["count", "sum", "avg", "min", "max"])
            return f + self.rng.choice(["(", " ( "]) + self.column() + ")" if f != "count" else "count(*)"
        return self.rng.choice(["true", "false", "null"])

    def arith(self):
        out = self.value()
        while self.rng.random() < 0.25:
            out += " " + self.rng.choice("+-*/%") + " " + self.value()
        return out if self.rng.random() > 0.08 else "(" + out + ")"

    def pred(self):
        r = self.rng.random()
        a = " " + self.arith()
        if r < 0.1:
            return a + self.rng.choice([" is null", " is not null"])
        if r < 0.15:
            return a + " like 'x y'"
        if r < 0.22:
            return a + " in (select " + self.column() + " from " + self.rng.choice(self.tables) + ")"
        if r < 0.27:
            return " not" + a + " = " + self.value()
        return a + " " + self.rng.choice(["=", "<>", "!=", "<", ">", "<=", ">="]) + " " + self.arith()

    def head(self, role):
        t = self.rng.choice(self.tables)
        r = self.rng.random()
        if role == "admin" and r < 0.15:
            return " update " + t + " set " + self.rng.choice(self.cols) + " = " + self.arith() + " where"
        if role == "admin" and r < 0.3:
            return " delete from " + t + " where"
        out = " select " + self.rng.choice(["", "", "distinct "]) + (self.arith() if r < 0.9 else "*")
        out += " from " + t
        if self.rng.random() < 0.3:
            out += " inner join " + self.rng.choice(self.tables) + " on " + self.column() + " = " + self.column()
        return out + " where"

    def segments(self, depth, role):
        """The segments of an endless statement: `depth` nested parentheses or
        subqueries, then a chain of predicates, select items or order keys."""
        chain = self.rng.choice(["where"] * 4 + ["items", "order"]) if depth == 0 else "where"
        if chain == "items":
            yield " select"
            while True:
                yield " " + self.arith() + ","
        if chain == "order":
            yield " select * from " + self.rng.choice(self.tables) + " order by"
            while True:
                yield " " + self.arith() + self.rng.choice([",", " asc,", " desc,"])
        yield self.head(role)
        for _ in range(depth):
            yield " (" if self.rng.random() < 0.75 else \
                " " + self.column() + " in (select " + self.column() + " from " + self.rng.choice(self.tables) + " where"
        some = [self.pred() for _ in range(40)]  # a long chain's predicates recur
        while True:
            yield self.rng.choice(some)
            yield self.rng.choice([" and", " and", " or"])

    def statement(self, preds, depth, role):
        out = self.head(role)
        for i in range(preds):
            out += (" and" if i else "") + self.pred()
        return out + ";"


def expr_segments(rng, depth):
    for _ in range(depth):
        yield "("
    while True:
        yield (rng.choice(["ab", "x", "count", "zeta"]) if rng.random() < 0.5 else str(rng.randrange(1000)))
        yield rng.choice(["+", "*", " + ", " * "])


class Tokenizer:
    """Greedy longest match over the vocabulary's spellings, segment by segment."""

    def __init__(self, tokens, eos, specials):
        skip = set(specials) | {eos}
        self.ids = {}
        for i, t in enumerate(tokens):
            if i not in skip:
                self.ids.setdefault(t, i)
        self.longest = max(map(len, self.ids))

        self.known = {}

    def encode(self, text):
        out = self.known.get(text)
        if out is None:
            data = text.encode()
            out, i = [], 0
            while i < len(data):
                L = next(L for L in range(self.longest, 0, -1) if data[i:i + L] in self.ids)
                out.append(self.ids[data[i:i + L]])
                i += len(data[i:i + L])
            self.known[text] = out
        return out


# ---------------------------------------------------------------------------
# handles that a program keeps for its lifetime, made once per (grammar,
# schema, vocabulary)
@functools.lru_cache(maxsize=None)
def vocab_handle(grammar, V, words):
    tokens, eos, specials = vocabulary(grammar, V, words)
    return G.Vocab(tokens, eos, specials), Tokenizer(tokens, eos, specials)


def compile_grammar(case, seed):
    if case["grammar"] == "expr":
        return G.Grammar(grammar_text("expr")), ([], [])
    tables, cols = schema(case["tables"], case["cols"], seed)
    lexicons = {"TABLE_NAME": tables, "COLUMN_NAME": cols}
    return G.Grammar(grammar_text("sql"), ROLES[case["role"]], lexicons, max_depth=4096), (tables, cols)


@functools.lru_cache(maxsize=None)
def kept(grammar, role, tables, cols, V, words):
    g, names = compile_grammar(dict(grammar=grammar, role=role, tables=tables, cols=cols), 1)
    vocab, tokenizer = vocab_handle(grammar, V, (tables, cols) if words else None)
    return G.Spec(g, vocab), tokenizer, names


# ---------------------------------------------------------------------------
# inputs
def segments(case, names, rng):
    """An endless text of the case's language, piece by piece."""
    if case["grammar"] == "expr":
        return expr_segments(rng, case["depth"])
    return Sentences(rng, *names).segments(case["depth"], case["role"])


def prompts(case, names, tokenizer, seed, whole):
    """Token ids [B, n] of random prefixes (-1 after the last) and the token
    that follows each.  Lengths are spread over [n / 40, n], all n if `whole`."""
    rng = random.Random(seed)
    B, n = case["B"], case["n"]
    fed = np.full((B, n), -1, dtype=np.int32)
    follow = np.zeros(B, dtype=np.int32)
    for b in range(B):
        want = n if whole else max(1, round(n * rng.uniform(1 / 40, 1)))
        ids = []
        for seg in segments(case, names, rng):
            ids += tokenizer.encode(seg)
            if len(ids) > want:
                break
        fed[b, :want] = ids[:want]
        follow[b] = ids[want]
    return fed, follow


def word_prompts(case, names, tokenizer, seed):
    """The same in whole words: statements cut after a random word."""
    rng = random.Random(seed)
    B, n = case["B"], case["n"]
    tables, cols = names
    fed = np.full((B, n), -1, dtype=np.int32)
    follow = np.zeros(B, dtype=np.int32)
    for b in range(B):
        words = ["select", rng.choice(cols), "from", rng.choice(tables)]
        if rng.random() < 0.5:
            words += ["left", "join", rng.choice(tables), "on", rng.choice(cols), "=", str(rng.randrange(10))]
        words += ["where", rng.choice(cols), "is", "not", "null"]
        while len(words) < n and rng.random() < 0.9:
            words += ["and", rng.choice(cols), "=", str(rng.randrange(10))]
        words += ["group", "by", rng.choice(cols), "order", "by", rng.choice(cols), "limit", "5"]
        ids = [tokenizer.encode(" " + w)[0] for w in words]
        want = rng.randint(1, min(n, len(ids) - 1))
        fed[b, :want] = ids[:want]
        follow[b] = ids[want]
    return fed, follow


def fill_logits(B, V, dtype, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn((B, V), generator=gen, device="cuda") * 3).to(DTYPES[dtype])


def prepare(case, seed):
    dev = torch.device("cuda")
    kind, B, V = case["kind"], case["B"], case["V"]
    state = dict(kind=kind)
    if kind == "apply":
        # masks admit a few to some twenty in a hundred tokens, as grammar masks do
        rng = np.random.default_rng(seed)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        share = torch.from_numpy(rng.uniform(0.01, 0.2, size=(B, 1)).astype(np.float32)).to(dev)
        W = (V + 31) // 32
        words = torch.zeros((B, W), dtype=torch.int64, device=dev)
        for j in range(32):
            words |= (torch.rand((B, W), generator=gen, device=dev) < share).to(torch.int64) << j
        state["mask"] = words.to(torch.int32)
        state["logits"] = fill_logits(B, V, case["dtype"], seed + 1)
        return state
    if kind == "specialize":
        state["grammar"], _ = compile_grammar(case, 1000 + seed)
        state["vocab"] = vocab_handle(case["grammar"], V, None)[0]
        state["B"] = B
        W = (V + 31) // 32
        state["mask"] = torch.zeros((B, W), dtype=torch.int32, device=dev)
        state["status"] = torch.zeros(B, dtype=torch.int32, device=dev)
        return state
    words = bool(case.get("words"))
    spec, tokenizer, names = kept(case["grammar"], case["role"], case["tables"], case["cols"], V, words)
    if words:
        fed, follow = word_prompts(case, names, tokenizer, seed)
    else:
        fed, follow = prompts(case, names, tokenizer, seed, kind in ("prefill", "masks"))
    fed = torch.from_numpy(fed).to(dev)
    state.update(spec=spec, tokens=torch.from_numpy(follow).to(dev), cin=G.Configs(spec, B),
                 mask=torch.zeros((B, spec.W), dtype=torch.int32, device=dev),
                 status=torch.zeros(B, dtype=torch.int32, device=dev))
    if kind == "prefill":
        state["fed"] = fed
        return state
    if kind == "audit":
        G.grid_configs_enable_audit(spec.h, state["cin"].h)
    G.grid_advance(spec, state["cin"], state["cin"], fed, state["status"])
    if int(state["status"].abs().max()) != G.GRID_ST_OK:
        raise RuntimeError("a prompt was refused: %s" % state["status"].tolist())
    if kind != "masks":
        state["cout"] = G.Configs(spec, B)
    if case.get("cache"):
        state["cache"] = G.Cache(spec, 1024)
    if kind == "step" and case["dtype"] != "none":
        state["logits"] = fill_logits(B, spec.V, case["dtype"], seed + 1)
    elif kind == "span":
        state["max_span"] = case["max_span"]
        state["span"] = torch.zeros((B, case["max_span"]), dtype=torch.int32, device=dev)
        state["span_len"] = torch.zeros(B, dtype=torch.int32, device=dev)
    elif kind == "reserve":
        rng = np.random.default_rng(seed)
        state["budget"] = torch.from_numpy(rng.integers(1, 400, size=B).astype(np.int32)).to(dev)
        state["cost"] = torch.zeros(B, dtype=torch.int32, device=dev)
        state["fire"] = torch.zeros(B, dtype=torch.int32, device=dev)
        state["rest"] = torch.zeros((B, case["cap"]), dtype=torch.int32, device=dev)
    elif kind == "audit":
        G.grid_configs_enable_audit(spec.h, state["cout"].h)
        state["next_mask"] = torch.zeros_like(state["mask"])
        state["records"] = torch.zeros((B, 80), dtype=torch.uint8, device=dev)
        G.grid_masks(spec, state["cin"], state["mask"], state["status"])
    torch.cuda.synchronize()
    return state


def run(state):
    kind = state["kind"]
    if kind == "step":
        G.grid_advance_masks(state["spec"], state["cin"], state["cout"], state["tokens"], state["mask"],
                             state["status"], state.get("logits"), cache=state.get("cache"))
        out = dict(mask=state["mask"], status=state["status"])
        if "logits" in state:
            out["logits"] = state["logits"]
        return out
    if kind == "masks":
        if "cache" in state:
            G.grid_masks_cached(state["spec"], state["cin"], state["cache"], state["mask"], state["status"])
        else:
            G.grid_masks(state["spec"], state["cin"], state["mask"], state["status"])
        return dict(mask=state["mask"], status=state["status"])
    if kind == "prefill":
        spec, cfg = state["spec"], state["cin"]
        cfg.reset()
        G.grid_advance(spec, cfg, cfg, state["fed"], state["status"])
        fed = state["status"].clone()
        G.grid_masks(spec, cfg, state["mask"], state["status"])
        return dict(fed=fed, mask=state["mask"], status=state["status"])
    if kind == "specialize":
        spec = G.Spec(state["grammar"], state["vocab"])
        cfg = G.Configs(spec, state["B"])
        G.grid_masks(spec, cfg, state["mask"], state["status"])
        state["spec"], state["cfg"] = spec, cfg
        return dict(mask=state["mask"], status=state["status"])
    if kind == "apply":
        G.grid_apply_mask(state["mask"], state["logits"])
        return state["logits"]
    if kind == "span":
        spec, cfg = state["spec"], state["cout"]
        G.grid_advance(spec, state["cin"], cfg, state["tokens"], state["status"])
        G.grid_forced_span(spec.h, cfg.h, state["max_span"], state["mask"], state["span"], state["span_len"],
                           state["status"])
        return dict(mask=state["mask"], span=state["span"], length=state["span_len"], status=state["status"])
    if kind == "reserve":
        G.grid_reserve(state["spec"].h, state["cin"].h, state["cost"], state["rest"], state["status"],
                       budget=state["budget"], safety=8, fire=state["fire"])
        return dict(cost=state["cost"], tokens=state["rest"], status=state["status"], fire=state["fire"])
    spec = state["spec"]
    G.grid_audit_append(spec.h, state["cin"].h, state["mask"], state["tokens"], 0, state["records"])
    G.grid_advance_masks(spec, state["cin"], state["cout"], state["tokens"], state["next_mask"], state["status"])
    return dict(records=state["records"], mask=state["next_mask"], status=state["status"])


# ---------------------------------------------------------------------------
def work(case):
    """Bytes of one pass: every input read once, every output written once."""
    kind, B, V = case["kind"], case["B"], case["V"]
    mask = 4 * B * ((V + 31) // 32)
    classes = 2 * V  # the class code of every token in the start state's table
    if kind == "apply":
        return dict(bytes=mask + B * V * (4 if case["dtype"] == "f32" else 2), flops=0)
    if kind == "specialize":
        # the spellings read, one class code written per token and table
        return dict(bytes=8 * V + 25 * classes + mask, flops=0)
    if kind == "step":
        return dict(bytes=classes + mask + B * V * {"f32": 4, "bf16": 2, "none": 0}[case["dtype"]], flops=0)
    if kind == "masks":
        return dict(bytes=classes + mask, flops=0)
    if kind == "prefill":
        # the tokens, their spellings' places and bytes
        return dict(bytes=classes + mask + 20 * B * case["n"], flops=0)
    if kind == "span":
        return dict(bytes=classes + mask + 4 * B * (case["max_span"] + 2), flops=0)
    if kind == "reserve":
        return dict(bytes=B * (4 * case["cap"] + 2 * 64 + 32), flops=0)
    return dict(bytes=classes + 2 * mask + 80 * B, flops=0)


def tolerance(case):
    """Masks, statuses, tokens and records are whole numbers; logits are either
    left as they are or become -inf."""
    return "exact"


def exact(case, seed):
    """The filled logits of the apply cases; the other outputs are whole
    numbers, and the logits of a step are its masks' work."""
    if case["kind"] != "apply":
        return None
    state = prepare(case, seed)
    bits = (state["mask"].unsqueeze(2) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1
    bits = bits.reshape(case["B"], -1)[:, :case["V"]]
    return torch.where(bits != 0, state["logits"].double(), torch.full((), -math.inf, dtype=torch.float64, device="cuda"))
