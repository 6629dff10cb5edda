"""Feeding several tokens in one call, 32 lexed at a time: the status and the
configuration that every row is left in, against the oracle's token-by-token
advance and against the same tokens fed one per call.  Batch edges, gaps (-1),
refused tokens, EOS inside and at the end, tokens that end several lexemes,
lexemes of more candidates than a list holds, stacks beyond the
shared-memory window, and chains over empty nonterminals."""
import numpy as np
import pytest

from workloads import configs, grammar_text

pytestmark = pytest.mark.gpu

MANY = "%token A0 /a/\n" + "".join("%%token A%d /[a-%s]/\n" % (i, "bcdefghijk"[i - 1]) for i in range(1, 10)) + """
%token SEMI ";"
%ignore WS /[ ]+/
%start s
s -> list SEMI
list -> list item
list -> item
item -> A9 opt opt2 A9
opt -> %empty
opt -> A0 SEMI
opt2 -> %empty
opt2 -> A1 SEMI SEMI
"""


def _world(name):
    """(grammar, role, lexicons, tokens, eos, specials, good prefixes)"""
    if name == "sql":
        wl = configs.sql_admin(B=8)
        return wl["grammar"], wl["role"], wl["lexicons"], wl["tokens"], wl["eos"], wl["specials"], wl["prefixes"]
    if name == "expr":
        wl = configs.tiny_expr(B=8)
        toks = list(wl["tokens"][:-1]) + [b"((((((((", b"a+b*c+d*e+f*g", b"x ", wl["tokens"][-1]]
        eos = len(toks) - 1
        lp, many = eos - 3, eos - 2
        x = toks.index(b"a")
        plus = toks.index(b"+")
        good = [list(p) for p in wl["prefixes"]]
        good += [[lp] * 5 + [x], [many, plus, many], [lp] * 160 + [x, plus, x, toks.index(b")")]]
        return wl["grammar"], wl["role"], wl["lexicons"], toks, eos, [], good
    toks = [bytes([c]) for c in b"abcdefghij; "] + [b"jj;", b"aj", b" j", b"a;"] + [b"<eos>"]
    t = {x: i for i, x in enumerate(toks)}
    good = [[t[b"j"], t[b" "], t[b"j"], t[b" j"], t[b" j"], t[b";"], t[b" "]] * 1,
            [t[b"j"], t[b" "], t[b"a;"], t[b" "], t[b"j"]] * 1]
    return MANY, None, {}, toks, len(toks) - 1, [], good


def _oracle_feed(og, toks, tokens, eos, specials):
    """(status, tokens taken in) of a row that starts empty."""
    from paper_2607_11951_gb300 import grid as G
    cfg, done = og.start_config(), 0
    for k, tok in enumerate(toks):
        if tok < 0:
            continue
        if cfg.complete:
            return G.GRID_ST_COMPLETE, toks[:k]
        nxt = og.advance(cfg, tok, tokens, eos, specials) if 0 <= tok < len(tokens) else None
        if nxt is None:
            return G.GRID_ST_TOKEN_NOT_ALLOWED, toks[:k]
        cfg, done = nxt, k + 1
    return G.GRID_ST_OK, toks


@pytest.mark.parametrize("name", ["sql", "expr", "many"])
def test_feed_matches_token_by_token(name):
    import torch
    from oracle import compile_grammar
    from paper_2607_11951_gb300 import grid as G
    grammar, role, lexicons, tokens, eos, specials, good = _world(name)
    if name == "expr":
        assert grammar == grammar_text("expr")
    og = compile_grammar(grammar, role, lexicons)
    rng = np.random.default_rng(3)
    rows = []
    for p in good:
        p = [int(x) for x in p]
        rows.append(p)
        for cut in (31, 32, 33, 64, 65):
            if cut < len(p):
                rows.append(p[:cut])
        at = int(rng.integers(0, len(p) + 1))
        rows.append(p[:at] + [int(rng.integers(0, len(tokens)))] + p[at:])       # most often refused there
        rows.append(p[:at] + [eos] + p[at:])                                     # EOS, rarely a sentence
        rows.append([x for t in p for x in (-1, t)])                             # gaps
        rows.append(p[:at] + [-1, len(tokens)] + p[at:])                         # no such token
        if specials:
            rows.append(p[:at] + [int(specials[0])] + p[at:])
    if name == "many":
        t = {x: i for i, x in enumerate(tokens)}
        rows += [good[0][:-1] + [eos], good[0][:-1] + [eos, t[b"j"]], [t[b"aj"]], [t[b"jj;"]]]
    B, n = len(rows), max(map(len, rows))
    fed = np.full((B, n), -1, np.int32)
    for b, r in enumerate(rows):
        fed[b, :len(r)] = r
    spec = G.Spec(G.Grammar(grammar, role, lexicons), G.Vocab(tokens, eos, specials))
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    cfg, other, one = G.Configs(spec, B), G.Configs(spec, B), G.Configs(spec, B)
    d = torch.from_numpy(fed).cuda()
    # in one call out of place, and inside a mask step
    G.grid_advance(spec, cfg, other, d, status)
    st = status.cpu().numpy().copy()
    mask = torch.zeros((B, (len(tokens) + 31) // 32), dtype=torch.int32, device="cuda")
    G.grid_advance_masks(spec, cfg, cfg, d, mask, status)
    st2 = status.cpu().numpy()
    # the tokens that the oracle takes in, one per call
    want = [_oracle_feed(og, r, tokens, eos, specials) for r in rows]
    took = np.full((B, n), -1, np.int32)
    for b, (_, r) in enumerate(want):
        took[b, :len(r)] = r
    for k in range(n):
        G.grid_advance(spec, one, one, torch.from_numpy(np.ascontiguousarray(took[:, k:k + 1])).cuda(), status)
        assert not status.any()
    for b in range(B):
        assert st[b] == want[b][0], (b, rows[b], st[b], want[b][0])
        if want[b][0] != G.GRID_ST_OK:
            assert st2[b] == want[b][0]
        ref = one.export(b)
        assert other.export(b) == ref and cfg.export(b) == ref, (b, rows[b])


@pytest.mark.parametrize("n", [1, 2, 8, 9, 40])
@pytest.mark.parametrize("name", ["sql", "expr", "many"])
def test_large_batch_feeds_as_a_small_one(name, n):
    """Rows whose blocks are not on the device at once: statuses,
    configurations and node hashes are those of the same rows in a small
    batch (fed as the test above checks against the oracle)."""
    import torch
    from paper_2607_11951_gb300 import grid as G
    grammar, role, lexicons, tokens, eos, specials, good = _world(name)
    rng = np.random.default_rng(n)
    rows = []
    for p in good * 8:
        p = [int(x) for x in p]
        at = int(rng.integers(0, len(p) + 1))
        rows.append((p[:at], (p[at:] + [eos] + p[:1])[:n]))
        rows.append((p[:at], (p[at:at + n // 2] + [int(rng.integers(0, len(tokens)))] + p[at + n // 2:])[:n]))
        rows.append((p[:at], (p[at:at + 1] + [-1, -1] + p[at + 1:])[:n]))
    times = 1 + 5000 // len(rows)
    spec = G.Spec(G.Grammar(grammar, role, lexicons), G.Vocab(tokens, eos, specials))

    def feed(rows):
        B, m = len(rows), max(1, max(len(a) for a, _ in rows))
        before, fed = np.full((B, m), -1, np.int32), np.full((B, n), -1, np.int32)
        for b, (a, x) in enumerate(rows):
            before[b, :len(a)] = a
            fed[b, :len(x)] = x
        st, cin, out = torch.zeros(B, dtype=torch.int32, device="cuda"), G.Configs(spec, B), G.Configs(spec, B)
        for c in (cin, out):
            G.grid_configs_enable_audit(spec.h, c.h)
        G.grid_advance(spec, cin, cin, torch.from_numpy(before).cuda(), st)
        assert not st.any()
        G.grid_advance(spec, cin, out, torch.from_numpy(fed).cuda(), st)
        records = torch.zeros((B, 80), dtype=torch.uint8, device="cuda")
        mask, zero = torch.zeros((B, spec.W), dtype=torch.int32, device="cuda"), torch.zeros_like(st)
        G.grid_audit_append(spec.h, out.h, mask, zero, 0, records)
        torch.cuda.synchronize()
        return st.cpu().numpy(), out, records.cpu().numpy()

    st, out, rec = feed(rows)
    st2, out2, rec2 = feed(rows * times)
    assert (st2 == np.tile(st, times)).all()
    assert (rec2 == np.tile(rec, (times, 1))).all()
    ref = [out.export(b) for b in range(len(rows))]
    for b in rng.integers(0, len(rows) * times, 300):
        assert out2.export(int(b)) == ref[int(b) % len(rows)], b


def test_batches_cut_by_their_bytes():
    """Tokens of 17 to 400 bytes: a batch that ends one byte below its 384
    bytes, at them and above; tokens of exactly 384 bytes and of more (which
    no batch holds) first, in the middle and last; spellings beyond the 16
    bytes that are kept with them."""
    import torch
    from oracle import compile_grammar
    from paper_2607_11951_gb300 import grid as G
    by_len = {2 * k + odd: b"a+" * k + b" " * odd for k in list(range(9, 31)) + [192, 193, 200] for odd in (0, 1)}
    tokens = [bytes([c]) for c in b"ab+*() "] + list(by_len.values()) + [b"b+" * 100 + b")", b"<eos>"]
    eos = len(tokens) - 1
    of = {n: tokens.index(t) for n, t in by_len.items()}
    bad = eos - 1  # refused after 200 bytes
    rows = []
    for last in (23, 24, 25):  # 6 x 60 + last = 383, 384, 385 bytes
        rows.append([of[60]] * 6 + [of[last]] + [of[41]] * 20)
        rows.append([of[19]] * 3 + [-1] + [of[60]] * 5 + [of[last + 3]] + [of[60]] * 5 + [of[last]] * 2)
        rows.append([of[18]] * 40 + [of[60]] * 6 + [of[last]])
    for n in (384, 385, 386, 387, 400):
        for at in (0, 9, 18):
            rows.append([of[17 + 2 * (i % 9) + 1] for i in range(at)] + [of[n]] + [of[20 + i] for i in range(18 - at)])
        rows.append([of[n], of[n], of[18], of[n]])
    rows += [[of[60]] * 7 + [bad, of[18]], [bad], [of[385], bad], [of[18]] * 33 + [bad], [of[60], eos], [of[384], eos]]
    og = compile_grammar(grammar_text("expr"))
    want = [_oracle_feed(og, r, tokens, eos, []) for r in rows]
    assert sorted({w[0] for w in want}) == [G.GRID_ST_OK, G.GRID_ST_TOKEN_NOT_ALLOWED]
    B, n = len(rows), max(map(len, rows))
    fed, took = np.full((B, n), -1, np.int32), np.full((B, n), -1, np.int32)
    for b, r in enumerate(rows):
        fed[b, :len(r)] = r
        took[b, :len(want[b][1])] = want[b][1]
    spec = G.Spec(G.Grammar(grammar_text("expr"), None, {}), G.Vocab(tokens, eos, []))
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    mask = torch.zeros((B, spec.W), dtype=torch.int32, device="cuda")
    cfg, other, one = G.Configs(spec, B), G.Configs(spec, B), G.Configs(spec, B)
    d = torch.from_numpy(fed).cuda()
    G.grid_advance(spec, cfg, other, d, st)
    assert st.cpu().tolist() == [w[0] for w in want]
    G.grid_advance_masks(spec, cfg, cfg, d, mask, st)
    for k in range(n):
        G.grid_advance(spec, one, one, torch.from_numpy(np.ascontiguousarray(took[:, k:k + 1])).cuda(), st)
        assert not st.any()
    for b in range(B):
        ref = one.export(b)
        assert other.export(b) == ref and cfg.export(b) == ref, (b, rows[b])
