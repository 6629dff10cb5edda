"""grid_reserve at the sizes where its split can go wrong: stacks and searches
that fit the warps' shared memory, that just do not, and that are far beyond
it, in one batch, against the oracle's reserve and a legal completion."""
import numpy as np
import pytest

from workloads import grammar_text

pytestmark = pytest.mark.gpu

ALPHA = b"abcdefghijklmnopqrstuvwxyz0123456789+*() "


@pytest.mark.parametrize("depths", [(0, 1, 40, 90), (120, 130, 200, 380), (1010, 1023, 1024, 1100)])
def test_reserve_of_deep_stacks(depths):
    import torch
    from oracle import compile_grammar
    from oracle.reserve import Reserve
    from paper_2607_11951_gb300 import grid as G
    toks = [bytes([c]) for c in ALPHA] + [b" )", b"<eos>"]
    eos = len(toks) - 1
    t = {x: i for i, x in enumerate(toks)}
    rows = []
    for d in depths:
        rows += [[t[b"("]] * d, [t[b"("]] * d + [t[b"a"]], [t[b"("]] * d + [t[b"a"], t[b"+"]]]
    B, n, cap = len(rows), max(1, max(map(len, rows))), 4 * max(depths) + 16
    fed = np.full((B, n), -1, np.int32)
    for b, r in enumerate(rows):
        fed[b, :len(r)] = r
    spec = G.Spec(G.Grammar(grammar_text("expr"), None, {}), G.Vocab(toks, eos, []))
    cfg = G.Configs(spec, B)
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    G.grid_advance(spec, cfg, cfg, torch.from_numpy(fed).cuda(), st)
    assert not st.any()
    cost = torch.zeros(B, dtype=torch.int32, device="cuda")
    out = torch.zeros((B, cap), dtype=torch.int32, device="cuda")
    G.grid_reserve(spec.h, cfg.h, cost, out, st)
    torch.cuda.synchronize()
    og = compile_grammar(grammar_text("expr"))
    R = Reserve(og, toks, eos, [])
    for b, r in enumerate(rows):
        c = og.config_from_ids(r, toks, eos, [])
        assert int(st[b]) == G.GRID_ST_OK and int(cost[b]) == R.reserve(c), b
        seq = [int(x) for x in out[b] if int(x) >= 0]
        assert len(seq) == int(cost[b])
        for x in seq:
            c = og.advance(c, x, toks, eos, [])
            assert c is not None, b
        assert c.complete


WAYS = "%token LP \"(\"\n%token RP \")\"\n" + "".join("%%token K%d \"k%s\"\n" % (i, "abcdefgh"[:i]) for i in range(9)) + """
%ignore WS /[ ]+/
%start e
e -> LP e RP
""" + "".join("e -> K%d\n" % i for i in range(8)) + """e -> u1
u1 -> u2
u2 -> u3
u3 -> u4
u4 -> K8
"""


def test_reserve_where_some_ways_fit():
    """Nine ways to end the pending lexeme (k, ka, .. kabcdefgh), of which the
    last visits more entries: over the depths at which a search outgrows a
    warp's space, for one way while the others still fit, for all, for none."""
    import torch
    from oracle import compile_grammar
    from oracle.reserve import Reserve
    from paper_2607_11951_gb300 import grid as G
    toks = [bytes([c]) for c in b"abcdefghk() "] + [b"<eos>"]
    eos = len(toks) - 1
    t = {x: i for i, x in enumerate(toks)}
    rows = [[t[b"("]] * d + [t[b"k"]] for d in list(range(120, 136)) + list(range(184, 200)) + list(range(374, 390))]
    B, n, cap = len(rows), max(map(len, rows)), 1024
    fed = np.full((B, n), -1, np.int32)
    for b, r in enumerate(rows):
        fed[b, :len(r)] = r
    spec = G.Spec(G.Grammar(WAYS, None, {}), G.Vocab(toks, eos, []))
    cfg = G.Configs(spec, B)
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    G.grid_advance(spec, cfg, cfg, torch.from_numpy(fed).cuda(), st)
    assert not st.any()
    cost = torch.zeros(B, dtype=torch.int32, device="cuda")
    out = torch.zeros((B, cap), dtype=torch.int32, device="cuda")
    og = compile_grammar(WAYS)
    R = Reserve(og, toks, eos, [])
    cfgs = [og.config_from_ids(r, toks, eos, []) for r in rows]
    want = [R.reserve(c) for c in cfgs]
    for _ in range(3):
        G.grid_reserve(spec.h, cfg.h, cost, out, st)
        torch.cuda.synchronize()
        assert not st.any() and cost.tolist() == want
        for b, c in enumerate(cfgs):
            seq = [int(x) for x in out[b] if int(x) >= 0]
            assert len(seq) == want[b]
            if b % 16 == 0:
                for x in seq:
                    c = og.advance(c, x, toks, eos, [])
                    assert c is not None, b
                assert c.complete
