"""A grammar whose tables are too large for shared memory: the kernels'
instances that read them from global memory (masks, token feed, spans,
reserve) against the oracle."""
import numpy as np
import pytest

from tests.harness import unpack

pytestmark = pytest.mark.gpu

N = 112


def _grammar():
    name = lambda i: "%s%s" % (chr(97 + i // 16), chr(97 + i % 16))
    toks = "".join("%%token T%d /%s/\n" % (i, name(i)) for i in range(N))
    prods = "".join("stmt -> T%d T%d opt T%d T%d\n" % (i, (i * 7 + 3) % N, (i * 5 + 1) % N, (i * 3 + 2) % N)
                    for i in range(N))
    return toks + "%token SEMI /;/\n%ignore WS /[ ]+/\n%start prog\nprog -> prog stmt\nprog -> stmt\n" + prods + \
        "opt -> %empty\nopt -> opt2 SEMI\nopt2 -> %empty\n", name


def test_tables_in_global_memory():
    import torch
    from oracle import compile_grammar
    from oracle.reserve import Reserve
    from paper_2607_11951_gb300 import grid as G
    text, name = _grammar()
    toks = [bytes([c]) for c in b"abcdefghijklmnop ;"] + [(" " + name(i)).encode() for i in range(N)] + \
        [(name(i) + " " + name((i * 7 + 3) % N)).encode() for i in range(0, N, 3)] + [b"<eos>"]
    eos = len(toks) - 1
    spec = G.Spec(G.Grammar(text, None, {}), G.Vocab(toks, eos, []))
    assert spec.info()["staged_bytes"] == 0
    w = lambda i: 18 + i % N
    rows = [[], [w(5)], [w(9), w(9 * 7 + 3)], [w(9), w(9 * 7 + 3), w(9 * 5 + 1), w(9 * 3 + 2), w(8)], [0], [w(9), 16]]
    og = compile_grammar(text)
    B, n = len(rows), max(map(len, rows))
    fed = np.full((B, n), -1, np.int32)
    for b, r in enumerate(rows):
        fed[b, :len(r)] = r
    cfg = G.Configs(spec, B)
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    mask = torch.zeros((B, spec.W), dtype=torch.int32, device="cuda")
    G.grid_advance_masks(spec, cfg, cfg, torch.from_numpy(fed).cuda(), mask, st)
    torch.cuda.synchronize()
    bits = unpack(mask.cpu().numpy().view(np.uint32), len(toks))
    cfgs = [og.config_from_ids(r, toks, eos, []) for r in rows]
    for b in range(B):
        assert int(st[b]) == 0
        assert (bits[b] == np.asarray(og.mask(cfgs[b], toks, eos, []), np.uint8)).all(), b
    cost = torch.zeros(B, dtype=torch.int32, device="cuda")
    out = torch.zeros((B, 64), dtype=torch.int32, device="cuda")
    G.grid_reserve(spec.h, cfg.h, cost, out, st)
    R = Reserve(og, toks, eos, [])
    assert cost.cpu().tolist() == [R.reserve(c) if R.reserve(c) is not None else -1 for c in cfgs]
    one = G.Configs(spec, B)
    G.grid_advance(spec, one, one, torch.from_numpy(np.ascontiguousarray(fed[:, :1])).cuda(), st)
    assert not st.any()
    span, length = torch.zeros((B, 4), dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda")
    G.grid_forced_span(spec.h, one.h, 4, mask, span, length, st)
    torch.cuda.synchronize()
    for b, r in enumerate(rows):
        want = og.forced_span(og.config_from_ids(r[:1], toks, eos, []), toks, eos, [], 4)[0]
        assert span[b].tolist()[:int(length[b])] == list(want), b


def test_largest_staged_tables():
    """The largest tables that are staged, in a batch that stages them and in one
    that reads them from global memory: every row's mask is the oracle's."""
    from oracle import compile_grammar
    from paper_2607_11951_gb300 import grid as G
    from tests.harness import GpuRun
    from tests.test_staging_host import grammar
    lexicons = {"C%d" % c: [b"qr" + bytes([113 + c])] for c in range(7)}
    text = grammar(82, 7)
    toks = [bytes([c]) for c in b"abcdefghijklmnopqrstuvwxyz ;"] + [b"aa ", b"aa ad", b" qrq", b"q ", b"rq ", b"rq ;", b"r",
                                                                     b"rq;aa ab ", b"; ", b"<eos>"]
    eos = len(toks) - 1
    byte = {t: i for i, t in enumerate(toks)}
    kinds = [[byte[bytes([c])] for c in x] for x in (b"", b"a", b"aa ad", b"q", b"qr", b"qrq", b"qrq;", b"qrq ; aa ")]
    og = compile_grammar(text, None, lexicons)
    cfgs = [og.config_from_ids(p, toks, eos) for p in kinds]
    assert all(c is not None for c in cfgs)
    for B in (152, 3200):
        run = GpuRun(dict(name="staging", grammar=text, role=None, lexicons=lexicons, tokens=toks, eos=eos, specials=[],
                          prefixes=[kinds[b % 8] for b in range(B)], max_depth=1024))
        assert run.spec.info()["staged_bytes"] > 104 * 1024
        assert not run.build_configs().any()
        words, status = run.masks()
        assert not status.any()
        bits = unpack(words, run.V)
        for k, c in enumerate(cfgs):
            assert (bits[k::8] == np.asarray(og.mask(c, toks, eos), np.uint8)).all(), (B, kinds[k])
