"""Which tables are staged in shared memory, and the launches that follow, on a
CUDA runtime without a GPU: lexer and parser tables of up to 96 KB are staged
whatever else goes with them, no launch asks for more shared memory than its
kernel was allowed, a batch whose spellings are all walked gets the walk's
largest blocks, and a mask row's chunk digests have room up to 25 M tokens."""
import ctypes

import pytest

from paper_2607_11951_gb300 import grid as G
from tests import fakes

SM_BYTES = 227 * 1024  # shared memory of one block, at most


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fakes.link(tmp_path_factory.mktemp("fake"))


def grammar(n, cats):
    """Statements led by n keywords, with `cats` categories of one regex."""
    name = lambda i: "%s%s" % (chr(97 + i // 16), chr(97 + i % 16))
    toks = "".join("%%token T%d /%s/\n" % (i, name(i)) for i in range(n))
    toks += "".join("%%token C%d /[q-z]+/\n" % c for c in range(cats))
    prods = "".join("stmt -> T%d T%d opt T%d T%d\n" % (i, (i * 7 + 3) % n, (i * 5 + 1) % n, (i * 3 + 2) % n)
                    for i in range(n))
    prods += "".join("stmt -> C%d SEMI T%d\n" % (c, c) for c in range(cats))
    return toks + "".join("%%category C%d\n" % c for c in range(cats)) + \
        "%token SEMI /;/\n%ignore WS /[ ]+/\n%start prog\nprog -> prog stmt\nprog -> stmt\n" + prods + \
        "opt -> %empty\nopt -> opt2 SEMI\nopt2 -> %empty\n"


def table_bytes(i):
    """Lexer and parser tables without the reduce groups."""
    Q, S, T1, N = i["dfa_states"], i["lalr_states"], i["terminals"] + 1, i["nonterminals"]
    return 256 + 2 * Q * i["byte_classes"] + 32 * Q + 2 * S * (T1 + N) + 2 * i["productions"] + 20 * S


@pytest.mark.parametrize("cats", [0, 7])
def test_tables_of_96_kb_are_staged(fake, cats):
    with fakes.use(fake) as rt:
        toks = [bytes([b]) for b in range(256)] + [b"%d" % i for i in range(10, 60000)] + [b"<eos>"]
        v = G.Vocab(toks, len(toks) - 1, [])
        seen = []
        for n in range(70, 92):
            g = G.Grammar(grammar(n, cats), None, {"C%d" % c: [b"qr" + bytes([113 + c])] for c in range(cats)})
            size = table_bytes(g.info())
            rt.reset(ones=1)
            s = G.Spec(g, v)
            staged = s.info()["staged_bytes"]
            seen.append((size > 94 * 1024, staged > 0))
            assert s.info()["ci_on"] and (staged > 0 or size > 96 * 1024), (n, size)
            one = ctypes.c_void_p(16)
            for B in (152, 4096):  # rows that stage large tables, and that do not; both want the walk's largest blocks
                c = G.Configs(s, B)
                rt.reset()
                assert G.lib().grid_masks(s.h, c.h, one, one, None) == G.GRID_OK
                assert G.lib().grid_reserve(s.h, c.h, one, one, 16, one, None, 0, None, None) == G.GRID_OK
                for name, grid, threads, smem, limit in rt.launches():
                    assert smem <= limit <= SM_BYTES, (name, smem, limit)
                    if "k_rowILi0E" in name or "k_walkILb0E" in name:
                        pair = 2 * (staged + 39 * 1024) <= 228 * 1024  # two blocks of k_row on an SM
                        assert ("0ELb1E" in name) == (staged > 0 and (B == 152 or pair)), (name, B, staged)
                    if "k_walk" in name:
                        assert threads >= 20 * 32
                del c
            del g, s
        assert (True, True) in seen and (True, False) in seen
        del v


def test_walk_without_ci_classes(fake):
    from workloads import configs
    wl = configs.manycat(12, 21, B=1)
    with fakes.use(fake) as rt:
        g = G.Grammar(wl["grammar"], wl["role"], wl["lexicons"])
        v = G.Vocab(wl["tokens"], wl["eos"], wl["specials"])
        s = G.Spec(g, v)
        assert not s.info()["ci_on"]
        warps = []
        for B in (1, 32):
            c = G.Configs(s, B)
            rt.reset()
            assert G.lib().grid_masks(s.h, c.h, ctypes.c_void_p(16), ctypes.c_void_p(16), None) == G.GRID_OK
            warps += [threads // 32 for name, _, threads, _, _ in rt.launches() if "k_walk" in name]
            del c
        assert warps == [8, 24]
        del g, v, s


def test_audit_record_of_the_largest_vocabulary(fake):
    chunks = 25_165_824 // 8192
    with fakes.use(fake) as rt:
        toks = [bytes([b]) for b in range(256)] + [b"<eos>"]
        v, g = G.Vocab(toks, 256, []), G.Grammar("%token A /a/\n%ignore WS /[ ]+/\n%start s\ns -> A\n")
        s = G.Spec(g, v)
        c = G.Configs(s, 1)
        one = ctypes.c_void_p(16)
        assert G.lib().grid_configs_enable_audit(s.h, c.h, None) == G.GRID_OK
        rt.reset()
        assert G.lib().grid_audit_append(s.h, c.h, one, one, 0, one, None) == G.GRID_OK
        # dynamic shared memory that the kernel may have beside its own: two words and two per chunk
        (limit,) = [limit for name, _, _, _, limit in rt.launches() if "k_audit_append" in name]
        assert limit != fakes.DEFAULT_SMEM and limit >= 8 * (2 + 2 * chunks)
        del c, s, g, v
