"""Rows of one forced span that stop at different positions: at once, in the
middle, at the span's bound, on a forced token that the stack has no room for
(its status is reported, the configuration stays as it was), and at the end of
the sentence; spans, masks and statuses as the steps one by one give them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GRAMMAR = "".join("%%token T%s /%s/\n" % (c, c) for c in "abcdefxy") + """
%ignore WS /[ ]+/
%start s
s -> Ta Tb Tc Td Te Tf tail
tail -> Tx
tail -> Ty
"""


@pytest.mark.parametrize("max_depth,max_span", [(64, 8), (64, 3), (5, 8), (64, 1)])
def test_rows_stop_at_their_own_positions(max_depth, max_span):
    import torch
    from paper_2607_11951_gb300 import grid as G
    toks = [c.encode() for c in "abcdefxy"] + [b"<eos>"]
    eos = len(toks) - 1
    spec = G.Spec(G.Grammar(GRAMMAR, None, {}, max_depth=max_depth), G.Vocab(toks, eos, []))
    starts = [[], [0, 1], [0, 1, 2, 3, 4, 5], [0, 1, 2, 3, 4, 5, 6], [0, 1, 2, 3, 4]]
    starts = [s for s in starts if len(s) < max_depth]
    B = len(starts)
    fed = np.full((B, 8), -1, np.int32)
    for b, s in enumerate(starts):
        fed[b, :len(s)] = s
    cfg, ref = G.Configs(spec, B), G.Configs(spec, B)
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    for c in (cfg, ref):
        G.grid_advance(spec, c, c, torch.from_numpy(fed).cuda(), st)
        assert not st.any()
    mask = torch.zeros((B, spec.W), dtype=torch.int32, device="cuda")
    span = torch.zeros((B, max_span), dtype=torch.int32, device="cuda")
    length = torch.zeros(B, dtype=torch.int32, device="cuda")
    G.grid_forced_span(spec.h, cfg.h, max_span, mask, span, length, st)
    # the same, one step per call
    m1, s1 = torch.zeros_like(mask), torch.zeros_like(st)
    want = [[] for _ in range(B)]
    fail = [0] * B
    live = [True] * B
    G.grid_masks(spec, ref, m1, s1)
    for _ in range(max_span):
        words, status = m1.cpu().numpy().view(np.uint32)[:, 0], s1.cpu().numpy()
        tok = np.full(B, -1, np.int32)
        for b in range(B):
            one = live[b] and status[b] == 0 and bin(int(words[b])).count("1") == 1
            live[b] = one
            if one:
                tok[b] = int(words[b]).bit_length() - 1
                want[b].append(int(tok[b]))
        G.grid_advance(spec, ref, ref, torch.from_numpy(tok).cuda(), s1)
        refused = s1.cpu().numpy()
        for b in range(B):
            if tok[b] >= 0 and refused[b]:
                fail[b], live[b] = int(refused[b]), False
        G.grid_masks(spec, ref, m1, s1)
    final = [fail[b] or int(s1[b]) for b in range(B)]
    assert st.cpu().tolist() == final
    assert (max_depth == 5) == (G.GRID_ST_STACK_OVERFLOW in final) or max_span < 5
    assert length.cpu().tolist() == [len(w) for w in want]
    for b in range(B):
        assert span[b].tolist() == want[b] + [-1] * (max_span - len(want[b]))
        assert cfg.export(b) == ref.export(b)
    assert torch.equal(mask, m1)
