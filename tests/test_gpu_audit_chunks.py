"""The audit kernels at the sizes where their split can go wrong: mask rows of
one block and less, of whole chunks and one word more, and of more chunks than
a block hashes at once; and node hashes made after several tokens were fed
(entries pushed, popped and pushed again) against the oracle's."""
import struct

import numpy as np
import pytest

from tests.harness import GpuRun, unpack
from workloads import configs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [64, 1024, 1025, 8192, 8193, 8192 * 8 + 40, 8192 * 33 + 31])
def test_mask_id_at_chunk_edges(V):
    import torch
    from oracle import audit
    from paper_2607_11951_gb300 import grid as G
    wl = configs.tiny_expr(B=1)
    alphabet = sorted({bytes([b]) for t in wl["tokens"] for b in t if t != wl["tokens"][wl["eos"]]})
    fill = [b"%x" % i for i in range(V)]
    tokens = list(dict.fromkeys(alphabet + fill))[:V - 1] + [b"<eos>"]
    g = G.Grammar(wl["grammar"], wl["role"], wl["lexicons"])
    spec = G.Spec(g, G.Vocab(tokens, V - 1, []))
    B = 3
    cfg = G.Configs(spec, B)
    G.grid_configs_enable_audit(spec.h, cfg.h)
    rng = np.random.default_rng(V)
    W = (V + 31) // 32
    words = rng.integers(0, 2 ** 32, size=(B, W), dtype=np.uint32)
    words[:, -1] &= np.uint32((1 << (V - 32 * (W - 1))) - 1 if V % 32 else 0xFFFFFFFF)
    bits = unpack(words, V)
    mask = torch.from_numpy(words.view(np.int32)).cuda()
    rec = torch.zeros((2, B, 80), dtype=torch.uint8, device="cuda")
    toks = torch.tensor([1, -1, 2], dtype=torch.int32, device="cuda")
    G.grid_audit_append(spec.h, cfg.h, mask, toks, 0, rec[0])
    G.grid_audit_append(spec.h, cfg.h, mask, toks, 1, rec[1])
    torch.cuda.synchronize()
    got = rec.cpu().numpy()
    for b in range(B):
        if int(toks[b]) < 0:
            assert not got[:, b].any()
            continue
        mid = audit.mask_id(bits[b].tolist())
        prev = audit.GENESIS
        for k in range(2):
            want = audit.record(k, 0, mid, int(toks[b]), V - int(bits[b].sum()), k, prev)
            assert got[k, b].tobytes() == want, (b, k)
            prev = audit.record_hash(want)


@pytest.mark.parametrize("out_of_place", [False, True])
def test_node_hashes_of_several_tokens(out_of_place):
    import torch
    from oracle import audit, compile_grammar
    from paper_2607_11951_gb300 import grid as G
    wl = configs.sql_admin(B=6)
    run = GpuRun(wl)
    og = compile_grammar(wl["grammar"], wl["role"], wl["lexicons"])
    out = G.Configs(run.spec, run.B) if out_of_place else run.cfg
    for c in {id(run.cfg): run.cfg, id(out): out}.values():
        G.grid_configs_enable_audit(run.spec.h, c.h)
    n = max(len(p) for p in wl["prefixes"])
    half = n // 2
    toks = np.full((run.B, n), -1, np.int32)
    for b, p in enumerate(wl["prefixes"]):
        toks[b, :len(p)] = p
    first, rest = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (toks[:, :half], toks[:, half:]))
    G.grid_advance(run.spec.h, run.cfg.h, run.cfg.h, first, run.status)
    # the rest inside a mask step (k_row feeds it)
    G.grid_advance_masks(run.spec.h, run.cfg.h, out.h, rest, run.mask, run.status)
    seal = torch.zeros((run.B, 80), dtype=torch.uint8, device="cuda")
    G.grid_audit_seal(run.spec.h, out.h, torch.zeros(run.B, dtype=torch.int32, device="cuda"), 0, seal)
    torch.cuda.synchronize()
    for b, p in enumerate(wl["prefixes"]):
        cfg = og.config_from_ids(p, wl["tokens"], wl["eos"], wl["specials"])
        assert struct.unpack("<Q", seal[b].cpu().numpy().tobytes()[8:16])[0] == audit.config_hash(og, cfg), b
