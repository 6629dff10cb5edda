"""The -inf fill at the places where its split can go wrong: rows at every
offset from a sector boundary, vocabularies of less than a sector, of whole
sectors and one element more, blocks' ends, masks of no bit, of every bit and
of single bits; standalone and in the step; neighbours of a row untouched."""
import numpy as np
import pytest

from tests.harness import pack_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V", [1, 7, 8, 15, 16, 17, 31, 32, 33, 8191, 8192, 8193, 8207, 40_001])
def test_apply_at_every_offset(dtype, V):
    import torch
    from paper_2607_11951_gb300 import grid as G
    tdt, idt = (torch.float32, torch.int32) if dtype == "f32" else (torch.bfloat16, torch.int16)
    per = 32 // tdt.itemsize
    rng = np.random.default_rng(V)
    B = 5
    bits = (rng.random((B, V)) < np.array([0.0, 1.0, 0.5, 0.05, 0.95])[:, None]).astype(np.uint8)
    mask = torch.from_numpy(pack_bits(bits).view(np.int32)).cuda()
    want_bits = torch.from_numpy(bits.astype(bool)).cuda()
    for off in range(0, per, 1 if V < 100 else 3):
        for stride in {V, (V + per - 1) // per * per, V + 3}:
            flat = torch.randn(off + B * stride + per, device="cuda").to(tdt)
            ref = flat.clone()
            rows = torch.as_strided(flat, (B, V), (stride, 1), off)
            torch.as_strided(ref, (B, V), (stride, 1), off).masked_fill_(~want_bits, float("-inf"))
            G.grid_apply_mask(mask, rows)
            assert torch.equal(flat.view(idt), ref.view(idt)), (off, stride)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V", [8191, 8192, 8225, 16_401])
def test_fused_fill_at_block_ends(dtype, V):
    import torch
    from paper_2607_11951_gb300 import grid as G
    from tests.harness import unpack
    from workloads import configs
    wl = configs.tiny_expr(B=4)
    fill = [b"%d" % i for i in range(V)] + [b"a%d" % i for i in range(V)]
    toks = list(dict.fromkeys([bytes([c]) for c in b"abcdefghijklmnopqrstuvwxyz0123456789+*() "] + fill))[:V - 1]
    spec = G.Spec(G.Grammar(wl["grammar"], wl["role"], wl["lexicons"]), G.Vocab(toks + [b"<eos>"], V - 1, []))
    B = 4
    cfg, out = G.Configs(spec, B), G.Configs(spec, B)
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    mask = torch.zeros((B, spec.W), dtype=torch.int32, device="cuda")
    tok = torch.tensor([0, 39, 1, 38], dtype=torch.int32, device="cuda")
    tdt, idt = (torch.float32, torch.int32) if dtype == "f32" else (torch.bfloat16, torch.int16)
    for stride, off in ((V, 0), (V + 7, 0), (V + 16 - V % 16, 0), (V, 1)):
        flat = torch.randn(off + B * stride + 32, device="cuda").to(tdt)
        ref = flat.clone()
        rows = torch.as_strided(flat, (B, V), (stride, 1), off)
        G.grid_advance_masks(spec, cfg, out, tok, mask, st, rows)
        bits = torch.from_numpy(unpack(mask.cpu().numpy().view(np.uint32), V).astype(bool)).cuda()
        torch.as_strided(ref, (B, V), (stride, 1), off).masked_fill_(~bits, float("-inf"))
        assert torch.equal(flat.view(idt), ref.view(idt)), (stride, off)
