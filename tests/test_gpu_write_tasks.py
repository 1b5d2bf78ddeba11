"""Writes on both sides of the line between one and two tasks per warp (csrc/dispatch.h): the
bytes of a write are those of the same tokens written a few at a time."""

import pytest
import torch

pytestmark = pytest.mark.gpu

FIELDS = ("k_codes", "v_codes", "k_scale", "v_scale", "k_witness", "k_bypass", "v_witness")


@pytest.mark.parametrize("scheme,bits,n_tok,hkv", [("int8", 10, 15, 8), ("int8", 10, 16, 8), ("int8", 10, 17, 1), ("int8", 10, 131, 3),
                                                   ("int8", 10, 1064, 8), ("int8", 10, 1065, 8), ("g32", 8, 16, 8),
                                                   ("g32", 8, 77, 5), ("g32", 8, 2047, 8), ("g32", 8, 2048, 8)])
@pytest.mark.parametrize("rope", [0, 1])
def test_whole_write_equals_small_writes(scheme, bits, n_tok, hkv, rope):
    import paper_2607_28699_gb300 as wc
    code = wc.SCHEME_DITHER_INT8_G32 if scheme == "g32" else wc.SCHEME_DITHER_INT8
    desc = wc.CacheDesc(num_q_heads=hkv, num_kv_heads=hkv, num_pages=(n_tok + 15) // 16 + 3, scheme=code, dither_bits=bits,
                        rope_layout=rope, seed=3)
    g = torch.Generator().manual_seed(n_tok + hkv)
    k, v = (torch.randn(n_tok, hkv, 128, generator=g).half().cuda() for _ in range(2))
    slots = torch.randperm(desc.num_pages * 16, generator=g)[:n_tok].int().cuda()
    slots[n_tok // 2] = -1                                   # a skipped token

    def cache():
        c = wc.LayerCache.empty(desc, value_witness=scheme != "g32", num_bypass_pairs=2)
        if c.bypass_pairs is not None:
            c.bypass_pairs.copy_(torch.tensor([[3, 40]] * hkv, dtype=torch.int32))
        return c

    whole, pieces = cache(), cache()
    wc.kv_quantize_witness(desc, 0, k, v, slots, whole)
    for i in range(0, n_tok, 15):
        wc.kv_quantize_witness(desc, 0, k[i:i + 15].contiguous(), v[i:i + 15].contiguous(), slots[i:i + 15].contiguous(), pieces)
    for f in FIELDS:
        a, b = getattr(whole, f), getattr(pieces, f)
        if a is not None:
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), f
    assert whole.k_codes.any()
