"""Batches with short block tables on both sides of the rule between the split and the flattened
plan (csrc/dispatch.h), against each sequence decoded on its own; the append's tokens against a
write before the decode."""

import numpy as np
import pytest
import torch

from tests._parity import assert_close
from tests.test_gpu_flat_batches import _batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [8, 10])
@pytest.mark.parametrize("batch,hkv,group", [(75, 8, 1), (76, 8, 1), (76, 8, 3), (76, 8, 4), (190, 8, 5), (190, 8, 6)])
@pytest.mark.parametrize("pages", [2, 5, 40])
@pytest.mark.parametrize("variant", ["plain", "tier_b", "value", "repair"])
def test_short_tables_match_each_sequence_alone(batch, hkv, group, pages, bits, variant):
    import paper_2607_28699_gb300 as wc
    rng = np.random.default_rng(batch + group + pages)
    lens = [int(x) for x in rng.integers(1, 16 * pages + 1, batch)]
    lens[0], lens[5], lens[batch - 1] = 16 * pages, 0, 1
    desc, table, ctx, q, cache = _batch(lens, wc.SCHEME_DITHER_INT8, group * hkv, hkv, variant == "value", bits)

    def decode(q, table, ctx):
        ws = wc.Workspace(desc, q.shape[0], table.shape[1])
        if variant == "tier_b":
            r = wc.metered_decode_attention_tier_b(desc, 0, q, table, ctx, cache, ws, 1e-4)
        elif variant == "value":
            r = wc.metered_decode_attention_v(desc, 0, q, table, ctx, cache, ws)
        elif variant == "repair":   # the pages' terms are relative to running maxima: their contributions are compared
            r = wc.metered_decode_attention_repair(desc, 0, q, table, ctx, cache, ws)
            r = (*r[:3], wc.repair_select(r[3], r[4], ctx, 0.05)[0])
        else:
            r = wc.metered_decode_attention(desc, 0, q, table, ctx, cache, ws)
        torch.cuda.synchronize()
        assert wc.read_status(ws) == 0
        return r

    got = decode(q, table, ctx)
    for b in sorted({0, 1, 5, batch // 2, batch - 1}):
        one = decode(q[b:b + 1].contiguous(), table[b:b + 1].contiguous(), ctx[b:b + 1].contiguous())
        for i, (x, y) in enumerate(zip(got, one)):
            assert_close(x[b:b + 1].cpu().numpy(), y.cpu().numpy(), f"output {i} of sequence {b}, {lens[b]} tokens")


@pytest.mark.parametrize("batch", [19, 20, 100])
@pytest.mark.parametrize("pages", [1, 5, 40])
def test_append_equals_write_then_decode(batch, pages):
    import paper_2607_28699_gb300 as wc
    rng = np.random.default_rng(batch + pages)
    lens = [int(x) for x in rng.integers(1, 16 * pages + 1, batch)]
    lens[0], lens[1] = 16 * pages, 1
    desc, table, ctx, q, cache = _batch(lens, wc.SCHEME_DITHER_INT8, 32, 8)
    g = torch.Generator().manual_seed(7)
    k, v = (torch.randn(batch, 8, 128, generator=g).half().cuda() for _ in range(2))
    last = [(x - 1) // 16 for x in lens]
    slots = torch.tensor([int(table[b, last[b]]) * 16 + (lens[b] - 1) % 16 for b in range(batch)], dtype=torch.int32).cuda()
    slots[3] = -1                                            # no new token
    ws = wc.Workspace(desc, batch, table.shape[1])
    got = [x.clone() for x in wc.metered_decode_attention_append(desc, 0, q, table, ctx, cache, ws, k, v, slots)]
    torch.cuda.synchronize()
    assert wc.read_status(ws) == 0
    stored = [t.clone() for t in (cache.k_codes, cache.v_codes, cache.k_scale, cache.v_scale, cache.k_witness)]
    wc.kv_quantize_witness(desc, 0, k, v, slots, cache)
    for a, b in zip(stored, (cache.k_codes, cache.v_codes, cache.k_scale, cache.v_scale, cache.k_witness)):
        assert torch.equal(a, b)
    for i, (x, y) in enumerate(zip(got, wc.metered_decode_attention(desc, 0, q, table, ctx, cache, ws))):
        assert_close(x.cpu().numpy(), y.cpu().numpy(), f"output {i}")
