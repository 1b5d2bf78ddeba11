"""Batches under the flattened split plan (whose cuts depend on every length) against each
sequence decoded on its own: one long sequence among short ones, empty ones, lengths
at the edges of pages and shares, at batch sizes that take every width of the merge; and
contexts that change between a captured step's replays."""

import numpy as np
import pytest
import torch

from tests._parity import assert_close

pytestmark = pytest.mark.gpu


def _lens(batch, kind):
    rng = np.random.default_rng(batch)
    lens = {"long_first": [6001] + [17] * (batch - 1),
            "ragged": list(rng.integers(1, 2500, batch)),
            "holes": [0 if i % 3 == 1 else 16 * (1 + i % 50) + i % 2 for i in range(batch)]}[kind]
    return [int(x) for x in lens]


def _batch(lens, scheme, hq, hkv, value=False, bits=8):
    import paper_2607_28699_gb300 as wc
    batch, mp = len(lens), max((x + 15) // 16 for x in lens)
    pages = sum((x + 15) // 16 for x in lens)
    desc = wc.CacheDesc(num_q_heads=hq, num_kv_heads=hkv, num_pages=pages, scheme=scheme, dither_bits=bits, seed=9)
    g = torch.Generator().manual_seed(batch + hq)
    table = torch.zeros(batch, mp, dtype=torch.int32)
    order, at = torch.randperm(pages, generator=g).int(), 0
    for b, x in enumerate(lens):
        n = (x + 15) // 16
        table[b, :n] = order[at:at + n]
        at += n
    n = 16 * pages
    k, v = (torch.randn(n, hkv, 128, generator=g).half().cuda() for _ in range(2))
    q = torch.randn(batch, hq, 128, generator=g).half().cuda()
    cache = wc.LayerCache.empty(desc, value_witness=value, num_bypass_pairs=2)
    if cache.bypass_pairs is not None:
        cache.bypass_pairs.copy_(torch.tensor([[3, 40]] * hkv, dtype=torch.int32))
    wc.kv_quantize_witness(desc, 0, k, v, torch.arange(n, dtype=torch.int32, device="cuda"), cache)
    return desc, table.cuda(), torch.tensor(lens, dtype=torch.int32, device="cuda"), q, cache


@pytest.mark.parametrize("kind", ["long_first", "ragged", "holes"])
@pytest.mark.parametrize("batch,hq,hkv", [(2, 28, 4), (5, 28, 4), (9, 16, 8), (20, 28, 4), (40, 8, 1), (600, 4, 2)])
@pytest.mark.parametrize("scheme,variant", [("int8", "plain"), ("int8", "value"), ("int8-10bit", "plain"), ("g32", "tier_b")])
def test_flat_batch_matches_its_sequences(batch, hq, hkv, kind, scheme, variant):
    import paper_2607_28699_gb300 as wc
    lens = _lens(batch, kind)
    code = wc.SCHEME_DITHER_INT8_G32 if scheme == "g32" else wc.SCHEME_DITHER_INT8
    desc, table, ctx, q, cache = _batch(lens, code, hq, hkv, variant == "value", 10 if "10" in scheme else 8)

    def decode(q, table, ctx):
        ws = wc.Workspace(desc, q.shape[0], table.shape[1])
        if variant == "value":
            r = wc.metered_decode_attention_v(desc, 0, q, table, ctx, cache, ws)
        elif variant == "tier_b":
            r = wc.metered_decode_attention_tier_b(desc, 0, q, table, ctx, cache, ws, 1e-4)
        else:
            r = wc.metered_decode_attention(desc, 0, q, table, ctx, cache, ws)
        torch.cuda.synchronize()
        assert wc.read_status(ws) == 0
        return r

    got = decode(q, table, ctx)
    for b in sorted({0, 1, 2, batch // 2, batch - 2, batch - 1} & set(range(batch))):
        one = decode(q[b:b + 1].contiguous(), table[b:b + 1].contiguous(), ctx[b:b + 1].contiguous())
        for i, (x, y) in enumerate(zip(got, one)):
            assert_close(x[b:b + 1].cpu().numpy(), y.cpu().numpy(), f"output {i} of sequence {b}, {lens[b]} tokens")


@pytest.mark.parametrize("scheme,bits", [("int8", 8), ("int8", 10), ("g32", 8)])
@pytest.mark.parametrize("tokens", [16, 128, 129, 480, 481, 640, 641])
@pytest.mark.parametrize("batch", [2, 33])
def test_short_block_tables_match_their_sequences(batch, tokens, scheme, bits):
    """Both sides of the longest block table that a batch splits instead of flattening (30 pages
    for the grouped cache, 40 otherwise), and of a split's pages."""
    import paper_2607_28699_gb300 as wc
    code = wc.SCHEME_DITHER_INT8_G32 if scheme == "g32" else wc.SCHEME_DITHER_INT8
    lens = [tokens] + [max(1, (tokens * i) // batch) for i in range(1, batch - 1)] + [0]
    desc, table, ctx, q, cache = _batch(lens, code, 28, 4, bits=bits)
    got = wc.metered_decode_attention(desc, 0, q, table, ctx, cache, wc.Workspace(desc, batch, table.shape[1]))
    for b in sorted({0, batch // 2, batch - 1}):
        one = wc.metered_decode_attention(desc, 0, q[b:b + 1].contiguous(), table[b:b + 1].contiguous(),
                                          ctx[b:b + 1].contiguous(), cache, wc.Workspace(desc, 1, table.shape[1]))
        for i, (x, y) in enumerate(zip(got, one)):
            assert_close(x[b:b + 1].cpu().numpy(), y.cpu().numpy(), f"output {i} of sequence {b}, {lens[b]} tokens")


def test_ten_bit_batch_in_a_workspace_of_one_partial_per_unit():
    """800 units, a split each: the flattened plan needs a partial per SM more than the split
    plan, which a workspace of that plan's size still gets; a smaller one is refused."""
    import paper_2607_28699_gb300 as wc
    lens = [700] + [int(x) for x in np.random.default_rng(4).integers(1, 120, 199)]
    desc, table, ctx, q, cache = _batch(lens, wc.SCHEME_DITHER_INT8, 8, 4, bits=10)
    ws = wc.Workspace(desc, 200, table.shape[1])
    least = (256 + 4 * 800 * 8 * 140 + 255) // 256 * 256
    assert ws.nbytes > least
    want = wc.metered_decode_attention(desc, 0, q, table, ctx, cache, ws)
    small = wc.Workspace(desc, 200, table.shape[1])
    small.nbytes = least
    got = wc.metered_decode_attention(desc, 0, q, table, ctx, cache, small)
    torch.cuda.synchronize()
    assert not small.view[least:].any()          # nothing written behind the given size
    for i, (x, y) in enumerate(zip(got, want)):
        assert_close(x.cpu().numpy(), y.cpu().numpy(), f"output {i}")
    small.nbytes = least - 256
    with pytest.raises(wc.WitCertError) as e:
        wc.metered_decode_attention(desc, 0, q, table, ctx, cache, small)
    assert e.value.status == 4


@pytest.mark.parametrize("scheme", ["int8", "g32"])
def test_contexts_change_between_replays(scheme):
    """A captured decode follows the lengths that the preceding kernel of the stream writes."""
    import paper_2607_28699_gb300 as wc
    code = wc.SCHEME_DITHER_INT8_G32 if scheme == "g32" else wc.SCHEME_DITHER_INT8
    full = [900, 33, 2400, 16]
    desc, table, ctx, q, cache = _batch(full, code, 28, 4)
    ws = wc.Workspace(desc, 4, table.shape[1])
    src = ctx.clone()
    outs = wc.metered_decode_attention(desc, 0, q, table, ctx, cache, ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.copy_(src)
        wc.metered_decode_attention(desc, 0, q, table, ctx, cache, ws, *outs)
    for lens in (full, [1, 33, 1999, 5], [0, 0, 2400, 0], [899, 32, 17, 16], full):
        src.copy_(torch.tensor(lens, dtype=torch.int32))
        graph.replay()
        torch.cuda.synchronize()
        assert wc.read_status(ws) == 0
        want = wc.metered_decode_attention(desc, 0, q, table, torch.tensor(lens, dtype=torch.int32, device="cuda"), cache,
                                           wc.Workspace(desc, 4, table.shape[1]))
        for x, y in zip(outs, want):
            assert torch.equal(x, y)
