"""Status reports under each of the decode's plans (csrc/dispatch.h): a length out of range, a page
outside the pool, an append slot that is not the context's last.  Block tables of 45 pages take the
flattened plan (its lengths are read by a thread each up to 512 sequences, by its merge's lanes
up to 32), or with the 10-bit dither and 600 units the kernel with two CTAs per SM."""

import numpy as np
import pytest
import torch

from tests._parity import assert_close
from tests.test_gpu_flat_batches import _batch

pytestmark = pytest.mark.gpu

PLANS = [("int8", 8, 2), ("int8", 8, 33), ("int8", 8, 513), ("int8", 10, 2), ("int8", 10, 33), ("int8", 10, 513), ("int8", 10, 600),
         ("g32", 8, 2), ("g32", 8, 33), ("g32", 8, 513), ("fp8", 8, 33)]


def _case(scheme, bits, batch):
    import paper_2607_28699_gb300 as wc
    code = {"int8": wc.SCHEME_DITHER_INT8, "g32": wc.SCHEME_DITHER_INT8_G32, "fp8": wc.SCHEME_FP8_E4M3}[scheme]
    lens = [int(x) for x in np.random.default_rng(batch).integers(20, 80, batch)]
    lens[batch // 2] = 16 * 45
    return wc, lens, _batch(lens, code, 4, 1, bits=bits)


def _decode(wc, desc, q, table, ctx, cache, ws):
    r = [x.clone() for x in wc.metered_decode_attention(desc, 0, q, table, ctx, cache, ws)]
    torch.cuda.synchronize()
    return r, wc.read_status(ws)


@pytest.mark.parametrize("scheme,bits,batch", PLANS)
def test_lengths_out_of_range(scheme, bits, batch):
    wc, lens, (desc, table, ctx, q, cache) = _case(scheme, bits, batch)
    ws = wc.Workspace(desc, batch, table.shape[1])
    want, status = _decode(wc, desc, q, table, ctx, cache, ws)
    assert status == 0
    for at in (0, batch - 1):
        for bad in (-1, 16 * 45 + 1, -(1 << 31), (1 << 31) - 1):
            lengths = ctx.clone()
            lengths[at] = bad
            got, status = _decode(wc, desc, q, table, lengths, cache, ws)
            assert status == wc.DEV_BAD_CTX
            clamped = lengths.clamp(0, 16 * 45)              # as if the length were this
            ref, status = _decode(wc, desc, q, table, clamped, cache, ws)
            assert status == 0
            for x, y, z in zip(got, ref, want):
                assert torch.equal(x, y)
                if bad < 0:
                    assert not x[at].any()
                others = [b for b in range(batch) if b != at]
                assert_close(x[others].cpu().numpy(), z[others].cpu().numpy(), "the other sequences")
    got, status = _decode(wc, desc, q, table, ctx, cache, ws)
    assert status == 0 and all(torch.equal(x, y) for x, y in zip(got, want))


@pytest.mark.parametrize("scheme,bits,batch", PLANS)
def test_pages_outside_the_pool(scheme, bits, batch):
    wc, lens, (desc, table, ctx, q, cache) = _case(scheme, bits, batch)
    ws = wc.Workspace(desc, batch, table.shape[1])
    want, _ = _decode(wc, desc, q, table, ctx, cache, ws)
    for at, page in ((0, 0), (batch // 2, 44), (batch // 2, 3)):
        for bad in (-1, desc.num_pages, 1 << 30):
            t = table.clone()
            t[at, page] = bad
            got, status = _decode(wc, desc, q, t, ctx, cache, ws)
            assert status == wc.DEV_BAD_PAGE
            others = torch.tensor([b for b in range(batch) if b != at], device="cuda")
            for x, y in zip(got, want):
                assert torch.equal(x[others], y[others])      # the cuts are the same
                assert torch.isfinite(x[at]).all() and not torch.equal(x[at], y[at])
    t = table.clone()
    t[batch // 2] = -1                                        # no page of it can be read
    got, status = _decode(wc, desc, q, t, ctx, cache, ws)
    assert status == wc.DEV_BAD_PAGE and not got[0][batch // 2].any()


@pytest.mark.parametrize("batch", [2, 33, 160, 513])
def test_append_slot_not_the_last(batch):
    wc, lens, (desc, table, ctx, q, cache) = _case("int8", 8, batch)
    g = torch.Generator().manual_seed(3)
    k, v = (torch.randn(batch, 1, 128, generator=g).half().cuda() for _ in range(2))
    slots = torch.tensor([int(table[b, (n - 1) // 16]) * 16 + (n - 1) % 16 for b, n in enumerate(lens)], dtype=torch.int32).cuda()
    ws = wc.Workspace(desc, batch, table.shape[1])
    before = cache.k_codes.clone()
    for at in (0, batch // 2, batch - 1):
        for bad in (int(slots[at]) - 1, 16 * desc.num_pages, (1 << 31) - 1):
            cache.k_codes.copy_(before)
            s = slots.clone()
            s[at] = bad
            wc.metered_decode_attention_append(desc, 0, q, table, ctx, cache, ws, k, v, s)
            torch.cuda.synchronize()
            assert wc.read_status(ws) == wc.DEV_BAD_APPEND
            changed = (cache.k_codes != before).any(-1).view(-1).nonzero().view(-1)
            allowed = torch.cat([slots[:at], slots[at + 1:]])
            assert torch.isin(changed.int(), allowed).all()   # the others' tokens and nothing else
            assert changed.numel() == batch - 1
