"""The warp-specialized decode where its halves can go wrong: every group size
(the CTA merge takes the heads of the 10-bit dither's batches four at a time), page
counts around the eight page streams, both dithers, one sequence and batches."""

import pytest
import torch

import workloads as W
from oracle import pipeline as OP
from tests._parity import assert_close, descs, make_inputs, numpy_cache_to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [8, 10])
@pytest.mark.parametrize("group", [1, 2, 3, 5, 7, 8])
@pytest.mark.parametrize("ctx_lens", [[1], [128], [129, 15, 2049], [16, 0, 17, 700]])
def test_decode_pairs_match_oracle(bits, group, ctx_lens):
    import paper_2607_28699_gb300 as wc
    wl = W.Workload("pairs", 1, 2 * group, 2, ctx_lens, shuffle_pages=True, seed=31 + group)
    bt, sm, k, v, q = make_inputs(wl, 0)
    od, gd = descs(2 * group, 2, wl.num_pages, bits=bits, layout=group % 2, seed=6)
    ocache = OP.empty_cache(od)
    OP.write_tokens(od, 0, k.numpy(), v.numpy(), sm, ocache)
    cache = numpy_cache_to_gpu(ocache, gd)   # the same stored inputs on both sides
    ws = wc.Workspace(gd, wl.batch, wl.max_pages)
    ctx = torch.tensor(ctx_lens, dtype=torch.int32, device="cuda")
    out, meter, raw = wc.metered_decode_attention(gd, 0, q.cuda(), torch.from_numpy(bt).cuda(), ctx, cache, ws)
    torch.cuda.synchronize()
    assert wc.read_status(ws) == 0
    for b, S in enumerate(ctx_lens):
        r = OP.decode_sequence(od, 0, q[b].numpy(), bt[b], S, ocache)
        for name, gpu in (("out", out), ("meter", meter), ("meter_raw", raw)):
            assert_close(gpu[b].cpu().numpy(), r[name], f"{name}[{b}]")
