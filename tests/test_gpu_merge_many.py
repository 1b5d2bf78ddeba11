"""The merge of batches that are too large for its hints (more than 32 sequences), against
each sequence decoded on its own: CTAs whose outputs belong to several sequences (one or
three query heads), batches at the edges of a CTA's threads, empty sequences, both plans."""

import numpy as np
import pytest
import torch

from tests._parity import assert_close
from tests.test_gpu_flat_batches import _batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [33, 255, 257, 513])
@pytest.mark.parametrize("hq,hkv", [(1, 1), (3, 1), (7, 1), (10, 2)])
@pytest.mark.parametrize("scheme,variant", [("int8", "plain"), ("int8", "value"), ("g32", "tier_b"), ("fp8", "plain")])
def test_many_sequences_match_each_alone(batch, hq, hkv, scheme, variant):
    import paper_2607_28699_gb300 as wc
    rng = np.random.default_rng(batch + hq)
    lens = [int(x) for x in rng.integers(1, 60, batch)]
    lens[0] = 16 * 45                       # longer than the block tables that a batch splits
    lens[2] = lens[batch - 2] = 0
    code = {"int8": wc.SCHEME_DITHER_INT8, "g32": wc.SCHEME_DITHER_INT8_G32, "fp8": wc.SCHEME_FP8_E4M3}[scheme]
    desc, table, ctx, q, cache = _batch(lens, code, hq, hkv, variant == "value")

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
    for b in sorted({0, 1, 2, 3, 31, 32, batch // 2, batch - 3, batch - 2, batch - 1}):
        one = decode(q[b:b + 1].contiguous(), table[b:b + 1].contiguous(), ctx[b:b + 1].contiguous())
        for i, (x, y) in enumerate(zip(got, one)):
            assert_close(x[b:b + 1].cpu().numpy(), y.cpu().numpy(), f"output {i} of sequence {b}, {lens[b]} tokens")
