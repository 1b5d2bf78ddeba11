"""The grouped write's grids and tasks: the edge between its one-index and its per-head grid,
and between one and two tasks per warp, bypassed channels at the fp16 range, against the
oracle."""

import numpy as np
import pytest
import torch

import workloads as W
from oracle import pipeline as OP
from oracle import quantizer as Q
from tests._parity import descs, gpu_cache_to_numpy, make_inputs, witness_step_up

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tok,m", [(n, m) for n in (15, 16, 17, 31, 33) for m in (0, 1, 16)] + [(8191, 4), (8203, 4)])
def test_grouped_write_bypass_at_the_fp16_range(n_tok, m):
    import paper_2607_28699_gb300 as wc
    wl = W.Workload("gx", 1, 8, 2, [n_tok], shuffle_pages=True, seed=n_tok + m)
    _, sm, k, v, _ = make_inputs(wl, 0)
    k, v = k.numpy().copy(), v.numpy()
    pairs = np.stack([np.arange(h, 64, 4)[:m] for h in range(2)]).astype(np.int64)
    for h in range(2):
        if m:
            d = Q.bypass_dims(pairs[h], 128, Q.ROPE_HALF)
            k[:, h, d] = np.where(np.arange(len(d)) % 2 == 0, 65504.0, -6e-8).astype(np.float16)
    od, gd = descs(8, 2, wl.num_pages, OP.SCHEME_DITHER_INT8_G32, 8, 0, 5, num_bypass_pairs=m)
    ref = OP.empty_cache(od)
    OP.write_tokens(od, 0, k, v, sm, ref, bypass_pairs=pairs if m else None)
    cache = wc.LayerCache.empty(gd, num_bypass_pairs=m)
    if m:
        cache.bypass_pairs.copy_(torch.from_numpy(pairs.astype(np.int32)))
    wc.kv_quantize_witness(gd, 0, torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda(),
                           torch.from_numpy(sm).cuda(), cache)
    got = gpu_cache_to_numpy(cache)
    for name in ("k_codes", "v_codes", "k_scale", "v_scale") + (("k_bypass",) if m else ()):
        assert np.array_equal(got[name].view(np.uint8), ref[name].view(np.uint8)), name
    w, up = ref["k_witness"], witness_step_up(ref["k_witness"])
    assert np.all((got["k_witness"] == w) | (got["k_witness"] == up))
