"""The pair calibration's wide cluster (4096 rows and more, 16-byte aligned keys) against
the narrow one, which keys that are only 8-byte aligned take at any length: the same
pairs on ragged row counts, with equal energies and with infinities."""

import numpy as np
import pytest
import torch

from oracle import quantizer as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", [Q.ROPE_HALF, Q.ROPE_INTERLEAVED])
@pytest.mark.parametrize("n,hkv", [(4095, 2), (4096, 3), (4097, 1), (8191, 9), (8449, 2)])
def test_wide_cluster_selects_the_narrow_ones_pairs(n, hkv, layout):
    import paper_2607_28699_gb300 as wc
    g = torch.Generator().manual_seed(n + hkv)
    k = torch.randn(n, hkv, 128, generator=g).half()
    last = n - 1
    k[:, :, 40] = k[:, :, 2]                      # equal channels: half layout pairs 2 and 40
    k[last, hkv - 1, 77] = 3000.0                 # decided by the last row alone
    if hkv > 1:
        k[0, 0, 5] = float("inf")
        k[n // 2, 0, 9] = float("nan")
    room = torch.empty(k.numel() + 4, dtype=torch.float16, device="cuda")
    aligned = k.cuda()
    shifted = room[4:].view(n, hkv, 128)
    shifted.copy_(aligned)
    assert aligned.data_ptr() % 16 == 0 and shifted.data_ptr() % 16 == 8
    for m in (1, 4, 16):
        wide = torch.full((hkv, m), -7, dtype=torch.int32, device="cuda")
        narrow = wide.clone()
        wc.select_bypass_pairs(aligned, m, layout, pairs=wide)
        wc.select_bypass_pairs(shifted, m, layout, pairs=narrow)
        assert torch.equal(wide, narrow)
        h = hkv - 1                               # finite in every case
        x = k[:, h].double().numpy()
        dims = Q.bypass_dims(np.arange(64), 128, layout).reshape(64, 2)
        e = np.sum(x[:, dims[:, 0]] ** 2 + x[:, dims[:, 1]] ** 2, axis=0)
        got = wide[h].cpu().numpy()
        # fp32 sums of n terms in 256 chains: n / 256 + 48 roundings at most
        assert e[got].min() >= np.delete(e, got).max() * (1 - (n / 256 + 48) * 2.0 ** -23)
