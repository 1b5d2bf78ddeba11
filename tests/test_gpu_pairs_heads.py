"""Pair selection on both sides of what decides its cluster (csrc/dispatch.h): rows, heads and
the alignment of k.  The pairs are those of the largest energies in float64."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [1, 14, 15, 16, 32])
@pytest.mark.parametrize("rows", [4095, 4096])
@pytest.mark.parametrize("rope", [0, 1])
@pytest.mark.parametrize("offset", [0, 4])                  # in elements: 16-byte or 8-byte aligned
def test_pairs_are_the_largest_energies(heads, rows, rope, offset):
    import paper_2607_28699_gb300 as wc
    g = torch.Generator().manual_seed(rows + heads)
    flat = torch.empty(rows * heads * 128 + 8, dtype=torch.float16, device="cuda")
    k = flat[offset:offset + rows * heads * 128].view(rows, heads, 128)
    scale = 1.0 + 0.05 * torch.stack([torch.randperm(128, generator=g) for _ in range(heads)]).float()
    k.copy_((torch.randn(rows, heads, 128, generator=g) * scale).half())
    assert k.data_ptr() % 16 == 2 * offset
    e = (k.double() ** 2).sum(0)
    pair = e[:, :64] + e[:, 64:] if rope == wc.ROPE_HALF else e[:, 0::2] + e[:, 1::2]
    want = pair.topk(5, dim=1).indices.sort(dim=1).values.int()
    assert torch.equal(wc.select_bypass_pairs(k, 5, rope), want)
