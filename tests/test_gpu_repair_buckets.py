"""The repair selection's bucket sort where it can go wrong: keys that share a
bucket, as many as it takes and one more (then the network sorts), a range
stretched by one large page, contexts that end inside the block table."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

MAX_BUCKET = 64   # kMaxBucket of csrc/repair_kernel.cu


def _rows(n, rng):
    spread = rng.lognormal(-6.0, 1.0, n)
    far = spread.copy()
    far[n // 2] = 1e30                                  # every other page in a few buckets
    rows = [spread, far]
    for tied in (MAX_BUCKET, MAX_BUCKET + 1):
        r = rng.lognormal(-6.0, 1.0, n)
        r[rng.permutation(n)[:tied]] = 1e-3
        rows.append(r)
    steps = 1e-3 * (1.0 + 2.0 ** -23 * rng.permutation(n))   # neighbouring floats: one bucket each or two
    rows.append(steps)
    return [x.astype(np.float32) for x in rows]


@pytest.mark.parametrize("max_pages", [3, 511, 512, 700, 2048, 4097, 16384])
@pytest.mark.parametrize("short", [0, 2])
def test_order_is_by_contribution_then_page(max_pages, short):
    import paper_2607_28699_gb300 as wc
    n = max_pages - short
    rows = _rows(n, np.random.default_rng(max_pages + short))
    pt = torch.full((1, len(rows), max_pages, 2), float("nan"))        # columns past the context are not read as pages
    norm = torch.zeros(1, len(rows), 2)
    norm[..., 1] = 1.0
    for i, c in enumerate(rows):
        pt[0, i, :n, 0] = 0.0
        pt[0, i, :n, 1] = torch.from_numpy(c)
    ctx = torch.tensor([16 * n - 5], dtype=torch.int32, device="cuda")
    contrib, pages, n_rep, d_after = wc.repair_select(pt.cuda(), norm.cuda(), ctx, 0.0)
    for i, c in enumerate(rows):
        assert torch.equal(contrib[0, i, :n].cpu(), torch.from_numpy(c))
        assert int(n_rep[0, i]) == n and float(d_after[0, i]) == 0.0    # tau = 0: every page
        assert np.array_equal(pages[0, i, :n].cpu().numpy(), np.argsort(-c.astype(np.float64), kind="stable"))
