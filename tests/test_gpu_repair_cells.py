"""The repair selection over table sizes and cell counts (few cells take wider CTAs), on
contributions that no bucket spreads: zeros, equal values, infinities and NaN, a few values many
times over.  Order, counts and the remaining sums against a stable sort in numpy; few cells
against many, bit for bit."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _rows(n, rng):
    """Contributions of one page-term row each (d with m = M = 0, L = 1, so C_j = d_j)."""
    spread = rng.lognormal(-6.0, 1.0, n)
    zeros = spread * (rng.random(n) < 0.5)
    few = rng.choice([0.0, 1e-3, 2e-3, 5e-3], n)
    tiny = np.where(rng.random(n) < 0.9, 0.0, 1e-40)         # subnormal beside zero
    infs = np.where(rng.random(n) < 0.3, np.inf, spread)
    nans = np.where(rng.random(n) < 0.3, np.nan, few)
    rows = [spread, zeros, few, np.full(n, 1e-3), np.zeros(n), tiny, infs, nans, np.full(n, np.inf)]
    return [r.astype(np.float32) for r in rows]


def _order(c):
    """Decreasing contribution (NaN above infinity), ties to the lower page."""
    bits = c.view(np.uint32).astype(np.int64)
    return np.argsort(-bits, kind="stable")


def _select(rows, n, max_pages, tau, copies):
    import paper_2607_28699_gb300 as wc
    pt = torch.full((copies, len(rows), max_pages, 2), float("nan"))   # columns past the context are not pages
    pt[:, :, :n, 0] = 0.0
    for i, c in enumerate(rows):
        pt[:, i, :n, 1] = torch.from_numpy(c)
    norm = torch.zeros(copies, len(rows), 2)
    norm[..., 1] = 1.0
    ctx = torch.full((copies,), 16 * n - 3, dtype=torch.int32, device="cuda")
    return wc.repair_select(pt.cuda(), norm.cuda(), ctx, tau)


@pytest.mark.parametrize("max_pages", [1, 31, 32, 33, 64, 65, 128, 129, 256, 257, 512, 513, 1024, 1025, 2048, 2049, 4096,
                                       4097, 8193])
@pytest.mark.parametrize("short", [0, 1])
def test_order_counts_and_sums(max_pages, short):
    n = max(1, max_pages - short)
    rows = _rows(n, np.random.default_rng(max_pages + short))
    for tau in (-1.0, 0.0, 0.02):
        contrib, pages, n_rep, d_after = (x.cpu().numpy() for x in _select(rows, n, max_pages, tau, 1))
        for i, c in enumerate(rows):
            order, k = _order(c), int(n_rep[0, i])
            assert np.array_equal(contrib[0, i, :n], c, equal_nan=True)
            assert np.array_equal(pages[0, i, :k], order[:k]), (i, tau)
            rest = c[order].astype(np.float64)
            if tau < 0:
                assert k == n and d_after[0, i] == 0.0
                continue
            left = rest[k:].sum() if k < n else 0.0
            assert abs(d_after[0, i] - left) <= 1e-5 * max(left, 1e-30)
            assert 0.5 * left * (left + 2.0) <= tau * (1 + 1e-4)             # the list is enough
            if k > 0:                                                        # and one page less is not
                more = left + rest[k - 1]
                assert not 0.5 * more * (more + 2.0) < tau * (1 - 1e-4)
            assert k <= np.count_nonzero(c)                                  # a page that adds nothing is not listed


@pytest.mark.parametrize("max_pages,copies", [(20, 3000), (64, 300), (128, 200), (200, 100), (256, 400), (512, 100), (1000, 60),
                                              (2048, 40), (4096, 30)])
def test_many_cells_select_as_few(max_pages, copies):
    rows = _rows(max_pages, np.random.default_rng(max_pages))
    for tau in (-1.0, 0.02):
        few = _select(rows, max_pages, max_pages, tau, 1)
        many = _select(rows, max_pages, max_pages, tau, copies)
        k = few[2].cpu()
        assert torch.equal(many[2].cpu(), k.expand(copies, -1))
        for at in (0, copies // 2, copies - 1):
            assert torch.equal(many[3][at].cpu().view(torch.int32), few[3][0].cpu().view(torch.int32))   # the same bits
            for i in range(len(rows)):
                assert torch.equal(many[1][at, i, :int(k[0, i])], few[1][0, i, :int(k[0, i])])
