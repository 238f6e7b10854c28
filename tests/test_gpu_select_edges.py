"""Truncation and radix sort at the edges of their tiles and of the one-CTA paths.

Both move values without arithmetic, so ranks and values are exact; the norm may
be summed in another order than numpy's, which moves a quotient by a few ulp.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TILE, SMALL = 2048, 8192


@pytest.mark.parametrize("n", [1, 31, 1024, TILE + 1, SMALL - 1, SMALL, SMALL + 1, 40 * TILE, 300007])
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0, 1.7])
@pytest.mark.parametrize("values", ["spread", "ties", "zeros"])
def test_truncate_exact(n, share, values):
    torch = pytest.importorskip("torch")
    import paper_2312_01846_gb300 as sf
    rng = np.random.default_rng(n + int(10 * share) + len(values))
    k = max(1, int(share * n))
    # high digits that all ranks share, and ranks beyond 2^32
    rank = rng.permutation(n).astype(np.uint64) * np.uint64(77777) + np.uint64(5 << 40)
    coef = rng.choice([-1.0, 1.0], n) * np.exp(-30.0 * rng.random(n))
    if values == "ties":
        coef = rng.choice([-0.5, 0.25, 0.5, 3e-310], n)
    if values == "zeros":
        coef[rng.random(n) < 0.6] = 0.0
        coef[rng.random(n) < 0.1] = -0.0
    live = np.nonzero(coef)[0]
    order = live[np.lexsort((rank[live], -np.abs(coef[live])))][:k]
    order = order[np.argsort(rank[order])]
    r = torch.from_numpy(rank.view(np.int64)).cuda()
    c = torch.from_numpy(coef).cuda()
    gr, gv = sf.sfci_truncate_topk(r, c, k, normalize=False)
    assert np.array_equal(gr.cpu().numpy().view(np.uint64), rank[order])
    assert np.array_equal(gv.cpu().numpy(), coef[order])
    gr, gv = sf.sfci_truncate_topk(r, c, k, normalize=True)
    assert np.array_equal(gr.cpu().numpy().view(np.uint64), rank[order])
    norm = np.sqrt(np.sum(coef[order] ** 2))
    if norm > 0:
        # a norm of non-negative terms summed in any order: relative error <= n * 2^-53
        np.testing.assert_allclose(gv.cpu().numpy(), coef[order] / norm, rtol=(n + 4) * 2.0 ** -52, atol=1e-320)


@pytest.mark.parametrize("n", [5, SMALL, SMALL + 1])
def test_nothing_asked_for(n):
    """k = 0 keeps nothing, whatever the values."""
    torch = pytest.importorskip("torch")
    import paper_2312_01846_gb300 as sf
    c = torch.full((n,), float("inf"), dtype=torch.float64, device="cuda")
    r, v = sf.sfci_truncate_topk(torch.arange(n, device="cuda"), c, 0, normalize=False)
    assert r.numel() == 0 and v.numel() == 0
