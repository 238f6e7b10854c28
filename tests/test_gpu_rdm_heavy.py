"""Density matrices of vectors with one long row: lookups, not comparisons within it.

Pairs within a row are found by comparing all of it, which lookups beat once most
determinants share a row of more than about 1e5.  Whether a vector that long is
spread over its rows is counted on the device.  The launches tell which way it went.
"""
import math

import numpy as np
import pytest

from test_gpu_rdm_rows import _rdm, _table_bytes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,lookups", [(1, True), (2, False), (20, False)])
def test_one_long_row(rows, lookups):
    torch = pytest.importorskip("torch")
    import paper_2312_01846_gb300 as sf
    n, na, nb, dets = 20, 1, 10, 130000  # rows of up to 184756; 26 pairs per excitation: 59346 a determinant
    rng = np.random.default_rng(rows)
    s = sf.System(n, na, nb, np.eye(n), np.zeros((n,) * 4))
    cb = math.comb(n, nb)
    rank = np.sort(np.concatenate([a * cb + rng.choice(cb, dets // rows, replace=False) for a in range(rows)]))
    coef = rng.normal(size=rank.size) * np.exp(-6.0 * rng.random(rank.size))
    r, c = torch.from_numpy(rank).cuda(), torch.from_numpy(coef).cuda()
    count = [sf.kernel_launches()]
    st1, p1, q1, n1 = _rdm(sf, torch, s, r, c)
    count.append(sf.kernel_launches())
    st2, p2, q2, n2 = _rdm(sf, torch, s, r, c, _table_bytes(rank.size))
    count.append(sf.kernel_launches())
    s.close()
    first, forced = count[1] - count[0], count[2] - count[1]
    # by rows: check, norm (2), marks, two scans (3 each), places, strings, a scan (3), pairs, images
    assert first == (12 + forced if lookups else 17)
    assert st1 == st2 == 0 and n1 == n2
    np.testing.assert_allclose(p1, p2, rtol=0, atol=1e-12 * np.abs(p2).max())
    np.testing.assert_allclose(q1, q2, rtol=0, atol=1e-12 * np.abs(q2).max())
