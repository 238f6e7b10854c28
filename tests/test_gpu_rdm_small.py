"""Density matrices of vectors with few or small rows: lookups, unless they are many or a determinant has
many excitations; and the rows of such spaces (no electrons of a spin, one hole, full) against lookups.

The launches tell which way a call went.
"""
import math

import numpy as np
import pytest

from test_gpu_rdm_lone import LOOKUPS, _scan
from test_gpu_rdm_rows import _rdm, _table_bytes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,na,nb,dets,rows", [
    (17, 0, 4, 1190, False),
    (16, 0, 8, 12000, True),      # no alpha electrons
    (12, 12, 4, 250, False),
    (24, 24, 4, 10626, True),     # every orbital alpha
    (20, 7, 0, 300, True),        # no beta electrons
    (9, 4, 0, 120, False),
    (40, 39, 39, 1500, True),     # one hole each
    (10, 9, 9, 90, False),
    (40, 1, 1, 1500, True),
    (10, 1, 4, 1050, False),
    (12, 4, 4, 100000, True),
    (8, 4, 4, 3000, True),
    (8, 4, 4, 300, False),
    (20, 5, 5, 30, True),
])
def test_path(orc, n, na, nb, dets, rows):
    torch = pytest.importorskip("torch")
    import paper_2312_01846_gb300 as sf
    rng = np.random.default_rng(n + dets)
    s = sf.System(n, na, nb, np.eye(n), np.zeros((n,) * 4))
    cb = math.comb(n, nb)
    rank = np.sort(rng.choice(s.dim, dets, replace=False)).astype(np.int64)
    coef = rng.normal(size=dets) * np.exp(-6.0 * rng.random(dets))
    r, c = torch.from_numpy(rank).cuda(), torch.from_numpy(coef).cuda()
    before = sf.kernel_launches()
    st1, p1, q1, n1 = _rdm(sf, torch, s, r, c)
    # by rows: check, norm (2), marks, two scans, places, strings, a scan, pairs, images
    assert sf.kernel_launches() - before == (8 + 2 * _scan(dets) + _scan(cb) if rows else LOOKUPS)
    other = _rdm(sf, torch, s, r, c, _table_bytes(dets))
    if other is None:
        osys = orc.System(n, na, nb, np.zeros((n, n)), np.zeros((n,) * 4))
        other = (0, *orc.rdm12(osys, rank.astype(np.uint64), coef), n1)
    st2, p2, q2, n2 = other
    assert st1 == st2 == 0 and n1 == n2
    np.testing.assert_allclose(p1, p2, rtol=0, atol=1e-12 * np.abs(p2).max())
    np.testing.assert_allclose(q1, q2, rtol=0, atol=1e-12 * np.abs(q2).max())
    s.close()
