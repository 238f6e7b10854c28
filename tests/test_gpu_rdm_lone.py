"""Density matrices of vectors whose rows hold a determinant each and whose opposite-spin
excitations are few: lookups, not a row's units that find nothing.

How many units the rows have is counted on the device.  The launches tell which way it went.
"""
import math

import numpy as np
import pytest

from test_gpu_rdm_rows import _rdm, _table_bytes

pytestmark = pytest.mark.gpu


LOOKUPS = 6  # check, norm (2), the table cleared and filled, lookups


def _scan(m):  # launches of a scan
    return 1 if m <= 8192 else 3


@pytest.mark.parametrize("nb,rows,dets,lookups", [
    (0, 5000, 5000, True),
    (28, 5000, 5000, True),     # no beta hops either
    (0, 300, 300, False),
    (1, 60000, 60000, True),
    (27, 60000, 60000, True),
    (1, 3000, 60000, False),    # 20 determinants to a row
    (1, 3000, 3000, False),     # too few for the lookups' warps
    (3, 60000, 60000, False),   # many opposite-spin lookups
])
def test_lone_rows(orc, nb, rows, dets, lookups):
    torch = pytest.importorskip("torch")
    import paper_2312_01846_gb300 as sf
    n, na = 28, 7
    rng = np.random.default_rng(nb)
    s = sf.System(n, na, nb, np.eye(n), np.zeros((n,) * 4))
    ca, cb = math.comb(n, na), math.comb(n, nb)
    a = rng.choice(ca, rows, replace=False)
    b = np.concatenate([rng.choice(cb, dets // rows, replace=False) for _ in range(rows)])
    rank = np.sort(np.repeat(a, dets // rows) * cb + b)
    coef = rng.normal(size=rank.size) * np.exp(-6.0 * rng.random(rank.size))
    r, c = torch.from_numpy(rank).cuda(), torch.from_numpy(coef).cuda()
    count = [sf.kernel_launches()]
    st1, p1, q1, n1 = _rdm(sf, torch, s, r, c)
    count.append(sf.kernel_launches())
    other = _rdm(sf, torch, s, r, c, _table_bytes(rank.size))
    count.append(sf.kernel_launches())
    first, forced = count[1] - count[0], count[2] - count[1]
    if cb == 1:  # no row can hold two: known without counting, and no more memory is asked for
        assert (other is None) == lookups
        assert first == (LOOKUPS if lookups else 8 + 2 * _scan(rank.size) + _scan(cb))
        osys = orc.System(n, na, nb, np.zeros((n, n)), np.zeros((n,) * 4))
        other = (0, *orc.rdm12(osys, rank.astype(np.uint64), coef), n1)
    else:
        # by rows: check, norm (2), marks, two scans, places, strings, a scan, pairs, images
        before = 6 + _scan(rank.size) + _scan(cb)
        assert forced == LOOKUPS and first == before + (forced if lookups else 2 + _scan(rank.size))
    st2, p2, q2, n2 = other
    assert st1 == st2 == 0 and n1 == n2
    np.testing.assert_allclose(p1, p2, rtol=0, atol=1e-12 * np.abs(p2).max())
    np.testing.assert_allclose(q1, q2, rtol=0, atol=1e-12 * np.abs(q2).max())
    # ranks out of order or beyond the space are refused
    for bad in (r.flip(0).contiguous(), torch.cat([r[:-1], torch.tensor([s.dim], device="cuda")])):
        assert _rdm(sf, torch, s, bad, c)[0] == sf.SFCI_E_INVALID
    s.close()
