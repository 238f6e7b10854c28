"""Density matrices from pairs met by rows against those from lookups.

A workspace just large enough for the lookups' table makes the library take them
(where the rows' buffers are smaller than that, the oracle takes their place).
Both add the same products, in any order: they agree to the rounding of sums of
products bounded by |c|^2 (1e-12 of the largest element, as against the oracle).
"""
import ctypes as C
import math

import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


def _table_bytes(m):
    slots = 1024
    while slots < 2 * m:
        slots *= 2
    return slots * 16 + 256 * 3 + (152 * 8 + 255) // 256 * 256


def _rdm(sf, torch, s, r, c, nbytes=None):
    nb = C.c_size_t()
    assert sf.lib().sfci_rdm12_workspace_bytes(s.handle, r.numel(), C.byref(nb)) == 0
    if nbytes is not None and nbytes >= nb.value:
        return None
    ws = torch.empty(nbytes or nb.value, dtype=torch.uint8, device="cuda")
    g1 = torch.full((s.n,) * 2, np.nan, dtype=torch.float64, device="cuda")
    g2 = torch.full((s.n,) * 4, np.nan, dtype=torch.float64, device="cuda")
    nrm = C.c_double()
    st = sf.lib().sfci_rdm12(s.handle, r.data_ptr(), c.data_ptr(), r.numel(), g1.data_ptr(), g2.data_ptr(),
                             C.byref(nrm), ws.data_ptr(), ws.numel(), None)
    return st, g1.cpu().numpy(), g2.cpu().numpy(), nrm.value


# orbitals, electrons, alpha strings with many determinants, lone determinants
CASES = {
    "dense": (8, 4, 4, 12, 0),
    "no_alpha": (9, 0, 4, 1, 0),
    "no_beta": (9, 4, 0, 126, 0),
    "one_each": (10, 1, 1, 4, 20),
    "full_alpha": (9, 9, 4, 1, 0),
    "one_hole_each": (10, 9, 9, 6, 12),
    "several_batches_of_hops": (14, 5, 3, 60, 4000),
    "row_longer_than_the_table": (15, 2, 6, 3, 3000),  # C(15, 6) = 5005 determinants a row
    "lone": (20, 5, 5, 0, 3000),
    "many_electrons": (17, 14, 13, 5, 2000),
    "sixty_four_orbitals": (64, 2, 2, 2, 900),
}


@pytest.mark.parametrize("name", CASES)
def test_rows_equal_lookups(orc, name):
    torch = pytest.importorskip("torch")
    import paper_2312_01846_gb300 as sf
    n, na, nb, full, lone = CASES[name]
    rng = np.random.default_rng(len(name))
    s = sf.System(n, na, nb, np.eye(n), np.zeros((n,) * 4))
    cb = math.comb(n, nb)
    rank = [np.arange(cb, dtype=np.int64)[rng.random(cb) < 0.97] + a * cb for a in range(full)]
    rank = np.unique(np.concatenate(rank + [rng.integers(0, s.dim, lone)]))
    coef = rng.normal(size=rank.size) * np.exp(-6.0 * rng.random(rank.size))
    coef[rng.random(rank.size) < 0.03] = 0.0
    r, c = torch.from_numpy(rank).cuda(), torch.from_numpy(coef).cuda()
    st1, p1, q1, n1 = _rdm(sf, torch, s, r, c)
    other = _rdm(sf, torch, s, r, c, _table_bytes(rank.size))
    if other is None:
        osys = orc.System(n, na, nb, np.zeros((n, n)), np.zeros((n,) * 4))
        other = (0, *orc.rdm12(osys, rank.astype(np.uint64), coef), n1)
    st2, p2, q2, n2 = other
    assert st1 == st2 == 0 and n1 == n2
    np.testing.assert_allclose(p1, p2, rtol=0, atol=1e-12 * np.abs(p2).max())
    np.testing.assert_allclose(q1, q2, rtol=0, atol=1e-12 * np.abs(q2).max())
    # ranks out of order or beyond the space are refused
    for bad in (r.flip(0).contiguous(), torch.cat([r[:-1], torch.tensor([s.dim], device="cuda")])):
        if rank.size > 1:
            assert _rdm(sf, torch, s, bad, c)[0] == sf.SFCI_E_INVALID
    s.close()
