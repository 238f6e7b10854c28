"""Unranking at the edges: no, one or all orbitals occupied, 64 orbitals, string counts on both
sides of 32 bits.  Whole numbers: the first, last and drawn ranks come back exactly, and the
strings have the index that the combinatorial number system gives them."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,na,nb", [(1, 1, 0), (5, 0, 5), (28, 7, 7), (35, 16, 3), (36, 18, 3), (64, 1, 63), (64, 7, 6)])
def test_unrank_edges(n, na, nb):
    torch = pytest.importorskip("torch")
    import paper_2312_01846_gb300 as sf
    s = sf.System(n, na, nb, np.eye(n), np.zeros((n,) * 4))
    rng = np.random.default_rng(n)
    ranks = {0, s.dim - 1, s.dim // 2} | {int(x * s.dim) for x in rng.random(500)}
    ranks = np.array(sorted(r for r in ranks if r < s.dim), dtype=np.uint64)
    a, b = (sf.to_u64(x) for x in sf.sfci_unrank(s, torch.from_numpy(ranks.view(np.int64)).cuda()))
    for r, x, y in zip(ranks, a, b):
        h = [sum(math.comb(p, k + 1) for k, p in enumerate(q for q in range(n) if int(v) >> q & 1)) for v in (x, y)]
        assert bin(int(x)).count("1") == na and bin(int(y)).count("1") == nb
        assert h[0] * math.comb(n, nb) + h[1] == int(r)
    s.close()
