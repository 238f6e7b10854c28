"""sigma = H psi by target rows against the hash table.

The standalone sigma sums by target rows when the lists fit in the workspace's
table space, which grows with out_cap: with out_cap just at the number of entries
a small space's lists do not fit (many elements to each entry) and the table is
used, with a large out_cap they do.  Both sum exactly and round once: ranks and
values agree bit for bit.
"""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2312_01846_gb300 as sf
    sf.lib()
    return sf


def _molecule(n, na, nb, seed=9):
    return dict(gen.molecular_integrals(n, 16, seed=seed), n=n, na=na, nb=nb)


def _run(sf, s, r, c, **kw):
    gr, gc = sf.sfci_sigma(s, r, c, **kw)
    return sf.to_u64(gr), gc.cpu().numpy()


CASES = {
    "no_beta_pairs": (_molecule(10, 3, 1), 0, {}),
    "no_alpha": (_molecule(10, 0, 2), 0, {}),
    "no_beta": (_molecule(10, 2, 0), 0, {}),
    "full_alpha": (_molecule(10, 10, 3), 0, {}),
    "one_hole_each": (_molecule(10, 9, 9), 0, {}),
    "past_the_limit": (_molecule(16, 13, 2), 0, {}),  # more electrons than the row path takes
    "whole_space": (gen.config_system(0), 0, {}),
    "classes": (_molecule(15, 3, 6), 0, {}),
    "ring": (gen.config_system(1), 0, {}),
    "ring_screened": (gen.config_system(1), 0, {"eps_screen": 1e-3}),
    "float32": (_molecule(12, 3, 4), 1, {}),
    "tiny_values": (_molecule(11, 3, 3), 0, {"scale": 1e-280}),
}


@pytest.mark.parametrize("name", CASES)
def test_rows_equal_table(sf, name):
    d, flags, kw = CASES[name]
    kw = dict(kw)
    scale = kw.pop("scale", 1.0)
    s = sf.System.from_dict(d, flags)
    rng = np.random.default_rng(len(name))
    n = min(s.dim, 20000)
    r = np.sort(rng.choice(s.dim, n, replace=False)).astype(np.uint64)
    c = rng.normal(size=n) * np.exp(-12.0 * rng.random(n)) * scale
    c[rng.random(n) < 0.05] = 0.0
    r1, c1 = _run(sf, s, r, c, out_cap=1 << 23, **kw)
    r2, c2 = _run(sf, s, r, c, out_cap=r1.size, **kw)
    s.close()
    assert np.all(np.diff(r1.astype(np.int64)) > 0)
    assert np.array_equal(r1, r2), name
    assert np.array_equal(c1.view(np.uint64), c2.view(np.uint64)), name


def test_capacity_and_refusals(sf):
    """One entry too few is a capacity error that names the count; bad inputs are refused as before."""
    s = sf.System.from_dict(gen.config_system(4))
    r, c = np.arange(0, 900, 300).astype(np.uint64), np.array([1.0, -0.5, 0.25])
    full, _ = _run(sf, s, r, c)
    exact, _ = _run(sf, s, r, c, out_cap=full.size)
    assert np.array_equal(full, exact)
    for bad in (dict(rank=r, coef=c, out_cap=full.size // 4), dict(rank=r[::-1].copy(), coef=c),
                dict(rank=np.array([0, 1, s.dim], dtype=np.uint64), coef=c),
                dict(rank=r, coef=np.array([1.0, np.inf, 0.0]))):
        cap = bad.pop("out_cap", None)
        if cap:  # grown by the caller until it fits
            grown, _ = _run(sf, s, r, c, out_cap=cap)
            assert np.array_equal(full, grown)
        else:
            with pytest.raises(sf.SfciError):
                _run(sf, s, bad["rank"], bad["coef"])
    s.close()
