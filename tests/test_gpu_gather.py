"""Sigma by target rows against the bucketed path.

The solver sums sigma by target rows unless the caller shapes the bucketed path
(here: bucket_elems).  Both sum every entry exactly and round once, and the dots
and the truncation that follow are the same kernels, so the kept vectors and the
scalars a and b must agree bit for bit.  The systems sit at the edges of the row
path: no, one or all orbitals of a spin occupied (no pairs, no hops), spaces
smaller and larger than one table, rows that are summed in classes and classes
that split, long runs of sources sharing a string and lone ones, the ring's
zero integrals, float32 elements, both screens, and a vector replaced mid-cycle.
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


def _run(sf, d, n_keep, steps, init, flags=0, **kw):
    s = sf.System.from_dict(d, flags)
    lz = sf.Lanczos(s, *init, n_keep, n_lanczos=5, **kw)
    out = []
    for k in range(steps):
        if k == 2:  # the same w_i handed back: its row pointers must be found again
            lz.set_input(*lz.vector())
        info = lz.step()
        r, c = lz.vector()
        out.append((info, sf.to_u64(r), c.cpu().numpy()))
    lz.close()
    s.close()
    return out


AUFBAU = (np.array([0], dtype=np.uint64), np.array([1.0]))
CASES = {
    "no_beta_pairs": (_molecule(10, 3, 1), 300, {}),
    "one_electron_each": (_molecule(10, 1, 1), 300, {}),
    "no_alpha": (_molecule(10, 0, 2), 300, {}),
    "no_beta": (_molecule(10, 2, 0), 300, {}),
    "full_alpha": (_molecule(10, 10, 3), 300, {}),
    "one_hole_each": (_molecule(10, 9, 9), 300, {}),
    "most_electrons": (_molecule(16, 12, 3), 900, {}),
    "whole_space": (gen.config_system(0), 4900, {}),
    "one_table": (_molecule(15, 4, 5), 2500, {}),           # C(15, 5) = 3003 < 4096 slots
    "just_past_one_table": (_molecule(15, 5, 6), 2500, {}),  # C(15, 6) = 5005
    "classes": (gen.config_system(4), 4000, {}),
    "classes_long_vector": (gen.batched_scan_instances()[5], 20000, {}),
    "ring": (gen.config_system(1), 3000, {}),
    "ring_screened": (gen.config_system(1), 3000, {"eps_screen": 5e-5}),
    "float32": (gen.config_system(4), 1500, {"flags": 1}),
    "element_screen": (gen.config_system(4), 1500, {"eps_element": 1e-4}),
}


@pytest.mark.parametrize("name", CASES)
def test_rows_equal_buckets(sf, name):
    d, n_keep, kw = CASES[name]
    rows = _run(sf, d, n_keep, 6, AUFBAU, **kw)
    buckets = _run(sf, d, n_keep, 6, AUFBAU, bucket_elems=1024, **kw)
    for k, ((i1, r1, c1), (i2, r2, c2)) in enumerate(zip(rows, buckets)):
        assert np.array_equal(r1, r2), (name, k)
        assert np.array_equal(c1.view(np.uint64), c2.view(np.uint64)), (name, k)
        for key in ("a", "b", "lambda_min", "n_kept", "n_in", "n_elements", "n_alpha_runs"):
            assert i1[key] == i2[key], (name, k, key)
        if not kw:  # (the ring's zero products and screened ones are counted by the buckets alone)
            assert i1["n_sigma"] == i2["n_sigma"], (name, k)


def test_scattered_sources(sf):
    """Lone sources: one determinant per alpha string, drawn over the whole space."""
    d = gen.config_system(4)
    a, b = gen.random_dets(d["n"], d["na"], d["nb"], 1500, seed=3)[:2]
    a, i = np.unique(a, return_index=True)
    s = sf.System.from_dict(d)
    r = np.sort(sf.to_u64(sf.sfci_rank(s, a, b[i])))
    s.close()
    c = np.random.default_rng(4).normal(size=r.size)
    rows = _run(sf, d, 1500, 2, (r, c))
    buckets = _run(sf, d, 1500, 2, (r, c), bucket_elems=1024)
    for (i1, r1, c1), (i2, r2, c2) in zip(rows, buckets):
        assert np.array_equal(r1, r2) and np.array_equal(c1.view(np.uint64), c2.view(np.uint64))
        assert (i1["a"], i1["n_sigma"]) == (i2["a"], i2["n_sigma"])
