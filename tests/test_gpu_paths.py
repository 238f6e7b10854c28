"""Which path a sigma took: by target rows, or the hash table / the buckets.

The tests that compare the paths mean something only while each side takes the
path it is meant to take (sfci_row_sigmas counts those summed by rows).
"""
import numpy as np
import pytest

import gen
import test_gpu_gather as solver
import test_gpu_sigma_rows as single

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2312_01846_gb300 as sf
    sf.lib()
    return sf


def _by_rows(sf, call):
    n0 = sf.row_sigmas()
    out = call()
    return sf.row_sigmas() - n0, out


@pytest.mark.parametrize("name", solver.CASES)
def test_solver(sf, name):
    d, n_keep, kw = solver.CASES[name]
    rows, out = _by_rows(sf, lambda: solver._run(sf, d, n_keep, 3, solver.AUFBAU, **kw))
    assert rows == len(out) + sum(i["redo"] for i, _, _ in out)
    assert _by_rows(sf, lambda: solver._run(sf, d, n_keep, 3, solver.AUFBAU, bucket_elems=1024, **kw))[0] == 0


def test_solver_past_the_limit(sf):
    d = single._molecule(16, 13, 2)
    assert _by_rows(sf, lambda: solver._run(sf, d, 900, 3, solver.AUFBAU))[0] == 0


# (classes: by 20000 determinants its lists fit even then; test_sigma_classes has a longer vector)
@pytest.mark.parametrize("name", [n for n in single.CASES if n != "classes"])
def test_sigma(sf, name):
    d, flags, kw = single.CASES[name]
    kw = {k: v for k, v in kw.items() if k != "scale"}
    s = sf.System.from_dict(d, flags)
    rng = np.random.default_rng(len(name))
    n = min(s.dim, 20000)
    r = np.sort(rng.choice(s.dim, n, replace=False)).astype(np.uint64)
    c = rng.normal(size=n)
    rows, (r1, _) = _by_rows(sf, lambda: single._run(sf, s, r, c, out_cap=1 << 23, **kw))
    assert rows == (0 if name == "past_the_limit" else 1)
    assert _by_rows(sf, lambda: single._run(sf, s, r, c, out_cap=r1.size, **kw))[0] == 0
    s.close()


def test_sigma_classes(sf):
    """Rows summed in classes against the table: 40000 determinants, each row's 5005 strings more than
    one table of sums, and lists of about 470 MB, which 2^24 slots of 32 bytes hold and 2^23 do not."""
    s = sf.System.from_dict(single._molecule(15, 3, 6))
    rng = np.random.default_rng(2)
    r = np.sort(rng.choice(s.dim, 40000, replace=False)).astype(np.uint64)
    c = rng.normal(size=r.size) * np.exp(-12.0 * rng.random(r.size))
    by_rows, (r1, c1) = _by_rows(sf, lambda: single._run(sf, s, r, c, out_cap=1 << 23))
    by_table, (r2, c2) = _by_rows(sf, lambda: single._run(sf, s, r, c, out_cap=r1.size))
    s.close()
    assert (by_rows, by_table) == (1, 0)
    assert np.array_equal(r1, r2) and np.array_equal(c1.view(np.uint64), c2.view(np.uint64))
