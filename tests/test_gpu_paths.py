"""Which path a sigma took: by target rows, or the hash table / the buckets.

The tests that compare the paths mean something only while each side takes the
path it is meant to take (sfci_row_sigmas counts those summed by rows).
"""
import math

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


# a batch, where the others' work hides what the buckets wait for
@pytest.mark.parametrize("n,na,nb,dets,alone,beside", [
    (24, 7, 0, 400, 1, 0),      # elements of one spin
    (24, 10, 10, 50, 1, 0),     # 2e6 rows for 50 determinants
    (24, 8, 8, 8, 1, 1),
    (14, 4, 4, 500, 1, 1),
])
def test_scan_takes_the_faster_path(sf, n, na, nb, dets, alone, beside):
    d = single._molecule(n, na, nb)
    r, c = _rows_vector(d, min(3 * dets, math.comb(n, na)), dets)
    out = []
    for workers, want in ((1, alone), (2, beside)):
        systems = [sf.System.from_dict(d) for _ in range(2)]
        scan = sf.Scan([(s, r, c, dets) for s in systems], n_lanczos=3, workers=workers)
        rows, infos = _by_rows(sf, scan.step)
        assert rows == (2 + sum(i["redo"] for i in infos) if want else 0)
        for i in range(2):
            rk, cf = scan.vector(i)
            out.append((infos[i]["a"], sf.to_u64(rk), cf.cpu().numpy().view(np.uint64)))
        scan.close()
        for s in systems:
            s.close()
    for a, rk, cf in out[1:]:
        assert a == out[0][0] and np.array_equal(rk, out[0][1]) and np.array_equal(cf, out[0][2])


def _restarts(sf, d, init, count, **kw):
    """Rows taken and launches of `count` restarts from one vector, and the last step's vector."""
    s = sf.System.from_dict(d)
    lz = sf.Lanczos(s, *init, max(len(init[0]), 100), n_lanczos=3, **kw)
    rows, launches = [], []
    for _ in range(count):
        lz.load(*init)
        n0, l0 = sf.row_sigmas(), sf.kernel_launches()
        info = lz.step()
        rows.append(sf.row_sigmas() - n0)
        launches.append(sf.kernel_launches() - l0)
    r, c = lz.vector()
    lz.close()
    s.close()
    return rows, launches, (info["a"], sf.to_u64(r), c.cpu().numpy().view(np.uint64))


def _rows_vector(d, rows, n, seed=4):
    """n determinants spread over `rows` alpha strings."""
    ca, cb = math.comb(d["n"], d["na"]), math.comb(d["n"], d["nb"])
    rng = np.random.default_rng(seed)
    a = rng.choice(ca, rows, replace=False)
    r = np.unique(rng.choice(a, 2 * n).astype(np.uint64) * np.uint64(cb) + rng.integers(0, cb, 2 * n).astype(np.uint64))
    r = np.sort(rng.choice(r, n, replace=False))
    return r, rng.normal(size=n)


# what pays by rows and what does not: a space of many rows takes a long vector, and heavy rows
# may not outnumber the excitations of a string by their classes
@pytest.mark.parametrize("n,na,nb,rows,dets,by_rows", [
    (28, 12, 2, 5, 30, 0),        # 3e7 rows for 30 determinants
    (26, 10, 3, 100, 300, 0),     # 5e6 rows, few elements
    (28, 1, 9, 8, 20000, 0),      # 2500 determinants to a row, 2000 classes
    (24, 0, 12, 1, 34000, 0),     # one row
    (28, 7, 0, 6000, 3000, 0),    # no opposite-spin elements
    (30, 1, 3, 7, 8000, 0),       # 30 rows, one class each
    (20, 5, 5, 500, 1000, 1),
    (28, 7, 7, 20, 30, 1),        # 1e6 rows
    (24, 1, 7, 6, 20000, 1),      # heavy rows of few classes
])
def test_solver_takes_the_faster_path(sf, n, na, nb, rows, dets, by_rows):
    d = single._molecule(n, na, nb)
    init = _rows_vector(d, rows, dets)
    got, launches, out = _restarts(sf, d, init, 5)
    _, want_launches, want = _restarts(sf, d, init, 5, emit_warps=8)
    assert got == [by_rows] * 5
    if not by_rows:  # and nothing is prepared again for a plan that did not pay (the order in which
        # the stream fills may cost either an attempt more)
        assert min(launches[1:]) <= min(want_launches[1:])
    assert out[0] == want[0] and np.array_equal(out[1], want[1]) and np.array_equal(out[2], want[2])


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


def test_solver_takes_rows_for_its_vectors(sf):
    """The vectors of a solver's own first steps, whose sources share beta strings: planned as if they
    were scattered, the second has 1.9 visits an element (0.3 in truth: 6 ms by rows, 10 by buckets)."""
    s = sf.System.from_dict(single._molecule(28, 2, 9))
    lz = sf.Lanczos(s, np.zeros(1, dtype=np.uint64), np.ones(1), 16000, n_lanczos=3)
    rows, infos = _by_rows(sf, lambda: [lz.step() for _ in range(2)])
    lz.close()
    s.close()
    assert infos[1]["n_in"] > 15000
    assert rows == 2 + sum(i["redo"] for i in infos)


# the standalone sigma: few elements a source, elements of one spin (both while the table is small),
# and heavy rows whose classes visit sources more than twice as often as there are elements
@pytest.mark.parametrize("n,na,nb,rows,dets,caps,by_rows", [
    (28, 1, 1, 28, 300, (1 << 19, (1 << 19) + 1), (0, 1)),
    (40, 1, 1, 40, 300, (1 << 19, 1 << 20), (1, 1)),
    (28, 7, 0, 6000, 1000, (1 << 22, (1 << 22) + 1), (0, 1)),
    (24, 0, 12, 1, 2000, (1 << 22, (1 << 22) + 1), (0, 1)),
    (24, 0, 12, 1, 300, (1 << 21, 1 << 22), (1, 1)),
    (28, 1, 7, 28, 3000, (18500000, 1 << 25), (1, 1)),
    (28, 1, 9, 28, 5000, (48000000, 50000000), (1, 1)),
    (28, 1, 9, 28, 12000, (110000000, 120000000), (0, 0)),
])
def test_sigma_takes_the_faster_path(sf, n, na, nb, rows, dets, caps, by_rows):
    s = sf.System.from_dict(single._molecule(n, na, nb))
    r, c = _rows_vector(dict(n=n, na=na, nb=nb), rows, dets)
    out = []
    for cap, want in zip(caps, by_rows):
        took, (rk, cf) = _by_rows(sf, lambda: sf.sfci_sigma(s, r, c, out_cap=cap))
        assert took == want, cap
        out.append((sf.to_u64(rk), cf.cpu().numpy().view(np.uint64)))
    s.close()
    (r1, c1), (r2, c2) = out
    assert np.array_equal(r1, r2) and np.array_equal(c1, c2)


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
