"""A solver whose target-row lists do not fit in memory takes the buckets.

It gives the same vectors as a solver that takes the buckets from the start,
within the same share of memory, and holds no buffer of the path it left.
share and alloc_limit stand in for a device that is nearly full (no test fills
one).  20 orbitals, 4000 determinants: the rows take about 0.3 GB, the elements
of the buckets 0.5 GB, in as many passes as the share asks for.
"""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu
SHARE = 260_000_000  # above the rows' first two stages, below all of them
KEEP, SHORT = 4000, 200


@pytest.fixture(scope="module")
def sf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2312_01846_gb300 as sf
    sf.lib()
    return sf


@pytest.fixture(scope="module")
def inputs(sf):
    s = sf.System.from_dict(gen.config_system(4))
    rng = np.random.default_rng(11)
    vecs = {}
    for n in (KEEP, SHORT):
        r = np.sort(rng.choice(s.dim, n, replace=False)).astype(np.uint64)
        vecs[n] = r, rng.normal(size=n)
    yield s, vecs
    s.close()


def _solver(sf, inputs, share=0, alloc_limit=0, **kw):
    s, vecs = inputs
    lz = sf.Lanczos(s, *vecs[KEEP], KEEP, n_lanczos=4, **kw)
    lz.debug_memory(share=share, alloc_limit=alloc_limit)
    return lz


def _step(sf, lz, vec):
    """(rows or not, launches, a, vector) of one restart and step."""
    lz.load(*vec)
    n0, l0 = sf.row_sigmas(), sf.kernel_launches()
    info = lz.step()
    n1, l1 = sf.row_sigmas(), sf.kernel_launches()
    r, c = lz.vector()
    return n1 - n0, l1 - l0, info["a"], sf.to_u64(r), c.cpu().numpy().view(np.uint64)


def _same(x, y):
    return x[2] == y[2] and np.array_equal(x[3], y[3]) and np.array_equal(x[4], y[4])


@pytest.mark.parametrize("alloc_limit", [500_000, 4_000_000, 30_000_000, 62_000_000])
def test_out_of_memory(sf, inputs, alloc_limit):
    """An allocation of the row path that fails, at each of its stages, is no error."""
    _, vecs = inputs
    lz, ref = _solver(sf, inputs, alloc_limit=alloc_limit), _solver(sf, inputs, emit_warps=8)
    want = _step(sf, ref, vecs[KEEP])
    got = _step(sf, lz, vecs[KEEP])
    assert got[0] == 0 and _same(got, want)
    lz.close()
    ref.close()


def test_declined_late(sf, inputs):
    _, vecs = inputs
    lz, ref = _solver(sf, inputs, share=SHARE), _solver(sf, inputs, share=SHARE, emit_warps=8)
    want = [_step(sf, ref, vecs[KEEP]) for _ in range(2)]
    got = _step(sf, lz, vecs[KEEP])
    assert got[0] == 0 and _same(got, want[0])
    assert lz.debug_memory() <= SHARE  # nothing of the rows is left beside the buckets
    again = _step(sf, lz, vecs[KEEP])
    assert again[0] == 0 and _same(again, want[1])
    assert again[1] == want[1][1]  # no preparation that is thrown away
    lz.debug_memory(share=0)  # memory came back
    assert _step(sf, lz, vecs[KEEP])[0] == 1
    lz.close()
    ref.close()


def test_short_after_long(sf, inputs):
    """A vector whose lists fit, after one whose lists did not: the buckets' regions make room."""
    _, vecs = inputs
    lz, ref = _solver(sf, inputs, share=SHARE), _solver(sf, inputs, emit_warps=8)
    assert _step(sf, lz, vecs[KEEP])[0] == 0
    assert lz.debug_memory() > SHARE // 2
    got, want = _step(sf, lz, vecs[SHORT]), _step(sf, ref, vecs[SHORT])
    assert got[0] == 1 and _same(got, want)
    assert lz.debug_memory() <= SHARE
    lz.close()
    ref.close()


def test_stream_of_the_buckets_counts(sf, inputs):
    """The same where the stream is longer than the rows want it (how long the buckets make it
    depends on the order in which it fills): it counts as it is."""
    _, vecs = inputs
    for _ in range(16):
        lz = _solver(sf, inputs, share=SHARE)
        assert _step(sf, lz, vecs[KEEP])[0] == 0
        assert _step(sf, lz, vecs[SHORT])[0] == 1
        assert lz.debug_memory() <= SHARE
        lz.close()


def test_allocation_time(sf, inputs):
    """ms_alloc: what a step by rows spends on growing its buffers, and nothing once they have grown."""
    _, vecs = inputs
    lz = _solver(sf, inputs)
    infos = []
    for _ in range(2):
        lz.load(*vecs[KEEP])
        n0 = sf.row_sigmas()
        infos.append(lz.step())
        assert sf.row_sigmas() == n0 + 1
    lz.close()
    assert 0.0 < infos[0]["ms_alloc"] <= infos[0]["ms_plan"]
    assert infos[1]["ms_alloc"] == 0.0
