"""The sort's workspace holds every count up to the one it was sized for.

sfci_sigma sorts the entries it found in a workspace sized for out_cap, so the
size may not fall as the capacity grows, and nothing behind the queried bytes
may be written.  524288 pairs (256 tiles of 2048) is where the sort's counters
change their layout.
"""
import ctypes as C

import numpy as np
import pytest

import gen

TILE, FUSED = 2048, 256 * 2048


def test_workspace_never_shrinks():
    import importlib
    build = importlib.import_module("paper_2312_01846_gb300.build")
    try:
        lib = C.CDLL(build.build())
    except RuntimeError as e:  # no nvcc on this machine
        pytest.skip(str(e))

    def room(k):
        nb = C.c_size_t()
        assert lib.sfci_truncate_topk_workspace_bytes(C.c_int64(1 << 22), C.c_int64(k), C.byref(nb)) == 0
        return nb.value

    ks = sorted(set(range(1, 3 * FUSED, 997)) | {FUSED + d for d in (-1, 0, 1, TILE, TILE + 1)})
    sizes = [room(k) for k in ks]
    assert all(a <= b for a, b in zip(sizes, sizes[1:]))


@pytest.mark.gpu
@pytest.mark.parametrize("out_cap", [FUSED + 1, 530000, 540000, FUSED])
def test_sigma_stays_in_its_workspace(out_cap):
    """120 x 4368 = 524160 determinants, nearly all reached: just below 256 tiles of entries in a
    workspace for as many or more.  What lies behind the queried bytes (here: the rest of the
    same, longer buffer) keeps its pattern."""
    torch = pytest.importorskip("torch")
    import paper_2312_01846_gb300 as sf
    d = dict(gen.molecular_integrals(16, 16, seed=9), n=16, na=2, nb=5)
    s = sf.System.from_dict(d)
    rng = np.random.default_rng(5)
    rank = np.sort(rng.choice(s.dim, 2000, replace=False)).astype(np.uint64)
    r = torch.from_numpy(rank.view(np.int64)).cuda()
    c = torch.from_numpy(rng.normal(size=rank.size)).cuda()
    want_r, want_c = sf.sfci_sigma(s, r, c, out_cap=1 << 21)
    assert 519000 < want_r.numel() <= FUSED
    need, behind = sf.sigma_workspace_bytes(s, r.numel(), out_cap), 2 << 20
    buf = torch.full((need + behind,), 0x5A, dtype=torch.uint8, device="cuda")
    outr = torch.empty(out_cap, dtype=torch.int64, device="cuda")
    outc = torch.empty(out_cap, dtype=torch.float64, device="cuda")
    n = C.c_int64()
    st = sf.lib().sfci_sigma(s.handle, sf._ptr(r), sf._ptr(c), r.numel(), 0.0, sf._ptr(outr), sf._ptr(outc),
                             out_cap, C.byref(n), sf._ptr(buf), need, sf._stream(None))
    s.close()
    assert st == 0 and n.value == want_r.numel()
    assert bool((buf[need:] == 0x5A).all())
    assert torch.equal(outr[: n.value], want_r) and torch.equal(outc[: n.value], want_c)
