"""The first capacity of sfci_sigma: what a call holds, and what it does where memory is short.

The capacities are made small (they are module constants), so that a small space
behaves as 2^24 to 2^25 entries do.
"""
import types

import numpy as np
import pytest

import gen


def test_table_systems_start_small():
    """Beyond the limits of the sum by target rows the hash table is cleared throughout."""
    import paper_2312_01846_gb300 as sf
    for n, na, nb, rows in ((28, 7, 7, True), (28, 12, 12, True), (32, 12, 12, False), (16, 13, 2, False),
                            (64, 5, 12, False), (64, 5, 5, True)):
        assert sf._rows_possible(types.SimpleNamespace(n=n, na=na, nb=nb)) == rows


@pytest.fixture
def small(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2312_01846_gb300 as sf
    monkeypatch.setattr(sf, "_SIGMA_ROOM", 1 << 14)
    monkeypatch.setattr(sf, "_SIGMA_ROOM_TABLE", 1 << 13)
    s = sf.System.from_dict(gen.config_system(0))  # 4900 determinants
    rng = np.random.default_rng(0)
    r = np.sort(rng.choice(s.dim, 257, replace=False)).astype(np.uint64)
    c = rng.normal(size=r.size)
    want = sf.sfci_sigma(s, r, c, out_cap=4900)
    yield sf, torch, s, r, c, want
    s.close()


@pytest.mark.gpu
def test_result_holds_its_own_size(small):
    sf, torch, s, r, c, want = small
    rank, coef = sf.sfci_sigma(s, r, c)
    assert torch.equal(rank, want[0]) and torch.equal(coef, want[1])
    assert rank.untyped_storage().nbytes() == coef.untyped_storage().nbytes() == 8 * rank.numel()


@pytest.mark.gpu
def test_smaller_room_where_memory_is_short(small, monkeypatch):
    sf, torch, s, r, c, want = small
    asked, empty = [], torch.empty

    def short(size, **kw):
        asked.append(size)
        if isinstance(size, int) and size == sf._SIGMA_ROOM:
            raise torch.OutOfMemoryError("injected")
        return empty(size, **kw)

    monkeypatch.setattr(torch, "empty", short)
    rank, coef = sf.sfci_sigma(s, r, c)
    monkeypatch.undo()
    assert 1 << 14 in asked and 1 << 13 in asked
    assert torch.equal(rank, want[0]) and torch.equal(coef, want[1])
