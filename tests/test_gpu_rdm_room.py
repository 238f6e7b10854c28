"""sfci_rdm12 where the workspace of the pairs by rows is not free: the vector's table does."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dets", [1, 511, 512, 513, 3000])
def test_table_where_memory_is_short(monkeypatch, dets):
    torch = pytest.importorskip("torch")
    import paper_2312_01846_gb300 as sf
    s = sf.System.from_dict(gen.config_system(4))
    rng = np.random.default_rng(dets)
    r = np.sort(rng.choice(s.dim, dets, replace=False)).astype(np.uint64)
    c = rng.normal(size=dets)
    want = sf.sfci_rdm12(s, r, c)
    asked, empty = [], torch.empty

    def short(size, **kw):
        if kw.get("dtype") == torch.uint8:
            asked.append(size)
            if len(asked) == 1:
                raise torch.OutOfMemoryError("injected")
        return empty(size, **kw)

    monkeypatch.setattr(torch, "empty", short)
    got = sf.sfci_rdm12(s, r, c)
    monkeypatch.undo()
    s.close()
    assert len(asked) == 2 and asked[1] < asked[0]
    assert got[2] == want[2]
    for x, y in zip(got[:2], want[:2]):  # (the same products, added in any order)
        np.testing.assert_allclose(x.cpu().numpy(), y.cpu().numpy(), rtol=0, atol=1e-12 * float(y.abs().max()))
