"""The packed interior field of a ghosted state and back: block by block through
views up to a number of blocks, by an index table beyond it; the same values."""
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims", [[(3, 4, 5)], [(1, 1, 1)], [(7, 2, 1)], [(2, 3, 1), (5, 1, 4)],
                                  [(k + 1, 3, 2) for k in range(9)]])
def test_views_and_table_agree(dims, monkeypatch):
    from paper_2012_02925_gb300 import autograd
    monkeypatch.setattr(torch.Tensor, "cuda", lambda self: self)
    size = sum(5 * (a + 4) * (b + 4) * (c + 4) for a, b, c in dims)
    q = torch.arange(size, dtype=torch.float64)
    out = []
    for limit in (0, 100):
        monkeypatch.setattr(autograd, "_VIEW_BLOCKS", limit)
        s = SimpleNamespace(block_dims=dims, state_size=size)
        field = autograd.interior(s, q)
        out.append((field, autograd.scatter_interior(s, field)))
    assert out[0][0].numel() == 5 * sum(a * b * c for a, b, c in dims)
    assert all(torch.equal(a, b) for a, b in zip(*out))
    assert torch.equal(autograd.interior(s, torch.stack([q, q], 1)[:, 0]), out[0][0])   # a strided state
