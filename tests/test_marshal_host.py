"""Host checks of the binding's argument marshalling that need no GPU: what its
Python path refuses."""
import pytest
import torch

from paper_1902_08755_gb300 import api


def _shapes(h, w, pitch):
    """Depth buffers of the colour's pitch with too few rows, too few columns, or
    one dimension only, and one of another pitch."""
    buf = torch.ones((h, pitch))
    yield buf[:h - 1, :w]
    yield buf[:0, :w]
    yield buf[:, :w - 1]
    yield buf.reshape(-1)
    yield torch.ones((h, pitch + 1))[:, :w]


@pytest.mark.parametrize("pvp", [None, (2, 3, 9, 7)])
def test_output_depth_covers_the_output(monkeypatch, pvp):
    """Every row and column of the output rectangle is written, so the output
    depth has to have them."""
    monkeypatch.setattr(api, "_on_device", lambda *a: None)
    h, w, pitch = 7, 9, 12
    color = torch.zeros((h, pitch), dtype=torch.int32)[:, :w]
    good = torch.ones((h, pitch))[:, :w]
    assert api._target(color, good, pvp, 0).depth == good.data_ptr()
    assert api._target(color, torch.ones((h + 2, pitch)), pvp, 0).depth
    for bad in _shapes(h, w, pitch):
        with pytest.raises(ValueError):
            api._target(color, bad, pvp, 0)
    # a smaller rectangle needs only its own rows and columns
    small = torch.ones((h, pitch))[:4, :5]
    assert api._target(color, small, (0, 0, 5, 4), 0).depth == small.data_ptr()
    with pytest.raises(ValueError):
        api._target(color, small, (0, 0, 5, 5), 0)
