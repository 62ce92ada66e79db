"""Strip height of served small grids that step side by side (host only): the
library's choice until their 16-row strips fill the resident warps, 16 rows
from there, set once per change and for small grids only."""
import pytest

from paper_1605_05320_gb300 import serve


@pytest.mark.parametrize("sizes,rows", [([], 0), ([512], 0), ([512] * 3, 0), ([512] * 4, 16),
                                        ([256] * 15, 0), ([256] * 16, 16), ([1024], 0),
                                        ([1024, 512], 16), ([64] * 16, 0)])
def test_rows_by_the_strips_in_flight(sizes, rows):
    assert serve.strip_rows(sizes, 2432) == rows


def test_height_is_set_once_per_change(monkeypatch):
    calls = []
    monkeypatch.setattr(serve.S, "swa_grid_set_strip_rows", lambda h, r: calls.append(r))
    sc = serve.Scenario.__new__(serve.Scenario)
    sc.rows = 0
    sc.grid = type("Grid", (), {"h": None})
    for r in (0, 16, 16, 0, 0, 16):
        sc.set_rows(r)
    assert calls == [16, 0, 16]
