"""Map descriptions given as arrays: what the binding hands to the library."""
import numpy as np
import pytest

from paper_1811_09711_gb300 import problems as P
from paper_1811_09711_gb300 import vamp as V


def maps(rows, slots, k=3):
    rng = np.random.default_rng(1)
    return P.MapSet(np.array([2, 0, 4])[:k], rng.integers(0, 9, (rows, slots)), rng.integers(0, 3, (rows, slots)),
                    rng.uniform(size=(rows, slots)), rng.uniform(size=(rows, slots)).astype(np.float32))


@pytest.mark.parametrize("rows,slots", [(3, 4), (5, 4), (3, 6)])
def test_fields(rows, slots):
    ms = maps(rows, slots)
    arr = V._map_array(ms)
    assert len(arr) == 3
    for q in range(3):
        assert arr[q].n_mapped == ms.n_mapped[q]
        for f in ("coord", "kind", "a", "b"):
            assert list(getattr(arr[q], f)) == list(getattr(ms, f)[q, :4]), f


@pytest.mark.parametrize("rows,slots", [(2, 4), (3, 1), (3, 3), (1, 4)])
def test_too_few_rows_or_slots(rows, slots):
    with pytest.raises(IndexError):
        V._map_array(maps(rows, slots))
