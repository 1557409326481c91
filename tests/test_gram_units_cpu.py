"""Units of a group in the shared-operand contraction, on CPU: its kernel gives
every 16-row unit of a step a producer warp of its own, 20 of them."""
import pytest

from test_gram_rows_cpu import _check, _closing, _layout, driver  # noqa: F401 (fixture)


@pytest.mark.parametrize("mode,nb,items", [
    ("P", 128, [(0, b, b) for b in range(64)] + [(0, 0, b) for b in range(64, 128)]),  # 64 pairs, 128 bins
    ("W", 64, _closing(64, 3, 1.0)),                                                   # 64 bins, groups of 256 pairs
    ("W", 64, _closing(64, 3, -0.08)),
    ("S", 16, _closing(16, 3, 0.0) + _closing(16, 4, 0.0)),                            # 16 bins, every quadruplet
    ("S", 21, _closing(21, 3, -0.5) + [(0, 0, a, b) for a in range(21) for b in range(a, 21)]),  # 252 rows
])
def test_a_producer_warp_for_every_unit(driver, mode, nb, items):  # noqa: F811
    ok, groups = _layout(driver, mode, nb, sorted(set(items)))
    assert ok
    _check(groups, sorted(set(items)))
    for _, _, rows, _ in groups:
        assert sum(any(x >= 0 for row in rows[u:u + 16] for x in row) for u in range(0, len(rows), 16)) <= 20
