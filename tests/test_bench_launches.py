"""How bench.py counts launches: from what the profiled steps launched, per solve."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def fam(**n):
    names = ("resident_bicg", "resident_cg", "mass", "amg", "amg_transfer")
    return {f: (n.get(f, 0), 0.0) for f in names}


@pytest.mark.parametrize("launches,inner,scalars,want", [
    (dict(), 1, 0, (False, False, False, False)),
    (dict(resident_bicg=2, resident_cg=2), 1, 0, (True, False, True, False)),
    # scalars fit in one launch on systems too large for three components
    (dict(resident_bicg=4, mass=60), 1, 2, (False, True, False, False)),
    (dict(resident_bicg=6, resident_cg=2, mass=2), 1, 2, (True, True, True, True)),
    (dict(resident_bicg=6, resident_cg=6), 3, 0, (True, False, True, False)),
])
def test_solves_in_one_launch(launches, inner, scalars, want):
    import bench
    assert bench.step_launches(fam(**launches), 2, inner, scalars) == want


def test_first_level_of_the_shared_launch():
    import bench
    info = {"levels": 5}
    assert bench.amg_tail(info, fam(amg=10, amg_transfer=40)) == 2
    assert bench.amg_tail(info, fam(amg=10, amg_transfer=80)) == 4
    assert bench.amg_tail(info, fam()) == 4
