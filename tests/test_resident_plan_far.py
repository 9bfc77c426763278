"""Resident plans whose two matrix copies both stay in global memory (csrc/resident_plan.cpp), on the CPU."""
import pytest

import lpgen
from tests.test_resident_plan import check, plan, runner  # noqa: F401  (runner: a fixture)


@pytest.mark.parametrize("esize,size", [(8, (66_667, 166_667, 1_000_000)), (4, (160_000, 400_000, 1_040_000))])
def test_both_sides_stay_in_global_memory(runner, tmp_path, esize, size):  # noqa: F811
    lp = lpgen.powerlaw(2, *size)
    p = plan(runner, tmp_path, lp, esize, 152)
    assert p["ok"] and p["far"] == 3 and p["G"] == 152 and p["ep"] == p["ed"] == 0
    check(p, lp, "far", 152, esize)


def test_larger_matrices_are_refused_rather_than_read_from_global_memory(runner, tmp_path):  # noqa: F811
    assert not plan(runner, tmp_path, lpgen.powerlaw(2, 100_000, 250_000, 1_500_000), 8, 152)["ok"]


@pytest.mark.parametrize("size,far", [((86_666, 216_666, 1_300_000), (1, 2)), ((100_000, 250_000, 1_500_000), (3,)),
                                      ((115_000, 285_000, 1_750_000), ())])
def test_far_sides_leave_room_for_the_l1_beyond_a_million_entries(runner, tmp_path, size, far):  # noqa: F811
    lp = lpgen.powerlaw(2, *size)
    p = plan(runner, tmp_path, lp, 4, 152)
    assert bool(p["ok"]) == bool(far)
    if far:
        assert p["far"] in far and p["smem"] <= 193 * 1024
        check(p, lp, "far", 152, 4)
