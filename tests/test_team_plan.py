"""The team plan of a batch: every unit in one class, its teams resident together, and planned in a time of the order
of one sort of the units, since it is part of the call."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1903_01665_gb300", "csrc")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("team_plan") / "team_plan")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "team_plan.cpp"), "-o", out], check=True)
    return out


def plan(exe, units, kinds, seed, spread):
    rows = subprocess.run([exe, str(units), str(kinds), str(seed), str(spread)], check=True, capture_output=True,
                          text=True).stdout.split("\n")
    return [tuple(map(int, r.split())) for r in rows[:kinds]], float(rows[kinds])


# the last two: the units' work is far more than 10^4 times that of the longest one on all CTAs
@pytest.mark.parametrize("units, kinds, spread", [(1, 1, 1), (7, 3, 2), (24, 2, 3), (1000, 3, 3), (1000, 1, 0),
                                                  (60000, 1, -6), (60000, 2, -6)])
def test_every_unit_planned_and_the_teams_fit(exe, units, kinds, spread):
    for seed in (1, 2):
        rows, _ = plan(exe, units, kinds, seed, spread)
        assert sum(r[2] for r in rows) == units
        assert all(planned == mine for _, _, mine, planned in rows)
        assert all(1 <= ctas <= capacity for capacity, ctas, _, _ in rows)
        assert sum(ctas / capacity for capacity, ctas, _, _ in rows) <= 1.0 + 1e-9


def test_more_kinds_than_fit_together_get_a_cta_each(exe):
    rows, _ = plan(exe, 40, 8, 1, 2)   # two of the eight have room for one CTA
    assert all(1 <= ctas <= capacity for capacity, ctas, _, _ in rows)
    assert all(planned == mine for _, _, mine, planned in rows)


def test_planning_takes_the_time_of_a_few_sorts(exe):
    assert min(plan(exe, 20000, 3, seed, 3)[1] for seed in (1, 2, 3)) < 30
