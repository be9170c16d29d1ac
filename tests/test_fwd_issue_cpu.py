"""The order in which the forward's issuing warp waits and issues, run on the host with stand-ins (fwd_issue_host.cpp): what a
whole run does, and that after a wait that failed nothing more is issued or waited for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WAITS = "uqkvp"


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("issue") / "fwd_issue")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2609_19242_b200", "csrc"),
                    os.path.join(ROOT, "tests", "fwd_issue_host.cpp"), "-o", exe], check=True)

    def go(fail, units):
        out = subprocess.run([exe, str(fail), *map(str, units)], check=True, capture_output=True, text=True, timeout=60).stdout
        events, done = out.split("\n")[:2]
        return events, done == "1"
    return go


UNITS = [[1], [3], [0], [2, 1], [0, 0, 2], [4, 0, 0, 1, 2, 0], []]


@pytest.mark.parametrize("units", UNITS, ids=str)
def test_a_whole_run_issues_every_tile_once(run, units):
    events, done = run(-1, units)
    assert done
    tiles, seen = sum(units), sum(u > 0 for u in units)
    for c in "STOPK":
        assert events.count(c) == tiles, c
    for first, rest in ("YA", "ZB"):   # two halves per tile; the first half of a unit's first tile starts O anew
        assert events.count(first) == seen and events.count(rest) == 2 * tiles - seen
    assert events.count("E") == events.count("q") == seen
    assert events.count("p") == 4 * tiles and events.count("k") == events.count("v") == tiles
    assert events.count("u") == len(units) + 1


@pytest.mark.parametrize("units", UNITS, ids=str)
def test_nothing_follows_a_failed_wait(run, units):
    whole, _ = run(-1, units)
    for fail in range(sum(c in WAITS for c in whole)):
        events, done = run(fail, units)
        assert not done
        assert whole.startswith(events) and events[-1] in WAITS
        assert sum(c in WAITS for c in events) == fail + 1
