"""The autotuner's default candidates are different launches."""
import re
import os

from paper_2603_08386_gb300 import tune

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def constant(name):
    src = open(os.path.join(ROOT, "paper_2603_08386_gb300", "csrc", "ddhf_internal.cuh")).read()
    return int(re.search(rf"constexpr int {name} = (\d+);", src).group(1))


def test_default_candidates_are_distinct_launches():
    team, big = constant("kTeamPixel"), constant("kBigPixel")
    seen = {}
    for c in tune.DEFAULT_CANDIDATES:
        hm = c["heavy_min"]
        launch = (min(hm, team), max(hm, big)) + tuple(sorted((k, v) for k, v in c.items()
                                                              if k != "heavy_min"))
        assert launch not in seen, (c, seen[launch])
        seen[launch] = c
