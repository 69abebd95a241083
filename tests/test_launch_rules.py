"""The launch planners' arithmetic, on the host: every team is whole warps
whatever the number of teams a CTA holds (512 and 1024 threads shared by 3, 5, 6
or 7 teams are not multiples of 32)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include "launch_rules.h"
int main() {
  for (int cta : {512, 1024})
    for (int teams = 1; teams <= 15; ++teams)
      for (long long rows : {1ll, 31ll, 32ll, 33ll, 330ll, 4000ll, 65535ll, 2147483647ll})
        for (long long per : {1ll, 2ll, 8ll, 2147483647ll})
          std::printf("%d %d %lld %lld %d\n", cta, teams, rows, per,
                      pccp::team_for_rows(rows, per, cta, teams));
}
"""


@pytest.fixture(scope="module")
def teams(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cc").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2207_12116_gb300", "csrc"),
                    str(d / "rules.cc"), "-o", str(d / "rules")], check=True)
    out = subprocess.run([str(d / "rules")], check=True, capture_output=True, text=True).stdout
    return [tuple(int(x) for x in line.split()) for line in out.splitlines()]


def test_teams_are_whole_warps_that_fit_the_cta(teams):
    assert len(teams) == 2 * 15 * 8 * 4
    for cta, n, rows, per, team in teams:
        assert team % 32 == 0 and 32 <= team and team * n <= cta, (cta, n, rows, per, team)
        # as many threads as the rows ask for, unless the CTA has no more
        want = -(-rows // per)
        assert team >= want or team + 32 > cta // n
        assert team - 32 < want
