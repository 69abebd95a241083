"""The team size of the mask form's propagation, on the host: a batch whose stores
fit the GPU's teams at once takes one turn, whatever the width of a store."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include "launch_rules.h"
int main() {
  for (int words : {0, 1, 2, 7, 20, 30, 68, 120, 128, 129, 270, 480, 8191})
    for (long long n : {1ll, 10ll, 152ll, 153ll, 304ll, 456ll, 608ll, 777ll, 1216ll, 1217ll, 2432ll, 2433ll,
                        3040ll, 5000ll, 10000ll, 2147483647ll})
      for (int sms : {1, 148, 152})
        std::printf("%d %lld %d %d\n", words, n, sms, pccp::propagation_team(n, sms, words));
}
"""


@pytest.fixture(scope="module")
def planned(tmp_path_factory):
    d = tmp_path_factory.mktemp("team")
    (d / "team.cc").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2207_12116_gb300", "csrc"),
                    str(d / "team.cc"), "-o", str(d / "team")], check=True)
    out = subprocess.run([str(d / "team")], check=True, capture_output=True, text=True).stdout
    return [tuple(int(x) for x in line.split()) for line in out.splitlines()]


def test_one_turn_where_the_teams_hold_the_batch(planned):
    assert len(planned) == 13 * 16 * 3
    for words, n, sms, team in planned:
        assert team % 32 == 0 and 64 <= team <= 1024
        pairs = (words + 1) // 2
        if pairs <= 40:  # larger stores take at least four warps, or eight
            assert team <= 32 * max(2, pairs)
            at_once = sms * min(16, 1024 // team)
            assert n <= at_once or n > 16 * sms, (words, n, sms, team)
        else:
            assert team >= (256 if pairs > 100 else 128) and team >= min(pairs, 1024)


def test_no_second_turn_of_a_few_stores(tmp_path):
    """Stores too large for one turn's share of warps: 1,314 of 78 tasks (195 words) in
    teams of 4 warps were a turn of 1,216 stores and one of 98."""
    (tmp_path / "few.cc").write_text(r"""
#include <cstdio>
#include "launch_rules.h"
int main() {
  for (int words : {130, 195, 255, 256, 270, 480, 511})
    for (long long n = 1; n <= 2432; ++n) std::printf("%d %lld %d\n", words, n, pccp::propagation_team(n, 152, words));
}
""")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2207_12116_gb300", "csrc"),
                    str(tmp_path / "few.cc"), "-o", str(tmp_path / "few")], check=True)
    out = subprocess.run([str(tmp_path / "few")], check=True, capture_output=True, text=True).stdout
    lines = [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    assert len(lines) == 7 * 2432
    for words, n, team in lines:
        assert team % 32 == 0 and 64 <= team <= 1024
        held = 152 * min(16, 1024 // team)
        assert not held < n <= held + held // 3, (words, n, team)
