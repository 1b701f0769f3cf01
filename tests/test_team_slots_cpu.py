"""The scratch slots of the team tier when there are fewer than CTAs (host build
of csrc/layout.h): teams of one level have slots and CTAs of their own, and a
team shares its slot only with coarser teams that hold all of its CTAs.  No
barrier sits between levels, so a CTA that is not in the slot's last team could
otherwise write to it while that team is at work."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_02423_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>
#include "layout.h"
using namespace cfsim;
typedef std::map<uint64_t, std::vector<uint32_t>> Slots;  // slot -> the CTAs of its team
int main(int argc, char** argv) {
  const uint32_t n_team = atoi(argv[1]);
  int bad = 0;
  for (uint64_t nslots = 1; nslots <= n_team; ++nslots) {
    const bool shared = nslots < n_team;
    const int finest = shared ? team_finest(n_team, nslots) : kTeamLevels - 1;
    bad += finest < 0 || finest >= kTeamLevels;
    std::vector<Slots> at(kTeamLevels);
    for (int L = 0; L <= finest; ++L) {
      std::vector<int> seen(n_team, 0);
      for (uint32_t b = 0; b < n_team; ++b) {
        const TeamSeat s = team_seat(b, L, n_team, n_team, shared, finest);
        if (!s.in) continue;
        bad += s.T == 0 || s.k >= s.teams || b < s.first || b >= s.first + s.T || s.first + s.T > n_team;
        bad += s.slot >= nslots;
        at[L][s.slot].push_back(b);
      }
      bad += at[L].empty();
      for (const auto& q : at[L]) {  // a whole team, one team a slot
        const TeamSeat s = team_seat(q.second[0], L, n_team, n_team, shared, finest);
        bad += q.second.size() != s.T || q.second[0] != s.first || q.second.back() != s.first + s.T - 1;
        for (uint32_t b : q.second) bad += seen[b]++ != 0;
      }
      for (int C = 0; C < L; ++C)
        for (const auto& q : at[L]) {
          const auto c = at[C].find(q.first);
          if (c == at[C].end()) continue;
          bad += q.second.front() < c->second.front() || q.second.back() > c->second.back();
        }
    }
  }
  printf("%d\n", bad);
  return 0;
}
"""


@pytest.mark.parametrize("ctas", [1, 2, 3, 60, 64, 100, 132, 148, 152, 208])
def test_shared_slots_nest(ctas, tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe), str(ctas)], check=True, capture_output=True, text=True).stdout == "0\n"
