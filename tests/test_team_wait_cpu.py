"""How long a CTA of the team tier waits for another one (host build of
csrc/layout.h): as long as that CTA passes barriers, however many pairs it still
has to do, and no longer than an iteration of the costliest pair after it has
stopped."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_02423_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "layout.h"
using namespace cfsim;
int main() {
  const uint64_t s = 1000000000ull, limit = team_wait_ns(0);
  int bad = limit < s || limit > 60 * s;
  // a barrier every `every` seconds, the last one at 3,600 s; polled every 50 ms
  for (uint64_t every = 1; every * s < limit; ++every) {
    TeamWait w{7, 1};
    uint64_t over = 0;
    for (uint64_t now = 7; now < 8000 * s && !over; now += s / 20) {
      const uint64_t passed = (now < 3600 * s ? now : 3600 * s) / (every * s);
      if (team_wait_over(w, now, 1 + passed, limit)) over = now;
    }
    const uint64_t last = 3600 / every * every * s;
    bad += over <= last + limit || over > last + limit + s;
  }
  // an iteration of two CFGs of 32,000 blocks with 2^20 edges each, on one CTA at one term per ns
  const int64_t cost = 32000ll * 32000 + 2 * (1ll << 40);
  bad += team_wait_ns(cost) < (uint64_t)cost;
  // the most a pair can have: no overflow
  const int64_t most = 32000ll * 32000 + 2 * (32000ll * 32000) * (32000ll * 32000);
  bad += team_wait_ns(2 * most) < team_wait_ns(most);
  printf("%d\n", bad);
  return 0;
}
"""


def test_waits_go_on_with_progress(tmp_path):
    src, exe = tmp_path / "wait.cpp", tmp_path / "wait"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.strip() == "0"
