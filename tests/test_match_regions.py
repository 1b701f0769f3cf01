"""The matching of given matrices stays inside its group's shared memory: the
matrix and the state of a pair of more than 256 lists take more room one way
round than the other, and the kernel works on the caller's orientation."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_02423_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "layout.h"
using namespace cfsim;
int main() {
  const int nt = 1024, z = 225280;
  ClassCfg c{nt, z, z / 2, z / 4, z / 8, (z / (nt / 32)) & ~15, kClassWarp, 0, 0, 2};
  long bad = 0;
  for (int cls = kClassCta; cls <= kClassWarp; ++cls) {
    c.min_cls = cls;
    for (int na = 1; na <= kMaxBlocks; na += na < 400 ? 1 : na / 100)
      for (int nb = 1; nb <= 70000 / na + 300 && nb <= kMaxBlocks; ++nb) {
        const Shape s = classify(na, nb, na, nb, c);
        if (s.cls != kClassGlobal) bad += s.tr != 0 || match_bytes(na, nb) > group_region(s.cls, c);
      }
  }
  printf("%ld\n", bad);
  return 0;
}
"""


def test_regions_hold_their_pairs(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "0\n"


# the last shape of a half CTA, shapes that only fit one the other way round, the
# other way round, the same at a whole CTA and a quarter
@pytest.mark.gpu
@pytest.mark.parametrize("na,nb,pairs", [(20, 1340, 304), (20, 1341, 304), (20, 1350, 304), (20, 1365, 304),
                                         (1350, 20, 304), (10, 2570, 304), (10, 1280, 800), (19, 2830, 20), (1, 28155, 3),
                                         (1, 28170, 3), (28170, 1, 3)])
def test_matchings(na, nb, pairs):
    import torch

    import oracle
    from gen.cfg_grammar import CFG
    from paper_1707_02423_gb300 import api

    z = np.zeros(0, np.int32)
    cfgs = [CFG(n, z, z, np.zeros(0, np.float32), np.ones((n, 4), np.float32)) for n in (na, nb)]
    pk = api.Pack(cfgs, 4, device="cuda")
    rng = np.random.default_rng([na, nb])
    xs = [(rng.integers(0, 1 << 15, size=(na, nb)) / 8.0).astype(np.float32) for _ in range(4)]
    refs = [oracle.greedy_match(x.astype(np.float64)) for x in xs]
    X = torch.from_numpy(np.concatenate([xs[p % 4].ravel() for p in range(pairs)])).cuda()
    r = api.match(pk, pk, [(0, 1)] * pairs, X)
    mt, sc = r.match.cpu().numpy().reshape(pairs, na), r.scores.cpu().numpy()
    for p in range(pairs):
        m_ref, s_ref = refs[p % 4]
        assert np.array_equal(mt[p], m_ref), p
        assert float(sc[p]) == s_ref
