"""Scores of the team tier's pairs that are too thin for its lists and are matched
by one CTA of the team: the sum over that CTA's warps, read by all of them before
the team's next barrier takes its place."""
import numpy as np
import pytest
import torch

from gen.cfg_grammar import CFG

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
DEV = "cuda"


@pytest.mark.parametrize("na,nb", [(3000, 5), (5, 3000), (1500, 10), (10, 1500), (15000, 1)])
@pytest.mark.parametrize("P", [1, 5, 40, 300])
def test_scores(na, nb, P):
    rng = np.random.default_rng([na, P])
    z = np.zeros(0, np.int32)
    pk = api.Pack([CFG(n, z, z, z.astype(np.float32), np.ones((n, 4), np.float32)) for n in (na, nb)], 4, device=DEV)
    x = rng.integers(0, 1 << 12, (P, na, nb)).astype(np.float32)  # sums are exact
    X = torch.from_numpy(x.ravel()).to(DEV)
    ws = api.Workspace(DEV)
    for _ in range(20):
        r = api.match(pk, pk, np.tile([[0, 1]], (P, 1)), X, ws=ws)
        m = r.match.cpu().numpy().reshape(P, na)
        p, i = np.nonzero(m >= 0)
        assert len(p) == P * min(na, nb)
        s = np.bincount(p, x[p, i, m[p, i]].astype(np.float64), P)
        assert np.array_equal(r.scores.cpu().numpy().astype(np.float64), s)
