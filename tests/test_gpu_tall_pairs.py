"""Global-class pairs of many rows and few columns, whose matrices the team tier
keeps transposed (n_a >= 4 n_b): on either side of the line, with lists of every
length in rows and columns, staged and not."""
import time

import numpy as np
import pytest
import torch

import oracle
from test_gpu_far_pairs import graph
from _helpers import eps_greedy, greedy_margin

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
B = pytest.importorskip("paper_1707_02423_gb300._binding")
DEV = "cuda"


@pytest.mark.parametrize("na,nb,ha,hb", [(399, 100, (), ()), (400, 100, (40,), (33,)), (401, 100, (5,), (17,)),
                                         (700, 25, (), ()), (3000, 7, (90,), ()), (4100, 33, (17, 90), (20,)),
                                         (19000, 1, (), ()), (9000, 2, (50,), ())])
@pytest.mark.parametrize("form", ["batch", "plain", "beside a wide one"])
def test_against_the_oracle(na, nb, ha, hb, form):
    rng = np.random.default_rng([na, nb])
    a, b = graph(rng, na, ha), graph(rng, nb, hb)
    pk = api.Pack([a, b], 13, device=DEV)
    om = torch.linspace(0.5, 1.5, 13, device=DEV)
    pairs = [(0, 1), (1, 0)] if form == "beside a wide one" else [(0, 1)]
    r = api.similarity(pk, pk, pairs, om, 0.8, 8, want_x=True, want_match=True, per_pair=form == "plain")
    ref = oracle.similarity(a, b, om.cpu().numpy(), 0.8, 8)["X"]
    got = r.X_of(0, na, nb).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-5
    m = r.match.cpu().numpy()[:na]
    m_own, s_own = oracle.greedy_match(got.astype(np.float64))
    assert np.array_equal(m, m_own)
    assert abs(float(r.scores[0]) - s_own) <= 1e-5
    if greedy_margin(ref) <= 1e-6:
        assert eps_greedy(got, ref, m, 2e-5)
    if len(pairs) == 2:
        assert np.abs(r.X_of(1, nb, na).cpu().numpy().T - ref).max() <= 1e-5


@pytest.mark.parametrize("na,nb", [(3000, 13), (20000, 2)])
def test_no_slower_than_wide(na, nb):
    rng = np.random.default_rng(4)
    pk = api.Pack([graph(rng, na), graph(rng, nb)], 13, device=DEV)
    om = torch.ones(13, device=DEV)

    def took(pair):
        pairs, ws, best = np.tile([pair], (304, 1)), api.Workspace(DEV), 1e9
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            api.similarity(pk, pk, pairs, om, ws=ws, want_x=True, want_scores=False)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best

    tall, wide = took((0, 1)), took((1, 0))
    print(f"\n  304 pairs, {na} x {nb}: {1e3 * tall:.2f} ms, the other way round {1e3 * wide:.2f} ms")
    assert tall <= 2 * wide
