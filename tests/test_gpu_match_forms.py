"""Greedy matching of given matrices far from rank one, by rounds, beside others
by steps: the groups of one CTA and a CTA of the team tier; and batches of large
ones, a CTA or a team each."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_large_match import greedy, near_rank_one, pack
from test_gpu_match_ties import took

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
DEV = "cuda"


# the smaller side at the 80 elements from which on the lists are looked at, up to
# the 256 lists of the steps; few pairs (large groups) and many (small ones)
@pytest.mark.parametrize("na,nb", [(8, 20), (79, 79), (79, 200), (80, 80), (80, 256), (256, 80), (200, 81), (120, 120),
                                   (139, 130), (200, 200), (250, 256)])
@pytest.mark.parametrize("P", [3, 1300])
def test_matchings(na, nb, P):
    rng = np.random.default_rng([na, nb])
    kinds = [rng.integers(0, 1 << 14, (na, nb)),                                             # rounds
             np.floor(120 * rng.random((na, 1)) * rng.random((1, nb)) * 120),                # steps
             np.where(rng.random((na, nb)) < 1.5 / nb, 9000, rng.integers(0, 9, (na, 1)))]   # some of both
    xs = [k.astype(np.float32) for k in kinds]
    pk = pack((na, nb))
    r = api.match(pk, pk, np.tile([(0, 1)], (P, 1)), torch.from_numpy(np.stack([xs[p % 3] for p in range(P)]).ravel()).to(DEV))
    mt, sc = r.match.cpu().numpy().reshape(P, na), r.scores.cpu().numpy()
    for q, x in enumerate(xs):
        m, s = oracle.greedy_match(x.astype(np.float64))
        assert (mt[q::3] == m).all() and (sc[q::3] == s).all()


@pytest.mark.parametrize("na,nb", [(300, 300), (20, 3000), (3000, 20), (700, 90)])
def test_large_matchings(na, nb):
    g = torch.Generator(device=DEV).manual_seed(5)
    xs = [torch.rand(na, nb, generator=g, device=DEV), near_rank_one(g, na, nb)]
    pk, P = pack((na, nb)), 310  # two pairs a CTA
    r = api.match(pk, pk, np.tile([(0, 1)], (P, 1)), torch.cat([xs[p % 2].flatten() for p in range(P)]))
    mt = r.match.cpu().numpy().reshape(P, na)
    for q, x in enumerate(xs):
        assert (mt[q::2] == greedy(x.cpu().numpy())).all()


@pytest.mark.parametrize("n,P,most", [(200, 1000, 0.6), (300, 304, 0.9)])
def test_random_ones_are_not_stepped(n, P, most):
    g = torch.Generator(device=DEV).manual_seed(8)
    pk, pairs = pack((n, n)), np.tile([(0, 1)], (P, 1))
    random = took(pk, pairs, torch.rand(n * n, generator=g, device=DEV).repeat(P))
    near = took(pk, pairs, near_rank_one(g, n, n).flatten().repeat(P))
    print(f"\n  {P} of {n} x {n}: random {1e3 * random:.2f} ms, near rank one {1e3 * near:.2f} ms")
    assert random <= most * near


@pytest.mark.parametrize("na,nb", [(1500, 1500), (13, 5000), (5000, 13)])
def test_noisy_ones_are_not_rounds(na, nb):
    """Near rank one, but with the best elements of most rows apart: by rounds 70, 4
    and 2 times what the phases take."""
    g = torch.Generator(device=DEV).manual_seed(8)
    pk, P = pack((na, nb)), torch.cuda.get_device_properties(0).multi_processor_count
    near = near_rank_one(g, na, nb).flatten()
    one, all_ = took(pk, [(0, 1)], near), took(pk, np.tile([(0, 1)], (P, 1)), near.repeat(P))
    print(f"\n  {na} x {nb}: one {1e3 * one:.2f} ms, {P} {1e3 * all_:.2f} ms")
    assert all_ <= 20 * one
