"""Greedy matching of large given matrices with many equal values in a row: more
of them than a row's list or its candidates hold."""
import time

import numpy as np
import pytest
import torch

from test_gpu_large_match import greedy, near_rank_one, pack

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
DEV = "cuda"


def check(xs):
    pk = pack([n for x in xs for n in x.shape])
    pairs = np.arange(2 * len(xs), dtype=np.int32).reshape(-1, 2)
    r = api.match(pk, pk, pairs, torch.from_numpy(np.concatenate([x.ravel() for x in xs])).to(DEV))
    mt, sc = r.match.cpu().numpy(), r.scores.cpu().numpy()
    for p, x in enumerate(xs):
        m = greedy(x)
        assert np.array_equal(mt[r.m_off[p]:r.m_off[p + 1]], m), x.shape
        k = np.flatnonzero(m >= 0)
        s = x[k, m[k]].astype(np.float64).sum()  # whole numbers: exact
        assert float(sc[p]) == s


def took(pk, pairs, X):
    ws, best = api.Workspace(DEV), 1e9
    for _ in range(5):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        api.match(pk, pk, pairs, X, ws=ws)
        best = min(best, time.perf_counter() - t0)
    return best


# values per entry; pairs of one matrix each (a team) and of many (a CTA)
@pytest.mark.parametrize("na,nb", [(13, 5000), (200, 1500), (500, 600), (2, 9000)])
@pytest.mark.parametrize("values", [1, 2, 3, 17, 1000])
@pytest.mark.parametrize("P", [1, 160])
def test_few_values(na, nb, values, P):
    rng = np.random.default_rng([na, values])
    xs = [rng.integers(0, values, (na, nb)).astype(np.float32) for _ in range(min(P, 4))]
    check(xs[:1] if P == 1 else [xs[p % 4] for p in range(P)])


@pytest.mark.parametrize("first", [0, 1, 70, 71, 72, 95, 96, 97, 500, 513])
@pytest.mark.parametrize("second", [20, 96, 600])
def test_runs(first, second):
    """`first` entries of one value and `second` of the next one in every row,
    around the list's length (96; from 72 on it may end early)."""
    rng = np.random.default_rng([first, second])
    x = rng.integers(0, 50, (60, 2000)).astype(np.float32)
    for row in x:
        at = rng.permutation(2000)
        row[at[:first]] = 100
        row[at[first:first + second]] = 90
    check([x])


@pytest.mark.parametrize("kind", ["few", "ones"])
def test_no_cliff(kind):
    g = torch.Generator(device=DEV).manual_seed(8)
    pk, pairs = pack((13, 5000)), np.tile([(0, 1)], (500, 1))
    x = torch.ones(13, 5000, device=DEV) if kind == "ones" else torch.floor(3 * torch.rand(13, 5000, generator=g, device=DEV))
    near = took(pk, pairs, near_rank_one(g, 13, 5000).flatten().repeat(500))
    tied = took(pk, pairs, x.flatten().repeat(500))
    print(f"\n  500 matrices of 13 x 5,000: near rank one {1e3 * near:.2f} ms, {kind} {1e3 * tied:.2f} ms")
    assert tied <= 4 * near
