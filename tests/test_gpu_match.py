"""Greedy matching of caller-given matrices, against the FP64 oracle on the same
float32 values: the sizes where its forms meet (a warp's lists per lane, the
256 lists of the sequential steps, one CTA's shared memory, a team's lists),
both orientations, exact ties; workspaces without scratch; entries that are
never taken."""
import ctypes as C

import numpy as np
import pytest
import torch

import oracle
from gen.cfg_grammar import structured_cfg

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
B = pytest.importorskip("paper_1707_02423_gb300._binding")
DEV = "cuda"


def draw(rng, na, nb, ties):
    # multiples of 1/8 below 2**12: a score of up to 512 such terms is exact in float32
    return (rng.integers(0, 6 if ties else 1 << 15, size=(na, nb)) / 8.0).astype(np.float32)


@pytest.mark.parametrize("ties", [True, False])
@pytest.mark.parametrize("sizes", [
    [(1, 1), (1, 300), (300, 1), (31, 33), (32, 32), (33, 31), (64, 65), (65, 64), (120, 129), (129, 120)],
    [(255, 20), (256, 20), (257, 20), (20, 255), (20, 256), (20, 257), (128, 128), (130, 139), (137, 137)],
    [(138, 140), (150, 150), (257, 260), (20, 1100), (1100, 20), (700, 90)],
    [(3000, 9), (9, 3000), (1500, 40)],
])
@pytest.mark.parametrize("scratch", [True, False])
def test_sizes(sizes, ties, scratch):
    rng = np.random.default_rng(5)
    cfgs = [structured_cfg(rng, n, 3, 3) for s in sizes for n in s]
    pairs = np.arange(2 * len(sizes), dtype=np.int32).reshape(-1, 2)
    pk = api.Pack(cfgs, 4, device=DEV)
    xs = [draw(rng, na, nb, ties) for na, nb in sizes]
    X = torch.from_numpy(np.concatenate([x.ravel() for x in xs])).to(DEV)
    if scratch:
        r = api.match(pk, pk, pairs, X)
        sc, mt, m_off = r.scores, r.match, r.m_off
    else:  # the fixed part of a workspace only: as much as this many pairs of one block need
        one = api.Pack([structured_cfg(rng, 1, 3, 3)], 4, device=DEV)
        n = api.ws_size(one, one, np.zeros_like(pairs), B.params())
        ws = torch.empty(n, dtype=torch.uint8, device=DEV)
        m_off = np.concatenate([[0], np.cumsum([s[0] for s in sizes])])
        sc = torch.empty(len(sizes), device=DEV)
        mt = torch.empty(int(m_off[-1]), dtype=torch.int32, device=DEV)
        d_pairs = torch.from_numpy(pairs).to(DEV)
        st = torch.cuda.current_stream().cuda_stream
        L = B.lib()
        B.check(L.cf_match(pk.dev.data_ptr(), pk.dev.data_ptr(), d_pairs.data_ptr(), len(pairs),
                           C.byref(B.params()), None, X.data_ptr(), mt.data_ptr(), sc.data_ptr(), ws.data_ptr(), n, st))
        B.check(L.cf_status_check(ws.data_ptr(), st))
    sc, mt = sc.cpu().numpy(), mt.cpu().numpy()
    for p, x in enumerate(xs):
        m_ref, s_ref = oracle.greedy_match(x.astype(np.float64))
        assert np.array_equal(mt[m_off[p]:m_off[p + 1]], m_ref), sizes[p]
        assert float(sc[p]) == s_ref, sizes[p]


@pytest.mark.parametrize("na,nb", [(6, 40), (40, 6), (200, 200), (300, 20)])
@pytest.mark.parametrize("bad", [float("nan"), float("-inf")])
def test_entries_never_taken(na, nb, bad):
    # one whole line of the shorter side cannot be matched; -0 counts as +0
    rng = np.random.default_rng(6)
    x = draw(rng, na, nb, True)
    x[x == 0] = -0.0
    k = min(na, nb) - 1
    y = np.delete(x, k, axis=0 if na <= nb else 1)
    x[(k, slice(None)) if na <= nb else (slice(None), k)] = bad
    pk = api.Pack([structured_cfg(rng, n, 3, 3) for n in (na, nb)], 4, device=DEV)
    pairs = np.array([[0, 1]], np.int32)
    ws = api.Workspace(DEV)
    X = torch.from_numpy(x.ravel()).to(DEV)
    with pytest.raises(B.CfsimError) as e:
        api.match(pk, pk, pairs, X, ws=ws)
    assert e.value.status == 6  # CF_ERR_NUMERIC
    mt = torch.empty(na, dtype=torch.int32, device=DEV)
    sc = torch.empty(1, device=DEV)
    d_pairs = torch.from_numpy(pairs).to(DEV)
    w = ws.get(0)
    st = torch.cuda.current_stream().cuda_stream
    B.check(B.lib().cf_match(pk.dev.data_ptr(), pk.dev.data_ptr(), d_pairs.data_ptr(), 1, C.byref(B.params()), None,
                             X.data_ptr(), mt.data_ptr(), sc.data_ptr(), w.data_ptr(), w.numel(), st))
    m_ref, s_ref = oracle.greedy_match(y.astype(np.float64))
    if na <= nb:
        m_ref = np.append(m_ref, -1)
    assert np.array_equal(mt.cpu().numpy(), m_ref)
    assert float(sc[0]) == s_ref
