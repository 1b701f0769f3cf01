"""The team tier with fewer scratch slots than CTAs: pairs on several team levels
in workspaces of few slots give what a workspace with a slot for every pair
gives, and the same bits every time."""
import ctypes as C

import numpy as np
import pytest
import torch

from gen.cfg_grammar import structured_cfg
from _helpers import valid_matching

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
B = pytest.importorskip("paper_1707_02423_gb300._binding")
DEV = "cuda"


def workload(large, small):
    """`large` pairs of 376 x 376 blocks, `small` of 230 x 230: two team levels
    and more, by the number of CTAs that are left for them."""
    rng = np.random.default_rng(11)
    cfgs = [structured_cfg(rng, n, 6, 12) for n in 4 * [376] + 8 * [230]]
    pairs = [(k % 4, (k + 1 + k // 4) % 4) for k in range(large)]
    pairs += [(4 + k % 8, 4 + (3 * k + 1 + k // 8) % 8) for k in range(small)]
    pairs = np.array(pairs, np.int32)
    pk = api.Pack(cfgs, 13, device=DEV)
    one = api.Pack([structured_cfg(rng, 1, 6, 12)], 13, device=DEV)
    fixed = api.ws_size(one, one, np.zeros_like(pairs), B.params())  # the part without slots
    full = api.ws_size(pk, pk, pairs, B.params())
    return cfgs, pairs, pk, fixed, (full - fixed) // len(pairs)


@pytest.mark.parametrize("large,small", [(4, 18), (12, 110), (60, 60)])
@pytest.mark.parametrize("slots", [2, 7, 16, 17, 19, 21, 43, 104])
def test_similarity(large, small, slots):
    cfgs, pairs, pk, fixed, slot = workload(large, small)
    if slots >= len(pairs):
        pytest.skip("a slot for every pair")
    om = torch.linspace(0.5, 1.5, 13, device=DEV)
    ref = api.similarity(pk, pk, pairs, om, want_x=True, want_match=True)
    first = None
    for _ in range(3):
        r = api.similarity(pk, pk, pairs, om, want_x=True, want_match=True, ws_bytes=fixed + slots * slot)
        # either side is within 1e-5 of the exact X
        assert (r.X - ref.X).abs().max().item() <= 2e-5
        if first is not None:
            assert torch.equal(r.X, first.X) and torch.equal(r.scores, first.scores) and torch.equal(r.match, first.match)
        first = r
    X, sc, mt = first.X.cpu().numpy().astype(np.float64), first.scores.cpu().numpy(), first.match.cpu().numpy()
    for p, (a, b) in enumerate(pairs):  # the score is the matching's, in the call's own X
        m = mt[r.m_off[p]:r.m_off[p + 1]]
        assert valid_matching(m, cfgs[a].n, cfgs[b].n)
        x = X[r.x_off[p]:r.x_off[p + 1]].reshape(cfgs[a].n, -1)
        assert abs(sc[p] - x[np.arange(len(m)), m].sum()) <= 1e-5


@pytest.mark.parametrize("slots", [7, 17, 19, 43])
def test_given_matrices(slots):
    cfgs, pairs, pk, fixed, slot = workload(12, 110)
    g = torch.Generator(device=DEV).manual_seed(3)
    x_off, m_off = api.out_offsets(pk, pk, pairs)
    # multiples of 1/8 below 2**12: the scores are exact
    X = torch.randint(0, 1 << 15, (int(x_off[-1]),), generator=g, device=DEV).float() / 8.0
    ref = api.match(pk, pk, pairs, X)
    ws = torch.empty(fixed + slots * slot, dtype=torch.uint8, device=DEV)
    sc = torch.empty(len(pairs), device=DEV)
    mt = torch.empty(int(m_off[-1]), dtype=torch.int32, device=DEV)
    d_pairs = torch.from_numpy(pairs).to(DEV)
    st = torch.cuda.current_stream().cuda_stream
    for _ in range(3):
        B.check(B.lib().cf_match(pk.dev.data_ptr(), pk.dev.data_ptr(), d_pairs.data_ptr(), len(pairs),
                                 C.byref(B.params()), None, X.data_ptr(), mt.data_ptr(), sc.data_ptr(), ws.data_ptr(),
                                 ws.numel(), st))
        B.check(B.lib().cf_status_check(ws.data_ptr(), st))
        assert torch.equal(sc, ref.scores) and torch.equal(mt, ref.match)


def test_noalloc():
    """The static workspace of 32 MiB: 19 slots for these 22 pairs."""
    cfgs, pairs, pk, _, _ = workload(4, 18)
    om = torch.ones(13, device=DEV)
    ref = api.similarity(pk, pk, pairs, om, want_x=True)
    d_pairs = torch.from_numpy(pairs).to(DEV)
    X, sc = torch.empty_like(ref.X), torch.empty_like(ref.scores)
    st = torch.full((1,), -7, dtype=torch.int32, device=DEV)
    for _ in range(3):
        B.check(B.lib().cf_similarity_noalloc(pk.dev.data_ptr(), pk.dev.data_ptr(), d_pairs.data_ptr(), len(pairs),
                                              C.byref(B.params(0.8, 40)), om.data_ptr(), X.data_ptr(), sc.data_ptr(),
                                              None, st.data_ptr(), torch.cuda.current_stream().cuda_stream))
        assert int(st.item()) == 0
        assert (X - ref.X).abs().max().item() <= 2e-5
