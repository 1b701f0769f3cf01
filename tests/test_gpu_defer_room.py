"""The default configuration at 32 pairs per SM and more in a workspace without
room for the ranked lists: the forward takes the matching's steps itself, with
the bits of the call that defers them; and on a pair list of the device in a
workspace for any pairs."""
import numpy as np
import pytest
import torch

from gen.cfg_grammar import structured_cfg

pytestmark = pytest.mark.gpu
api = pytest.importorskip("paper_1707_02423_gb300.api")
B = pytest.importorskip("paper_1707_02423_gb300._binding")
DEV = "cuda"


def test_same_bits():
    rng = np.random.default_rng(9)
    P = 32 * torch.cuda.get_device_properties(0).multi_processor_count + 5
    cfgs = [structured_cfg(rng, int(n), 5, 7) for n in rng.integers(20, 45, 30)] + [structured_cfg(rng, 300, 5, 7)]
    pairs = rng.integers(0, 30, (P, 2)).astype(np.int32)
    pairs[7], pairs[8] = (30, 3), (30, 30)
    pk = api.Pack(cfgs, 8, device=DEV)
    om = torch.linspace(0.5, 1.5, 8, device=DEV)
    small = api.ws_size(pk, pk, pairs, B.params(tune=1))
    full = api.ws_size(pk, pk, pairs, B.params())
    assert small < full <= api.ws_size_any(pk, pk, P, B.params())
    ref = api.similarity(pk, pk, pairs, om, want_match=True)
    for size in (small, full - 1):
        ws = api.Workspace(DEV)  # one of this size: Workspace keeps the largest it was asked for
        for flags in (0, B.CF_FLAG_REUSE_PLAN):
            r = api.similarity(pk, pk, pairs, om, want_match=True, ws=ws, ws_bytes=size, flags=flags)
            assert ws.buf.numel() == size
            assert torch.equal(r.scores, ref.scores) and torch.equal(r.match, ref.match)
    sc, mt = torch.empty_like(ref.scores), torch.empty_like(ref.match)
    api.similarity_dev(pk, pk, torch.from_numpy(pairs).to(DEV), om, scores=sc, match=mt, ws=api.Workspace(DEV),
                       ws_bytes=api.ws_size_any(pk, pk, P, B.params()))
    assert torch.equal(sc, ref.scores) and torch.equal(mt, ref.match)
