"""Packing of a request trace by Server.replay: no request, one request, codes
of several sizes in any order, syndromes of other integer types, outputs in
page-locked or pageable memory; every result equals bpq_decode's."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [0, 1, 37])
@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("dtype", [np.uint32, np.int64])
def test_replay_packs_any_trace(R, pinned, dtype):
    import paper_2407_11523_gb300 as bpq
    codes = [bpq.Tanner("planar", 5), bpq.Tanner("toric", 8), bpq.Tanner("xzzx", 7)]
    ch = oracle.depolarizing(0.06)
    priors = [bpq.prior_tensor(t.upload(), *ch) for t in codes]
    code = np.random.default_rng(R).integers(0, len(codes), R)
    syns, refs = [], []
    for r, c in enumerate(code):
        _, syn = bpq.sample(codes[c], *ch, seed=r, shot0=0, B=1)
        refs.append([x.cpu().numpy()[0] for x in bpq.decode(codes[c], syn, priors[c], "ewainit", max_iter=50)])
        syns.append(syn.cpu().numpy().view(np.uint32)[0].astype(dtype))
    srv = bpq.Server(codes, priors, "ewainit", max_iter=50, mode="slots", slots_per_code=8)
    ests, conv, iters, done, _ = srv.replay(code, np.zeros(R), syns, pinned=pinned)
    assert len(ests) == conv.size == iters.size == done.size == R
    for r in range(R):
        assert ests[r].dtype == np.uint8 and np.array_equal(ests[r], refs[r][0])
        assert conv[r] == refs[r][1] and iters[r] == refs[r][2]
    if R == 37:
        with pytest.raises(IndexError):
            srv.replay(np.full(R, 3), np.zeros(R), syns, pinned=pinned)
        with pytest.raises(ValueError):
            srv.replay(code, np.zeros(R), syns[:-1], pinned=pinned)
