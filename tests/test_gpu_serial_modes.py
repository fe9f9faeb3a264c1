"""The serial kernels' ways to decode (a whole warp, 16 or 8 lanes per shot)
give the same results bit for bit, at the sizes where the automatic choice and
the number of warps per CTA change, on codes with fewer qubits than lanes, on
ragged graphs in both table layouts, and whatever the batch leaves idle."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bpq():
    import paper_2407_11523_gb300 as bpq
    return bpq


def ragged(y):
    """Checks of 0 to 4 qubits, qubits on no check; with y, a Y entry (generic layout)."""
    H = np.zeros((9, 20), dtype=np.uint8)
    for i, (row, p) in enumerate([([0], 1), ([0, 1], 3), ([1, 2, 3], 1), ([2, 3, 4, 5], 3), ([5, 6], 1),
                                  ([6, 7, 8], 3), ([8], 3), ([9, 10, 11, 12], 1), ([], 1)]):
        H[i, row] = p
    if y:
        H[3, 4] = 2
    return H


def graphs(bpq):
    return [bpq.Tanner("planar", 2), bpq.Tanner("toric", 3), bpq.Tanner("xzzx", 6), bpq.Tanner("planar", 14),
            bpq.Tanner(H=ragged(False)), bpq.Tanner(H=ragged(True))]


@pytest.mark.parametrize("variant", ["plain", "momentum", "adagrad", "ewainit"])
def test_modes_agree(bpq, variant):
    for t in graphs(bpq):
        rng = np.random.default_rng(t.N)
        prior = torch.from_numpy(rng.uniform(0.01, 0.1, (t.N, 3)).astype(np.float32)).cuda()
        _, syn = bpq.sample(t, 0.03, 0.02, 0.03, seed=t.N, shot0=0, B=40000)
        for B, max_iter in ((1, 30), (3, 1), (153, 30), (2433, 30), (40000, 12)):
            s = syn[:B].contiguous()
            out = []
            for k in (0, 1, 2):
                t.set_serial_shots_per_warp(k)
                out.append(bpq.decode(t, s, prior, variant, max_iter=max_iter, schedule="serial"))
            t.set_serial_shots_per_warp(0)
            for o in out[1:]:
                for a, b in zip(out[0], o):
                    assert torch.equal(a, b), (t.N, variant, B)


def test_ragged_graphs_match_the_oracle(bpq):
    """Checks of one and two qubits and qubits on no check, against the float64 oracle's serial sweep (posteriors
    within 4e-4, the bound of the message tests)."""
    for y in (False, True):
        H = ragged(y)
        t = bpq.Tanner(H=H)
        rng = np.random.default_rng(1 + y)
        prior = rng.uniform(0.01, 0.2, (t.N, 3)).astype(np.float32)
        bits = rng.integers(0, 2, (12, t.M)).astype(np.uint8)
        bits[:, 8] = 0  # the empty check
        words = (bits.astype(np.int64) << np.arange(t.M)).sum(1).astype(np.int32)[:, None]
        rec = bpq.decode_trace(t, torch.from_numpy(words).cuda(), torch.from_numpy(prior).cuda(), variant="plain", T=4,
                               schedule="serial")
        for b in range(12):
            ref = oracle.trace(H, bits[b], prior.astype(np.float64), variant="plain", T=4, schedule="serial")
            q = rec["Q"][b].cpu().numpy()
            assert (np.abs(q - ref["Q"]) <= 4e-4 + 1e-6 * np.abs(ref["Q"])).all()
