"""Serial schedule, two shots per warp, on codes whose two shots just fit in
shared memory."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


# Check i on qubits i, i + 1, i + 37, i + 211 (mod N) with Paulis X, Y, Z, X: the generic table layout
@pytest.mark.parametrize("N", [2001, 2002])
def test_two_shots_per_warp_at_the_limit(N):
    import paper_2407_11523_gb300 as bpq

    M = N * 7 // 8
    H = np.zeros((M, N), np.uint8)
    for k, step in enumerate((0, 1, 37, 211)):
        H[np.arange(M), (np.arange(M) + step) % N] = k % 3 + 1
    t = bpq.Tanner(H=H)
    _, syn = bpq.sample(t, 0.01, 0.01, 0.01, seed=2, shot0=0, B=5)
    prior = bpq.prior_tensor(t, 0.01, 0.01, 0.01)
    outs = []
    for k in (1, 2):
        t.set_serial_shots_per_warp(k)
        outs.append(bpq.decode(t, syn, prior, "ewainit", max_iter=6, schedule="serial"))
    assert all(torch.equal(x, y) for x, y in zip(*outs))
