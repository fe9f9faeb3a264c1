"""Small batches take kernels of their own (one CTA per shot and several lanes
per node, or one node per thread): their results equal the queue kernels' bit
for bit, for every variant, at the sizes where the choice of lanes changes and
on graphs with ragged checks, checks of one qubit and qubits without checks."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bpq():
    import paper_2407_11523_gb300 as bpq
    return bpq


def both(bpq, t, syn, prior, variant, max_iter):
    """Outputs of the automatic choice and of the queue kernel with two nodes per thread."""
    work = bpq.workspace()
    work.fill_(0xFF)  # need not be initialised
    auto = bpq.decode(t, syn, prior, variant, max_iter=max_iter, work=work)
    assert bpq.decode_status(work) == 0
    nodes = max(t.N, t.M)
    t.set_shots_per_thread(1)
    t.set_launch(((nodes + 1) // 2 + 31) // 32 * 32, 1)
    queue = bpq.decode(t, syn, prior, variant, max_iter=max_iter)
    t.set_launch(0, 0)
    t.set_shots_per_thread(0)
    return auto, queue


def check(bpq, t, syn, prior, variant, max_iter):
    auto, queue = both(bpq, t, syn, prior, variant, max_iter)
    for a, b in zip(auto, queue):
        assert torch.equal(a, b), (t.N, variant, syn.shape[0], max_iter)


# lanes per node at one shot per SM: 4 up to 160 nodes, 2 up to 320, then 1; none above 1024
@pytest.mark.parametrize("kind,d", [("planar", 2), ("planar", 9), ("toric", 8), ("planar", 10), ("xzzx", 13),
                                    ("toric", 13), ("toric", 15), ("planar", 23), ("planar", 24)])
@pytest.mark.parametrize("variant", ["plain", "momentum", "adagrad", "ewainit", "aewa"])
def test_small_batches_equal_the_queue(bpq, kind, d, variant):
    t = bpq.Tanner(kind, d)
    ch = oracle.depolarizing(0.07)
    prior = bpq.prior_tensor(t, *ch, jitter=2.0 ** -6)
    _, syn = bpq.sample(t, *ch, seed=0x51A + d, shot0=0, B=1300)
    for B in (1, 2, 153, 305, 457, 1300):  # shots per SM: 1, 1, 2, 3, 4, 9
        check(bpq, t, syn[:B].contiguous(), prior, variant, 30)
    for max_iter in (1, 255):
        check(bpq, t, syn[:7].contiguous(), prior, variant, max_iter)
    zero = torch.zeros((3, t.W), dtype=torch.int32, device="cuda")
    check(bpq, t, zero, prior, variant, 5)


@pytest.mark.parametrize("variant", ["plain", "momentum", "adagrad", "ewainit"])
def test_small_batches_on_ragged_graphs(bpq, variant):
    rng = np.random.default_rng(3)
    H = np.zeros((9, 20), dtype=np.uint8)  # at most two X and two Z edges a qubit: the split layout
    for i, (row, p) in enumerate([([0], 1), ([0, 1], 3), ([1, 2, 3], 1), ([2, 3, 4, 5], 3), ([5, 6], 1),
                                  ([6, 7, 8], 3), ([8], 3), ([9, 10, 11, 12], 1), ([], 1)]):
        H[i, row] = p  # qubits 13 .. 19 are on no check; the last check is empty
    t = bpq.Tanner(H=H)
    assert t.layout() == 1
    prior = torch.from_numpy(rng.uniform(0.01, 0.2, (20, 3)).astype(np.float32)).cuda()
    syn = torch.from_numpy(rng.integers(0, 2 ** 8, (40, 1)).astype(np.int32)).cuda()
    for B in (1, 40):
        check(bpq, t, syn[:B].contiguous(), prior, variant, 20)
