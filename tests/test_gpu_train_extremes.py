"""Training losses and gradients where the channel or the code is extreme:
noise of one Pauli only (two of a qubit's prior probabilities are 0, so two of
its log-likelihoods are infinite), no checks, messages near the top of their
range."""
import numpy as np
import pytest
import torch

from oracle import unrolled
from test_gpu_train import oracle_inputs, params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bpq():
    import paper_2407_11523_gb300 as bpq
    return bpq


# The reference has 1e-30 in place of 0: log-likelihoods of 66 and more instead of infinity, beyond the
# clip of 30 in every message, and probabilities that change no sum of fp32 or of the bars below (those of
# the planar d = 9 tests; losses under 1e-9, where every qubit is certain, count as equal).  The gradient for alpha multiplies an infinite prior by 0 and is no number.
@pytest.mark.parametrize("kind,d", [("planar", 5), ("toric", 4), ("xzzx", 5)])
@pytest.mark.parametrize("ch", [(0.06, 0.0, 0.0), (0.0, 0.06, 0.0), (0.0, 0.0, 0.06), (0.04, 0.0, 0.03)])
@pytest.mark.parametrize("kind_of_loss", ["posterior", "coset"])
def test_noise_of_some_paulis_only(bpq, kind, d, ch, kind_of_loss):
    T, B = 6, 16
    t = bpq.Tanner(kind, d)
    err, syn = bpq.sample(t, *ch, seed=5, shot0=0, B=B)
    prior = bpq.prior_tensor(t, *ch)
    H, s, e, pri = oracle_inputs(t, err, syn, np.maximum(ch, 1e-30))
    Lg = t.logicals()
    a, b, w = params(T, t.E, 6, spread=0.1)
    ts = [torch.tensor(x, device="cuda", dtype=torch.float32, requires_grad=True) for x in (a, b, w)]
    kw = dict(loss="coset", logicals=Lg) if kind_of_loss == "coset" else {}
    L = bpq.unrolled_loss(t, syn, err, prior, *ts, T=T, ckpt_every=4, **kw)
    L.backward()
    kw = dict(kind="coset", logicals=Lg) if kind_of_loss == "coset" else {}
    ref = unrolled.loss_and_grads(H, s, e, pri, a, b, w, T, **kw)
    assert L.item() == pytest.approx(ref[0], rel=2e-4, abs=1e-9)
    for x, r in zip(ts[1:], ref[2:]):
        g = x.grad.cpu().numpy().astype(np.float64)
        assert np.abs(g - r).max() <= 2e-3 * np.abs(r).max() + 1e-7, (np.abs(g - r).max(), np.abs(r).max())


# A code without checks: every posterior is the prior, the coset loss has no check terms, and -log P of the
# logical operator Z on qubit 0 is that of its X and Y errors.  rel 1e-6: a few roundings of fp32.
def test_code_without_checks(bpq):
    import ctypes

    t = bpq.Tanner(H=np.zeros((0, 3), np.uint8)).upload()
    prior = torch.tensor([[0.03, 0.02, 0.05], [0.1, 0.2, 0.1], [0.2, 0.1, 0.3]], device="cuda")
    err = torch.tensor([[0, 1, 2], [1, 0, 0]], dtype=torch.uint8, device="cuda")
    some = torch.full((4,), 0.5, device="cuda")  # weights of each of the T = 2 iterations; unused syndromes and edges
    lg = torch.tensor([[3, 0, 0]], dtype=torch.uint8, device="cuda")
    nbytes = bpq.lib().bpq_train_workspace_bytes(t.handle, 0, 2, 2, 1)
    work, loss = torch.empty(nbytes, dtype=torch.uint8, device="cuda"), torch.empty(1, device="cuda")
    p = lambda x: ctypes.c_void_p(x.data_ptr())
    ld = bpq._binding.TrainLoss(1, lg.data_ptr(), 1)
    rc = bpq.lib().bpq_train_forward(t.handle, 0, p(some), p(err), p(prior), 2, 2, 1, p(some), p(some), None, p(some),
                                     30.0, ctypes.byref(ld), p(loss), None, p(work), nbytes,
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, bpq.lib().bpq_last_error()
    assert loss.item() == pytest.approx(-(np.log(0.95) + np.log(0.05)) / 2, rel=1e-6)


# Messages of 88.0 (both anticommuting Paulis of an edge have probability 3e-39), for which expm1 is above
# 2^126: one iteration of checks of degree 2, 3 and 4 with weights of 1/2 against float64.  Bar: the largest
# sum is about 260, of which fp32 holds 1.5e-5; expm1 and log1p are within a few such steps.
def test_messages_near_the_top_of_the_range(bpq):
    H = np.zeros((3, 7), np.uint8)
    H[0, [0, 1]] = H[1, [1, 2, 3]] = H[2, [3, 4, 5, 6]] = 3
    t = bpq.Tanner(H=H)
    prior = np.full((7, 3), 3e-39, dtype=np.float32)
    syn = np.array([[0], [5], [7]], np.int32)
    a, b, w = np.full(1, 0.5), np.zeros(1), np.full(t.E, 0.5)
    dev = lambda x, dt=torch.float32: torch.tensor(x, dtype=dt, device="cuda")
    Q, _ = bpq.unrolled_posterior(t, dev(syn, torch.int32), torch.zeros((3, 7), dtype=torch.uint8, device="cuda"),
                                  torch.from_numpy(prior).cuda(), dev(a), dev(b), dev(w), T=1, ckpt_every=1,
                                  msg_clip=88.5)
    s = (syn >> np.arange(3)) & 1
    ref = unrolled.forward(unrolled.Graph(H), s, prior.astype(np.float64), *map(torch.tensor, (a, b, w)), T=1,
                           clip=88.5).numpy()
    assert np.abs(Q.cpu().numpy() - ref).max() <= 2e-4
