"""Loss and gradients of the unrolled decoders at the edges of the training
kernels' shapes, against the float64 oracle: fewer nodes than a warp, node
counts around a CTA's 320 threads (the kernels' two register budgets), two and
four logical operators, Pauli Y entries, and batches of one and of odd size
(the sums over shots).  Bars: those of the planar d = 9 tests (loss 2e-4,
gradients 2e-3 of their largest entry), which hold for fp32 messages of any
code at these depths."""
import numpy as np
import pytest
import torch

import oracle
from oracle import codes, unrolled
from test_gpu_batch import y_rotated
from test_gpu_train import oracle_inputs, params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,d,B", [("planar", 2, 1), ("planar", 3, 65), ("generic", 5, 3), ("toric", 4, 5),
                                      ("planar", 13, 2), ("toric", 13, 1)])
@pytest.mark.parametrize("model", ["ewainit", "momentum"])
@pytest.mark.parametrize("kind_of_loss", ["posterior", "coset"])
def test_training_shapes(kind, d, B, model, kind_of_loss):
    import paper_2407_11523_gb300 as bpq
    T = 6
    if kind == "generic":
        H = bpq.Tanner("planar", d).dense()
        t = bpq.Tanner(H=y_rotated(H, np.random.default_rng(d).choice(H.shape[1], 12, replace=False)))
    else:
        t = bpq.Tanner(kind, d)
    ch = oracle.depolarizing(0.06)
    err, syn = bpq.sample(t, *ch, seed=71 + d, shot0=0, B=B)
    prior = bpq.prior_tensor(t, *ch)
    H, s, e, pri = oracle_inputs(t, err, syn, ch)
    Lg = codes.logical_operators(H)
    a, b, w = params(T, t.E, 72 + d, spread=0.1)
    gm = 0.3 + 0.05 * np.random.default_rng(73).standard_normal(T) if model == "momentum" else None
    ts = [torch.tensor(x, device="cuda", dtype=torch.float32, requires_grad=True)
          for x in (a, b, w) + ((gm,) if gm is not None else ())]
    kw = dict(loss="coset", logicals=Lg) if kind_of_loss == "coset" else {}
    L = bpq.unrolled_loss(t, syn, err, prior, *ts[:3], T=T, ckpt_every=4, model=model,
                          gamma=ts[3] if gm is not None else None, **kw)
    L.backward()
    kw = dict(kind="coset", logicals=Lg) if kind_of_loss == "coset" else {}
    ref = unrolled.loss_and_grads(H, s, e, pri, a, b, w, T, model=model, gamma=gm, **kw)
    assert L.item() == pytest.approx(ref[0], rel=2e-4)
    for x, r in zip(ts, ref[1:]):
        g = x.grad.cpu().numpy().astype(np.float64)
        assert np.abs(g - r).max() <= 2e-3 * np.abs(r).max() + 1e-7, (np.abs(g - r).max(), np.abs(r).max())
