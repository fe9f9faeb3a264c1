"""What one shot under the serial schedule costs beside its sweeps: staging the
tables and making the initial messages, which the warps of a CTA share."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def microseconds(call):
    call()
    ts = []
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(20):
            call()
        b.record()
        b.synchronize()
        ts.append(a.elapsed_time(b) * 50)
    return float(np.median(ts))


# One warp alone took 2.35 and 2.15 sweeps of these codes for it (start and launch included), sixteen take
# 1.14 and 0.99; bar 1.6.  The syndrome is of noise that nine sweeps do not converge on.
@pytest.mark.parametrize("kind,d", [("planar", 25), ("toric", 27)])
def test_start_of_one_shot(kind, d):
    import paper_2407_11523_gb300 as bpq

    t = bpq.Tanner(kind, d)
    _, syn = bpq.sample(t, 0.07, 0.07, 0.07, seed=3, shot0=0, B=1)
    prior, work = bpq.prior_tensor(t, 0.02, 0.02, 0.02), bpq.workspace()
    out = bpq.decode(t, syn, prior, "ewainit", max_iter=9, schedule="serial")
    assert out[2].item() == 9
    one, nine = (microseconds(lambda: bpq.decode(t, syn, prior, "ewainit", max_iter=n, schedule="serial", out=out,
                                                 work=work)) for n in (1, 9))
    sweep = (nine - one) / 8
    assert one - sweep <= 1.6 * sweep, (one, nine)
