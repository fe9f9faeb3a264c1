"""The sampler's two kernels, one CTA per shot for few shots and one per 32
shots for many: a batch above the line equals the same shots drawn in batches
below it, bit for bit, at the edges of the 32-shot tiles and with an error
buffer off the 4-byte boundary."""
import numpy as np
import pytest
import torch

from test_gpu_batch import y_rotated

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,d", [("planar", 2), ("planar", 7), ("toric", 8), ("xzzx", 13), ("generic", 9),
                                    ("planar", 25), ("toric", 32)])
@pytest.mark.parametrize("ch", [(0.05, 0.02, 0.1), (0.0, 0.0, 0.3)])
def test_many_shots_equal_few_at_a_time(kind, d, ch):
    import paper_2407_11523_gb300 as bpq

    if kind == "generic":
        H = bpq.Tanner("planar", d).dense()
        t = bpq.Tanner(H=y_rotated(H, np.random.default_rng(d).choice(H.shape[1], 30, replace=False)))
    else:
        t = bpq.Tanner(kind, d)
    line = 12 * torch.cuda.get_device_properties(0).multi_processor_count
    for B in (line, line + 1, line + 63):
        err = torch.full((B * t.N + 1,), 77, dtype=torch.uint8, device="cuda")[B % 2:][:B * t.N].view(B, t.N)
        err, syn = bpq.sample(t, *ch, seed=9, shot0=2 ** 40 + 5, B=B, err=err)
        cuts = [0, 1, 34, line // 2, line - 1, line, B]
        for a, b in zip(cuts, cuts[1:]):
            if b > a:
                e, s = bpq.sample(t, *ch, seed=9, shot0=2 ** 40 + 5 + a, B=b - a)
                assert torch.equal(e, err[a:b]) and torch.equal(s, syn[a:b]), (B, a, b)


# The fault that this mends: few shots of a large code took 36 us whatever their number.  Bar: twice the
# time of the smallest code, whose calls are nothing but launches (1.05 times measured; 4 with the tiles).
def test_few_shots_of_a_large_code_cost_a_launch():
    import paper_2407_11523_gb300 as bpq

    codes = [(bpq.Tanner("planar", d).upload(), d) for d in (3, 31)]
    us = []
    for t, _ in codes:
        err, syn = bpq.sample(t, 0.02, 0.02, 0.02, seed=1, shot0=0, B=40)
        ts = []
        for _ in range(15):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for _ in range(20):
                bpq.sample(t, 0.02, 0.02, 0.02, seed=1, shot0=0, B=40, err=err, syn=syn)
            b.record()
            b.synchronize()
            ts.append(a.elapsed_time(b))
        us.append(np.median(ts))
    assert us[1] <= 2 * us[0], us
