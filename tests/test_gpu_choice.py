"""The launch that bpq_decode and the batched plan choose by themselves against
others that can be asked for: never much slower.  Each case is one that an
earlier rule got wrong; the ratio it had then stands beside it, and the bar lies
between that and what the rule that replaced it has (1.0 to 1.04)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bpq():
    import paper_2407_11523_gb300 as bpq
    return bpq


def milliseconds(call):
    call()
    ts = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(5):
            call()
        b.record()
        b.synchronize()
        ts.append(a.elapsed_time(b) / 5)
    return float(np.median(ts))


def inputs(bpq, kind, d, p, B):
    t = bpq.Tanner(kind, d)
    _, syn = bpq.sample(t, p / 3, p / 3, p / 3, seed=1, shot0=0, B=B)
    return t, syn, bpq.prior_tensor(t, p / 3, p / 3, p / 3, jitter=2.0 ** -16)


def decoding(bpq, t, syn, prior, variant):
    work, out = bpq.workspace(), bpq.decode(t, syn, prior, variant, max_iter=100)
    return out, lambda: bpq.decode(t, syn, prior, variant, max_iter=100, out=out, work=work)


# Against one shot per thread
@pytest.mark.parametrize("kind,d,variant,p,B,bar", [
    ("planar", 22, "ewainit", 0.08, 40000, 1.12),   # 1.22: the table of byte offsets left one CTA per SM
    ("planar", 23, "momentum", 0.03, 20000, 1.12),  # 1.24: one CTA per SM against two
])
def test_pairs_against_one_shot(bpq, kind, d, variant, p, B, bar):
    t, syn, prior = inputs(bpq, kind, d, p, B)
    out, call = decoding(bpq, t, syn, prior, variant)
    ref = [x.clone() for x in out]
    ms = milliseconds(call)
    t.set_shots_per_thread(1)
    assert ms <= bar * milliseconds(call)
    assert all(torch.equal(x, y) for x, y in zip(ref, out))


@pytest.mark.parametrize("kind,d,variant,p,B,bar", [
    ("planar", 4, "plain", 0.03, 1000000, 1.08),    # 1.18: one-warp groups either way
    ("toric", 13, "adagrad", 0.03, 60000, 1.04),    # 1.09: 64 shots per group
    ("planar", 16, "ewainit", 0.03, 60000, 1.05),   # 1.12: 64 shots per group
])
def test_when_pairs_start(bpq, kind, d, variant, p, B, bar):
    test_pairs_against_one_shot(bpq, kind, d, variant, p, B, bar)


# Against two nodes per thread
@pytest.mark.parametrize("kind,d,variant,p,B,bar", [
    ("toric", 20, "plain", 0.03, 700, 1.06),        # 1.14: one node per thread
    ("toric", 15, "adagrad", 0.03, 300, 1.02),      # 1.05: one CTA per shot
])
def test_small_batches_against_two_nodes_per_thread(bpq, kind, d, variant, p, B, bar):
    t, syn, prior = inputs(bpq, kind, d, p, B)
    out, call = decoding(bpq, t, syn, prior, variant)
    ref = [x.clone() for x in out]
    ms = milliseconds(call)
    t.set_shots_per_thread(1)
    t.set_launch((max(t.N, t.M) + 63) // 64 * 32, 0)
    assert ms <= bar * milliseconds(call)
    assert all(torch.equal(x, y) for x, y in zip(ref, out))


# A plan just above eight CTA loads per SM against one just below, per shot: the ones above form a group of
# the threads left over where there are one or two full groups
@pytest.mark.parametrize("d,groups,bar", [(7, 10, 1.12), (15, 4, 1.08)])  # 1.31, 1.13
def test_plan_above_and_below_eight_loads(bpq, d, groups, bar):
    line = 8 * torch.cuda.get_device_properties(0).multi_processor_count * groups
    ms = []
    for B in (line - groups, line + groups):
        t, syn, prior = inputs(bpq, "planar", d, 0.05, B)
        assert t.batch_launch("ewainit")[1] == groups
        plan = bpq.BatchPlan([(t, syn, prior)], variant="ewainit", max_iter=100)
        ms.append(milliseconds(plan.run))
    assert ms[1] <= bar * ms[0], ms
