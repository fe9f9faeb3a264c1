"""Bounds-checked decoding of small batches (bpq_set_debug_checks): the copy
that runs is that of the kernel that runs without the checks, one CTA per shot
with 4, 2 or 1 lanes per node.  That kernel takes no shot from the queue, so the
queue word of the workspace stays 0, which tells it from the others."""
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,d", [("planar", 5), ("toric", 4), ("planar", 9), ("xzzx", 13), ("toric", 15)])
@pytest.mark.parametrize("variant", ["plain", "momentum", "adagrad", "ewainit"])
@pytest.mark.parametrize("per_sm", [0, 1, 2])
def test_small_batches_run_their_own_checked_copy(kind, d, variant, per_sm):
    import paper_2407_11523_gb300 as bpq

    t = bpq.Tanner(kind, d)
    ch = oracle.depolarizing(0.08)
    B = max(1, per_sm * torch.cuda.get_device_properties(0).multi_processor_count)
    _, syn = bpq.sample(t, *ch, seed=31, shot0=0, B=B)
    prior = bpq.prior_tensor(t, *ch)
    runs = []
    for on in (False, True):
        t.set_debug_checks(on)
        work = bpq.workspace()
        out = bpq.decode(t, syn, prior, variant, max_iter=30, work=work)
        assert bpq.decode_status(work) == 0
        runs.append((out, int(work[:4].view(torch.int32).item())))
    (ref, taken), (got, taken_checked) = runs
    assert (taken == 0) == (taken_checked == 0)
    assert all(torch.equal(x, y) for x, y in zip(ref, got))
