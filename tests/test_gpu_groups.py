"""Shapes of shot groups that only some codes take: the smaller group made of
the batched kernel's left-over threads, threads that read more than two nodes
from the staged table, and the automatic shapes of two shots per thread.
Every result equals that of the one-shot kernel with two nodes per thread bit
for bit."""
import numpy as np
import pytest
import torch

import oracle
from inputs import random_tree_code
from test_gpu_batch import y_rotated

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bpq():
    import paper_2407_11523_gb300 as bpq
    return bpq


def make(bpq, kind, d):
    if kind == "generic":
        H = bpq.Tanner("planar", d).dense()
        return bpq.Tanner(H=y_rotated(H, np.random.default_rng(d).choice(H.shape[1], 30, replace=False)))
    if kind == "tree":
        return bpq.Tanner(H=random_tree_code(d, seed=d))
    return bpq.Tanner(kind, d)


def inputs(bpq, t, B, seed):
    ch = oracle.depolarizing(0.06)
    _, syn = bpq.sample(t, *ch, seed=seed, shot0=0, B=B)
    return syn, bpq.prior_tensor(t, *ch, jitter=2.0 ** -6)


def reference(bpq, t, syn, prior, variant, max_iter):
    t.set_shots_per_thread(1)
    t.set_launch(((max(t.N, t.M) + 1) // 2 + 31) // 32 * 32, 1)
    out = bpq.decode(t, syn, prior, variant, max_iter=max_iter)
    t.set_launch(0, 0)
    t.set_shots_per_thread(0)
    return out


def same(a, b, what):
    for x, y in zip(a, b):
        assert torch.equal(x, y), what


# threads of the groups + left over: 352 x 2 + 320, 384 x 2 + 256, 608 + 416, 640 + 384 (no padding), 1024 + 0;
# the left-over groups and the tables of initial messages need eight CTA loads of shots per SM
@pytest.mark.parametrize("variant", ["plain", "momentum", "adagrad", "ewainit"])
def test_left_over_threads_decode(bpq, variant):
    items = []
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for k, (kind, d, B) in enumerate([("planar", 25, 8 * sms), ("planar", 19, 700), ("generic", 19, 500), ("toric", 19, 300),
                                      ("planar", 25, 400), ("generic", 25, 1), ("toric", 25, 0), ("toric", 25, 350),
                                      ("planar", 5, 900), ("tree", 8, 600)]):
        t = make(bpq, kind, d)
        items.append((t, *inputs(bpq, t, B, 60 + k)))
    outs = bpq.BatchPlan(items, variant=variant, max_iter=40).run()
    for (t, syn, prior), got in zip(items, outs):
        if syn.shape[0]:
            same(got, reference(bpq, t, syn, prior, variant, 40), (t.N, variant))


# three and four nodes per thread, with a last pass that is full, partial or empty for some warps
@pytest.mark.parametrize("kind,d,T", [("planar", 9, 64), ("planar", 11, 64), ("generic", 9, 64), ("toric", 8, 32),
                                      ("toric", 15, 128), ("toric", 16, 128), ("xzzx", 11, 64), ("planar", 25, 320)])
@pytest.mark.parametrize("variant", ["plain", "momentum", "adagrad", "ewainit", "aewa"])
def test_more_nodes_per_thread_equal_two(bpq, kind, d, T, variant):
    t = make(bpq, kind, d)
    syn, prior = inputs(bpq, t, 300, 5)
    ref = reference(bpq, t, syn, prior, variant, 40)
    t.set_shots_per_thread(1)
    t.set_launch(T, 2)
    same(bpq.decode(t, syn, prior, variant, max_iter=40), ref, (kind, d, T, variant))


# one warp up to 96 nodes, two nodes per thread, 256 threads above 512 nodes where two CTAs fit, one group
# with a 32-bit or (where that is too large) a 16-bit slot table
@pytest.mark.parametrize("kind,d", [("planar", 2), ("planar", 7), ("toric", 4), ("planar", 8), ("toric", 9),
                                    ("planar", 17), ("planar", 18), ("toric", 18), ("planar", 25), ("toric", 27),
                                    ("planar", 31)])
@pytest.mark.parametrize("variant", ["plain", "momentum", "adagrad", "ewainit"])
def test_automatic_pair_shapes(bpq, kind, d, variant):
    t = make(bpq, kind, d)
    syn, prior = inputs(bpq, t, 401, 9)
    ref = reference(bpq, t, syn, prior, variant, 40)
    try:
        t.set_shots_per_thread(2)
        got = bpq.decode(t, syn, prior, variant, max_iter=40)
    except bpq.BPQError:
        # no pair shape fits: the automatic choice then keeps to one shot per thread
        t.set_shots_per_thread(0)
        assert t.shots_per_thread(variant) == 1
        return
    same(got, ref, (kind, d, variant))
