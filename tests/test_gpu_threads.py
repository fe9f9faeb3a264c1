"""Calls from several host threads at once, each thread on a code, a stream
and buffers of its own."""
import ctypes
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def in_threads(calls, rounds):
    """calls: one list of (entry point, arguments) per thread, made over and
    over; returns the error codes that are not 0 with their messages."""
    import paper_2407_11523_gb300 as bpq

    failures, go = set(), threading.Barrier(len(calls))

    def loop(mine):
        go.wait()
        for _ in range(rounds):
            for f, args in mine:
                rc = f(*args)
                if rc:
                    failures.add((rc, bpq.lib().bpq_last_error()))

    ts = [threading.Thread(target=loop, args=(c,)) for c in calls]
    for th in ts:
        th.start()
    for th in ts:
        th.join()
    torch.cuda.synchronize()
    return failures


def p(x):
    return ctypes.c_void_p(x.data_ptr())


# Codes whose needs of shared memory differ, all above the 48 KB that a launch gets without asking (enough
# shots for the sampler's tiles)
def test_sample_and_check_logical_of_two_large_codes():
    import paper_2407_11523_gb300 as bpq

    calls, kept = [], []
    B = 12 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    for kind, d in [("planar", 26), ("toric", 32)] * 2:
        t, stream = bpq.Tanner(kind, d).upload(), torch.cuda.Stream()
        err, syn = bpq.sample(t, 0.02, 0.02, 0.02, seed=1, shot0=0, B=B)
        out = [torch.empty_like(err), torch.empty_like(syn), torch.empty(B, dtype=torch.uint8, device="cuda")]
        s, c = ctypes.c_void_p(stream.cuda_stream), ctypes.c_double(0.02)
        kept.append((t, stream, err, syn, out))
        calls.append([(bpq.lib().bpq_sample, (t.handle, c, c, c, 1, 0, B, p(out[0]), p(out[1]), s)),
                      (bpq.lib().bpq_check_logical, (t.handle, p(out[0]), p(out[0]), B, p(out[2]), s))])
    torch.cuda.synchronize()
    assert not in_threads(calls, 4000)
    for t, stream, err, syn, out in kept:
        assert torch.equal(out[0], err) and torch.equal(out[1], syn) and not out[2].any()


# One decode kernel (one shot per thread, two nodes per thread) on codes of 27 to 78 KB of shared memory
@pytest.mark.parametrize("schedule", ["bpq_decode", "bpq_decode_serial"])
def test_decode_of_two_codes_of_one_kernel(schedule):
    import paper_2407_11523_gb300 as bpq

    calls, kept, params = [], [], bpq.make_params("ewainit")
    for d in [15, 26] * 2:
        t, stream = bpq.Tanner("planar", d).upload(), torch.cuda.Stream()
        t.set_shots_per_thread(1)
        t.set_launch((t.N + 63) // 64 * 32, 1)
        prior = bpq.prior_tensor(t, 0.01, 0.01, 0.01)
        _, syn = bpq.sample(t, 0.01, 0.01, 0.01, seed=1, shot0=0, B=20)
        work = bpq.workspace()
        ref = bpq.decode(t, syn, prior, "ewainit", max_iter=4, work=work,
                         schedule="serial" if "serial" in schedule else "parallel")
        out = [torch.empty_like(x) for x in ref]
        kept.append((t, stream, syn, prior, work, ref, out))
        calls.append([(getattr(bpq.lib(), schedule),
                       (t.handle, p(syn), p(prior), bpq.EWAINIT, ctypes.byref(params), 4, 20, *map(p, out), p(work),
                        ctypes.c_void_p(stream.cuda_stream)))])
    torch.cuda.synchronize()
    assert not in_threads(calls, 8000)
    for *_, ref, out in kept:
        assert all(torch.equal(x, y) for x, y in zip(ref, out))


# A plan of a small code made between another plan's making and its launch
def test_batch_plan_after_another_plan():
    import paper_2407_11523_gb300 as bpq

    plans, refs = [], []
    for d in (25, 3):
        t = bpq.Tanner("planar", d)
        _, syn = bpq.sample(t, 0.01, 0.01, 0.01, seed=1, shot0=0, B=50)
        prior = bpq.prior_tensor(t, 0.01, 0.01, 0.01)
        refs.append(bpq.decode(t, syn, prior, "ewainit", max_iter=20))
        plans.append(bpq.BatchPlan([(t, syn, prior)], variant="ewainit", max_iter=20))
    for plan, ref in zip(plans, refs):
        assert all(torch.equal(x, y) for x, y in zip(ref, plan.run()[0]))
