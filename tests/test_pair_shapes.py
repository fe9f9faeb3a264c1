"""Two shots per thread have a launch shape on every code that the GPU tests of
the automatic shapes go through, for every variant (no GPU needed), and none on
the largest torus with variant state."""
import pytest

import paper_2407_11523_gb300 as bpq


@pytest.mark.parametrize("kind,d", [("planar", 2), ("planar", 7), ("toric", 4), ("planar", 8), ("toric", 9),
                                    ("planar", 17), ("planar", 18), ("toric", 18), ("planar", 22), ("planar", 25),
                                    ("toric", 27), ("planar", 31)])
def test_pair_shape_fits(kind, d):
    t = bpq.Tanner(kind, d)
    assert [t.shots_per_thread(v) for v in ("plain", "momentum", "adagrad", "ewainit")] == [2, 2, 2, 2]
    t.set_shots_per_thread(2)  # raises if Momentum BP's shape does not fit
    threads, groups = t.launch()
    assert threads % 32 == 0 and threads * groups <= 1024


def test_largest_torus_has_none_with_state():
    t = bpq.Tanner("toric", 32)
    assert t.shots_per_thread("momentum") == 1
    with pytest.raises(bpq.BPQError):
        t.set_shots_per_thread(2)
