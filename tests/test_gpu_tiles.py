"""The sampler and the classifier work on tiles of 32 shots: odd sizes around
the tile, buffers off a 4-byte boundary, qubit counts that are and are not
multiples of 4 (of 128: padded rows), Y checks, the largest graph, and codes
above 3 (which count as I).  Whole numbers: equal to the oracle's exactly."""
import numpy as np
import pytest
import torch

import oracle
from inputs import pack_bits, random_tree_code

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bpq():
    import paper_2407_11523_gb300 as bpq
    return bpq


def at_offset(shape, off, fill=0):
    """uint8 CUDA tensor whose data starts off bytes past an aligned address."""
    n = int(np.prod(shape))
    return torch.full((n + 16,), fill, dtype=torch.uint8, device="cuda")[off:off + n].view(shape)


def graph(bpq, kind, d):
    if kind == "tree":  # Y entries, ragged checks
        H = random_tree_code(30, d)
        return bpq.Tanner(H=H), H
    t = bpq.Tanner(kind, d)
    return t, t.dense()


@pytest.mark.parametrize("kind,d", [("planar", 2), ("planar", 7), ("toric", 8), ("xzzx", 5), ("planar", 32),
                                    ("tree", 9)])
@pytest.mark.parametrize("B,off", [(1, 0), (31, 1), (33, 2), (64, 0), (97, 3)])
def test_sample_tiles(bpq, kind, d, B, off):
    t, H = graph(bpq, kind, d)
    ch = (0.05, 0.11, 0.02)
    err = at_offset((B, t.N), off, 77)
    bpq.sample(t, *ch, seed=2**63 + 5, shot0=2**33 - 7, B=B, err=err)
    _, syn = bpq.sample(t, *ch, seed=2**63 + 5, shot0=2**33 - 7, B=B)
    e_ref, s_ref = oracle.sample(H, *ch, seed=2**63 + 5, shot0=2**33 - 7, B=B)
    assert (err.cpu().numpy() == e_ref).all()
    assert (syn.cpu().numpy().view(np.uint32) == pack_bits(s_ref)).all()


def parities(R, H):
    """<R_b, H_i> of every row pair (symplectic product, by matrix products)."""
    x, z = lambda c: ((c == 1) | (c == 2)).astype(np.float32), lambda c: (c >= 2).astype(np.float32)
    return (x(R) @ z(H).T + z(R) @ x(H).T).astype(np.int64) & 1


@pytest.mark.parametrize("kind,d", [("planar", 2), ("planar", 7), ("toric", 8), ("toric", 3), ("xzzx", 5),
                                    ("planar", 32)])
@pytest.mark.parametrize("B,off", [(1, 0), (31, 1), (33, 2), (97, 0)])
def test_check_logical_tiles(bpq, kind, d, B, off):
    t, H = graph(bpq, kind, d)
    L = t.logicals()
    rng = np.random.default_rng(17 * d + B)
    err = rng.integers(0, 4, (B, t.N)).astype(np.uint8)
    est = err.copy()
    xz = np.array([0, 1, 3, 2])  # code <-> (x, z) bits packed so that products are XORs

    def times(code, op):
        return np.array([0, 1, 3, 2])[xz[code] ^ xz[op]]

    for b in range(B):  # a stabilizer (0), a logical operator (2) or a single-qubit error (1) times the error
        op = [H[rng.integers(t.M)], L[rng.integers(len(L))]][b % 2] if b % 3 else np.eye(t.N, dtype=int)[b % t.N]
        est[b] = times(err[b], op)
    bad = err.copy()
    bad[::5, 0] = 4 + (bad[::5, 0] | 3)  # no Pauli code: counts as I
    for e in (err, bad):
        good = np.where(e > 3, 0, e)
        r = times(good, est)
        want = np.where(parities(r, H).any(1), 1, np.where(parities(r, L).any(1), 2, 0))
        de, dh, out = at_offset((B, t.N), off), at_offset((B, t.N), (off * 3) % 4), at_offset((B,), off)
        de.copy_(torch.from_numpy(e))
        dh.copy_(torch.from_numpy(est))
        got = bpq.check_logical(t, de, dh, out=out).cpu().numpy()
        assert (got == want).all()
