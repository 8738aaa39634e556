"""A batch of very different lengths: the constant-coefficient build's grid
follows the boundaries of all problems together, not the longest one times their
number.  Against the oracle, and the long problem against itself in a batch of
its own."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests.test_gpu_parity import TOL, relerr as rel, to_np

pytestmark = pytest.mark.gpu


def member(n, T, seed=3):
    if n > 1:
        return W.batched_member(seed, T=T, n=n)
    p = W.batched_member(seed, T=T, n=2)
    return dataclasses.replace(p, n=1, nr=1, F=W.const(p.F.values[0][:1, :1]), L=W.const(np.array([[0.7]])),
                               X=W.const(np.array([[1.3]])), r=W.Coef(p.r.values[:, :1].copy(), p.r.mode),
                               Xf=np.array([[1.3]]), rf=p.rf[:1], x0=p.x0[:1])


@pytest.mark.parametrize("n", [1, 2, 8, 16])
def test_lengths_around_the_chunks(n):
    """Problems that start and end anywhere in a chunk, several in one chunk,
    one over many chunks, with and without a table."""
    from paper_2212_11744_gb300.batch import Batch
    Ts = [64, 1, 1, 130, 64, 63, 3000, 2, 16, 200, 65, 513]
    ps = [member(n, T, 3 + i) for i, T in enumerate(Ts)]
    b = Batch(ps)
    out = b.solve()
    torch.cuda.synchronize()
    for i, p in enumerate(ps):
        ref, got = oracle.solve(p), b.problem_slice(out, i)
        for k in ("S", "v", "zeta", "x", "u"):
            assert rel(to_np(got[k]), ref[k]) <= TOL, (i, k)


def test_longest_times_count_beyond_the_grid_limit():
    """2^16 problems, one of 2^21 + 64 sub-intervals: 2^31 chunks of the longest."""
    from paper_2212_11744_gb300.batch import Batch
    long, short = member(1, (1 << 21) + 64), member(1, 1)
    B = 1 << 16
    b = Batch([short] * (B - 1) + [long])
    out = b.solve()
    torch.cuda.synchronize()
    alone = Batch([long])
    want = alone.solve()
    ref = oracle.solve(short)
    for i in (0, B - 2):
        got = b.problem_slice(out, i)
        for k in ("S", "v", "zeta", "x", "u"):
            assert rel(to_np(got[k]), ref[k]) <= TOL, (i, k)
    got = b.problem_slice(out, B - 1)
    for k in ("S", "v", "x", "u"):
        assert rel(to_np(got[k]), to_np(want[k])) <= TOL, k
