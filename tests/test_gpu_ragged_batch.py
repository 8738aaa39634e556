"""A batch of very different lengths: the constant-coefficient build's grid
follows the boundaries of all problems together, not the longest one times their
number.  Against the oracle, and the long problem against itself in a batch of
its own."""
import dataclasses

import pytest
import torch

import oracle
import workloads as W
from tests.test_gpu_parity import TOL, relerr as rel, relerr_one, to_np

pytestmark = pytest.mark.gpu


def member(n, T, seed=3):
    """A member of the workloads' batch; n = 1 and 3: its first states, one input."""
    if n not in (1, 3):
        return W.batched_member(seed, T=T, n=n)
    p = W.batched_member(seed, T=T, n=n + 1)
    cut = lambda c: W.const(c.values[0][:n, :n])
    return dataclasses.replace(p, n=n, nr=n, m=1, F=cut(p.F), L=W.const(p.L.values[0][:n, :1]), X=cut(p.X),
                               U=W.const(p.U.values[0][:1, :1]), r=W.Coef(p.r.values[:, :n].copy(), p.r.mode),
                               Xf=p.Xf[:n, :n], rf=p.rf[:n], x0=p.x0[:n])


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
    # scalars that cross zero: against the whole trajectory's norm
    got = b.problem_slice(out, B - 1)
    for k in ("S", "v", "x", "u"):
        assert relerr_one(to_np(got[k]), to_np(want[k])) <= TOL, k


# n, T, problems: either side of the shortest problem that has a table, and of
# the fewest sub-intervals for which a batch makes tables
@pytest.mark.parametrize("n,T,B", [(1, 1023, 129), (1, 1024, 127), (1, 1024, 128), (2, 255, 129), (2, 256, 127),
                                   (2, 256, 128), (3, 63, 3), (3, 64, 3)])
def test_lines_of_the_table_rule(n, T, B):
    from paper_2212_11744_gb300.batch import Batch
    p = member(n, T)
    b = Batch([p] * B)
    out = b.solve()
    torch.cuda.synchronize()
    ref = oracle.solve(p)
    for i in (0, B // 2, B - 1):
        got = b.problem_slice(out, i)
        for k in ("S", "v", "zeta", "x", "u"):
            assert rel(to_np(got[k]), ref[k]) <= TOL, (i, k)
