"""The n = 16 composition of one-sub-interval maps on split products
(reduce_maps_w16_kernel) where it can go wrong: a single map, groups of one and
of ragged length, every chunk length of a batch with its jumps between problems
(maps of zero Psi).  Bound 1e-9 against the oracle, the parity tests'."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests.test_gpu_parity import TOL, relerr as rel, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 2, 3, 31, 33, 1025])
def test_trajectory_matches_oracle(T):
    import paper_2212_11744_gb300 as lqt
    p = W.batched_member(5, T=T, n=16)
    out = lqt.lqt_solve(lqt.DeviceProblem(p))
    torch.cuda.synchronize()
    assert lqt.lqt_get_status() == 0
    ref = oracle.solve(p)
    for k in ("x", "u"):
        assert rel(to_np(out[k]), ref[k]) <= TOL, k


@pytest.mark.parametrize("chunk", [0, 2, 8, 32])
def test_batch_chunks_match_oracle(chunk):
    from paper_2212_11744_gb300.batch import Batch
    ps = [W.batched_member(40 + i, T=T, n=16) for i, T in enumerate((1, 37, 64, 200, 5))]
    b = Batch(ps)
    out = b.solve(chunk=chunk)
    torch.cuda.synchronize()
    for i, p in enumerate(ps):
        ref = oracle.solve(p)
        got = b.problem_slice(out, i)
        for k in ("x", "u"):
            assert rel(to_np(got[k]), ref[k]) <= TOL, (i, k)
