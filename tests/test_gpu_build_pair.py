"""The element build by two warps per 32 sub-intervals (n = 2..4, T <= 2^17)
against the oracle (1e-11 per element, the bound of the general build's tests)
at ragged T, with coefficients per interval and per stage, and against the
build by one thread per sub-interval bit for bit."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests.test_gpu_parity import relerr as rel, to_np
from tests.test_gpu_uniform import make

pytestmark = pytest.mark.gpu
FIELDS = ("A", "b", "C", "eta", "J", "zeta")


def build(p):
    import paper_2212_11744_gb300 as lqt
    el = lqt.lqt_build_elements(lqt.DeviceProblem(p))
    torch.cuda.synchronize()
    assert lqt.lqt_get_status() == 0
    return el


@pytest.mark.parametrize("n,m", [(2, 1), (2, 2), (3, 1), (3, 3), (4, 2), (4, 3)])
@pytest.mark.parametrize("T,K", [(1, 3), (31, 2), (33, 1), (1025, 2)])
@pytest.mark.parametrize("mode", ["const", "interval", "stages"])
def test_elements_match_oracle(n, m, T, K, mode):
    p = make(n, m, T, K, "uneven", "interval")
    rng = np.random.default_rng(n + T)
    p.c = W.const(rng.standard_normal(n))
    if mode != "const":
        cnt = T if mode == "interval" else 2 * K * T + 1
        vary = lambda a: W.Coef(np.asarray(a)[None] * rng.uniform(0.7, 1.3, (cnt,) + (1,) * np.ndim(a)),
                                W.PER_INTERVAL if mode == "interval" else W.PER_STAGE)
        p.F, p.L, p.c = vary(p.F.values.reshape(n, n)), vary(p.L.values.reshape(n, m)), vary(p.c.values.reshape(n))
    el = build(p)
    ref = oracle.build_elements(p, 0, T + 1)
    for k in FIELDS:
        assert rel(to_np(el[k]), ref[k]) <= 1e-11, k


@pytest.mark.parametrize("n", [2, 3, 4])
def test_same_bits_as_one_thread_per_subinterval(n):
    T = (1 << 17) + 1
    p = make(n, 2, T, 2, "uneven", "const")
    one = build(p)
    p.T, p.t = T - 1, p.t[:-1]
    two = build(p)
    for k in FIELDS:
        assert torch.equal(one[k][:T - 1], two[k][:T - 1]), k
