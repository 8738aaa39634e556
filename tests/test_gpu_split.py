"""FP64 combinations on split products (csrc/lqt_split.cuh, n = 16): against the
oracle's fold on elements in units that differ by up to 2^8,
whose I + C J needs row exchanges or is ill conditioned, and on horizons around
the chunk and level edges.  Bounds: 1e-9 per boundary (the parity bound); an
ill-conditioned system (condition number kappa) is held to 64 eps kappa."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests.test_gpu_parity import TOL, relerr as rel, to_np

pytestmark = pytest.mark.gpu


def lqt():
    import paper_2212_11744_gb300 as m
    return m


def check(p, n, el_np, tol, keys=("S", "v", "zeta")):
    m = lqt()
    dp = m.DeviceProblem(p)
    el = {k: torch.tensor(np.ascontiguousarray(v), device="cuda") for k, v in el_np.items()}
    out = m.lqt_scan_value(dp, el)
    torch.cuda.synchronize()
    ref_of = dict(zip(keys, oracle.suffix_values(n, el_np)))
    for k in keys:
        ref = ref_of[k]
        assert rel(to_np(out[k]), ref) <= tol, k


def elements(n, T, seed, cond=1.0, graded=False, swap=False):
    rng = np.random.default_rng(seed)
    G = rng.standard_normal((2, T + 1, n, n))
    A = rng.standard_normal((T + 1, n, n)) / (2 * np.sqrt(n))
    C, J = (g @ g.transpose(0, 2, 1) / n * cond for g in G)
    b, eta, z = rng.standard_normal((T + 1, n)), rng.standard_normal((T + 1, n)), rng.standard_normal(T + 1)
    if graded:  # states of very different units: x = D x'
        D = 2.0 ** rng.integers(-4, 5, n)
        A, C, J = A * D[:, None] / D[None, :], C * np.outer(D, D), J / np.outer(D, D)
        b, eta = b * D, eta / D
    if swap:  # small diagonal next to large off-diagonal entries
        C = C + 50.0 * np.roll(np.eye(n), 1, 1) + 50.0 * np.roll(np.eye(n), -1, 1) + 100.0 * np.eye(n)
    A[T], b[T], C[T] = 0.0, 0.0, 0.0
    return {"A": A, "b": b, "C": C, "eta": eta, "J": J, "zeta": z}


@pytest.mark.parametrize("n", [16, 64])
@pytest.mark.parametrize("kind", ["plain", "graded", "swap", "cond"])
@pytest.mark.parametrize("T", [1, 2, 3, 37, 130])
def test_scan_of_random_elements(n, kind, T):
    p = W.batched_member(7, T=T, n=16) if n == 16 else W.large_state_n64(T=T)
    el = elements(n, T, 100 * T + n, cond=1e3 if kind == "cond" else 1.0, graded=kind == "graded", swap=kind == "swap")
    if kind == "cond":
        W1 = np.eye(n) + el["C"][:-1] @ el["J"][1:]
        kappa = np.linalg.cond(W1).max()
        check(p, n, el, max(TOL, 64 * 2.2e-16 * kappa))
    else:
        check(p, n, el, TOL)


@pytest.mark.parametrize("T", [1367, 1368, 2735, 2736, 4104])
def test_n16_solve_around_the_chunk_edges(T):
    p = W.batched_member(9, T=T, n=16)
    out = lqt().lqt_solve(lqt().DeviceProblem(p))
    ref = oracle.solve(p)
    for k in ("S", "v", "zeta", "x", "u"):
        assert rel(to_np(out[k]), ref[k]) <= TOL, k


def test_non_finite_elements_are_reported():
    n, T = 16, 5
    p = W.batched_member(7, T=T, n=n)
    el = elements(n, T, 3)
    el["J"][2, 3, 4] = el["J"][2, 4, 3] = np.nan
    m = lqt()
    out = m.lqt_scan_value(m.DeviceProblem(p), {k: torch.tensor(v, device="cuda") for k, v in el.items()})
    torch.cuda.synchronize()
    assert m.lqt_get_status() == 3
    assert not np.isfinite(to_np(out["S"][0])).all()
    assert np.isfinite(to_np(out["S"][3:])).all()
