"""Workspaces hold what their call uses: the kept products of the mixed-precision
solve's build (n = 64, in proportion to K) are in no other call's workspace, and the
solves' own share them with the scan.  Host functions only."""
import dataclasses

import pytest

import workloads as W

KINDS = ("LQT_WS_BUILD", "LQT_WS_VALUE", "LQT_WS_TRAJ", "LQT_WS_SOLVE_METHOD2")


def sizes(T, K):
    import paper_2212_11744_gb300 as m
    hp = m.HostProblem(dataclasses.replace(W.large_state_n64(T=T), K=K), pinned=False)
    return {k: m.lqt_workspace_size(hp, getattr(m, k)) for k in KINDS + ("LQT_WS_SOLVE",)}


@pytest.mark.parametrize("T", [128, 1000, 4096, 4097])
def test_independent_of_the_steps(T):
    """The problem is constant and its grid equal, so only the mixed build depends on K."""
    one, eight = sizes(T, 1), sizes(T, 8)
    for k in KINDS:
        assert one[k] == eight[k], k
    assert eight["LQT_WS_SOLVE"] >= one["LQT_WS_SOLVE"]


def test_solve_workspace_holds_the_mixed_build():
    """Kept products: 4 K stages of 2 n M doubles for up to 152 lengths."""
    base = sizes(128, 1)["LQT_WS_BUILD"]
    assert sizes(128, 8)["LQT_WS_SOLVE"] - base >= 128 * 4 * 8 * 2 * 64 * 16 * 8
