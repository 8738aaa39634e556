"""Calls from several host threads at once, each on its own stream and buffers:
sizes whose kernels take different amounts of dynamic shared memory."""
import threading

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def run_threads(jobs, times):
    errors = []

    def loop(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(times):
                    job()
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(repr(e))

    threads = [threading.Thread(target=loop, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_grid_values_of_different_sizes():
    import paper_2212_11744_gb300 as lqt
    jobs, checks = [], []
    for G, T in ((31, 30001), (300, 3000), (40, 16000), (300, 3000)):  # 18 to 58 KB, the same kernel
        g = W.falling_body(G=G, T=T)
        Vb = lqt.lqt_grid_block(g)
        want = lqt.lqt_grid_values(g, Vb)
        out = torch.empty_like(want)
        ws = torch.empty(lqt.lqt_grid_workspace_size(g, 1), dtype=torch.uint8, device="cuda")
        jobs.append(lambda g=g, Vb=Vb, out=out, ws=ws: lqt.lqt_grid_values(g, Vb, out=out, ws=ws))
        checks.append((out, want))
    torch.cuda.synchronize()
    run_threads(jobs, 100)
    torch.cuda.synchronize()
    for out, want in checks:
        assert torch.equal(out, want)


def test_gradients_of_different_sizes():
    from tests.test_gpu_adjoint import gpu_grads, weights
    from tests.test_gpu_uniform import make
    ps = [make(8, 4, 1056, 8, "equal", "const"), make(4, 1, 8192, 1, "equal", "const")]
    ws = [weights(p, 5) for p in ps]
    want = [gpu_grads(p, *w) for p, w in zip(ps, ws)]
    got = [None, None]

    def job(i):
        got[i] = gpu_grads(ps[i], *ws[i])

    run_threads([lambda i=i: job(i) for i in range(2)], 50)
    for a, b in zip(got, want):
        for k in b:
            np.testing.assert_array_equal(a[k], b[k])
