"""Solvers stepped at once from threads of their own, each on its stream, with calls that take
turns between the graphs of a context (one step, several steps, run): the handles, tables and
counters that a graph's kernels read have to be in place before it starts."""
import threading

import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_common import hc  # noqa: F401

pytestmark = pytest.mark.gpu
LIMIT = 60.0  # seconds; each thread runs for well below one


def make(hc, n, seed, **kw):
    import torch
    L = (1.0, 1.0)
    g = O.Grid(n, L)
    s = hc.Solver(n, L, c=10.0, D=0.05, gamma=0.75, dt=1e-3, cg_rtol=1e-8, cg_maxit=500,
                  device="cuda:0", stream=torch.cuda.Stream("cuda:0"), **kw)
    s.set_r(W.smooth_r(n, seed, L))
    s.set_source(W.minus_mean(W.gaussian(n, (0.3, 0.4), 0.1, L) - W.gaussian(n, (0.7, 0.6), 0.1, L)))
    return s, W.uniform_m(g.shape, 2, 0.0, 0.5, seed), np.zeros(g.shape)


def drive(s, m0, p0):
    s.set_state(m0, p0)
    its = [s.step(3).total_cg_iters, s.step(1).cg_iters, s.step(2).total_cg_iters]
    s.run(2, eps=0.0, stop_on_energy=False)
    its.append(s.step(3).total_cg_iters)
    return [np.array(a) for a in s.get_state()] + [np.array(its)]


# (2048, 16) and (8, 8): no loop kernel; the others take one.
@pytest.mark.parametrize("precision", ["fp32_refined", "fp32_refined_df", "fp64"])
@pytest.mark.parametrize("n", [(2048, 16), (8, 8), (128, 128)])
def test_alternating_graphs_on_threads(hc, n, precision):
    """Every solver ends, and as it does alone, bit for bit, iteration counts included."""
    members = [make(hc, n, k, precision=precision) for k in range(8)]
    alone = [drive(*x) for x in members]
    for _ in range(6):
        out, err = [None] * len(members), []

        def go(k):
            try:
                out[k] = drive(*members[k])
            except Exception as e:  # reported below, in the main thread
                err.append(e)

        threads = [threading.Thread(target=go, args=(k,), daemon=True) for k in range(len(members))]
        for t in threads:
            t.start()
        for t in threads:
            t.join(LIMIT)
        assert not any(t.is_alive() for t in threads), "a call did not return"
        assert not err, err
        for a, b in zip(out, alone):
            assert all(np.array_equal(x, y) for x, y in zip(a, b))
    for s, _, _ in members:
        s.close()
