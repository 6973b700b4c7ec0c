"""Loop kernels of several callers on one device: calls that step inside another call, and
solvers on threads of their own.  Every wait of a test ends: what should have returned is
joined with a limit."""
import threading

import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_common import hc  # noqa: F401

pytestmark = pytest.mark.gpu
LIMIT = 120.0  # seconds that a joined thread may take; each runs for well below one


def make(hc, n, precision, seed, **kw):
    import torch
    L = (1.0, 1.0)
    g = O.Grid(n, L)
    opt = dict(c=10.0, D=0.05, gamma=0.75, dt=1e-3, cg_rtol=1e-8, cg_maxit=500)
    opt.update(kw)
    s = hc.Solver(n, L, precision=precision, device="cuda:0", stream=torch.cuda.Stream("cuda:0"),
                  **opt)
    s.set_r(W.smooth_r(n, seed, L))
    s.set_source(W.minus_mean(W.gaussian(n, (0.3, 0.4), 0.1, L) - W.gaussian(n, (0.7, 0.6), 0.1, L)))
    return s, W.uniform_m(g.shape, 2, 0.0, 0.5, seed), np.zeros(g.shape)


def in_threads(calls):
    """The calls' results, each from a thread of its own; fails if one does not return."""
    out, err = [None] * len(calls), []

    def go(k):
        try:
            out[k] = calls[k]()
        except Exception as e:  # reported below, in the main thread
            err.append(e)

    threads = [threading.Thread(target=go, args=(k,), daemon=True) for k in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(LIMIT)
    assert not any(t.is_alive() for t in threads), "a call did not return"
    assert not err, err
    return out


def gradients(s, m0, p0, steps=3, every=2):
    s.set_state(m0, p0)
    g = s.adjoint(steps, 2.0 * m0, every)
    return [np.asarray(g[k]).copy() for k in ("dc2", "dD2", "dr", "dS", "dm0")]


def stepped(s, m0, p0, steps=4):
    s.set_state(m0, p0)
    st = s.step(steps)
    assert st.status == 0
    return [np.array(a) for a in s.get_state()]


def same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
def test_adjoint_returns_and_leaves_the_device_free(hc, precision):
    """The adjoint steps forward inside its own call, on a grid whose solves are loop kernels:
    it returns, repeats itself, and neither disturbs nor waits for ever on a solver that steps
    beside it."""
    a, ma, pa = make(hc, (64, 64), precision, 1)
    b, mb, pb = make(hc, (64, 64), precision, 2)
    alone = in_threads([lambda: gradients(a, ma, pa)])[0]
    step_alone = stepped(b, mb, pb)
    for _ in range(3):
        both = in_threads([lambda: gradients(a, ma, pa), lambda: stepped(b, mb, pb)])
        assert same(both[0], alone) and same(both[1], step_alone)
    a.close()
    b.close()
