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


# (size, precision, how many): loops that fit an SM together in twos, fours and eights, loops that
# take the device for themselves, and more of each than fit at a time.
CROWDS = [
    [((64, 64), "fp64")] * 16,
    [((256, 256), "fp64")] * 6,
    [((256, 256), "fp32_refined")] * 8,
    [((512, 512), "fp32_refined"), ((512, 512), "fp64"), ((64, 64), "fp64"), ((128, 64), "fp64"),
     ((32, 8), "fp64"), ((256, 128), "fp32_refined"), ((512, 512), "fp32_refined_df"),
     ((1024, 512), "fp32_refined")],
]


@pytest.mark.parametrize("crowd", range(len(CROWDS)))
def test_crowd_on_threads(hc, crowd):
    """Solvers stepped at once, each from its thread on its stream: as each is alone, bit for bit,
    whether its loops find room at once or have to wait for it."""
    members = [make(hc, n, precision, k) for k, (n, precision) in enumerate(CROWDS[crowd])]
    alone = [stepped(*x) for x in members]
    for _ in range(3):
        out = in_threads([lambda x=x: stepped(*x) for x in members])
        assert all(same(a, b) for a, b in zip(out, alone))
    for s, _, _ in members:
        s.close()


# Loops that share the device, and refined ones that would take it in turns: those run the separate
# kernels in a batch, with the same results.
@pytest.mark.parametrize("n, precision, count", [((64, 64), "fp64", 16), ((256, 256), "fp64", 6),
                                                 ((512, 512), "fp32_refined_df", 3),
                                                 ((1024, 512), "fp32_refined_df", 3)])
def test_crowd_in_a_batch(hc, n, precision, count):
    """Contexts outside a size class, each on a chain of its own."""
    members = [make(hc, n, precision, k) for k in range(count)]
    alone = [stepped(*x) for x in members]
    with hc.Batch([s for s, _, _ in members]) as b:
        assert b.classes() == (0, 0)
        for _ in range(3):
            for s, m0, p0 in members:
                s.set_state(m0, p0)
            assert all(st.status == 0 for st in b.step(4))
            assert all(same(s.get_state(), w) for (s, _, _), w in zip(members, alone))
    for s, _, _ in members:
        s.close()


def test_large_loop_is_not_starved(hc):
    """A solver whose loops need every SM, beside eight small ones that never rest: it returns
    while they still step."""
    big, mb, pb = make(hc, (512, 512), "fp64", 0)
    small = [make(hc, (64, 64), "fp64", k) for k in range(1, 9)]
    want = stepped(big, mb, pb)
    for x in small:
        stepped(*x)
    stop = threading.Event()
    ran = [0] * len(small)

    def keep(k):
        while not stop.is_set():
            small[k][0].step(1)
            ran[k] += 1

    threads = [threading.Thread(target=keep, args=(k,), daemon=True) for k in range(len(small))]
    for t in threads:
        t.start()
    try:
        got = in_threads([lambda: stepped(big, mb, pb)])[0]
    finally:
        stop.set()
        for t in threads:
            t.join(LIMIT)
    assert not any(t.is_alive() for t in threads)
    assert same(got, want) and min(ran) > 0
    big.close()
    for s, _, _ in small:
        s.close()
