"""The bounded waits of the CG loop kernels: a launch whose barrier wait runs out leaves the solve
as it was for every one of its CTAs, is repeated while the caller's patience lasts, and is then
reported, after which the context goes on as any other.  The limits are made so short that waits
run out; nothing waits longer than them."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_common import hc  # noqa: F401

pytestmark = pytest.mark.gpu
STEPS = 3


def make(hc, n, precision, use_graph):
    L = (1.0, 1.0)
    g = O.Grid(n, L)
    s = hc.Solver(n, L, c=10.0, D=0.05, gamma=0.75, dt=1e-3, precision=precision, cg_rtol=1e-8,
                  use_graph=use_graph, device="cuda:0")
    s.set_r(W.smooth_r(n, 3, L))
    s.set_source(W.minus_mean(W.gaussian(n, (0.3, 0.4), 0.1, L) - W.gaussian(n, (0.7, 0.6), 0.1, L)))
    return s, W.uniform_m(g.shape, 2, 0.0, 0.5, 3), np.zeros(g.shape)


def stepped(s, m0, p0):
    s.set_state(m0, p0)
    s.step(STEPS)
    return [np.array(a) for a in s.get_state()]


@pytest.mark.parametrize("use_graph", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
def test_wait_that_runs_out_is_reported(hc, precision, use_graph):
    """No polls at all: no barrier completes."""
    s, m0, p0 = make(hc, (64, 64), precision, use_graph)
    want = stepped(s, m0, p0)
    for patience in (0.0, 0.02):
        s.set_loop_wait(0, patience)
        for _ in range(2):
            s.set_state(m0, p0)
            with pytest.raises(hc.HuCaiError) as e:
                s.step(STEPS)
            assert e.value.code == hc.HC_ETIMEOUT
        with pytest.raises(hc.HuCaiError) as e:
            s.run(STEPS)
        assert e.value.code == hc.HC_ETIMEOUT
        with pytest.raises(hc.HuCaiError) as e:
            s.adjoint(STEPS, m0, 2)
        assert e.value.code == hc.HC_ETIMEOUT
        s.set_loop_wait()
        got = stepped(s, m0, p0)
        assert all(np.array_equal(a, b) for a, b in zip(got, want))
    s.close()


@pytest.mark.parametrize("use_graph", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
@pytest.mark.parametrize("n", [(64, 64), (256, 256)])
def test_no_answer_from_a_launch_given_up(hc, n, precision, use_graph):
    """Waits that sometimes run out, at any barrier and in any CTA: every call either reports it
    or returns what it returns undisturbed, bit for bit."""
    s, m0, p0 = make(hc, n, precision, use_graph)
    want = stepped(s, m0, p0)
    ends = set()
    for polls in [0, 1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 64, 1 << 20]:
        s.set_loop_wait(polls, 0.002)
        for _ in range(8):
            try:
                got = stepped(s, m0, p0)
            except hc.HuCaiError as e:
                assert e.code == hc.HC_ETIMEOUT
                ends.add("reported")
                continue
            ends.add("answered")
            assert all(np.array_equal(a, b) for a, b in zip(got, want)), polls
    assert ends == {"reported", "answered"}
    s.close()


def test_batch_reports_it(hc):
    a, ma, pa = make(hc, (64, 64), "fp64", True)
    b, mb, pb = make(hc, (128, 64), "fp64", True)
    want = [stepped(a, ma, pa), stepped(b, mb, pb)]
    with hc.Batch([a, b]) as batch:
        a.set_loop_wait(0, 0.01)
        a.set_state(ma, pa)
        b.set_state(mb, pb)
        with pytest.raises(hc.HuCaiError) as e:
            batch.step(STEPS)
        assert e.value.code == hc.HC_ETIMEOUT
        a.set_loop_wait()
        a.set_state(ma, pa)
        b.set_state(mb, pb)
        batch.step(STEPS)
    for s, w in zip((a, b), want):
        assert all(np.array_equal(x, y) for x, y in zip(s.get_state(), w))
        s.close()


def test_limits_are_checked(hc):
    s, _, _ = make(hc, (64, 64), "fp64", True)
    for bad in (-1.0, float("nan"), float("inf")):
        with pytest.raises(hc.HuCaiError) as e:
            s.set_loop_wait(1, bad)
        assert e.value.code == hc.HC_EINVAL
    s.close()
