"""The CG loop as one cooperative kernel (2D solves up to about 10^6 points): the sizes at the
ends of its range and of its tiles against the oracle, and several of its launches at once."""
import threading

import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2606_06720_gb300 as m
    return m


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def setup(n, seed):
    L = (1.0, 1.0)
    g = O.Grid(n, L)
    S = W.minus_mean(W.gaussian(n, (0.3, 0.4), 0.1, L) - W.gaussian(n, (0.7, 0.6), 0.1, L))
    r = W.smooth_r(n, seed, L)
    m0 = W.uniform_m(g.shape, 2, 0.0, 0.5, seed)
    return g, L, S, r, m0


# One CTA; one column or one row group a CTA; 32 columns a CTA; long rows (a row on a thread in
# the separate kernels); transforms below and at the fixed-point lengths; the largest grids that
# take the loop and the smallest that do not (FP32: 512 threads, 2^20 points; FP64: 256, 2^18).
SIZES = [(32, 8), (32, 16), (64, 64), (16, 512), (512, 16), (64, 32), (2048, 32), (256, 128),
         (512, 512), (1024, 512)]


@pytest.mark.parametrize("use_graph", [False, True])
@pytest.mark.parametrize("precond", ["scalar", "kbar"])
@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
@pytest.mark.parametrize("n", SIZES)
def test_step_against_oracle(hc, n, precision, precond, use_graph):
    """One step from m0.  The pressure solves meet 1e-10, so FP64 agrees to the solve (1e-8 in
    p through the operator's inverse); the refined mode keeps m in FP32 (1e-5)."""
    g, L, S, r, m0 = setup(n, 3)
    prm = O.Params(c=10.0, D=0.05, gamma=0.75, dt=1e-3, cg_rtol=1e-10, cg_maxit=500)
    m_ref, p_ref, _ = O.step(g, prm, r, S, m0, np.zeros(g.shape))
    with hc.Solver(n, L, c=prm.c, D=prm.D, gamma=prm.gamma, dt=prm.dt, precision=precision,
                   cg_rtol=1e-10, precond=precond, use_graph=use_graph, device="cuda:0") as s:
        s.set_r(r)
        s.set_source(S)
        s.set_state(m0, np.zeros(g.shape))
        st = s.step(1)
        m, p = s.get_state()
    assert st.status == 0 and st.rel_residual <= 1e-10
    assert rel(m, m_ref) < (1e-8 if precision == "fp64" else 1e-5)
    assert rel(p, p_ref) < (1e-7 if precision == "fp64" else 1e-4)


def test_iteration_cap(hc):
    """A solve that may take three iterations takes three and says so."""
    n = (64, 64)
    g, L, S, r, m0 = setup(n, 1)
    with hc.Solver(n, L, c=10.0, D=0.05, gamma=0.75, dt=1e-3, precision="fp64", cg_rtol=1e-12,
                   cg_maxit=3, device="cuda:0") as s:
        s.set_r(r)
        s.set_source(S)
        s.set_m(m0)
        st = s.step(1)
    assert st.cg_iters == 3 and st.status == -4


@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
def test_loops_side_by_side(hc, precision):
    """Six solvers of 512^2, each loop launch on most of the SMs, stepped from six threads on
    six streams: every one as it is alone, bit for bit."""
    import torch
    n = (512, 512)
    solvers, init, alone = [], [], []
    for k in range(6):
        g, L, S, r, m0 = setup(n, k)
        s = hc.Solver(n, L, c=25.0, D=0.02, gamma=0.5, dt=5e-4, precision=precision, cg_rtol=1e-8,
                      device="cuda:0", stream=torch.cuda.Stream("cuda:0"))
        s.set_r(r)
        s.set_source(S)
        solvers.append(s)
        init.append((m0, np.zeros(g.shape)))
        s.set_state(*init[k])
        s.step(4)
        alone.append([np.array(a) for a in s.get_state()])
    for _ in range(3):
        for s, i in zip(solvers, init):
            s.set_state(*i)
        out, err = [None] * 6, []

        def go(k):
            try:
                solvers[k].step(4)
                out[k] = [np.array(a) for a in solvers[k].get_state()]
            except Exception as e:  # reported below, in the main thread
                err.append(e)

        threads = [threading.Thread(target=go, args=(k,)) for k in range(6)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not err, err
        for a, b in zip(out, alone):
            assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    for s in solvers:
        s.close()
