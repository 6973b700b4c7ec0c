"""The refinement loop's prediction that its next residual ends it, where it does not: the
fixed-point residual has added the correction and misses the tolerance, and the FP64 residual
follows from the pressure as it is.  Inner solves are asked for far more than FP32 gives, so their
own residual promises what the true one does not hold."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_common import hc, rel_l2  # noqa: F401

pytestmark = pytest.mark.gpu
RTOLS = [1e-11, 1e-12, 1e-13, 3e-14]


def solver(hc, n, rtol, use_graph, sync_cert=True, **kw):
    L = (1.0,) * len(n)
    shape = tuple(reversed(n))
    s = hc.Solver(n, L, c=10.0, D=0.05, gamma=0.75, dt=1e-3, precision="fp32_refined", cg_rtol=rtol,
                  inner_rtol=1e-9, max_sweeps=12, use_graph=use_graph, sync_cert=sync_cert,
                  device="cuda:0", **kw)
    s.set_r(W.smooth_r(n, 3, L) if len(n) == 2 else np.full(shape, 0.1))
    s.set_source(W.minus_mean(W.gaussian(n, (0.3,) * len(n), 0.1, L) -
                              W.gaussian(n, (0.7,) * len(n), 0.1, L)))
    s.set_state(W.uniform_m(shape, len(n), 0.0, 0.5, 3), np.zeros(shape))
    return s


@pytest.mark.parametrize("n", [(128, 64), (2048, 16), (32, 32, 16)])
def test_missed_prediction(hc, n):
    """One step at each tolerance, graph and host loop alike bit for bit, against the loop with
    FP64 residuals alone: a correction added twice would cost further sweeps and move p.  The
    graph's kernel count tells the residuals that missed (three or five kernels each)."""
    per_iter, per_res = (4, 3) if len(n) == 2 else (6, 5)
    extras = []
    for rtol in RTOLS:
        with solver(hc, n, rtol, True, fp64_mid_residual=True) as s:
            ref = s.step(1)
            p_ref = s.get_state()[1]
        out = []
        for use_graph in (True, False):
            with solver(hc, n, rtol, use_graph) as s:
                before = s.launch_count()
                st = s.step(1)
                if use_graph:
                    extras.append(s.launch_count() - before - per_iter * st.cg_iters
                                  - per_res * (st.refine_residuals + st.mid_residual_df))
                out.append((st, [np.array(a) for a in s.get_state()]))
        (g, gs), (h, hs) = out
        assert all(np.array_equal(a, b) for a, b in zip(gs, hs))
        assert (g.cg_iters, g.refine_sweeps, g.refine_residuals, g.status) == \
               (h.cg_iters, h.refine_sweeps, h.refine_residuals, h.status)
        # a tolerance below what FP64 residuals reach is reported by both loops
        assert g.status == ref.status, (rtol, g, ref)
        if g.status == 0:
            assert g.rel_residual <= rtol
            # p to the tolerances of both, through the operator's inverse, and FP64's own rounding
            assert rel_l2(gs[1], p_ref) <= 1e3 * rtol + 1e-12
            assert g.refine_sweeps <= ref.refine_sweeps + 1
    assert all((e - min(extras)) % per_res == 0 for e in extras)
    assert max(extras) > min(extras), (n, extras)


def test_missed_prediction_in_a_class(hc):
    """Members of a batch's size class take the same turns as their solo runs."""
    n = (128, 64)
    solo = []
    for rtol in RTOLS:
        with solver(hc, n, rtol, True) as s:
            st = s.step(1)
            solo.append((st.cg_iters, st.refine_sweeps, st.refine_residuals,
                         [np.array(a) for a in s.get_state()]))
    members = [solver(hc, n, rtol, True) for rtol in RTOLS]
    with hc.Batch(members) as b:
        assert b.classes() == (1, len(RTOLS))
        stats = b.step(1)
    for s, st, w in zip(members, stats, solo):
        assert (st.cg_iters, st.refine_sweeps, st.refine_residuals) == w[:3]
        assert all(np.array_equal(x, y) for x, y in zip(s.get_state(), w[3]))
        s.close()
