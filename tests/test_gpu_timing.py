"""hc_time_kernel: it times the kernels that a step runs (the fused divergence pass of plain FP64,
the fixed-point residual, the loop kernel) and leaves the problem as it was."""
import numpy as np
import pytest

import workloads as W
from gpu_common import hc  # noqa: F401

pytestmark = pytest.mark.gpu

COMMON = ["cg_grad", "cg_apply", "cg_div", "cg_update", "res_grad", "res_apply", "res_div",
          "split_grad", "split_row", "split_heat", "split_c2r"]
REFINED = COMMON + ["first_grad", "first_apply", "first_div", "mid_grad", "mid_apply", "mid_div"]


@pytest.mark.parametrize("n, precision, names, loop", [
    ((64, 64), "fp64", COMMON, True), ((512, 1024), "fp64", COMMON, False),
    ((128, 64), "fp32_refined", REFINED, True), ((2048, 16), "fp32_refined", REFINED, False),
    ((32, 16, 16), "fp32_refined", REFINED + ["cg_ypass", "res_ypass", "mid_ypass"], False),
    ((16, 16, 32), "fp64", COMMON + ["cg_ypass", "res_ypass"], False)])
def test_every_kernel_is_timed_and_nothing_moves(hc, n, precision, names, loop):
    L = (1.0,) * len(n)
    shape = tuple(reversed(n))
    with hc.Solver(n, L, c=10.0, D=0.05, gamma=0.75, dt=1e-3, precision=precision, cg_rtol=1e-8,
                   device="cuda:0") as s:
        s.set_source(W.minus_mean(W.gaussian(n, (0.4,) * len(n), 0.1, L)))
        s.set_m(W.uniform_m(shape, len(n), 0.0, 0.5, 1))
        s.step(2)
        before = [np.array(a) for a in s.get_state()]
        for name in names + (["cg_loop"] if loop else []):
            ms = s.time_kernel(name, 25)
            if name == "cg_update" and precision == "fp64" and len(n) == 2:
                assert ms == 0.0  # part of cg_div
            else:
                assert 0.0 < ms < 50.0, (name, ms)
        if not loop:
            with pytest.raises(hc.HuCaiError) as e:
                s.time_kernel("cg_loop", 5)
            assert e.value.code == hc.HC_ENOTSUP
        after = s.get_state()
        assert all(np.array_equal(a, b) for a, b in zip(before, after))
        assert s.step(1).status == 0
