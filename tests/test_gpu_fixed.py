"""The FP64 transforms' fixed-point passes: every length 64 .. 4096 along both
axes (each mix of radix-8, radix-4 and radix-2 passes, groups of less than a
warp up to 16 warps), inputs of very different magnitudes, the ends of FP64's
range, zeros and non-finite values.

Tolerance.  A pass rounds to one unit where the output's rms is at least 2^54
units: at most 2^-54 relative to the norm per pass, two axes of at most four
passes; the FP64 results of the two axes are rounded to at most 2^-53 each, and
so are the reference's.  The sum is below 8 * 2^-53.
"""
import numpy as np
import pytest

from gpu_common import hc, packed  # noqa: F401

sf = pytest.importorskip("scipy.fft")

pytestmark = pytest.mark.gpu
TOL = 8 * 2.0 ** -53


def _solver(hc, nx, ny):
    return hc.Solver((nx, ny), c=1.0, D=0.1, gamma=0.5, dt=1e-3, precision="fp64")


def _field(kind, ny, nx):
    rng = np.random.default_rng(nx * 8192 + ny)
    f = rng.standard_normal((ny, nx))
    if kind == "range":
        f = f * 10.0 ** rng.uniform(-14, 4, (ny, nx))
    elif kind == "point":
        f[:] = 0.0
        f[ny // 3, nx // 5] = -1.5
    elif kind == "constant":
        f[:] = 0.75
    return f


@pytest.mark.parametrize("kind", ["normal", "range", "point", "constant"])
@pytest.mark.parametrize("n", [(64, 64), (128, 32), (8, 256), (512, 128), (64, 1024), (2048, 16),
                               (16, 2048), (4096, 8), (8, 4096)])
def test_transform_error_is_that_of_rounding(hc, n, kind):
    nx, ny = n
    f = _field(kind, ny, nx)
    ref = packed(sf.fft2(f.astype(np.clongdouble)))
    with _solver(hc, nx, ny) as s:
        got = s.spectrum(f)
    err = np.sqrt(float((np.abs(got - ref) ** 2).sum()) / float((np.abs(ref) ** 2).sum()))
    assert err < TOL, (n, kind, err)


@pytest.mark.parametrize("n", [(64, 64), (256, 128)])
@pytest.mark.parametrize("e", [-1000, -880, 1008])
def test_powers_of_two_scale_exactly(hc, n, e):
    nx, ny = n
    f = _field("normal", ny, nx)
    with _solver(hc, nx, ny) as s:
        base = s.spectrum(f)
        got = s.spectrum(np.ldexp(f, e))
    assert np.isfinite(got).all()
    want = np.empty_like(base)
    want.real = np.ldexp(base.real, e)
    want.imag = np.ldexp(base.imag, e)
    if e > -1000:
        assert (got == want).all()
    else:  # subnormal results are rounded once more
        assert np.abs(got - want).max() <= np.ldexp(1.0, -1073)


def test_zero_and_non_finite_inputs(hc):
    with _solver(hc, 128, 64) as s:
        assert (s.spectrum(np.zeros((64, 128))) == 0).all()
        for bad in (np.nan, np.inf):
            f = _field("normal", 64, 128)
            f[5, 7] = bad
            assert not np.isfinite(s.spectrum(f)).any()
