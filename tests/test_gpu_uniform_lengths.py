"""Uniform solves of square and ragged grids whose transforms have lengths 5/4 and 3/2
of a power of two (320 to 3072): caller slopes against the oracle's FFT route, central
slopes against the same plan's caller slopes fed with the oracle's central differences
(on noise these are of order 1/h, and the rounding of the oracle's own tables, 1e-16
d ln d an entry, then reaches 1e-11 of the force). Tolerances as in test_gpu_uniform.py
(FP64 1e-12, FP32 1e-5)."""
import numpy as np
import pytest

from oracle.fftconv import central_slopes
from oracle.norms import rel_l2
from paper_2001_02765_gb300 import workloads as W
from tests.test_gpu_uniform import F32_TOL, F64_TOL, _oracle, _solve, sg  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec, tol", [("fp64", F64_TOL), ("fp32", F32_TOL)])
@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("nx, ny", [(150, 150), (310, 190), (380, 601), (700, 640), (1100, 1030), (1500, 777)])
def test_uniform_at_the_odd_lengths(sg, nx, ny, mode, prec, tol):  # noqa: F811
    geom = (nx, ny, -0.4, 0.2, 1.7 / nx)
    dt = np.float64 if prec == "fp64" else np.float32
    s, sx, sy = W.random_fields(ny, nx, seed=nx + 3 * ny)
    fx, fy = _solve(sg, geom, prec, mode, s, sx, sy)
    if mode == sg.SG_SLOPES_CENTRAL:
        cx, cy = central_slopes(np.asarray(s, dt).astype(np.float64), geom[4])
        ox, oy = _solve(sg, geom, prec, sg.SG_SLOPES_CALLER, s, cx, cy)
    else:
        ox, oy = _oracle(sg, geom, mode, s, sx, sy, dt)
    err = rel_l2(fx, fy, ox, oy)
    print("rel L2 %d x %d %s mode %d: %.2e" % (nx, ny, prec, mode, err))
    assert err < tol
