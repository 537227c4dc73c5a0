"""Potential and off-plane force with central slopes (formed in the column pass from
the transform of sigma) against the same plan fed those slopes by the caller (three
transforms), at the edges of every transform length, along either axis.

Tolerances, relative to the norm of the result: FP64 1e-12; FP32 2e-6, about
log2(4096) stages of 2^-24 rounding, doubled for the three transforms in a row."""
import numpy as np
import pytest

from paper_2001_02765_gb300 import workloads as W
from tests._lib import ensure_built, to_dev

pytestmark = pytest.mark.gpu
LENGTHS = [2, 16, 64, 128, 256, 320, 384, 512, 640, 768, 1024, 1280, 1536, 2048, 2560, 3072, 4096]


@pytest.mark.parametrize("prec, tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("what", ["potential", "offplane"])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("length", LENGTHS)
def test_central_slopes_equal_caller_slopes(length, axis, what, prec, tol):
    import torch
    ensure_built()
    from paper_2001_02765_gb300 import sg
    dt = np.float32 if prec == "fp32" else np.float64
    for n in {length // 2, min(2048, length // 2 + 1)}:
        nx, ny = (n, 9) if axis == 0 else (9, n)
        h = 1.0 / n
        s = W.random_fields(ny, nx, seed=nx + 7 * ny)[0].astype(dt).astype(np.float64)
        p = np.pad(s, 1)
        sx, sy = (p[1:-1, 2:] - p[1:-1, :-2]) / (2 * h), (p[2:, 1:-1] - p[:-2, 1:-1]) / (2 * h)
        out = []
        for mode, fields in ((1, (s,)), (2, (s, sx, sy))):
            plan = sg.Plan([(0, nx, ny, 0.0, 0.0, h)], precision=prec, slope_mode=mode,
                           z=3 * h if what == "offplane" else 0.0)
            args = [to_dev(a, dt) for a in fields]
            got = plan.force3(*args) if what == "offplane" else (plan.potential(*args),)
            torch.cuda.synchronize()
            out.append(np.stack([t.cpu().numpy().astype(np.float64).ravel() for t in got]))
            plan.close()
        assert np.linalg.norm(out[0] - out[1]) < tol * np.linalg.norm(out[1]), (nx, ny)
