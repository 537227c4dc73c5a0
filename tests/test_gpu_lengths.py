"""Uniform solves at the edges of every transform length (2^k, 5/4 2^k, 3/2 2^k):
the largest patch of each length and the smallest of the next, along either axis,
against numpy's FFT convolution of the plan's own FP64 kernel tables (which other
tests hold to the oracle's; the oracle's entries round at 1e-16 d ln d, which on
these thin grids reaches 1e-12 of the force); batches of such members against
single solves.

Tolerances: FP64 1e-12; FP32 2e-6, about log2(4096) stages of 2^-24 rounding,
doubled for the three transforms in a row."""
import numpy as np
import pytest

from oracle.fftconv import _wrap_correlation_kernel
from paper_2001_02765_gb300 import workloads as W
from tests._lib import ensure_built, to_dev

pytestmark = pytest.mark.gpu
LENGTHS = [128, 256, 320, 384, 512, 640, 768, 1024, 1280, 1536, 2048, 2560, 3072, 4096]


@pytest.fixture(scope="module")
def sg():
    import torch
    assert torch.cuda.is_available()
    ensure_built()
    from paper_2001_02765_gb300 import sg as mod
    return mod


def _central(s, h):
    p = np.pad(s, 1)
    return (p[1:-1, 2:] - p[1:-1, :-2]) / (2 * h), (p[2:, 1:-1] - p[:-2, 1:-1]) / (2 * h)


def _reference(plan, fields):
    ny, nx = fields[0].shape
    p = (2 * ny, 2 * nx)
    spec = [np.fft.rfft2(f, s=p) for f in fields]
    out = []
    for names in (("x0", "xx", "xy"), ("y0", "yx", "yy")):
        k = [np.fft.rfft2(_wrap_correlation_kernel(plan.kernel_table(0, n), *p)) for n in names]
        out.append(np.fft.irfft2(sum(a * b for a, b in zip(spec, k)), s=p)[:ny, :nx])
    return out


def _fields(nx, ny, dt):
    s, sx, sy = W.random_fields(ny, nx, seed=nx + 7 * ny)
    return [a.astype(dt).astype(np.float64) for a in (s, sx, sy)]


@pytest.mark.parametrize("prec, tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("length", LENGTHS)
def test_uniform_at_length_edges(sg, length, axis, mode, prec, tol):
    import torch
    dt = np.float32 if prec == "fp32" else np.float64
    for n in {length // 2, min(2048, length // 2 + 1)}:
        nx, ny = (n, 9) if axis == 0 else (9, n)
        h = 1.0 / n
        s, sx, sy = _fields(nx, ny, dt)
        plan = sg.Plan([(0, nx, ny, 0.0, 0.0, h)], precision=prec, slope_mode=mode)
        fx, fy = plan.force(*[to_dev(a, dt) for a in ((s, sx, sy) if mode == 2 else (s,))])
        torch.cuda.synchronize()
        if mode == 1:
            sx, sy = _central(s, h)
        if mode == 0:
            sx, sy = np.zeros_like(s), np.zeros_like(s)
        rx, ry = _reference(plan, (s, sx, sy))
        gx, gy = (t.cpu().numpy().astype(np.float64).reshape(ny, nx) for t in (fx, fy))
        plan.close()
        err = np.sqrt((np.sum((gx - rx) ** 2) + np.sum((gy - ry) ** 2)) / (np.sum(rx ** 2) + np.sum(ry ** 2)))
        assert err < tol, (n, err)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("layout", [1, 2], ids=["persistent", "grouped"])
def test_batches_of_these_lengths_equal_single_solves(sg, layout, mode, prec):
    import torch
    dt = np.float32 if prec == "fp32" else np.float64
    sizes = [(150, 140), (160, 160), (170, 300), (192, 150), (300, 310), (384, 17), (600, 21), (23, 700), (128, 768)]
    plans, ins, outs, refs = [], [], [], []
    for nx, ny in sizes + sizes[1:3]:
        plan = sg.Plan([(0, nx, ny, 0.0, 0.0, 1.0 / nx)], precision=prec, slope_mode=mode)
        f = [to_dev(a, dt) for a in _fields(nx, ny, dt)][:3 if mode == 2 else 1]
        refs.append([t.clone() for t in plan.force(*f)])
        plans.append(plan)
        ins.append(f + [None] * (3 - len(f)))
        outs.append([torch.full_like(f[0], float("nan")) for _ in range(2)])
    ptr = lambda k, v: [x[k].data_ptr() if x[k] is not None else 0 for x in v]
    batch = sg.sg_batch_create([p.handle for p in plans], ptr(0, ins), ptr(1, ins), ptr(2, ins), ptr(0, outs),
                               ptr(1, outs), mode=layout)
    sg.sg_batch_launch(batch, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert sg.sg_batch_check_error(batch) == sg.SG_OK
    if layout == sg.SG_BATCH_PERSISTENT:
        assert sg.sg_batch_launches(batch) == 1
    sg.sg_batch_destroy(batch)
    for o, r, (nx, ny) in zip(outs, refs, sizes + sizes[1:3]):
        assert torch.equal(o[0], r[0]) and torch.equal(o[1], r[1]), (nx, ny)
    for p in plans:
        p.close()
