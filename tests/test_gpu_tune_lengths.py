"""Launch-shape tuning at the lengths that solves run at: every compiled shape of
every pass of 320 ... 3072 points (5/4 and 3/2 of the powers of two) and of 512,
1024 and 2048 points (shared-memory and register forms of the row passes) gives
the same result bit for bit, and sg_autotune covers the lengths between its bounds."""
import itertools

import numpy as np
import pytest

from paper_2001_02765_gb300 import workloads as W
from tests._lib import ensure_built, to_dev

pytestmark = pytest.mark.gpu
LENGTHS = {150: 320, 190: 384, 250: 512, 310: 640, 380: 768, 500: 1024, 600: 1280, 700: 1536, 1000: 2048, 1100: 2560,
           1500: 3072}


@pytest.fixture(scope="module")
def sg():
    import torch
    assert torch.cuda.is_available()
    ensure_built()
    from paper_2001_02765_gb300 import sg as mod

    def defaults():
        for prec in (mod.SG_FP32, mod.SG_FP64):
            for p in [64, 128, 256, 4096] + list(LENGTHS.values()):
                mod.sg_tune_set(prec, p, [0, 0, 0, 0])
    defaults()  # other tests may have tuned lengths between powers of two
    yield mod
    defaults()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("n", sorted(LENGTHS))
def test_every_shape_gives_identical_results(sg, n, mode, prec):
    import torch
    precision = sg.SG_FP32 if prec == "fp32" else sg.SG_FP64
    dt = np.float32 if prec == "fp32" else np.float64
    plan = sg.Plan([(0,) + W.unit_grid(n)], precision=precision, slope_mode=mode)
    pad = plan.info["max_pad"]
    assert pad == LENGTHS[n]
    f = [to_dev(a, dt) for a in W.random_fields(n, n, seed=n)][:3 if mode == 2 else 1]
    ref = [t.clone() for t in plan.force(*f)]
    d = sg.sg_tune_get(precision, pad)
    knobs = ["row_fwd", "row_inv", "col_central" if mode == 1 else "col"]
    tried = 0
    for combo in itertools.product(*[sorted({d[k] // 2, d[k], 2 * d[k]} - {0}) for k in knobs]):
        shape = dict(zip(knobs, combo))
        try:
            sg.sg_tune_set(precision, pad, shape)
        except sg.SgError:
            continue  # not a compiled candidate at this length
        assert sg.sg_tune_get(precision, pad) == dict(d, **shape)
        out = plan.force(*f)
        torch.cuda.synchronize()
        assert torch.equal(out[0], ref[0]) and torch.equal(out[1], ref[1]), shape
        tried += 1
    sg.sg_tune_set(precision, pad, [0, 0, 0, 0])
    plan.close()
    assert tried >= 4


def test_autotune_covers_the_lengths_between(sg):
    res = sg.sg_autotune(sg.SG_FP32, 320, 1280, reps=3)
    assert sorted(res) == [320, 640, 1280] and all(ms > 0 for _, ms in res.values())
    with pytest.raises(sg.SgError):
        sg.sg_autotune(sg.SG_FP32, 320, 900, reps=3)  # 900 is no transform length
