"""The FP32 cross-patch sum (clusters, middle cells, near tables or the corner
form) against the oracle's plain leaf sum, on shapes where its index rules can go
wrong: patches ending inside a cluster, several patches per level, the
smallest patches, width ratios beyond the near tables, budgets that leave them out.

Tolerance 2e-6 (relative L2 over the leaves): the stated truncations of the middle
cells (1.02e-6) and of the clusters on both sides (2 x 2e-7) plus the FP32 transforms'
4.4e-7, rounded up."""
import numpy as np
import pytest

from oracle import amr as oamr
from oracle.direct import direct_force3
from oracle.potential import amr_direct_potential
from paper_2001_02765_gb300 import workloads as W
from tests._lib import concat_dev, ensure_built, gather_leaves

pytestmark = pytest.mark.gpu
TOL = 2e-6

H = 1.0 / 32
SHAPES = {
    # 41 x 27 with two level-1 patches, one of them with a child; ends one past, on and before a cluster's edge
    "ragged": [(0, 41, 27, 0.0, 0.0, H), (1, 34, 18, 5 * H, 3 * H, H / 2), (1, 16, 32, 25 * H, 4 * H, H / 2),
               (2, 18, 16, 5 * H + 3 * H, 3 * H + 0.5 * H, H / 4)],
    # two level-0 patches side by side (same cell width) and a 2 x 2 child
    "side": [(0, 9, 8, 0.0, 0.0, H), (0, 7, 23, 9 * H, -2 * H, H), (1, 2, 2, 4 * H, 3 * H, H / 2)],
    # eight nested levels: width ratios up to 2^7
    "deep": [(lev,) + p for lev, p in enumerate(W.centred_nested_patches(16, 8))],
    # four cluster levels on the coarse patch, clusters wider than the fine blocks
    "wide": [(0, 130, 121, -1.0, -1.0, 2.0 / 128), (1, 24, 40, 0.0, 0.25, 1.0 / 128)],
}


@pytest.fixture(scope="module")
def sg():
    import torch
    assert torch.cuda.is_available()
    ensure_built()
    from paper_2001_02765_gb300 import sg as mod
    return mod


def _fields(patches, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    r = lambda lo, w: [rng.uniform(lo, 1, (p[2], p[1])).astype(np.float32).astype(np.float64) * w / p[5] ** (w != 1)
                       for p in patches]
    f32 = lambda a: [x.astype(np.float32).astype(np.float64) for x in a]
    return r(-1, 1), f32(r(-1, 0.5)), f32(r(-1, 0.5))


def _reference(patches, kind, f, z):
    P = oamr.make_patches(patches)
    if kind == "force":
        leaves, rx, ry = oamr.amr_direct_force(P, *f)
        return leaves, [rx, ry]
    if kind == "potential":
        leaves, ref = amr_direct_potential(P, *f)
        return leaves, [ref]
    leaves = oamr.leaf_cells(P)
    off = np.cumsum([0] + [p.nx * p.ny for p in P])
    idx = np.array([off[k] + j * P[k].nx + i for k, j, i in zip(leaves["patch"], leaves["j"], leaves["i"])])
    flat = [np.concatenate([a.ravel() for a in g])[idx] for g in f]
    return leaves, list(direct_force3((leaves["xl"], leaves["xr"], leaves["yd"], leaves["yu"]), *flat, leaves["xc"],
                                      leaves["yc"], z))


def _solve(plan, kind, f):
    import torch
    a = [concat_dev(g, np.float32) for g in f]
    out = {"force": plan.force, "potential": lambda *x: [plan.potential(*x)], "force3": plan.force3}[kind](*a)
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in out]


@pytest.mark.parametrize("kind", ["force", "potential", "force3"])
@pytest.mark.parametrize("shape", sorted(SHAPES))
@pytest.mark.parametrize("tight", [False, True], ids=["tables", "corner-form"])
def test_cross_sum_matches_plain_sum(sg, shape, kind, tight):
    patches = SHAPES[shape]
    z = 0.4 * patches[-1][5] if kind == "force3" else 0.0
    f = _fields(patches, seed=len(shape))
    budget = 0
    if tight:
        # a budget that holds everything but the largest near tables
        with pytest.raises(sg.SgError) as e:
            sg.Plan(patches, cross_mode=sg.SG_CROSS_DIRECT, z=z, hbm_budget=1)
        assert e.value.status == sg.SG_EBUDGET
        budget = sg.sg_plan_bytes(patches, sg.SG_FP32, z=z, cross_mode=sg.SG_CROSS_DIRECT) - 1
    plan = sg.Plan(patches, cross_mode=sg.SG_CROSS_DIRECT, z=z, hbm_budget=budget)
    assert plan.info["cross_mode"] == sg.SG_CROSS_DIRECT
    got = _solve(plan, kind, f)
    again = _solve(plan, kind, f)
    leaves, ref = _reference(patches, kind, f, z)
    g = [gather_leaves(plan, v, leaves) for v in got]
    h = [gather_leaves(plan, v, leaves) for v in again]
    plan.close()
    assert all(np.array_equal(a, b) for a, b in zip(g, h))
    err = np.sqrt(sum(np.sum((a - b) ** 2) for a, b in zip(g, ref)) / sum(np.sum(b ** 2) for b in ref))
    print("rel L2 %s %s: %.2e" % (shape, kind, err))
    assert err < TOL
