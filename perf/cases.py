"""Performance cases of the thin-disk self-gravity library.

A case is one solve (or one batch of solves) through the public Python binding,
as a simulation calls it once per time step: the plan is made once per grid, the
density changes from step to step. Inputs are seeded: a Kuzmin, spiral or
exponential disk with a random centre, scale and small noise, evaluated at the
cell centres in FP64 and rounded to the plan's precision; caller slopes are the
analytic gradient.

Kinds of cases:
* uniform: one patch of nx x ny cells (force, potential or off-plane force);
* nested:  centred ratio-2 patches of base x base cells, level l on
           [-2^-l, 2^-l]^2 (a zoom-in run);
* zones:   the zone-by-zone hierarchies refined along the disk edge (independent
           or variable level refinement);
* batch:   many uneven uniform disks bound into one batch.
"""
import functools
import math

import numpy as np
import torch

from paper_2001_02765_gb300 import sg
from paper_2001_02765_gb300 import workloads as W

SLOPES = {"none": sg.SG_SLOPES_NONE, "central": sg.SG_SLOPES_CENTRAL, "caller": sg.SG_SLOPES_CALLER}


def _uniform(nx, ny, precision="fp32", slopes="central", quantity="force", disk="spiral"):
    return dict(kind="uniform", nx=nx, ny=ny, precision=precision, slopes=slopes, quantity=quantity, disk=disk)


def _nested(base, levels, precision="fp32", quantity="force"):
    return dict(kind="nested", base=base, levels=levels, precision=precision, slopes="caller", quantity=quantity,
                disk="exponential")


def listed():
    cases = [
        # the smallest grid in use (a 64^2 galaxy model stepped many times): launch and latency bound
        ("uniform_64", _uniform(64, 64, disk="kuzmin")),
        # the ordinary production step: a 1024^2 spiral disk, slopes by central differences
        ("uniform_1024", _uniform(1024, 1024)),
        # a ragged grid with slopes from the caller's reconstruction
        ("uniform_1100x1030_caller", _uniform(1100, 1030, slopes="caller")),
        # the largest single patch
        ("uniform_2048", _uniform(2048, 2048)),
        # a double-precision run at an ordinary size of the serving mix
        ("uniform_704_fp64", _uniform(704, 704, precision="fp64")),
        # the potential (energy diagnostics) beside the force
        ("potential_1024", _uniform(1024, 1024, quantity="potential")),
        # forces on a layer above the plane
        ("offplane_1024", _uniform(1024, 1024, slopes="caller", quantity="force3")),
        # three nested levels, the ordinary zoom-in hierarchy (level convolutions)
        ("nested_3x256", _nested(256, 3)),
        # six nested levels: the finest extent exceeds the level convolutions (cross-patch sum)
        ("nested_6x256_deep", _nested(256, 6)),
        # off-plane forces on a hierarchy (cross-patch sum)
        ("offplane_nested_3x256", _nested(256, 3, quantity="force3")),
        # the paper's edge-refined disk, N = 512, three levels, zone by zone
        ("zones_ilr_512", dict(kind="zones", n=512, levels=3, rule="ilr", disk="d2", precision="fp32", slopes="caller",
                               quantity="force")),
        # 64 uneven disks of a parameter study in one batch launch
        ("batch_64", dict(kind="batch", count=64, lo=64, hi=512, size_seed=4, precision="fp32", slopes="central",
                          quantity="force", disk="spiral")),
    ]
    return [dict(c, name=n) for n, c in cases]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    known = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        c = _draw(rng)
        if c not in known:
            return c


def _draw(rng):
    u = rng.random()
    if u < 0.55:
        n = _log_int(rng, 64, 2048)
        nx, ny = n, n
        if rng.random() < 0.5:  # ragged grids, aspect up to 1.5
            ny = max(64, min(2048, int(round(n * rng.uniform(2.0 / 3.0, 1.5)))))
        if rng.random() < 0.3:  # multiples of 64, the grids of the serving mix
            nx, ny = max(128, nx // 64 * 64), max(128, ny // 64 * 64)
        precision = "fp64" if rng.random() < 0.2 else "fp32"
        slopes = rng.choice(["central", "central", "caller", "none"])
        quantity = rng.choice(["force", "force", "force", "potential", "force3"])
        return _uniform(nx, ny, precision, slopes, quantity, rng.choice(["kuzmin", "spiral", "exponential"]))
    if u < 0.8:
        quantity = rng.choice(["force", "force", "potential", "force3"])
        levels = rng.randint(2, 3 if quantity == "force3" else 6)
        base = 4 * (_log_int(rng, 64, 256) // 4)
        precision = "fp64" if quantity != "force3" and levels <= 3 and rng.random() < 0.15 else "fp32"
        return _nested(base, levels, precision, quantity)
    if u < 0.88:
        rule = rng.choice(["ilr", "vlr"])
        return dict(kind="zones", n=64 * rng.randint(2, 8), levels=rng.randint(2, 3), rule=rule,
                    disk=rng.choice(["d2", "d22"]), precision="fp32", slopes="caller",
                    quantity=rng.choice(["force", "potential"]))
    lo = _log_int(rng, 64, 256)
    return dict(kind="batch", count=_log_int(rng, 8, 64), lo=lo, hi=max(lo + 32, _log_int(rng, 128, 512)),
                size_seed=rng.randint(0, 1 << 20), precision="fp32", slopes=rng.choice(["central", "caller"]),
                quantity="force", disk="spiral")


# ---------------------------------------------------------------- geometry --

def _unit(n):
    return 2.0 / n


@functools.lru_cache(maxsize=4)
def _hierarchy(n, levels, rule, disk):
    """The zone list of a zones case (seeded by nothing: the refinement follows the disk edge)."""
    return W.band_hierarchy(n, levels, rule, disk)


def _patches(case):
    """(level, nx, ny, x0, y0, h) of every patch of a uniform or nested case."""
    if case["kind"] == "uniform":
        h = _unit(max(case["nx"], case["ny"]))
        return [(0, case["nx"], case["ny"], -0.5 * case["nx"] * h, -0.5 * case["ny"] * h, h)]
    b = case["base"]
    return [(lev, b, b, -(2.0 ** -lev), -(2.0 ** -lev), _unit(b) / 2 ** lev) for lev in range(case["levels"])]


def _height(case):
    """Targets one finest cell above the plane for off-plane cases."""
    return _patches(case)[-1][5] if case["quantity"] == "force3" else 0.0


def _sizes(case):
    """Grid sizes of a batch's members."""
    rng = np.random.Generator(np.random.PCG64(case["size_seed"]))
    u = rng.uniform(math.log(case["lo"]), math.log(case["hi"]), size=case["count"])
    return [int(v) for v in np.rint(np.exp(u))]


def _leaf_patches(case):
    """Leaf masks (bool [ny, nx], on the GPU) of the patches of a nested case."""
    b, out = case["base"], []
    for lev in range(case["levels"]):
        m = torch.ones(b, b, dtype=torch.bool, device="cuda")
        if lev + 1 < case["levels"]:
            m[b // 4:b // 4 + b // 2, b // 4:b // 4 + b // 2] = False
        out.append(m)
    return out


# ------------------------------------------------------------------ inputs --

class _Disk:
    """A seeded disk: density and gradient at given points (FP64, on the GPU)."""

    def __init__(self, disk, seed):
        g = np.random.Generator(np.random.PCG64(seed))
        self.disk = disk
        self.cx, self.cy = g.uniform(-0.02, 0.02, 2)
        self.a = g.uniform(0.08, 0.2)
        self.amp = g.uniform(0.05, 0.2) if disk == "spiral" else 0.0
        self.radius = g.uniform(0.48, 0.52)
        self.noise = torch.Generator(device="cuda")
        self.noise.manual_seed(int(seed) & 0x7fffffff)

    def at(self, x, y):
        x, y = x - self.cx, y - self.cy
        r2 = x * x + y * y
        if self.disk == "exponential":
            r = torch.sqrt(r2).clamp_min(1e-12)
            s = torch.exp(-r / self.a)
            g = -s / (self.a * r)
            sx, sy = g * x, g * y
        elif self.disk in ("d2", "d22"):
            # the smooth-edged disk(s) of the refinement hierarchies
            s = sx = sy = 0.0
            for oy in ((0.0,) if self.disk == "d2" else (0.5, -0.5)):
                rad = self.radius if self.disk == "d2" else 0.8 * self.radius
                q = (1.0 - (x * x + (y - oy) ** 2) / rad ** 2).clamp_min(0.0)
                g = -3.0 * torch.sqrt(q) / rad ** 2
                s, sx, sy = s + q ** 1.5, sx + g * x, sy + g * (y - oy)
        else:
            q = r2 + self.a ** 2
            s = self.a / (2.0 * math.pi * q ** 1.5)
            sx, sy = -3.0 * s / q * x, -3.0 * s / q * y
            if self.amp:
                k = 1.0 / math.tan(math.radians(15.0))
                r2s = r2.clamp_min(1e-12)
                ph = 2.0 * torch.atan2(y, x) - 0.5 * k * torch.log(r2s)
                m, sn = 1.0 + self.amp * torch.cos(ph), self.amp * torch.sin(ph)
                sx, sy = sx * m - s * sn * (-2.0 * y - k * x) / r2s, sy * m - s * sn * (2.0 * x - k * y) / r2s
                s = s * m
        s = s + (torch.rand(s.shape, generator=self.noise, dtype=s.dtype, device=s.device) - 0.5) * 2e-3
        return s, sx, sy


def _centres(p):
    _, nx, ny, x0, y0, h = p
    x = x0 + (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) * h
    y = y0 + (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) * h
    return x[None, :].expand(ny, nx), y[:, None].expand(ny, nx)


def _dtype(case):
    return torch.float32 if case["precision"] == "fp32" else torch.float64


def _patch_fields(case, patches, seed, disk=None):
    """sigma, dx, dy over the concatenated patches, in the plan's precision."""
    d = _Disk(disk or case["disk"], seed)
    parts = [d.at(*_centres(p)) for p in patches]
    return [torch.cat([q[k].reshape(-1) for q in parts]).to(_dtype(case)) for k in range(3)]


def _zone_fields(case, seed):
    hier = _hierarchy(case["n"], case["levels"], case["rule"], case["disk"])
    xc, yc, _ = W.zone_geometry(hier)
    d = _Disk(case["disk"], seed)
    f = d.at(torch.from_numpy(xc).cuda(), torch.from_numpy(yc).cuda())
    return [v.to(_dtype(case)) for v in f]


def _member_fields(case, seed):
    """Flat fields of a batch's members, each starting on a 256-byte boundary: (offsets, sizes, sigma, dx, dy)."""
    sizes, offs, total = _sizes(case), [], 0
    for n in sizes:
        offs.append(total)
        total += (n * n + 63) // 64 * 64
    flat = [torch.zeros(total, dtype=_dtype(case), device="cuda") for _ in range(3)]
    for k, (n, o) in enumerate(zip(sizes, offs)):
        f = _patch_fields(case, [(0, n, n, -1.0, -1.0, _unit(n))], seed * 1000 + k)
        for a, b in zip(flat, f):
            a[o:o + n * n] = b
    return offs, sizes, flat


# ------------------------------------------------------------------ states --

class _Batch:
    """A batch with its plans and buffers; released in order."""

    def __init__(self, case, seed):
        offs, sizes, (s, dx, dy) = _member_fields(case, seed)
        self.inputs = (s, dx, dy)
        self.fx, self.fy = torch.zeros_like(s), torch.zeros_like(s)
        self.plans = [sg.Plan([(0, n, n, -1.0, -1.0, _unit(n))], precision=case["precision"],
                              slope_mode=SLOPES[case["slopes"]]) for n in sizes]
        es = s.element_size()
        at = lambda t: [t.data_ptr() + o * es for o in offs]
        caller = case["slopes"] == "caller"
        torch.cuda.synchronize()
        self.handle = sg.sg_batch_create([p.handle for p in self.plans], at(s), at(dx) if caller else [0] * len(offs),
                                         at(dy) if caller else [0] * len(offs), at(self.fx), at(self.fy))

    def __del__(self):
        if getattr(self, "handle", None):
            sg.sg_batch_destroy(self.handle)
        for p in getattr(self, "plans", []):
            p.close()


def prepare(case, seed):
    if case["kind"] == "batch":
        return dict(case=case, batch=_Batch(case, seed))
    if case["kind"] == "zones":
        hier = _hierarchy(case["n"], case["levels"], case["rule"], case["disk"])
        plan = sg.ZonePlan(case["n"], case["n"], hier["x0"], hier["y0"], hier["h0"], hier["level"], hier["ix"],
                           hier["iy"], precision=case["precision"], slope_mode=SLOPES[case["slopes"]])
        fields, leaf = _zone_fields(case, seed), None
    else:
        patches = _patches(case)
        plan = sg.Plan(patches, precision=case["precision"], slope_mode=SLOPES[case["slopes"]], z=_height(case))
        fields = _patch_fields(case, patches, seed)
        leaf = torch.cat([m.reshape(-1) for m in _leaf_patches(case)]) if case["kind"] == "nested" else None
    if case["slopes"] != "caller":
        fields = [fields[0], None, None]
    return dict(case=case, plan=plan, fields=fields, leaf=leaf, zero=torch.zeros((), dtype=_dtype(case), device="cuda"))


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        sg.sg_batch_launch(b.handle, torch.cuda.current_stream().cuda_stream)
        return [b.fx, b.fy]
    plan, f, q = state["plan"], state["fields"], case["quantity"]
    if case["kind"] == "zones":
        return list(plan.force_zones(*f)) if q == "force" else [plan.potential_zones(*f)]
    if q == "force":
        out = list(plan.force(*f))
    elif q == "force3":
        out = list(plan.force3(*f))
    else:
        out = [plan.potential(*f)]
    if state["leaf"] is not None:
        # values at covered cells are unspecified: a simulation takes the leaves'
        out = [torch.where(state["leaf"], v, state["zero"]) for v in out]
    return out


# ------------------------------------------------------------------- work --

def _conv_flops(nx, ny, fields, outs):
    """Real transforms of the doubled lengths (2.5 P log2 P each way) and the products."""
    p = 4.0 * nx * ny
    return 2.5 * p * math.log2(p) * (fields + outs) + 2.0 * p * fields * outs


def work(case):
    es = 4 if case["precision"] == "fp32" else 8
    fields = {"none": 1, "central": 1, "caller": 3}[case["slopes"]]
    outs = {"force": 2, "force3": 3, "potential": 1}[case["quantity"]]
    if case["kind"] == "uniform":
        grids = [(case["nx"], case["ny"])]
    elif case["kind"] == "nested":
        grids = [(case["base"], case["base"])] * case["levels"]
    elif case["kind"] == "batch":
        grids = [(n, n) for n in _sizes(case)]
    else:
        lev = _hierarchy(case["n"], case["levels"], case["rule"], case["disk"])["level"]
        grids = [(math.sqrt(c), math.sqrt(c)) for c in np.bincount(lev)]
    cells = sum(a * b for a, b in grids)
    return {"bytes": es * cells * (fields + outs), "flops": sum(_conv_flops(a, b, fields, outs) for a, b in grids)}


# ------------------------------------------------------------------ exact --
#
# The same sums in FP64 from the closed-form cell integrals, by FFTs of torch:
# every pair of levels is a set of plain convolutions, one per residue class of
# the finer level's cells modulo the ratio of the cell widths.

def _asinh_ratio(v, u):
    """asinh(v / |u|), on the line u = 0 its limit inside a double difference, sgn(v) ln|v|."""
    au = u.abs()
    safe = torch.where(au > 0, au, torch.ones_like(au))
    on = torch.sign(v) * torch.log(v.abs())
    return torch.where(au > 0, torch.asinh(v / safe), on)


def _dd(f, u, v):
    """Double difference of f over the corners (u[0], u[1]) x (v[0], v[1])."""
    return f(u[1], v[1]) - f(u[1], v[0]) - f(u[0], v[1]) + f(u[0], v[0])


def _integrals(cx, cy, h, z, quantity):
    """Cell integrals of a cell of width h centred at (cx, cy) from the target: per output, the
    factors of sigma, dx and dy."""
    cx, cy = torch.broadcast_tensors(cx, cy)
    u, v = (cx - 0.5 * h, cx + 0.5 * h), (cy - 0.5 * h, cy + 0.5 * h)
    clean = lambda t: torch.nan_to_num(t, nan=0.0, posinf=0.0, neginf=0.0)
    if quantity == "potential":
        prod = lambda a, g: torch.where(a == 0, torch.zeros_like(g), a * g)
        p0 = _dd(lambda a, b: prod(a, _asinh_ratio(b, a)) + prod(b, _asinh_ratio(a, b)), u, v)
        px = _dd(lambda a, b: 0.5 * (b * torch.hypot(a, b) + a * prod(a, _asinh_ratio(b, a))), u, v) - cx * p0
        py = _dd(lambda a, b: 0.5 * (a * torch.hypot(a, b) + b * prod(b, _asinh_ratio(a, b))), u, v) - cy * p0
        return [[clean(-p0), clean(-px), clean(-py)]]
    az = abs(z)
    rad = lambda a, b: torch.sqrt(a * a + b * b + z * z)
    if z == 0.0:
        gx, gy = (lambda a, b: _asinh_ratio(b, a)), (lambda a, b: _asinh_ratio(a, b))
        at = None
    else:
        gx = lambda a, b: torch.asinh(b / torch.sqrt(a * a + z * z))
        gy = lambda a, b: torch.asinh(a / torch.sqrt(b * b + z * z))
        at = _dd(lambda a, b: torch.atan(a * b / (az * rad(a, b))), u, v)
    prod = lambda a, g: torch.where(a == 0, torch.zeros_like(g), a * g)
    x0, y0 = -_dd(gx, u, v), -_dd(gy, u, v)
    r = _dd(rad, u, v)
    xx = _dd(lambda a, b: prod(b, gy(a, b)), u, v) - cx * x0
    yy = _dd(lambda a, b: prod(a, gx(a, b)), u, v) - cy * y0
    if at is not None:
        xx, yy = xx - az * at, yy - az * at
    out = [[x0, xx, -r - cy * x0], [y0, -r - cx * y0, yy]]
    if quantity == "force3":
        sz = math.copysign(1.0, z)
        z0 = -sz * at
        out.append([z0, -cx * z0 - z * x0, -cy * z0 - z * y0])
    return [[clean(t) for t in row] for row in out]


def _convolve(src, shape, step, off, h, z, quantity):
    """Sums over the cells of src ([3][ny][nx], spacing step, width h) at targets [shape] of the same
    spacing; off: source cell (0, 0) centre minus target (0, 0)."""
    sy, sx = src[0].shape
    ty, tx = shape
    ly, lx = (sy + ty + 14) // 16 * 16, (sx + tx + 14) // 16 * 16
    ar = lambda n, l: torch.where(torch.arange(l, device="cuda") < n, torch.arange(l, device="cuda"),
                                  torch.arange(l, device="cuda") - l).double()
    # entry e of the wrapped table: target index minus source index
    ex, ey = ar(tx, lx), ar(ty, ly)
    tabs = _integrals((off[0] - ex * step)[None, :], (off[1] - ey * step)[:, None], h, z, quantity)
    spec = [torch.fft.rfft2(f, s=(ly, lx)) if f is not None else None for f in src]
    out = []
    for row in tabs:
        acc = sum(torch.fft.rfft2(t) * s for t, s in zip(row, spec) if s is not None)
        out.append(torch.fft.irfft2(acc, s=(ly, lx))[:ty, :tx])
    return out


def _central(s, h):
    """Central differences, zero outside the patch."""
    p = torch.nn.functional.pad(s, (1, 1, 1, 1))
    return (p[1:-1, 2:] - p[1:-1, :-2]) / (2 * h), (p[2:, 1:-1] - p[:-2, 1:-1]) / (2 * h)


def _exact_uniform(case, patch, fields):
    """One patch: fields [sigma, dx, dy] flat, rounded to the plan's precision."""
    _, nx, ny, _, _, h = patch
    f = [t.double().reshape(ny, nx) for t in fields]
    if case["slopes"] == "central":
        f[1], f[2] = _central(f[0], h)
    elif case["slopes"] == "none":
        f[1] = f[2] = None
    z = h if case["quantity"] == "force3" else 0.0
    return [t.reshape(-1) for t in _convolve(f, (ny, nx), h, (0.0, 0.0), h, z, case["quantity"])]


def _exact_levels(levels, z, quantity):
    """levels: per level dict(h, i0, j0, src [3][ny][nx] zero off the leaves, leaf [ny][nx]) on images of
    its own lattice (cell (i0, j0) first; all lattices start at the same corner). Returns per level the
    outputs [ny][nx], zero off the leaves."""
    outs = []
    for t in levels:
        tj, ti = t["leaf"].shape
        res = None
        for s in levels:
            f = max(1, int(round(s["h"] / t["h"])))   # coarser source: targets in f x f classes
            c = max(1, int(round(t["h"] / s["h"])))   # finer source: sources in c x c classes
            for a in range(max(f, c)):
                for b in range(max(f, c)):
                    # cells whose global index is b mod the ratio along x, a along y
                    fi = lambda first, m, r: (r - first) % m
                    if f > 1:
                        ox, oy = fi(t["i0"], f, b), fi(t["j0"], f, a)
                        if ox >= ti or oy >= tj:
                            continue
                        sub, src, step = t["leaf"][oy::f, ox::f], s["src"], s["h"]
                        sx0, sy0, tx0, ty0 = s["i0"], s["j0"], t["i0"] + ox, t["j0"] + oy
                    else:
                        ox, oy = fi(s["i0"], c, b), fi(s["j0"], c, a)
                        src = [v[oy::c, ox::c] for v in s["src"]]
                        if 0 in src[0].shape:
                            continue
                        sub, step = t["leaf"], t["h"]
                        sx0, sy0, tx0, ty0 = s["i0"] + ox, s["j0"] + oy, t["i0"], t["j0"]
                    off = ((sx0 + 0.5) * s["h"] - (tx0 + 0.5) * t["h"], (sy0 + 0.5) * s["h"] - (ty0 + 0.5) * t["h"])
                    got = _convolve(src, sub.shape, step, off, s["h"], z, quantity)
                    if res is None:
                        res = [torch.zeros(tj, ti, dtype=torch.float64, device="cuda") for _ in got]
                    for r, g in zip(res, got):
                        if f > 1:
                            r[oy::f, ox::f] += g
                        else:
                            r += g
        outs.append([torch.where(t["leaf"], r, torch.zeros_like(r)) for r in res])
    return outs


def exact(case, seed):
    if case["kind"] == "uniform":
        p = _patches(case)
        return _exact_uniform(case, p[0], _patch_fields(case, p, seed))
    if case["kind"] == "batch":
        offs, sizes, flat = _member_fields(case, seed)
        out = [torch.zeros(flat[0].numel(), dtype=torch.float64, device="cuda") for _ in range(2)]
        for n, o in zip(sizes, offs):
            got = _exact_uniform(case, (0, n, n, -1.0, -1.0, _unit(n)), [t[o:o + n * n] for t in flat])
            for a, b in zip(out, got):
                a[o:o + n * n] = b
        return out
    levels = []
    if case["kind"] == "nested":
        patches, b = _patches(case), case["base"]
        fields, leaf = _patch_fields(case, patches, seed), _leaf_patches(case)
        for k, p in enumerate(patches):
            f = [t[k * b * b:(k + 1) * b * b].double().reshape(b, b) * leaf[k] for t in fields]
            i0 = int(round((p[3] + 1.0) / p[5]))
            levels.append(dict(h=p[5], i0=i0, j0=i0, src=f, leaf=leaf[k]))
        outs = _exact_levels(levels, _height(case), case["quantity"])
        return [torch.cat([o[k].reshape(-1) for o in outs]) for k in range(len(outs[0]))]
    # zones: every level's zones on the image of their bounding box
    hier = _hierarchy(case["n"], case["levels"], case["rule"], case["disk"])
    fields = [t.double() for t in _zone_fields(case, seed)]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    lev, ix, iy, isleaf = dev(hier["level"]), dev(hier["ix"]).long(), dev(hier["iy"]).long(), dev(hier["leaf"])
    places = []
    for m in range(int(hier["level"].max()) + 1):
        k = torch.nonzero(lev == m).reshape(-1)
        i0, j0 = int(ix[k].min()), int(iy[k].min())
        nx, ny = int(ix[k].max()) - i0 + 1, int(iy[k].max()) - j0 + 1
        slot = (iy[k] - j0) * nx + ix[k] - i0
        img = lambda v: torch.zeros(ny * nx, dtype=v.dtype, device="cuda").index_put_((slot,), v).reshape(ny, nx)
        leaf = img(isleaf[k])
        levels.append(dict(h=hier["h0"] / 2 ** m, i0=i0, j0=j0, src=[img(f[k]) * leaf for f in fields], leaf=leaf))
        places.append((k, slot))
    outs = _exact_levels(levels, 0.0, case["quantity"])
    res = [torch.zeros(lev.numel(), dtype=torch.float64, device="cuda") for _ in outs[0]]
    for (k, slot), o in zip(places, outs):
        for r, v in zip(res, o):
            r[k] = v.reshape(-1)[slot]
    return res
