"""The measured cases of the PLIC hot path: what a user of this framework has it do.

Six kinds of work, each through the public entry points of
``paper_2006_12838_gb300`` as a program calls them:

* ``offset``     -- plane offsets of a batch of cells (``plic.offset``), the
  inversion that every VOF step makes;
* ``roundtrip``  -- the same with the forward volume of the result
  (``plic.offset_roundtrip``), the benchmark's step;
* ``offset_grad`` -- forward and backward through ``autograd.offset``;
* ``field``      -- one curvature step of a simulation: the list of interface
  cells of a fill field and their mean curvature, chained on the device
  (``plic.interface_compact`` and ``plic.curvature`` with the device count);
* ``batched``    -- the curvature of many fields of uneven size in one call
  (``plic.curvature_batched``);
* ``curvature_grad`` -- forward and backward through ``autograd.curvature``.

``listed()`` names the fixed cases, ``draw()`` gives others of the same ranges.
Inputs are made on the GPU from the seed.  The formulas in this file (plane-cube
volume, its inverse by bisection, the paraboloid fit) are plain torch in 64 bits
and share nothing with the library.
"""
import math

import torch

from paper_2006_12838_gb300 import autograd, plic

DEV = "cuda"
F64 = torch.float64
CHUNK = 1 << 24                        # cells per step of input making and of exact()
DTYPES = {"fp32": torch.float32, "fp32p": torch.float32, "fp64": F64, "fp64r": F64}


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    """Twelve cases; the sizes are those of the tests, the benchmark and the README."""
    return [
        # a small solver's call: a few thousand interface cells, launch and call latency
        {"name": "offset_4099", "kind": "offset", "n": 4099, "method": "sz_opt", "precision": "fp32p",
         "rows": False},
        # the paper's own solver on the rows of one (3, n) tensor of normals (the README's use);
        # an odd n leaves the rows on 4-byte boundaries
        {"name": "offset_analytic_rows_odd", "kind": "offset", "n": 10_000_019, "method": "analytic",
         "precision": "fp32p", "rows": True},
        # double precision, the default for double tensors
        {"name": "offset_fp64_2p24", "kind": "offset", "n": 1 << 24, "method": "sz_opt", "precision": "fp64",
         "rows": False},
        # double precision refined from a single-precision solve, an odd count
        {"name": "offset_fp64r_odd", "kind": "offset", "n": 16_000_057, "method": "sz_opt",
         "precision": "fp64r", "rows": False},
        # the benchmark's step at its full size
        {"name": "roundtrip_2p28", "kind": "roundtrip", "n": 1 << 28, "method": "sz_opt", "precision": "fp32p"},
        # a training step through the inversion: forward and all four gradients
        {"name": "offset_grad_32m", "kind": "offset_grad", "n": 32_000_003, "dtype": "fp32"},
        # the curvature step of a small field (tests, two-dimensional studies): latency
        {"name": "field_64", "kind": "field", "nx": 64, "ny": 64, "nz": 64, "drops": 2, "rmin": 6.0, "rmax": 14.0},
        # the benchmark's curvature field
        {"name": "field_256", "kind": "field", "nx": 256, "ny": 256, "nz": 256, "drops": 8, "rmin": 6.0,
         "rmax": 40.0},
        # odd edges: rows that are neither aligned nor whole words
        {"name": "field_odd", "kind": "field", "nx": 301, "ny": 203, "nz": 257, "drops": 12, "rmin": 5.0,
         "rmax": 30.0},
        # the benchmark's largest field (1 GiB), a spray of many droplets
        {"name": "field_1gib", "kind": "field", "nx": 1024, "ny": 512, "nz": 512, "drops": 60, "rmin": 5.0,
         "rmax": 40.0},
        # many fields of uneven size in one launch
        {"name": "batched_64", "kind": "batched", "fields": 64, "edges": "32,64,96,128,192,256"},
        # a training step through the curvature: forward and the dense gradient of the field
        {"name": "curvature_grad_drop", "kind": "curvature_grad", "nx": 400, "ny": 300, "nz": 350, "ax": 60.0,
         "ay": 80.0, "az": 100.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["offset", "offset", "offset", "roundtrip", "offset_grad", "field", "field", "field",
                       "batched", "curvature_grad"])
    if kind == "offset":
        p = rng.choice(["fp32", "fp32p", "fp64", "fp64r"])
        return {"kind": kind, "n": _log_int(rng, 1000, 16_000_000 if p.startswith("fp64") else 64_000_000),
                "method": rng.choice(["sz_opt", "analytic"]), "precision": p, "rows": rng.random() < 0.4}
    if kind == "roundtrip":
        return {"kind": kind, "n": _log_int(rng, 10_000, 1 << 28), "method": "sz_opt", "precision": "fp32p"}
    if kind == "offset_grad":
        return {"kind": kind, "n": _log_int(rng, 1000, 32_000_000), "dtype": rng.choice(["fp32", "fp64"])}
    if kind == "field":
        e = [_log_int(rng, 40, 800) for _ in range(3)]
        while e[0] * e[1] * e[2] > 1 << 27:
            e[rng.randrange(3)] = _log_int(rng, 40, 800)
        if rng.random() < 0.5:
            e[0] = (e[0] + 31) // 32 * 32
        big = min(40.0, min(e) / 4)
        return {"kind": kind, "nx": e[0], "ny": e[1], "nz": e[2], "drops": _log_int(rng, 1, 60), "rmin": 4.0,
                "rmax": round(rng.uniform(6.0, max(7.0, big)), 2)}
    if kind == "batched":
        return {"kind": kind, "fields": _log_int(rng, 4, 64),
                "edges": ",".join(str(_log_int(rng, 32, 256)) for _ in range(4))}
    e = [_log_int(rng, 48, 400) for _ in range(3)]
    return {"kind": kind, "nx": e[0], "ny": e[1], "nz": e[2],
            "ax": round(rng.uniform(5.0, e[0] / 3), 2), "ay": round(rng.uniform(5.0, e[1] / 3), 2),
            "az": round(rng.uniform(5.0, e[2] / 3), 2)}


# ---------------------------------------------------------------------------
# The plane-cube problem in 64 bits (cube [-1/2, 1/2]^3, plane n.x = d0)
# ---------------------------------------------------------------------------
def _reduced_volume(d, n1, n2, n3):
    """Volume below the plane at distance d from the corner, n1 <= n2 <= n3, 0 <= d <= (n1+n2+n3)/2."""
    n12 = n1 + n2
    i1 = torch.where(n1 > 0, 1.0 / n1, torch.zeros_like(n1))
    e2, e3 = (d - n2).clamp(min=0), (d - n3).clamp(min=0)
    mid = (3.0 * d * (d - n1) + n1 * n1 - (e2 * e2 * e2 + e3 * e3 * e3) * i1) / (6.0 * n2 * n3)
    v = torch.where(d < n1, d * d * d / (6.0 * n1 * n2 * n3), mid)
    return torch.where(d >= n12, (d - 0.5 * n12) / n3, v)


def _solve(n, V0):
    """d0 of unit normals n (3, k) and volumes V0 (k), by bisection."""
    s = n.abs().sort(dim=0).values
    n1, n2, n3 = s[0], s[1], s[2]
    half = 0.5 * (n1 + n2 + n3)
    V = torch.minimum(V0, 1.0 - V0)
    lo, hi = torch.zeros_like(half), half.clone()
    for _ in range(60):
        m = 0.5 * (lo + hi)
        below = _reduced_volume(m, n1, n2, n3) < V
        lo, hi = torch.where(below, m, lo), torch.where(below, hi, m)
    d = 0.5 * (lo + hi)
    d = torch.where(V <= 0, torch.zeros_like(d), d)
    return torch.where(V0 >= 0.5, half - d, d - half)


def _volume(n, d0):
    s = n.abs().sort(dim=0).values
    half = 0.5 * (s[0] + s[1] + s[2])
    v = _reduced_volume((half - d0.abs()).clamp(min=0), s[0], s[1], s[2])
    v = torch.where(d0.abs() >= half, torch.zeros_like(v), v)
    return torch.where(d0 > 0, 1.0 - v, v)


def _area_centroid(n, d0):
    """Area (k) and centroid (3, k) of the cut polygon: derivatives of the volume."""
    a = n.abs()
    s, order = a.sort(dim=0)
    n1, n2, n3 = s[0], s[1], s[2]
    d = 0.5 * (n1 + n2 + n3) - d0.abs()
    n12 = n1 + n2
    i1 = torch.where(n1 > 0, 1.0 / n1, torch.zeros_like(n1))
    i2 = torch.where(n2 > 0, 1.0 / n2, torch.zeros_like(n2))
    e2, e3 = (d - n2).clamp(min=0), (d - n3).clamp(min=0)
    cub = (e2 ** 3 + e3 ** 3) * i1
    N = 3 * d * (d - n1) + n1 * n1 - cub
    G = 6 * d - 3 * n1 - 3 * (e2 * e2 + e3 * e3) * i1
    c1, c5 = d < n1, d >= n12
    third = torch.full_like(d, 0.5)
    vp = torch.where(c5, 1 / n3, torch.where(c1, 0.5 * d * d * i1 * i2 / n3, G * i2 / (6 * n3)))
    k0 = torch.where(c5, third, torch.where(c1, d * i1 / 3, (3 * d - 2 * n1 - cub * i1) / G))
    k1 = torch.where(c5, third, torch.where(c1, d * i2 / 3, (N * i2 - 3 * e2 * e2 * i1) / G))
    k2 = torch.where(c5, (d - 0.5 * n12) / n3, torch.where(c1, d / (3 * n3), (N / n3 - 3 * e3 * e3 * i1) / G))
    c = torch.zeros_like(n).scatter(0, order, torch.stack([k0, k1, k2]))
    c = torch.where(d0 > 0, 0.5 - c, c - 0.5) * torch.where(n < 0, -1.0, 1.0)
    return vp * (n * n).sum(0).sqrt(), c


# ---------------------------------------------------------------------------
# Inputs: cells
# ---------------------------------------------------------------------------
def _cells(n, seed, dtype, rows=False, edges=True):
    """Normals (three arrays of n) and volumes of a batch: directions uniform on
    the sphere and V0 ~ U[0, 1]; with ``edges``, 10 % of the cells sit within 1e-6 of a
    boundary between two intersection cases and 2 % are the special cells of
    simple flows (V0 in {0, 1, 1/2}; normals along an axis, in a coordinate
    plane, along a diagonal).  ``rows``: the normals are the rows of one tensor."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    if rows:
        nn = torch.empty(3, n, dtype=dtype, device=DEV)
        nx, ny, nz = nn[0], nn[1], nn[2]
    else:
        nx, ny, nz = (torch.empty(n, dtype=dtype, device=DEV) for _ in range(3))
    V0 = torch.empty(n, dtype=dtype, device=DEV)
    for a in range(0, n, CHUNK):
        k = min(CHUNK, n - a)
        v = torch.randn(3, k, dtype=F64, device=DEV, generator=g)
        f = torch.rand(k, dtype=F64, device=DEV, generator=g)
        if edges:
            u = torch.rand(k, dtype=F64, device=DEV, generator=g)
            which = torch.randint(0, 5, (k,), device=DEV, generator=g)
            axis = torch.randint(0, 3, (k,), device=DEV, generator=g)
            keep = torch.arange(3, device=DEV)[:, None] == axis
            special = u < 0.02
            v = torch.where((special & ((which == 1) | (which == 3))) & ~keep, torch.zeros_like(v), v)
            v = torch.where((special & (which == 2)) & keep, torch.zeros_like(v), v)
            v = torch.where(special & (which == 4), v.sign(), v)
            ends = (special & (which == 0)) | (special & (which == 3) & (f < 0.4))
            f = torch.where(ends, torch.tensor([0.0, 1.0, 0.5], dtype=F64, device=DEV)[axis], f)
        v = v / (v * v).sum(0).sqrt()
        if edges:
            s = v.abs().sort(dim=0).values
            near = (u >= 0.02) & (u < 0.12)
            upper = (which & 1) == 1
            d = torch.where(upper, torch.minimum(s[2], s[0] + s[1]), s[1])
            d = torch.minimum(d, 0.5 * (s[0] + s[1] + s[2]))
            vb = _reduced_volume(d, s[0], s[1], s[2]) + (f - 0.5) * 2e-6
            vb = vb.clamp(0.0, 0.5)
            f = torch.where(near, torch.where(axis == 0, 1.0 - vb, vb), f)
        else:
            f = f.clamp(2e-4, 1 - 2e-4)
        nx[a:a + k], ny[a:a + k], nz[a:a + k] = v[0].to(dtype), v[1].to(dtype), v[2].to(dtype)
        V0[a:a + k] = f.to(dtype)
    return nx, ny, nz, V0


# ---------------------------------------------------------------------------
# Inputs: fill fields
# ---------------------------------------------------------------------------
def _add_ellipsoid(phi, c, semi):
    """Union of the field with an ellipsoid: each cell's fraction below the
    tangent plane of the level set through its centre (fractions under 1e-5 cut)."""
    nz, ny, nx = phi.shape
    lo = [max(0, int(ck - ak) - 2) for ck, ak in zip(c, semi)]
    hi = [min(e, int(ck + ak) + 4) for ck, ak, e in zip(c, semi, (nx, ny, nz))]
    if any(h <= l for l, h in zip(lo, hi)):
        return
    x, y, z = (torch.arange(l, h, dtype=F64, device=DEV) - ck for l, h, ck in zip(lo, hi, c))
    g = [x[None, None, :] / semi[0] ** 2, y[None, :, None] / semi[1] ** 2, z[:, None, None] / semi[2] ** 2]
    f = (g[0] * x[None, None, :] + g[1] * y[None, :, None] + g[2] * z[:, None, None]).sqrt().clamp(min=1e-3)
    gl = (g[0] ** 2 + g[1] ** 2 + g[2] ** 2).sqrt().clamp(min=1e-9) / f
    dist = (1 - f) / gl                                # signed distance to the tangent plane, > 0 inside
    sub = phi[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
    sub[dist > 0.9] = 1.0
    at = (dist.abs() <= 0.9).nonzero(as_tuple=True)
    n = torch.stack([(gk.expand_as(f)[at] / (f[at] * gl[at])) for gk in g])
    v = _volume(n / (n * n).sum(0).sqrt(), dist[at]).to(torch.float32)
    v = torch.where(v < 1e-5, torch.zeros_like(v), torch.where(v > 1 - 1e-5, torch.ones_like(v), v))
    sub[at] = torch.maximum(sub[at], v)


def _droplets(shape, drops, rmin, rmax, g, inside=True):
    """A (nz, ny, nx) field of spherical droplets, R ~ U[rmin, rmax], four cells or
    more apart (one that finds no room in 30 tries is left out: surface tension merges droplets that touch)."""
    nz, ny, nx = shape
    phi = torch.zeros(shape, dtype=torch.float32, device=DEV)
    placed = []
    for tries in torch.rand(drops, 30, 4, dtype=F64, generator=g).tolist():
        for ux, uy, uz, ur in tries:
            r = min(rmin + (rmax - rmin) * ur, min(shape) / 2 - 3)
            m = r + 2 if inside else 0.0
            c = [m + t * (e - 1 - 2 * m) for t, e in zip((ux, uy, uz), (nx, ny, nz))]
            if all(math.dist(c, q[:3]) > r + q[3] + 4 for q in placed):
                placed.append((*c, r))
                _add_ellipsoid(phi, c, (r, r, r))
                break
    return phi


def _interface(phi):
    """Ascending linear indices of the interior cells with 0 < phi < 1 (int32)."""
    m = (phi > 0) & (phi < 1)
    m[0], m[-1] = False, False
    m[:, 0], m[:, -1] = False, False
    m[:, :, 0], m[:, :, -1] = False, False
    return m.view(-1).nonzero().squeeze(1).to(torch.int32)


def _capacity(case):
    """List entries that a program holds for these droplets: 1.6 cells per unit of the largest area."""
    cells = case["nx"] * case["ny"] * case["nz"]
    return min(cells, int(case["drops"] * 1.6 * 4 * math.pi * case["rmax"] ** 2) + 1024)


def _batch_capacity(case):
    return 160_000 * case["fields"] + 600_000


def _field(case, seed):
    g = torch.Generator().manual_seed(int(seed))
    return _droplets((case["nz"], case["ny"], case["nx"]), case["drops"], case["rmin"], case["rmax"], g)


def _fields(case, seed):
    """The batch: cubic fields with edges drawn from the list, 1 to 20 droplets of
    radius 4 to 40 each, anywhere (some clipped by the boundary)."""
    g = torch.Generator().manual_seed(int(seed))
    edges = [int(e) for e in case["edges"].split(",")]
    out = []
    for _ in range(case["fields"]):
        e = edges[int(torch.randint(0, len(edges), (1,), generator=g))]
        k = int(torch.randint(1, 21, (1,), generator=g))
        out.append(_droplets((e, e, e), k, 4.0, 40.0, g, inside=False))
    return out


def _grad_field(case, seed):
    """One ellipsoid with 1e-3 noise on its interface cells (the set of cells stays that of the
    ellipsoid), and the weight of each cell's curvature."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    phi = torch.zeros(case["nz"], case["ny"], case["nx"], dtype=torch.float32, device=DEV)
    c = [0.5 * e + t for e, t in zip((case["nx"], case["ny"], case["nz"]), (0.31, -0.17, 0.07))]
    _add_ellipsoid(phi, c, (case["ax"], case["ay"], case["az"]))
    m = (phi > 0) & (phi < 1)
    noise = 1e-3 * torch.randn(phi.shape, device=DEV, generator=g)
    phi = torch.where(m, (phi + noise).clamp(2e-4, 1 - 2e-4), phi)
    idx = _interface(phi)
    w = torch.randn(idx.numel(), device=DEV, generator=g)
    return phi, idx, w


# ---------------------------------------------------------------------------
# What a program has in hand, and one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    """Inputs and the buffers that a program keeps over its steps."""
    kind = case["kind"]
    s = dict(case)
    if kind in ("offset", "roundtrip"):
        s["in"] = _cells(case["n"], seed, DTYPES[case["precision"]], rows=case.get("rows", False))
        s["out"] = [torch.zeros_like(s["in"][3]) for _ in range(1 if kind == "offset" else 2)]
    elif kind == "offset_grad":
        s["in"] = [t.requires_grad_() for t in _cells(case["n"], seed, DTYPES[case["dtype"]], edges=False)]
        g = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
        s["g"] = torch.randn(case["n"], dtype=DTYPES[case["dtype"]], device=DEV, generator=g)
    elif kind == "field":
        # a simulation keeps its list, count, scratch and result buffers, with
        # room for a growing interface
        s["phi"] = _field(case, seed)
        cap = _capacity(case)
        s["idx"] = torch.zeros(cap, dtype=torch.int32, device=DEV)
        s["count"] = torch.zeros(1, dtype=torch.int64, device=DEV)
        s["kappa"] = torch.zeros(cap, dtype=torch.float32, device=DEV)
        s["ws"] = torch.empty(plic.workspace_bytes(plic.WS_COMPACT, s["phi"].numel()), dtype=torch.uint8,
                              device=DEV)
    elif kind == "batched":
        fields = _fields(case, seed)
        lists = [_interface(p) for p in fields]
        s["kappa"] = torch.zeros(_batch_capacity(case), dtype=torch.float32, device=DEV)
        rows = []
        at = 0
        for p, i in zip(fields, lists):
            rows.append((p, i, i.numel(), s["kappa"][at:at + i.numel()]))
            at += i.numel()
        s["batch"] = plic.BatchedFields(rows)
    else:
        phi, s["idx"], s["w"] = _grad_field(case, seed)
        s["phi"] = phi.requires_grad_()
    return s


def run(s):
    """One pass through the public entry points."""
    kind = s["kind"]
    if kind == "offset":
        return plic.offset(*s["in"], method=s["method"], precision=s["precision"], out=s["out"][0])
    if kind == "roundtrip":
        return plic.offset_roundtrip(*s["in"], method=s["method"], precision=s["precision"], out=s["out"][0],
                                     out_rt=s["out"][1])
    if kind == "offset_grad":
        d0 = autograd.offset(*s["in"])
        return (d0.detach(),) + torch.autograd.grad(d0, s["in"], s["g"])
    if kind == "field":
        plic.interface_compact(s["phi"], idx=s["idx"], count=s["count"], workspace=s["ws"])
        plic.curvature(s["phi"], s["idx"], count=s["count"], kappa=s["kappa"])
        return s["idx"], s["count"], s["kappa"]
    if kind == "batched":
        plic.curvature_batched(s["batch"])
        return s["kappa"]
    kappa = autograd.curvature(s["phi"], s["idx"])
    return kappa.detach(), torch.autograd.grad(kappa, s["phi"], s["w"])[0]


def work(case):
    """Bytes and operations that one pass cannot do without.  Operations per
    cell: 80 for an inversion, 25 for a forward volume, 50 for an adjoint,
    1571 for the curvature of one cell (13 neighbours), three times that for
    its reverse pass; interface cells of a droplet: 1.5 per unit of its area
    (a third of a batch's droplets find room and lie inside their field)."""
    kind = case["kind"]
    area = lambda r0, r1: 4 * math.pi * (r0 * r0 + r0 * r1 + r1 * r1) / 3 * 1.5  # noqa: E731
    if kind in ("offset", "roundtrip"):
        e, k = (8 if case["precision"].startswith("fp64") else 4), (5 if kind == "offset" else 6)
        return {"bytes": k * e * case["n"], "flops": (80 if kind == "offset" else 105) * case["n"]}
    if kind == "offset_grad":
        e = 8 if case["dtype"] == "fp64" else 4
        return {"bytes": (5 + 9) * e * case["n"], "flops": 130 * case["n"]}
    if kind == "field":
        cells = case["nx"] * case["ny"] * case["nz"]
        k = case["drops"] * area(case["rmin"], case["rmax"])
        return {"bytes": 4 * cells + 8 * k, "flops": 1571 * k + cells}
    if kind == "batched":
        edges = [int(e) for e in case["edges"].split(",")]
        k = case["fields"] * min(10.5 * 0.35 * area(4.0, 40.0), 1.5 * sum(e ** 3 for e in edges) / len(edges) / 20)
        return {"bytes": 12 * k, "flops": 1571 * k}
    cells = case["nx"] * case["ny"] * case["nz"]
    k = 1.5 * 4 * math.pi * ((case["ax"] * case["ay"]) ** 1.6 / 3 + (case["ax"] * case["az"]) ** 1.6 / 3
                             + (case["ay"] * case["az"]) ** 1.6 / 3) ** (1 / 1.6)
    return {"bytes": 4 * cells + 24 * k, "flops": 4 * 1571 * k}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
# the 26 neighbours, in the D3Q27 order of the paper's Appendix B
_E = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, -1), (0, 1, 1), (0, -1, -1),
      (1, -1, 0), (-1, 1, 0), (1, 0, -1), (-1, 0, 1), (0, 1, -1), (0, -1, 1),
      (1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]


def _unit(v):
    return v / (v * v).sum(0).sqrt()


def _curvature(phi, shape, idx):
    """Mean curvature of the listed cells (positive for a convex fluid region):
    Parker-Youngs normal, plane offsets with the centre's normal, paraboloid
    fit, reduced where a pivot falls to 1e-6 of the trace.  ``phi`` flat, 64 bits;
    differentiable in phi (the interface set held fixed)."""
    nz, ny, nx = shape
    e = torch.tensor(_E, dtype=F64, device=DEV)
    w = torch.tensor([{1: 4.0, 2: 2.0, 3: 1.0}[sum(t * t for t in v)] for v in _E], dtype=F64, device=DEV)
    off = torch.tensor([v[0] + nx * (v[1] + ny * v[2]) for v in _E], device=DEV)
    c = idx.to(torch.int64)
    p0, p = phi[c], phi[c[:, None] + off]                              # (k), (k, 26)
    g = torch.einsum("j,jd,kj->dk", w, e, p)
    good = (g * g).sum(0) > 0
    g = torch.where(good, g, torch.ones_like(g))
    n = -_unit(g)
    r = torch.tensor([0.562709, 0.32704452, 0.75921047], dtype=F64, device=DEV)[:, None].expand_as(n)
    by = _unit(torch.linalg.cross(n, r, dim=0))
    bx = torch.linalg.cross(by, n, dim=0)
    here = (p > 0) & (p < 1)

    def offsets(nn, v):
        """d0 with its derivatives 1/A and c (implicit function theorem)."""
        with torch.no_grad():
            d = _solve(nn.detach(), v.detach())
            A, cc = _area_centroid(nn.detach(), d)
        if not torch.is_grad_enabled():
            return d
        return d + (v - v.detach()) / A + (cc * (nn - nn.detach())).sum(0)

    k = c.numel()
    d00 = offsets(n, p0)
    safe = torch.where(here, p, torch.full_like(p, 0.5)).T.reshape(-1)  # (26 k), neighbour-major
    di = offsets(n.repeat(1, 26), safe).view(26, k)
    x, y = e @ bx, e @ by                                              # (26, k)
    z = e @ n + di - d00
    m = here.T.to(F64)
    Q = torch.stack([x * x, y * y, x * y, x, y]) * m                   # (5, 26, k)
    M = torch.einsum("ajk,bjk->kab", Q, Q)
    b = torch.einsum("ajk,jk->ka", Q, z)
    # elimination with the dimension cut at the first pivot <= 1e-6 trace
    tol = 1e-6 * M.diagonal(dim1=1, dim2=2).sum(1)
    dim = here.sum(1).clamp(max=5)
    L, D = [[None] * 5 for _ in range(5)], []
    for j in range(5):
        dj = M[:, j, j] - sum((L[j][q] ** 2 * D[q] for q in range(j)), torch.zeros_like(tol))
        dim = torch.where((dim > j) & ~(dj > tol), torch.full_like(dim, j), dim)
        dj = torch.where(dim > j, dj, torch.ones_like(dj))
        D.append(dj)
        for i in range(j + 1, 5):
            L[i][j] = (M[:, i, j] - sum((L[i][q] * L[j][q] * D[q] for q in range(j)), torch.zeros_like(tol))) / dj
    t = []
    for i in range(5):
        v = b[:, i] - sum((L[i][q] * t[q] for q in range(i)), torch.zeros_like(tol))
        t.append(torch.where(dim > i, v, torch.zeros_like(v)))
    s = [None] * 5
    for i in reversed(range(5)):
        v = t[i] / D[i] - sum((L[q][i] * s[q] for q in range(i + 1, 5)), torch.zeros_like(tol))
        s[i] = torch.where(dim > i, v, torch.zeros_like(v))
    A, B, C, H, I = s
    kap = -(A * (I * I + 1) + B * (H * H + 1) - C * H * I) / (H * H + I * I + 1) ** 1.5
    return torch.where(good, kap, torch.zeros_like(kap))


def _curvature_list(phi, idx):
    flat = phi.reshape(-1).to(F64) if phi.numel() < 1 << 27 else phi.reshape(-1)
    out = torch.empty(idx.numel(), dtype=F64, device=DEV)
    with torch.no_grad():
        for a in range(0, idx.numel(), 1 << 18):
            part = idx[a:a + (1 << 18)]
            if flat.dtype == F64:
                out[a:a + part.numel()] = _curvature(flat, phi.shape, part)
            else:                                       # a window of a very large field
                plane = phi.shape[1] * phi.shape[2]
                z0, z1 = int(part[0]) // plane - 1, int(part[-1]) // plane + 2
                win = flat[z0 * plane:z1 * plane].to(F64)
                out[a:a + part.numel()] = _curvature(win, (z1 - z0,) + tuple(phi.shape[1:]),
                                                     part.to(torch.int64) - z0 * plane)
    return out


def exact(case, seed):
    """What run() returns for these inputs, in 64 bits; None for the lists and counts."""
    kind = case["kind"]
    if kind in ("offset", "roundtrip"):
        nx, ny, nz, V0 = _cells(case["n"], seed, DTYPES[case["precision"]], rows=case.get("rows", False))
        out = torch.empty(case["n"], dtype=F64, device=DEV)
        for a in range(0, case["n"], CHUNK):
            k = slice(a, a + CHUNK)
            out[k] = _solve(torch.stack([nx[k], ny[k], nz[k]]).to(F64), V0[k].to(F64))
        return out if kind == "offset" else (out, V0.to(F64))
    if kind == "offset_grad":
        nx, ny, nz, V0 = _cells(case["n"], seed, DTYPES[case["dtype"]], edges=False)
        g = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
        w = torch.randn(case["n"], dtype=DTYPES[case["dtype"]], device=DEV, generator=g).to(F64)
        n = torch.stack([nx, ny, nz]).to(F64)
        d0 = _solve(n, V0.to(F64))
        A, c = _area_centroid(n, d0)
        return (d0, w * c[0], w * c[1], w * c[2], w / A)
    if kind == "field":
        phi = _field(case, seed)
        idx = _interface(phi)
        kappa = torch.zeros(_capacity(case), dtype=F64, device=DEV)
        kappa[:idx.numel()] = _curvature_list(phi, idx)
        return (None, None, kappa)
    if kind == "batched":
        kappa = torch.zeros(_batch_capacity(case), dtype=F64, device=DEV)
        at = 0
        for p in _fields(case, seed):
            k = _curvature_list(p, _interface(p))
            kappa[at:at + k.numel()] = k
            at += k.numel()
        return kappa
    phi, idx, w = _grad_field(case, seed)
    p64 = phi.to(F64).requires_grad_()
    kappa = _curvature(p64.reshape(-1), phi.shape, idx)
    return (kappa.detach(), torch.autograd.grad(kappa, p64, w.to(F64))[0])
