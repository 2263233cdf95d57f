"""Cases that the near-field operator is timed on.

A case is one call pattern of the package's public API (`paper_2403_01596_gb300.api`) on one seeded geometry:

  apply   out = A lam (or A^H lam) with a plan the program holds: one right-hand side (the matrix-vector product
          inside an iterative solver) or several (block solvers)
  step    the autograd step of a shape or source optimisation: A lam, the residual norm, dL/dlam and dL/dx
  setup   new geometry: leaf binning, neighbour lists, plan and the first product
  batch   a problem cut into pieces, all of them applied in one replayed launch

Geometries are drawn on the GPU from the seed: points uniform on the unit sphere, on the 2:1:1 ellipsoid, on a
square plate, in the unit cube, and on a cylinder between two plates with half of the points in clusters.  Grids
and wavenumbers are those of `workloads.py`: the leaf edge is 0.25 wavelengths on spheres and assemblies, 0.2 on
ellipsoids and 0.5 in cubes.
"""
import math

import numpy as np
import torch

from paper_2403_01596_gb300 import api

TWO_PI = 2.0 * math.pi
INV_4PI = 1.0 / (4.0 * math.pi)

#: origin and edge of the cube that holds each shape's leaf grid, and the leaf edge in wavelengths
SHAPES = {"sphere": (-1.0, 2.0, 0.25), "ellipsoid": (-2.0, 4.0, 0.2), "plate": (0.0, 1.0, 0.25),
          "cube": (0.0, 1.0, 0.5), "assembly": (-1.3, 2.6, 0.25)}


def _case(name, op, shape, n, ng, kernel="helmholtz", nrhs=1, layout="indexed", path="auto", adjoint=False, pieces=1):
    case = {"op": op, "shape": shape, "n": n, "ng": ng, "kernel": kernel, "nrhs": nrhs, "layout": layout,
            "path": path, "adjoint": adjoint, "pieces": pieces}
    return {"name": name, **case} if name else case


def listed():
    return [
        # the smallest call: one product on a small scatterer, as often as a solver iterates; launches and latency
        _case("small_sphere", "apply", "sphere", 4_099, 12),
        # one product on a large sphere at the occupancies of the benchmark's sweep (8, 32 and 64 points per box);
        # 32 in the layout that keeps every box's neighbourhood contiguous
        _case("sphere_8_per_box", "apply", "sphere", 1 << 20, 180),
        _case("sphere_32_per_box_redundant", "apply", "sphere", 1 << 20, 86, layout="redundant"),
        _case("sphere_64_per_box", "apply", "sphere", 1 << 20, 61),
        # electrostatics on the plate of the layout comparison: four points per box, real kernel
        _case("plate_laplace", "apply", "plate", 1 << 20, 512, kernel="laplace"),
        # a volume: 27 full neighbours, 64 points per box
        _case("cube_volume", "apply", "cube", 32_768, 8),
        # eight excitations of an assembly whose boxes hold 1 to ~100 points
        _case("assembly_8_rhs", "apply", "assembly", 500_000, 141, nrhs=8),
        # a block of 64 excitations on the large ellipsoid (the largest call)
        _case("ellipsoid_64_rhs", "apply", "ellipsoid", 1 << 21, 188, nrhs=64),
        # an odd block width in the accurate split, adjoint direction (block least squares)
        _case("sphere_24_rhs_adjoint", "apply", "sphere", 200_003, 54, nrhs=24, path="tc_bf16x6", adjoint=True),
        # one step of a gradient-based optimisation of strengths and positions
        _case("gradient_step", "step", "sphere", 1 << 18, 62),
        # a new geometry up to its first product
        _case("new_geometry", "setup", "sphere", 1 << 20, 86),
        # a problem cut into pieces of 65 536 points, replayed as one launch
        _case("sixteen_pieces", "batch", "sphere", 65_536, 31, pieces=16),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid_for(shape, n, per_box):
    """Boxes per axis at which occupied boxes hold about per_box points."""
    if shape == "cube":
        return max(2, round((n / per_box) ** (1.0 / 3.0)))
    if shape == "plate":
        return max(2, round(math.sqrt(n / per_box)))
    area = {"sphere": 4.0 * math.pi, "ellipsoid": 21.48, "assembly": 2.0 * math.pi + 8.0}[shape]
    # a surface cuts about 1.29 boxes per h^2 of its area; the assembly's clustered half fills few boxes
    boxes = n / per_box * (0.5 if shape == "assembly" else 1.0)
    return max(2, round(SHAPES[shape][1] * math.sqrt(boxes / (1.29 * area))))


def draw(rng):
    op = rng.choice(["apply", "apply", "apply", "block", "block", "step", "setup", "batch"])
    kernel = rng.choice(["helmholtz", "helmholtz", "laplace"])
    if op == "apply":
        shape = rng.choice(["sphere", "sphere", "ellipsoid", "plate", "cube", "assembly"])
        n = int(_log_uniform(rng, 4_000, 1_000_000)) | 1
        per_box = _log_uniform(rng, 3.0, 24.0 if shape in ("cube", "assembly") else 64.0)
        return _case(None, "apply", shape, n, _grid_for(shape, n, per_box), kernel,
                     layout=rng.choice(["indexed", "indexed", "redundant"]), adjoint=rng.random() < 0.25)
    if op == "block":
        shape = rng.choice(["sphere", "ellipsoid", "assembly"])
        nrhs = int(_log_uniform(rng, 2, 100))
        n = int(_log_uniform(rng, 8_000, 500_000)) | 1
        per_box = _log_uniform(rng, 6.0, 12.0 if shape == "assembly" else 48.0)
        return _case(None, "apply", shape, n, _grid_for(shape, n, per_box), kernel, nrhs=nrhs,
                     path=rng.choice(["auto", "auto", "tc_bf16x6"]) if nrhs >= 16 else "auto",
                     adjoint=rng.random() < 0.25)
    shape = rng.choice(["sphere", "ellipsoid"])
    per_box = _log_uniform(rng, 6.0, 48.0)
    if op == "step":
        n = int(_log_uniform(rng, 10_000, 500_000)) | 1
        return _case(None, "step", shape, n, _grid_for(shape, n, per_box), kernel)
    if op == "setup":
        n = int(_log_uniform(rng, 10_000, 1_000_000)) | 1
        return _case(None, "setup", shape, n, _grid_for(shape, n, per_box), kernel)
    n = int(_log_uniform(rng, 20_000, 150_000)) | 1
    return _case(None, "batch", shape, n, _grid_for(shape, n, per_box), kernel, pieces=rng.randint(2, 16))


# ------------------------------------------------------------------------------------------------ inputs --

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed))


def _unit_vectors(n, gen):
    v = torch.randn(n, 3, generator=gen, device=gen.device, dtype=torch.float64)
    return v / v.norm(dim=1, keepdim=True)


def _mirror(x):
    """Reflects values that leave [-1, 1] at its ends."""
    return 1.0 - (torch.remainder(x + 1.0, 4.0) - 2.0).abs()


def _points(case, gen):
    """(n, 3) float32 points of the case's shape."""
    n, shape, dev = case["n"], case["shape"], gen.device
    if shape == "sphere":
        p = _unit_vectors(n, gen)
    elif shape == "cube":
        p = torch.rand(n, 3, generator=gen, device=dev, dtype=torch.float64)
    elif shape == "plate":
        p = torch.rand(n, 3, generator=gen, device=dev, dtype=torch.float64)
        p[:, 2] = 0.5
    elif shape == "ellipsoid":
        # area-uniform: a sphere sample is kept with the ratio of the ellipsoid's area element to its largest
        parts, have = [], 0
        while have < n:
            u = _unit_vectors(int(1.5 * (n - have)) + 1024, gen)
            w = torch.sqrt(u[:, 0] ** 2 + 4.0 * (u[:, 1] ** 2 + u[:, 2] ** 2)) / 2.0
            u = u[torch.rand(u.shape[0], generator=gen, device=dev, dtype=torch.float64) < w]
            parts.append(u)
            have += u.shape[0]
        p = torch.cat(parts)[:n] * torch.tensor([2.0, 1.0, 1.0], device=dev, dtype=torch.float64)
    else:
        # cylinder of radius 0.5 between two 2 x 2 plates; half of the points in clusters of ~2000, std two leaf edges
        h = SHAPES["assembly"][1] / case["ng"]
        n_clu = n // 2
        clusters = max(1, n_clu // 2000)
        m = n - n_clu + clusters
        u = torch.rand(m, 3, generator=gen, device=dev, dtype=torch.float64)
        cyl_share = TWO_PI / (TWO_PI + 8.0)
        part = torch.where(u[:, 0] < cyl_share, 0, torch.where(u[:, 0] < 0.5 * (1.0 + cyl_share), 1, 2))
        s = torch.where(part == 0, u[:, 1] * math.pi, 2.0 * u[:, 1] - 1.0)
        t = 2.0 * u[:, 2] - 1.0
        which = torch.randint(0, clusters, (n_clu,), generator=gen, device=dev) + (n - n_clu)
        off = torch.randn(n_clu, 2, generator=gen, device=dev, dtype=torch.float64) * (2.0 * h)
        part = torch.cat([part[:n - n_clu], part[which]])
        sc = s[which] + off[:, 0]
        s = torch.cat([s[:n - n_clu], torch.where(part[n - n_clu:] == 0, torch.remainder(sc, math.pi), _mirror(sc))])
        t = torch.cat([t[:n - n_clu], _mirror(t[which] + off[:, 1])])
        cyl = part == 0
        p = torch.stack([torch.where(cyl, 0.5 * torch.cos(2.0 * s), s),
                         torch.where(cyl, 0.5 * torch.sin(2.0 * s), t),
                         torch.where(cyl, t, torch.where(part == 1, -1.25, 1.25))], dim=1)
        p = p[torch.randperm(n, generator=gen, device=dev)]
    return p.to(torch.float32).contiguous()


def _strengths(n, nrhs, gen):
    """Complex64 strengths, Re and Im i.i.d. N(0, 1): (n,) or (n, nrhs)."""
    v = torch.view_as_complex(torch.randn(n, nrhs, 2, generator=gen, device=gen.device))
    return v[:, 0].contiguous() if nrhs == 1 else v


def _grid(case):
    """Grid origin, leaf edge, boxes per axis and wavenumber."""
    lo, edge, wavelengths = SHAPES[case["shape"]]
    h = edge / case["ng"]
    return (lo, lo, lo), h, case["ng"], TWO_PI * wavelengths / h if case["kernel"] == "helmholtz" else 0.0


def _inputs(case, seed):
    """Per piece: points, strengths and (for a step) the data the product is fitted to."""
    gen = _generator(seed)
    got = []
    for _ in range(case["pieces"]):
        points = _points(case, gen)
        lam = _strengths(case["n"], case["nrhs"], gen)
        data = _strengths(case["n"], 1, gen) * 10.0 if case["op"] == "step" else None
        got.append((points, lam, data))
    return got


# --------------------------------------------------------------------------------------------------- runs --

def _plan(case, points):
    lo, h, ng, k = _grid(case)
    return api.Plan(points, lo, h, ng, k, kernel=case["kernel"], layout=case["layout"], max_nrhs=case["nrhs"])


def prepare(case, seed):
    inputs = _inputs(case, seed)
    state = {"case": case, "op": case["op"], "points": inputs[0][0], "lam": inputs[0][1]}
    if case["op"] == "apply":
        state["plan"] = _plan(case, state["points"])
    elif case["op"] == "step":
        state["plan"] = _plan(case, state["points"])
        state["points"].requires_grad_()
        state["lam"].requires_grad_()
        state["data"] = inputs[0][2]
    elif case["op"] == "batch":
        state["plans"] = [_plan(case, p) for p, _, _ in inputs]
        state["batch"] = api.Batch(state["plans"], nrhs=case["nrhs"])
        state["batch"].capture([lam for _, lam, _ in inputs])
    return state


def run(state):
    case = state["case"]
    if case["op"] == "apply":
        return state["plan"].apply(state["lam"], adjoint=case["adjoint"], path=case["path"])
    if case["op"] == "step":
        lam, points = state["lam"], state["points"]
        out = api.p2p(lam, points, state["plan"])
        loss = torch.view_as_real(out - state["data"]).square().sum()
        glam, gx = torch.autograd.grad(loss, (lam, points))
        return {"out": out, "lam_grad": glam, "points_grad": gx}
    if case["op"] == "setup":
        plan = _plan(case, state["points"])
        st = plan.structure
        return {"out": plan.apply(state["lam"]), "perm": st.perm, "point_box": st.point_box}
    return list(state["batch"].replay())


# ------------------------------------------------------------------------- the same results in 64 bits --

class _Boxes:
    """Leaf boxes of a point set in plain torch: points sorted by cell, box offsets, the 27 neighbours of a box."""

    def __init__(self, points, lo, h, ng):
        cells = torch.floor((points.double() - lo[0]) / h).clamp(0, ng - 1).long()
        key = (cells[:, 2] * ng + cells[:, 1]) * ng + cells[:, 0]
        key, self.order = torch.sort(key, stable=True)
        keys, self.count = torch.unique_consecutive(key, return_counts=True)
        self.start = torch.cumsum(self.count, 0) - self.count
        cell = torch.stack([keys % ng, (keys // ng) % ng, keys // (ng * ng)], dim=1)
        step = torch.arange(-1, 2, device=points.device)
        offset = torch.cartesian_prod(step, step, step)
        near = cell[:, None, :] + offset[None]
        ok = ((near >= 0) & (near < ng)).all(dim=2)
        want = (near[..., 2] * ng + near[..., 1]) * ng + near[..., 0]
        at = torch.searchsorted(keys, want.reshape(-1)).clamp(max=keys.numel() - 1).reshape(want.shape)
        ok &= keys[at] == want
        self.near = torch.where(ok, at, -1)
        self.near_count = torch.where(ok, self.count[at], 0)      # sources per neighbour, 0 where there is none
        self.sources = self.near_count.sum(dim=1)

    def pairs(self):
        return int((self.count * self.sources).sum().item())

    def blocks(self, most):
        """Groups of boxes as padded index blocks (targets (b, T), sources (b, S)); -1 pads."""
        by_size = torch.argsort(self.count * 1_000_000 + self.sources.clamp(max=999_999), descending=True)
        size = torch.stack([self.count[by_size], self.sources[by_size]]).cpu().numpy()
        i, total = 0, by_size.numel()
        while i < total:
            j, t, s = i, 0, 0
            while j < total:
                t2, s2 = max(t, int(size[0, j])), max(s, int(size[1, j]))
                if j > i and (j + 1 - i) * t2 * s2 > most:
                    break
                j, t, s = j + 1, t2, s2
            boxes = by_size[i:j]
            i = j
            a = torch.arange(t, device=boxes.device)
            tgt = torch.where(a[None] < self.count[boxes][:, None], self.start[boxes][:, None] + a[None], -1)
            # sources: position p of the list lies in the neighbour whose running count first exceeds p
            run_up = torch.cumsum(self.near_count[boxes], dim=1)
            p = torch.arange(s, device=boxes.device).expand(boxes.numel(), s).contiguous()
            q = torch.searchsorted(run_up, p, right=True)
            ok = q < 27
            q = q.clamp(max=26)
            first = torch.gather(run_up - self.near_count[boxes], 1, q)
            box = torch.gather(self.near[boxes], 1, q).clamp(min=0)
            src = torch.where(ok, self.start[box] + p - first, -1)
            yield tgt, src


def _distances(x, tgt, src):
    d = x[tgt.clamp(min=0)][:, :, None, :] - x[src.clamp(min=0)][:, None, :, :]
    r2 = (d * d).sum(dim=3)
    keep = (r2 > 0) & (tgt >= 0)[:, :, None] & (src >= 0)[:, None, :]
    return d, torch.sqrt(torch.where(keep, r2, 1.0)), keep


def _green(r, keep, k):
    """exp(ikr) / (4 pi r), 0 where there is no pair."""
    a = torch.where(keep, INV_4PI / r, 0.0)
    return torch.complex(a * torch.cos(k * r), a * torch.sin(k * r))


def _product(boxes, x, lam, k, adjoint=False):
    """A lam (or A^H lam) in complex128, sorted order in and out; lam (n, nrhs)."""
    out = torch.zeros_like(lam)
    for tgt, src in boxes.blocks(max(1, 24_000_000 // (1 + lam.shape[1] // 8))):
        _, r, keep = _distances(x, tgt, src)
        g = _green(r, keep, -k if adjoint else k)
        part = torch.bmm(g, lam[src.clamp(min=0)])
        out[tgt[tgt >= 0]] = part[tgt >= 0]
    return out


def _points_gradient(boxes, x, lam, g, k):
    """d/dx of Re <g, A lam> for sorted strengths and gradient (n,)."""
    out = torch.zeros_like(x)
    for tgt, src in boxes.blocks(8_000_000):
        d, r, keep = _distances(x, tgt, src)
        s, t = src.clamp(min=0), tgt.clamp(min=0)
        c = g[t].conj()[:, :, None] * lam[s][:, None, :] + g[s].conj()[:, None, :] * lam[t][:, :, None]
        slope = _green(r, keep, k) * torch.complex(-1.0 / r, torch.full_like(r, k))
        w = (slope * c).real / r
        part = (w[..., None] * d).sum(dim=2)
        out[tgt[tgt >= 0]] = part[tgt >= 0]
    return out


def _unsort(order, v):
    out = torch.empty_like(v)
    out[order] = v
    return out


def exact(case, seed):
    lo, h, ng, k = _grid(case)
    k = float(np.float32(k))
    got = []
    for points, lam, data in _inputs(case, seed):
        boxes = _Boxes(points, lo, h, ng)
        x = points.double()[boxes.order]
        lam2 = lam.reshape(case["n"], case["nrhs"]).to(torch.complex128)[boxes.order]
        out = _product(boxes, x, lam2, k, case["adjoint"])
        if case["op"] == "step":
            g = 2.0 * (out[:, 0] - data.to(torch.complex128)[boxes.order])
            glam = _product(boxes, x, g[:, None], k, adjoint=True)[:, 0]
            gx = _points_gradient(boxes, x, lam2[:, 0], g, k)
            return {"out": _unsort(boxes.order, out[:, 0]), "lam_grad": _unsort(boxes.order, glam),
                    "points_grad": _unsort(boxes.order, gx)}
        got.append(_unsort(boxes.order, out))
    if case["op"] == "batch":
        return got
    out = got[0].reshape(case["n"]) if case["nrhs"] == 1 else got[0]
    if case["op"] == "setup":
        return {"out": out, "perm": None, "point_box": None}
    return out


# --------------------------------------------------------------------------------------------------- work --

def work(case):
    """Strengths, coordinates and results once each; per pair the distance and the kernel (22 operations with sin
    and cos, 8 without) and 8 (4) per right-hand side.  A gradient step sweeps the pairs three times."""
    lo, h, ng, _ = _grid(case)
    pairs = 0
    gen = _generator(0)
    for _ in range(case["pieces"]):
        pairs += _Boxes(_points(case, gen), lo, h, ng).pairs()
    n, nrhs = case["n"] * case["pieces"], case["nrhs"]
    helm = case["kernel"] == "helmholtz"
    per_pair = (22 if helm else 8) + (8 if helm else 4) * nrhs
    rows = n * (12 + 16 * nrhs)
    if case["op"] == "step":
        return {"bytes": n * (12 + 8 * 4 + 12), "flops": pairs * (2 * per_pair + per_pair + 24)}
    return {"bytes": rows, "flops": pairs * per_pair}
