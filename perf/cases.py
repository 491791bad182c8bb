"""The work this framework does for its users, as a list of measured cases.

Every case is one pass through the public entry points: the densities of a
hierarchy handed over and the hierarchy solved, potentials and forces of every
level written to the caller's arrays (``mg_set_density`` + ``mg_solve``, or
``mg_box_set_density`` + ``mg_box_solve`` + ``mg_box_forces``), or one forward
pass or training step of the learned-guess network.  ``prepare`` builds what a
program keeps between passes: the inputs, the handle and the output arrays.

The densities are sums of compact polynomial spheres (disks in 2D) with
seeded centres, radii and masses, the outer boundary their closed-form
potential, as in the repository's benchmark; ``exact`` solves the same
discrete problem directly (sine transforms) in 64 bits.
"""
import math
import random

import numpy as np
import torch

from paper_2001_02327_gb300 import mg
from paper_2001_02327_gb300 import unet as U

TOL = 1e-10
MAX_CYCLES = 60
DEV = "cuda"
F64 = torch.float64


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def listed():
    return [
        # the smallest calls: a coarse 3D hierarchy solved with the paper's default options inside a larger
        # program's time step; launches and latency count
        nest("3d_3x16_fp64", 3, [16, 16, 16], "fp64", 2, 1, 2),
        # a 2D disk problem at the resolution of the repository's 2D workload
        nest("2d_3x64_fp64", 2, [64, 64, 64], "fp64", 2, 2, 1),
        # 2D at the largest resolution of the paper's tables, four levels
        nest("2d_4x1024_fp64", 2, [1024] * 4, "fp64", 2, 1, 3),
        # the benchmark workload, plain and mixed precision
        nest("3d_4x64_fp64", 3, [64] * 4, "fp64", 2, 2, 1),
        nest("3d_4x64_mixed", 3, [64] * 4, "mixed", 2, 2, 1, inner_max=8),
        # levels of different sizes, none a power of two, in plain FP64
        nest("3d_ragged_fp64", 3, [131, 114, 98], "fp64", 2, 1, 4),
        # the large workload: four levels of 256^3, DRAM-resident
        nest("3d_4x256_mixed", 3, [256] * 4, "mixed", 2, 2, 8, inner_max=8),
        # many small independent hierarchies in one call
        batch("batch_256_small", 256, "16,24,32", 7),
        # an uneven batch of middle-sized hierarchies
        batch("batch_32_uneven", 32, "32,48,64,96,128", 11),
        # non-cubic patches
        box("box_512x256x256_mixed", 3, "512x256x256", 3, "mixed", 2, 2, 1, inner_max=8),
        # the learned guess: inference and training on a batch of 64^3 samples
        net("unet_forward_4x64", "forward", 4, 64),
        net("unet_train_4x64", "train", 4, 64),
    ]


def nest(name, dim, edges, precision, nu_pre, nu_post, sources, inner_max=0):
    return {"name": name, "kind": "nest", "dim": dim, "edges": ",".join(map(str, edges)), "precision": precision,
            "nu_pre": nu_pre, "nu_post": nu_post, "sources": sources, "inner_max": inner_max}


def batch(name, count, edges, pick):
    return {"name": name, "kind": "batch", "count": count, "edges": edges, "pick": pick}


def box(name, dim, cells, levels, precision, nu_pre, nu_post, sources, inner_max=0):
    return {"name": name, "kind": "box", "dim": dim, "cells": cells, "levels": levels, "precision": precision,
            "nu_pre": nu_pre, "nu_post": nu_post, "sources": sources, "inner_max": inner_max}


def net(name, kind, samples, edge):
    return {"name": name, "kind": kind, "samples": samples, "edge": edge}


def log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the ranges above: 2D edges 32..1024, 3D edges 16..224,
    2 to 4 levels of equal or different edges, both precisions, the benchmark's
    and the paper's sweep counts, fixed and adaptive correction steps."""
    kind = rng.choice(["nest2", "nest3", "nest3", "nest3", "batch", "box", "net"])
    precision = rng.choice(["fp64", "mixed"])
    nu_post = rng.choice([1, 2])
    inner_max = rng.choice([0, 8]) if precision == "mixed" else 0
    if kind in ("nest2", "nest3"):
        dim = 2 if kind == "nest2" else 3
        levels = rng.randint(2, 4)
        top = 1024 if dim == 2 else 224 if precision == "mixed" else 160
        n0 = int(log_uniform(rng, 32 if dim == 2 else 16, top))
        edges = [n0]
        for _ in range(1, levels):
            edges.append(n0 // 2 * 2 if rng.random() < 0.5 else max(8, int(edges[-1] * rng.uniform(0.7, 1.2)) // 2 * 2))
        edges = [min(e, top) for e in edges]
        c = nest("", dim, edges, precision, 2, nu_post, rng.randint(1, 8), inner_max)
    elif kind == "batch":
        if rng.random() < 0.5:
            c = batch("", int(log_uniform(rng, 32, 320)), "16,24,32", rng.randrange(10 ** 6))
        else:
            c = batch("", int(log_uniform(rng, 4, 24)), "32,48,64,96,128", rng.randrange(10 ** 6))
    elif kind == "box":
        cells = "x".join(str(int(log_uniform(rng, 24, top)) // 2 * 2) for top in (384, 224, 224))
        c = box("", 3, cells, rng.randint(2, 3), precision, 2, nu_post, rng.randint(1, 4), inner_max)
    else:
        c = net("", rng.choice(["forward", "train"]), rng.randint(1, 4), rng.choice([16, 32, 64]))
        c["pick"] = rng.randrange(10 ** 6)   # tells two draws of one size apart
    del c["name"]
    return c


# --------------------------------------------------------------------------
# geometry: patches of n_a cells per axis, cells of one size per level, each
# patch inside its parent at a whole number of parent cells
# --------------------------------------------------------------------------
class Geometry:
    def __init__(self, dim, cells):
        self.dim, self.n = dim, [tuple(c) for c in cells]
        self.h = [2.0 / max(self.n[0]) / 2 ** l for l in range(len(cells))]
        self.lo, self.off = [], [None]
        self.lo.append([-0.5 * na * self.h[0] for na in self.n[0]])
        for l in range(1, len(cells)):
            o = [(p - c // 2) // 2 for p, c in zip(self.n[l - 1], self.n[l])]
            self.off.append(o)
            self.lo.append([x + oa * self.h[l - 1] for x, oa in zip(self.lo[l - 1], o)])

    @property
    def levels(self):
        return len(self.n)

    def zones(self, l):
        return math.prod(self.n[l])

    def axis(self, l, a, pad):
        i = torch.arange(-pad, self.n[l][a] + pad, dtype=F64, device=DEV)
        return self.lo[l][a] + (i + 0.5) * self.h[l]

    def finest_centre(self):
        l = self.levels - 1
        return [x + 0.5 * n * self.h[l] for x, n in zip(self.lo[l], self.n[l])]

    def finest_half(self):
        l = self.levels - 1
        return 0.5 * min(self.n[l]) * self.h[l]


def batch_geometries(case):
    """Two to four levels, edges drawn from the list (a centred child needs
    an even gap of at least two parent cells)."""
    rng = random.Random(case["pick"])
    edges = [int(e) for e in case["edges"].split(",")]
    out = []
    for _ in range(case["count"]):
        levels = rng.randint(2, 4)
        while True:
            ns = [rng.choice(edges) for _ in range(levels)]
            if all((ns[l - 1] - ns[l] // 2) % 2 == 0 and ns[l - 1] - ns[l] // 2 >= 2 for l in range(1, levels)):
                break
        out.append(Geometry(3, [(n,) * 3 for n in ns]))
    return out


def geometries(case):
    if case["kind"] == "batch":
        return batch_geometries(case)
    if case["kind"] == "box":
        cells = tuple(int(v) for v in case["cells"].split("x"))
        return [Geometry(case["dim"], [cells] * case["levels"])]
    return [Geometry(case["dim"], [(int(n),) * case["dim"] for n in case["edges"].split(",")])]


# --------------------------------------------------------------------------
# densities and closed-form potentials (G = 1)
# --------------------------------------------------------------------------
def sources_of(geo, count, rng):
    """Spheres (3D, (1 - r^2/R^2)^3) or disks (2D, (1 - r^2/R^2)^4) with
    centres in the finest patch and masses U[0.5, 2]: (centre, R, rho0, m, mass)."""
    width = 0.5 * min(geo.n[0]) * geo.h[0]
    c0, w = geo.finest_centre(), min(0.4 * width, geo.finest_half())
    out = []
    for _ in range(count):
        c = [x + rng.uniform(-w, w) for x in c0]
        if geo.dim == 3:
            R, m = rng.uniform(0.04, 0.2) * width, 3
            factor = 4 * math.pi * R ** 3 * sum(math.comb(m, j) * (-1) ** j / (2 * j + 3) for j in range(m + 1))
        else:
            R, m = rng.uniform(0.1, 0.5) * width, 4
            factor = R ** 2 / (2 * (m + 1))
        mass = rng.uniform(0.5, 2.0)
        out.append((c, R, mass / factor, m, mass))
    return out


def r2_of(axes, c):
    """Squared distances over the grid of the axes (x, y[, z]); C order, x fastest."""
    dim = len(axes)
    r2 = 0.0
    for a, ax in enumerate(axes):
        shape = [1] * dim
        shape[dim - 1 - a] = -1
        r2 = r2 + ((ax - c[a]) ** 2).reshape(shape)
    return r2


def density(axes, sources):
    rho = 0.0
    for c, R, rho0, m, _ in sources:
        rho = rho + rho0 * (1.0 - r2_of(axes, c) / R ** 2).clamp_min(0.0) ** m
    return rho.contiguous()


def potential(axes, sources):
    """Closed form inside and outside the sources."""
    phi = 0.0
    for c, R, rho0, m, mass in sources:
        r2 = r2_of(axes, c)
        if len(axes) == 3:
            v = (r2 / R ** 2).clamp_max(1.0)
            s = sum(math.comb(m, j) * (-1) ** j * v ** (j + 1) / (2 * j + 3) for j in range(m + 1))
            inside = -4 * math.pi * rho0 * R ** 2 * (s + (1 - v) ** (m + 1) / (2 * (m + 1)))
            phi = phi + torch.where(r2 < R * R, inside, -mass / r2.clamp_min(1e-300).sqrt())
        else:   # only evaluated outside the disks (the outer boundary)
            phi = phi + 2 * math.pi * mass * torch.log(r2.clamp_min(1e-300))
    return phi.contiguous()


def inputs_of(geo, sources):
    """rho of every level, and the base's density and potential with one and two rings."""
    ax = lambda l, pad: [geo.axis(l, a, pad) for a in range(geo.dim)]
    rho = [density(ax(l, 0), sources) for l in range(geo.levels)]
    return rho, density(ax(0, 1), sources), potential(ax(0, 2), sources)


def problem(case, seed):
    """[(geometry, rho per level, bc_rho, bc_phi)] of a solver case."""
    rng = random.Random(seed)
    out = []
    for geo in geometries(case):
        count = case["sources"] if "sources" in case else rng.randint(1, 4)
        out.append((geo, *inputs_of(geo, sources_of(geo, count, rng))))
    return out


def output_layout(geos):
    """Offsets of every level's potential and force in two flat arrays, each slot 256-byte aligned."""
    up = lambda v: -(-v // 32) * 32
    pos, p, f = [], 0, 0
    for geo in geos:
        for l in range(geo.levels):
            z = geo.zones(l)
            pos.append((p, f))
            p, f = p + up(z), f + up(geo.dim * z)
    return pos, p, f


# --------------------------------------------------------------------------
# prepare and run
# --------------------------------------------------------------------------
class Solver:
    """A hierarchy (or batch) handle with its inputs and registered outputs."""

    def __init__(self, case, seed):
        self.problems = problem(case, seed)
        geos = [p[0] for p in self.problems]
        descs = [self.desc(g) for g in geos]
        mixed = case.get("precision", "mixed") == "mixed"
        opt = mg.options(nu_pre=case.get("nu_pre", 2), nu_post=case.get("nu_post", 2), max_cycles=MAX_CYCLES,
                         rel_tol=TOL, precision=mg.MG_MIXED if mixed else mg.MG_FP64, inner_cycles=3,
                         inner_max=case.get("inner_max", 8))
        self.handle = mg.mg_create_hierarchy(descs, opt)
        pos, np_, nf = output_layout(geos)
        self.phi = torch.zeros(np_, dtype=F64, device=DEV)
        self.force = torch.zeros(nf, dtype=F64, device=DEV)
        it = iter(pos)
        for b, geo in enumerate(geos):
            for l in range(geo.levels):
                p, f = next(it)
                z = geo.zones(l)
                mg.mg_set_outputs(self.handle, b, l, self.phi[p:p + z], self.force[f:f + geo.dim * z])

    @staticmethod
    def desc(geo):
        d = mg.mg_hierarchy_desc()
        d.dim, d.num_levels, d.h0, d.G = geo.dim, geo.levels, geo.h[0], 1.0
        for l in range(geo.levels):
            d.n[l] = geo.n[l][0]
            for a in range(geo.dim):
                d.lo[l][a] = geo.lo[l][a]
        return d

    def step(self):
        for b, (geo, rho, bc_rho, bc_phi) in enumerate(self.problems):
            mg.mg_set_density(self.handle, b, 0, rho[0], bc_rho, bc_phi)
            for l in range(1, geo.levels):
                mg.mg_set_density(self.handle, b, l, rho[l])
        mg.mg_solve(self.handle, len(self.problems))
        return {"phi": self.phi, "force": self.force}

    def __del__(self):
        if getattr(self, "handle", None):
            mg.mg_destroy(self.handle)


class BoxSolver:
    """A hierarchy of box patches with its inputs and output arrays."""

    def __init__(self, case, seed):
        (self.geo, self.rho, self.bc_rho, self.bc_phi), = problem(case, seed)
        geo = self.geo
        d = mg.mg_box_desc()
        d.dim, d.num_patches, d.h0, d.G = geo.dim, geo.levels, geo.h[0], 1.0
        for l in range(geo.levels):
            for a in range(geo.dim):
                d.n[l][a] = geo.n[l][a]
                d.lo[l][a] = geo.lo[l][a]
        mixed = case["precision"] == "mixed"
        opt = mg.options(nu_pre=case["nu_pre"], nu_post=case["nu_post"], max_cycles=MAX_CYCLES, rel_tol=TOL,
                         precision=mg.MG_MIXED if mixed else mg.MG_FP64, inner_cycles=3, inner_max=case["inner_max"])
        self.handle = mg.mg_box_create(d, opt)
        self.pos, np_, nf = output_layout([geo])
        self.phi = torch.zeros(np_, dtype=F64, device=DEV)
        self.force = torch.zeros(nf, dtype=F64, device=DEV)

    def step(self):
        geo = self.geo
        mg.mg_box_set_density(self.handle, 0, self.rho[0], self.bc_rho, self.bc_phi)
        for l in range(1, geo.levels):
            mg.mg_box_set_density(self.handle, l, self.rho[l])
        mg.mg_box_solve(self.handle, geo.levels)
        for l, (p, f) in enumerate(self.pos):
            z = geo.zones(l)
            mg.mg_box_forces(self.handle, l, self.phi[p:p + z], self.force[f:f + geo.dim * z])
        return {"phi": self.phi, "force": self.force}

    def __del__(self):
        if getattr(self, "handle", None):
            mg.mg_box_destroy(self.handle)


CONVS = [(3, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (128, 32), (64, 16), (32, 16)]
CONV_SCALE = [1, 1, 2, 2, 4, 8, 4, 2, 1]


def net_params(seed):
    """Uniform, fan-in scaled parameters in the network's flat layout (per
    convolution [27][Cin][Cout] weights and biases, then the 1x1x1 output)."""
    rng = np.random.default_rng(seed)
    parts = []
    for cin, cout in CONVS:
        b = math.sqrt(3.0 / (27 * cin))
        parts += [rng.uniform(-b, b, 27 * cin * cout) * math.sqrt(2.0), rng.uniform(-b, b, cout)]
    parts += [rng.uniform(-0.25, 0.25, 16), rng.uniform(-0.1, 0.1, 1)]
    return np.concatenate(parts).astype(np.float32)


def net_samples(case, seed):
    """Densities of refinement-level patches, the true potential, its trilinear
    interpolation from cells twice the size (the guess the network corrects)
    and the h^2-scaled residual of that guess."""
    B, n = case["samples"], case["edge"]
    rng = random.Random(seed)
    rho, guess, resid, true = [], [], [], []
    geo = Geometry(3, [(n,) * 3])
    h = geo.h[0]
    for _ in range(B):
        src = sources_of(geo, rng.randint(1, 8), rng)
        fine = [geo.axis(0, a, 1) for a in range(3)]
        coarse = [geo.lo[0][a] + (torch.arange(-2, n // 2 + 2, dtype=F64, device=DEV) + 0.5) * 2 * h for a in range(3)]
        up = torch.nn.functional.interpolate(potential(coarse, src)[None, None], scale_factor=2, mode="trilinear",
                                             align_corners=False)[0, 0]
        g = up[3:3 + n + 2, 3:3 + n + 2, 3:3 + n + 2]      # one ring around the patch
        r = density(fine, src)
        c = g[1:-1, 1:-1, 1:-1]
        lap = (g[:-2, 1:-1, 1:-1] + g[2:, 1:-1, 1:-1] + g[1:-1, :-2, 1:-1] + g[1:-1, 2:, 1:-1]
               + g[1:-1, 1:-1, :-2] + g[1:-1, 1:-1, 2:]) - 6.0 * c
        inner = r[1:-1, 1:-1, 1:-1]
        rho.append(inner)
        guess.append(c)
        resid.append(4 * math.pi * h * h * inner - lap)
        true.append(potential([ax[1:-1] for ax in fine], src))
    return [torch.stack(v).contiguous() for v in (rho, guess, resid, true)], np.full(B, 4 * math.pi * h * h)


class Net:
    """The learned-guess network with a batch of samples."""

    def __init__(self, case, seed):
        self.case = case
        self.data, self.frho = net_samples(case, seed)
        self.net = U.mg_unet_create(case["edge"], case["samples"], seed=1)
        U.mg_unet_set_params(self.net, net_params(seed))

    def step(self):
        B, n = self.case["samples"], self.case["edge"]
        rho, guess, resid, true = self.data
        if self.case["kind"] == "forward":
            return U.mg_unet_forward(self.net, B, n, rho, guess, resid, self.frho)
        loss = U.mg_unet_train_step(self.net, B, n, rho, guess, resid, true, self.frho, lr=1e-4, wd=1e-5)
        return {"loss": loss, "grad": U.mg_unet_get_grad(self.net)}

    def __del__(self):
        if getattr(self, "net", None):
            U.mg_unet_destroy(self.net)


def prepare(case, seed):
    if case["kind"] in ("forward", "train"):
        state = Net(case, seed)
    elif case["kind"] == "box":
        state = BoxSolver(case, seed)
    else:
        state = Solver(case, seed)
    torch.cuda.synchronize()
    return state


def run(state):
    return state.step()


# --------------------------------------------------------------------------
# the least one pass has to do
# --------------------------------------------------------------------------
def work(case):
    if case["kind"] in ("forward", "train"):
        B, n = case["samples"], case["edge"]
        flops = sum(2.0 * 27 * ci * co * B * (n // d) ** 3 for (ci, co), d in zip(CONVS, CONV_SCALE))
        params = sum(27 * a * b + b for a, b in CONVS) + 17
        cells = float(B * n ** 3)
        if case["kind"] == "forward":
            return {"bytes": cells * (3 * 8 + 4) + 4 * params, "flops": flops}
        return {"bytes": cells * 4 * 8 + 4 * params * 7, "flops": 3 * flops}
    nu = case.get("nu_pre", 2) + case.get("nu_post", 2)
    total = {"bytes": 0.0, "flops": 0.0}
    for geo in geometries(case):
        d = geo.dim
        for l in range(geo.levels):
            z = float(geo.zones(l))
            ring1 = math.prod(n + 2 for n in geo.n[l]) - z
            ring2 = math.prod(n + 4 for n in geo.n[l]) - z - ring1
            total["bytes"] += 8 * z * (2 + d) + (8 * (ring1 + ring2) if l == 0 else 0)
            # ten V-cycles: sweeps, residual, transfers, on all multigrid levels; Eq. 2 forces
            per_cycle = (nu * (2 * d + 2) + 6 * d) * 2 ** d / (2 ** d - 1)
            total["flops"] += z * (10 * per_cycle + 5 * d)
    return total


# --------------------------------------------------------------------------
# exact: the discrete problem solved directly in 64 bits
# --------------------------------------------------------------------------
def along(A, M, axis):
    """M applied along one axis of A."""
    return torch.movedim(torch.tensordot(M, A, dims=([1], [axis])), 0, axis)


def poisson(rhs):
    """Solve the (2d+1)-point Laplacian (unit spacing, zero boundary) for rhs by sine transforms."""
    x = rhs
    lam = 0.0
    sines = {}
    for a, M in enumerate(rhs.shape):
        if M not in sines:
            k = torch.arange(1, M + 1, dtype=F64, device=DEV)
            sines[M] = (torch.sin(math.pi * torch.remainder(torch.outer(k, k), 2 * (M + 1)) / (M + 1)),
                        -4.0 * torch.sin(0.5 * math.pi * k / (M + 1)) ** 2)
        S, ev = sines[M]
        x = along(x, S, a)
        shape = [1] * rhs.dim()
        shape[a] = -1
        lam = lam + ev.reshape(shape)
    x = x / lam
    for a, M in enumerate(rhs.shape):
        x = along(x, sines[M][0], a) * (2.0 / (M + 1))
    return x


def from_parent(A, geo, l, pad):
    """The parent's block A (two rings) interpolated (3/4, 1/4 per axis) at the cells of level l with `pad` rings."""
    for a in range(geo.dim):
        axis = geo.dim - 1 - a
        i = torch.arange(-pad, geo.n[l][a] + pad, device=DEV)
        near = geo.off[l][a] + torch.div(i, 2, rounding_mode="floor") + 2
        far = near + torch.where(i % 2 == 0, -1, 1)
        A = 0.75 * A.index_select(axis, near) + 0.25 * A.index_select(axis, far)
    return A


def ring_only(A):
    out = A.clone()
    out[tuple(slice(1, -1) for _ in range(A.dim()))] = 0.0
    return out


def solve_exactly(geo, rho, bc_rho, bc_phi):
    """Potential and Eq. 2 force of every level on its own cells."""
    d = geo.dim
    inner = tuple(slice(1, -1) for _ in range(d))
    phi_blk = rho_blk = None
    out = []
    for l in range(geo.levels):
        if l == 0:
            ring_phi, ring_rho = bc_phi, bc_rho
        else:
            ring_phi, ring_rho = from_parent(phi_blk, geo, l, 2), from_parent(rho_blk, geo, l, 1)
        r = ring_rho.clone()
        r[inner] = rho[l]
        ring = ring_only(ring_phi)
        rhs = 4 * math.pi * geo.h[l] ** 2 * r
        for a in range(d):
            m = ring.shape[a] - 2
            for s in (0, 2):
                rhs = rhs - ring[tuple(slice(s, s + m) if b == a else slice(1, -1) for b in range(d))]
        blk = ring
        blk[inner] = poisson(rhs)
        force = []
        for a in range(d):
            axis = d - 1 - a
            n = geo.n[l][a]
            at = lambda o: blk[tuple(slice(2 + o, 2 + o + n) if b == axis else slice(2, -2) for b in range(d))]
            force.append(-(8.0 * (at(1) - at(-1)) - (at(2) - at(-2))) / (12.0 * geo.h[l]))
        out.append((blk[tuple(slice(2, -2) for _ in range(d))], torch.stack(force)))
        phi_blk = blk
        rho_blk = torch.nn.functional.pad(r, (1,) * (2 * d))
    return out


def net_exactly(case, seed):
    """The network in 64 bits (plain convolutions), and with training the loss and its gradient."""
    Fn = torch.nn.functional
    (rho, guess, resid, true), frho = net_samples(case, seed)
    p = torch.from_numpy(net_params(seed)).to(DEV).double().requires_grad_(case["kind"] == "train")
    convs, off = [], 0
    for cin, cout in CONVS:
        w = p[off:off + 27 * cin * cout].reshape(27, cin, cout).permute(2, 1, 0).reshape(cout, cin, 3, 3, 3)
        off += 27 * cin * cout
        convs.append((w, p[off:off + cout]))
        off += cout
    biggest = lambda t: t.abs().amax(dim=(1, 2, 3), keepdim=True)
    s, sr = biggest(guess), biggest(resid)
    x = torch.stack([torch.from_numpy(frho).to(DEV).reshape(-1, 1, 1, 1) * rho / s, guess / s, resid / sr], dim=1)
    conv = lambda t, i: torch.relu(Fn.conv3d(t, convs[i][0], convs[i][1], padding=1))
    pool = lambda t: Fn.avg_pool3d(t, 2)
    up = lambda t: Fn.interpolate(t, scale_factor=2, mode="nearest")
    with torch.backends.cudnn.flags(enabled=False):
        s0 = conv(conv(x, 0), 1)
        s1 = conv(conv(pool(s0), 2), 3)
        s2 = conv(pool(s1), 4)
        d2 = conv(torch.cat([up(conv(pool(s2), 5)), s2], dim=1), 6)
        d1 = conv(torch.cat([up(d2), s1], dim=1), 7)
        d0 = conv(torch.cat([up(d1), s0], dim=1), 8)
        y = torch.einsum("bczyx,c->bzyx", d0, p[off:off + 16]) + p[off + 16]
        if case["kind"] == "forward":
            return y.detach()
        n = case["edge"]
        loss = ((y - (true - guess) / (sr * (n * n / 16.0))) ** 2).mean()
        loss.backward()
    return {"loss": float(loss.detach()), "grad": p.grad}


def exact(case, seed):
    if case["kind"] in ("forward", "train"):
        return net_exactly(case, seed)
    problems = problem(case, seed)
    pos, np_, nf = output_layout([p[0] for p in problems])
    phi = torch.zeros(np_, dtype=F64, device=DEV)
    force = torch.zeros(nf, dtype=F64, device=DEV)
    it = iter(pos)
    for geo, rho, bc_rho, bc_phi in problems:
        for v, f in solve_exactly(geo, rho, bc_rho, bc_phi):
            p, q = next(it)
            phi[p:p + v.numel()] = v.reshape(-1)
            force[q:q + f.numel()] = f.reshape(-1)
    return {"phi": phi, "force": force}
