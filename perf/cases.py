"""Performance cases: the work a user of the framework has it do.

Every case goes through the public Python interface (``solver.DoctorsProblem``,
``solver.solve_batch``, ``solver.ct_to_materials``, ``autograd.RoiDose``) with
the schedule the library picks by default.  Inputs are seeded synthetic
phantoms, cross sections, spectra and beams of the shapes the method is used
on (a water cylinder, an abdomen at liver level, the paper's coarse and fine
water meshes).  ``exact`` is an independent FP64 solution in plain torch.

A case is a dict of plain values:
  kind       solve     set the beams, solve, fluence and dose out
             gradients gradients of a region-of-interest dose (adjoint) of a
                       problem that has been solved
             train     one step of an optimisation over beam weights, spectrum
                       and densities: RoiDose forward and backward
             batch     several problems in one call of solve_batch
             ct        CT numbers to materials and densities
  phantom    cube, cylinder or abdomen; nx, ny, nz voxels over fov x fov cm
             in plane (cube: 1 cm voxels), dz cm slices
  sn, legendre, groups   angular quadrature order, scattering order, energy groups
  beams      number of sources; beam = "point" (isotropic) or "fan" (collimated)
  scheme     0 step, 1 diamond differencing
"""
from __future__ import annotations

import functools
import itertools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1811_12391_gb300 import autograd, solver

TOL = 1e-6


def _problem(name, kind, phantom, nx, ny, nz, sn, legendre, groups, beams=1, beam="fan", scheme=0, fov=35.2, dz=0.5):
    return {"name": name, "kind": kind, "phantom": phantom, "nx": nx, "ny": ny, "nz": nz, "sn": sn,
            "legendre": legendre, "groups": groups, "beams": beams, "beam": beam, "scheme": scheme,
            "fov": fov, "dz": dz}


def listed():
    return [
        # the smallest solve: a 16^3 water cube with one point source, as used to try a cross-section set;
        # launches and host turnaround
        _problem("tiny_cube_s4p1", "solve", "cube", 16, 16, 16, 4, 1, 4, 1, "point", 0, 16.0, 1.0),
        # the paper's coarse water mesh, seven groups: a CT scan of 16 superposed cone beams, S6 P0
        _problem("coarse_ct_s6p0", "solve", "cylinder", 64, 64, 16, 6, 0, 7, 16, "fan", 0, 50.0, 0.78125),
        # the same mesh, single projection with anisotropic scattering, S8 P1
        _problem("coarse_s8p1", "solve", "cylinder", 64, 64, 16, 8, 1, 7, 1, "point", 0, 50.0, 0.78125),
        # the ordinary diagnostic case: one cone-beam view of a 35 cm water cylinder, S8 P3, 19 groups
        _problem("cylinder_s8p3", "solve", "cylinder", 64, 64, 32, 8, 3, 19),
        # a cropped field of view: sides that no tile divides, three views, S4 P3
        _problem("ragged_s4p3", "solve", "cylinder", 75, 61, 37, 4, 3, 12, 3),
        # diamond differencing of the ordinary case
        _problem("diamond_s8p3", "solve", "cylinder", 64, 64, 32, 8, 3, 19, 1, "fan", 1),
        # the paper's fine water mesh, single projection, S6 P0
        _problem("fine_s6p0", "solve", "cylinder", 256, 256, 64, 6, 0, 7, 1, "point", 0, 50.0, 0.1953125),
        # the largest: an abdomen with a fine quadrature against ray effects, S16 P3
        _problem("abdomen_s16p3", "solve", "abdomen", 128, 128, 48, 16, 3, 19, 1, "fan", 0, 32.0, 0.25),
        # the backward direction alone: gradients of the mean dose of a region, one view
        _problem("gradients_s8p3", "gradients", "cylinder", 64, 64, 32, 8, 3, 19),
        # one step of dose optimisation over eight views: new densities and weights in, gradients out
        _problem("train_s8p3", "train", "abdomen", 64, 64, 24, 8, 3, 19, 8, "fan", 0, 32.0, 0.5),
        # views and patients of unequal size in one batch, each with its own solution
        {**_problem("batch_s8p3", "batch", "cylinder", 64, 64, 32, 8, 3, 19), "instances": 6},
        # the input path: a CT volume to materials and densities
        {"name": "ct_volume", "kind": "ct", "nx": 512, "ny": 512, "nz": 160},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _updates(c):
    """Cell updates (voxel x direction x group) of one sweep, all instances."""
    n = sum(d[0] * d[1] * d[2] for d in _batch_dims(c)) if c["kind"] == "batch" else c["nx"] * c["ny"] * c["nz"]
    return n * c["sn"] * (c["sn"] + 2) * c["groups"]


_SWEEPS = {"solve": 14, "batch": 14, "gradients": 22, "train": 38}   # sweeps a solution takes at least, about


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["gradients", "train", "batch", "ct"])
    if kind == "ct":
        return {"kind": "ct", "nx": _log_int(rng, 32, 512), "ny": _log_int(rng, 32, 512), "nz": _log_int(rng, 1, 160)}
    most = 14 * 128 * 128 * 48 * 288 * 19
    while True:
        nx, ny, nz = _log_int(rng, 12, 256), _log_int(rng, 12, 256), _log_int(rng, 8, 64)
        if kind != "solve":
            nx, ny, nz = _log_int(rng, 16, 96), _log_int(rng, 16, 96), _log_int(rng, 8, 48)
        c = _problem("", kind, rng.choice(["cylinder", "abdomen"]), nx, ny, nz,
                     rng.choice([2, 4, 4, 6, 6, 8, 8, 12, 16]) if kind == "solve" else rng.choice([4, 6, 8, 8]),
                     rng.choice([0, 0, 1, 1, 2, 3, 3, 3]), rng.randint(4, 24),
                     rng.choice([1, 1, 2, 3, 8, 16]), rng.choice(["fan", "fan", "point"]),
                     rng.choice([0, 0, 0, 0, 0, 1]) if kind == "solve" else 0,
                     rng.uniform(32.0, 50.0), rng.uniform(0.2, 0.8))
        if kind == "batch":
            c["instances"], c["beams"] = rng.randint(2, 8), 1
        if c["legendre"] == 0 and c["sn"] > 8 or c["sn"] == 2 and c["legendre"] == 3:
            continue    # orders nobody pairs
        if 4e5 <= _updates(c) and _SWEEPS[kind] * _updates(c) <= most:
            del c["name"]
            return c


# ---------------------------------------------------------------------------
# inputs (host arrays, from the seed alone)
# ---------------------------------------------------------------------------

# water-like attenuation A (20 keV / E)^3 + B: mean free paths 13.9 mm at 20 keV, 60.6 mm at 100 keV
_B = (1.0 / 6.06 - (1.0 / 1.39) / 125.0) / (1.0 - 1.0 / 125.0)
_A = 1.0 / 1.39 - _B


def _tables(rng, groups, legendre, photo):
    """sigma_t [nmat][G], sigma_s [nmat][L+1][G][G] (downscatter), group mid-energies."""
    edges = np.linspace(120.0, 10.0, groups + 1)
    e = 0.5 * (edges[1:] + edges[:-1])
    st = np.zeros((len(photo), groups))
    ss = np.zeros((len(photo), legendre + 1, groups, groups))
    for m, pe in enumerate(photo):
        st[m] = pe * rng.uniform(0.95, 1.05) * _A * (20.0 / e) ** 3 + _B
        out = _B * rng.uniform(0.9, 1.0, groups)
        within, aniso = rng.uniform(0.3, 0.6, groups), rng.uniform(0.1, 0.4, groups)
        s0 = np.diag(within * out)
        for g in range(groups - 1):
            tail = 0.5 ** np.arange(groups - 1 - g)
            s0[g, g + 1:] = (1.0 - within[g]) * out[g] * tail / tail.sum()
        for l in range(legendre + 1):
            ss[m, l] = s0 * aniso[:, None] ** l
    return st, ss, e


def _one(case, rng, dims, diameter=35.0, theta=None):
    nx, ny, nz = dims
    cube = case["phantom"] == "cube"
    d = (1.0, 1.0, 1.0) if cube else (case["fov"] / nx, case["fov"] / ny, case["dz"])
    origin = -0.5 * np.array([nx * d[0], ny * d[1], nz * d[2]])
    x = (origin[0] + (np.arange(nx) + 0.5) * d[0])[None, :]
    y = (origin[1] + (np.arange(ny) + 0.5) * d[1])[:, None]
    if cube:
        photo, rho, plane = [1.0], [1.0], np.zeros((ny, nx), np.uint8)
    elif case["phantom"] == "cylinder":
        photo, rho = [0.9, 1.0], [0.0012, 1.0]
        plane = (x * x + y * y <= (0.5 * diameter) ** 2).astype(np.uint8)
    else:   # air, fat, soft tissue, liver, bone
        photo, rho = [0.9, 0.6, 1.0, 1.05, 6.0], [0.0012, 0.92, 1.03, 1.06, 1.85]
        plane = np.zeros((ny, nx), np.uint8)
        for m, cx, cy, ax, ay in ((1, 0, 0, 16, 12), (2, 0, 0, 15, 11), (3, -6, 0, 5, 4), (4, 0, -8, 2, 1.5),
                                  (0, 5, 7, 2.5, 1.5), (0, -5, 7, 2.5, 1.5)):
            plane[((x - cx) / ax) ** 2 + ((y - cy) / ay) ** 2 <= 1.0] = m
    st, ss, e = _tables(rng, case["groups"], case["legendre"], photo)
    mat = np.broadcast_to(plane, (nz, ny, nx)).reshape(-1).copy()
    # reconstructed densities vary a little from voxel to voxel
    density = (np.asarray(rho)[mat] * rng.uniform(0.97, 1.03, mat.size)).astype(np.float32)
    spectrum = (125.0 - e) / e * 2.0 ** -((30.0 / e) ** 3) * rng.uniform(0.95, 1.05, e.size)
    spectrum /= spectrum.sum()
    sid = 54.0
    start = rng.uniform(0.0, 2.0 * math.pi) if theta is None else theta
    z_half = 0.5 * nz * d[2] if case["phantom"] == "abdomen" else min(2.0, 0.5 * nz * d[2])
    sources = []
    for b in range(case["beams"]):
        a = start + 2.0 * math.pi * b / case["beams"]
        pos = sid * np.array([math.sin(a), -math.cos(a), 0.0])
        sources.append(SimpleNamespace(kind=0 if case["beam"] == "point" else 1, pos=pos, axis=-pos / np.linalg.norm(pos),
                                       fan_deg=40.0, z_half_iso=z_half, iso_dist=sid,
                                       weight=float(rng.uniform(0.5, 1.5)), spectrum=spectrum.copy()))
    k_dep = e[None, :] * (st - ss[:, 0].sum(axis=2))
    cx, cy = (-6.0, 0.0) if case["phantom"] == "abdomen" else (0.0, 0.0)
    roi = np.zeros((nz, ny, nx))
    box = (np.abs(x - cx) <= 3.0) & (np.abs(y - cy) <= 3.0)
    roi[nz // 4:max(nz // 4 + 1, 3 * nz // 4)] = box
    roi /= max(1.0, roi.sum())
    return SimpleNamespace(nx=nx, ny=ny, nz=nz, dx=d[0], dy=d[1], dz=d[2], origin=origin, mat=mat, density=density,
                           sigma_t=st, sigma_s=ss, sn=case["sn"], legendre=case["legendre"], sources=sources,
                           differencing=case["scheme"], k_dep=k_dep, roi=roi.reshape(-1))


def _batch_dims(case):
    """Instances alternate between the stated mesh and a taller, narrower one."""
    big, small = (case["nx"], case["ny"], case["nz"]), (max(8, 3 * case["nx"] // 4), max(8, 3 * case["ny"] // 4),
                                                       max(8, 3 * case["nz"] // 2))
    return [big if q % 2 == 0 else small for q in range(case["instances"])]


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        return [_one(case, rng, dims, 35.0 - 4.0 * (q % 3)) for q, dims in enumerate(_batch_dims(case))]
    return _one(case, rng, (case["nx"], case["ny"], case["nz"]))


# a piecewise calibration for air, fat, soft tissue, liver and bone
_CT_THRESHOLDS = np.array([-500.0, -30.0, 45.0, 150.0], np.float32)
_CT_BINS = np.array([0, 1, 2, 3, 4], np.uint8)
_CT_HU = np.array([-1000.0, -100.0, 20.0, 60.0, 1000.0], np.float32)
_CT_RHO = np.array([0.0012, 0.93, 1.03, 1.06, 1.85], np.float32)


def _ct_image(case, seed):
    """CT numbers: half air, the rest tissue with noise and some bone (float32, on the GPU)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = case["nx"] * case["ny"] * case["nz"]
    kind = torch.rand(n, device="cuda", generator=gen)
    noise = torch.randn(n, device="cuda", generator=gen)
    centre = torch.where(kind < 0.5, -1000.0, torch.where(kind < 0.6, -100.0, torch.where(kind < 0.95, 40.0, 700.0)))
    return centre + 25.0 * noise


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def _on_gpu(p):
    """The problem with its voxel arrays in device memory, as a CT reconstruction leaves them."""
    q = SimpleNamespace(**p.__dict__)
    q.mat = torch.as_tensor(p.mat, device="cuda")
    q.density = torch.as_tensor(p.density, device="cuda")
    return q


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ct":
        return {"kind": kind, "hu": _ct_image(case, seed)}
    p = _inputs(case, seed)
    if kind == "batch":
        return {"kind": kind, "problems": p, "handles": [solver.DoctorsProblem(_on_gpu(q), tol=TOL) for q in p]}
    if kind == "train":
        dev = lambda a: torch.as_tensor(a, device="cuda").requires_grad_()    # noqa: E731
        return {"kind": kind, "handle": autograd.DoseProblem(p, p.roi, tol=TOL),
                "leaves": [dev(np.array([s.weight for s in p.sources])), dev(p.sources[0].spectrum.copy()),
                           dev(p.density)]}
    state = {"kind": kind, "problem": p, "handle": solver.DoctorsProblem(_on_gpu(p), tol=TOL)}
    if kind == "gradients":
        state["roi"] = torch.as_tensor(p.roi, device="cuda")
        state["handle"].solve()
    return state


def run(state):
    kind = state["kind"]
    if kind == "ct":
        mat, rho = solver.ct_to_materials(state["hu"], _CT_THRESHOLDS, _CT_BINS, _CT_HU, _CT_RHO)
        return {"mat": mat, "rho": rho}
    if kind == "batch":
        solver.solve_batch(state["handles"])
        return [{"fluence": h.fluence(), "dose": h.dose(p.k_dep)} for h, p in zip(state["handles"], state["problems"])]
    if kind == "train":
        leaves = state["leaves"]
        J = autograd.RoiDose.apply(*leaves, state["handle"])
        grads = torch.autograd.grad(J, leaves)
        return {"J": J.detach(), "weights": grads[0], "spectrum": grads[1], "density": grads[2]}
    h, p = state["handle"], state["problem"]
    if kind == "gradients":
        g = h.roi_gradients(p.k_dep, state["roi"])
        return {"J": g["J"], "weights": g["weights"], "spectrum": g["spectrum"], "density": g["density"]}
    h.set_sources(p.sources)
    h.solve()
    return {"fluence": h.fluence(), "dose": h.dose(p.k_dep)}


def work(case):
    """Per cell update: 2 (L+1)^2 multiply-adds into and out of the direction and about 8 operations for the cell;
    the bytes are the voxel data in and the fluence, dose or gradients out."""
    if case["kind"] == "ct":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 9 * n, "flops": 4 * n}
    up = _updates(case)
    cells = up // (case["sn"] * (case["sn"] + 2) * case["groups"])
    flops = _SWEEPS[case["kind"]] * up * (4 * (case["legendre"] + 1) ** 2 + 8)
    if case["kind"] in ("gradients", "train"):
        return {"bytes": cells * (1 + 4 + 8 + 8), "flops": flops}
    return {"bytes": cells * (1 + 4 + 8 + 4 * case["groups"]), "flops": flops}


# ---------------------------------------------------------------------------
# the same results in FP64, plain torch
# ---------------------------------------------------------------------------

def exact(case, seed):
    if case["kind"] == "ct":
        hu = _ct_image(case, seed).cpu().numpy()
        mat = _CT_BINS[np.searchsorted(_CT_THRESHOLDS, hu, side="right")]
        return {"mat": mat, "rho": np.interp(hu.astype(np.float64), _CT_HU.astype(np.float64), _CT_RHO.astype(np.float64))}
    if _SWEEPS[case["kind"]] * _updates(case) > 2.5e10:
        return None     # takes longer than a comparison is worth
    p = _inputs(case, seed)
    if case["kind"] == "batch":
        return [_forward_result(_Fp64(q)) for q in p]
    if case["kind"] in ("gradients", "train"):
        return _Fp64(p).gradients()
    return _forward_result(_Fp64(p))


def _forward_result(f):
    phi = f.solve()
    return {"fluence": phi.T.contiguous(), "dose": (f.k[f.mat] * phi).sum(1) * f.rho}


@functools.lru_cache(maxsize=None)
def _octant_directions(sn):
    """First-octant directions and weights of the level-symmetric set: point weights per permutation class
    that integrate every even monomial of degree <= N - 2 exactly."""
    mu1 = {2: 1.0 / math.sqrt(3.0), 4: 0.3500212, 6: 0.2666355, 8: 0.2182179, 12: 0.1672126, 16: 0.1389568}[sn]
    half = sn // 2
    step = 2.0 * (1.0 - 3.0 * mu1 ** 2) / (sn - 2) if sn > 2 else 0.0
    mu = np.sqrt(mu1 ** 2 + step * np.arange(half))
    tri = [t for t in itertools.product(range(half), repeat=3) if sum(t) == half - 1]
    classes = sorted({tuple(sorted(t)) for t in tri})
    pts = np.array([[mu[a] for a in t] for t in tri])
    member = np.array([[tuple(sorted(t)) == c for c in classes] for t in tri], float)
    rows, rhs = [], []
    for a, b, c in itertools.product(range(half), repeat=3):
        if a + b + c < half:
            rows.append((pts[:, 0] ** (2 * a) * pts[:, 1] ** (2 * b) * pts[:, 2] ** (2 * c)) @ member)
            rhs.append(math.gamma(a + .5) * math.gamma(b + .5) * math.gamma(c + .5) / (4.0 * math.gamma(a + b + c + 1.5)))
    return pts, member @ np.linalg.lstsq(np.array(rows), np.array(rhs), rcond=None)[0]


def _harmonics(legendre, d):
    """Real harmonics of unit vectors d [..., 3] with sum_m R_lm(a) R_lm(b) = P_l(a . b)."""
    x, y, z = d[..., 0], d[..., 1], d[..., 2]
    r = [torch.ones_like(x)]
    if legendre > 0:
        r += [x, y, z]
    if legendre > 1:
        s = math.sqrt(3.0)
        r += [s * x * y, s * y * z, s * x * z, 0.5 * s * (x * x - y * y), 1.5 * z * z - 0.5]
    if legendre > 2:
        a, b, c = math.sqrt(5.0 / 8.0), math.sqrt(15.0), math.sqrt(3.0 / 8.0)
        r += [a * y * (3 * x * x - y * y), a * x * (x * x - 3 * y * y), b * x * y * z, 0.5 * b * z * (x * x - y * y),
              c * y * (5 * z * z - 1), c * x * (5 * z * z - 1), 0.5 * z * (5 * z * z - 3)]
    return torch.stack(r, -1)


class _Fp64:
    """One problem in FP64: arrays are voxel first, [V][G] and [V][G][M]."""

    def __init__(self, p):
        t = lambda a: torch.as_tensor(np.asarray(a, np.float64), device="cuda")    # noqa: E731
        self.p = p
        self.V, (self.nmat, self.G), self.L = p.nx * p.ny * p.nz, p.sigma_t.shape, p.legendre
        self.M = (p.legendre + 1) ** 2
        self.mat = torch.as_tensor(p.mat.astype(np.int64), device="cuda")
        self.rho, self.st, self.ss, self.k = t(p.density), t(p.sigma_t), t(p.sigma_s), t(p.k_dep)
        self.sigma = self.rho[:, None] * self.st[self.mat]
        self.voxels = [torch.nonzero(self.mat == m)[:, 0] for m in range(self.nmat)]
        pts, w = _octant_directions(p.sn)
        sign = np.array([[-1.0 if o >> a & 1 else 1.0 for a in range(3)] for o in range(8)])
        R = _harmonics(self.L, t(sign[:, None, :] * pts[None]))                       # [8][A8][M]
        C = t([(2 * l + 1) / (4.0 * math.pi) for l in range(self.L + 1) for _ in range(2 * l + 1)])
        self.A8 = len(w)
        self.to_dir, self.to_mom = (R * C).transpose(1, 2).contiguous(), R * t(w)[None, :, None]
        f = 2.0 if p.differencing else 1.0
        self.c = [t(f * pts[:, a] / (p.dx, p.dy, p.dz)[a]) for a in range(3)]
        # hyperplanes i + j + k = h in every octant's sweep order
        k, j, i = np.meshgrid(np.arange(p.nz), np.arange(p.ny), np.arange(p.nx), indexing="ij")
        i, j, k = (torch.as_tensor(a.reshape(-1), device="cuda") for a in (i, j, k))
        order = torch.argsort(i + j + k, stable=True)
        counts = torch.bincount(i + j + k).tolist()
        self.planes = []
        for sel in torch.split(order, counts):
            a, b, c = i[sel], j[sel], k[sel]
            v = torch.stack([((p.nz - 1 - c if o & 4 else c) * p.ny + (p.ny - 1 - b if o & 2 else b)) * p.nx +
                             (p.nx - 1 - a if o & 1 else a) for o in range(8)])
            self.planes.append((v, b * p.nz + c, a * p.nz + c, a * p.ny + b))

    def sweep(self, s, into, out, reverse=False, g0=0, keep=None):
        """Source moments s [V][G'][M] of groups g0.. to angular fluences (into [8][M][A8]) and back (out)."""
        p, n = self.p, s.shape[1]
        face = [torch.zeros(8, m, n, self.A8, dtype=torch.float64, device="cuda")
                for m in (p.ny * p.nz, p.nx * p.nz, p.nx * p.ny)]
        mom = torch.zeros_like(s)
        csum = sum(self.c)
        if reverse:     # directions -Omega: octant o sweeps with the tables of the opposite octant
            into, out = into.flip(0), out.flip(0)
        for v, *cols in self.planes:
            m = v.shape[1]
            q = torch.bmm(s[v].reshape(8, m * n, -1), into).reshape(8, m, n, self.A8)
            inflow = [f[:, col] for f, col in zip(face, cols)]
            for a in range(3):
                q += self.c[a] * inflow[a]
            q /= self.sigma[v][:, :, g0:g0 + n, None] + csum
            for a in range(3):
                face[a][:, cols[a]] = 2.0 * q - inflow[a] if p.differencing else q
            mom.index_add_(0, v.reshape(-1), torch.bmm(q.reshape(8, m * n, -1), out).reshape(8 * m, n, -1))
            if keep is not None:    # [V][8][G][A8], by the octant of the direction
                for o in range(8):
                    keep[v[o], 7 - o if reverse else o] = q[o]
        return mom

    def scatter(self, x, transpose=False, with_density=True, g0=0, g1=None):
        out = torch.zeros_like(x)
        for m, sel in enumerate(self.voxels):
            for l in range(self.L + 1):
                tab = self.ss[m, l].T if transpose else self.ss[m, l]
                lm = slice(l * l, (l + 1) * (l + 1))
                out[sel, :, lm] = torch.einsum("vgm,gh->vhm", x[sel][:, :, lm], tab)
        return out * self.rho[:, None, None] if with_density else out

    def iterate(self, fixed, into, out, transpose=False):
        """Fixed point of x = sweep(fixed + scatter(x)); groups that are final are not swept again."""
        x = torch.zeros_like(fixed)
        g0, g1 = 0, self.G
        for _ in range(400):
            s = fixed + self.scatter(x, transpose)
            new = self.sweep(s[:, g0:g1].contiguous(), into, out, transpose, g0)
            change = (new[:, :, 0] - x[:, g0:g1, 0]).norm(dim=0) / new[:, :, 0].norm(dim=0).clamp_min(1e-300)
            x[:, g0:g1] = new
            final = (change < 1e-11).tolist()
            while final and final[-1 if transpose else 0]:
                final.pop(-1 if transpose else 0)
                g0, g1 = (g0, g1 - 1) if transpose else (g0 + 1, g1)
            if not final:
                break
        return x

    def walk(self, src, visit):
        """Follow the rays from every voxel centre back to the source: visit(ray, voxel, length)."""
        p = self.p
        n = (p.nx, p.ny, p.nz)
        d = (p.dx, p.dy, p.dz)
        v = torch.arange(self.V, device="cuda")
        cell = [v % p.nx, (v // p.nx) % p.ny, v // (p.nx * p.ny)]
        ray = [float(p.origin[a]) + (cell[a].double() + 0.5) * d[a] - float(src.pos[a]) for a in range(3)]
        length = torch.sqrt(sum(r * r for r in ray))
        step = [torch.where(r > 0, -1, 1) for r in ray]
        at = torch.ones_like(length)
        for _ in range(sum(n) + 3):
            cross = []
            for a in range(3):
                plane = float(p.origin[a]) + (cell[a] + (step[a] > 0)).double() * d[a] - float(src.pos[a])
                cross.append(torch.where(ray[a] == 0, -math.inf, plane / ray[a]))
            cross = torch.stack(cross)
            nxt, axis = cross.max(0)
            seg = at - nxt.clamp_min(0.0)
            visit(v, (cell[2] * p.ny + cell[1]) * p.nx + cell[0], (seg * length).clamp_min(0.0))
            cell = [cell[a] + torch.where(axis == a, step[a], 0) for a in range(3)]
            alive = nxt > 0
            for a in range(3):
                alive &= (cell[a] >= 0) & (cell[a] < n[a])
            if not bool(alive.any()):
                break
            v, length, at = v[alive], length[alive], nxt[alive]
            cell, ray, step = [c[alive] for c in cell], [r[alive] for r in ray], [s[alive] for s in step]

    def lit(self, src):
        """The collimator's mask, decided in FP32 like the geometry it is given in."""
        p, f = self.p, np.float32
        if src.kind == 0:
            return torch.ones(self.V, device="cuda")
        ax = src.axis
        h = math.hypot(ax[0], ax[1])
        perp = np.array([-ax[1] / h, ax[0] / h, 0.0])
        up = np.cross(ax, perp)
        axis = [((f(p.origin[a]) + (np.arange(n, dtype=f) + f(0.5)) * f(d)) - f(src.pos[a])).astype(f)
                for a, (n, d) in enumerate(zip((p.nx, p.ny, p.nz), (p.dx, p.dy, p.dz)))]
        uz, uy, ux = np.meshgrid(axis[2], axis[1], axis[0], indexing="ij")
        dot = lambda e: (ux * f(e[0]) + uy * f(e[1])) + uz * f(e[2])      # noqa: E731
        along, across, vert = dot(ax), dot(perp), dot(up)
        tan, slope = f(math.tan(0.5 * src.fan_deg * (math.pi / 180.0))), f(src.z_half_iso / src.iso_dist)
        on = (along > 0) & (np.abs(across) <= tan * along) & (np.abs(vert) <= slope * along)
        return torch.as_tensor(on.reshape(-1).astype(np.float64), device="cuda")

    def uncollided(self, src):
        """Fluence per emitted photon [V][G] and harmonics [V][M] of the direction of flight."""
        p = self.p
        depth = torch.zeros(self.V * self.nmat, dtype=torch.float64, device="cuda")

        def visit(ray, u, length):
            depth[ray * self.nmat + self.mat[u]] += self.rho[u] * length
        self.walk(src, visit)
        v = torch.arange(self.V, device="cuda")
        i, j, k = (v % p.nx).double(), (v // p.nx % p.ny).double(), (v // (p.nx * p.ny)).double()
        pos = torch.stack([float(p.origin[0]) + (i + 0.5) * p.dx - float(src.pos[0]),
                           float(p.origin[1]) + (j + 0.5) * p.dy - float(src.pos[1]),
                           float(p.origin[2]) + (k + 0.5) * p.dz - float(src.pos[2])], -1)
        r2 = (pos * pos).sum(1)
        u = (self.lit(src) / (4.0 * math.pi * r2))[:, None] * torch.exp(-depth.reshape(self.V, self.nmat) @ self.st)
        return u, _harmonics(self.L, pos / r2.sqrt()[:, None])

    def solve(self):
        """Total scalar fluence [V][G]."""
        chi = [torch.as_tensor(s.weight * s.spectrum, device="cuda") for s in self.p.sources]
        self.phiu = torch.zeros(self.V, self.G, dtype=torch.float64, device="cuda")
        self.U = torch.zeros(self.V, self.G, self.M, dtype=torch.float64, device="cuda")
        for src, e in zip(self.p.sources, chi):
            u, R = self.uncollided(src)
            self.phiu += u * e
            self.U += (u * e)[:, :, None] * R[:, None, :]
        self.Q = self.scatter(self.U)
        self.x = self.iterate(self.Q, self.to_dir, self.to_mom)
        return self.phiu + self.x[:, :, 0]

    def gradients(self):
        """J = sum_v roi(v) dose(v) and its gradients, by the transposed equations."""
        p = self.p
        phi = self.solve()
        roi = torch.as_tensor(p.roi, device="cuda")
        per_rho = roi[:, None] * self.k[self.mat]
        r = per_rho * self.rho[:, None]
        # b = dJ/d(source moments) solves b = transposed sweep (r in l = 0 + transposed scatter b)
        into, out = self.to_mom.transpose(1, 2).contiguous(), self.to_dir.transpose(1, 2).contiguous()
        r0 = torch.zeros_like(self.x)
        r0[:, :, 0] = r
        # iterate x = r0 + scatter^T(sweep^T x) in the form it knows: b = sweep^T(r0 + scatter^T b)
        b = self.iterate(r0, into, out, True)
        shape = (self.V, 8, self.G, self.A8)
        psi, chi = (torch.empty(shape, dtype=torch.float64, device="cuda") for _ in range(2))
        self.sweep(self.Q + self.scatter(self.x), self.to_dir, self.to_mom, keep=psi)
        back = self.scatter(b, True)
        self.sweep(r0 + back, into, out, True, keep=chi)
        rho_grad = (per_rho * phi).sum(1)
        rho_grad -= (self.st[self.mat] * torch.einsum("voga,voga->vg", psi, chi)).sum(1)
        del psi, chi
        rho_grad += (b * self.scatter(self.x + self.U, with_density=False)).sum((1, 2))
        weights, spectrum = [], torch.zeros(self.G, dtype=torch.float64, device="cuda")
        for src in p.sources:
            u, R = self.uncollided(src)
            imp = u * (r + torch.einsum("vgm,vm->vg", back, R))
            e = torch.as_tensor(src.spectrum, device="cuda")
            weights.append((imp.sum(0) * e).sum())
            spectrum += src.weight * imp.sum(0)
            h = (imp * (src.weight * e)) @ self.st.T                    # [V][nmat]

            def visit(ray, v, length):
                rho_grad.index_add_(0, v, -length * h[ray, self.mat[v]])
            self.walk(src, visit)
        return {"J": (roi * (self.k[self.mat] * phi).sum(1) * self.rho).sum(), "weights": torch.stack(weights),
                "spectrum": spectrum, "density": rho_grad}
