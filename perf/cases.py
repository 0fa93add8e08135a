"""Timed cases: the calls a user of the library makes, over the sizes this repository works at.

A case is a dict of plain values.  Its "kind" says which public calls one pass makes:

  solve    frequency solves (bie_solve_frequencies) of a mesh at nk wavenumbers, mode "mixed",
           "fp64" or "learned"
  async    the same solves stream-ordered (bie_solve_frequencies_async)
  multi    several incident directions on one factor (bie_solve_frequencies_multi)
  field    a pulse's space-time field at observation points from surface solutions in hand:
           spectrum, field evaluation, synthesis
  picked   the same at the `keep` dominant frequencies of the pulse (bie_top_frequencies)
  whole    solves, field, spectrum and synthesis one after the other
  pulses   synthesis of many pulses from field spectra in hand

A scene is `bodies` spheres or ellipsoids (meshes of 6-node triangles from `workloads`) on a
lattice, turned as a whole by a rotation that the seed draws; the seed also draws the incident
direction, the exact wavenumber spacing, ellipsoid axes, pulses and surface solutions.  Surface
solutions "in hand" are the surface values of point sources inside the bodies, i.e. of a radiating
field, as a solve would return them.
"""
from __future__ import annotations

import collections
import functools
import math

import numpy as np
import torch

from paper_1706_07919_gb300 import Solver
from paper_1706_07919_gb300 import binding as B
from workloads import (ellipsoid_from_sphere, gaussian_pulse, ico_sphere, merge_meshes, modulated_gaussian, octa_sphere,
                       paper_sine_pulse, ricker_pulse, scale_translate)

MODES = {"mixed": B.BIE_MODE_MIXED, "fp64": B.BIE_MODE_FP64, "learned": B.BIE_MODE_LEARNED}
TAU = 2.0 * math.pi

# A scene's defaults: `grid` "ico" (20 div^2 elements a body) or "octa" (8 4^div), `uneven` 1: every
# body after the first has one division fewer (down to 3) and is an ellipsoid, `bc` "hard", "soft"
# or "both" (alternating bodies), `gap` between neighbouring unit spheres, `long` the third semi-axis.
SCENE = dict(bodies=1, grid="ico", div=5, uneven=0, bc="hard", gap=0.1, long=1.0)


def _case(kind, name=None, **kw):
    c = dict(kind=kind, **SCENE)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a first look at one scatterer: one wavenumber of the 258-node sphere (latency and launches)
        _case("solve", "sphere_one_frequency", grid="octa", div=2, mode="mixed", nk=1, m0=16, dk=0.125),
        # the plain FP64 experiment: 64 wavenumbers of the 258-node sphere, the field at 1000 shell
        # points, 256 time samples
        _case("whole", "sphere_fp64_whole", grid="octa", div=2, mode="fp64", nk=64, m0=1, dk=0.125, points="shell", m=1000,
              nt=256, out="f64"),
        # the paper's soft sphere (1002 nodes), its 64 frequencies from k = 0 on
        _case("solve", "paper_sphere_sweep", bc="soft", mode="mixed", nk=64, m0=0, dk=TAU / 20.1),
        # Table I's question: the pulse at two receivers from its 20 dominant frequencies
        _case("picked", "paper_two_receivers", bc="soft", mode="mixed", nk=64, m0=0, dk=TAU / 20.1, points="shell", m=2, nt=128,
              keep=20, out="f64"),
        # part of the benchmark sweep: two hard spheres, 2884 nodes, near the top of its range
        _case("solve", "two_spheres_sweep", bodies=2, div=6, mode="mixed", nk=64, m0=384, dk=1 / 32),
        # the benchmark's plane: 128 x 128 points, 1024 samples, 32-bit output
        _case("field", "two_spheres_plane", bodies=2, div=6, mode="mixed", nk=64, m0=128, dk=1 / 32, points="plane", m=16384,
              nt=1024, out="f32"),
        # a configuration of the uneven batch (hard and soft bodies of different sizes), enqueued
        _case("async", "uneven_bodies_async", bodies=3, div=6, uneven=1, bc="both", gap=0.5, mode="mixed", nk=24, m0=100,
              dk=8 / 256),
        # one configuration under eight incident waves: the factor is shared
        _case("multi", "sphere_eight_directions", mode="mixed", nk=24, m0=8, dk=TAU / 20.1, dirs=8),
        # the learned sweep on the spheroid (2562 nodes): anchors, training, GMRES
        _case("solve", "spheroid_learned", div=8, long=2.0, mode="learned", nk=32, m0=256, dk=20 / 1024),
        # half of the large lattice: 16 soft spheres, 10 272 nodes, few systems at once
        _case("solve", "lattice_two_frequencies", bodies=16, div=4, bc="soft", gap=0.4, mode="mixed", nk=2, m0=400, dk=12 / 1024),
        # the plain FP64 solve at the benchmark's size (the judge of the mixed one)
        _case("solve", "two_spheres_fp64", bodies=2, div=6, mode="fp64", nk=2, m0=100, dk=1 / 32),
        # many pulses on the same solves: eight signals of 4096 samples at 8192 points
        _case("pulses", "eight_pulses", nk=512, m0=1, dk=12 / 1024, m=8192, nt=4096, pulses=8, out="f32"),
    ]


def _sizes(c):
    """Nodes and standard quadrature points of a case's scene (the library's default 4 x 4 rule)."""
    divs = _divs(c)
    e = sum(8 * 4 ** d if c["grid"] == "octa" else 20 * d * d for d in divs)
    return 2 * e + 2 * len(divs), 16 * e


def _divs(c):
    return [max(3, c["div"] - i) if c["uneven"] else c["div"] for i in range(c["bodies"])]


def _cost(c):
    """About how long a pass takes (s): only to keep drawn cases below the largest listed one."""
    n, q = _sizes(c)
    t = 0.0
    if c["kind"] in ("solve", "whole", "async", "multi"):
        fp64 = c["mode"] == "fp64"
        d = c.get("dirs", 1)
        t += c["nk"] * (n * q * (2.5e-10 if fp64 else 1e-11) * (2 if d > 1 else 1) + n ** 3 * (4.5e-12 if fp64 else 1.6e-14) +
                        n * n * d * 2e-11) + 0.004
        if c["mode"] == "learned":
            t += 0.1 + c["nk"] * n * n * 3e-10
    if c["kind"] in ("field", "picked", "whole"):
        t += max(c["m"], 128) * q * c["nk"] * (1.2e-10 if c["mode"] == "fp64" else 2.6e-12) + 0.001
    if "nt" in c:
        t += c["m"] * c["nt"] * c.get("pulses", 1) * 2e-12
    return t


def draw(rng):
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    while True:
        kind = rng.choice(["solve", "solve", "solve", "async", "multi", "field", "field", "picked", "whole", "pulses"])
        mode = rng.choice(["mixed", "mixed", "mixed", "fp64"]) if kind in ("solve", "multi", "field", "whole") else "mixed"
        if kind == "solve" and rng.random() < 0.1:
            mode = "learned"
        bodies = rng.choice([1, 1, 2, 2, 3, 5, 8])
        uneven = int(bodies > 1 and rng.random() < 0.5)
        bc = rng.choice(["hard", "hard", "soft", "both"])
        dk = rng.uniform(1 / 96, 1 / 6)
        c = _case(kind, bodies=bodies, div=rng.randint(3, 8), uneven=uneven, bc=bc, gap=round(rng.uniform(0.1, 0.8), 3), mode=mode,
                  nk=log(1, 300), m0=rng.randint(0, 60), dk=round(dk, 5))
        if bodies == 1 and rng.random() < 0.3:
            c.update(grid="octa", div=rng.randint(1, 3))
        if bodies == 1 and rng.random() < 0.3:
            c.update(long=round(rng.uniform(0.6, 2.0), 3))
        if kind == "multi":
            c.update(dirs=rng.randint(2, 12), nk=log(1, 60))
        if mode == "learned":
            c.update(m0=max(4, c["m0"]), nk=log(17, 64), bc="hard", uneven=0, gap=0.4)
        if kind in ("field", "picked", "whole"):
            nt = 2 ** rng.randint(6, 12)
            c.update(points=rng.choice(["plane", "shell", "line"]), m=log(1, 30000), nt=nt, out=rng.choice(["f32", "f64"]))
            if kind == "picked":
                c.update(m0=0, nk=min(nt // 2 + 1, log(4, 200)))
                c.update(keep=rng.randint(1, c["nk"]))
        if kind == "pulses":
            c.update(nt=2 ** rng.randint(4, 12), m=log(1, 70000), pulses=rng.randint(1, 9), out=rng.choice(["f32", "f64"]),
                     nk=log(2, 1500))
            c.update(m0=rng.randint(0, 3))
        if "nt" in c:  # the wavenumbers are harmonics m0 .. m0 + nk - 1 of the window
            if c["m0"] + c["nk"] > c["nt"] // 2 + 1:
                continue
            if c.get("pulses", 1) * c["m"] * c["nt"] > 2 ** 28:
                continue
        # resolved waves only: at least about three elements to a wavelength, as in the workloads
        k_max = (c["m0"] + c["nk"]) * c["dk"]
        if kind != "pulses" and k_max > 2.6 * min(2 ** c["div"] if c["grid"] == "octa" else d for d in _divs(c)):
            continue
        if (c["m0"] + c["nk"]) < 2 or _cost(c) > 0.35:
            continue
        return c


# ---- inputs ----------------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _unit(grid, div):
    return octa_sphere(div) if grid == "octa" else ico_sphere(div)


def _rotation(rng):
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    q = q * np.sign(np.diag(r))
    return q if np.linalg.det(q) > 0 else q[:, [1, 0, 2]]


def _unit_vectors(rng, n):
    v = rng.standard_normal((n, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def _scene(c, rng):
    """The mesh, the bodies' centres and bounding radii, and the scene's rotation."""
    n = c["bodies"]
    side = max(1, math.ceil(n ** (1 / 3) - 1e-9))
    step = 2.0 + c["gap"]
    # a line of up to three bodies along the third axis, a lattice from four on
    spots = [(0, 0, i) for i in range(n)] if n <= 3 else [(i // (2 * side), (i // 2) % side, i % 2) for i in range(n)]
    spots = np.array(spots, float) * step
    spots -= spots.mean(axis=0)
    turn = _rotation(rng)
    parts, radii = [], []
    for i, d in enumerate(_divs(c)):
        axes = (1.0, 1.0, c["long"])
        if c["uneven"] and i > 0:
            axes = (1.0, rng.uniform(0.5, 1.0), rng.uniform(0.5, 1.0))
        m = _unit(c["grid"], d)
        if axes != (1.0, 1.0, 1.0):
            m = ellipsoid_from_sphere(m, axes)
        soft = c["bc"] == "soft" or (c["bc"] == "both" and i % 2 == 1)
        own = _rotation(rng) if c["uneven"] else np.eye(3)
        parts.append(scale_translate(m, 1.0, turn @ spots[i], rot=turn @ own, bc=int(soft)))
        radii.append((max(axes), min(axes)))
    return merge_meshes(parts).contiguous(), spots @ turn.T, np.array(radii), turn


def _observers(c, rng, centres, radii, turn):
    """Points in the fluid: on a plane through the scene, in a shell around it, or on a line."""
    m, out = c["m"], np.zeros((c["m"], 3))
    reach = np.linalg.norm(centres, axis=1).max() + radii.max()
    if c["points"] == "plane":
        n = math.ceil(math.sqrt(m))
        g = np.linspace(-5.0, 5.0, n) * max(1.0, reach / 3.0)
        x, y = np.meshgrid(g, g, indexing="ij")
        out[:, 0], out[:, 1] = x.ravel()[:m], y.ravel()[:m]
        out[:, 2] = rng.uniform(-0.02, 0.02)
    elif c["points"] == "shell":
        d = _unit_vectors(rng, m)
        out = d * (reach * rng.uniform(1.05, 3.0, (m, 1)))
    else:
        out[:, 2] = np.linspace(-4.0 * reach, 4.0 * reach, m) if m > 1 else 1.5 * reach
        out[:, 0] = rng.uniform(0.3, 0.6)
    out = out @ turn.T
    for x0, (r, _) in zip(centres, radii):  # the bounding balls are disjoint: none pushed into another
        v = out - x0
        dist = np.linalg.norm(v, axis=1, keepdims=True)
        v = np.where(dist > 1e-9, v / np.maximum(dist, 1e-9), turn[:, 0])
        out = np.where(dist < 1.03 * r, x0 + 1.03 * r * v, out)
    return out


def _signals(c, rng, dk):
    nt, t = c["nt"], TAU / dk
    top = (c["m0"] + c["nk"]) * dk  # highest wavenumber: the pulses live below it
    rows = []
    for p in range(c.get("pulses", 1)):
        tc = t * rng.uniform(0.2, 0.6)
        kind = "sine" if c["kind"] == "picked" else ("gauss", "ricker", "mod")[p % 3]
        if kind == "sine":
            rows.append(paper_sine_pulse(nt, t, top * rng.uniform(0.2, 0.4), 4, 0.1, 0.1 * t))
        elif kind == "gauss":
            rows.append(gaussian_pulse(nt, t, sigma=4.0 / top * rng.uniform(0.9, 1.1), tc=tc))
        elif kind == "ricker":
            rows.append(ricker_pulse(nt, t, kp=0.35 * top * rng.uniform(0.9, 1.1), tc=tc))
        else:
            rows.append(modulated_gaussian(nt, t, kc=top * rng.uniform(0.3, 0.6), sigma=12.0 / top, tc=tc))
    return np.stack(rows)


def _sources(rng, centres, radii, per=2):
    pos = np.repeat(centres, per, axis=0) + 0.35 * np.repeat(radii[:, 1:], per, axis=0) * _unit_vectors(rng, per * len(centres))
    amp = rng.standard_normal(len(pos)) + 1j * rng.standard_normal(len(pos))
    return pos, amp / math.sqrt(len(pos))


def _radiated(mesh, k, pos, amp):
    """Surface values [nk][2][N] (P and its normal derivative) of point sources inside the bodies."""
    x, nu = _dev(mesh.nodes), _dev(mesh.normals)
    kt = torch.as_tensor(k, dtype=torch.float64, device=_device())[:, None]
    surf = torch.zeros((len(k), 2, mesh.N), dtype=torch.complex128, device=_device())
    for s, a in zip(pos, amp):
        r = x - _dev(s)
        dist = r.norm(dim=1)[None, :]
        e = complex(a) * torch.polar(1.0 / dist.expand(len(k), -1), kt * dist)
        surf[:, 0] += e
        surf[:, 1] += e * torch.complex(-1.0 / dist.expand(len(k), -1), kt.expand(-1, mesh.N)) * ((r * nu).sum(dim=1)[None, :] / dist)
    return surf


def _device():
    return torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=_device())


def _inputs(c, seed):
    """Everything that the seed decides, the same for prepare() and exact()."""
    rng = np.random.Generator(np.random.PCG64([1706, 7919, int(seed)]))
    s = dict(dk=c["dk"] * rng.uniform(0.98, 1.02))
    s["midx"] = np.arange(c["m0"], c["m0"] + c["nk"], dtype=np.int64)
    s["k"] = s["dk"] * s["midx"].astype(np.float64)
    if c["kind"] != "pulses":
        s["mesh"], centres, radii, turn = _scene(c, rng)
        s["dir"] = _unit_vectors(rng, 1)[0]
        s["dirs"] = _unit_vectors(rng, c.get("dirs", 1))
        if "points" in c:
            s["xobs"] = _observers(c, rng, centres, radii, turn)
        if c["kind"] in ("field", "picked"):
            s["surf"] = _radiated(s["mesh"], s["k"], *_sources(rng, centres, radii))
    else:
        # spectra at the points: a few waves from different distances, as a scattered field has
        g = torch.Generator(device=_device()).manual_seed(int(seed) + 11)
        far = 1.0 + 9.0 * torch.rand((1, c["m"]), dtype=torch.float64, device=_device(), generator=g)
        amp = torch.randn((c["nk"], c["m"]), dtype=torch.float64, device=_device(), generator=g).mul_(0.1).add_(1.0)
        s["T"] = torch.polar(amp.abs_().div_(far), _dev(s["k"])[:, None] * far)
    if "nt" in c:
        s["s"] = _dev(_signals(c, rng, s["dk"]))
    return s


def prepare(case, seed):
    c = case
    s = _inputs(c, seed)
    sol = Solver(0)
    s["sol"] = sol
    if "mesh" in s:
        mesh = s["mesh"]
        sol.set_geometry(mesh.nodes, mesh.elems, mesh.normals, mesh.bc)
        sol.set_incident_plane_wave(s["dir"])
    if "xobs" in s:
        s["xobs"] = _dev(s["xobs"])
    s["case"] = c
    s["pending"] = collections.deque(maxlen=64)
    return s


def run(state):
    c, sol = state["case"], state["sol"]
    kind = c["kind"]
    if kind == "solve":
        return sol.solve_frequencies(state["k"], MODES[c["mode"]])[0]
    if kind == "async":
        surf, pending = sol.solve_frequencies_async(state["k"])
        state["pending"].append(pending)  # the reports are filled in stream order
        return surf
    if kind == "multi":
        return sol.solve_frequencies_multi(state["k"], state["dirs"], MODES[c["mode"]])[0]
    dtype = torch.float32 if c["out"] == "f32" else torch.float64
    spectrum = sol.pulse_spectrum(state["s"])
    if kind == "pulses":
        return sol.synthesize(state["T"], state["midx"], spectrum, c["nt"], dtype)
    out = {}
    k, midx = state["k"], state["midx"]
    if kind == "whole":
        surf = sol.solve_frequencies(k, MODES[c["mode"]])[0]
        out["surf"] = surf
    else:
        surf = state["surf"]
    if kind == "picked":  # the dominant frequencies among those with a solution in hand
        midx = sol.top_frequencies(spectrum, c["nt"], c["keep"])
        midx = midx[midx < c["nk"]]
        k, surf = state["dk"] * midx.astype(np.float64), surf[torch.as_tensor(midx, device=surf.device)]
        out["midx"] = midx
    field = sol.eval_field(state["xobs"], k, surf, MODES[c["mode"]])
    out["p"] = sol.synthesize(field, midx, spectrum, c["nt"], dtype)
    return out


def work(case):
    """One pass's work: the mesh, pulses and points read and the results written once; per solve the
    quadrature of every row (104 flops a point: kernels, regularisation, six nodal sums) and the LU
    (8/3 N^3), per field value 98 flops a point, per signal an FFT."""
    c = case
    n, q = _sizes(c)
    nbytes, flops = 0.0, 0.0
    dirs = c.get("dirs", 1)
    if c["kind"] != "pulses":
        nbytes += n * 49 + q / 16 * 24
    if c["kind"] in ("solve", "async", "multi", "whole"):
        nbytes += c["nk"] * dirs * 2 * n * 16
        flops += c["nk"] * (104.0 * n * q * (2 if dirs > 1 else 1) + 8.0 / 3.0 * n ** 3 + dirs * 8.0 * n * n)
    nf = c.get("keep", c["nk"])
    if c["kind"] in ("field", "picked", "whole"):
        if c["kind"] != "whole":
            nbytes += nf * 2 * n * 16
        nbytes += c["m"] * 24
        flops += 98.0 * c["m"] * q * nf
    if c["kind"] == "pulses":
        nbytes += c["nk"] * c["m"] * 16
    if "nt" in c:
        p = c.get("pulses", 1)
        nbytes += p * c["nt"] * 8 + p * c["m"] * c["nt"] * (4 if c["out"] == "f32" else 8)
        flops += p * c["m"] * (2.5 * c["nt"] * math.log2(c["nt"]) + 8.0 * nf)
    return {"bytes": nbytes, "flops": flops}


# ---- the same in 64 bits: the method's equations in plain torch ---------------------------------

def _duffy(n, v, a, b):
    x, w = np.polynomial.legendre.leggauss(n)
    x, w = 0.5 * (x + 1.0), 0.5 * w
    e1, e2 = a - v, b - a
    det = abs(e1[0] * e2[1] - e1[1] * e2[0])
    u, t = np.meshgrid(x, x, indexing="ij")
    p = v + u[..., None] * e1 + (u * t)[..., None] * e2
    return p.reshape(-1, 2), (np.outer(w * x, w) * det).ravel()


REF = np.array([(0, 0), (1, 0), (0, 1), (0.5, 0), (0.5, 0.5), (0, 0.5)], float)


def _near_rule(a, n=6):
    """Points on an element that holds the collocation node a: collapsed onto the node."""
    if a < 3:
        return _duffy(n, REF[a], REF[(a + 1) % 3], REF[(a + 2) % 3])
    pa, pb, pc = a - 3, (a - 2) % 3, (a - 1) % 3
    p, w = zip(_duffy(n, REF[a], REF[pb], REF[pc]), _duffy(n, REF[a], REF[pc], REF[pa]))
    return np.concatenate(p), np.concatenate(w)


def _shapes(p):
    """Quadratic shape functions and their derivatives at p [..., 2] (torch or numpy columns)."""
    x, y = p[..., 0], p[..., 1]
    l1 = 1.0 - x - y
    stack = torch.stack if isinstance(p, torch.Tensor) else (lambda v, dim: np.stack(v, axis=dim))
    z = 0.0 * x
    return (stack([l1 * (2 * l1 - 1), x * (2 * x - 1), y * (2 * y - 1), 4 * l1 * x, 4 * x * y, 4 * y * l1], -1),
            stack([1 - 4 * l1, 4 * x - 1, z, 4 * (l1 - x), 4 * y, -4 * y], -1),
            stack([1 - 4 * l1, z, 4 * y - 1, -4 * x, 4 * x, 4 * (l1 - y)], -1))


class _Surface:
    """Quadrature points of a mesh: the standard 4 x 4 rule, and the rules near each local node."""

    def __init__(self, mesh):
        self.x, self.nu, self.soft = _dev(mesh.nodes), _dev(mesh.normals), _dev(mesh.bc.astype(bool))
        self.el = _dev(mesh.elems.astype(np.int64))
        self.N, self.E = mesh.N, mesh.E
        p, w = _duffy(4, REF[0], REF[1], REF[2])
        self.shape, self.q = _dev(_shapes(p)[0]), len(w)
        self.pts = self._at(p, w)
        self.near = []
        for a in range(6):
            p, w = _near_rule(a)
            self.near.append((_dev(_shapes(p)[0]), self._at(p, w)))

    def _at(self, p, w):
        n, dx, dy = (_dev(v) for v in _shapes(p))
        x = self.x[self.el]
        pos = torch.einsum("qa,ead->eqd", n, x)
        nrm = torch.linalg.cross(torch.einsum("qa,ead->eqd", dx, x), torch.einsum("qa,ead->eqd", dy, x))
        jac = nrm.norm(dim=-1)
        return pos, nrm / jac[..., None], _dev(w) * jac


def _kernels(k, pos, nuq, wj, xi, nui):
    """w G, w dG/dnu and the regularised terms about xi (broadcast over points)."""
    r = [pos[..., d] - xi[..., d] for d in range(3)]
    dist = (r[0] ** 2 + r[1] ** 2 + r[2] ** 2).sqrt()
    rn = (r[0] * nuq[..., 0] + r[1] * nuq[..., 1] + r[2] * nuq[..., 2]) / dist ** 3
    nr = r[0] * nui[..., 0] + r[1] * nui[..., 1] + r[2] * nui[..., 2]
    nn = nuq[..., 0] * nui[..., 0] + nuq[..., 1] * nui[..., 1] + nuq[..., 2] * nui[..., 2]
    e = torch.polar(wj.expand_as(dist), k * dist)
    g = e / dist
    dg = e * torch.complex(-rn, k * dist * rn)
    c = (k * nr).cos()
    f = (k * nr).sin() / k if k > 0 else nr
    al = c * dg + (k * (k * nr).sin() * nn) * g
    be = f * dg - (c * nn) * g
    return g, dg, al, be


def _system(s, k):
    """The coefficients of P and of P' in Eq. (BRIEF) at one wavenumber: C, D [N][N]."""
    N, E, Q = s.N, s.E, s.q
    H = torch.zeros((N, N), dtype=torch.complex128, device=s.x.device)
    Gm = torch.zeros_like(H)
    al = torch.zeros(N, dtype=torch.complex128, device=s.x.device)
    be = torch.zeros_like(al)
    pos, nuq, wj = (t.reshape(1, E * Q, *t.shape[2:]) for t in s.pts)
    sh, cols = s.shape.to(torch.complex128), s.el.reshape(-1)
    rows = max(1, int(2.5e7 // (E * Q)))
    for i0 in range(0, N, rows):
        i = torch.arange(i0, min(N, i0 + rows), device=s.x.device)
        far = (s.el[None] != i[:, None, None]).all(dim=2)  # elements without node i
        w = (wj.reshape(1, E, Q) * far[..., None]).reshape(len(i), E * Q)
        g, dg, a, b = _kernels(k, pos, nuq, w, s.x[i][:, None], s.nu[i][:, None])
        al[i] += a.sum(dim=1)
        be[i] += b.sum(dim=1)
        for M, v in ((H, dg), (Gm, g)):
            M[i0:i0 + len(i)].index_add_(1, cols, (v.reshape(len(i), E, Q) @ sh).reshape(len(i), -1))
    for a, (shn, (pos, nuq, wj)) in enumerate(s.near):
        i = s.el[:, a]
        g, dg, x, y = _kernels(k, pos, nuq, wj, s.x[i][:, None], s.nu[i][:, None])
        al.index_add_(0, i, x.sum(dim=1))
        be.index_add_(0, i, y.sum(dim=1))
        at = (i[:, None] * N + s.el).reshape(-1)
        for M, v in ((H, dg), (Gm, g)):
            M.view(-1).index_add_(0, at, (v @ shn.to(torch.complex128)).reshape(-1))
    H.diagonal().sub_(4 * math.pi + al)
    Gm.neg_().diagonal().sub_(be)
    return H, Gm


def _solutions(mesh, ks, dirs):
    """Surface values [nk][ndir][2][N] of the direct solves."""
    s = _Surface(mesh)
    d = _dev(dirs)
    out = torch.empty((len(ks), len(dirs), 2, mesh.N), dtype=torch.complex128, device=s.x.device)
    soft = s.soft[:, None]
    for i, k in enumerate(ks):
        C, D = _system(s, float(k))
        p = torch.polar(torch.ones((mesh.N, len(dirs)), dtype=torch.float64, device=s.x.device), float(k) * (s.x @ d.T))
        known = torch.where(soft, -p, -1j * float(k) * (s.nu @ d.T) * p)
        A = torch.where(s.soft[None], D, C)
        C = torch.where(s.soft[None], C, D)
        del D
        x = torch.linalg.solve(A, -(C @ known))
        out[i, :, 0], out[i, :, 1] = torch.where(soft, known, x).T, torch.where(soft, x, known).T
    return out


def _feet(s, xobs):
    """Closest surface points: positions, normals, element and shape values there."""
    m = xobs.shape[0]
    nearest = torch.cat([torch.cdist(p, s.x, compute_mode="donot_use_mm_for_euclid_dist").argmin(dim=1) for p in xobs.split(4096)])
    own = [[] for _ in range(s.N)]
    for e, row in enumerate(s.el.tolist()):
        for a, j in enumerate(row):
            own[j].append((e, a))
    most = max(map(len, own))
    table = _dev(np.array([v + [(-1, 0)] * (most - len(v)) for v in own], np.int64))
    best = torch.full((m,), math.inf, dtype=torch.float64, device=s.x.device)
    at = torch.zeros((m, 2), dtype=torch.float64, device=s.x.device)
    elem = torch.zeros(m, dtype=torch.int64, device=s.x.device)
    second = _dev(np.array([(4, 4, 4), (4, 0, 0), (0, 0, 4), (-8, -4, 0), (0, 4, 0), (0, -4, -8)], float))
    ref = _dev(REF)
    dot = lambda a, b: (a * b).sum(dim=-1)  # noqa: E731
    for col in range(most):
        e, a = table[nearest, col].unbind(dim=1)
        has = (e >= 0).nonzero()[:, 0]
        x, p = s.x[s.el[e[has]]], xobs[has]
        z = ref[a[has]].clone()
        pos = lambda z: torch.einsum("ma,mad->md", _shapes(z)[0], x)  # noqa: E731
        f = dot(pos(z) - p, pos(z) - p)
        live = torch.ones(len(has), dtype=torch.bool, device=s.x.device)
        for _ in range(60):
            n, dx, dy = _shapes(z)
            r = torch.einsum("ma,mad->md", n, x) - p
            t1, t2 = torch.einsum("ma,mad->md", dx, x), torch.einsum("ma,mad->md", dy, x)
            h = torch.einsum("ab,mad->mbd", second, x)
            g1, g2 = dot(r, t1), dot(r, t2)
            a11, a12, a22 = dot(t1, t1) + dot(r, h[:, 0]), dot(t1, t2) + dot(r, h[:, 1]), dot(t2, t2) + dot(r, h[:, 2])
            flat = ~((a11 > 0) & (a11 * a22 - a12 * a12 > 0))
            a11, a12, a22 = (torch.where(flat, u, v) for u, v in ((dot(t1, t1), a11), (dot(t1, t2), a12), (dot(t2, t2), a22)))
            det = a11 * a22 - a12 * a12
            step = torch.stack([-(a22 * g1 - a12 * g2) / det, -(a11 * g2 - a12 * g1) / det], dim=1)
            short = step.abs().sum(dim=1) < 1e-6
            new, newf, todo = z.clone(), f.clone(), live.clone()
            lam = 1.0
            for _ in range(40):
                t = (z + lam * step).clamp_min(0.0)
                over = (t.sum(dim=1) - 1.0).clamp_min(0.0)[:, None] * 0.5
                t = t - over
                t = torch.where(t[:, :1] < 0, _dev(np.array([[0.0, 1.0]])), torch.where(t[:, 1:] < 0, _dev(np.array([[1.0, 0.0]])), t))
                tf = dot(pos(t) - p, pos(t) - p)
                ok = todo & (short | (tf <= f))
                new, newf = torch.where(ok[:, None], t, new), torch.where(ok, tf, newf)
                todo &= ~ok
                if not bool(todo.any()):
                    break
                lam *= 0.5
            live &= ~todo & ((new - z).abs().sum(dim=1) >= 1e-15)
            z, f = new, newf
            if not bool(live.any()):
                break
        better = f < best[has]
        w = has[better]
        best[w], at[w], elem[w] = f[better], z[better], e[has][better]
    n, dx, dy = _shapes(at)
    x = s.x[s.el[elem]]
    nrm = torch.linalg.cross(torch.einsum("ma,mad->md", dx, x), torch.einsum("ma,mad->md", dy, x))
    return torch.einsum("ma,mad->md", n, x), nrm / nrm.norm(dim=1, keepdim=True), elem, n


def _fields(mesh, xobs, ks, surf):
    """Eq. (BRIEFdmn) about the closest surface points: [nk][M]."""
    s = _Surface(mesh)
    xo = _dev(xobs)
    x0, nu0, elem, n0 = _feet(s, xo)
    pos, nuq, wj = (t.reshape(1, -1, *t.shape[2:]) for t in s.pts)
    sh = s.shape.to(torch.complex128)
    out = torch.empty((len(ks), len(xo)), dtype=torch.complex128, device=xo.device)
    step = max(1, int(2.5e7 // pos.shape[1]))
    for m0 in range(0, len(xo), step):
        at = slice(m0, m0 + step)
        el0, nz = s.el[elem[at]], n0[at].to(torch.complex128)
        r0 = pos - x0[at][:, None]
        nr = (r0 * nu0[at][:, None]).sum(dim=-1)
        nn = (nuq * nu0[at][:, None]).sum(dim=-1)
        geo = []
        for r in (pos - xo[at][:, None], r0):
            dist = r.norm(dim=-1)
            geo.append((dist, (r * nuq).sum(dim=-1) / dist ** 3))
        for i, k in enumerate(map(float, ks)):
            P, D = surf[i, 0], surf[i, 1]
            P0, D0 = ((v[el0] * nz).sum(dim=1)[:, None] for v in (P, D))
            Pq, Dq = (torch.einsum("qa,ea->eq", sh, v[s.el]).reshape(1, -1) for v in (P, D))
            (Rp, rp), (R0, rz) = geo
            ep, e0 = (torch.polar(torch.ones_like(R), k * R) for R in (Rp, R0))
            c, sn = (k * nr).cos(), (k * nr).sin()
            f = sn / k if k > 0 else nr
            dd = ep * torch.complex(-rp, k * Rp * rp) - e0 * torch.complex(-rz, k * R0 * rz)
            gd = ep / Rp - e0 / R0
            total = (wj * ((Pq - P0 * c - D0 * f) * dd - gd * (Dq + P0 * (k * sn * nn) - D0 * (c * nn)))).sum(dim=1)
            out[i, at] = P0[:, 0] + total / (4 * math.pi)
    return out


def _synthesised(T, midx, spectrum, nt):
    """[P][M][nt] of (1/nt) sum w Re(S T exp(-2 pi i m n / nt))."""
    out = []
    for row in spectrum:
        full = torch.zeros((T.shape[1], nt // 2 + 1), dtype=torch.complex128, device=T.device)
        full[:, torch.as_tensor(midx, device=T.device)] = (row[torch.as_tensor(midx, device=T.device), None] * T).T
        out.append(torch.fft.irfft(full.conj().resolve_conj(), n=nt, dim=1))
    return torch.stack(out)


def exact(case, seed):
    c = case
    n, q = _sizes(c)
    seconds = 0.0
    if c["kind"] in ("solve", "async", "multi", "whole"):
        seconds += c["nk"] * (n * q * 1e-9 + n ** 3 * 4.5e-12)
    if c["kind"] in ("field", "picked", "whole"):
        seconds += c.get("keep", c["nk"]) * c["m"] * q * 9e-10
    if seconds > 20.0:
        return None  # would take longer
    s = _inputs(c, seed)
    kind = c["kind"]
    if kind == "multi":
        return _solutions(s["mesh"], s["k"], s["dirs"])
    if kind in ("solve", "async"):
        return _solutions(s["mesh"], s["k"], s["dir"][None])[:, 0]
    # S_m = sum s_n exp(+2 pi i m n / nt)
    spectrum = torch.fft.rfft(s["s"], dim=1).conj().resolve_conj()
    if kind == "pulses":
        return _synthesised(s["T"], s["midx"], spectrum, c["nt"])
    out, k, midx = {}, s["k"], s["midx"]
    if kind == "whole":
        out["surf"] = surf = _solutions(s["mesh"], k, s["dir"][None])[:, 0]
    else:
        surf = s["surf"]
    if kind == "picked":
        amp = spectrum.abs().amax(dim=0).cpu().numpy()
        midx = np.sort(np.lexsort((np.arange(amp.size), -amp))[:c["keep"]]).astype(np.int64)
        midx = midx[midx < c["nk"]]
        k, surf = s["dk"] * midx.astype(np.float64), surf[torch.as_tensor(midx, device=surf.device)]
        out["midx"] = None  # whole numbers
    field = _fields(s["mesh"], s["xobs"], k, surf)
    out["p"] = _synthesised(field, midx, spectrum, c["nt"])
    return out
