"""Performance cases of the geometric VoF framework: what a user's program has it do.

A case is a dict of plain values.  Its ``what`` names the call:

* ``step``         one time step of a simulation, ``VofContext.advect``: band
                   classification, reconstruction, flux correction, phase
                   fluxes, update and redistribution (``host``: the same step
                   through ``vof_advect_host`` from pinned host buffers);
* ``batch``        one step of many uneven cases, ``VofBatch.advect``;
* ``reconstruct``  the PLIC planes of a field, ``vof_reconstruct``;
* ``gradient``     forward and backward pass of the initial-guess network,
                   ``Mlp.gradient``, as its training loop calls it.

Meshes are those of ``inputs.make_workload``: jittered hexahedra, the periodic
one-cell-thick disc mesh, fully periodic jittered hexahedra, Kuhn tetrahedra
and 2:1 octrees.  They depend on the case alone; the volume fractions, the
velocity's strength and phase and the body's place come from the seed.  A body
is a ``sphere`` (the start of the deformation case) or a ``sheet`` (a bent thin
film, what the field has stretched the sphere into later in the run: the band
is several times larger).
"""
from __future__ import annotations

import functools
import math
import types

import numpy as np
import torch

from paper_1305_3417_gb300 import inputs as I
from paper_1305_3417_gb300 import vof

PRECISION = {"fp64": vof.FP64, "mixed": vof.MIXED}
DEV = "cuda"


# ------------------------------------------------------------------ the cases

def _step(name, mesh, nx, ny, nz, precision, body="sphere", lsq=False, host=False):
    return {"name": name, "what": "step", "mesh": mesh, "nx": nx, "ny": ny, "nz": nz,
            "precision": precision, "body": body, "lsq": lsq, "host": host}


def listed():
    return [
        # the 2D disc of the validation runs: the smallest step, launches and latency
        _step("disc2d_32_fp64", "disc2d", 32, 32, 1, "fp64"),
        # a coarse 3D run, as used to check a set-up before the production mesh
        _step("hex_24_mixed", "hex", 24, 24, 24, "mixed"),
        # an ordinary production step in the middle of a run: the body is a film
        _step("hex_64_sheet_mixed", "hex", 64, 64, 64, "mixed", body="sheet"),
        # the benchmark's own mesh: 2.1M cells, the early steps
        _step("hex_128_mixed", "hex", 128, 128, 128, "mixed"),
        # the plain FP64 form, for reference runs and convergence tables
        _step("hex_64_fp64", "hex", 64, 64, 64, "fp64"),
        # tetrahedra (half the benchmark's lattice): long stencils, triangular faces
        _step("tet_48_mixed", "tet", 48, 48, 48, "mixed"),
        # the octree (half the benchmark's base lattice): faces of 4 to 8 points,
        # cells of up to 78 tetrahedra
        _step("octree_32_mixed", "octree", 32, 32, 32, "mixed"),
        # a ragged periodic box with the least-squares normals
        _step("periodic_45x37x51_lsq_mixed", "periodic", 45, 37, 51, "mixed", lsq=True),
        # a solver that keeps its arrays on the host: transfers in the call
        _step("host_hex_64_mixed", "hex", 64, 64, 64, "mixed", host=True),
        # an ensemble: uneven hexahedral and tetrahedral cases in one graph launch
        {"name": "batch_32_mixed", "what": "batch", "cases": 32, "hex_lo": 16, "hex_hi": 40, "tet_lo": 8,
         "tet_hi": 24, "layout": 1304, "precision": "mixed"},
        # the planes alone, for output and for the mapping of an adaptive mesh
        {"name": "reconstruct_96_fp64", "what": "reconstruct", "nx": 96, "ny": 96, "nz": 96, "precision": "fp64",
         "body": "sphere"},
        # a training batch of the initial-guess network
        {"name": "gradient_4096", "what": "gradient", "samples": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choices(["hex", "disc2d", "periodic", "tet", "octree", "batch", "reconstruct", "gradient"],
                       [6, 2, 2, 3, 2, 2, 2, 1])[0]
    if what == "gradient":
        return {"what": "gradient", "samples": _log_int(rng, 64, 16384)}
    if what == "batch":
        hl, tl = rng.randint(10, 18), rng.randint(6, 9)
        return {"what": "batch", "cases": _log_int(rng, 4, 32), "hex_lo": hl, "hex_hi": rng.randint(hl + 4, 40),
                "tet_lo": tl, "tet_hi": rng.randint(tl + 4, 22), "layout": rng.randint(1, 10 ** 6),
                "precision": "mixed"}
    body = rng.choice(["sphere", "sphere", "sheet"])
    if what == "reconstruct":
        n = _log_int(rng, 16, 96)
        return {"what": "reconstruct", "nx": n, "ny": rng.randint(max(12, 3 * n // 4), n), "nz": n,
                "precision": rng.choice(["fp64", "mixed"]), "body": body}
    if what == "octree":
        n = _log_int(rng, 8, 28)
        return _unnamed(_step("", "octree", n, n, n, "mixed"))
    if what == "disc2d":
        n = _log_int(rng, 24, 200)
        return _unnamed(_step("", "disc2d", n, n, 1, rng.choice(["fp64", "mixed"])))
    precision = rng.choice(["fp64", "mixed", "mixed", "mixed"])
    hi = {"hex": 56 if precision == "fp64" else 104, "periodic": 32 if precision == "fp64" else 64,
          "tet": 20 if precision == "fp64" else 44}[what]
    n = _log_int(rng, {"hex": 14, "periodic": 12, "tet": 8}[what], hi)
    dims = [n, rng.randint(max(8, 4 * n // 5), n), rng.randint(max(8, 4 * n // 5), n)]
    rng.shuffle(dims)
    return _unnamed(_step("", what, *dims, precision, body=body, lsq=rng.random() < 0.2,
                          host=what == "hex" and rng.random() < 0.15))


def _unnamed(case):
    case.pop("name")
    return case


# ------------------------------------------------------------ meshes (no seed)

def _sizes(case):
    return tuple(int(case[k]) for k in ("nx", "ny", "nz"))


@functools.lru_cache(maxsize=64)
def _mesh(kind, nx, ny, nz):
    n = (nx, ny, nz)
    if kind == "hex":
        return I.hex_mesh(n, jitter=0.2, seed=1302)
    if kind == "open":
        return I.hex_mesh(n, open_sides=("x-", "x+", "y-", "y+", "z-", "z+"))
    if kind == "periodic":
        return I.hex_mesh(n, jitter=0.2, seed=1304, periodic="xyz")
    if kind == "disc2d":
        return I.hex_mesh(n, (1.0, 1.0, 1.0 / nx), dim=2, periodic="xy")
    if kind == "tet":
        return I.kuhn_tet_mesh(n, jitter=0.15, seed=1303)
    if kind == "open_tet":
        m = I.kuhn_tet_mesh(n)
        m.wall = np.zeros(m.n_faces - m.n_internal, np.uint8)
        return m
    return I.octree_mesh(nx, 2, (0.35, 0.35, 0.35), 0.15)


@functools.lru_cache(maxsize=64)
def _on_device(kind, nx, ny, nz):
    """(points, cell vertices, per face-point slot the edge's low and high end and its sign, 0 in the padding)."""
    m = _mesh(kind, nx, ny, nz)
    ptr = torch.from_numpy(m.face_ptr.astype(np.int64)).to(DEV)
    pts = torch.from_numpy(m.face_pts.astype(np.int64)).to(DEV)
    cnt = ptr[1:] - ptr[:-1]
    j = torch.arange(int(cnt.max()), device=DEV)[None, :]
    live = j < cnt[:, None]
    a = pts[ptr[:-1, None] + torch.where(live, j, 0)]
    b = pts[ptr[:-1, None] + torch.where(live, (j + 1) % cnt[:, None], 0)]
    sign = torch.where(a < b, 1.0, -1.0).double() * live
    return (torch.from_numpy(m.points).to(DEV), torch.from_numpy(m.cell_verts.astype(np.int64)).to(DEV),
            torch.minimum(a, b), torch.maximum(a, b), sign)


# ------------------------------------------------- fields and bodies (by seed)

def _fields(kind, rng):
    """(velocity, vector potential) of the mesh's test field, on (..., 3) tensors."""
    pi, s = math.pi, float(rng.uniform(0.7, 1.0))
    if kind == "disc2d":
        th = float(rng.uniform(0.0, 2.0 * pi))
        U = torch.tensor([s * math.cos(th), s * math.sin(th), 0.0], dtype=torch.float64, device=DEV)
        return lambda x: U.expand(x.shape), lambda x: 0.5 * torch.linalg.cross(U.expand(x.shape), x)
    if kind == "periodic":
        def u(x):
            return s * torch.sin(2 * pi * x[..., [1, 2, 0]])

        def A(x):
            return -s * torch.cos(2 * pi * x[..., [2, 0, 1]]) / (2 * pi)
        return u, A
    if kind == "tet":                                  # the single vortex
        def u(x):
            X, Y = pi * x[..., 0], pi * x[..., 1]
            return s * torch.stack([-torch.sin(X) ** 2 * torch.sin(2 * Y), torch.sin(2 * X) * torch.sin(Y) ** 2,
                                    torch.zeros_like(X)], -1)

        def A(x):
            X, Y = pi * x[..., 0], pi * x[..., 1]
            z = torch.zeros_like(X)
            return torch.stack([z, z, -(s / pi) * torch.sin(X) ** 2 * torch.sin(Y) ** 2], -1)
        return u, A
    if kind in ("open", "open_tet"):                   # solid-body rotation, |u| <= s on the box
        w = rng.normal(size=3)
        w = torch.from_numpy(w * (s / (np.linalg.norm(w) * 0.5 * math.sqrt(3.0)))).to(DEV)
        return (lambda x: torch.linalg.cross(w.expand(x.shape), x - 0.5),
                lambda x: -0.5 * ((x - 0.5) ** 2).sum(-1, keepdim=True) * w)

    def u(x):                                          # the deformation case
        X, Y, Z = pi * x[..., 0], pi * x[..., 1], pi * x[..., 2]
        return s * torch.stack([2 * torch.sin(X) ** 2 * torch.sin(2 * Y) * torch.sin(2 * Z),
                                -torch.sin(2 * X) * torch.sin(Y) ** 2 * torch.sin(2 * Z),
                                -torch.sin(2 * X) * torch.sin(2 * Y) * torch.sin(Z) ** 2], -1)

    def A(x):
        X, Y, Z = pi * x[..., 0], pi * x[..., 1], pi * x[..., 2]
        q = (s / pi) * torch.sin(X) ** 2
        return torch.stack([torch.zeros_like(X), -q * torch.sin(2 * Y) * torch.sin(Z) ** 2,
                            q * torch.sin(Y) ** 2 * torch.sin(2 * Z)], -1)
    return u, A


def _body(kind, body, rng):
    """Signed distance (about) to the body, negative inside, and |gradient| <= 1.3."""
    r = rng.uniform(-1.0, 1.0, 4)
    if kind == "disc2d":
        c = torch.tensor([0.5 + 0.3 * r[0], 0.5 + 0.3 * r[1]], dtype=torch.float64, device=DEV)
        return lambda x: torch.linalg.vector_norm(_wrap(x[..., :2] - c), dim=-1) - (0.15 + 0.01 * r[3])
    if body == "sheet":
        c = torch.tensor([0.5 + 0.05 * r[0], 0.5 + 0.05 * r[1]], dtype=torch.float64, device=DEV)
        z0, ph, w = 0.5 + 0.05 * r[2], math.pi * r[3], 0.04

        def sdf(x):
            q = x[..., :2] - c
            mid = z0 + 0.1 * torch.sin(2 * math.pi * x[..., 0] + ph) * torch.cos(2 * math.pi * x[..., 1])
            return torch.maximum((x[..., 2] - mid).abs() - 0.5 * w, torch.linalg.vector_norm(q, dim=-1) - 0.35)
        return sdf
    if kind == "octree":                               # inside the refined shell
        c, R = 0.35 + 0.004 * r[:3], 0.15
    elif kind == "periodic":                           # across the seams
        c, R = np.array([0.9, 0.15, 0.5]) + 0.1 * r[:3], 0.25 + 0.01 * r[3]
    elif kind == "tet":
        c, R = np.array([0.5, 0.75, 0.0]) + [0.02 * r[0], 0.02 * r[1], 0.0], 0.15 + 0.005 * r[3]
        c2 = torch.from_numpy(c[:2].copy()).to(DEV)
        return lambda x: torch.linalg.vector_norm(x[..., :2] - c2, dim=-1) - R
    elif kind in ("open", "open_tet"):
        c, R = 0.5 + 0.15 * r[:3], 0.17 + 0.06 * r[3]
    else:
        c, R = 0.35 + 0.05 * r[:3], 0.15 + 0.005 * r[3]
    ct = torch.from_numpy(np.asarray(c, float)).to(DEV)
    if kind == "periodic":
        return lambda x: torch.linalg.vector_norm(_wrap(x - ct), dim=-1) - R
    return lambda x: torch.linalg.vector_norm(x - ct, dim=-1) - R


def _wrap(d):
    return d - torch.round(d)


def _fractions(dev, sdf, m=4):
    """Volume fractions: each cell near the surface sampled at m^3 (tetrahedra: as many) points
    of its parametrisation, each the middle of a small box that the surface cuts about linearly."""
    P, cv = dev[0], dev[1]
    X = P[cv]
    cen = X.mean(1)
    rad = torch.linalg.vector_norm(X - cen[:, None], dim=-1).amax(1)
    d = sdf(cen)
    out = (d < 0).double()
    near = torch.nonzero(d.abs() <= 1.4 * rad)[:, 0]
    g = (torch.arange(m, device=DEV, dtype=torch.float64) + 0.5) / m
    xi = torch.cartesian_prod(g, g, g)
    if cv.shape[1] == 8:
        lo = 1.0 - xi
        f = [(xi if c else lo) for c in (0, 1)]
        corner = [(0, 0, 0), (1, 0, 0), (1, 1, 0), (0, 1, 0), (0, 0, 1), (1, 0, 1), (1, 1, 1), (0, 1, 1)]
        N = torch.stack([f[a][:, 0] * f[b][:, 1] * f[c][:, 2] for a, b, c in corner], 1)
    else:
        t = torch.sort(xi, dim=1, descending=True)[0]
        N = torch.stack([1 - t[:, 0], t[:, 0] - t[:, 1], t[:, 1] - t[:, 2], t[:, 2]], 1)
    for part in near.split(1 << 16):
        x = (N[None, :, :, None] * X[part][:, None]).sum(2)
        w = (2.0 / m) * rad[part][:, None]
        f = torch.clamp(0.5 - sdf(x) / w, 0.0, 1.0).mean(1)
        # slivers and wisps: every other nearly empty or nearly full cell holds
        # (lacks) much less than its share, down to 1e-8
        thin = torch.where(part % 2 == 0, 10.0 ** (-6.0 * torch.frac(part * 0.6180339887498949)), 1.0)
        f = torch.where(f < 0.02, f * thin, torch.where(f > 0.98, 1.0 - (1.0 - f) * thin, f))
        out[part] = f
    return out


def _inputs(kind, sizes, body, seed, co):
    """(alpha, U [3 x cells], F, dt) of one step, on the device."""
    rng = np.random.default_rng([int(seed), 17])
    dev = _on_device(kind, *sizes)
    mesh = _mesh(kind, *sizes)
    u, A = _fields(kind, rng)
    alpha = _fractions(dev, _body(kind, body, rng))
    P, cv, lo, hi, sign = dev
    U = u(P[cv].mean(1)).T.contiguous()
    # circulation of the potential round each face: 4-point Gauss-Legendre per
    # edge, from its lower to its higher point for both its faces
    x, wx = np.polynomial.legendre.leggauss(4)
    F = torch.empty(lo.shape[0], dtype=torch.float64, device=DEV)
    for a in range(0, lo.shape[0], 1 << 20):
        sl = slice(a, a + (1 << 20))
        p0 = P[lo[sl]]
        e = P[hi[sl]] - p0
        acc = torch.zeros(p0.shape[:-1], dtype=torch.float64, device=DEV)
        for t, w in zip(x, wx):
            acc += (0.5 * float(w)) * (A(p0 + 0.5 * (float(t) + 1.0) * e) * e).sum(-1)
        F[sl] = (acc * sign[sl]).sum(1)
    h = mesh.h if mesh.kind == "octree" else 1.0 / max(sizes)
    if mesh.kind == "tet":
        h /= 6.0 ** (1.0 / 3.0)
    speed = {"hex": 2.0, "octree": 2.0, "periodic": math.sqrt(3.0)}.get(kind, 1.0)  # the fields' largest
    return alpha, U, F, co * h / speed


# ---------------------------------------------------------------------- cases

def _batch_layout(case):
    rng = np.random.default_rng([int(case["layout"]), 5])
    out = []
    for i in range(int(case["cases"])):
        kind, lo, hi = ("open", "hex_lo", "hex_hi") if i % 2 == 0 else ("open_tet", "tet_lo", "tet_hi")
        n = int(rng.integers(int(case[lo]), int(case[hi]) + 1))
        out.append((kind, (n, n, n), float(rng.uniform(0.3, 0.8))))
    return out


@functools.lru_cache(maxsize=8)
def _joined(layout):
    return I.concat_meshes([_mesh(kind, *sizes) for kind, sizes, _ in layout])


def prepare(case, seed):
    if case["what"] == "gradient":
        return _prepare_gradient(int(case["samples"]), int(seed))
    if case["what"] == "batch":
        layout = _batch_layout(case)
        mesh, cells, _ = _joined(tuple(layout))
        ins = [_inputs(kind, sizes, "sphere", int(seed) * 1009 + i, co)
               for i, (kind, sizes, co) in enumerate(layout)]
        ni = [_mesh(kind, *sizes).n_internal for kind, sizes, _ in layout]
        F = torch.cat([x[2][:k] * x[3] for x, k in zip(ins, ni)] + [x[2][k:] * x[3] for x, k in zip(ins, ni)])
        U = torch.cat([x[1] * x[3] for x in ins], 1).reshape(-1).contiguous()
        alpha0 = torch.cat([x[0] for x in ins])
        batch = vof.VofBatch(types.SimpleNamespace(mesh=mesh, cases=layout, cell_off=cells),
                             precision=PRECISION[case["precision"]])
        return {"what": "batch", "ctx": batch, "alpha0": alpha0, "alpha": alpha0.clone(), "U": U, "F": F,
                "mass": torch.zeros(len(layout), dtype=torch.float64, device=DEV)}
    sizes = _sizes(case)
    if case["what"] == "reconstruct":
        mesh = _mesh("hex", *sizes)
        rng = np.random.default_rng([int(seed), 17])
        alpha = _fractions(_on_device("hex", *sizes), _body("hex", case["body"], rng))
        nc = mesh.n_cells
        return {"what": "reconstruct", "ctx": vof.VofContext(mesh, precision=PRECISION[case["precision"]]),
                "alpha": alpha, "n": torch.zeros(3 * nc, dtype=torch.float64, device=DEV),
                "d": torch.zeros(nc, dtype=torch.float64, device=DEV),
                "flags": torch.zeros(nc, dtype=torch.uint8, device=DEV)}
    kind = case["mesh"]
    alpha0, U, F, dt = _inputs(kind, sizes, case["body"], seed, 0.5)
    ctx = vof.VofContext(_mesh(kind, *sizes), precision=PRECISION[case["precision"]])
    if case["lsq"]:
        vof.vof_set_gradient(ctx.h, vof.GRAD_LSQ)
    st = {"what": "host" if case["host"] else "step", "ctx": ctx, "dt": dt}
    if case["host"]:
        st.update(alpha0=alpha0.cpu(), alpha=alpha0.cpu().pin_memory(), U=U.cpu().reshape(-1).pin_memory(),
                  F=F.cpu().pin_memory(), stats=torch.zeros(vof.S_LEN, dtype=torch.float64).pin_memory())
    else:
        st.update(alpha0=alpha0, alpha=alpha0.clone(), U=U.reshape(-1), F=F,
                  stats=torch.zeros(vof.S_LEN, dtype=torch.float64, device=DEV))
    return st


def run(state):
    """One pass.  A step works in place on the state's volume fractions, as in
    a time loop; they are set back first, so that every pass is the same step."""
    what = state["what"]
    if what == "gradient":
        loss, grad = state["net"].gradient(state["feat"], state["target"])
        return {"loss": loss, "grad": grad}
    ctx = state["ctx"]
    if what == "reconstruct":
        vof.vof_reconstruct(ctx.h, state["alpha"], state["n"], state["d"], state["flags"])
        return {"n": state["n"], "d": state["d"], "flags": state["flags"]}
    alpha = state["alpha"]
    alpha.copy_(state["alpha0"])
    if what == "batch":
        ctx.advect(alpha, state["U"], state["F"], case_mass=state["mass"])
        return {"alpha": alpha, "mass": state["mass"]}
    if what == "host":
        vof.vof_advect_host(ctx.h, alpha, state["U"], state["F"], state["dt"], state["stats"])
        torch.cuda.current_stream().synchronize()     # the caller reads the arrays on the host
        return {"alpha": alpha}
    # (the statistics also hold the solvers' iteration counts, which are no result)
    ctx.advect(alpha, state["U"], state["F"], state["dt"], state["stats"])
    return {"alpha": alpha}


def _area(kind, body, sizes):
    if kind == "disc2d":
        return 2 * math.pi * 0.15 / sizes[0]
    if kind == "tet":
        return 2 * math.pi * 0.15
    if body == "sheet":
        return 2.3 * math.pi * 0.35 ** 2
    return 4 * math.pi * {"periodic": 0.25, "open": 0.17, "open_tet": 0.17}.get(kind, 0.15) ** 2


def _step_work(kind, body, sizes):
    """A step reads and writes every cell's fraction and reads every face's flux
    once; a face near the interface clips its flux polyhedron against the
    cells around it, about 5e4 operations (counted on the hexahedral meshes,
    which have about 13 such faces per cell-sized patch of the interface;
    tetrahedra and octrees taken the same per patch of their smaller cells)."""
    nx, ny, nz = sizes
    boxes = nx * ny * nz
    h2 = (1.0 / boxes) ** (2.0 / 3.0) if kind != "disc2d" else 1.0 / (nx * nx)
    cells, faces = boxes, 3 * boxes
    if kind in ("tet", "open_tet"):
        cells, faces, h2 = 6 * boxes, 12 * boxes, h2 / 6.0 ** (2.0 / 3.0)
    elif kind == "octree":
        cells, faces, h2 = 3 * boxes, 9 * boxes, h2 / 16.0
    return 16.0 * cells + 8.0 * faces, 13.0 * _area(kind, body, sizes) / h2 * 5e4


def work(case):
    if case["what"] == "gradient":
        n, mac = float(case["samples"]), 33 * 64 + 64 * 64 + 64 * 4
        return {"bytes": n * (33 + 4) * 4 + 2 * 4 * mac, "flops": 2 * n * (3 * mac - 33 * 64)}
    if case["what"] == "batch":
        each = [_step_work(kind, "sphere", sizes) for kind, sizes, _ in _batch_layout(case)]
        return {"bytes": sum(e[0] for e in each), "flops": sum(e[1] for e in each)}
    sizes = _sizes(case)
    if case["what"] == "reconstruct":
        # fractions in, planes and flags out; per interface cell (1.5 per
        # patch) about 15 fill evaluations of 24 tetrahedra, 30 operations each
        cells = sizes[0] * sizes[1] * sizes[2]
        patches = _area("hex", case["body"], sizes) * cells ** (2.0 / 3.0)
        return {"bytes": (8.0 + 32.0 + 1.0) * cells, "flops": 1.5 * patches * 15 * 24 * 30}
    b, f = _step_work(case["mesh"], case["body"], sizes)
    return {"bytes": b, "flops": f}


# ------------------------------------------------- the initial-guess network

_SHAPES = [(33, 64), (64,), (64, 64), (64,), (64, 4), (4,)]


def _prepare_gradient(n, seed):
    """Samples as the training set has them: the fractions of a 3x3x3 neighbourhood cut by a plane,
    near-cubic shape numbers, the plane as the target; He-uniform weights."""
    rng = np.random.default_rng([seed, 29])
    nn = rng.normal(size=(n, 3))
    nn /= np.linalg.norm(nn, axis=1, keepdims=True)
    s = rng.uniform(-0.6, 0.6, n)
    off = np.array([(i, j, k) for k in (-1, 0, 1) for j in (-1, 0, 1) for i in (-1, 0, 1)], float)
    frac = np.clip(0.5 + s[:, None] - nn @ off.T, 0.0, 1.0)
    geo = np.array([1, 1, 1, 1, 0.25, 1.0]) * rng.uniform(0.9, 1.1, (n, 6))
    feat = np.concatenate([frac, geo], 1).astype(np.float32)
    target = np.concatenate([nn, 0.5 + s[:, None]], 1).astype(np.float32)
    params = np.concatenate([(rng.uniform(-1, 1, sh) * math.sqrt(6.0 / sh[0]) if len(sh) == 2
                              else 0.01 * rng.uniform(-1, 1, sh)).reshape(-1) for sh in _SHAPES]).astype(np.float32)
    return {"what": "gradient", "net": vof.Mlp(params, max_batch=max(n, 16)), "params": params,
            "feat": torch.from_numpy(feat).to(DEV), "target": torch.from_numpy(target).to(DEV)}


# ----------------------------------------------------------- 64-bit references

def _exact_gradient(n, seed):
    st = _prepare_gradient(n, seed)
    p, o = [], 0
    for sh in _SHAPES:
        k = int(np.prod(sh))
        p.append(torch.from_numpy(st["params"][o:o + k].astype(np.float64).reshape(sh)).to(DEV).requires_grad_())
        o += k
    x = st["feat"].double()
    h = torch.relu(x @ p[0] + p[1])
    h = torch.relu(h @ p[2] + p[3])
    y = h @ p[4] + p[5]
    loss = ((y - st["target"].double()) ** 2).sum() / n
    g = torch.autograd.grad(loss, p)
    return {"loss": float(loss), "grad": torch.cat([v.reshape(-1) for v in g])}


def _below(h, level):
    """Fraction of tetrahedra (cells, k) with sorted vertex values h (cells, k, 4) below each cell's level."""
    d = level[:, None]
    h0, h1, h2, h3 = h.unbind(-1)
    low = (d - h0) ** 3 / ((h1 - h0) * (h2 - h0) * (h3 - h0))
    top = 1.0 - (h3 - d) ** 3 / ((h3 - h0) * (h3 - h1) * (h3 - h2))
    a, b = (d - h0) / (h2 - h0), (d - h0) / (h3 - h0)
    c, e = (d - h1) / (h2 - h1), (d - h1) / (h3 - h1)
    mid = a * b + a * (1 - b) * e + (1 - a) * c * e
    v = torch.where(d <= h1, low, torch.where(d >= h2, top, mid))
    return torch.where(d <= h0, torch.zeros_like(v), torch.where(d >= h3, torch.ones_like(v), v))


def _exact_reconstruct(case, seed):
    """Node-averaged Gauss gradient and the plane offset by bisection, from their definitions, on the hexahedral mesh."""
    sizes = _sizes(case)
    m = _mesh("hex", *sizes)
    rng = np.random.default_rng([int(seed), 17])
    dev = _on_device("hex", *sizes)
    alpha = _fractions(dev, _body("hex", case["body"], rng))
    P, cv = dev[0], dev[1]
    nc, npnt = m.n_cells, m.n_points
    fp = torch.from_numpy(m.face_pts.astype(np.int64)).to(DEV).view(-1, 4)
    own = torch.from_numpy(m.owner.astype(np.int64)).to(DEV)
    nei = torch.from_numpy(m.neighbour.astype(np.int64)).to(DEV)
    ni = m.n_internal
    # inverse-distance point values
    cen = P[cv].mean(1)
    w = 1.0 / torch.linalg.vector_norm(P[cv] - cen[:, None], dim=-1)
    num = torch.zeros(npnt, dtype=torch.float64, device=DEV).index_add_(0, cv.reshape(-1), (w * alpha[:, None]).reshape(-1))
    den = torch.zeros(npnt, dtype=torch.float64, device=DEV).index_add_(0, cv.reshape(-1), w.reshape(-1))
    phi = (num / den)[fp]
    # face values, area weighted over the fan about the point mean
    X = P[fp]
    fc = X.mean(1)
    a, b = X - fc[:, None], torch.roll(X, -1, 1) - fc[:, None]
    tri = 0.5 * torch.linalg.cross(a, b)
    S, ar = tri.sum(1), torch.linalg.vector_norm(tri, dim=-1)
    val = (ar * (phi.mean(1, keepdim=True) + phi + torch.roll(phi, -1, 1)) / 3.0).sum(1) / ar.sum(1)
    flux = S * val[:, None]
    g = torch.zeros(nc, 3, dtype=torch.float64, device=DEV).index_add_(0, own, flux).index_add_(0, nei, -flux[:ni])
    # the faces of each cell, as the outward fans that make its tetrahedra
    code = torch.cat([own * 2, nei * 2 + 1])
    face = torch.cat([torch.arange(fp.shape[0], device=DEV), torch.arange(ni, device=DEV)])
    order = torch.argsort(code // 2, stable=True)
    cf, side = face[order].view(nc, 6), (code[order] % 2).view(nc, 6)
    eps = 1e-9
    cells = torch.nonzero((alpha > eps) & (alpha < 1.0 - eps))[:, 0]
    n = torch.zeros(3, nc, dtype=torch.float64, device=DEV)
    dd = torch.zeros(nc, dtype=torch.float64, device=DEV)
    flags = torch.where(alpha >= 1.0 - eps, 4, 0).to(torch.uint8)
    for part in cells.split(1 << 15):
        c = cen[part]
        f = cf[part]
        c0, t1 = fc[f][:, :, None].expand(-1, -1, 4, -1), X[f]
        t2 = torch.roll(t1, -1, 2)
        vol = (torch.linalg.cross(t1 - c0, t2 - c0) * (c0 - c[:, None, None])).sum(-1) / 6.0
        vol = (vol * torch.where(side[part] == 0, 1.0, -1.0)[:, :, None]).reshape(part.numel(), 24)
        V = vol.sum(1)
        nn = -g[part] / torch.linalg.vector_norm(g[part], dim=-1, keepdim=True)
        verts = torch.stack([c[:, None, None].expand_as(t1), c0, t1, t2], -2).reshape(part.numel(), 24, 4, 3)
        h = torch.sort((verts * nn[:, None, None]).sum(-1), dim=-1)[0]
        lo, hi = h.amin((1, 2)), h.amax((1, 2))
        for _ in range(64):
            mid = 0.5 * (lo + hi)
            fill = (vol * _below(h, mid)).sum(1) / V
            up = fill < alpha[part]
            lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
        n[:, part] = nn.T
        dd[part] = 0.5 * (lo + hi)
        flags[part] = 3
    return {"n": n.reshape(-1), "d": dd, "flags": flags}


def exact(case, seed):
    """The network's gradient and the planes; a whole step's clipping has no short 64-bit form."""
    if case["what"] == "gradient":
        return _exact_gradient(int(case["samples"]), int(seed))
    if case["what"] == "reconstruct":
        return _exact_reconstruct(case, seed)
    return None
