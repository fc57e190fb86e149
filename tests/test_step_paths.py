"""The step's paths by size: bands of a few faces (dealt in parts), of hundreds
and of every face (more clip jobs than the queue holds), reconstruction of few
and of many cells, redistribution in one cluster and over the whole chip,
network gradients and case masses at the edges of their tiles.

A step is compared with its stages called one by one, which take every cell and
face, and with the oracle where that is quick.  FP64: the replay tolerance
against the oracle (1e-11).  Mixed: the replay tolerance too (2e-5, from 2e-6 of
a cell volume per face on either side).
"""
import numpy as np
import pytest

from paper_1305_3417_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = {0: 1e-11, 1: 2e-5}


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1305_3417_gb300 import build
    build.build()
    return torch


def T(torch, x, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(x).reshape(-1).copy())
    return (t if dtype is None else t.to(dtype)).cuda()


def _alpha(w, n, kind):
    if kind == "all":      # every cell cut: the band is every face
        return np.random.default_rng(n).uniform(0.05, 0.95, w.mesh.n_cells)
    if kind == "one":      # one cut cell among empty ones
        a = np.zeros(w.mesh.n_cells)
        a[w.mesh.n_cells // 2 + n // 2] = 0.4
        return a
    return w.alpha0


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,kind", [(5, "one"), (6, "all"), (9, "body"), (16, "body"), (32, "body"), (32, "all")])
def test_step_equals_its_stages(torch, oracle_lib, n, kind, precision):
    from paper_1305_3417_gb300 import vof
    w = I.make_workload("deform3d", n=n)
    m = w.mesh
    F, U, dt = w.step_inputs(1)
    a0 = _alpha(w, n, kind)
    ctx = vof.VofContext(m, precision=precision, bound=False)
    tF, tU, ta = T(torch, F), T(torch, U), T(torch, a0)
    ctx.advect(ta, tU, tF, dt)
    got = ta.cpu().numpy()

    f64 = dict(dtype=torch.float64, device="cuda")
    b = T(torch, a0)
    nn, d = torch.zeros(3 * m.n_cells, **f64), torch.zeros(m.n_cells, **f64)
    fl = torch.zeros(m.n_cells, dtype=torch.uint8, device="cuda")
    Up, lam, Va = torch.zeros(3 * m.n_points, **f64), torch.zeros(m.n_faces, **f64), torch.zeros(m.n_faces, **f64)
    vof.vof_reconstruct(ctx.h, b, nn, d, fl)
    vof.vof_point_velocity(ctx.h, tU, Up)
    vof.vof_correct_flux(ctx.h, Up, tF, dt, lam)
    vof.vof_phase_flux(ctx.h, b, nn, d, fl, Up, tF, lam, dt, Va)
    vof.vof_update(ctx.h, b, Va)
    assert ctx.status() == 0
    assert np.abs(got - b.cpu().numpy()).max() < TOL[precision]
    if n <= 16:
        want, _, st = oracle_lib.OracleMesh(m).advect(a0, U, F, dt, bound=False)
        assert st == 0
        assert np.abs(got - want).max() < TOL[precision]
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", [(1, 1, 1), (31, 1, 1), (8, 4, 1), (11, 3, 1), (7, 6, 5)])
def test_reconstruct_chunk_edges(torch, oracle_lib, shape, precision):
    """Every cell is cut: the plane's fill is the cell's (3e-13, the stopping
    residual of 1e-13 on both sides and roundings), its normal the oracle's."""
    from paper_1305_3417_gb300 import vof
    m = I.hex_mesh(shape, jitter=0.1, seed=3)
    a = np.random.default_rng(7).uniform(0.02, 0.98, m.n_cells)
    om = oracle_lib.OracleMesh(m)
    on, _, ofl, _, _ = om.reconstruct(a)
    ctx = vof.VofContext(m, precision=precision)
    n, d, fl = ctx.reconstruct(T(torch, a))[:3]
    n, d, fl = n.cpu().numpy().reshape(3, -1), d.cpu().numpy(), fl.cpu().numpy()
    assert np.array_equal(fl, ofl)
    _, vc, _, _ = om.geometry()
    cells = np.flatnonzero(ofl & oracle_lib.ORIENTED)
    assert np.abs(n - np.asarray(on).reshape(3, -1))[:, cells].max(initial=0.0) < 1e-11
    for c in cells:
        assert abs(om.cut_volume(c, n[:, c], d[c]) / vc[c] - a[c]) <= 3e-13
    ctx.close()


@pytest.mark.parametrize("nz", [32, 33])            # 2^15 cells: one cluster; above: every SM
@pytest.mark.parametrize("kind", ["local", "global"])
def test_redistribution_by_size(torch, oracle_lib, nz, kind):
    """Zero fluxes.  local: room next to every excess; global: excess whose
    neighbours are full, shared over the mesh.  Sums of 3e4 terms of order one
    share at most one unit of alpha: 1e-12."""
    from paper_1305_3417_gb300 import vof
    m = I.hex_mesh((32, 32, nz))
    rng = np.random.default_rng(nz)
    if kind == "local":
        a = rng.uniform(-0.1, 1.1, m.n_cells)
    else:
        a = np.where(rng.uniform(size=m.n_cells) < 0.01, 1.05, 1.0)
        a[: 32 * 32 * 4] = 0.5
    zero = np.zeros(m.n_faces)
    want, ost, _ = oracle_lib.OracleMesh(m).update(a, zero, bound=True)
    ctx = vof.VofContext(m)
    ta = T(torch, a)
    st = ctx.update(ta, T(torch, zero)).cpu().numpy()
    assert ctx.status() == 0
    if kind == "global":
        assert st[vof.S["bound_global"]] > 0
    assert np.abs(ta.cpu().numpy() - want).max() < 1e-12
    assert st[1] == pytest.approx(ost[1], rel=1e-13)
    ctx.close()


def test_case_masses_at_segment_edges(torch):
    """Cases of 1, 255, 256, 257 and 600 cells at rest: each one's mass is its
    own cells' (1e-14: at most 600 terms)."""
    from paper_1305_3417_gb300 import vof
    meshes = [I.hex_mesh(s) for s in [(1, 1, 1), (17, 15, 1), (16, 16, 1), (257, 1, 1), (30, 20, 1)]]
    joined, off = I.concat_meshes(meshes)[:2]
    h = vof.vof_batch_create(joined, off)
    a = np.random.default_rng(1).uniform(0.0, 1.0, joined.n_cells)
    ta, mass = T(torch, a), torch.zeros(len(meshes), dtype=torch.float64, device="cuda")
    U, F = T(torch, np.zeros(3 * joined.n_cells)), T(torch, np.zeros(joined.n_faces))
    vof.vof_batch_advect(h, ta, U, F, case_mass=mass)
    torch.cuda.synchronize()
    got = mass.cpu().numpy()
    vof.vof_batch_destroy(h)
    for i, m in enumerate(meshes):
        V = 1.0 / m.n_cells
        assert got[i] == pytest.approx(V * a[off[i]:off[i + 1]].sum(), rel=1e-14)


@pytest.mark.parametrize("rows", [1, 63, 64, 65, 64 * 160 + 1])
def test_mlp_gradient_row_edges(torch, rows):
    """Rows below, at and above a tile of 64, and more tiles than SMs; samples
    whose BF16 roundings are decided, repeated: 1e-3 of the gradient's norm, the
    bound of the gradient against the reference in general."""
    from oracle import mlp_ref as M
    from paper_1305_3417_gb300 import vof
    from .test_mlp import _forward_bound, _params
    p = _params(5)
    rng = np.random.default_rng(6)
    X = rng.uniform(0.0, 1.2, (3000, M.N_IN)).astype(np.float32)
    Y = rng.normal(0.0, 1.0, (3000, M.N_OUT)).astype(np.float32)
    _, ok = _forward_bound(M, p, X.astype(np.float64))
    idx = np.resize(np.flatnonzero(ok), rows)
    X, Y = X[idx], Y[idx]
    net = vof.Mlp(p, max_batch=max(rows, 128))
    loss, g = net.gradient(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda())
    lr, gr = M.backward(p, X.astype(np.float64), Y.astype(np.float64))
    assert abs(loss - lr) <= 1e-5 * abs(lr)
    assert np.linalg.norm(g.cpu().numpy() - gr) < 1e-3 * np.linalg.norm(gr)


def test_step_under_capture(torch):
    """A captured step (its dependent launches and second stream in the graph)
    replays to the state of direct steps bit for bit."""
    from paper_1305_3417_gb300 import vof
    w = I.make_workload("deform3d", n=12)
    F, U, dt = w.step_inputs(0)
    ctx = vof.VofContext(w.mesh, precision=1)
    tF, tU = T(torch, F), T(torch, U)
    a, b = T(torch, w.alpha0), T(torch, w.alpha0)
    st = torch.zeros(vof.S_LEN, dtype=torch.float64, device="cuda")
    for _ in range(3):
        vof.vof_advect(ctx.h, a, tU, tF, dt, st)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        vof.vof_advect(ctx.h, b, tU, tF, dt, st)
    b.copy_(T(torch, w.alpha0))
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert ctx.status() == 0
    assert torch.equal(a, b)
    ctx.close()
