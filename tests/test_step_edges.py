"""What a step does at its edges: shared memory handed between the lanes of a
warp, settings changed between batch steps, cells of any aspect ratio,
NaN fractions, what the positioning's stop leaves of an offset,
wisps in cells along the mesh,
a band beyond the queue of clip jobs,
a context made, or a network attached, where memory is short, network outputs
written over their inputs.

FP64 is held to the replay tolerance against the oracle (1e-11).
"""
import os
import re

import numpy as np
import pytest

from paper_1305_3417_gb300 import inputs as I

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1305_3417_gb300", "csrc")


def test_queue_write_waits_for_its_shared_inputs():
    """The pair stage's lanes write the queue from what other lanes have put
    into shared memory (candidate map, job codes): a warp barrier lies between
    (shuffles and ballots do not order shared memory).  Read from the source: a
    missing barrier shows in no result that could be waited for."""
    src = open(os.path.join(SRC, "vof_phase_flux.cu")).read()
    body = src[src.index("void pf_pairs_body("):src.index("struct __align__(16) ClipShared")]
    body = re.sub(r"//[^\n]*", "", body)
    stored = body.index("sh.Kmap[__popc(used & lt)] =")
    for read in ("sh.Kmap[i / 5]", "sh.Kmap[lane]", "sh.Q[i]"):
        first = body.index(read)
        assert first > stored and "__syncwarp();" in body[stored:first], read


def test_marks_move_on_before_the_redistribution():
    """The numbers that the redistribution marks cells with move on where a
    step's (an update's) counters are cleared, not at its end, which a launch
    whose waits ran out does not reach: its marks would be taken for the next
    step's own and their cells left out.  Read from the source: no wait runs out
    in a sound step."""
    src = open(os.path.join(SRC, "vof_kernels.cu")).read()

    def body(name):
        i = src.index(name)
        return src[i:src.index("\n}\n", i)]
    for kernel in ("void k_point_state(", "void k_zero_update("):
        assert "cnt[CNT_EPOCH]" in body(kernel) and "EPOCH_STEP" in body(kernel)
    step = body("k_bound_step(DevMesh m, BoundStep a)")
    assert "*a.epoch" in step and not re.search(r"\*a\.epoch\s*=[^=]", step)
    assert "EPOCH_STEP = BOUND_PASSES_MAX + 2" in src       # a launch's marks: one a pass, and the segments'


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1305_3417_gb300 import build
    build.build()
    return torch


def T(torch, x):
    return torch.from_numpy(np.ascontiguousarray(x).reshape(-1).copy()).cuda()


@pytest.mark.gpu
@pytest.mark.parametrize("what", ["gradient", "count", "guess"])
def test_batch_follows_its_context(torch, what):
    """A setting of the batch's context changed between two steps on the same
    arrays holds from the next step on, as it does for direct steps: bit for
    bit.  Networks are detached and destroyed, and larger ones attached, between
    the steps."""
    from paper_1305_3417_gb300 import mlp, vof
    b = I.make_batch(4, seed=1304, hex_range=(8, 10), tet_range=(5, 6), steps=3)
    B = vof.VofBatch(b, precision=1)
    ctx = B.context()
    U, F = T(torch, b.U_dt), T(torch, b.F_dt)
    s, a = T(torch, b.alpha0), T(torch, b.alpha0)
    seen = []

    def step():
        s.copy_(T(torch, b.alpha0))
        a.copy_(s)
        vof.vof_work_counts(ctx)
        B.advect(s, U, F)
        counted = vof.vof_work_counts(ctx)
        vof.vof_advect(ctx, a, U, F, 1.0)
        torch.cuda.synchronize()
        assert torch.equal(s, a)
        # where the iterations differ, so do they in the batch's step
        assert counted == vof.vof_work_counts(ctx)
        seen.append((s.clone(), counted["fill32"], counted["faces"]))

    step()
    if what == "gradient":
        for kind in (vof.GRAD_LSQ, vof.GRAD_NAG):
            vof.vof_set_gradient(ctx, kind)
            step()
        assert not torch.equal(seen[0][0], seen[1][0]) and torch.equal(seen[0][0], seen[2][0])
    elif what == "count":
        for on in (True, False):
            vof.vof_count_work(ctx, on)
            step()
        assert [x[2] > 0 for x in seen] == [False, True, False]
    else:
        vof.vof_count_work(ctx, True)
        step()
        net = None
        for k, cap in enumerate((1 << 12, 1 << 14)):   # (more than the interface cells)
            old, net = net, vof.Mlp(mlp.init_params(5 + k), max_batch=cap)
            vof.vof_set_guess(ctx, net)
            if old:
                old.close()
            step()
            assert seen[-1][1] != seen[-2][1]
        vof.vof_set_guess(ctx, None)
        net.close()
        step()
        assert seen[-1][1] == seen[1][1]
    B.close()


@pytest.mark.gpu
@pytest.mark.parametrize("aspect", [1, 30, 300, 1000, 3000])
def test_sliver_along_needle_cells(torch, oracle_lib, aspect):
    """A plane just inside the far end of a sweep along needle cells: the flux is
    the sliver between the two (of phase, or of void), 3e-10 to 1e-6 cells thick,
    in the step and in its stages called one by one."""
    from paper_1305_3417_gb300 import vof
    n = (6, 3, 3)
    m = I.hex_mesh(n, (6.0, 3.0 / aspect, 3.0 / aspect), periodic="xyz")
    om = oracle_lib.OracleMesh(m)
    F = np.asarray(om.geometry()[3]).reshape(3, -1)[0]      # u = (1, 0, 0)
    U = np.zeros((3, m.n_cells))
    U[0] = 1.0
    i = np.arange(m.n_cells) % n[0]
    ctx = vof.VofContext(m, precision=0, bound=False)
    tF, tU = T(torch, F), T(torch, U)
    Up = ctx.point_velocity(tU)
    for dt in (0.3, 0.5, 0.61, 0.97):
        lam = ctx.correct_flux(Up, tF, dt)[0]
        for thick in (3e-10, 1e-9, 3e-9, 1e-8, 3e-8, 5e-8, 1e-7, 1e-6):
            for phase in (True, False):
                a = np.where((i >= 1) & (i < 3), 1.0, 0.0)
                if phase:
                    a[i == 3] = 1.0 - dt + thick
                else:
                    a[i == 0] = dt - thick
                want, _, st = om.advect(a.copy(), U, F, dt, bound=False)
                assert st == 0
                t, b = T(torch, a), T(torch, a)
                ctx.advect(t, tU, tF, dt)
                ctx.update(b, ctx.phase_flux(b, *ctx.reconstruct(b)[:3], Up, tF, lam, dt))
                for got in (t, b):
                    assert np.abs(got.cpu().numpy() - want).max() < 1e-11, (dt, thick, phase)
    assert ctx.status() == 0
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("nz", [32, 33])            # 2^15 cells: one cluster; above: every SM
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_nan_stays_out_of_the_redistribution(torch, nz, sign):
    """A NaN fraction is neither source nor receiver of a local pass: every
    other cell comes out as if that cell were full, bit for bit; the mesh-wide
    fallback then sets it to 1 (0 with the sign bit set)."""
    from paper_1305_3417_gb300 import vof
    m = I.hex_mesh((32, 32, nz))
    rng = np.random.default_rng(nz)
    a = rng.uniform(0.2, 0.8, m.n_cells)
    a[rng.uniform(size=m.n_cells) < 0.02] = 1.01    # excess with room all around
    cells = [0, 32 * 32 * 16 + 500, m.n_cells - 1]
    Va = T(torch, np.zeros(m.n_faces))
    ctx = vof.VofContext(m)
    out = []
    for x in (1.0, np.copysign(np.nan, sign)):
        b = a.copy()
        b[cells] = x
        t = T(torch, b)
        st = ctx.update(t, Va).cpu().numpy()
        out.append((t.cpu().numpy(), int(st[vof.S["bound_passes"]])))
    ctx.close()
    (full, p0), (got, p1) = out
    assert p0 == p1 > 0 and full.max() <= 1.0 + 1e-13
    assert np.all(got[cells] == (1.0 if sign > 0 else 0.0))
    rest = np.setdiff1d(np.arange(m.n_cells), cells)
    assert np.array_equal(got[rest], full[rest])


@pytest.mark.gpu
def test_fp64_offsets_beyond_the_stop(torch, oracle_lib):
    """Alg. 1 stops at a residual of 1e-13; the offset handed out is good to the
    fill's roundings: two fill evaluations over 24 tetrahedra at a few 1e-16 of
    the cell's volume each, 1e-14 at most."""
    from paper_1305_3417_gb300 import vof
    m = I.hex_mesh((8, 8, 8), jitter=0.2, seed=5)
    rng = np.random.default_rng(11)
    a = rng.uniform(0.0, 1.0, m.n_cells)
    thin = rng.uniform(size=m.n_cells) < 0.5            # half of them nearly empty or nearly full
    a[thin] = np.where(a[thin] < 0.5, 1e-7, 1.0 - 1e-7) ** rng.uniform(0.2, 1.0, int(thin.sum()))
    om = oracle_lib.OracleMesh(m)
    vc = om.geometry()[1]
    ctx = vof.VofContext(m)
    n, d, fl = (t.cpu().numpy() for t in ctx.reconstruct(T(torch, a))[:3])
    n = n.reshape(3, -1)
    cells = np.flatnonzero(fl & oracle_lib.ORIENTED)
    assert cells.size > 400
    res = np.array([abs(om.cut_volume(c, n[:, c], d[c]) / vc[c] - a[c]) for c in cells])
    assert res.max() <= 1e-14, res.max()
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
def test_no_room_in_the_queue_changes_no_bit(torch, precision):
    """A step whose band (every face) has more clip jobs than the context's queue
    holds: the same bits from run to run, and as in a joined mesh
    with an empty case whose faces make the queue large enough."""
    from paper_1305_3417_gb300 import vof
    w = I.make_workload("deform3d", n=16)
    rest = I.hex_mesh((64, 64, 64))
    F, U, dt = w.step_inputs(1)
    a0 = np.random.default_rng(3).uniform(0.05, 0.95, w.mesh.n_cells)
    joined, off = I.concat_meshes([w.mesh, rest])[:2]
    ni = w.mesh.n_internal
    Fj = np.concatenate([F[:ni], np.zeros(rest.n_internal), F[ni:], np.zeros(rest.n_faces - rest.n_internal)])
    Uj = np.concatenate([U.reshape(3, -1), np.zeros((3, rest.n_cells))], axis=1)

    def run(h, a, u, f):
        ta, tU, tF = T(torch, a), T(torch, u), T(torch, f)
        vof.vof_count_work(h)
        out = []
        for _ in range(3):
            t = ta.clone()
            vof.vof_work_counts(h)
            vof.vof_advect(h, t, tU, tF, dt)
            out.append((t[:w.mesh.n_cells].clone(), vof.vof_work_counts(h)))
        assert vof.vof_status(h) == 0
        return out

    ctx = vof.VofContext(w.mesh, precision=precision, bound=False)
    few = run(ctx.h, a0, U, F)
    ctx.close()
    b = vof.vof_batch_create(joined, off, precision=precision, bound=False)
    all_ = run(vof.vof_batch_context(b), np.concatenate([a0, np.zeros(rest.n_cells)]), Uj, Fj)
    vof.vof_batch_destroy(b)
    # ("reserved" counts the faces without room)
    assert all(c["reserved"] > 100 for _, c in few) and all(c["reserved"] == 0 for _, c in all_)
    for t, c in few[1:] + all_:
        assert torch.equal(few[0][0], t)
        # and no face's work is done, or counted, twice
        assert {k: v for k, v in c.items() if k != "reserved"} == {k: v for k, v in few[0][1].items() if k != "reserved"}


@pytest.mark.gpu
def test_context_where_memory_is_short(torch):
    """With all but a part of what a context likes to take allocated elsewhere, a
    smaller queue serves: the same step, and memory left for the buffers that the
    caller and the least-squares gradient take afterwards."""
    from paper_1305_3417_gb300 import vof
    w = I.make_workload("deform3d", n=64)
    F, U, dt = w.step_inputs(1)
    a0 = np.random.default_rng(3).uniform(0.05, 0.95, w.mesh.n_cells)   # (every face in the band)
    tF, tU, t0 = T(torch, F), T(torch, U), T(torch, a0)

    def step():
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ctx = vof.VofContext(w.mesh, precision=1)
        took = before - torch.cuda.mem_get_info()[0]
        t = t0.clone()
        ctx.advect(t, tU, tF, dt)
        vof.vof_set_gradient(ctx.h, vof.GRAD_LSQ)
        b = t0.clone()
        ctx.advect(b, tU, tF, dt)
        assert ctx.status() == 0
        ctx.close()
        return took, t, b

    step()
    took, t, b = step()
    queue = 512 * w.mesh.n_faces                # preferred size, and 16 bytes of tables a batch of 224
    queue += 16 * (queue // 224)
    # room for the rest, 200 MB for what the step's second half takes, and parts of a queue
    for part in (0.9, 0.5, 0.0):
        leave = took - queue + (200 << 20) + int(part * queue)
        torch.cuda.empty_cache()
        hog = torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")
        try:
            less, u, v = step()
        finally:
            del hog
            torch.cuda.empty_cache()
        assert less < took - queue // 4
        assert torch.equal(t, u) and torch.equal(b, v)


@pytest.mark.gpu
@pytest.mark.parametrize("at", [0, 29 * 12801])      # over the first rows, or the last ones
def test_forward_over_its_own_features(torch, at):
    """More tiles than blocks; the same bits as into a buffer of its own."""
    from paper_1305_3417_gb300 import mlp, vof
    n = 12801
    net = vof.Mlp(mlp.init_params(3), max_batch=n)
    feat = torch.rand((n, vof.MLP_IN), generator=torch.Generator().manual_seed(1)).cuda()
    want = net.forward(feat)
    flat = feat.reshape(-1).clone()
    out = flat[at:at + n * vof.MLP_OUT]
    assert vof.lib().vof_mlp_forward(net.h, vof._ptr(flat), n, vof._ptr(out), vof._stream(None)) == 0
    torch.cuda.synchronize()
    assert torch.equal(out.reshape(n, -1), want)
    net.close()


@pytest.mark.gpu
def test_network_that_finds_no_room(torch):
    """A network whose offsets' buffer cannot be had is refused, and the one
    attached before goes on as it was."""
    from paper_1305_3417_gb300 import mlp, vof
    w = I.make_workload("deform3d", n=16)
    F, U, dt = w.step_inputs(1)
    tF, tU, t0 = T(torch, F), T(torch, U), T(torch, w.alpha0)
    ctx = vof.VofContext(w.mesh, precision=1)
    nets = [vof.Mlp(mlp.init_params(k), max_batch=b) for k, b in ((1, 1 << 12), (2, 1 << 26))]
    vof.vof_set_guess(ctx.h, nets[0])
    a = t0.clone()
    ctx.advect(a, tU, tF, dt)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (128 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(vof.VofError):
            vof.vof_set_guess(ctx.h, nets[1])          # 256 MB
    finally:
        del hog
        torch.cuda.empty_cache()
    b = t0.clone()
    ctx.advect(b, tU, tF, dt)
    assert ctx.status() == 0 and torch.equal(a, b)
    ctx.close()
    for net in nets:
        net.close()


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [15, 16])
def test_wisps_along_the_mesh(torch, oracle_lib, precision, n):
    """Cells of 1.1e-9 to 1e-3 (and as much below 1) on uniform hexahedra, next to
    a boundary or to a slab, so that their normals lie along the mesh up to
    roundings: every offset converges, to the stopping residual of 1e-13 (3e-13
    with the roundings of both sides)."""
    from paper_1305_3417_gb300 import vof
    m = I.hex_mesh((n, n, n), open_sides=("x-", "x+", "y-", "y+", "z-", "z+"))
    om = oracle_lib.OracleMesh(m)
    vc = om.geometry()[1]
    rng = np.random.default_rng(n)
    ctx = vof.VofContext(m, precision=precision)
    worst = 0
    for up in (False, True):
        for layer in (False, True):
            a = np.zeros((n, n, n))                     # [z, y, x]
            if layer:
                a[:, :, :4] = 1.0
                a[:, :, 4] = 10.0 ** rng.uniform(-8.9, -3.0, (n, n))
                a[::2, ::2, 4] = 3e-9
            else:
                t = 10.0 ** np.linspace(-8.9, -3.0, 3 * (n // 3) ** 2).reshape(3, n // 3, n // 3)
                k = 3 * np.arange(n // 3) + 1
                a[np.ix_(k, k, [0])] = t[0][:, :, None]
                a[np.ix_(k, [n - 1], k)] = t[1][:, None, :]
                a[np.ix_([0], k, k)] = t[2][None]
            a = a.reshape(-1)
            if up:
                a = 1.0 - a
            nn, d, fl, it = (x.cpu().numpy() for x in ctx.reconstruct(T(torch, a)))
            nn = nn.reshape(3, -1)
            cells = np.flatnonzero(fl & oracle_lib.ORIENTED)
            assert cells.size >= 3 * (n // 3) ** 2 - 3
            assert ctx.status() == 0
            worst = max(worst, int(it[cells].max()))
            for c in cells:
                assert abs(om.cut_volume(c, nn[:, c], d[c]) / vc[c] - a[c]) <= 3e-13
    assert worst < 60                                   # Alg. 1 ends within 50; Newton well before
    ctx.close()
