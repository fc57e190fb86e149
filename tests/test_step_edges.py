"""What a step does at its edges: shared memory handed between the lanes of a
warp, settings changed between batch steps.
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
