"""What a step does at its edges: shared memory handed between the lanes of a
warp.
"""
import os
import re

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
