"""The tensor-memory accesses' preconditions, read off the source.

tcgen05.{ld,st,wait}.sync.aligned are instructions of a whole warp: one that
its threads reach in different groups is undefined, whatever a compiler makes of
it, so every access reconverges the warp first.  The deallocation comes after
every thread's accesses: wait, fence, barrier, fence."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_10987_gb300", "csrc")


def _source():
    with open(os.path.join(CSRC, "hydro_tmem.cuh")) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _body(src, name):
    """The body of the one function `name` defines."""
    m = re.search(r"\b%s\([^)]*\)\s*(?:const\s*)?\{" % name, src)
    assert m, name
    depth, i = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
    return src[m.end():i - 1]


@pytest.mark.parametrize("name", ["next", "record", "store", "tmem_free"])
def test_accesses_reconverge_first(name):
    body = _body(_source(), name)
    first = re.search(r"tcgen05\.\S*\.sync\.aligned", body)
    assert first and "__syncwarp();" in body[:first.start()]


def test_deallocation_is_fenced():
    body = _body(_source(), "tmem_free")
    order = ["tcgen05.wait::st", "tcgen05.fence::before_thread_sync", "__syncthreads();",
             "tcgen05.fence::after_thread_sync", "tcgen05.dealloc"]
    at = [body.find(x) for x in order]
    assert -1 not in at and at == sorted(at)


def test_no_other_file_touches_tensor_memory():
    for f in os.listdir(CSRC):
        if f.endswith((".cu", ".cuh")) and f != "hydro_tmem.cuh":
            with open(os.path.join(CSRC, f)) as s:
                assert not re.search(r"asm[^;]*tcgen05", s.read()), f


def test_predictions_reconverge_between_the_guarded_loads_and_the_matrix_instructions():
    """mma.sync.aligned is an instruction of a whole warp too; the predictions'
    loads are guarded per lane (the padding columns)."""
    with open(os.path.join(CSRC, "hydro_gate.cu")) as f:
        body = _body(re.sub(r"//[^\n]*", "", f.read()), "hydro_mlp_forward_kernel")
    guard, sync, mma = body.find("if (c < kGateIn)"), body.find("__syncwarp();"), body.find("mma_bf16_16816(")
    assert 0 <= guard < sync < mma
