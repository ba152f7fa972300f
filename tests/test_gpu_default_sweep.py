"""Which sweep the mixed step takes by default, read off a captured graph's
kernel nodes (640 threads: planes, 192: rows): planes for at most one tile per
SM with nine flux points per face, rows for more, for the single-point face flux
and for the indicator."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2107_10987_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
PLANES, ROWS = 640, 192


class KernelNode(C.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def _blocks(call):
    """The block sizes of the kernels that `call` launches on the current stream."""
    cu = C.CDLL("libcuda.so.1")

    def ok(name, *args):
        assert getattr(cu, name)(*args) == 0, name

    stream = torch.cuda.Stream()
    st, graph, n = C.c_void_p(stream.cuda_stream), C.c_void_p(), C.c_size_t()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        ok("cuStreamBeginCapture_v2", st, 1)  # thread-local
        call()
        ok("cuStreamEndCapture", st, C.byref(graph))
    ok("cuGraphGetNodes", graph, None, C.byref(n))
    nodes = (C.c_void_p * n.value)()
    ok("cuGraphGetNodes", graph, nodes, C.byref(n))
    out = []
    for node in nodes:
        kind, p = C.c_int(), KernelNode()
        ok("cuGraphNodeGetType", C.c_void_p(node), C.byref(kind))
        if kind.value == 0:
            ok("cuGraphKernelNodeGetParams_v2", C.c_void_p(node), C.byref(p))
            out.append(p.block[0] * p.block[1] * p.block[2])
    ok("cuGraphDestroy", graph)
    return out


@pytest.mark.parametrize("N", [8, 16])
@pytest.mark.parametrize("points,gate,over,want", [(9, 0, 0, PLANES), (9, 0, 1, ROWS), (1, 0, 0, ROWS), (1, 0, 1, ROWS),
                                                   (9, 1, 0, ROWS)])
def test_step(N, points, gate, over, want):
    from paper_2107_10987_gb300 import hydro as H

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per = (N // 8) ** 3
    for n in ((sms // per + 1,) if over else (1, sms // per)):
        U = torch.zeros((n, 10, N + 6, N + 6, N + 6), dtype=torch.float64, device="cuda")
        o = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        h = torch.ones(n, dtype=torch.float64, device="cuda")
        dU = torch.empty((n, 10, N, N, N), dtype=torch.float64, device="cuda")
        am = torch.empty(n, dtype=torch.float64, device="cuda")
        ctx = H.Context(5 / 3, 0.0, N=N)
        H.hydro_set_mode(ctx, H.HYDRO_PREC_MIXED, flux_points=points)
        if gate:
            H.hydro_set_indicator(ctx, torch.zeros(H.HYDRO_GATE_NPARAM, device="cuda"), 0.5)
        B = H.make_batch(U, o, h)
        H.hydro_step(ctx, B, 0.0, dU, am)  # allocates what it needs
        assert _blocks(lambda: H.hydro_step(ctx, B, 0.0, dU, am)) == [want], n


@pytest.mark.parametrize("points,want", [(9, PLANES), (1, ROWS)])
def test_fused_step(points, want):
    from paper_2107_10987_gb300 import hydro as H
    from paper_2107_10987_gb300.uniform import UniformRun

    ctx = H.Context(5 / 3, 0.0)
    H.hydro_set_mode(ctx, H.HYDRO_PREC_MIXED, flux_points=points)
    run = UniformRun(ctx, W.random_subgrids(8, 5, 5 / 3), np.zeros((8, 3)), 0.05, 2, H.HYDRO_BC_PERIODIC, fused=True)
    run.step()
    blocks = _blocks(lambda: H.hydro_rk3_step(ctx, run.desc, run.parity))
    assert len(blocks) == 4 and blocks.count(want) == 2
    run.close()
