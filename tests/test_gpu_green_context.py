"""The FP64 step on a stream that owns part of the SMs (a green context): its
teams of CTAs wait for one another, so they have to fit what the stream has.
Eager and captured steps give the bits of the ordinary stream."""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")

from paper_2107_10987_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
SM, DEFAULT_STREAM, NON_BLOCKING = 1, 1, 1  # CU_DEV_RESOURCE_TYPE_SM, CU_GREEN_CTX_DEFAULT_STREAM, ...


class Resource(C.Structure):  # CUdevResource
    _fields_ = [("type", C.c_int), ("pad", C.c_ubyte * 92), ("sm", C.c_uint * 3), ("rest", C.c_ubyte * 148)]


@pytest.fixture(scope="module")
def green_stream():
    """A stream of a green context of 16 SMs."""
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")

    def call(name, *args):
        if getattr(cu, name)(*args):
            pytest.skip(f"{name}: green contexts are not to be had here")

    dev, all_sms, part, rest = C.c_int(), Resource(), Resource(), Resource()
    n, desc, ctx, stream = C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
    call("cuCtxGetDevice", C.byref(dev))
    call("cuDeviceGetDevResource", dev, C.byref(all_sms), SM)
    call("cuDevSmResourceSplitByCount", C.byref(part), C.byref(n), C.byref(all_sms), C.byref(rest), 0, 16)
    call("cuDevResourceGenerateDesc", C.byref(desc), C.byref(part), 1)
    call("cuGreenCtxCreate", C.byref(ctx), desc, dev, DEFAULT_STREAM)
    call("cuGreenCtxStreamCreate", C.byref(stream), ctx, NON_BLOCKING, 0)
    assert part.sm[0] < all_sms.sm[0]
    yield torch.cuda.ExternalStream(stream.value)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("n", [1, 3, 40])
@pytest.mark.parametrize("how", ["eager", "capture"])
def test_step_on_a_green_stream(green_stream, n, how):
    from paper_2107_10987_gb300 import hydro as H

    U = torch.tensor(W.random_subgrids(n, 5, 5 / 3), device="cuda")
    o = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    h = torch.full((n,), 0.05, dtype=torch.float64, device="cuda")
    ctx = H.Context(5 / 3, 0.2)
    H.hydro_set_mode(ctx, H.HYDRO_PREC_FP64)
    B = H.make_batch(U, o, h)

    def outputs():
        return (torch.full((n, 10, 8, 8, 8), float("nan"), dtype=torch.float64, device="cuda"),
                torch.full((n,), float("nan"), dtype=torch.float64, device="cuda"))

    want, got = outputs(), outputs()
    H.hydro_step(ctx, B, 0.0, *want)
    torch.cuda.synchronize()
    if how == "eager":
        H.hydro_step(ctx, B, 0.0, *got, stream=green_stream)
    else:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=green_stream):
            H.hydro_step(ctx, B, 0.0, *got)
        with torch.cuda.stream(green_stream):
            graph.replay()
    green_stream.synchronize()
    assert H.hydro_status(ctx) == 0
    for x, y in zip(got, want):
        assert torch.equal(x.view(torch.int64), y.view(torch.int64))
