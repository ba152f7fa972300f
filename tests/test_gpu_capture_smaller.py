"""A stream capture of hydro_step on a batch no larger than one the context has
stepped allocates nothing: the FP64 step divides a smaller batch among more
teams of CTAs, or among the first teams at all, whose buffers are there.  The
replay gives the bits of the call outside a capture."""
import pytest

torch = pytest.importorskip("torch")

from paper_2107_10987_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first,then", [(152, 1), (512, 130), (304, 77)])
def test_capture_after_a_larger_batch(first, then):
    from paper_2107_10987_gb300 import hydro as H

    base = torch.tensor(W.random_subgrids(16, 5, 5 / 3), device="cuda")

    def batch(n):
        U = base.repeat((n + 15) // 16, 1, 1, 1, 1)[:n].contiguous()
        o = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        h = torch.full((n,), 0.05, dtype=torch.float64, device="cuda")
        out = (torch.full((n, 10, 8, 8, 8), float("nan"), dtype=torch.float64, device="cuda"),
               torch.full((n,), float("nan"), dtype=torch.float64, device="cuda"))
        return (U, o, h), H.make_batch(U, o, h), out

    keep, B, out = batch(first)
    ctx = H.Context(5 / 3, 0.2)
    H.hydro_set_mode(ctx, H.HYDRO_PREC_FP64)
    H.hydro_step(ctx, B, 0.0, *out)
    small, b, got = batch(then)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        H.hydro_step(ctx, b, 0.0, *got)
    graph.replay()
    torch.cuda.synchronize()
    _, b2, want = batch(then)
    H.hydro_step(ctx, b2, 0.0, *want)
    torch.cuda.synchronize()
    assert H.hydro_status(ctx) == 0
    for x, y in zip(got, want):
        assert torch.equal(x.view(torch.int64), y.view(torch.int64))
