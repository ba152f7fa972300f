"""The FP64 step on teams of CTAs.

A batch that does not fill whole rounds of the SMs is worked on by teams of
several CTAs per tile, which share its primitives, lines, faces and cells
through global memory.  The team size follows from the number of tiles alone,
so the counts below cover teams from the whole chip to pairs, single CTAs, and
teams that loop over several tiles.  The results may not depend on it: dU/dt,
amax and the boundary faces equal those of single CTAs (a fixed grid) bit for
bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2107_10987_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
GAMMA = 5.0 / 3.0


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2107_10987_gb300 import _build, hydro
    _build.build()
    return hydro


def _run(H, ctx, U, o, h, g, N):
    n = U.shape[0]
    dU = torch.full((n, 10, N, N, N), float("nan"), dtype=torch.float64, device="cuda")
    am = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    ff = torch.full((n, 6, 13, N, N), float("nan"), dtype=torch.float64, device="cuda")
    H.hydro_step(ctx, H.make_batch(U, o, h, g), 0.0, dU, am, ff)
    torch.cuda.synchronize()
    return dU, am, ff


@pytest.mark.parametrize("n,N,points,contact,spin", [
    (1, 8, 9, 0, 0), (2, 8, 9, 1, 0), (3, 8, 1, 0, 0), (19, 8, 9, 0, 1), (50, 8, 9, 0, 0), (77, 8, 1, 1, 1),
    (105, 8, 9, 1, 1), (152, 8, 9, 0, 0), (153, 8, 9, 0, 0), (1, 16, 9, 0, 0), (13, 16, 9, 1, 0)])
def test_teams_equal_single_ctas(H, n, N, points, contact, spin):
    U = torch.tensor(W.random_subgrids(n, 300 + n, GAMMA, N=N), device="cuda")
    rng = np.random.default_rng(n)
    o = torch.tensor(rng.uniform(-1, 1, (n, 3)), device="cuda")
    h = torch.tensor(rng.uniform(0.01, 0.1, n), device="cuda")
    g = torch.tensor(rng.normal(0, 0.1, (n, 3, N, N, N)), device="cuda")
    ctx = H.Context(GAMMA, 0.17, N=N)
    H.hydro_set_mode(ctx, H.HYDRO_PREC_FP64, flux_points=points, contact=contact, spin=spin)
    got = _run(H, ctx, U, o, h, g, N)
    again = _run(H, ctx, U, o, h, g, N)
    H.hydro_set_launch(ctx, H.HYDRO_DECOMP_AUTO, 37)
    want = _run(H, ctx, U, o, h, g, N)
    assert H.hydro_status(ctx) == 0
    for a, b, c in zip(got, want, again):
        assert torch.isfinite(b).all()
        assert torch.equal(a.view(torch.int64), b.view(torch.int64))
        assert torch.equal(c.view(torch.int64), b.view(torch.int64))


def test_teams_with_the_indicator_and_in_a_graph(H):
    """The indicator's decisions are every CTA's own; a captured step replays
    with the team's buffers of its capture.  (The random network marks blast
    cells smooth, so the states need not stay physical: bits and status bits
    are compared.)"""
    from test_gpu_fused import blast_mesh
    from paper_2107_10987_gb300.uniform import UniformRun
    U, o, h = blast_mesh(3, 2, 1)
    rng = np.random.default_rng(3)
    params = torch.tensor(rng.normal(0, 0.3, H.HYDRO_GATE_NPARAM), dtype=torch.float32, device="cuda")
    out = []
    for ctas, graph in ((0, False), (37, False), (0, True)):
        ctx = H.Context(GAMMA, 0.0)
        H.hydro_set_indicator(ctx, params, 0.5)
        H.hydro_set_launch(ctx, H.HYDRO_DECOMP_AUTO, ctas)
        run = UniformRun(ctx, U, o, h, (3, 2, 1), H.HYDRO_BC_OUTFLOW)
        for _ in range(2):
            run.step(use_graph=graph)
        torch.cuda.synchronize()
        out.append((run.interior().view(torch.int64), H.hydro_status(ctx)))
        run.close()
    for bits, status in out[1:]:
        assert torch.equal(bits, out[0][0]) and status == out[0][1]
