"""Row sweeps that share the SMs (each CTA holds half of an SM's tensor memory
from start to end): two contexts on two streams give the bits that each gives
alone, at once and in turn."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2107_10987_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 153, 700])
def test_two_streams(n):
    from paper_2107_10987_gb300 import hydro as H

    rng = np.random.default_rng(n)
    base = W.random_subgrids(32, 3, 5 / 3)
    o = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    h = torch.full((n,), 0.05, dtype=torch.float64, device="cuda")
    runs = []
    for _ in range(2):
        U = torch.tensor(base[rng.integers(0, len(base), n)], device="cuda")
        ctx = H.Context(5 / 3, 0.2)
        H.hydro_set_mode(ctx, H.HYDRO_PREC_MIXED)
        H.hydro_set_launch(ctx, H.HYDRO_DECOMP_ROWS, 0)
        runs.append((ctx, H.make_batch(U, o, h), U))

    def step(run):
        dU = torch.full((n, 10, 8, 8, 8), float("nan"), dtype=torch.float64, device="cuda")
        am = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        H.hydro_step(run[0], run[1], 0.0, dU, am)
        return dU, am

    alone = []
    for r in runs:
        alone.append(step(r))
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in runs]
    for _ in range(3):
        both = []
        for r, s in zip(runs, streams):
            with torch.cuda.stream(s):
                both.append(step(r))
        torch.cuda.synchronize()
        for (dU, am), (dU0, am0) in zip(both, alone):
            assert torch.equal(dU.view(torch.int64), dU0.view(torch.int64))
            assert torch.equal(am, am0)
    for r in runs:
        assert H.hydro_status(r[0]) == 0
