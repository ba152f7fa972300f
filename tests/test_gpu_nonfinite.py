"""The FP64 step around a cell whose values are infinite, NaN or too large for
PPM's squares: what reaches the other cells, and how far, is the formula's.

Each state is smooth but for one value of one cell that raises no status bit
(tracer, spin, species, momentum).  With an infinity or a large number the
comparisons decide as the oracle's do: the same cells of dU/dt are finite, with
the oracle's values there, and the same amax.  With a NaN, of either sign, no
comparison holds: the values next to the cell are NaN, and the 3 x 3 x 3 block of
cells that share a face point with it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import core as orc  # noqa: E402
from paper_2107_10987_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
GAMMA = 5.0 / 3.0
H_CELL = 0.05
CELL = (6, 7, 8)  # padded (z, y, x): interior (3, 4, 5)


def _state(field, value):
    U = W.random_subgrids(1, 7, GAMMA, smooth=True)
    U[(0, field) + CELL] = value
    return U


def _steps(U, omega, **mode):
    """dU/dt and amax of one tile by a team of CTAs, by one CTA and by the
    axis-sweep kernel."""
    from paper_2107_10987_gb300 import hydro as H
    Ud = torch.tensor(U, device="cuda")
    o = torch.zeros((1, 3), dtype=torch.float64, device="cuda")
    h = torch.full((1,), H_CELL, dtype=torch.float64, device="cuda")
    for how in ("team", "single", "static"):
        ctx = H.Context(GAMMA, omega)
        H.hydro_set_mode(ctx, H.HYDRO_PREC_FP64, **mode)
        H.hydro_set_launch(ctx, H.HYDRO_DECOMP_AUTO, 1 if how == "single" else 0)
        dU = torch.zeros((1, 10, 8, 8, 8), dtype=torch.float64, device="cuda")
        am = torch.zeros(1, dtype=torch.float64, device="cuda")
        B = H.make_batch(Ud, o, h)
        if how == "static":
            H.hydro_step_static(ctx, B, 0.0, dU, am)
        else:
            H.hydro_step(ctx, B, 0.0, dU, am)
        torch.cuda.synchronize()
        yield how, dU.cpu().numpy(), am.cpu().numpy()


def _check(U, omega=0.2, **mode):
    with np.errstate(all="ignore"):
        P = orc.OracleParams(gamma=GAMMA, omega=omega, **mode)
        want, wam, _ = orc.step(P, U, np.zeros((1, 3)), np.array([H_CELL]))
        fin = np.isfinite(want)
        scale = np.array([np.abs(want[0, k][fin[0, k]]).max() for k in range(10)]).reshape(1, 10, 1, 1, 1)
        for how, dU, am in _steps(U, omega, **mode):
            assert np.array_equal(np.isfinite(dU), fin), how
            assert (np.abs(dU / scale - want / scale)[fin] <= 1e-12).all(), how
            assert am[0] == wam[0] or abs(am[0] / wam[0] - 1.0) <= 1e-12, how


@pytest.mark.parametrize("field", [5, 6, 9])
@pytest.mark.parametrize("value", [np.inf, -np.inf, 1e308, -1e308, 1e200])
def test_infinities_and_large_values(field, value):
    _check(_state(field, value))


@pytest.mark.parametrize("value", [np.inf, -np.inf, 1e200])
def test_infinities_with_contact_steepening_and_spin(value):
    _check(_state(9, value), contact=1, spin=1)


@pytest.mark.parametrize("field", [5, 9])
@pytest.mark.parametrize("value", [np.nan, -np.nan])
def test_nan(field, value):
    block = np.zeros((10, 8, 8, 8), dtype=bool)
    z, y, x = (c - 3 for c in CELL)
    block[field, z - 1:z + 2, y - 1:y + 2, x - 1:x + 2] = True
    for how, dU, am in _steps(_state(field, value), 0.0):
        assert np.array_equal(np.isnan(dU[0]), block), how
        assert np.isfinite(dU[0][~block]).all() and np.isfinite(am).all(), how
