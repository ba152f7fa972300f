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


@pytest.mark.parametrize("rho", [1e-308, 1e-300, 1e300, 1.7e308])
@pytest.mark.parametrize("speed", [0.0, 0.5])
def test_extreme_densities(rho, speed):
    U = _state(0, rho)
    U[(0, slice(1, 4)) + CELL] = 0.0
    U[(0, 1) + CELL] = speed * rho
    _check(U)


@pytest.mark.parametrize("rho", [1e-309, 5e-324])
def test_densities_below_the_reciprocals_range(rho):
    """The reciprocal overflows, the quotients do not: dU/dt and amax stay finite,
    and the oracle's values wherever its sound speed, a root of an
    overflowing quotient, is finite."""
    U = _state(0, rho)
    U[(0, slice(1, 4)) + CELL] = 0.0
    with np.errstate(all="ignore"):
        want, _, _ = orc.step(orc.OracleParams(gamma=GAMMA, omega=0.2), U, np.zeros((1, 3)), np.array([H_CELL]))
    fin = np.isfinite(want)
    for how, dU, am in _steps(U, 0.2):
        assert np.isfinite(dU).all() and 1e150 < am[0] < np.inf, how
        assert (np.abs(dU - want)[fin] <= 1e-12 * np.abs(want[fin]).max()).all(), how


@pytest.mark.parametrize("value", [np.inf, -np.inf])
def test_infinite_momentum_shows_in_amax(value):
    U = _state(1, value)
    with np.errstate(all="ignore"):
        want, wam, _ = orc.step(orc.OracleParams(gamma=GAMMA, omega=0.2), U, np.zeros((1, 3)), np.array([H_CELL]))
    fin = np.isfinite(want)
    assert wam[0] == np.inf
    for how, dU, am in _steps(U, 0.2):
        assert am[0] == np.inf, how
        assert np.isfinite(dU[fin]).all(), how  # nothing but what the oracle has
        assert (np.abs(dU[fin] - want[fin]) <= 1e-12 * np.abs(want[fin]).max()).all(), how


@pytest.mark.parametrize("sweep", ["rows", "planes"])
@pytest.mark.parametrize("field", [1, 5, 6, 9])
@pytest.mark.parametrize("value", [np.inf, -np.inf])
def test_infinities_in_the_mixed_form(field, value, sweep):
    """The same in FP32: the oracle's finite cells, their values to the mixed form's
    rounding (about 1e-6 of a field's largest), and an infinite momentum in amax."""
    from paper_2107_10987_gb300 import hydro as H
    U = _state(field, value)
    with np.errstate(all="ignore"):
        want, wam, _ = orc.step(orc.OracleParams(gamma=GAMMA, omega=0.2), U, np.zeros((1, 3)), np.array([H_CELL]))
    fin = np.isfinite(want)
    ctx = H.Context(GAMMA, 0.2)
    H.hydro_set_mode(ctx, H.HYDRO_PREC_MIXED)
    H.hydro_set_launch(ctx, H.HYDRO_DECOMP_ROWS if sweep == "rows" else H.HYDRO_DECOMP_PLANES, 0)
    dU = torch.zeros((1, 10, 8, 8, 8), dtype=torch.float64, device="cuda")
    am = torch.zeros(1, dtype=torch.float64, device="cuda")
    H.hydro_step(ctx, H.make_batch(torch.tensor(U, device="cuda"), torch.zeros((1, 3), dtype=torch.float64, device="cuda"),
                                   torch.full((1,), H_CELL, dtype=torch.float64, device="cuda")), 0.0, dU, am)
    torch.cuda.synchronize()
    dU, am = dU.cpu().numpy(), am.cpu().numpy()
    assert np.array_equal(np.isfinite(dU), fin)
    for k in range(10):
        f = fin[0, k]
        assert np.abs(dU[0, k][f] - want[0, k][f]).max() <= 2e-5 * max(np.abs(want[0, k][f]).max(), 1.0), k
    assert am[0] == wam[0] or abs(am[0] / wam[0] - 1.0) <= 1e-5
