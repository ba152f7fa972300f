"""The step kernels' scalar helpers against the operations they stand for.

  * momenta over density: from one reciprocal with a correction inside a range of
    exponents, by division outside: the division's bits everywhere;
  * 1 / sqrt: an FP32 start y and one third-order step.  y^2 is exact, the residual
    e = 1 - x y^2 (2^-20 at most) and e y round once each, and the last fused
    step once: half an ulp, 2 x 2^-53 of the correction (2^-21 ulp) and 5/16 e^3
    (2^-62, 2^-9 ulp) make less than 0.51.  Outside FP32's exponents the
    library's function, within an ulp;
  * conversions between FP32 and FP64 on the integer pipes: the conversions' bits;
  * the dual-energy comparison with its FP32 pre-test: the FP64 decision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
TINY, MIN, MAX = 5e-324, 2.0 ** -1022, np.finfo(np.float64).max


def _run(x, y, eta=0.1):
    from paper_2107_10987_gb300 import hydro as H
    x, y = np.broadcast_arrays(np.asarray(x, dtype=np.float64), np.asarray(y, dtype=np.float64))
    out = torch.full((5 * x.size,), float("nan"), dtype=torch.float64, device="cuda")
    H.hydro_selftest_scalar(torch.tensor(x.ravel(), device="cuda"), torch.tensor(y.ravel(), device="cuda"), eta, out)
    torch.cuda.synchronize()
    return x.ravel(), y.ravel(), out.cpu().numpy().reshape(-1, 5)


def _same(got, want):
    nan = np.isnan(want)
    return np.array_equal(np.isnan(got), nan) and np.array_equal(got[~nan].view(np.int64), want[~nan].view(np.int64))


def _random(rng, n, lo, hi):
    return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n)) * rng.choice([-1.0, 1.0], n)


def _near(values):
    """The values, their neighbours and their negatives, with the specials."""
    v = np.array(values, dtype=np.float64)
    v = np.concatenate([v, np.nextafter(v, 0.0), np.nextafter(v, np.inf)])
    v = np.concatenate([v, [0.0, TINY, 3 * TINY, MIN, MAX, np.inf, np.nan, 1.0, 3.0]])
    return np.concatenate([v, -v])


def test_quotients():
    rng = np.random.default_rng(1)
    edges = _near([2.0 ** e for e in (-1074, -1024, -1021, -969, -900, -520, -500, -120, -1, 0, 119, 120, 499, 500, 519, 520,
                                   899, 900, 1021, 1023)])
    pairs = np.meshgrid(edges, edges)
    n = 300_000
    x = np.concatenate([pairs[0].ravel(), _random(rng, n, -1074, 1024), _random(rng, n, -30, 30)])
    y = np.concatenate([pairs[1].ravel(), np.abs(_random(rng, n, -1074, 1024)), np.abs(_random(rng, n, -30, 30))])
    x, y, out = _run(x, y)
    with np.errstate(all="ignore"):
        assert _same(out[:, 0], x / y)


def test_quotients_near_rounding_boundaries():
    """x = (m y + j) / 2^k exactly for a quotient m / 2 between two doubles and
    j = +-1 .. 3 units of the product: the closest that x / y comes to m / 2."""
    rng = np.random.default_rng(2)
    x, y = [], []
    while len(x) < 20_000:
        r = int(rng.integers(2 ** 52, 2 ** 53)) | 1
        for k in (52, 53, 54):
            inv = pow(r, -1, 2 ** k)
            for j in (-3, -2, -1, 1, 2, 3):
                m0 = (-j * inv) % 2 ** k
                for m in range(m0, 2 ** 54, 2 ** k):
                    s = (m * r + j) >> k
                    if m % 2 and m >= 2 ** 53 and 2 ** 50 <= s < 2 ** 53:
                        x.append(float(s))
                        y.append(float(r))
    x, y, out = _run(np.array(x), np.array(y))
    assert _same(out[:, 0], x / y)


def test_reciprocal_square_root():
    rng = np.random.default_rng(3)
    y = np.concatenate([_near([2.0 ** e for e in (-1022, -200, -127, -126, -125, 0, 1, 126, 127, 128, 200, 1023)]),
                        np.abs(_random(rng, 400_000, -126, 127)), np.abs(_random(rng, 100_000, -1074, 1024))])
    y = np.abs(y[np.isfinite(y) & (y != 0.0)])
    _, y, out = _run(np.zeros_like(y), y)
    want = 1.0 / np.sqrt(y.astype(np.longdouble))
    ulps = np.abs((out[:, 1].astype(np.longdouble) - want) / np.spacing(want.astype(np.float64)))
    inside = (y >= 2.0 ** -126) & (y < 2.0 ** 127)
    assert float(ulps[inside].max()) <= 0.51
    assert float(ulps[~inside].max()) <= 1.01


def _fp32_cases():
    rng = np.random.default_rng(4)
    f = np.concatenate([rng.integers(0, 2 ** 32, 300_000, dtype=np.uint64).astype(np.uint32).view(np.float32),
                        np.array([0, 1, 2, 0x7fffff, 0x800000, 0x800001, 0x7f7fffff, 0x7f800000, 0x3f800000],
                                 dtype=np.uint32).view(np.float32)])
    with np.errstate(all="ignore"):
        d = f.astype(np.float64)
        d = d[~np.isnan(d)]
        half = (np.nextafter(np.abs(d).astype(np.float32), np.float32(np.inf)).astype(np.float64) + np.abs(d)) / 2
    half = half[np.isfinite(half)]  # midway between two FP32 numbers, and its neighbours
    top = 2.0 ** 128 - 2.0 ** 103   # the tie that rounds to infinity
    return np.concatenate([d, half, -half, np.nextafter(half, 0.0), np.nextafter(half, np.inf),
                           _near([top, 2.0 ** -149, 2.0 ** -150, 2.0 ** -126, 2.0 ** 128, 1e300, 1e-300]),
                           _random(rng, 300_000, -160, 140), _random(rng, 100_000, -1074, 1024)])


def test_conversions():
    x = _fp32_cases()
    x, _, out = _run(x, np.ones_like(x))
    with np.errstate(all="ignore"):
        want = x.astype(np.float32).astype(np.float64)
    assert _same(out[:, 2], want)
    assert _same(out[:, 3], want)


@pytest.mark.parametrize("eta", [1e-3, 0.1, 1.0])
def test_dual_energy_comparison(eta):
    rng = np.random.default_rng(5)
    y = np.concatenate([_random(rng, 100_000, -140, 130), _random(rng, 100_000, -20, 20),
                        _near([1e-30, 1e-27, 2.0 ** -126, 2.0 ** 127, 1e300])])
    with np.errstate(all="ignore"):
        lim = eta * y
        x = [lim, np.nextafter(lim, np.inf), np.nextafter(lim, -np.inf), y, np.zeros_like(y), -y]
        x += [lim * (1.0 + s * d) for s in (1, -1) for d in (1e-12, 1e-7, 9.9e-5, 1e-4, 1.01e-4, 1e-3)]
        x = np.concatenate(x)
        y = np.tile(y, x.size // y.size)
        x, y, out = _run(x, y, eta)
        want = x > eta * y
    assert np.array_equal(out[:, 4] == 1.0, want)
