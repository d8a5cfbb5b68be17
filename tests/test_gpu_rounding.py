"""The integer product, square root and division round as IEEE 754 does: compared with numpy to the bit on random
operands of every exponent, exact results, exact ties, results next to the middle between two doubles, powers of two and
their neighbours, and what is left to the FP64 unit (needs a GB300)."""
import numpy as np
import pytest

from paper_2509_15117_gb300 import binding as Bd

pytestmark = pytest.mark.gpu

N = 1 << 19
SPECIAL = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -1022, 1.7976931348623157e308,
                    2.0 ** 500, 2.0 ** -500, 2.0 ** 501, 2.0 ** -501, np.nextafter(2.0 ** 500, 0), 1.0, -1.0])


def _run(op, a, b):
    torch = pytest.importorskip("torch")
    ad, bd = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (a, b))
    y, g = torch.empty_like(ad), torch.empty(len(a), dtype=torch.int32, device="cuda")
    Bd.ia_rounding_check(op, ad, bd, y, g)
    return y.cpu().numpy(), g.cpu().numpy()


def _same(y, ref):
    nan = np.isnan(ref)
    assert np.isnan(y[nan]).all()
    np.testing.assert_array_equal(y[~nan].view(np.int64), ref[~nan].view(np.int64))


def _random(rng, n, e):
    """Mantissas uniform or with few bits set, exponents up to 2^+-e."""
    m = rng.integers(1 << 52, 1 << 53, n, dtype=np.int64)
    m = np.where(rng.random(n) < 0.3, (1 << 52) | (np.int64(1) << rng.integers(0, 52, n)), m)
    m = np.where(rng.random(n) < 0.2, (1 << 53) - 1 - rng.integers(0, 4, n), m)
    return np.ldexp(m.astype(np.float64), rng.integers(-e, e + 1, n) - 52)


def _neighbours(x, rng):
    d = rng.integers(-1, 2, len(x))
    return np.where(d < 0, np.nextafter(x, 0.0), np.where(d > 0, np.nextafter(x, np.inf), x))


def test_product():
    rng = np.random.default_rng(1)
    sign = rng.choice([-1.0, 1.0], (2, N))
    a, b = _random(rng, N, 498) * sign[0], _random(rng, N, 498) * sign[1]
    # exact ties: odd factors whose product has 54 bits
    p, q = rng.integers(1 << 26, 1 << 27, (2, N), dtype=np.int64) | 1
    powers = _neighbours(np.ldexp(1.0, rng.integers(-400, 400, N)), rng)
    grid = [v.ravel() for v in np.meshgrid(SPECIAL, np.concatenate([SPECIAL, a[:50]]))]
    for x, y in ((a, b), (p.astype(np.float64), -q.astype(np.float64)), (powers, powers[::-1].copy()), (a, powers)):
        z, g = _run(0, x, y)
        assert not g.any()
        _same(z, x * y)
    for x, y in (grid, grid[::-1]):
        z, g = _run(0, x, y)
        with np.errstate(all="ignore"):
            ref = x * y
        out = (x == 0) | (y == 0) | ~np.isfinite(x) | ~np.isfinite(y)
        assert g[out].all()
        _same(z[g == 0], ref[g == 0])


def test_square_root():
    rng = np.random.default_rng(2)
    r = rng.integers(1, 1 << 26, N, dtype=np.int64).astype(np.float64)
    m = rng.integers(1 << 52, 1 << 53, N, dtype=np.int64).astype(np.longdouble) + np.longdouble(0.5)
    middle = np.ldexp((m * m).astype(np.float64), 2 * rng.integers(-200, 200, N))
    for x in (_random(rng, N, 520), _random(rng, N, 3), r * r, np.ldexp(r * r, 2 * rng.integers(-200, 200, N)),
              _neighbours(r * r, rng), _neighbours(middle, rng), _neighbours(np.ldexp(1.0, rng.integers(-520, 520, N)), rng),
              SPECIAL, -_random(rng, 100, 5)):
        with np.errstate(all="ignore"):
            ref = np.sqrt(x)
        _same(_run(1, x, np.ones_like(x))[0], ref)


def test_division():
    rng = np.random.default_rng(3)
    sign = rng.choice([-1.0, 1.0], N)
    b = _random(rng, N, 490)
    q = rng.integers(1, 1 << 26, N, dtype=np.int64).astype(np.float64)
    d = rng.integers(1, 1 << 27, N, dtype=np.int64).astype(np.float64)
    m = rng.integers(1 << 52, 1 << 53, N, dtype=np.int64).astype(np.longdouble) + np.longdouble(0.5)
    b1 = _random(rng, N, 0)
    middle = (m * b1.astype(np.longdouble)).astype(np.float64)
    for x, y in ((_random(rng, N, 490) * sign, b), (sign * _random(rng, N, 2), b1), (q * d, d), (_neighbours(q * d, rng), d),
                 (_neighbours(middle, rng) * sign, b1), (_neighbours(np.ldexp(1.0, rng.integers(-520, 520, N)), rng), b),
                 (b, _neighbours(np.ldexp(1.0, rng.integers(-520, 520, N)), rng)), (SPECIAL, np.full(len(SPECIAL), 3.0)),
                 (np.full(len(SPECIAL), 3.0), np.abs(SPECIAL)), (b, b)):
        with np.errstate(all="ignore"):
            ref = x / y
        _same(_run(2, x, y)[0], ref)
