"""Device functions of the FP64 local solve, element by element."""
import decimal
import math

import numpy as np
import pytest

import device_lib

pytestmark = pytest.mark.gpu

D = decimal.Decimal


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    return device_lib.load(tmp_path_factory.mktemp("dev"))


def powers(dev, x, y):
    torch, lib = dev
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    t, c = torch.empty_like(xd), torch.empty_like(xd)
    rc = lib.dev_pow(x.size, xd.data_ptr(), yd.data_ptr(), t.data_ptr(), c.data_ptr(),
                     torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    torch.cuda.synchronize()
    return t.cpu().numpy(), c.cpu().numpy()


def relative_errors(x, y, got):
    """|got / x^y - 1| with 60-digit powers."""
    with decimal.localcontext() as ctx:
        ctx.prec = 60
        out = np.empty(x.size)
        for i in range(x.size):
            want = (D(float(y[i])) * D(float(x[i])).ln()).exp()
            out[i] = float(abs(D(float(got[i])) / want - 1))
    return out


# The last rounding is at most 2^-53 = 1.11e-16 of the power; the exponential's series stops before (ln2/128)^6/720 =
# 3.5e-17; its product s q of at most 0.0055 carries three roundings (2e-18); the logarithm's truncation and roundings,
# 2.5e-20, are scaled by y ln2 (y <= 30: 5e-19). Sum 1.5e-16; one unit 2^-52 is asked for.
TOL = 2.0 ** -52


def test_power_in_every_bin_of_the_table(dev):
    """All 128 mantissa bins at their edges and inside, exponents of two between 2^-20 and 2^7, y from below 1 to 30."""
    rng = np.random.default_rng(11)
    bins = np.arange(128)
    m = np.concatenate([1 + bins / 128, np.nextafter(1 + bins / 128, 0), 1 + (bins + rng.random(128)) / 128,
                        1 + (bins + rng.random(128)) / 128])
    m = np.tile(m, 4)
    x = np.ldexp(m, rng.integers(-20, 8, m.size))
    y = np.concatenate([rng.uniform(0.6, 30.0, m.size - 256), rng.uniform(-0.9, 0.6, 256)])
    table, _ = powers(dev, x, y)
    err = relative_errors(x, y, table)
    assert err.max() < TOL, (err.max(), x[err.argmax()], y[err.argmax()])


def test_power_next_to_one(dev):
    """Both sides of x = 1, where e = -1 and the table's logarithm cancel."""
    k = np.arange(0, 53)
    x = np.concatenate([1 + 2.0 ** -k, 1 - 2.0 ** -k[1:], 1 + 3 * 2.0 ** -k[2:], 1 - 3 * 2.0 ** -k[3:]])
    x = np.repeat(x, 4)
    y = np.tile(np.array([0.6, 3.5, 9.37, 29.9]), x.size // 4)
    table, _ = powers(dev, x, y)
    err = relative_errors(x, y, table)
    assert err.max() < TOL, (err.max(), x[err.argmax()], y[err.argmax()])


def test_power_towards_the_ends_of_the_range(dev):
    """Results up to 2^+-990 by the tables: the logarithm's error (2.5e-20, scaled by y ln2) stays below 1e-18 for y up
    to 50, so the bound is the same."""
    rng = np.random.default_rng(12)
    y = rng.uniform(5.0, 50.0, 512)
    x = np.exp2(rng.uniform(-990, 990, 512) / y)
    table, _ = powers(dev, x, y)
    err = relative_errors(x, y, table)
    assert err.max() < TOL, (err.max(), x[err.argmax()], y[err.argmax()])


def test_power_outside_the_tables_is_cudas(dev):
    """Subnormal, infinite and NaN arguments, results that leave the range of doubles or come close to it: the bits of
    CUDA's pow."""
    tiny, big = np.finfo(np.float64).tiny, np.finfo(np.float64).max
    x = np.array([5e-324, tiny / 2, np.nextafter(tiny, 0), np.inf, np.nan, 1e-200, 1e200, big, tiny, 2.0, 0.5, 2.0, 2.0,
                  0.5, 1.5, 1.5])
    y = np.array([9.37, 0.6, 2.5, 9.37, 9.37, 9.37, 9.37, 1.5, 1.5, 1000.5, 1023.5, 1e300, np.inf, np.inf, np.nan, -np.inf])
    table, cuda = powers(dev, x, y)
    assert np.array_equal(table.view(np.int64), cuda.view(np.int64)), list(zip(x, y, table, cuda))


@pytest.mark.parametrize("exponent", [10.0, 7.0, 10.37])
def test_fp32_tangent_is_the_rounded_fp64_one(dev, exponent):
    """The FP32 tangent of the FP64 residual against the FP64 one: an entry is built from slopes rounded once from FP64,
    by at most eight more roundings of terms no larger than the entry's elastic part plus ks/6 of the sum of all
    slopes, 2^-24 each."""
    torch, lib = dev
    rng = np.random.default_rng(13)
    n, tauc, gdot0, dt = 1 << 16, 20.0, 1e-3, 1.0
    C11, C12, C44 = 168400.0, 121400.0, 75400.0
    den = (C11 - C12) * (C11 + 2 * C12)
    d, s12, s44 = (C11 + 2 * C12) / den, -C12 / den, 1 / (2 * C44)
    sg = rng.standard_normal((6, n))

    def ratios(s):   # |tau| / tau_c of the 12 systems, in families of four
        h = np.concatenate([s[:3] / math.sqrt(6), s[3:] / math.sqrt(12)]) / tauc
        out = []
        for f, (i, j) in enumerate(((1, 2), (0, 2), (0, 1))):
            dd, a, b = h[i] - h[j], h[4] if f == 2 else h[5], h[4] if f == 0 else h[3]
            out += [dd + a - b, dd - a + b, dd + a + b, dd - a - b]
        return np.abs(np.array(out))

    sg *= rng.uniform(0.3, 1.5, n) / ratios(sg).max(axis=0)   # the hardest system at 0.3 to 1.5 of its strength
    s = torch.from_numpy(sg).cuda()
    k32 = torch.empty((21, n), dtype=torch.float32, device="cuda")
    k64 = torch.empty((21, n), dtype=torch.float64, device="cuda")
    rc = lib.dev_tangent(n, s.data_ptr(), d, s12, s44, tauc, gdot0, dt, exponent,
                         int(exponent) if exponent == int(exponent) else 0, k32.data_ptr(), k64.data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    torch.cuda.synchronize()
    slopes = gdot0 * dt * exponent / tauc / 6 * (ratios(sg) ** (exponent - 1)).sum(axis=0)
    elastic = np.zeros(21)
    elastic[[0, 2, 5]], elastic[[1, 3, 4]], elastic[[9, 14, 20]] = d + abs(s12), abs(s12), s44
    size = elastic[:, None] + slopes
    err = np.abs(k32.cpu().numpy().astype(np.float64) - k64.cpu().numpy()) / size
    assert err.max() < 8 * 2.0 ** -24, err.max() * 2 ** 24
