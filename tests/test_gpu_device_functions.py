"""Device functions of the FP64 local solve, element by element."""
import math

import numpy as np
import pytest

import device_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    return device_lib.load(tmp_path_factory.mktemp("dev"))


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
