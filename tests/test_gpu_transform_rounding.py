"""Rounding of the transforms, measured without the zero frequency: zero-mean noise, root-mean-square errors against
the same transform in extended precision. A radix-2 butterfly rounds its product twice and its sum once and has one rounding
in its twiddle, 2^-p / sqrt3 rms each where they are of full size, so the error grows by at most 2 / sqrt3 of 2^-p a
stage in quadrature; 3 log2 n stages and the split of the packed rows (one more). The bound is twice that (three in the
inverse direction's two transforms, forward and back)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def modules():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    return torch, evp


def noise(n, fields, dtype):
    x = np.random.default_rng(100 * n + fields).standard_normal((fields, n, n, n))
    x -= x.mean(axis=(1, 2, 3), keepdims=True)
    return x.astype(dtype)


def reference(x, extended):
    return np.fft.rfftn(x.astype(np.longdouble if extended else np.float64), axes=(1, 2, 3))


def rms(a):
    a = a.copy()
    a[:, 0, 0, 0] = 0   # the zero frequency is compared on its own
    return math.sqrt(float((a.real ** 2 + a.imag ** 2).mean()))


@pytest.mark.parametrize("n", [8, 16, 32, 64])
@pytest.mark.parametrize("fields", [1, 6])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_rms_error_is_a_rounding_per_stage(n, fields, prec):
    torch, evp = modules()
    u = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    x = noise(n, fields, np.float64 if prec == "fp64" else np.float32)
    want = reference(x, prec == "fp64")
    spec = evp.rfft3d(torch.from_numpy(x).cuda())
    got = spec.cpu().numpy()
    stages = 3 * math.log2(n) + 1
    assert rms(got - want) < 2 * 2 / math.sqrt(3) * math.sqrt(stages) * u * rms(want)
    # the zero frequency: a sum of n^3 values of size one in log2(n^3) + 1 levels, each level at the size of its sums
    assert np.abs(got[:, 0, 0, 0] - want[:, 0, 0, 0]).max() < 4 * math.sqrt(stages) * u * n ** 1.5
    back = evp.irfft3d(spec.clone()).cpu().numpy() / n ** 3
    assert math.sqrt(float(((back - x) ** 2).mean())) < 3 * 2 / math.sqrt(3) * math.sqrt(2 * stages) * u
    if fields == 6:
        assert torch.equal(evp.stress_residual(torch.from_numpy(x).cuda())[0], spec)
