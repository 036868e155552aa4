"""FP64 transforms round no more than a network of plain products and sums: that network's root-mean-square errors on these
inputs (standard normal noise, seed n; relative, against extended precision) are the bounds, for the forward transform,
the inverse of a given spectrum, and one after the other."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def rel(got, want):
    d = got - want
    return math.sqrt(float((d.real ** 2 + d.imag ** 2).sum() / (want.real ** 2 + want.imag ** 2).sum()))


@pytest.mark.parametrize("n,forward,inverse,pair", [(16, 2.1102e-16, 2.2165e-16, 3.1483e-16),
                                                    (32, 2.4126e-16, 2.4390e-16, 3.4361e-16),
                                                    (64, 2.6607e-16, 2.6809e-16, 3.7449e-16),
                                                    (128, 3.1308e-16, 3.1349e-16, 4.7628e-16)])
def test_errors_are_at_most_those_of_products_and_sums(n, forward, inverse, pair):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    x = np.random.default_rng(n).standard_normal((1, n, n, n))
    want = np.fft.rfftn(x.astype(np.longdouble), axes=(1, 2, 3))
    spec = evp.rfft3d(torch.from_numpy(x).cuda())
    assert rel(spec.cpu().numpy(), want) <= forward
    assert rel(evp.irfft3d(spec).cpu().numpy() / n ** 3, x) <= pair
    given = want.astype(np.complex128)
    back = np.fft.irfftn(given.astype(np.clongdouble), s=(n, n, n), axes=(1, 2, 3))
    assert rel(evp.irfft3d(torch.from_numpy(given).cuda()).cpu().numpy() / n ** 3, back) <= inverse
