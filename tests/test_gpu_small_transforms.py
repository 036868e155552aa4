"""The radix-8 transforms of 16^3 and 32^3 grids (the last stage of the radix-16 network in their second pass) and their
neighbours, forward and inverse, for every number of fields, against torch.fft in FP64. Bounds: FP32 a few roundings per
radix stage (3 axes x 5 stages, 2^-24 each, random: 2e-6 of the largest coefficient covers them), FP64 the same at
2^-53."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 16, 32, 64])
@pytest.mark.parametrize("fields", [1, 5, 6])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_transforms_match_fp64(n, fields, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    gen = torch.Generator(device="cuda").manual_seed(7 * n + fields)
    x = torch.randn((fields, n, n, n), generator=gen, device="cuda", dtype=torch.float64) + 3.0
    dt, tol = (torch.float64, 4e-15) if prec == "fp64" else (torch.float32, 2e-6)
    x = x.to(dt)
    want = torch.fft.rfftn(x.double(), dim=(1, 2, 3))
    spec = evp.rfft3d(x)
    assert ((spec - want).abs().max() / want.abs().max()).item() < tol
    back = evp.irfft3d(spec.clone())
    assert ((back.double() / n ** 3 - x.double()).abs().max() / x.abs().max()).item() < tol
    if fields == 6:   # the residual of the same field: its spectrum and mean stress
        spec6, out = evp.stress_residual(x)
        assert torch.equal(spec6, spec)
        mean = x.double().mean(dim=(1, 2, 3))
        assert ((out[:6] - mean).abs().max() / mean.abs().max()).item() < tol
