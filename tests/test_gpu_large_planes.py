"""The 256^3 FP32 transforms, whose planes are held by clusters of four blocks and whose z pass takes the Nyquist column in
blocks of its own, for numbers of fields between the one and the six that other tests run, against torch.fft in FP64. The
bound is a few roundings per radix-2 stage (24 stages of 2^-24 each, random: 2e-6 of the largest coefficient covers
them). The Nyquist planes are compared on their own, against their own largest coefficient: their coefficients are as large
as the others here (noise), and their rounding is relative to the same sums, so ten times the bound holds."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fields", [2, 5])
def test_transforms_match_fp64(fields):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    n, tol = 256, 2e-6
    gen = torch.Generator(device="cuda").manual_seed(fields)
    x = torch.randn((fields, n, n, n), generator=gen, device="cuda")
    spec = evp.rfft3d(x)
    back = evp.irfft3d(spec.clone())
    for f in range(fields):
        want = torch.fft.rfftn(x[f].double())
        assert ((spec[f] - want).abs().max() / want.abs().max()).item() < tol
        nyq = want[..., n // 2]
        assert ((spec[f][..., n // 2] - nyq).abs().max() / nyq.abs().max()).item() < 10 * tol
        assert ((back[f].double() / n ** 3 - x[f].double()).abs().max() / x[f].abs().max()).item() < tol


def test_residual_keeps_the_spectrum():
    """The residual's z pass keeps the Nyquist column on its tiles: the same line transforms, so the same bits."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((6, 256, 256, 256), generator=gen, device="cuda")
    assert torch.equal(evp.stress_residual(x)[0], evp.rfft3d(x))


def test_transform_runs_on_the_current_stream():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    assert evp._stream(torch) == torch.cuda.current_stream().cuda_stream
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert evp._stream(torch) == s.cuda_stream
        x = torch.randn((1, 8, 8, 8), device="cuda")
        spec = evp.rfft3d(x)
    s.synchronize()
    want = torch.fft.rfftn(x[0].double())
    assert ((spec[0] - want).abs().max() / want.abs().max()).item() < 2e-6
