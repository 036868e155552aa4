"""k = sum of the 12 densities as set_fields refreshes it: the FP64 sum, also where the densities or FP32 sums of them are
infinite."""
import numpy as np
import pytest

from paper_1509_04953_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_refreshed_k_of_infinite_and_overflowing_densities(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    n, G, seed = 8, 5, synth.BASE_SEED
    g0 = evp.voronoi(n, synth.voronoi_seeds(n, G, seed)).cpu().numpy()
    s = evp.Solver(n, G, g0, synth.orientations(G, seed), synth.Material(), seed, precision=precision)
    rho = s.get("rho").astype(s.dtype)
    v = rho.reshape(12, -1)
    v[3, 5] = np.inf
    v[:, 6] = 3e38            # twelve of them pass the largest FP32 number
    v[0, 7] = 3.4e38
    v[1, 7] = 1e31            # one sum does
    v[2, 8], v[5, 8] = np.inf, np.nan
    v[:, 9] = 0.0
    v[:, 10] = 1e-42          # FP32 subnormals
    v[0, 11], v[1, 11] = 1e12, 1e-30
    s.set("rho", rho)
    want = v.astype(np.float64).sum(axis=0)
    got = s.get("k").reshape(-1)
    ok = np.isfinite(want)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
    assert (np.abs(got[ok] - want[ok]) <= 12 * 2.0 ** -52 * want[ok]).all()   # eleven additions on either side
    s.close()
