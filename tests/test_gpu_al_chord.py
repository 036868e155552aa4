"""The augmented-Lagrangian step of the FP32 path with stored factors (the chord loop with its out-of-line solver) against
the step with the exact local Newton: both solve every local problem to newton_tol (1e-5 of the stress; no adaptive
tolerance here), so after five iterations the stresses agree to a few times that. 4^3 is half a block of threads, 8^3 four
blocks, 16^3 spans every multiprocessor; both laws."""
import numpy as np
import pytest

from paper_1509_04953_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,grains", [(4, 3), (8, 5), (16, 8)])
@pytest.mark.parametrize("law", ["power", "mr"])
@pytest.mark.parametrize("precision", ["mixed", "mixed_fast"])
def test_chord_step_matches_exact_newton(n, grains, law, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    mat = synth.ma_roters_material() if law == "mr" else synth.Material()
    seed = synth.BASE_SEED + n
    g0 = evp.voronoi(n, synth.voronoi_seeds(n, grains, seed)).cpu().numpy()
    quat = synth.orientations(grains, seed)
    sig = {}
    for newton in ("reuse", "exact"):
        s = evp.Solver(n, grains, g0, quat, mat, seed, precision=precision, scheme="al", al_scale=8.0, law=law, tol=0.0,
                       max_iter=5, allow_unconverged=1, newton=newton, newton_adapt=0.0)
        for _ in range(2):
            rc, st = s.increment(-1e-3, 1.0)
            assert rc == 1 and st.iterations == 5
        sig[newton] = s.get("sig").astype(np.float64)
        solves, evals, _ = s.newton_counts()
        assert solves >= 12 * n ** 3 and evals >= solves   # (1 + 5) local steps an increment, at least one solve each
        s.close()
    assert np.abs(sig["reuse"] - sig["exact"]).max() < 1e-4 * np.abs(sig["exact"]).max()
