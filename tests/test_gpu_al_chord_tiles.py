"""The augmented-Lagrangian chord step of the FP32 path where a block walks several tiles of voxels: 64^3 is 2048 tiles of
128 voxels on at most 7 blocks per multiprocessor (1064 of them on 152), so the slots of the staged factors are used again
and the blocks' FP64 sums run over more than one tile, and the control adds up a thousand blocks' sums. Against the step
with the exact local Newton: both solve every local problem to newton_tol (1e-5 of the stress; no adaptive tolerance), so
after five iterations stress and mean stress agree to a few times that, and the residuals, which measure changes of the
stress by the same solves, to a few times that of the stress."""
import numpy as np
import pytest

from paper_1509_04953_gb300 import synth

pytestmark = pytest.mark.gpu


def test_chord_step_over_several_tiles_matches_exact_newton():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    n, grains = 64, 64
    assert n ** 3 // 128 > 7 * torch.cuda.get_device_properties(0).multi_processor_count
    seed = synth.BASE_SEED + n
    g0 = evp.voronoi(n, synth.voronoi_seeds(n, grains, seed)).cpu().numpy()
    quat = synth.orientations(grains, seed)
    sig, stats = {}, {}
    for newton in ("reuse", "exact"):
        s = evp.Solver(n, grains, g0, quat, synth.Material(), seed, precision="mixed", scheme="al", al_scale=8.0, tol=0.0,
                       max_iter=5, allow_unconverged=1, newton=newton, newton_adapt=0.0)
        for _ in range(2):
            rc, st = s.increment(-1e-3, 1.0)
            assert rc == 1 and st.iterations == 5
        sig[newton], stats[newton] = s.get("sig").astype(np.float64), st
        s.close()
    scale = np.abs(sig["exact"]).max()
    assert np.abs(sig["reuse"] - sig["exact"]).max() < 1e-4 * scale
    mean = {k: np.array(v.sig_mean[:]) for k, v in stats.items()}
    assert np.abs(mean["reuse"] - mean["exact"]).max() < 1e-4 * np.abs(mean["exact"]).max()
    # the device's sums against the field they are taken over: FP32 values, five-level trees, FP64 above
    for k in mean:
        want = sig[k].reshape(6, -1).mean(axis=1)
        assert np.abs(mean[k] - want).max() < 1e-6 * np.abs(sig[k]).max()
    assert abs(stats["reuse"].err_eq - stats["exact"].err_eq) < 1e-4
    assert abs(stats["reuse"].err_bc - stats["exact"].err_bc) < 1e-4
