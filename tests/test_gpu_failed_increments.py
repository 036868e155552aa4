"""Statistics that an increment reports when it fails: after a local failure in the augmented Lagrangian's initial step
there is no iteration to report residuals or a mean stress of, and a mean stress that is not a number leaves err_bc at
zero, as the status says what happened."""
import numpy as np
import pytest

from paper_1509_04953_gb300 import synth

pytestmark = pytest.mark.gpu


def solver(precision, **kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    n, G, seed = 8, 4, synth.BASE_SEED
    g0 = evp.voronoi(n, synth.voronoi_seeds(n, G, seed)).cpu().numpy()
    return evp.Solver(n, G, g0, synth.orientations(G, seed), synth.Material(), seed, precision=precision, **kw)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("newton", ["exact", "reuse"])
def test_failed_initial_step_of_the_augmented_lagrangian(precision, newton):
    s = solver(precision, scheme="al", newton=newton, newton_max=1)
    rc, st = s.increment(-1e-3, 1.0, check=False)
    assert rc == -3 and st.iterations == 1 and "local Newton failed" in s.last_error()
    assert (st.err_eq, st.err_bc) == (0.0, 0.0) and not any(st.sig_mean)
    s.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_mean_stress_that_is_not_a_number(precision):
    s = solver(precision)
    sig = s.get("sig")
    sig[1, 7] = np.nan
    s.set("sig", sig)
    rc, st = s.increment(-1e-3, 1.0, check=False)
    assert rc < 0 and np.isnan(st.err_eq) and st.err_bc == 0.0
    s.close()
