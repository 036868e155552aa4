"""The FP64 local problems in the crystal frame against the oracle, which works in the sample frame: every solver that
evaluates them, at the workloads' exponent (its own products), another integer exponent (the bit loop) and a
non-integer one. Same number of fixed-point iterations on both sides; the stress agrees to the local tolerance (1e-12
of the stress, below the parity tests' 1e-10), the rates to n times that."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_1509_04953_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-10


def rel(a, b):
    return np.abs(np.asarray(a) - np.asarray(b)).max() / max(np.abs(np.asarray(b)).max(), 1e-300)


@pytest.mark.parametrize("exponent", [10.0, 7.0, 10.37, 4.5])
@pytest.mark.parametrize("newton,scheme", [("f32_tangent", "basic"), ("exact", "basic"), ("reuse", "basic"),
                                           ("reuse", "al"), ("exact", "al")])
def test_fp64_local_solves_at_other_exponents_match_the_oracle(newton, scheme, exponent):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    mat = dataclasses.replace(synth.Material(), n=exponent)
    n, G, seed = 8, 5, synth.BASE_SEED + 1
    seeds, quat = synth.voronoi_seeds(n, G, seed), synth.orientations(G, seed)
    g0 = O.voronoi(n, seeds)
    kw = dict(tol=0.0, max_iter=5, allow_unconverged=1)
    gpu = evp.Solver(n, G, g0, quat, mat, seed, precision="fp64", newton=newton, scheme=scheme, al_scale=6.0, **kw)
    ref = O.State(n, G, g0, quat, mat, seed=seed, scheme=1 if scheme == "al" else 0, al_scale=6.0, **kw)
    for _ in range(3):
        rc, st = gpu.increment(-1e-3, 1.0)
        rco, sto = ref.increment(-1e-3, 1.0)
        assert rc == 1 and rco == 1 and st.iterations == sto.iterations
        assert rel(st.sig_mean, sto.sig_mean) < TOL
        for f in ("sig", "epsp", "rho"):
            assert rel(gpu.get(f), ref.field(f)) < TOL, f
