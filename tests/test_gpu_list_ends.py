"""Active sets as set_fields takes them. Any negative id ends a list (what follows it, ids and values, counts for nothing),
whichever negative number it is: the steps and statistics equal, bit by bit, those of the same lists ended by -1 and
zeros."""
import numpy as np
import pytest

from paper_1509_04953_gb300 import synth

pytestmark = pytest.mark.gpu


def solver(n, precision, **kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_04953_gb300 import build
    build.build()
    from paper_1509_04953_gb300 import evp
    G, seed = 9, synth.BASE_SEED + n
    g0 = evp.voronoi(n, synth.voronoi_seeds(n, G, seed)).cpu().numpy()
    return evp.Solver(n, G, g0, synth.orientations(G, seed), synth.Material(), seed, precision=precision, **kw)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,kmax", [(16, 3), (32, 3), (32, 8), (64, 5)])
def test_any_negative_id_ends_a_list(n, kmax, precision):
    s = solver(n, precision, kmax=kmax)
    s.pf_step(3)
    ids, eta = s.get("ids"), s.get("eta")
    ended = ids < 0
    assert ended.any() and (ids[1] >= 0).any()
    rng = np.random.default_rng(n)
    other_ids = np.where(ended, rng.integers(-9, -1, ids.shape), ids)
    other_eta = np.where(ended, 0.5, eta)
    out = []
    for i, e in ((ids, eta), (other_ids, other_eta)):
        s.set("ids", i)
        s.set("eta", e)
        stats = []
        for _ in range(2):
            _, st = s.pf_step(1)
            stats.append((st.F_tot, st.X_rex, st.n_grains, st.overflow))
        out.append((stats, s.get("ids"), s.get("eta"), s.get("g")))
    a, b = out
    used = a[1] >= 0
    assert np.array_equal(used, b[1] >= 0) and np.array_equal(a[1][used], b[1][used])
    assert np.array_equal(a[2][used], b[2][used]) and np.array_equal(a[3], b[3])
    assert a[0] == b[0]
    s.close()


def test_statistics_of_lists_ended_by_other_negative_ids():
    """pf_step(0) counts the lists as they were set."""
    s = solver(32, "fp64", kmax=4)
    s.pf_step(3)
    ids, eta = s.get("ids"), s.get("eta")
    _, want = s.pf_step(0)
    s.set("ids", np.where(ids < 0, -3, ids))
    s.set("eta", np.where(ids < 0, 0.25, eta))
    _, got = s.pf_step(0)
    assert (got.F_tot, got.X_rex, got.n_grains) == (want.F_tot, want.X_rex, want.n_grains)
    s.close()
