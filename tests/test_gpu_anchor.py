"""Re-anchoring in the block solver's mixed mode: the anchor x0 + d of the next refinement is a unit
vector however large the correction d was."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from workloads import random_system, synthetic_molecule  # noqa: E402


@pytest.fixture(scope="module")
def eng():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1910_03527_gb300 as e
    e.build()
    return e


@pytest.fixture(scope="module")
def ctx(eng):
    c = eng.Context(0)
    yield c
    c.close()


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


# (seed of the couplings, place among the molecule's 34 tuples of 7 orbitals, anchors that the
# refinement takes when the anchors' images are float64 sums): tuples whose first correction is
# larger than the anchor.  An image whose fixed-point vector had elements above 1 cost two more.
LARGE_CORRECTIONS = [(0, 3, 4), (4, 9, 4), (6, 24, 2), (8, 32, 4), (17, 13, 2), (25, 26, 4), (33, 13, 2)]


@pytest.mark.parametrize("seed,place,anchors", LARGE_CORRECTIONS)
def test_corrections_larger_than_the_anchor(eng, ctx, seed, place, anchors):
    h0, e0, occ = synthetic_molecule(1910)
    rng = np.random.default_rng(seed)
    noise = np.triu(rng.normal(0.0, 0.01, size=h0.shape), 1)
    h1, eri = h0 + noise + noise.T, e0 * (1.0 + 0.02 * rng.uniform(-1, 1))
    ref = list(range(5, 11))
    exp = [p for p in range(40) if p not in ref]
    t = dev(np.array([[exp[place]]], dtype=np.int32))
    args = (dev(h1), dev(eri), dev(occ), ref, 0.0, 1, t)
    eps, st, it = ctx.casci_batch(*args, eng.Opts(precision="mixed"))
    want, sw, _ = ctx.casci_batch(*args, eng.Opts(precision="fp64"))
    assert int(st[0]) == 0 and int(sw[0]) == 0
    assert abs(float(eps[0] - want[0])) <= 1e-10
    assert int(it[0]) >> 16 <= anchors


@pytest.mark.parametrize("n,k", [(7, 3), (8, 4), (10, 2)])
def test_mixed_density_matrix_belongs_to_a_unit_vector(eng, ctx, n, k):
    """The trace of a tuple's 1-RDM is its number of electrons, as Phi's is: no tolerance of the solver
    enters, only the norm of the vector (its square has a rounding error of a few 1e-16 per electron;
    a correction of the accepted size, 3e-4, would show as 1e-7)."""
    h1, eri, occ = random_system(20, 10, seed=n, eri_scale=0.3)
    t = np.array([list(range(i, i + k)) + list(range(10 + j, 10 + j + n - k))
                  for i in range(0, 10 - k, 2) for j in range(0, 10 - n + k + 1, 2)], dtype=np.int32)
    for row in t:
        gh = torch.zeros((20, 20), dtype=torch.float64, device="cuda")
        st = ctx.casci_rdm_batch(dev(h1), dev(eri), dev(occ), [], n, dev(row[None]), None, gh, None,
                                 eng.Opts(precision="mixed"))
        assert int(st[0]) in (0, 4)
        assert abs(float(gh.trace())) <= 1e-13 * 2 * k


@pytest.mark.parametrize("n,k", [(2, 1), (3, 1), (3, 2), (4, 2), (5, 2), (5, 4), (6, 1)])
def test_two_body_density_matrices_of_small_spaces(eng, ctx, n, k):
    """Mixed mode takes the float64 solver there: the same gradients, up to the order of the sums."""
    h1, eri, occ = random_system(20, 10, seed=n, eri_scale=0.3)
    t = dev(np.array([list(range(i, i + k)) + list(range(10 + i, 10 + i + n - k)) for i in range(0, 5)], dtype=np.int32))
    got = []
    for prec in ("fp64", "mixed"):
        gh = torch.zeros((20,) * 2, dtype=torch.float64, device="cuda")
        ge = torch.zeros((20,) * 4, dtype=torch.float64, device="cuda")
        st = ctx.casci_rdm_batch(dev(h1), dev(eri), dev(occ), [], n, t, None, gh, ge, eng.Opts(precision=prec, tol=1e-9))
        assert np.isin(st.cpu().numpy(), (0, 4)).all()
        got.append((gh, ge))
    assert float((got[0][0] - got[1][0]).abs().max()) <= 1e-13 and float((got[0][1] - got[1][1]).abs().max()) <= 1e-13


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,k", [(3, 1), (4, 2), (5, 2), (6, 1)])
def test_density_matrices_within_few_iterations(eng, ctx, n, k, prec):
    """20 iterations are enough for these spaces with a Davidson basis of 20 vectors, and so for the
    solver of three that takes their two-body density matrices."""
    h1, eri, occ = random_system(20, 10, seed=n, eri_scale=0.3)
    t = dev(np.array([list(range(i, i + k)) + list(range(10 + i, 10 + i + n - k)) for i in range(0, 5)], dtype=np.int32))
    gh = torch.zeros((20,) * 2, dtype=torch.float64, device="cuda")
    ge = torch.zeros((20,) * 4, dtype=torch.float64, device="cuda")
    st = ctx.casci_rdm_batch(dev(h1), dev(eri), dev(occ), [], n, t, None, gh, ge, eng.Opts(precision=prec, tol=1e-9, max_iter=20))
    assert np.isin(st.cpu().numpy(), (0, 4)).all()
