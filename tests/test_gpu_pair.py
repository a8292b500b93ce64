"""Both classes of three orbitals go to one launch: any share of either, against the oracle."""

import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import mbe as omb  # noqa: E402
from workloads import random_system  # noqa: E402

TOL = {"fp64": 1e-9, "mixed": 1e-8}


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


NORB, NOCC = 24, 12
ONE = [(o, *v) for o in range(NOCC) for v in itertools.combinations(range(NOCC, NORB), 2)]  # 792 with k = 1
TWO = [(*o, v) for o in itertools.combinations(range(NOCC), 2) for v in range(NOCC, NORB)]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n1,n2", [(1, 0), (0, 1), (1, 1), (5, 2), (792, 1), (3, 792), (792, 792)])
def test_both_classes_in_one_launch(eng, ctx, n1, n2, prec):
    h1, eri, occ = random_system(NORB, NOCC, seed=3, eri_scale=0.3)
    rng = np.random.default_rng(n1 + n2)
    t = [ONE[i] for i in rng.permutation(792)[:n1]] + [TWO[i] for i in rng.permutation(792)[:n2]]
    t = np.array([t[i] for i in rng.permutation(len(t))], dtype=np.int32)
    args = (dev(h1), dev(eri), dev(occ), [], 0.0, 3, dev(t), eng.Opts(precision=prec))
    ctx.casci_batch(*args)
    before = ctx.launches()
    eps, st, _ = ctx.casci_batch(*args)
    # core Fock, classes, lists; one determinant (two kernels in mixed mode); both classes (the same)
    assert ctx.launches() - before <= (5 if prec == "fp64" else 7)
    assert np.isin(st.cpu().numpy(), (0, 4)).all()
    eps = eps.cpu().numpy()
    e_phi = omb.phi_energy(h1, eri, occ)
    for i in rng.permutation(len(t))[:40]:
        assert abs(eps[i] - omb.tuple_energy(h1, eri, occ, [], tuple(int(p) for p in t[i]), e_phi, 0.0)) <= TOL[prec]
    # every tuple once: those of a list with one class only
    for k in (1, 2):
        sel = np.nonzero(occ[t].sum(1) == k)[0]
        if 0 < len(sel) < len(t):
            alone, _, _ = ctx.casci_batch(*args[:6], dev(t[sel]), eng.Opts(precision=prec))
            assert np.abs(alone.cpu().numpy() - eps[sel]).max() <= 1e-13


def test_gradients_of_both_classes(eng, ctx):
    h1, eri, occ = random_system(NORB, NOCC, seed=3, eri_scale=0.3)
    got = []
    for lists in ([ONE[:50] + TWO[:70]], [ONE[:50], TWO[:70]]):
        gh = torch.zeros((NORB,) * 2, dtype=torch.float64, device="cuda")
        ge = torch.zeros((NORB,) * 4, dtype=torch.float64, device="cuda")
        for t in lists:
            st = ctx.casci_rdm_batch(dev(h1), dev(eri), dev(occ), [], 3, dev(np.array(t, dtype=np.int32)), None, gh, ge,
                                     eng.Opts(precision="fp64", tol=1e-10))
            assert np.isin(st.cpu().numpy(), (0, 4)).all()
        got.append((gh, ge))
    # (sums of 120 tuples' terms of order one, in any order)
    assert float((got[0][0] - got[1][0]).abs().max()) <= 1e-12 and float((got[0][1] - got[1][1]).abs().max()) <= 1e-12
