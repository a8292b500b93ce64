"""casci_sigma_large in float64 is float64-accurate element by element, also for vectors whose elements
span many orders of magnitude."""

import itertools
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from workloads import random_system  # noqa: E402
from workloads.hamiltonians import hubbard_site_integrals  # noqa: E402


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


def _levels(n, k):
    """Excitation level of every determinant against the first."""
    s = sorted(sum(1 << p for p in c) for c in itertools.combinations(range(n), k))
    ex = np.array([bin(x & ~s[0]).count("1") for x in s])
    return (ex[:, None] + ex[None, :]).reshape(-1)


@pytest.mark.parametrize("n,k", [(6, 3), (8, 4), (10, 5), (11, 4)])
def test_tails_do_not_see_the_largest_element(eng, ctx, n, k):
    # c = e_0 + 1e-12 z: by linearity the rows that H does not connect with determinant 0 are those of
    # 1e-12 z alone, to the rounding of a float64 sum
    h1, eri, occ = random_system(n, k, seed=n)
    rng = np.random.default_rng(n)
    z = 1e-12 * rng.normal(size=math.comb(n, k) ** 2)
    far = _levels(n, k) > 2
    z[0] = 0.0
    both = z.copy()
    both[0] = 1.0
    a = (dev(h1), dev(eri), dev(occ), list(range(n)))
    want = ctx.casci_sigma_large(*a, dev(z), "fp64")[0].cpu().numpy()[far]
    got = ctx.casci_sigma_large(*a, dev(both), "fp64")[0].cpu().numpy()[far]
    assert np.abs(got - want).max() <= 1e-13 * np.abs(want).max()


@pytest.mark.parametrize("system", ["random", "site"])
@pytest.mark.parametrize("fall", [0.0, 0.5, 2.0, 4.0])
def test_rows_of_graded_vectors(eng, ctx, system, fall):
    # elements falling by 10^fall per excitation, as those of a CI vector do; rows of H from its columns
    # (sigma of unit vectors), their sums in extended precision.  A float64 sum of T terms is within
    # T 2^-53 of the sum of its terms' magnitudes; those are at most 2^3 of the row's.
    n, k = 8, 4
    if system == "random":
        h1, eri, occ = random_system(n, k, seed=2)
    else:  # most of V is zero
        h1, eri = hubbard_site_integrals(n, 1.0, 4.0)[:2]
        occ = np.array([1] * k + [0] * (n - k), dtype=np.uint8)
    a = (dev(h1), dev(eri), dev(occ), list(range(n)))
    lev = _levels(n, k)
    rng = np.random.default_rng(7)
    N = lev.size
    c = rng.normal(size=N) * 10.0 ** (-fall * lev)
    got = ctx.casci_sigma_large(*a, dev(c), "fp64")[0].cpu().numpy()
    terms = (k * (n - k + 1)) ** 2 + 2 * (1 + k * (n - k) + math.comb(k, 2) ** 2)
    for row in (0, 1, N // 3, N // 2, N - 2, N - 1):
        e = np.zeros(N)
        e[row] = 1.0
        h = ctx.casci_sigma(*a, dev(e))[0].cpu().numpy()  # (H is symmetric)
        assert abs(got[row] - math.fsum(h * c)) <= terms * 2.0 ** -50 * float(np.abs(h * c).sum()), row


def test_no_launches_for_a_form_that_is_not_used(eng, ctx):
    # set-up: 8 kernels; float64 sigma of few strings: opposite-spin, two same-spin, transpose; float32:
    # scatter lists, conversion, opposite-spin, two same-spin, transpose
    h1, eri, occ = random_system(8, 4, seed=2)
    a = (dev(h1), dev(eri), dev(occ))
    for A, prec, most in ((list(range(2, 7)), "fp64", 12), (list(range(8)), "mixed", 14)):
        k = int(sum(occ[p] for p in A))
        c = dev(np.random.default_rng(1).normal(size=math.comb(len(A), k) ** 2))
        ctx.casci_sigma_large(*a, A, c, prec)
        before = ctx.launches()
        ctx.casci_sigma_large(*a, A, c, prec)
        assert ctx.launches() - before <= most
