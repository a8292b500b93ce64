"""The sector solvers (tuples of 2-6 orbitals) and the block solver's tiled sigma.

Every string class (n, k) of the sector solvers, and classes of 7-10 orbitals of
the block solver on both sides of the size where its sigma changes form, against
the oracle on random Hamiltonians, whose ground states lie in either spin-flip
sector; the integrals also scaled up and down, since the float64 sigma is formed
in fixed point with a scale taken from them.
"""

import itertools
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import adjoint as oad  # noqa: E402
from oracle import fci  # noqa: E402
from oracle import mbe as omb  # noqa: E402
from workloads import random_system  # noqa: E402

TOL = {"fp64": 1e-9, "mixed": 1e-8}  # E_h at integrals of order one; relative to their scale below


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


def _tuples(n, k, nocc, norb, count, rng):
    """`count` tuples of n orbitals, k of them occupied."""
    occ = list(itertools.combinations(range(nocc), k))
    vir = list(itertools.combinations(range(nocc, norb), n - k))
    got = {occ[rng.integers(len(occ))] + vir[rng.integers(len(vir))] for _ in range(4 * count)}
    return sorted(got)[:count]


def _check(eng, ctx, h1, eri, occ, tuples, prec, scale):
    n = len(tuples[0])
    opts = eng.Opts(precision=prec, tol=1e-7 * scale, tol_switch=1e-5 * scale)
    eps, st, _ = ctx.casci_batch(dev(h1), dev(eri), dev(occ), [], 0.0, n, dev(np.array(tuples, dtype=np.int32)), opts)
    e_phi = omb.phi_energy(h1, eri, occ)
    want = np.array([omb.tuple_energy(h1, eri, occ, [], t, e_phi, 0.0) for t in tuples])
    assert np.isin(st.cpu().numpy(), (0, 4)).all()
    assert np.abs(eps.cpu().numpy() - want).max() <= TOL[prec] * scale


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,k", [(n, k) for n in range(2, 7) for k in range(1, n)])
def test_sector_classes(eng, ctx, n, k, prec):
    rng = np.random.default_rng(100 * n + k)
    h1, eri, occ = random_system(12, 6, seed=10 * n + k, eri_scale=0.8)
    _check(eng, ctx, h1, eri, occ, _tuples(n, k, 6, 12, 7, rng), prec, 1.0)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("scale", [0.1, 37.0, 4096.0])
@pytest.mark.parametrize("n,k", [(4, 2), (6, 3), (7, 3)])
def test_scaled_integrals(eng, ctx, n, k, scale, prec):
    rng = np.random.default_rng(5)
    h1, eri, occ = random_system(12, 6, seed=3)
    _check(eng, ctx, scale * h1, scale * eri, occ, _tuples(n, k, 6, 12, 4, rng), prec, scale)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,k,count", [(7, 2, 5), (7, 3, 5), (7, 5, 5), (8, 3, 3), (8, 4, 3), (8, 6, 3), (9, 2, 3),
                                       (9, 4, 1), (9, 7, 3), (10, 2, 3), (10, 8, 3)])
def test_block_classes(eng, ctx, n, k, count, prec):
    rng = np.random.default_rng(100 * n + k)
    h1, eri, occ = random_system(18, 9, seed=10 * n + k, eri_scale=0.5)
    _check(eng, ctx, h1, eri, occ, _tuples(n, k, 9, 18, count, rng), prec, 1.0)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [2, 4, 5, 6, 7])
def test_density_matrices(eng, ctx, n, prec):
    """Gradients of single tuples of every class against the oracle's density matrices."""
    h1, eri, occ = random_system(9, 4, seed=n, eri_scale=0.3)
    for k in range(max(1, n - 5), min(n, 5)):
        t = tuple(range(4 - k, 4)) + tuple(range(4, 4 + n - k))
        gh = torch.zeros((9, 9), dtype=torch.float64, device="cuda")
        ge = torch.zeros((9,) * 4, dtype=torch.float64, device="cuda")
        st = ctx.casci_rdm_batch(dev(h1), dev(eri), dev(occ), [], n, dev(np.array([t], dtype=np.int32)), None, gh, ge,
                                 eng.Opts(precision=prec, tol=1e-10))
        assert int(st[0]) == 0
        _, wh, we = oad.cas_gradient(h1, eri, occ, list(t))
        _, ph, pe = oad.cas_gradient(h1, eri, occ, [])
        # (first order in the residual, 1e-10, over a gap of a few tenths)
        assert np.abs(gh.cpu().numpy() - (wh - ph)).max() <= 1e-8
        assert np.abs(ge.cpu().numpy() - (we - pe)).max() <= 1e-8


def test_integrals_that_are_not_finite(eng, ctx):
    h1, eri, occ = random_system(12, 6, seed=3)
    for n, t in ((4, (4, 5, 6, 7)), (6, (3, 4, 5, 6, 7, 8)), (7, (3, 4, 5, 6, 7, 8, 9))):
        bad = eri.copy()
        bad[6, 6, 6, 6] = np.nan
        for prec in ("fp64", "mixed"):
            eps, st, _ = ctx.casci_batch(dev(h1), dev(bad), dev(occ), [], 0.0, n, dev(np.array([t], dtype=np.int32)),
                                         eng.Opts(precision=prec))
            assert int(st[0]) == 2 and np.isnan(float(eps[0]))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,k", [(13, 1), (13, 2), (13, 11), (14, 13), (15, 2), (15, 13), (16, 14), (16, 15)])
def test_wide_spaces_of_few_strings(eng, ctx, n, k, prec):
    """Tuple spaces of 13-16 orbitals with at most 128 strings go to the block solver; with a
    determinant limit of one they go to casci_solve. One order-1 tuple of each kind in the list
    where the space allows it, so that the lists are gathered and scattered."""
    h1, eri, occ = random_system(18, 15 if k > 2 else 3, seed=n + k, eri_scale=0.2)
    nocc = int(occ.sum())
    ref = list(range(nocc - k, nocc)) + list(range(nocc, nocc + n - k - 1))
    if len([p for p in ref if p < 18]) < n - 1:  # not enough virtuals: fill with lower occupied ones
        ref = list(range(18 - (n - 1), 18))
    ref = sorted(p for p in ref if p < 18)[:n - 1]
    exp = [p for p in range(18) if p not in ref]
    tup = dev(np.array([[p] for p in exp], dtype=np.int32))
    args = (dev(h1), dev(eri), dev(occ), ref, 0.0, 1, tup, eng.Opts(precision=prec, tol=1e-8))
    a, sa, _ = ctx.casci_batch_routed(*args)
    b, sb, _ = ctx.casci_batch_routed(*args, large_ndet=1)
    assert np.isin(sa.cpu().numpy(), (0, 4)).all() and np.isin(sb.cpu().numpy(), (0, 4)).all()
    assert np.abs((a - b).cpu().numpy()).max() <= 2 * TOL[prec]


@pytest.mark.parametrize("n,k", [(1, 1), (3, 1), (5, 2), (7, 4), (9, 3), (10, 8), (11, 5), (13, 2), (14, 3)])
@pytest.mark.parametrize("scale", [1.0, 1e-150, 1e150])
def test_large_sigma_on_digits(eng, ctx, n, k, scale):
    # float64 sigma of one large space from products of 8-bit digits; integrals whose scale is
    # near the ends of the range (1e-150, 1e150) stay on the plain float64 kernels.  Per term the
    # operands are rounded to 2^-56 of their largest and what is left out is below 2^-53.
    h1, eri, occ = random_system(n + 1, k, seed=n)
    h1, eri = h1 * scale, eri * scale
    A = list(range(k)) + list(range(k + 1, n + 1)) if n > k else list(range(n))
    rng = np.random.default_rng(k)
    N = math.comb(n, k) ** 2
    c = rng.normal(size=N)
    got = ctx.casci_sigma_large(dev(h1), dev(eri), dev(occ), A, dev(c), "fp64")[0].cpu().numpy()
    rows = rng.choice(N, size=min(N, 200), replace=False)
    _, h_eff, eri_a = omb.frozen_core(h1, eri, occ, A)
    want = fci.sigma_rows(h_eff, eri_a, k, k, c, rows)
    terms = (k * (n - k + 1)) ** 2 + 2 * (1 + k * (n - k) + math.comb(k, 2) * math.comb(n - k, 2))
    bound = terms * 2.0 ** -50 * max(np.abs(eri_a).max(), np.abs(h_eff).max()) * np.abs(c).max()
    assert np.abs(got[rows] - want).max() <= bound


def test_large_sigma_keeps_a_nan_where_it_belongs(eng, ctx):
    # a NaN in c reaches the determinants that it is connected to, and only those
    n, k = 8, 4
    h1, eri, occ = random_system(n, k, seed=1)
    c = np.random.default_rng(1).normal(size=math.comb(n, k) ** 2)
    c[0] = np.nan
    got = ctx.casci_sigma_large(dev(h1), dev(eri), dev(occ), list(range(n)), dev(c), "fp64")[0].cpu().numpy()
    assert np.isnan(got[0]) and np.isfinite(got).sum() > got.size // 4
