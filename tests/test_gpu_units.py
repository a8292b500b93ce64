"""The solvers do not depend on the unit of the integrals (tolerances given in the same unit)."""

import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from workloads import random_system  # noqa: E402


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


UNITS = [1e-18, 1e-14, 1e-10, 1e14, 1e18, 1e22]
VALID = (0, 4)  # (4: energies within 1e-8 of each other, always so in the small units)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,k", [(7, 3), (8, 4), (10, 2)])
@pytest.mark.parametrize("unit", UNITS)
def test_block_solver_in_any_unit(eng, ctx, n, k, unit, prec):
    # (the preconditioner keeps its absolute floor of 1e-4, so small units take more iterations; the
    # energies' errors are of second order in the residual, 1e-7, over gaps of a few tenths)
    h1, eri, occ = random_system(18, 9, seed=3, eri_scale=0.3)
    t = np.array([list(range(9 - k, 9)) + list(range(9, 9 + n - k)), list(range(0, k)) + list(range(18 - n + k, 18))],
                 dtype=np.int32)
    want, sw, _ = ctx.casci_batch(dev(h1), dev(eri), dev(occ), [], 0.0, n, dev(t), eng.Opts(precision="fp64"))
    eps, st, _ = ctx.casci_batch(dev(unit * h1), dev(unit * eri), dev(occ), [], 0.0, n, dev(t),
                                 eng.Opts(precision=prec, tol=1e-7 * unit, tol_switch=1e-5 * unit))
    assert np.isin(sw.cpu().numpy(), VALID).all() and np.isin(st.cpu().numpy(), VALID).all()
    assert float((eps / unit - want).abs().max()) <= 1e-9


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("unit", UNITS)
def test_large_solver_in_any_unit(eng, ctx, unit, prec):
    h1, eri, occ = random_system(8, 4, seed=3, eri_scale=0.3)
    want = ctx.casci_solve(dev(h1), dev(eri), dev(occ), list(range(8)), eng.Opts(precision="fp64"))
    got = ctx.casci_solve(dev(unit * h1), dev(unit * eri), dev(occ), list(range(8)),
                          eng.Opts(precision=prec, tol=1e-7 * unit, tol_switch=1e-5 * unit))
    assert want["status"] in VALID and got["status"] in VALID
    assert abs(got["lam"] / unit - want["lam"]) <= 1e-9


@pytest.mark.parametrize("n,k", [(7, 3), (9, 5), (10, 2)])
def test_no_interaction(eng, ctx, n, k):
    # a diagonal h and no (pq|rs): the unit of the float32 residuals is the diagonal's.  The lowest energy
    # is that of the lowest k orbitals, Phi's (h rises with the orbital)
    h1, eri, occ = random_system(18, 9, seed=3)
    t = np.array([list(range(9 - k, 9)) + list(range(9, 9 + n - k)), list(range(0, k)) + list(range(18 - n + k, 18))],
                 dtype=np.int32)
    eps, st, _ = ctx.casci_batch(dev(np.diag(np.diag(h1))), dev(0.0 * eri), dev(occ), [], 0.0, n, dev(t),
                                 eng.Opts(precision="mixed"))
    assert np.isin(st.cpu().numpy(), VALID).all()
    assert float(eps.abs().max()) <= 1e-9
