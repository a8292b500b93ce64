"""Tolerances near what the arithmetic can reach, in the block solver."""

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


def _solve(eng, ctx, n, k, count, scale, prec, tol):
    h1, eri, occ = random_system(24, 12, seed=4, eri_scale=scale)
    rng = np.random.default_rng(7)
    t = set()
    while len(t) < count:
        t.add(tuple(sorted(rng.choice(12, k, replace=False).tolist()) + sorted((12 + rng.choice(12, n - k, replace=False)).tolist())))
    _, st, it = ctx.casci_batch(dev(h1), dev(eri), dev(occ), [], 0.0, n, dev(np.array(sorted(t), dtype=np.int32)),
                                eng.Opts(precision=prec, tol=tol, max_iter=400))
    return st.cpu().numpy(), it.cpu().numpy()


@pytest.mark.parametrize("n,k,count", [(7, 3, 60), (8, 4, 20), (9, 4, 8), (10, 2, 20), (10, 4, 4)])
def test_mixed_refinements_reach_1e12(eng, ctx, n, k, count):
    # within the 8 anchors that a sector may take, without the float64 fallback (dozens of products)
    st, it = _solve(eng, ctx, n, k, count, 1.0, "mixed", 1e-12)
    assert np.isin(st, (0, 4)).all()
    assert (it >> 16).max() <= 16 and (it >> 16).mean() <= 8


@pytest.mark.parametrize("n,k,count,scale,tol", [(10, 2, 76, 1.0, 1e-13), (8, 4, 76, 0.5, 5e-14)])
def test_float64_reaches_its_rounding_error(eng, ctx, n, k, count, scale, tol):
    st, _ = _solve(eng, ctx, n, k, count, scale, "fp64", tol)
    assert np.isin(st, (0, 4)).all()
