"""Where casci_batch_routed sends active spaces of 13-16 orbitals with few strings: to the block solver
only where there are enough of them for the precision, and both routes agree."""

import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from workloads import random_system  # noqa: E402

VALID = (0, 4)
TOL = {"fp64": 1e-9, "mixed": 1e-8}  # E_h, the solvers' own


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


def _spaces(n, k, count):
    """Arguments of `count` spaces (n, k): a reference of the k occupied orbitals and virtual ones."""
    order = 2 if k < n - 1 else 1
    h1, eri, occ = random_system(40, k, seed=n, eri_scale=0.2)
    ref = list(range(n - order))
    t = np.array(list(itertools.combinations(range(n - order, 40), order))[:count], dtype=np.int32)
    assert len(t) == count
    return (dev(h1), dev(eri), dev(occ), ref, 0.0, order, dev(t))


@pytest.mark.parametrize("n,k,count,prec", [(15, 13, 1, "fp64"), (15, 13, 4, "mixed"), (16, 14, 8, "mixed"), (13, 2, 4, "fp64"),
                                            (16, 2, 16, "fp64")])
def test_few_spaces_go_to_the_whole_gpu(eng, ctx, n, k, count, prec):
    args = _spaces(n, k, count)
    got, launches = [], []
    for ndet in (0, 0, 1):  # (the first call warms up)
        before = ctx.launches()
        got.append(ctx.casci_batch_routed(*args, eng.Opts(precision=prec), large_ndet=ndet))
        launches.append(ctx.launches() - before)
    (a, sa, ia), (b, sb, ib) = got[1:]
    assert np.isin(sa.cpu().numpy(), VALID).all() and np.isin(sb.cpu().numpy(), VALID).all()
    assert float((a - b).abs().max()) <= 2 * TOL[prec]
    if prec == "fp64":  # (float32 sums of casci_solve are atomic: its last bits vary)
        assert torch.equal(a, b) and torch.equal(ia, ib)
    assert min(launches[1:]) >= 100 * count  # (a casci_solve takes hundreds, the block solver a handful)


@pytest.mark.parametrize("n,k,count,prec", [(14, 13, 1, "fp64"), (13, 1, 1, "mixed"), (13, 2, 16, "mixed"), (15, 13, 16, "mixed"),
                                            (16, 14, 32, "mixed"), (16, 2, 32, "mixed"), (13, 2, 20, "fp64")])
def test_many_spaces_go_to_the_block_solver(eng, ctx, n, k, count, prec):
    args = _spaces(n, k, count)
    ctx.casci_batch_routed(*args, eng.Opts(precision=prec))
    before = ctx.launches()
    a, sa, _ = ctx.casci_batch_routed(*args, eng.Opts(precision=prec))
    assert ctx.launches() - before <= 10  # (a casci_solve takes hundreds)
    b, sb, _ = ctx.casci_batch_routed(*args, eng.Opts(precision=prec), large_ndet=1)
    assert np.isin(sa.cpu().numpy(), VALID).all() and np.isin(sb.cpu().numpy(), VALID).all()
    assert float((a - b).abs().max()) <= 2 * TOL[prec]
