"""Sums over rows of K, columns and rows of A and entries of A Theta~ A^T run
one thread, one warp or one CTA each by their length.  Rows at the edges of
the classes (32 and 2048 terms), both forms: the norm against numpy, the
refined solution against a dense solve."""
import numpy as np
import pytest

from synth.lp import _from_coo

pytestmark = pytest.mark.gpu

RHO = DELTA = 1e-2


@pytest.fixture(scope="module")
def pkg():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_04370_gb300.build import build

    build()
    import paper_2508_04370_gb300 as p

    return p


def lp_with_rows(lengths, n, seed):
    """Row i holds lengths[i] entries in its first columns of a common shuffle
    (so entries of A A^T also sum min(lengths) terms), every column at least one."""
    rng = np.random.default_rng(seed)
    order = rng.permutation(n)
    rows = np.concatenate([np.full(k, i) for i, k in enumerate(lengths)] + [np.full(n, len(lengths))])
    cols = np.concatenate([order[:k] for k in lengths] + [np.arange(n)])
    keep = np.unique(np.stack([rows, cols]), axis=1)
    return _from_coo(len(lengths) + 1, n, keep[0], keep[1], rng.standard_normal(keep.shape[1]) / 8.0, "classes")


@pytest.mark.parametrize("form", [1, 2])
@pytest.mark.parametrize("lengths", [(1, 30, 31, 32, 33, 34), (2046, 2047, 2048, 2049), (64, 2500, 7)])
def test_row_lengths_at_class_edges(pkg, lengths, form):
    n = 2600
    lp = lp_with_rows(lengths, n, 3)
    rng = np.random.default_rng(5)
    theta = 10.0 ** rng.uniform(-1, 1, n)
    r7, r1 = rng.standard_normal(n), rng.standard_normal(lp.m)
    A = np.zeros((lp.m, n))
    A[lp.rowidx, np.repeat(np.arange(n), np.diff(lp.colptr))] = lp.vals
    h = 1.0 / theta + RHO
    S = (A / h) @ A.T + DELTA * np.eye(lp.m)
    K = np.block([[-np.diag(h), A.T], [A, DELTA * np.eye(lp.m)]])
    s = pkg.Solver.from_lp(lp, form=form)
    s.factorise(theta, RHO, DELTA)
    dx, dy = s.solve(r7, r1)
    info = s.info()
    M = S if form == 2 else K
    assert info["norm_K1"] == pytest.approx(np.abs(M).sum(axis=0).max(), rel=1e-12)
    assert info["rc"] >= 0 and info["refine_steps"] <= 10
    x = np.concatenate([dx.cpu().numpy(), dy.cpu().numpy()])
    ref = np.linalg.solve(K, np.concatenate([r7, r1]))
    # omega <= 1e-12 on the system solved bounds the error by cond times it
    assert np.abs(x - ref).max() <= 4e-12 * np.linalg.cond(K, np.inf) * np.abs(ref).max()
    s.close()
