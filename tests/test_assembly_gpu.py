"""Assembly of large fronts: children of up to 64 contribution rows go in as
lists of positions per destination, larger ones by columns and row blocks.
Children at the edges of the two classes and of the 32-column and 64-row
blocks, in the level kernel, the per-step launches and the dependency order:
the factor against the oracle, and the three equal bit for bit."""
import numpy as np
import pytest

import synth
from synth.lp import _from_coo
from test_parity_gpu import check_pair, run_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_04370_gb300.build import build

    build()
    import paper_2508_04370_gb300 as p

    return p


def lp_with_columns(m, lengths, seed):
    """Column j holds lengths[j] entries; eliminated first (natural order), it is
    a front with that many contribution rows, and the dense rows are one front
    of about m rows."""
    rng = np.random.default_rng(seed)
    rows = np.concatenate([np.sort(rng.choice(m, size=k, replace=False)) for k in lengths])
    cols = np.repeat(np.arange(len(lengths)), lengths)
    return _from_coo(m, len(lengths), rows, cols, rng.standard_normal(rows.size), "columns")


@pytest.mark.parametrize("m,lengths", [
    (130, [63, 64, 65, 66, 31, 32, 33, 130, 1, 2] * 3 + [128, 129, 130]),
    (192, [64, 65, 100, 191, 192] + [6] * 120),
    (257, [257, 64, 65, 127, 129] + [1, 5, 33] * 90),
])
def test_children_at_class_and_block_edges(pkg, m, lengths):
    lp = lp_with_columns(m, lengths, m)
    theta = synth.theta_loguniform(lp.n, 5, -3.0, 3.0)
    r7, r1 = synth.rhs_normal(lp.n, 6), synth.rhs_normal(lp.m, 7)
    base = None
    for opts in (dict(), dict(level_kernel=0), dict(schedule=pkg.IPM_SCHED_DEPENDENCY)):
        r = run_pair(pkg, lp, theta, r7, r1, ordering=pkg.IPM_ORD_NATURAL, **opts)
        assert r["info"]["nfronts_large"] > 0
        check_pair(r, lp)
        if base is None:
            base = r
        else:
            assert np.array_equal(base["D"], r["D"]) and np.array_equal(base["L"], r["L"])
        r["s"].close()


def lp_with_thin_fronts(nlink, groups, private, seed):
    """One column per group with `private` rows of its own and nlink dense rows:
    leaves of 1 + private pivots and nlink more rows."""
    rng = np.random.default_rng(seed)
    rows, cols = [], []
    for g in range(groups):
        rows += list(private * g + np.arange(private)) + list(private * groups + np.arange(nlink))
        cols += [g] * (private + nlink)
    return _from_coo(private * groups + nlink, groups, rows, cols, rng.standard_normal(len(rows)), "thin")


@pytest.mark.parametrize("nlink,groups,private", [(129, 6, 0), (130, 5, 3), (161, 4, 4), (300, 3, 12), (150, 3, 31),
                                                  (490, 2, 20), (130, 1040, 3), (161, 1030, 5), (170, 1030, 31)])
def test_thin_fronts(pkg, nlink, groups, private):
    lp = lp_with_thin_fronts(nlink, groups, private, nlink)
    theta = synth.theta_loguniform(lp.n, 5, -2.0, 2.0)
    r7, r1 = synth.rhs_normal(lp.n, 6), synth.rhs_normal(lp.m, 7)
    # each column first, then its private rows, then the dense rows
    perm = [v for g in range(groups) for v in [g] + [lp.n + private * g + i for i in range(private)]]
    perm = np.array(perm + list(lp.n + private * groups + np.arange(nlink)), dtype=np.int32)
    base = None
    for opts in (dict(schedule=pkg.IPM_SCHED_LEVELS, level_kernel=0), dict(schedule=pkg.IPM_SCHED_DEPENDENCY)):
        r = run_pair(pkg, lp, theta, r7, r1, ordering=pkg.IPM_ORD_USER, user_perm=perm, amalg_zero_frac=0.0,
                     **opts)
        if groups >= 1024 or private == 0:  # fewer go through the steps
            assert r["info"]["nfronts_thin"] > 0
        check_pair(r, lp)
        if base is None:
            base = r
        else:
            assert np.array_equal(base["D"], r["D"]) and np.array_equal(base["L"], r["L"])
        r["s"].close()


@pytest.mark.parametrize("m,lengths", [(129, [129, 128, 129]), (160, [159, 131, 140, 129, 64, 160, 150]), (193, [193, 130, 160, 161, 192]),
                                       (300, [129 + 7 * j for j in range(24)] + [65, 64, 1])])
def test_rank_one_leaves(pkg, m, lengths):
    """One-column leaves on subsets of m dense rows (runs and scattered rows, so
    that blocks take all, some and none of a child's rows), beside stored ones."""
    lp = lp_with_columns(m, lengths, m)
    theta = synth.theta_loguniform(lp.n, 5, -3.0, 3.0)
    r7, r1 = synth.rhs_normal(lp.n, 6), synth.rhs_normal(lp.m, 7)
    base = None
    for opts in (dict(schedule=pkg.IPM_SCHED_LEVELS, level_kernel=0), dict(schedule=pkg.IPM_SCHED_LEVELS, level_kernel=1),
                 dict(schedule=pkg.IPM_SCHED_DEPENDENCY)):
        r = run_pair(pkg, lp, theta, r7, r1, ordering=pkg.IPM_ORD_NATURAL, amalg_zero_frac=0.0, **opts)
        assert r["info"]["nfronts_thin"] > 0
        check_pair(r, lp)
        if base is None:
            base = r
        else:
            assert np.array_equal(base["D"], r["D"]) and np.array_equal(base["L"], r["L"])
        r["s"].close()


@pytest.mark.parametrize("m", [5, 32, 33, 64, 65, 66, 97])
def test_small_front_children(pkg, m):
    """A front of m rows under children of 1 to m contribution rows (lists up to
    64 rows, one by one beyond), every CTA width with the same bits."""
    lp = lp_with_columns(m, [1 + (7 * j) % m for j in range(3 * m)] + [m, max(m - 1, 1)], m)
    theta = synth.theta_loguniform(lp.n, 5, -3.0, 3.0)
    r = run_pair(pkg, lp, theta, synth.rhs_normal(lp.n, 6), synth.rhs_normal(lp.m, 7), ordering=pkg.IPM_ORD_NATURAL)
    assert r["info"]["nfronts_small"] > 0
    check_pair(r, lp)
    s = r["s"]
    for width in (32, 64, 128, 256):
        pkg.ipm_set_launch_shapes(s.ctx, [width] * 3)
        s.factorise(theta, 1e-8, 1e-8)
        L, D, _ = s.factor()
        assert np.array_equal(D, r["D"]) and np.array_equal(L, r["L"])
    s.close()
