"""Which large fronts run whole in one CTA: ipm_get_info tells the rank-one leaves
from the other thin leaves, and a level of 1,024 leaves takes the thin kernel up to
4 columns or 224 rows and the steps beyond, with the same bits either way."""
import numpy as np
import pytest

import synth
from test_assembly_gpu import lp_with_thin_fronts
from test_parity_gpu import DELTA, RHO

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


@pytest.mark.parametrize("nlink,private,thin", [(250, 3, True), (251, 4, False), (219, 4, True), (220, 4, False),
                                                (192, 31, True), (193, 31, False), (450, 1, True)])
def test_thin_leaf_edges(pkg, nlink, private, thin):
    groups = 1026
    lp = lp_with_thin_fronts(nlink, groups, private, nlink)
    theta = synth.theta_loguniform(lp.n, 5, -2.0, 2.0)
    perm = [v for g in range(groups) for v in [g] + [lp.n + private * g + i for i in range(private)]]
    perm = np.array(perm + list(lp.n + private * groups + np.arange(nlink)), dtype=np.int32)
    out = []
    for opts in (dict(schedule=pkg.IPM_SCHED_LEVELS, level_kernel=0), dict(schedule=pkg.IPM_SCHED_DEPENDENCY)):
        s = pkg.Solver.from_lp(lp, ordering=pkg.IPM_ORD_USER, user_perm=perm, amalg_zero_frac=0.0, **opts)
        s.factorise(theta, RHO, DELTA)
        info = s.info()
        assert info["status"] & ~2 == 0 and info["nfronts_rank_one"] == 0
        # (one group's leaf may join the front of the dense rows)
        assert (info["nfronts_thin"] >= groups - 1) if thin else (info["nfronts_thin"] == 0)
        out.append(s.factor())
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_rank_one_leaves_are_told_apart(pkg):
    lp = synth.block_angular(blocks=20, bm=60, bn=160, density=0.05, linking=150, seed=5)
    s = pkg.Solver.from_lp(lp, ordering=pkg.IPM_ORD_ND, schedule=pkg.IPM_SCHED_LEVELS, level_kernel=0)
    s.factorise(synth.theta_loguniform(lp.n, 51), RHO, DELTA)
    info = s.info()
    # (no level has 1,024 other thin leaves)
    assert info["nfronts_thin"] == info["nfronts_rank_one"] > 100
    s.close()
