"""The sliced update's runs of tiles: dense fronts at the edges of the 32-column
panels and pairs of panels, of the 128-row blocks, and large enough that a CTA
goes over several row blocks; the level order and the dependency order give
the same bits, and the factor meets the parity bar against the oracle."""
import numpy as np
import pytest

import synth
from test_assembly_gpu import lp_with_columns
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


@pytest.mark.parametrize("m", [97, 128, 129, 160, 161, 192, 255, 257, 289, 1600])
def test_dense_front(pkg, m):
    lp = lp_with_columns(m, [m, m - 1, m // 2] + [4] * m, m)
    theta = synth.theta_loguniform(lp.n, 11, -3.0, 3.0)
    r7, r1 = synth.rhs_normal(lp.n, 12), synth.rhs_normal(lp.m, 13)
    base = None
    for schedule in (pkg.IPM_SCHED_LEVELS, pkg.IPM_SCHED_DEPENDENCY):
        r = run_pair(pkg, lp, theta, r7, r1, ordering=pkg.IPM_ORD_NATURAL, level_kernel=0, schedule=schedule,
                     precision=pkg.IPM_PREC_SLICED, mixed_min_front=64)
        assert r["info"]["max_front"] >= m and r["info"]["precision_fallbacks"] == 0
        check_pair(r, lp, rowwise=True)
        if base is None:
            base = r
        else:
            assert np.array_equal(base["D"], r["D"]) and np.array_equal(base["L"], r["L"])
        r["s"].close()
