"""Widths of the small-front CTAs: by each launch's number of fronts unless one
width was set or tuned for the class; what ipm_get_info reports, and what the
autotuner tries."""
import numpy as np
import pytest

import synth


@pytest.fixture(scope="module")
def pkg():
    from paper_2508_04370_gb300.build import build

    build()
    import paper_2508_04370_gb300 as p

    return p


def test_info_tells_the_rule_from_a_fixed_width(pkg):
    ctx = pkg.ipm_create()

    def widths():
        info = pkg.ipm_get_info(ctx)[1].as_dict()
        return info["tune_small_threads"], info["tune_small_by_count"]

    assert widths() == ([32, 64, 128], [True] * 3)
    assert pkg.ipm_set_launch_shapes(ctx, [32, 0, 256]) == 0
    assert widths() == ([32, 64, 256], [False, True, False])
    assert pkg.ipm_set_launch_shapes(ctx, [32, 64, 128]) == 0
    assert widths() == ([32, 64, 128], [False] * 3)
    assert pkg.ipm_set_launch_shapes(ctx, [0, 0, 0]) == 0
    assert widths() == ([32, 64, 128], [True] * 3)
    pkg.ipm_destroy(ctx)


@pytest.mark.gpu
@pytest.mark.parametrize("start", [0, 32, 64])
def test_autotuner_tries_rule_and_both_widths(pkg, start):
    """On an LP with small fronts of one class the autotuner factorises with the
    state it finds, the other five level ratios (they change nothing here) and the
    two widths it is not at; each choice keeps the factor."""
    lp = synth.random_lp(12, 30, 3, seed=1)
    theta = synth.theta_loguniform(lp.n, 1, -2.0, 2.0)
    s = pkg.Solver.from_lp(lp)
    info = s.info()
    assert info["max_front"] <= 32 and info["nfronts_large"] == 0
    assert pkg.ipm_set_launch_shapes(s.ctx, [start, 0, 0]) == 0

    def launches(run):
        pkg.ipm_kernel_stats(s.ctx, reset=True)
        pkg.ipm_set_profiling(s.ctx, True)
        run()
        pkg.ipm_set_profiling(s.ctx, False)
        return pkg.ipm_kernel_stats(s.ctx, reset=True)["small_fronts"]["launches"]

    one = launches(lambda: s.factorise(theta, 1e-8, 1e-8))
    before = s.factor()
    tuned = launches(lambda: s.autotune(theta, 1e-8, 1e-8, reps=1))
    per_sm = s.info()["tune_level_ctas_per_sm"]
    # 2 factorisations (one untimed) per candidate; one level-kernel CTA per SM
    # is a candidate where more fit
    pkg.ipm_set_level_ctas(s.ctx, 0)
    more_fit = s.info()["tune_level_ctas_per_sm"] > 1
    assert per_sm >= 1
    assert tuned == 2 * one * (1 + 5 + 2 + more_fit)
    for a, b in zip(before, s.factor()):
        assert np.array_equal(a, b)
    s.close()
