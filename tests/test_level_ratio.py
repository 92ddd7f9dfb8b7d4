"""Which levels take the FP64 level kernel by default: with sliced updates in use the
steps win earlier (0.65 instead of 1), and a ratio that was set holds on every
level."""
import pytest

import synth


@pytest.fixture(scope="module")
def pkg():
    from paper_2508_04370_gb300.build import build

    build()
    import paper_2508_04370_gb300 as p

    return p


def test_reported_default(pkg):
    for precision, ratio in ((pkg.IPM_PREC_FP64, 1.0), (pkg.IPM_PREC_MIXED, 1.0), (pkg.IPM_PREC_SLICED, 0.65)):
        opt = pkg.ipm_default_options()
        opt.precision = precision
        ctx = pkg.ipm_create(opt)
        assert pkg.ipm_get_info(ctx)[1].tune_level_ratio == ratio
        assert pkg.ipm_set_launch_shapes(ctx, None, 0.5) == 0
        assert pkg.ipm_get_info(ctx)[1].tune_level_ratio == 0.5
        pkg.ipm_destroy(ctx)


@pytest.mark.gpu
@pytest.mark.parametrize("m,tensor", [(1200, False), (2100, True)])
def test_sliced_dense_root(pkg, m, tensor):
    """The dense root front (0.83 m rows) of a random LP: work over chain 0.3 at
    m = 1200, 0.99 at 2100."""
    lp = synth.random_lp(m, m * 5 // 2, 5, seed=m)
    theta = synth.theta_loguniform(lp.n, 3, -2.0, 2.0)
    s = pkg.Solver.from_lp(lp, precision=pkg.IPM_PREC_SLICED, schedule=pkg.IPM_SCHED_LEVELS)

    def tensor_launches():
        pkg.ipm_kernel_stats(s.ctx, reset=True)
        pkg.ipm_set_profiling(s.ctx, True)
        s.factorise(theta, 1e-8, 1e-8)
        pkg.ipm_set_profiling(s.ctx, False)
        return pkg.ipm_kernel_stats(s.ctx, reset=True)["large_update_tc"]["launches"]

    assert (tensor_launches() > 0) == tensor
    assert s.info()["tune_level_ratio"] == 0.65
    assert pkg.ipm_set_launch_shapes(s.ctx, None, 2.0) == 0
    assert tensor_launches() == 0
    s.close()
