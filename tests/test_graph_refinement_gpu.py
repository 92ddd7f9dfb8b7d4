"""Classical refinement inside a captured graph: three steps in line, the others in
a conditional node.  Inputs that need more steps than are in line, then inputs that
need fewer, then the first again, on one graph: every replay equals the direct
calls bit for bit, in steps and backward errors too."""
import numpy as np
import pytest

import synth
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


@pytest.mark.parametrize("refine_max", [3, 4, 5, 6, 10])
def test_steps_beyond_those_in_line(pkg, refine_max):
    import torch

    lp = synth.staircase(periods=3, seed=3)
    n, m = lp.n, lp.m
    sched = synth.theta_schedule(n, 40, 3)
    s = pkg.Solver.from_lp(lp, ordering=pkg.IPM_ORD_AMD, gmres_restarts=0, refine_max=refine_max)
    r7 = np.concatenate([synth.rhs_normal(n, 52), synth.rhs_normal(n, 53)])
    r1 = np.concatenate([synth.rhs_normal(m, 54), synth.rhs_normal(m, 55)])
    theta = torch.as_tensor(sched[39], device=s.dev)
    r7d, r1d = torch.as_tensor(r7, device=s.dev), torch.as_tensor(r1, device=s.dev)
    dx = torch.zeros(2 * n, dtype=torch.float64, device=s.dev)
    dy = torch.zeros(2 * m, dtype=torch.float64, device=s.dev)
    assert pkg.ipm_graph_capture(s.ctx, theta, RHO, DELTA, r7d, r1d, dx, dy, nsolves=2) == 0
    steps = []
    for it in (39, 5, 39):
        theta.copy_(torch.as_tensor(sched[it], device=s.dev))
        dx.fill_(np.nan)
        dy.fill_(np.nan)
        assert pkg.ipm_graph_launch(s.ctx) == 0
        torch.cuda.synchronize()
        got = s.info()
        gx, gy = dx.cpu().numpy(), dy.cpu().numpy()
        s.factorise(sched[it], RHO, DELTA)
        for k in range(2):
            ex, ey = s.solve(r7[k * n:(k + 1) * n], r1[k * m:(k + 1) * m])
            np.testing.assert_array_equal(gx[k * n:(k + 1) * n], ex.cpu().numpy())
            np.testing.assert_array_equal(gy[k * m:(k + 1) * m], ey.cpu().numpy())
        want = s.info()
        assert got["refine_steps"] == want["refine_steps"] and got["omega"] == want["omega"]
        assert got["omega_hist"] == want["omega_hist"]
        steps.append(got["refine_steps"])
    assert steps[0] == steps[2] == min(refine_max, steps[0]) and steps[1] <= 2
    # omega falls about tenfold a step: the limit ends the refinement up to six steps
    assert steps[0] == refine_max if refine_max <= 6 else steps[0] > 6
    s.close()
