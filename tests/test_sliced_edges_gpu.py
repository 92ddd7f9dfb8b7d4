"""Sliced updates of dense fronts of exactly k columns and f rows at the edges of the
32-column panels, the pairs of panels and the 128-row blocks, and of one front so
large that each CTA works through several tiles and row blocks, so that both groups
of warps and every buffer go round more than once.  The factor against the
oracle's, or for the large front against the FP64 path's, to the parity bar."""
import numpy as np
import pytest

import synth
from synth.lp import _from_coo
from oracle import Oracle
from test_parity_gpu import DELTA, EPS_PIV, RHO, check_pair, propagated_scales

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


def lp_with_front(k, r, seed):
    """Rows [0, k) become one front of k columns and k + r rows: columns that cover
    row 0 and the evens or odds of the rest fill it.  Of the r + 1 rows behind it the
    last is left out, which keeps the two fronts apart (a merged one would store a
    zero in every column).  Columns of four entries besides, so that there are more
    columns than rows."""
    rng = np.random.default_rng(seed)
    mine = np.arange(k + r)
    rest = k + np.arange(r + 1)
    cols = [np.union1d([0], mine[0::2]), np.union1d([0], mine[1::2])]
    if r > 0:
        cols += [np.union1d([k], rest[0::2]), np.union1d([k], rest[1::2])]
    m = k + r + (1 if r > 0 else 0)
    for j in range(m + 10):
        pool = mine if j % 2 or r < 4 else rest
        cols.append(np.sort(rng.choice(pool, size=min(4, len(pool)), replace=False)))
    rows = np.concatenate(cols)
    return _from_coo(m, len(cols), rows, np.repeat(np.arange(len(cols)), [len(c) for c in cols]),
                     rng.standard_normal(rows.size), "front")


def fronts(sym):
    """(columns, rows) of the supernodes."""
    return set(zip(np.diff(sym["snode_ptr"]).tolist(), np.diff(sym["sn_rptr"]).tolist()))


OPTS = dict(amalg_width=1, amalg_zero_frac=0.0, level_kernel=0, mixed_min_front=64)


def solve_pair(pkg, lp, theta, r7, r1, schedule):
    """The sliced factor and solution beside the oracle's with the same supernodes, and
    the tensor-core launches."""
    s = pkg.Solver.from_lp(lp, ordering=pkg.IPM_ORD_NATURAL, schedule=schedule, precision=pkg.IPM_PREC_SLICED, **OPTS)
    pkg.ipm_kernel_stats(s.ctx, reset=True)
    pkg.ipm_set_profiling(s.ctx, True)
    s.factorise(theta, RHO, DELTA)
    pkg.ipm_set_profiling(s.ctx, False)
    launches = pkg.ipm_kernel_stats(s.ctx, reset=True)["large_update_tc"]["launches"]
    dx, dy = s.solve(r7, r1)
    info, sym = s.info(), s.symbolic()
    L, D, dyn = s.factor()
    s.close()
    x = np.concatenate([dx.cpu().numpy(), dy.cpu().numpy()])
    o = Oracle.from_lp(lp)
    assert np.array_equal(o.analyse(sym["perm"], amalg_width=1, amalg_zero_frac=0.0)["sn_rows"], sym["sn_rows"])
    o.factorise(theta, RHO, DELTA, eps_piv=EPS_PIV)
    ofac = o.factor()
    ox, oy, _ = o.solve(r7, r1, omega_target=1e-12, max_steps=10)
    w = o.omega_K(theta, RHO, DELTA, r7, r1, x[: lp.n], x[lp.n:])
    return dict(info=info, sym=sym, L=L, D=D, dyn=dyn, x=x, ofac=ofac, ref=np.concatenate([ox, oy]), w_gpu=w,
                theta=theta), launches


@pytest.mark.parametrize("k,r", [(32, 128), (32, 127), (33, 128), (64, 128), (64, 129), (64, 255), (65, 63), (95, 161),
                                 (96, 160), (97, 159), (128, 128), (128, 0), (129, 1), (160, 97), (256, 256), (257, 0)])
def test_front_at_the_edges(pkg, k, r):
    lp = lp_with_front(k, r, 1000 * k + r)
    theta = synth.theta_loguniform(lp.n, 11, -3.0, 3.0)
    r7, r1 = synth.rhs_normal(lp.n, 12), synth.rhs_normal(lp.m, 13)
    base = None
    for schedule in (pkg.IPM_SCHED_LEVELS, pkg.IPM_SCHED_DEPENDENCY):
        p, launches = solve_pair(pkg, lp, theta, r7, r1, schedule)
        assert (k, k + r) in fronts(p["sym"])
        assert launches > 0 and p["info"]["flops_tensor"] > 0 and p["info"]["precision_fallbacks"] == 0
        check_pair(p, lp, rowwise=True)
        if base is None:
            base = p
        else:
            assert np.array_equal(base["D"], p["D"]) and np.array_equal(base["L"], p["L"])


def test_front_with_many_tiles_per_cta(pkg):
    k, r = 2850, 0
    lp = lp_with_front(k, r, 3)
    theta = synth.theta_loguniform(lp.n, 11, -3.0, 3.0)
    # tiles of 128 x 32 in the first pair's rest (columns from 128 on): the launch has
    # one CTA per SM at most
    tiles = sum((k - c + 127) // 128 for c in range(128, k, 32))
    import torch

    assert tiles >= 6 * torch.cuda.get_device_properties(0).multi_processor_count
    out = {}
    for precision in (pkg.IPM_PREC_FP64, pkg.IPM_PREC_SLICED):
        s = pkg.Solver.from_lp(lp, ordering=pkg.IPM_ORD_NATURAL, schedule=pkg.IPM_SCHED_LEVELS, precision=precision, **OPTS)
        s.factorise(theta, RHO, DELTA)
        info, sym = s.info(), s.symbolic()
        assert (k, k) in fronts(sym) and info["precision_fallbacks"] == 0
        assert (info["flops_tensor"] > 0) == (precision == pkg.IPM_PREC_SLICED)
        out[precision] = s.factor()
        s.close()
    (L, D, dyn), (Ls, Ds, dyns) = out[pkg.IPM_PREC_FP64], out[pkg.IPM_PREC_SLICED]
    assert np.array_equal(dyn != 0, dyns != 0)
    S = propagated_scales(sym, L, D)
    assert (np.abs(Ds - D) / S).max() <= 1e-10
    # L_ip: 1e-10 (sqrt(S_i S_p) + |L_ip| S_p) / |D_p|
    off = 0
    for sn in range(len(sym["sn_parent"])):
        c0, c1 = sym["snode_ptr"][sn], sym["snode_ptr"][sn + 1]
        R = sym["sn_rows"][sym["sn_rptr"][sn]:sym["sn_rptr"][sn + 1]]
        kk, f = c1 - c0, len(R)
        a, b = (x[off:off + f * kk].reshape(kk, f) for x in (L, Ls))
        Sp, Dp = S[c0:c1, None], np.abs(D[c0:c1])[:, None]
        low = np.arange(f)[None, :] > np.arange(kk)[:, None]
        bound = 1e-10 * (np.sqrt(S[R][None, :] * Sp) + np.abs(a) * Sp) / Dp
        assert (np.abs(a - b) <= bound)[low].all()
        off += f * kk
