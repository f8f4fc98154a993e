"""The default re-solve margin of PTCA_MIXED contexts grows as beta does: at low
temperature a given dF error is a larger part of the Metropolis threshold.

Small cone moves, so that many decisions fall near the threshold."""
import numpy as np
import pytest

import paper_1502_07028_gb300 as P

pytestmark = pytest.mark.gpu


def _sweep(cfg, n=1, margin=None, T=None, launch=None):
    ctx = P.Context(cfg)
    if launch is not None:
        P.ptca_set_launch_config(ctx.h, *launch)
    if T is not None:
        P.ptca_set_T(ctx.h, T)
    if margin is not None:
        P.ptca_set_resolve_margin(ctx.h, margin)
    st = ctx.sweep(n)
    rec = [x.cpu().numpy() for x in ctx.record()]
    ctx.close()
    return st.resolved, rec


@pytest.mark.parametrize("launch", [None, (P.PIPELINE_STAGES, 4, 0, P.REDUCTION_TILED)], ids=["rows", "tiled"])
def test_per_matrix_reductions_take_the_fp64_decisions_at_low_temperature(launch):
    # below the determinants' range; dF of n = 128 is off by 2.7e-5 rms, 1.4e-2 T
    T = 0.002
    base = dict(Lx=64, Ly=64, L_c=8, schedule=P.SCHEDULE_BLOCK, proposal=P.PROPOSAL_CONE, cone_deg=0.05, J_H=8.0, mu=-6.5,
                T=T, seed=2)
    n0 = len(P.ptca_schedule(P.Config(**base))[0])   # stage 0 reads the common start alone
    _, (site64, Fo, Fn, lnu, acc64) = _sweep(P.Config(**base, precision=P.FP64))
    resolved, (site, _, _, _, acc) = _sweep(P.Config(**base, precision=P.MIXED), launch=launch)
    sure = np.abs(lnu + (Fn - Fo) / T)[:n0] > 1e-6
    assert np.array_equal(site, site64) and resolved > 0
    assert np.array_equal(acc[:n0][sure], acc64[:n0][sure])


@pytest.mark.parametrize("T", [0.001, 0.005])
def test_large_clusters_default_margin_follows_the_temperature(T):
    # shared reduction at T = 0.001, determinants at 0.005: 4e-7 (J + 4 t) / T
    base = dict(Lx=96, Ly=96, L_c=12, schedule=P.SCHEDULE_BLOCK, proposal=P.PROPOSAL_CONE, cone_deg=0.2, J_H=8.0, mu=-6.5,
                seed=6, precision=P.MIXED)
    cfg = P.Config(**base, T=T)
    r, rec = _sweep(cfg)
    r_rule, rec_rule = _sweep(cfg, margin=4e-7 * 12 / T)
    r_low, _ = _sweep(cfg, margin=1e-4)
    r_set, rec_set = _sweep(P.Config(**base, T=0.05), T=T)   # set after the start
    assert r == r_rule == r_set and r > r_low
    for a, b, c in zip(rec, rec_rule, rec_set):
        assert np.array_equal(a, b) and np.array_equal(a, c)
