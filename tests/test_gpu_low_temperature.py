"""Mixed sweeps below the determinants' range (|mu - H| / T of a window of unit
vectors above 4096: T = 0.004 here): the Householder stage kernels of every CTA
width, the persistent kernels and the large-cluster reductions, which a context
runs there by default, against the oracle and against one another."""
import numpy as np
import pytest

import oracle
import paper_1502_07028_gb300 as P
from tests.test_gpu_parity import _check_sweep_against_oracle

pytestmark = pytest.mark.gpu
LOW = dict(J_H=8.0, mu=-6.5, T=0.004, schedule=P.SCHEDULE_BLOCK, proposal=P.PROPOSAL_CONE, cone_deg=2.0, precision=P.MIXED)
PIPELINES = [P.PIPELINE_STAGES, P.PIPELINE_OVERLAP, P.PIPELINE_PERSISTENT, P.PIPELINE_GRAPH]


@pytest.mark.parametrize("nw", [8, 4, 1])
@pytest.mark.parametrize("pipeline", PIPELINES)
def test_small_clusters_of_every_width_and_pipeline(pipeline, nw):
    cfg = P.Config(Lx=16, Ly=16, L_c=4, seed=3, **LOW)
    _check_sweep_against_oracle(cfg, sweeps=2, sample=12, near=6, launch=(pipeline, nw, 0))


@pytest.mark.parametrize("nw", [8, 4])
def test_pipelines_of_one_width_compute_the_same_chain(nw):
    # n = 128.  Bit for bit where the same kernels run: a launch per stage and per
    # re-solve (8 warps), or both inside the persistent kernel (nw warps); spins
    # and decisions in all four.
    cfg = P.Config(Lx=32, Ly=32, L_c=8, seed=5, **LOW)
    runs = []
    for pipeline in PIPELINES:
        ctx = P.Context(cfg)
        P.ptca_set_launch_config(ctx.h, pipeline, nw)
        resolved = ctx.sweep(2).resolved
        runs.append([resolved, ctx.spins().cpu().numpy(), *(x.cpu().numpy() for x in ctx.record())])
        ctx.close()
    assert runs[0][0] > 0
    for a, b in ((runs[0], runs[1]), (runs[2], runs[3])):
        assert all(np.array_equal(x, y) for x, y in zip(a, b))
    for run in runs[1:]:   # spins, sites, decisions
        assert all(np.array_equal(run[k], runs[0][k]) for k in (1, 2, 6))


@pytest.mark.parametrize("launch", [None, (P.PIPELINE_OVERLAP, 16, 0, P.REDUCTION_SHARED), (P.PIPELINE_STAGES, 16, 0),
                                    (P.PIPELINE_STAGES, 8, 0)], ids=["default", "overlap", "rows", "cluster"])
def test_large_clusters(launch):
    cfg = P.Config(Lx=24, Ly=24, L_c=12, seed=4, **LOW)
    _check_sweep_against_oracle(cfg, sweeps=1, sample=3, near=1, launch=launch)


def test_large_shared_reduction_keeps_its_dF_error():
    # n = 288, unguarded, stage 0: rounding common to both matrices and chases in
    # double-float, where one FP32 reduction per matrix leaves 2e-4
    cfg = P.Config(Lx=48, Ly=48, L_c=12, seed=1, **LOW)
    err = {}
    n0 = len(P.ptca_schedule(cfg)[0])
    m = oracle.Model(Lx=48, Ly=48, Lc=12, JH=8.0, mu=-6.5, T=0.004, schedule=P.SCHEDULE_BLOCK, seed=1,
                     proposal=P.PROPOSAL_CONE, cone_deg=2.0)
    for red in (P.REDUCTION_ROWS, P.REDUCTION_SHARED):
        ctx = P.Context(cfg)
        P.ptca_set_launch_config(ctx.h, P.PIPELINE_STAGES, 16, 0, red)
        P.ptca_set_resolve_margin(ctx.h, 0.0)
        S0 = ctx.spins().cpu().numpy()
        ctx.sweep(1)
        site, Fo, Fn, _, _ = (x.cpu().numpy() for x in ctx.record())
        ctx.close()
        d = []
        for k in range(0, n0, n0 // 6):
            s = int(site[k])
            ref = oracle.cluster_free_energy(m, S0, s, oracle.propose(m, 0, s, S0[s])) - oracle.cluster_free_energy(m, S0, s)
            d.append(Fn[k] - Fo[k] - ref)
        err[red] = np.max(np.abs(d))
    assert err[P.REDUCTION_SHARED] < 5e-6 and err[P.REDUCTION_SHARED] < 0.2 * err[P.REDUCTION_ROWS], err
