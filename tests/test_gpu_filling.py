"""Filling of PTCA_MIXED visits, whose free energies and fillings come from
determinants, against the Fermi function of the oracle's spectra and against FP64
contexts.

Tolerances.  One visit, per site: in double-float the nodes' error is at most
2.5e-10 on each of two levels, doubled for what both matrices and the phases'
rounding add.  In FP32 a phase carries a few 2^-24 of |x| up to 500 per level near
mu, and the filling's weights amount to 7: 4e-6.  The mean over a sweep of 2500
visits must lie within half an FP32 spacing of a value in [0.5, 1): 2^-25."""
import numpy as np
import pytest
import torch

import oracle
import paper_1502_07028_gb300 as P
from tests import inputs
from tests.test_gpu_parity import _oracle_model
from tests.test_gpu_resolvent import HOL, HUB

pytestmark = pytest.mark.gpu
BLOCK = dict(schedule=P.SCHEDULE_BLOCK)
DE = dict(J_H=8.0, mu=-6.5, T=0.05)
SHAPES = [
    dict(Lx=6, Ly=6, L_c=3, stride=3, **DE), dict(Lx=16, Ly=16, L_c=8, stride=8, **DE),
    dict(Lx=7, Ly=5, L_c=3, periodic=0, stride=3, **DE), dict(Lx=8, Ly=8, L_c=4, stride=4, J_H=8.0, mu=-6.5, T=0.6),
    dict(Lx=8, Ly=8, L_c=2, J_H=8.0, mu=-6.5, T=0.01), dict(Lx=24, Ly=24, L_c=8, t=0.7, **BLOCK, **DE),
    dict(Lx=24, Ly=24, L_c=4, **BLOCK, **DE), dict(Lx=24, Ly=24, L_c=12, **BLOCK, **DE), dict(Lx=26, Ly=26, L_c=13, **BLOCK, **DE),
    dict(Lx=12, Ly=12, Lz=12, L_c=3, J_H=6.0, mu=2.0, T=0.15, **BLOCK), dict(Lx=12, Ly=12, Lz=12, L_c=4, J_H=6.0, mu=2.0, T=0.1, **BLOCK),
    dict(Lx=24, Ly=24, L_c=5, T=0.1, t=-1.3, **BLOCK, **{**HUB, "mu": 1.0}), dict(Lx=1024, Ly=1, L_c=8, stride=8, T=0.1, **{**HOL, "mu": -1.0}),
]


@pytest.mark.parametrize("margin,tol", [(0.0, 4e-6), (1e6, 1e-9)])
@pytest.mark.parametrize("kw", SHAPES, ids=lambda d: "-".join(str(d[k]) for k in ("Lx", "Ly", "Lz", "L_c", "T") if k in d))
def test_one_visit_against_the_oracle(kw, margin, tol):
    cfg = P.Config(**kw, seed=2, precision=P.MIXED)
    m = _oracle_model(cfg)
    first = P.ptca_schedule(cfg)[0]
    for s in inputs.rng(7).choice(first, size=min(4, len(first)), replace=False):
        ctx = P.Context(cfg)   # observables: the visits recorded since the start, one here
        if cfg.model == P.MODEL_HUBBARD_MF:
            ctx.set_spins(torch.from_numpy(inputs.random_fields(5, cfg.N, 1.0)))
        S0 = ctx.spins().cpu().numpy()
        P.ptca_set_resolve_margin(ctx.h, margin)
        P.ptca_stage_run(ctx.h, 0, [int(s)])
        accepted = bool(ctx.record()[4].cpu().numpy()[0])
        filling = ctx.observables().filling
        ctx.close()
        H, _ = oracle.cluster_hamiltonian(m, S0, int(s), oracle.propose(m, 0, int(s), S0[s]) if accepted else None)
        x = (oracle.eigvalsh(H) - cfg.mu) / cfg.T
        ref = np.sum(0.5 - 0.5 * np.tanh(x / 2)) / (len(x) / 2)
        assert abs(filling - ref) <= tol, (filling, ref)


def _filling(cfg, margin):
    ctx = P.Context(cfg)
    if margin is not None:
        P.ptca_set_resolve_margin(ctx.h, margin)
    ctx.sweep(1)
    acc, filling = ctx.record()[4].cpu().numpy(), ctx.observables().filling
    ctx.close()
    return acc, filling


@pytest.mark.parametrize("kw", [dict(Lx=50, Ly=50, L_c=8, **BLOCK, **DE), dict(Lx=50, Ly=50, L_c=8, J_H=8.0, mu=-6.5, T=0.1, **BLOCK),
                                dict(Lx=12, Ly=12, Lz=12, L_c=3, J_H=8.0, mu=4.0, T=0.15, **BLOCK)],
                         ids=["square-0.05", "square-0.1", "cube"])
def test_mean_filling_of_a_sweep(kw):
    acc, ref = _filling(P.Config(**kw, seed=0, precision=P.FP64), None)
    for margin, tol in ((None, 2.0 ** -25), (1e6, 2e-11)):
        acc2, got = _filling(P.Config(**kw, seed=0, precision=P.MIXED), margin)
        assert np.array_equal(acc, acc2)
        assert abs(got - ref) <= tol, (margin, got - ref)
