"""Sweeps whose free energies come from determinants (the default reduction of
PTCA_MIXED contexts): FP32 nodes by one warp and by a group of threads, the
double-float re-solve, and the FP64 fallback for windows beyond the node
classes, against the oracle's spectra.

Shapes: window extents at and around the tiles' edges (4, 8, 12 and 16 sites
per layer), rings of two and three layers, single layers (clipped windows),
chains, ragged open windows; |x| just inside and outside a node class.

Tolerances.  A node's logarithm carries about sqrt(n) roundings of 2^-24 per
pivot, its weight a_j sums to less than X, so T X 2^-24 sqrt(n) bounds F's
error up to a small factor: 2e-7 T X with T X <= 2 |mu - H|_max, plus the
1e-6 |F| that FP32 input terms may lose.  dF keeps only the update site's last
pivot: 2e-6 of J + 2 d t.  Double-float and FP64: 1e-9."""
import os
import re

import numpy as np
import pytest

import oracle
import paper_1502_07028_gb300 as P
from paper_1502_07028_gb300 import _build
from tests import inputs
from tests.test_gpu_parity import _oracle_model

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_node_tables_reproduce_the_grand_canonical_functions():
    text = open(os.path.join(ROOT, "paper_1502_07028_gb300", "csrc", "fermi_nodes.cuh")).read()
    # the errors that the tables are made for, as their comments state them
    for name, tol_f, tol_t, tol_s in (("PTCA_FERMI_NODES", 3e-7, 2e-6, 1e-8), ("PTCA_FERMI_NODES_DF", 6e-11, 1e-7, 1e-9)):
        body = text.split(f"#define {name} ")[1].split("#define")[0].replace("\\", "")
        rows = re.findall(r"\{\s*(\d+), ([^,{]+), ([^,{]+), ([^,{]+),\s*\{([^}]*)\},\s*\{([^}]*)\},\s*\{([^}]*)\}\}", body)
        assert len(rows) >= 9
        for M, X, c, e, y, a, b in rows:
            X, c, e = float(X), float(c), float(e)
            y, a, b = (np.array([float(v) for v in q.split(",")]) for q in (y, a, b))
            assert y.size == a.size == b.size == int(M) <= 32
            x = np.concatenate([np.linspace(0, 12, 4001), np.geomspace(12, X, 4001)])
            lncosh = x / 2 + np.log1p(np.exp(-x)) - np.log(2.0)
            fit = c + e / 2 * x ** 2 + 0.5 * np.log1p(x[:, None] ** 2 / y ** 2) @ a
            assert np.max(np.abs(fit - lncosh)) < tol_f + 4e-15 * X * np.abs(a).sum(), (name, X)
            d = np.abs(np.arctan(x[:, None] / y) @ b - 0.5 * np.tanh(x / 2))
            assert d.max() < tol_t and d[x > 14].max() < tol_s, (name, X, d.max())




def _stage0(cfg, start, margin, sample=None):
    """Records of stage 0 (it reads the start alone) against the oracle."""
    _build.build()
    ctx = P.Context(cfg)
    if start is not None:
        ctx.set_spins(start)
    S0 = ctx.spins().cpu().numpy()
    P.ptca_set_resolve_margin(ctx.h, margin)
    ctx.sweep(1)
    site, Fo, Fn, lnu, acc = (x.cpu().numpy() for x in ctx.record())
    filling = ctx.observables().filling
    ctx.close()
    m = _oracle_model(cfg)
    n0 = len(P.ptca_schedule(cfg)[0])
    idx = np.arange(n0) if sample is None or n0 <= sample else inputs.rng(n0).choice(n0, size=sample, replace=False)
    eF = edF = 0.0
    Fmax = 1.0
    for k in idx:
        s = int(site[k])
        sn = oracle.propose(m, 0, s, S0[s])
        Fo_ref, Fn_ref = oracle.cluster_free_energy(m, S0, s), oracle.cluster_free_energy(m, S0, s, sn)
        Fmax = max(Fmax, abs(Fo_ref))
        eF = max(eF, abs(Fo[k] - Fo_ref), abs(Fn[k] - Fn_ref))
        edF = max(edF, abs((Fn[k] - Fo[k]) - (Fn_ref - Fo_ref)))
    return eF, edF, Fmax, filling, acc


HUB = dict(model=P.MODEL_HUBBARD_MF, U=8.0, mu=4.0, m_step=0.5)
HOL = dict(model=P.MODEL_HOLSTEIN, lam=1.5, K=1.0, mu=0.0, m_step=0.4)
SHAPES = [
    # few visits per stage: a group of threads per node
    dict(Lx=6, Ly=6, L_c=2, stride=2), dict(Lx=9, Ly=9, L_c=3, stride=3), dict(Lx=10, Ly=10, L_c=5, stride=5),
    dict(Lx=14, Ly=14, L_c=7, stride=7), dict(Lx=16, Ly=16, L_c=8, stride=8), dict(Lx=18, Ly=18, L_c=9, stride=9),
    dict(Lx=7, Ly=5, L_c=3, periodic=0, stride=3), dict(Lx=9, Ly=1, L_c=3, periodic=0, stride=3),
    dict(Lx=8, Ly=1, L_c=2, stride=2), dict(Lx=9, Ly=1, L_c=3, stride=3), dict(Lx=6, Ly=6, Lz=6, L_c=3, stride=3),
    dict(Lx=4, Ly=4, Lz=4, L_c=2, stride=2), dict(Lx=8, Ly=8, L_c=4, stride=4, cluster_periodic=0),
    # many: nodes packed into warps
    dict(Lx=26, Ly=24, L_c=2, schedule=P.SCHEDULE_BLOCK), dict(Lx=25, Ly=24, L_c=3, schedule=P.SCHEDULE_BLOCK),
    dict(Lx=24, Ly=24, L_c=4, schedule=P.SCHEDULE_BLOCK), dict(Lx=24, Ly=26, L_c=5, schedule=P.SCHEDULE_BLOCK),
    dict(Lx=24, Ly=24, L_c=8, schedule=P.SCHEDULE_BLOCK), dict(Lx=24, Ly=24, L_c=9, schedule=P.SCHEDULE_BLOCK),
    dict(Lx=30, Ly=28, L_c=2, periodic=0, stride=2), dict(Lx=37, Ly=37, L_c=3, periodic=0, stride=3),
    dict(Lx=1024, Ly=1, L_c=4, stride=4), dict(Lx=600, Ly=1, L_c=3, periodic=0, stride=3),
    dict(Lx=12, Ly=12, Lz=12, L_c=2, stride=2), dict(Lx=12, Ly=12, Lz=12, L_c=3, schedule=P.SCHEDULE_BLOCK),
    dict(Lx=24, Ly=24, L_c=4, schedule=P.SCHEDULE_BLOCK, cluster_periodic=0),
]


@pytest.mark.gpu
@pytest.mark.parametrize("mdl", ["exchange", "hubbard", "holstein"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda d: "x".join(str(v) for v in d.values()))
def test_free_energies_of_stage_0(shape, mdl):
    if mdl == "exchange":
        kw, scale, start = dict(J_H=8.0, mu=-6.5, T=0.05), 8.0 + 6.0, None
    elif mdl == "hubbard":
        kw, scale = dict(T=0.1, **HUB), 2 * 4.0 + 6.0
        start = inputs.random_fields(5, shape["Lx"] * shape["Ly"] * shape.get("Lz", 1), 2.0)
    else:
        kw, scale, start = dict(T=0.1, **HOL), 3.0 + 6.0, None
    cfg = P.Config(**shape, **kw, seed=3, precision=P.MIXED)
    eF, edF, Fmax, fill, _ = _stage0(cfg, start, 0.0, sample=24)
    assert eF <= 1e-6 * Fmax + 2e-7 * 2 * (scale + abs(cfg.mu)), (eF, Fmax)
    assert edF <= 2e-6 * scale, edF
    eF, edF, Fmax, fill2, _ = _stage0(cfg, start, 1e6, sample=24)
    assert eF <= 1e-9 * Fmax and edF <= 1e-9 * scale, (eF, edF, Fmax)
    assert abs(fill - fill2) <= 2e-5 * max(1.0, abs(fill2)), (fill, fill2)


@pytest.mark.gpu
@pytest.mark.parametrize("T", [0.0363, 0.0361, 0.0181, 0.0180, 0.3, 3.0, 0.0046])
def test_temperatures_at_the_edges_of_the_node_classes(T):
    # 8x8 torus, 4x4 clusters: |mu - H| <= 18.5, so |x| crosses 512 near
    # T = 0.0361 and 1024 near 0.0181; 0.0046 lies just inside the path.
    cfg = P.Config(Lx=8, Ly=8, L_c=4, J_H=8.0, mu=-6.5, T=T, seed=1, precision=P.MIXED)
    eF, edF, Fmax, _, _ = _stage0(cfg, None, 0.0)
    assert eF <= 1e-6 * Fmax + 2e-7 * 40 and edF <= 2e-6 * 12, (eF, edF)
    eF, edF, Fmax, _, _ = _stage0(cfg, None, 1e6)
    assert eF <= 1e-9 * Fmax and edF <= 1e-9 * 12, (eF, edF)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [dict(Lx=8, Ly=8, L_c=4, stride=4), dict(Lx=24, Ly=24, L_c=4, schedule=P.SCHEDULE_BLOCK)])
def test_windows_beyond_the_node_classes_are_solved_exactly(shape):
    # mean fields of length up to 4000 at T = 0.1: |x| up to 1.6e5
    cfg = P.Config(**shape, T=0.1, seed=2, precision=P.MIXED, **HUB)
    start = inputs.random_fields(8, cfg.N, 4000.0)
    eF, edF, Fmax, _, _ = _stage0(cfg, start, 1e-2, sample=24)
    assert eF <= 1e-12 * Fmax and edF <= 1e-12 * Fmax, (eF, edF, Fmax)
