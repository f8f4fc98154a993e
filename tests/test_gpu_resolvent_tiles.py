"""The largest tiles of the determinant kernels, against the oracle: windows of 12
to 16 sites per layer and 4x4x4 windows split by parity, in stages small enough
for one visit per CTA and large enough for several.

Tolerances as in test_gpu_resolvent.py: F to 1e-6 of itself plus 2e-7 of twice
the spectrum's reach, dF to 2e-6 of the couplings; double-float to 1e-9."""
import pytest

import paper_1502_07028_gb300 as P
from tests import inputs
from tests.test_gpu_resolvent import HUB, _stage0

pytestmark = pytest.mark.gpu
BLOCK = dict(schedule=P.SCHEDULE_BLOCK)


@pytest.mark.parametrize("L_c,T", [(15, 0.2), (16, 0.2), (16, 0.6), (15, 0.01)])
def test_large_clusters_on_lattices_of_many_visits(L_c, T):
    # 3136 visits a stage: several share a CTA where its shared memory holds them
    cfg = P.Config(Lx=112, Ly=112, L_c=L_c, J_H=8.0, mu=-6.5, T=T, seed=L_c, precision=P.MIXED, **BLOCK)
    eF, edF, Fmax, _, _ = _stage0(cfg, None, 0.0, sample=1)
    assert eF <= 1e-6 * Fmax + 2e-7 * 2 * 20.5 and edF <= 2e-6 * 14, (eF, edF, Fmax)


@pytest.mark.parametrize("margin", [0.0, 1e6])
@pytest.mark.parametrize("shape", [dict(Lx=24, Ly=24, L_c=12, **BLOCK), dict(Lx=26, Ly=27, L_c=13, **BLOCK),
                                   dict(Lx=32, Ly=34, L_c=16, **BLOCK), dict(Lx=33, Ly=31, L_c=15, periodic=0, stride=15)],
                         ids=lambda d: "x".join(str(v) for v in d.values()))
def test_large_windows(shape, margin):
    cfg = P.Config(**shape, J_H=8.0, mu=-6.5, T=0.05, seed=4, precision=P.MIXED)
    eF, edF, Fmax, _, _ = _stage0(cfg, None, margin, sample=1 if cfg.L_c == 16 else 3)
    if margin:
        assert eF <= 1e-9 * Fmax and edF <= 1e-9 * 14, (eF, edF, Fmax)
    else:
        assert eF <= 1e-6 * Fmax + 2e-7 * 2 * 20.5 and edF <= 2e-6 * 14, (eF, edF, Fmax)


@pytest.mark.parametrize("margin", [0.0, 1e6])
@pytest.mark.parametrize("L", [12, 24])
def test_cubes_of_parity_split_windows(L, margin):
    # 216 visits a stage, and 1728 with several visits per CTA
    cfg = P.Config(Lx=L, Ly=L, Lz=L, L_c=4, T=0.15, seed=5, precision=P.MIXED, **BLOCK, **HUB)
    start = inputs.random_fields(6, cfg.N, 1.5)
    eF, edF, Fmax, _, _ = _stage0(cfg, start, margin, sample=6)
    if margin:
        assert eF <= 1e-9 * Fmax and edF <= 1e-9 * 14, (eF, edF, Fmax)
    else:
        assert eF <= 1e-6 * Fmax + 2e-7 * 2 * 18 and edF <= 2e-6 * 14, (eF, edF, Fmax)


@pytest.mark.parametrize("Lx,Ly,L_c,T", [(57, 61, 9, 0.04), (60, 60, 11, 0.0375), (59, 59, 10, 0.013), (60, 60, 12, 0.007)])
def test_two_visits_of_two_node_warps_in_a_cta(Lx, Ly, L_c, T):
    # 899 or 900 visits a stage of 15, 17 or 19 nodes, on seven warps of two nodes
    cfg = P.Config(Lx=Lx, Ly=Ly, L_c=L_c, J_H=8.0, mu=-6.5, T=T, seed=L_c, precision=P.MIXED, **BLOCK)
    eF, edF, Fmax, _, _ = _stage0(cfg, None, 0.0, sample=2)
    assert eF <= 1e-6 * Fmax + 2e-7 * 2 * 20.5 and edF <= 2e-6 * 14, (eF, edF, Fmax)
