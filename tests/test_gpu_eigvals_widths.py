"""Batched FP32 eigenvalues at the counts where the CTA width changes (2, 3, 4
and 6 matrices per SM), orders up to 32 and above, open lattices (ragged
orders): every matrix against LAPACK on the oracle's matrix, at the bound of the
small batches."""
import numpy as np
import pytest
import torch

import oracle
import paper_1502_07028_gb300 as P
from paper_1502_07028_gb300 import _build
from tests import inputs

pytestmark = pytest.mark.gpu
TOL = 1e-5  # per J_H + 4t, as the small batches


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    assert torch.cuda.is_available()
    P.lib()


@pytest.mark.parametrize("per_sm, extra", [(2, 0), (2, 1), (3, 1), (4, 0), (4, 1), (6, 1)])
@pytest.mark.parametrize("L_c", [3, 4, 5, 8])
def test_batched_eigenvalues_at_width_changes(L_c, per_sm, extra):
    cfg = P.Config(Lx=12, Ly=11, L_c=L_c, periodic=0, schedule=P.SCHEDULE_BLOCK, precision=P.MIXED)
    m = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + extra
    ctx = P.Context(cfg)
    S = inputs.random_unit_spins(60 + L_c, cfg.N)
    ctx.set_spins(S)
    sites = np.arange(m) % cfg.N
    H, offs, n = ctx.build_clusters(sites)
    eig = ctx.cluster_eigvals(H, offs, n)[0].cpu().numpy()
    ctx.close()
    om = oracle.Model(Lx=12, Ly=11, Lc=L_c, lattice_periodic=0, schedule=oracle.SCHEDULE_BLOCK, JH=cfg.J_H, t=cfg.t)
    ref = [np.linalg.eigvalsh(oracle.cluster_hamiltonian(om, S, s)[0]) for s in range(min(m, cfg.N))]
    for i, s in enumerate(sites):
        assert np.max(np.abs(eig[i, : ref[s].size] - ref[s])) <= TOL * (cfg.J_H + 4 * cfg.t)
