"""Mixed sweeps so hot that the scales 1 / (T y) of the determinants' nodes are below
the smallest float: every level is at the middle of the Fermi function, and the
free energy of a matrix of order n is -n T ln 2 to the nodes' 3e-7 per level."""
import numpy as np
import pytest

import paper_1502_07028_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1e36, 1e44, 1e50])
@pytest.mark.parametrize("kw", [dict(Lx=8, Ly=8, L_c=4), dict(Lx=32, Ly=32, L_c=4, schedule=P.SCHEDULE_BLOCK),
                                dict(Lx=32, Ly=32, L_c=8, schedule=P.SCHEDULE_BLOCK)], ids=["few", "small", "square"])
def test_scales_below_the_floats(kw, T):
    ctx = P.Context(P.Config(**kw, T=T, J_H=8.0, mu=-6.5, seed=1, precision=P.MIXED))
    ctx.sweep(1)
    _, Fo, Fn, _, acc = (x.cpu().numpy() for x in ctx.record())
    filling = ctx.observables().filling
    ctx.close()
    n = 2 * kw["L_c"] ** 2
    for F in (Fo, Fn):
        assert np.max(np.abs(F / (-n * T * np.log(2.0)) - 1.0)) <= 3e-7 / np.log(2.0) * 1.01
    assert np.all(acc == 1) and abs(filling - 1.0) <= 1e-9
