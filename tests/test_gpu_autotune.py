"""Autotuning of sweeps whose free energies come from determinants, where CTA width
and grid change nothing: a pipeline is timed once for all its candidates, and the
other reductions by themselves."""
import pytest

import paper_1502_07028_gb300 as P

pytestmark = pytest.mark.gpu


def test_candidates_that_are_the_same_launches_share_one_timing():
    ctx = P.Context(P.Config(Lx=16, Ly=16, L_c=4, schedule=P.SCHEDULE_BLOCK, T=0.05, seed=1, precision=P.MIXED))
    _, table = P.ptca_autotune(ctx.h, 2)
    ctx.close()
    times = {}
    for c in table["candidates"]:
        assert c["ms_per_sweep"] is not None
        own = (c["reduction"], c["panel_width"]) if c["reduction"] or c["panel_width"] > 1 else "determinants"
        times.setdefault((c["pipeline"], own), []).append(c["ms_per_sweep"])
    for pipeline in ("stages", "overlap", "persistent", "graph"):
        t = times[pipeline, "determinants"]
        assert len(t) >= 3 and len(set(t)) == 1, (pipeline, t)
    assert any(own != "determinants" for _, own in times)
