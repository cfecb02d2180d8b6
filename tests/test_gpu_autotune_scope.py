"""qed_autotune_groups times only what the context's step reads.  An FP32 table
context runs the single pass: of the groups only the photon stage has a launch
to size, and no scheduling value is read, so the rest keep 8 CTAs per SM (as
many as fit) and their defaults instead of what noise favours.  The library's
own launch count tells how many steps were timed: one configuration as it is and
one per candidate, each with an untimed step and `reps` timed ones."""
import numpy as np
import pytest
import torch

from _parity import to32

pytestmark = pytest.mark.gpu

DEFAULTS = {"emit_lanes": 16, "round_lanes": 12, "scan_draws": 8, "scan_left": 8, "queue_trigger": 32}


@pytest.mark.parametrize("precision,order,tuned,candidates", [
    (0, 0, ("photon",), 8), (0, 1, ("photon",), 8), (1, 0, ("stream", "chains", "order", "photon"), 4 * 8 + 5 + 4)])
def test_only_what_the_step_reads_is_timed(precision, order, tuned, candidates):
    import __graft_entry__ as ge
    ge.build()
    from paper_1608_06356_gb300 import api, workloads as W
    n, reps = 3000, 2
    dt = torch.float64 if precision else torch.float32
    st = W.ensemble(n, seed=4)
    st = st if precision else to32(st)
    ctx = api.qed_init_tables(api.config(dt=0.01, seed=2, precision=precision, append_order=order, max_particles=1 << 18))
    F = api.Fields.per_particle()

    def species():
        return (api.Species.empty(n, -1, dtype=dt, fields=True).load(**st),
                api.Species.empty(1000, 1, dtype=dt, fields=True), api.Species.empty(1 << 17, 0, dtype=dt, fields=True))

    e, p, g = species()
    before = ctx.launches
    api.qed_step_fused(ctx, e, p, g, F, 0)
    api.qed_compact_fill(ctx, g)
    per_step = ctx.launches - before
    e, p, g = species()
    before = ctx.launches
    t = api.qed_autotune_groups(ctx, e, p, g, F, reps=reps)
    assert ctx.launches - before == (1 + candidates) * (1 + reps) * per_step
    for name, f in t["grid_factor"].items():
        ms = t["ms"][name]
        if name in tuned:
            assert ms[f - 1] == min(ms) and len(set(ms)) > 1
        else:
            assert f == 8 and len(set(ms)) == 1, name
    for name, v in t["sched"].items():
        if not (precision and name in ("emit_lanes", "scan_draws")):
            assert v == DEFAULTS[name], name
    assert t["ms_per_step"] > 0 and np.isfinite(t["ms_per_step"])
