"""qed_autotune_groups times only what the context's step reads.  An FP32 table
context runs the single pass: of the groups only the photon stage has a launch
to size, and no scheduling value is read, so the rest keep 8 CTAs per SM (as
many as fit) and their defaults instead of what noise favours.  The
library's own launch count tells how many steps were timed: one
configuration as it is and, per setting, its default before and after each of its
m candidates (2 m + 1), each with an untimed step and `reps` timed ones.

The population grows while it is tuned; a value must not win for having been
timed first."""
import numpy as np
import pytest
import torch

from _parity import to32

pytestmark = pytest.mark.gpu

DEFAULTS = {"emit_lanes": 16, "round_lanes": 12, "scan_draws": 8, "scan_left": 8, "queue_trigger": 32}


@pytest.mark.parametrize("precision,order,tuned,timed", [
    (0, 0, ("photon",), 17), (0, 1, ("photon",), 17),
    (1, 0, ("stream", "chains", "order", "photon"), 4 * 17 + 11 + 9)])
def test_only_what_the_step_reads_is_timed(precision, order, tuned, timed):
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
    assert ctx.launches - before == (1 + timed) * (1 + reps) * per_step
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


def test_growth_of_the_population_does_not_decide():
    """Electrons that emit about half a photon a step, tuned from no photons: by
    absolute times the candidates grow dearer as they are timed.  Relative to the
    default, 8 CTAs per SM, which is as many as fit, has the time of the step as it
    is within a tenth."""
    import __graft_entry__ as ge
    ge.build()
    from paper_1608_06356_gb300 import api, workloads as W
    n = 1 << 20
    st, _, _ = W.chi_target(n, seed=6, chi_lo=5.0, chi_hi=20.0, g_lo=2000.0, g_hi=9000.0)
    ctx = api.qed_init_tables(api.config(dt=0.02, seed=2, append_order=1, max_particles=1 << 24))
    e = api.Species.empty(1 << 22, -1, fields=True).load(**to32(st))
    p = api.Species.empty(1 << 22, 1, fields=True)
    g = api.Species.empty(1 << 24, 0, fields=True)
    t = api.qed_autotune_groups(ctx, e, p, g, api.Fields.per_particle(), reps=3)
    assert g.count() > n
    assert abs(t["ms"]["photon"][7] / t["ms"]["stream"][7] - 1) < 0.1, t["ms"]
