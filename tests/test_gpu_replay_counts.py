"""Ordered appends, leptons replayed because the photon records ran out: a replay
that disagrees with the photon count of its lepton (here because its emission
rate is changed, qed_test_replay_rate) keeps to the places the count gave it.
Every photon's weight names its parent, so the places of a step can be compared
with those of a context whose records all fit: the same parents at the same
indices, the same leptons' order and count.  A replay without events fills its
places with photons of zero energy and sets QED_STATUS_REPLAY; one with more
events than places stops; one that agrees leaves the status clean."""
import numpy as np
import pytest
import torch

from _parity import to32
from test_gpu_onepass import W, api  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["per_particle", "uniform"])
@pytest.mark.parametrize("factor", [1.0, 0.0, 50.0])
def test_replays_keep_to_their_places(api, W, mode, factor):  # noqa: F811
    from paper_1608_06356_gb300 import _binding as B
    n, fields = 50_001, mode == "per_particle"
    st, _, _ = W.chi_target(n, seed=8, chi_lo=5.0, chi_hi=50.0, g_lo=300.0, g_hi=900.0)
    st = to32(dict(st, w=np.arange(1.0, n + 1)))
    if not fields:
        st = {k: v for k, v in st.items() if k not in ("ex", "ey", "ez", "bx", "by", "bz")}
    F = api.Fields.per_particle() if fields else api.Fields.uniform((0.0, 50.0, 0.0), (0.0, 0.0, 9000.0))
    got = []
    for max_particles, f in ((1 << 16, factor), (1 << 22, 1.0)):
        ctx = api.qed_init_tables(api.config(dt=0.08, seed=4, max_particles=max_particles))
        api.qed_test_replay_rate(ctx, f)
        e = api.Species.empty(n, -1, fields=fields).load(**st)
        g = api.Species.empty(1 << 16, 0, fields=True)
        api.qed_step_fused(ctx, e, api.Species.empty(1, 1, fields=fields), g, F, 1)
        torch.cuda.synchronize()
        got.append((g.host(), api.qed_read_counters(ctx)))
    (g, c), (ref, cr) = got
    assert cr["emit_events"] > (1 << 20) // (16 if mode == "uniform" else 24)  # more than the records
    for k in ("emit_events", "dropped", "substeps", "hist"):
        assert c[k] == cr[k], k
    assert not cr["status"] & B.QED_STATUS_REPLAY
    np.testing.assert_array_equal(g["w"], ref["w"])
    assert (g["alive"] == 1).all()
    soft = (g["px"] == 0) & (g["py"] == 0) & (g["pz"] == 0)
    replayed = bool(c["status"] & B.QED_STATUS_REPLAY)
    if factor == 1.0:
        assert not replayed and not soft.any()
        np.testing.assert_array_equal(g["id"], ref["id"])
    elif factor == 0.0:
        assert replayed and 0 < soft.sum() < len(soft)
        np.testing.assert_array_equal(g["id"][~soft], ref["id"][~soft])
    else:  # the leptons that were not replayed have their photons
        assert (g["id"] == ref["id"]).mean() > 0.1
