"""Ordered appends of the single-pass lepton step: where its records of photons
find no room (more photons in a step than max_particles), the leptons concerned
are replayed from their stored state.  The result is the one of a context whose
records all fit: the same counts, ids and order, and the values within the xi
tolerance of two kernels that round the same expressions (1e-5,
tests/test_gpu_onepass.py).  Sizes: a few records too many, most of them, tiles
and chunks of 2048 slots with ragged ends, two species, grid fields (records of
96 bytes)."""
import numpy as np
import pytest
import torch

from _parity import to32
from test_gpu_onepass import _close_all, _same_counters, W, api  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


def _step(api, max_particles, e_st, p_st, cap_g, F, fields, dt, steps):  # noqa: F811
    ctx = api.qed_init_tables(api.config(dt=dt, seed=4, max_particles=max_particles))
    e = api.Species.empty(len(e_st["x"]), -1, fields=fields).load(**e_st)
    p = api.Species.empty(max(len(p_st["x"]), 1), 1, fields=fields).load(**p_st)
    g = api.Species.empty(cap_g, 0, fields=True)
    for s in range(steps):  # the second step finds the counters as the first left them
        api.qed_step_fused(ctx, e, p, g, F, s)
    torch.cuda.synchronize()
    return e.host(), p.host(), g.host(), api.qed_read_counters(ctx)


@pytest.mark.parametrize("mode,ne,npos,dt", [("per_particle", 40_001, 2_300, 0.05), ("per_particle", 60_000, 1, 0.15),
                                             ("uniform", 20_003, 20_001, 0.1), ("grid", 30_001, 511, 0.1)])
def test_lost_records_are_replayed(api, W, mode, ne, npos, dt):  # noqa: F811
    fields = mode == "per_particle"
    st, _, _ = W.chi_target(ne + npos, seed=8, chi_lo=5.0, chi_hi=50.0, g_lo=300.0, g_hi=900.0)
    st = to32(st)
    if not fields:
        st = {k: v for k, v in st.items() if k not in ("ex", "ey", "ez", "bx", "by", "bz")}
    if mode == "grid":
        rng = np.random.default_rng(2)
        grid = torch.from_numpy(rng.normal(scale=6000.0, size=(5, 6, 7, 8)).astype(np.float32)).cuda()
        F = api.Fields.grid(grid, 0.7, 0.8, 0.9)
    else:
        F = api.Fields.per_particle() if fields else api.Fields.uniform((0.0, 50.0, 0.0), (0.0, 0.0, 9000.0))
    a, b = {k: v[:ne] for k, v in st.items()}, {k: v[ne:] for k, v in st.items()}
    cap_g = 1 << 16
    # (grid: the leptons' stage only)
    steps = 1 if mode == "grid" else 2
    small = _step(api, 1 << 16, a, b, cap_g, F, fields, dt, steps)
    large = _step(api, 1 << 22, a, b, cap_g, F, fields, dt, steps)
    _same_counters(small[3], large[3])
    records = (1 << 20) // (16 if mode == "uniform" else 24)
    assert large[3]["emit_events"] > records and large[3]["dropped"] > 0
    for i, what in enumerate(("electrons", "positrons", "photons")):
        assert len(small[i]["x"]) == len(large[i]["x"])
        _close_all(small[i], large[i], what)
