"""The photon stage when every photon of a full species converts in one step: a
record for each pair, at the values of max_particles where the records are
fewest (qed_scratch.h: the minimum sizes hold 16384 and 131072 pairs) and one
below them.  The result is that of a larger context with the same photons, bit
for bit (the same kernels, appends in photon order), in both precisions and
with the records' field words (grid fields)."""
import numpy as np
import pytest
import torch

from _parity import to32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_1608_06356_gb300 import api as A
    return A


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,mode", [(16384, "per_particle"), (16385, "per_particle"), (16387, "grid"),
                                    (131073, "per_particle"), (131073, "grid")])
def test_every_photon_converts(api, precision, n, mode):
    from paper_1608_06356_gb300 import workloads as W
    st = W.ensemble(n, seed=n, photons=True, g_lo=1e3, g_hi=3e3, f_lo=2000.0, f_hi=4000.0)
    if mode == "grid":
        st = {k: v for k, v in st.items() if k not in ("ex", "ey", "ez", "bx", "by", "bz")}
        grid = np.zeros((4, 4, 4, 8), dtype=np.float32)
        grid[..., 3:6] = np.random.default_rng(1).uniform(2000.0, 4000.0, (4, 4, 4, 3))
        F = api.Fields.grid(torch.from_numpy(grid).cuda(), 0.5, 0.5, 0.5)
    else:
        F = api.Fields.per_particle()
    st = st if precision else to32(st)
    dt = torch.float64 if precision else torch.float32
    got = []
    for max_particles in (n, 1 << 19):
        ctx = api.qed_init_tables(api.config(dt=300.0, seed=6, precision=precision, max_particles=max_particles))
        g = api.Species.empty(n, 0, dtype=dt, fields=mode == "per_particle").load(**st)
        e, p = (api.Species.empty(n, q, dtype=dt, fields=True) for q in (-1, 1))
        api.qed_pair(ctx, g, e, p, F, 2)
        torch.cuda.synchronize()
        got.append((e.host(), p.host(), g.host(), api.qed_read_counters(ctx)))
    # parallel photons and fields may leave a few below the pair threshold
    assert got[0][3]["pair_events"] > n - n // 100 and got[0][3]["dropped"] == 0
    assert len(got[0][0]["x"]) == len(got[0][1]["x"]) == got[0][3]["pair_events"]
    for a, b in zip(got[0][:3], got[1][:3]):
        for k in a:
            np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    assert got[0][3] == got[1][3]
