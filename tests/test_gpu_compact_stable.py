"""qed_compact (stable in-place removal of dead particles) against its
definition, exactly: the live particles in their order, in front.  Sizes at
the edges of its tiles (512 particles in FP32, 256 in FP64), of the single
launch it uses for capacities of up to 512 tiles and of the rounds of its scan
(8192 tiles), fewer particles than the capacity, no and only dead particles,
a leading part that stays where it is, and twice in a row on one context (the
scratch must be back at zero)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

FIELDS = ("x", "y", "z", "px", "py", "pz", "w", "ex", "ey", "ez", "bx", "by", "bz")


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_1608_06356_gb300 import api as A
    return A


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("n,spare,dead", [
    (0, 5, 0.0), (1, 0, 0.0), (1, 0, 1.0), (255, 0, 0.3), (256, 1, 0.3), (257, 0, 0.01), (512, 0, 0.3), (513, 0, 0.5),
    (5000, 300_000, 0.3), (131_072, 0, 0.02), (131_073, 0, 0.02), (262_144, 0, 0.02), (262_145, 0, 0.02), (524_288, 0, 0.1), (524_289, 0, 0.1),
    (300_001, 0, 1.0), (300_001, 0, 0.0), (4_194_305, 0, 0.001), (4_300_000, 7, 0.5)])
def test_stable_compaction(api, precision, n, spare, dead):
    dt, npdt = (torch.float32, np.float32) if precision == 32 else (torch.float64, np.float64)
    rng = np.random.default_rng(n + precision)
    ctx = api.qed_init_tables(api.config(precision=0 if precision == 32 else 1, max_particles=max(n + spare, 1)))
    with_fields, with_tag = n % 2 == 1, n % 3 != 0
    for again in range(2):
        st = {k: rng.standard_normal(n).astype(npdt) for k in (FIELDS if with_fields else FIELDS[:7])}
        st["id"] = rng.integers(0, 1 << 63, size=n, dtype=np.uint64)
        if with_tag:
            st["tag"] = rng.integers(0, 1 << 31, size=n).astype(np.uint32)
        alive = (rng.uniform(size=n) >= dead).astype(np.uint8)
        if again:
            alive[: n // 3] = 1
        g = api.Species.empty(n + spare, 0, dtype=dt, fields=with_fields, tag=with_tag).load(**st)
        g.alive[:n].copy_(torch.tensor(alive))
        api.qed_compact(ctx, g)
        torch.cuda.synchronize()
        keep = np.flatnonzero(alive)
        assert g.count() == len(keep)
        h = g.host()
        for k, v in st.items():
            np.testing.assert_array_equal(h[k].view(v.dtype), v[keep], err_msg=k)
        assert bool((g.alive[: len(keep)] == 1).all())
        assert api.qed_read_counters(ctx)["status"] == 0
