"""Failure detection of the stable compaction's bounded waits, with no GPU fault:
it runs with its first tile taken by nobody (qed_test_compact_expiry), in the
single launch (up to 1024 tiles) and in the two of a larger species, in both
precisions.  The tiles that wait for the first give up at the iteration limit,
within seconds, set QED_STATUS_TIMEOUT and return; the count stays as it was,
and the same context then compacts with a clean status.

Collected last, as tests/test_zz_wait_expiry.py."""
import time

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n", [(0, 20_000), (1, 20_000), (0, 600_000), (1, 300_000)])
def test_compaction_waits_expire_with_status(precision, n):
    import __graft_entry__ as ge
    ge.build()
    from paper_1608_06356_gb300 import _binding as B, api
    dt = torch.float64 if precision else torch.float32
    ctx = api.qed_init_tables(api.config(precision=precision, max_particles=n))
    rng = np.random.default_rng(n)
    alive = (rng.uniform(size=n) < 0.9).astype(np.uint8)
    alive[:3] = 0

    def species():
        g = api.Species.empty(n, 0, dtype=dt)
        g.id.copy_(torch.arange(n, device="cuda"))
        g.x.copy_(torch.arange(n, device="cuda").to(dt))
        g.alive.copy_(torch.from_numpy(alive))
        g.n.fill_(n)
        return g

    g = species()
    api.qed_reset_counters(ctx)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    api.qed_test_compact_expiry(ctx, g)
    bits, _ = api.qed_last_device_status(ctx)  # waits for the kernels
    assert time.perf_counter() - t0 < 60.0
    assert bits == B.QED_STATUS_TIMEOUT
    assert g.count() == n
    api.qed_reset_counters(ctx)
    for _ in range(2):
        g = species()
        api.qed_compact(ctx, g)
        assert api.qed_last_device_status(ctx)[0] == 0
        keep = np.flatnonzero(alive)
        assert g.count() == len(keep)
        np.testing.assert_array_equal(g.host(["id"])["id"], keep.astype(np.uint64))
        np.testing.assert_array_equal(g.host(["x"])["x"], keep.astype(np.float64 if precision else np.float32))
