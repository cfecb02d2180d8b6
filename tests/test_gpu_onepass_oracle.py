"""The single-pass lepton step against the FP64 oracle, in both append orders (one
kernel since ordered appends take it too, so comparing the orders with each other
tests the order and the positions, not the chains).

- Full pools: 400,003 leptons of chi 10 to 100, four in five deferred, six
  sub-steps and more on average, several slices a warp.  Draws are keyed by particle id, so
  the oracle steps a sample of them alone: 384 leptons from all over the ensemble,
  whole neighbouring slices and scattered ones.
- The classic photon model in FP32 contexts, whose default path (ordered appends)
  is the single pass with the rate bound taken from its tables.

Tolerances: 1e-5 relative in xi and 1 - xi per event (tests/test_gpu_step.py), ten
events of a lepton at most in the samples: 1e-4 for energies.  A draw within the
rate tolerance of its threshold (1e-4 of at most 0.2, per sub-step) may fall on the
other side; of 384 leptons with ten sub-steps 0.08 are expected to, 3 are allowed
(in the classic sample those of `ambiguous` besides)."""
import numpy as np
import pytest
import torch

from _parity import ambiguous, by_id, oracle_host, oracle_species, to32
from test_gpu_onepass import W, _gamma, _run, api  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu
RTOL, FLIPS = 1e-4, 3


def _against_oracle(orc, cfg, st, pick, e, g, step, dt, skip=None):
    """Leptons `pick` of the step's output (e by slot, g the photons) against the
    oracle's step of those leptons alone; returns the oracle's photons."""
    sub = {k: v[pick] for k, v in st.items()}
    oe = oracle_species(orc, len(pick), -1.0, sub, fields=True)
    og = oracle_species(orc, 64 * len(pick), 0.0, {k: v[:0] for k, v in sub.items()}, fields=True, alive=True)
    orc.step(cfg, orc.per_particle_fields(), oe, orc.Species(1, 1.0), og, step)
    o = oracle_host(oe)
    ok = np.abs(_gamma({k: e[k][pick] for k in ("px", "py", "pz")}) / _gamma(o) - 1) <= RTOL
    if skip is not None:
        ok |= skip
    assert (~ok).sum() <= FLIPS, np.flatnonzero(~ok)
    for c in ("x", "y", "z"):  # (the push comes before the emissions)
        np.testing.assert_allclose(e[c][pick], o[c], rtol=1e-6, atol=1e-5)
    # photons by id: the oracle's that are missing belong to the flipped leptons
    oi, os_ = by_id(oracle_host(og))
    gi, gs = by_id(g)
    common, io, ig = np.intersect1d(oi, gi, return_indices=True)
    lost = len(oi) - len(common)
    assert lost <= 10 * (FLIPS + (0 if skip is None else int(skip.sum()))), lost
    same = np.abs(_gamma({k: gs[k][ig] for k in ("px", "py", "pz")}, True) /
                  _gamma({k: os_[k][io] for k in ("px", "py", "pz")}, True) - 1) <= RTOL
    assert (~same).sum() <= 10 * (FLIPS + (0 if skip is None else int(skip.sum())))
    for c in ("x", "y", "z"):
        np.testing.assert_allclose(gs[c][ig], os_[c][io], rtol=1e-6, atol=1e-5)
    return oi


@pytest.mark.parametrize("order", [0, 1])
def test_full_pools_match_oracle(api, orc, W, order):  # noqa: F811
    n, dt, step, seed = 400_003, 0.02, 2, 12345
    st, _, _ = W.chi_target(n, seed=5, chi_lo=10.0, chi_hi=100.0)
    st = to32(st)
    e, _, g, c = _run(api, order, st, None, None, (n, 1, 8 * n), step, dt=dt, seed=seed)
    assert c["substeps"] > 6 * n and c["deferred"] > 0.75 * n and c["dropped"] == 0
    assert len(np.unique(g["id"])) == len(g["id"]) == c["emit_events"]
    rng = np.random.default_rng(1)
    pick = np.unique(np.concatenate([np.arange(32), 200_000 + np.arange(64), n - 1 - np.arange(32),
                                     rng.integers(0, n, 256)]))
    oi = _against_oracle(orc, orc.make_config(dt=dt, seed=seed), st, pick, e, g, step, dt)
    assert len(oi) > len(pick) // 2


@pytest.mark.parametrize("order", [0, 1])
def test_classic_model_matches_oracle(api, orc, W, order):  # noqa: F811
    n, dt, step, seed = 600, 0.02, 3, 77
    st, _, _ = W.chi_target(n, seed=9, chi_lo=1e-2, chi_hi=2.9, g_lo=200.0, g_hi=2000.0)
    st = to32(st)
    ctx = api.qed_init_tables(api.config(dt=dt, seed=seed, append_order=order, model=1))
    e = api.Species.empty(n, -1, fields=True).load(**st)
    g = api.Species.empty(20 * n, 0, fields=True)
    api.qed_step_fused(ctx, e, api.Species.empty(0, 1, fields=True), g, api.Fields.per_particle(), step)
    torch.cuda.synchronize()
    cfg = orc.make_config(dt=dt, seed=seed, model=orc.MODEL_CLASSIC)

    def fields(i):
        return (np.array([st["ex"][i], st["ey"][i], st["ez"][i]]), np.array([st["bx"][i], st["by"][i], st["bz"][i]]))

    amb = ambiguous(orc, cfg, st, fields, -1.0, step)
    oi = _against_oracle(orc, cfg, st, np.arange(n), e.host(), g.host(), step, dt, skip=amb)
    assert len(oi) > 20  # (35)
    c = api.qed_read_counters(ctx)
    assert abs(c["emit_events"] - len(oi)) <= 10 * (FLIPS + int(amb.sum())) and c["dropped"] == 0
