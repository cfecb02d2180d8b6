"""The single-pass lepton step's pool of chains and its slice copies.

- Pools that stay full (four leptons in five deferred, ten sub-steps each, several
  slices per warp) against the ordered path: the leptons and the photons as a
  set, within the xi tolerance of the two paths (1e-5, tests/test_gpu_onepass.py).
- Arrays off a 16-byte boundary take their words one by one instead of by
  16-byte copies: the same kernel on the same values, so bit for bit the same
  leptons and photons, with ragged last slices of both species."""
import numpy as np
import pytest
import torch

from _parity import to32
from test_gpu_onepass import _close_all, _run, _same_counters, _sorted, W, api  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


def test_full_pools_equal_ordered(api, W):  # noqa: F811
    n = 400_003
    st, _, _ = W.chi_target(n, seed=5, chi_lo=10.0, chi_hi=100.0)
    caps = (n, 1, 8 * n)
    o = _run(api, 0, to32(st), None, None, caps, 2, dt=0.02)
    u = _run(api, 1, to32(st), None, None, caps, 2, dt=0.02)
    assert o[3]["substeps"] > 6 * n and o[3]["deferred"] > 0.75 * n and o[3]["dropped"] == 0
    _close_all(o[0], u[0], "leptons")
    _close_all(_sorted(o[2]), _sorted(u[2]), "photons")
    _same_counters(o[3], u[3])


@pytest.mark.parametrize("mode", ["per_particle", "uniform"])
@pytest.mark.parametrize("ne,npos", [(1, 0), (31, 33), (4099, 257)])
def test_unaligned_arrays_give_the_same_bits(api, W, mode, ne, npos):  # noqa: F811
    fields = mode == "per_particle"
    names = ("x", "y", "z", "px", "py", "pz", "w", "id") + (("ex", "ey", "ez", "bx", "by", "bz") if fields else ())
    got = []
    for off in (0, 1):
        ctx = api.qed_init_tables(api.config(dt=0.05, seed=9, append_order=1))
        F = api.Fields.per_particle() if fields else api.Fields.uniform((0.0, 30.0, 0.0), (0.0, 0.0, 900.0))
        sp = []
        for n, q, seed in ((ne, -1, 31), (npos, 1, 32)):
            s = api.Species.empty(n + 1, q, fields=fields)
            for k in names:  # the same values, `off` elements into the allocation
                setattr(s, k, getattr(s, k)[off:off + n])
            if n:
                st = to32(W.ensemble(n, seed=seed, id0=0 if q < 0 else 10**6))
                s.load(**{k: st[k] for k in names})
            sp.append(s)
        g = api.Species.empty(40 * (ne + npos) + 64, 0, fields=fields)
        api.qed_step_fused(ctx, sp[0], sp[1], g, F, 3)
        torch.cuda.synchronize()
        got.append([sp[0].host(), sp[1].host(), _sorted(g.host())])
    assert got[0][2]["id"].size > 0 or ne == 1
    for a, b in zip(*got):
        for k in a:
            np.testing.assert_array_equal(a[k], b[k], err_msg=k)
