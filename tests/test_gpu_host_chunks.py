"""qed_lepton_step_host takes the chunks the caller names: with ordered appends
the photons of a call lie chunk by chunk, each as qed_emit's step of those
leptons alone appends them -- compared bit for bit, on the device species and on
the host mirror, with one qed_step_fused call per chunk (without photons at its
start, so that its photon stage does nothing).  Chunks that are no multiple of
four start off a 16-byte boundary of the host arrays; all element sizes (FP32,
FP64, ids, tags), one and three leptons a chunk, and arrays the device maps at
an odd element (copied without the SMs) are covered."""
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


@pytest.mark.parametrize("precision,order,n,chunk,shift", [
    (0, 0, 10_001, 1001, 0), (0, 0, 10_001, 1002, 0), (0, 0, 3_000, 1000, 0), (0, 0, 101, 3, 0), (0, 0, 7, 1, 0),
    (0, 0, 5_003, 999, 1), (1, 0, 5_001, 1003, 0), (0, 1, 10_001, 1001, 0)])
def test_chunks_are_the_callers(api, precision, order, n, chunk, shift):
    from paper_1608_06356_gb300 import workloads as W
    st, _, _ = W.chi_target(n, seed=n + chunk, chi_lo=0.1, chi_hi=30.0)
    st = dict(st if precision else to32(st), tag=np.arange(n, dtype=np.uint32))
    dt = torch.float64 if precision else torch.float32
    ctx = api.qed_init_tables(api.config(dt=0.05, seed=5, precision=precision, append_order=order,
                                         max_particles=1 << 17))
    F, cap = api.Fields.per_particle(), 1 << 16
    host = api.Species.empty(n + shift, -1, dtype=dt, fields=True, tag=True, pinned=True)
    for k in [k for k in st if shift]:
        setattr(host, k, getattr(host, k)[shift:])
    host.load(**st)
    g = api.Species.empty(cap, 0, dtype=dt, fields=True, tag=True)
    mirror = api.Species.empty(cap, 0, dtype=dt, fields=True, tag=True, pinned=True)
    api.qed_lepton_step_host(ctx, host, g, mirror, F, 4, chunk)
    got, m = g.host(), int(mirror.n[0])
    assert m == g.count() > 0 or n < 10
    ref, leptons = [], []
    none = api.Species.empty(0, 1, dtype=dt, fields=True, tag=True)
    for a in range(0, n, chunk):
        part = {k: v[a:a + chunk] for k, v in st.items()}
        e = api.Species.empty(len(part["x"]), -1, dtype=dt, fields=True, tag=True).load(**part)
        gp = api.Species.empty(cap, 0, dtype=dt, fields=True, tag=True)
        api.qed_step_fused(ctx, e, none, gp, F, 4)
        torch.cuda.synchronize()
        ref.append(gp.host())
        leptons.append(e.host())
    ref, leptons = ({k: np.concatenate([r[k] for r in rs]) for k in rs[0]} for rs in (ref, leptons))
    for k in got:  # the mirror is the device species
        np.testing.assert_array_equal(getattr(mirror, k)[:m].numpy().view(got[k].dtype), got[k], err_msg=k)
    if order == 1:  # any order within a chunk, the chunks in order
        first = np.cumsum([0] + [np.count_nonzero(ref["tag"] // chunk == c) for c in range((n + chunk - 1) // chunk)])
        for s in (ref, got):
            o = np.concatenate([a + np.argsort(s["id"][a:b], kind="stable") for a, b in zip(first, first[1:])])
            s.update({k: v[o] for k, v in s.items()})
    for k in ref:
        np.testing.assert_array_equal(got[k], ref[k], err_msg=k)
    for k in leptons:
        a = getattr(host, k)[:n].numpy()
        np.testing.assert_array_equal(a.view(leptons[k].dtype), leptons[k], err_msg=k)
