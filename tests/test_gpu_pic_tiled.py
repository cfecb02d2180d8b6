"""The tiled current deposit (2^18 particles and more) against the
FP64 oracle of oracle/pic.py and against the direct deposit.

Tolerance, from the arithmetic: a float weight carries the rounding of a
reduced coordinate of up to 128 cells, 128 * 2^-24 = 8e-6 of the particle's
current; N particles of a cell add as sqrt(N), as their currents of either sign
do, so a cell is within about 8e-6 / 0.35 (the rms CIC weight) = 2e-5 of the
largest J, taken as 3e-5.  FP64 contexts add doubles and round to float once
per tile, at most 27 tiles to a cell: 27 * 2^-24 = 2e-6; with particles left
to the direct deposit (about 3500 float additions to a cell, their roundings of
either sign) that deposit's 1e-5."""
import numpy as np
import pytest
import torch

from _parity import to32

pytestmark = pytest.mark.gpu
STATE = ("x", "y", "z", "px", "py", "pz", "w")


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_1608_06356_gb300 import api as A
    return A


def _particles(n, box, seed):
    rng = np.random.default_rng(seed)
    st = {k: rng.uniform(-0.3 * b, 1.3 * b, n) for k, b in zip("xyz", box)}  # also outside the box
    st.update({k: rng.normal(scale=2.0, size=n) for k in ("px", "py", "pz")})
    return dict(st, w=rng.uniform(0.5, 2.0, n), id=np.arange(n, dtype=np.uint64))


# ragged tiles, one cell along an axis, two particles a cell, 60
# particles a cell, and more particles than records (65536 max_particles:
# 131072 records)
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape,n,max_particles", [
    ((257, 3, 41), 262144, 1 << 20), ((1, 70, 64), 270001, 1 << 20), ((67, 65, 5), 262147, 1 << 20),
    ((96, 81, 17), 264385, 1 << 20), ((16, 16, 132), 270001, 1 << 16)])
def test_tiled_deposit_matches_oracle(api, precision, shape, n, max_particles):
    from oracle import pic as P
    d, o = (0.5, 0.3, 0.45), (0.2, -0.4, 1.0)
    ctx = api.qed_init_tables(api.config(dt=0.1, precision=precision, max_particles=max_particles))
    y, g = api.Yee(*shape, *d, *o), P.Grid(*shape, *d, *o)
    st = _particles(n, [s * c for s, c in zip(shape, d)], n + precision)
    st = st if precision else to32(st)
    st["px"][5] = np.nan  # reported and left out
    e = api.Species.empty(n, -1, dtype=torch.float64 if precision else torch.float32).load(**st)
    api.qed_pic_deposit(ctx, e, y, 1.7)
    keep = np.arange(n) != 5
    tol = 3e-5 if not precision else 1e-5 if max_particles == 1 << 16 else 2e-6
    P.deposit(g, *(st[k][keep] for k in STATE), -1.0, 0.1, 1.7)
    torch.cuda.synchronize()
    for nm in ("jx", "jy", "jz"):
        ref = getattr(g, nm)
        np.testing.assert_allclose(getattr(y, nm).cpu().numpy(), ref, rtol=0,
                                   atol=tol * np.abs(ref).max(), err_msg=nm)
    assert api.qed_read_counters(ctx)["status"] & 4


def test_infinite_weight_reaches_the_same_nodes(api):
    """A particle of infinite weight makes the same elements of J non-finite
    on the direct path (alone) and on the tiled one (among many)."""
    ctx = api.qed_init_tables(api.config(dt=0.1, max_particles=1 << 19))
    bad = []
    for n in (1, 1 << 18):
        st = _particles(n, (48 * 0.5, 36 * 0.5, 20 * 0.5), 3)
        for k in ("x", "y", "z", "px", "py", "pz"):
            st[k][0] = 1.3
        st["w"][0] = np.inf
        y = api.Yee(48, 36, 20, 0.5, 0.5, 0.5)
        api.qed_pic_deposit(ctx, api.Species.empty(n, -1).load(**to32(st)), y, 1.0)
        bad.append([~torch.isfinite(getattr(y, nm)).cpu().numpy() for nm in ("jx", "jy", "jz")])
    for a, b in zip(*bad):
        assert a.sum() == 8
        np.testing.assert_array_equal(a, b)
