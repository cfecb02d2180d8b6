"""The tiled current deposit of clustered plasmas against the FP64 oracle of
oracle/pic.py: cells with more particles than a thread sums (24 of a batch of
2048), with more than a warp's chunk of 256, batches of one cell alone, tiles of
several parts (8192 records), light and heavy cells in the same batch, and
clusters on the edges of tiles and of the periodic box.

Tolerance: that of tests/test_gpu_pic_tiled.py, 3e-5 of the largest J.  It is
the rounding of a particle's coordinates against its own current; the sums of
a cell are shorter here than there (at most 24 in a row by a thread, 8 by a lane
and 5 over the lanes)."""
import numpy as np
import pytest
import torch

from _parity import to32

pytestmark = pytest.mark.gpu
STATE = ("x", "y", "z", "px", "py", "pz", "w")
N, SHAPE, D, O = 1_000_003, (66, 61, 70), (0.5, 0.3, 0.45), (0.2, -0.4, 1.0)


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_1608_06356_gb300 import api as A
    return A


def _cells(kind, rng):
    """Cell coordinates of the particles."""
    u = rng.uniform(0.0, SHAPE, (N, 3))
    if kind == "one cell":
        u = np.array([9.0, 17.0, 6.0]) + rng.uniform(0, 1, (N, 3))
    elif kind == "half in one cell":
        u[::2] = np.array([7.0, 8.0, 3.0]) + rng.uniform(0, 1, (len(u[::2]), 3))
    elif kind == "box corner":
        u[: N // 2] = rng.normal(0.0, 1.5, (N // 2, 3))
    elif kind == "ball":
        u = np.array([33.0, 30.0, 35.0]) + rng.normal(0.0, 4.0, (N, 3))
    elif kind == "sheet":
        u[:, 0] = 31.0 + rng.uniform(0, 1, N)
    elif kind == "sorted lines":  # 25 and 24 a cell in places, by cell
        u[:, 1] = np.floor(u[:, 1] / 8) * 8 + rng.uniform(0, 1, N)
        u[:, 0] = np.floor(u[:, 0] / 4) * 4 + rng.uniform(0, 1, N)
        u = u[np.lexsort(np.floor(u).T)]
    return u


@pytest.mark.parametrize("kind", ["one cell", "half in one cell", "box corner", "ball", "sheet", "sorted lines"])
def test_clustered_deposit_matches_oracle(api, kind):
    from oracle import pic as P
    rng = np.random.default_rng(len(kind))
    u = _cells(kind, rng)
    st = {k: o + d * v for k, v, d, o in zip("xyz", u.T, D, O)}
    st.update({k: rng.normal(scale=2.0, size=N) for k in ("px", "py", "pz")})
    st = to32(dict(st, w=rng.uniform(0.5, 2.0, N), id=np.arange(N, dtype=np.uint64)))
    ctx = api.qed_init_tables(api.config(dt=0.1, max_particles=1 << 20))
    y, g = api.Yee(*SHAPE, *D, *O), P.Grid(*SHAPE, *D, *O)
    e = api.Species.empty(N, -1).load(**st)
    before = ctx.launches
    api.qed_pic_deposit(ctx, e, y, 1.7)
    assert ctx.launches - before > 1  # the tiled path's
    P.deposit(g, *(st[k] for k in STATE), -1.0, 0.1, 1.7)
    torch.cuda.synchronize()
    for nm in ("jx", "jy", "jz"):
        ref = getattr(g, nm)
        np.testing.assert_allclose(getattr(y, nm).cpu().numpy(), ref, rtol=0, atol=3e-5 * np.abs(ref).max(), err_msg=nm)
    assert api.qed_read_counters(ctx)["status"] == 0
