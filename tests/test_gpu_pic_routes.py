"""Which current deposit a call takes, and the same J by each.  FP64 contexts
deposit directly, by one launch, at every size: the tiled sums took twice the
time there (2369 us against 1093 at 128^3 cells and 2^22 electrons).  FP32
contexts take tiles from 3 2^17 particles on (and two per cell; for a J larger
than L2 half of one where their order is scattered)."""
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


def _electrons(api, n, box, dtype=torch.float32, seed=1, capacity=None):
    gen = torch.Generator("cuda").manual_seed(seed)
    e = api.Species.empty(capacity or n, -1, dtype=dtype)
    for k in ("x", "y", "z", "px", "py", "pz", "w"):
        r = torch.rand(n, generator=gen, device="cuda", dtype=dtype)
        getattr(e, k)[:n] = r * box if k in "xyz" else r + 0.5 if k == "w" else 4 * r - 2
    e.n.fill_(n)
    return e


def test_fp64_deposits_directly(api):
    n = 1 << 20
    ctx = api.qed_init_tables(api.config(dt=0.1, precision=1, max_particles=n))
    y = api.Yee(64, 64, 64, 1.0, 1.0, 1.0)
    e = _electrons(api, n, 64.0, torch.float64)
    before = ctx.launches
    api.qed_pic_deposit(ctx, e, y, 1.0)
    torch.cuda.synchronize()
    assert ctx.launches - before == 1


def _time(fn, n=5):
    ms = []
    for _ in range(n + 2):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b))
    return sorted(ms[2:])[n // 2]


def test_a_full_cell_does_not_hold_up_the_tiled_deposit(api):
    """2^20 electrons, half of them in one cell: while a cell was one thread's
    work this took about a thousand times as long as a uniform plasma; summed by
    warps and by several CTAs it is of the same order (30 times allowed)."""
    n = 1 << 20
    ctx = api.qed_init_tables(api.config(dt=0.1, max_particles=n))
    y = api.Yee(64, 64, 64, 1.0, 1.0, 1.0)
    e = _electrons(api, n, 64.0)
    uniform = _time(lambda: api.qed_pic_deposit(ctx, e, y, 1.0))
    for k in "xyz":
        getattr(e, k)[: n // 2].mul_(1.0 / 64).add_(5.0)
    clustered = _time(lambda: api.qed_pic_deposit(ctx, e, y, 1.0))
    assert clustered < 30 * uniform, (clustered, uniform)


def _deposit(api, ctx, e, shape, count=None):
    y = api.Yee(*shape, 1.0, 1.0, 1.0)
    before = ctx.launches
    api.qed_pic_deposit(ctx, e, y, 1.0, count)
    torch.cuda.synchronize()
    return torch.stack([y.jx, y.jy, y.jz]), ctx.launches - before


def test_few_particles_of_a_large_capacity(api):
    """A species with room for the tiled path and few particles in it: four
    launches (the scatter pass deposits directly, the others return at once;
    five and a clear before), the J of the same particles in a species of their
    own size, and tiled calls between leave the scratch as it was.  The two add
    the same floats in another order: 2^-24 per addition, at most 8 n of them to
    a cell, random signs (at 3000 particles in 2^18 cells a few: 1e-6 of the
    largest J)."""
    shape, cap = (64, 64, 64), 1 << 20
    ctx = api.qed_init_tables(api.config(dt=0.1, max_particles=cap))
    full = _electrons(api, cap, 64.0, seed=2)
    ref_full = None
    for n in (1, 255, 3000):
        few, alone = _electrons(api, n, 64.0, seed=n, capacity=cap), _electrons(api, n, 64.0, seed=n)
        a, la = _deposit(api, ctx, few, shape)
        b, lb = _deposit(api, ctx, alone, shape)
        assert (la, lb) == (4, 1)
        torch.testing.assert_close(a, b, rtol=0, atol=1e-6 * float(b.abs().max()))
        # the same through the count, of a species that is full
        few.n.fill_(cap)
        c, lc = _deposit(api, ctx, few, shape, torch.tensor([n], dtype=torch.int64, device="cuda"))
        assert lc == 4
        torch.testing.assert_close(c, b, rtol=0, atol=1e-6 * float(b.abs().max()))
        f, lf = _deposit(api, ctx, full, shape)
        assert lf == 4
        ref_full = f if ref_full is None else ref_full
        torch.testing.assert_close(f, ref_full, rtol=0, atol=1e-5 * float(f.abs().max()))


# ragged tiles, one cell along an axis, 50 particles a cell, more particles than
# records (65536 max_particles: 131072 records), and an infinite weight
@pytest.mark.parametrize("shape,max_particles", [
    ((257, 3, 41), 1 << 19), ((1, 140, 128), 1 << 19), ((131, 65, 5), 1 << 19), ((67, 65, 5), 1 << 19),
    ((96, 81, 17), 1 << 19), ((16, 16, 132), 1 << 16)])
def test_tiled_deposit_matches_oracle(api, shape, max_particles):
    """Tolerance as in tests/test_gpu_pic_tiled.py: 3e-5 of the largest J."""
    from oracle import pic as P
    n, d, o = 400_003, (0.5, 0.3, 0.45), (0.2, -0.4, 1.0)
    rng = np.random.default_rng(n)
    st = {k: rng.uniform(-0.3 * s * c, 1.3 * s * c, n) for k, s, c in zip("xyz", shape, d)}
    st.update({k: rng.normal(scale=2.0, size=n) for k in ("px", "py", "pz")})
    st = to32(dict(st, w=rng.uniform(0.5, 2.0, n), id=np.arange(n, dtype=np.uint64)))
    st["px"][5] = np.nan  # reported and left out
    ctx = api.qed_init_tables(api.config(dt=0.1, max_particles=max_particles))
    y, g = api.Yee(*shape, *d, *o), P.Grid(*shape, *d, *o)
    before = ctx.launches
    api.qed_pic_deposit(ctx, api.Species.empty(n, -1).load(**st), y, 1.7)
    assert ctx.launches - before == 4
    keep = np.arange(n) != 5
    P.deposit(g, *(st[k][keep] for k in ("x", "y", "z", "px", "py", "pz", "w")), -1.0, 0.1, 1.7)
    torch.cuda.synchronize()
    for nm in ("jx", "jy", "jz"):
        ref = getattr(g, nm)
        np.testing.assert_allclose(getattr(y, nm).cpu().numpy(), ref, rtol=0, atol=3e-5 * np.abs(ref).max(), err_msg=nm)
    assert api.qed_read_counters(ctx)["status"] & 4


def test_infinite_weight_reaches_the_same_nodes(api):
    ctx = api.qed_init_tables(api.config(dt=0.1, max_particles=1 << 19))
    bad = []
    for n in (1, 1 << 19):
        e = _electrons(api, n, 10.0)
        for k in ("x", "y", "z", "px", "py", "pz"):
            getattr(e, k)[0] = 1.3
        e.w[0] = float("inf")
        J, launches = _deposit(api, ctx, e, (48, 36, 20))
        assert launches == (1 if n == 1 else 4)
        bad.append(~torch.isfinite(J))
    assert int(bad[0].sum()) == 24 and bool((bad[0] == bad[1]).all())


@pytest.mark.parametrize("per_cell", [0.6, 1.3])
def test_order_does_not_change_the_current(api, per_cell):
    """A J beyond L2 (190^3 cells), fewer than two particles a cell: stored by
    cell they are deposited directly, shuffled by tiles -- the same J within the
    rounding of a coordinate (3e-5 of the largest J, as above)."""
    nx = 190
    n = int(per_cell * nx ** 3)
    ctx = api.qed_init_tables(api.config(dt=0.1, max_particles=n))
    e = _electrons(api, n, float(nx))
    cell = (e.z.floor().long() * nx + e.y.floor().long()) * nx + e.x.floor().long()
    J = []
    for order in (torch.argsort(cell), torch.randperm(n, device="cuda", generator=torch.Generator("cuda").manual_seed(1))):
        for k in ("x", "y", "z", "px", "py", "pz", "w"):
            getattr(e, k).copy_(getattr(e, k)[order])
        j, launches = _deposit(api, ctx, e, (nx, nx, nx))
        assert launches == 4
        J.append(j)
    assert float((J[0] - J[1]).abs().max()) <= 3e-5 * float(J[0].abs().max())
