"""Which current deposit a call takes.  FP64 contexts deposit directly, by one
launch, at every size: the tiled sums took twice the time there (2369 us
against 1093 at 128^3 cells and 2^22 electrons)."""
import pytest
import torch

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
