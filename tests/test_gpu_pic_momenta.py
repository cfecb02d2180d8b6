"""The deposit of momenta whose square overflows the working precision: 1 / gamma
is 0 there, so the particle stands still, adds nothing to J and is no error
(QED_STATUS_NONFINITE is for momenta that are not finite).  In both precisions,
alone (the direct deposit) and among as many others as the tiled one takes;
momenta just below keep |v| = 1."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_1608_06356_gb300 import api as A
    return A


@pytest.mark.parametrize("precision,big,ok", [(0, 1e25, 1e18), (1, 1e200, 1e150)])
@pytest.mark.parametrize("n", [4, 1 << 20])
def test_overflowing_momentum_stands_still(api, precision, big, ok, n):
    from paper_1608_06356_gb300 import _binding as B
    dt = torch.float64 if precision else torch.float32
    ctx = api.qed_init_tables(api.config(dt=0.1, precision=precision, max_particles=1 << 20))
    e = api.Species.empty(n, -1, dtype=dt)
    gen = torch.Generator("cuda").manual_seed(3)
    for k in "xyz":
        getattr(e, k).copy_(16.0 + 48.0 * torch.rand(n, generator=gen, device="cuda", dtype=dt))
    for k, v in (("x", 5.5), ("y", 5.5), ("z", 5.5)):
        getattr(e, k)[:4] = v
    e.w.fill_(1.0)
    e.n.fill_(n)
    J = {}
    for what, px in (("none", 0.0), ("big", big), ("ok", ok)):
        e.px[:4] = 0.0
        e.px[1] = px
        y = api.Yee(64, 64, 64, 1.0, 1.0, 1.0)
        api.qed_pic_deposit(ctx, e, y, 1.0)
        torch.cuda.synchronize()
        J[what] = y.jx.double()
        assert api.qed_read_counters(ctx)["status"] == 0, what
        assert not bool(y.jy.any()) and not bool(y.jz.any())
    assert float(J["none"].abs().max()) == 0.0 and float(J["big"].abs().max()) == 0.0
    np.testing.assert_allclose(float(J["ok"].sum()), -1.0, rtol=1e-6)
    e.px[1] = float("inf")
    api.qed_pic_deposit(ctx, e, api.Yee(64, 64, 64, 1.0, 1.0, 1.0), 1.0)
    assert api.qed_read_counters(ctx)["status"] == B.QED_STATUS_NONFINITE
