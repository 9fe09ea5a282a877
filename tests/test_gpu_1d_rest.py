"""GPU: an instance at rest beside a moving one.

A solve with b = 0 ends at once with u = 0.  The right-hand side that follows it in a time step
takes u_x from the solve, in the layout's scratch, which another state on the layout has used
in between."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def S():
    from paper_2506_16045_gb300 import sgn
    ctx = sgn.Context(0)
    yield sgn, ctx
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,ctas", [(64, 1), (96, 1), (256, 1), (1024, 1), (4096, 1), (4096, 2),
                                    (8192, 2)])
def test_still_water_stays_still(S, n, ctas, prec):
    """eta = h, u = 0: every term of the equations is exactly zero, so nothing may move."""
    sgn, ctx = S
    L, g = 50.0, 9.81
    p = sgn.PREC_FP64 if prec == "fp64" else sgn.PREC_MIXED
    x = np.arange(n) * (L / n)
    h = 1.0 - 0.2 * np.cos(2 * np.pi * x / L)
    lay = sgn.Layout(ctx, [sgn.Grid(1, n, L, g=g)])
    if ctas == 2:
        lay.set_form(n.bit_length() - 1, 2)
    dev = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")

    def state(eta, u):
        f = [dev(eta), dev(np.zeros(n)), dev(u), dev(h), dev(np.zeros(n))]
        st = sgn.State(lay, *f)
        st.init()
        return st, f

    moving, mf = state(h + 0.1 * np.sin(2 * np.pi * x / L), 0.3 * np.sin(2 * np.pi * x / L))
    still, sf = state(h, np.zeros(n))
    dt = 0.05 * (L / n) / np.sqrt(g * 1.2)
    for _ in range(7):                                   # RK4 starts the four-step scheme
        moving.abk(4, dt, 1, rtol=1e-11, prec=p)
        still.abk(4, dt, 1, rtol=1e-11, prec=p)
    torch.cuda.synchronize()
    assert np.array_equal(sf[0].cpu().numpy(), h)
    assert not sf[1].cpu().numpy().any() and not sf[2].cpu().numpy().any()
    assert mf[2].cpu().numpy().any()
    moving.close()
    still.close()
    lay.close()
