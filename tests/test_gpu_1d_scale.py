"""GPU: mixed 1d solves whose b.A^{-1}b lies at the ends of the float32 range.

The sums of the mixed solve are float32 products in double-float; what is decided from them
(converged, the scale of the inner solve, the reported ratio) must hold over the whole range."""
import numpy as np
import pytest

from oracle import sgn_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def S():
    from paper_2506_16045_gb300 import sgn
    ctx = sgn.Context(0)
    yield sgn, ctx
    ctx.close()


def problem(n, L):
    x = np.arange(n) * (L / n)
    h = 1.0 - 0.2 * np.exp(-((x - 0.5 * L) / (0.08 * L)) ** 2)
    eta = h + 0.2 * np.exp(-((x - 0.4 * L) / (0.06 * L)) ** 2)
    u = 0.3 * np.sin(2 * np.pi * x / L) + 0.1 * np.cos(4 * np.pi * x / L)
    hx = O.deriv(h, L)
    b = O.apply_G_1d(eta, hx, u, L)
    P = O.precond_coeffs(eta, hx)
    k = 2 * np.pi * np.fft.rfftfreq(n, L / n)
    k[-1] = 0.0
    w = np.full(k.size, 2.0)
    w[0] = w[-1] = 1.0
    bb = float(np.sum(w * abs(np.fft.rfft(b)) ** 2 / (P["sigma"] + P["alpha"] * k * k)))
    return eta, hx, b, u, bb, P["kappa_ub"]


def solve(S, n, L, eta, hx, b, rtol):
    sgn, ctx = S
    lay = sgn.Layout(ctx, [sgn.Grid(1, n, L)])
    dev = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    info = sgn.pcg(lay, dev(eta), dev(hx), dev(b), x, rtol=rtol, prec=sgn.PREC_MIXED,
                   check=False)[0]
    lay.close()
    return x.cpu().numpy(), info


@pytest.mark.parametrize("n", [256, 1024, 4096])
@pytest.mark.parametrize("target", [1e-40, 1e-30, 1e37])
def test_small_and_large_right_hand_sides(S, n, target):
    """rtol 1e-5: the squared residuals at 1e-30 are 1e-40, still float32 numbers; at 1e-40 they
    are zero and the solve ends with its first correction, solved to 1e-6 (the tightest inner
    tolerance).  Either way the error is below sqrt(kappa_ub) 1e-5 and the subnormals' rounding
    (2^-16 at 1e-40) of the norms."""
    L = 50.0
    eta, hx, b, u, bb, kappa = problem(n, L)
    c = np.sqrt(target / bb)
    x, info = solve(S, n, L, eta, hx, c * b, 1e-5)
    assert info["status"] == 0 and info["ratio"] <= 1e-5, info
    assert np.linalg.norm(x / c - u) <= np.sqrt(kappa) * (1e-5 + 2.0 ** -16) * np.linalg.norm(u)


@pytest.mark.parametrize("n", [256, 4096])
def test_a_tolerance_that_everything_meets(S, n):
    """x0 = 0 has the ratio 1: no inner solve is due, and the ratio is reported.  x holds the
    rounding (2^-47) of the transform that it shares with b."""
    eta, hx, b, u, bb, kappa = problem(n, 50.0)
    for rtol in (2.0, 1e30, np.inf):
        x, info = solve(S, n, 50.0, eta, hx, b, rtol)
        assert info["status"] == 0 and info["iters"] == 0, (rtol, info)
        assert np.abs(x).max() <= 1e-12 * np.abs(b).max()
        assert abs(info["ratio"] - 1.0) < 1e-6
