"""GPU: NaN, infinities, non-positive depths and fields beyond the float32 range, 1d and 2d, both
precisions: a status, never a wrong answer, and the coefficients' extrema over the whole range."""
import numpy as np
import pytest

from oracle import sgn_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GRIDS = [(4096, 1), (256, 1), (96, 1), (64, 64), (48, 20)]
BREAKDOWN, NONPOSITIVE = 6, 7


@pytest.fixture(scope="module")
def S():
    from paper_2506_16045_gb300 import sgn
    ctx = sgn.Context(0)
    yield sgn, ctx
    ctx.close()


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64).ravel(), device="cuda")


def problem(nx, ny, L=20.0):
    x, y = np.arange(nx) / nx, np.arange(ny)[:, None] / ny
    if ny == 1:
        h = 1.0 + 0.2 * np.cos(2 * np.pi * x)
        eta, u = h + 0.05 * np.sin(4 * np.pi * x), np.sin(2 * np.pi * x)
        return eta, O.grad(h, L), u, O.make_grid(1, nx, L, 9.81)
    h = 1.0 + 0.2 * np.cos(2 * np.pi * x) * np.cos(2 * np.pi * y)
    eta = h + 0.05 * np.cos(2 * np.pi * (x - y))
    u = np.stack([np.sin(2 * np.pi * (x + y)), np.cos(2 * np.pi * y) + 0 * x])
    return eta, O.grad(h, (L, L)), u, O.make_grid(2, nx, L, 9.81, ny=ny, Ly=L)


def layout(sgn, ctx, nx, ny, L=20.0):
    return sgn.Layout(ctx, [sgn.Grid(1, nx, L, g=9.81) if ny == 1
                            else sgn.Grid(2, nx, L, ny=ny, Ly=L, g=9.81)])


def solve(sgn, lay, eta, gh, b, prec):
    x = torch.zeros(b.size, dtype=torch.float64, device="cuda")
    info = sgn.pcg(lay, dev(eta), dev(gh), dev(b), x, rtol=1e-10, prec=prec, check=False)[0]
    return x.cpu().numpy(), info


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("nx,ny", GRIDS)
def test_bad_points_end_with_a_status(S, nx, ny, mixed):
    sgn, ctx = S
    prec = sgn.PREC_MIXED if mixed else sgn.PREC_FP64
    eta, gh, u, _ = problem(nx, ny)
    lay = layout(sgn, ctx, nx, ny)
    at = lambda a, v: np.where(np.arange(a.size).reshape(a.shape) == a.size // 3, v, a)
    for v in (np.nan, 0.0, -1.0, -np.inf):
        assert solve(sgn, lay, at(eta, v), gh, u, prec)[1]["status"] == NONPOSITIVE, v
    assert solve(sgn, lay, eta, at(gh, np.nan), u, prec)[1]["status"] == NONPOSITIVE
    for v in (np.nan, np.inf):
        assert solve(sgn, lay, eta, gh, at(u, v), prec)[1]["status"] == BREAKDOWN, v
    x, info = solve(sgn, lay, eta, gh, u, prec)              # and the layout is as before
    assert info["status"] == 0 and np.isfinite(x).all()
    lay.close()


@pytest.mark.parametrize("host_driven", [0, 1])
def test_one_bad_instance_of_a_2d_batch(S, host_driven):
    """The instance with NaN ends with a breakdown and x = 0; the others are solved as alone."""
    sgn, ctx = S
    eta, gh, u, _ = problem(64, 64)
    ref = solve(sgn, layout(sgn, ctx, 64, 64), eta, gh, u, sgn.PREC_MIXED)[0].reshape(2, -1)
    count = 1 if host_driven else 3
    lay = sgn.Layout(ctx, [sgn.Grid(2, 64, 20.0, ny=64, Ly=20.0, g=9.81)] * count)
    if host_driven:
        lay.profile_inner2d(True)
    b = np.repeat(u.reshape(2, 1, -1), count, axis=1)
    b[0, count // 2, 5] = np.nan
    x = torch.zeros(b.size, dtype=torch.float64, device="cuda")
    info = sgn.pcg(lay, dev(np.tile(eta.ravel(), count)),
                   dev(np.repeat(gh.reshape(2, 1, -1), count, axis=1)), dev(b), x, rtol=1e-10,
                   prec=sgn.PREC_MIXED, check=False)
    x = x.cpu().numpy().reshape(2, count, -1)
    for i in range(count):
        if i == count // 2:
            assert info[i]["status"] == BREAKDOWN and not x[:, i].any()
        else:
            assert info[i]["status"] == 0
            assert np.linalg.norm(x[:, i] - ref) <= 1e-9 * np.linalg.norm(ref)
    lay.close()


@pytest.mark.parametrize("nx,ny", GRIDS)
def test_beyond_the_float32_range(S, nx, ny):
    """eta^3 above 2^128: the mixed form says that it cannot."""
    sgn, ctx = S
    eta, gh, u, _ = problem(nx, ny)
    lay = layout(sgn, ctx, nx, ny)
    assert solve(sgn, lay, 1e14 * eta, gh, 1e14 * u, sgn.PREC_MIXED)[1]["status"] != 0
    lay.close()


@pytest.mark.parametrize("nx,ny", GRIDS)
def test_extrema_over_the_range(S, nx, ny):
    """sigma, alpha and kappa_ub follow from extrema of eta, |grad h| and eta (1 + l |grad h|^2):
    fields over sixty decades, signs of grad h included, against the oracle's."""
    sgn, ctx = S
    lay = layout(sgn, ctx, nx, ny)
    rng = np.random.default_rng(5)
    shape = (nx,) if ny == 1 else (ny, nx)
    gshape = shape if ny == 1 else (2,) + shape
    for _ in range(4):
        eta = 10.0 ** rng.uniform(-30, 30, shape)
        gh = rng.choice([-1.0, 1.0], gshape) * 10.0 ** rng.uniform(-30, 30, gshape)
        p, w = sgn.precond_coeffs(lay, dev(eta), dev(gh))[0], O.precond_coeffs(eta, gh)
        for k in ("sigma", "alpha"):
            assert abs(p[k] - w[k]) <= 1e-14 * abs(w[k]), k
    lay.close()
