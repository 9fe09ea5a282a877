"""Gradient and right-hand side on 2d power-of-two grids against the CPU oracle at the edges of
the derivative passes: the smallest and largest sides, even and odd powers of two (the radix-2
stage), one, two and four columns per CTA, few rows and few columns."""
import numpy as np
import pytest

from oracle import sgn_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(8, 8), (8, 1024), (1024, 8), (16, 32), (128, 16), (256, 64), (512, 16), (64, 512),
          (1024, 128)]


def dev(x):
    return torch.as_tensor(np.ascontiguousarray(x, dtype=np.float64).ravel(), device="cuda")


def host(t, shape):
    torch.cuda.synchronize()
    return t.cpu().numpy().reshape(shape)


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.fixture(scope="module")
def S():
    from paper_2506_16045_gb300 import sgn
    ctx = sgn.Context(0)
    yield sgn, ctx
    ctx.close()


def fields(nx, ny, Lx, Ly):
    """Random, with every mode present (the n/2 modes too)."""
    rng = np.random.default_rng(nx * 1024 + ny)
    h = 1.0 + 0.1 * rng.standard_normal((ny, nx))
    eta = 1.0 + 0.2 * rng.random((ny, nx))
    u = rng.standard_normal((2, ny, nx))
    return h, eta, u


@pytest.mark.parametrize("nx,ny", SHAPES)
def test_gradient_and_rhs(S, nx, ny):
    sgn, ctx = S
    Lx, Ly = 0.3 * nx, 0.5 * ny
    h, eta, u = fields(nx, ny, Lx, Ly)
    lay = sgn.Layout(ctx, [sgn.Grid(2, nx, Lx, ny=ny, Ly=Ly, g=9.81)])
    P = nx * ny
    gh = torch.zeros(2 * P, dtype=torch.float64, device="cuda")
    sgn.spectral_grad(lay, dev(h), gh)
    ref = O.grad(h, (Lx, Ly))
    # one transform of at most 2^10 points and back: a few ulp per stage
    assert rel(host(gh, (2, ny, nx)), ref) < 1e-13
    # the field may be either plane of the result
    for k in (0, 1):
        buf = torch.zeros(2 * P, dtype=torch.float64, device="cuda")
        buf[k * P:(k + 1) * P] = dev(h)
        sgn.spectral_grad(lay, buf[k * P:(k + 1) * P], buf)
        assert torch.equal(buf, gh)
    fe, fU = torch.zeros(P, dtype=torch.float64, device="cuda"), torch.zeros_like(gh)
    sgn.rhs(lay, dev(eta), dev(u), dev(h), dev(ref), fe, fU)
    re, rU = O.rhs_2d(eta, u, h, ref, Lx, Ly, 9.81)
    # three derivatives in turn of a field with energy up to the highest mode
    assert rel(host(fe, (ny, nx)), re) < 1e-13
    assert rel(host(fU, (2, ny, nx)), rU) < 1e-12


@pytest.mark.parametrize("nx,ny", [(8, 16), (128, 8), (256, 32), (512, 8)])
def test_mixed_step(S, nx, ny):
    """One RK4 step in mixed precision against float64: both solves stop at a residual of 1e-12,
    which the operator's condition (a few hundred here) turns into less than 1e-9 of u."""
    sgn, ctx = S
    Lx, Ly = 0.5 * nx, 0.5 * ny
    x, y = np.arange(nx) / nx, np.arange(ny)[:, None] / ny
    h = 1.0 + 0.2 * np.cos(2 * np.pi * x) * np.cos(2 * np.pi * y)
    eta = h + 0.05 * np.cos(2 * np.pi * (x - y))
    u = np.stack([0.1 * np.sin(2 * np.pi * (x + y)), 0.1 * np.cos(2 * np.pi * y) + 0 * x])
    out = []
    for prec in (sgn.PREC_FP64, sgn.PREC_MIXED):
        lay = sgn.Layout(ctx, [sgn.Grid(2, nx, Lx, ny=ny, Ly=Ly, g=9.81)])
        t = [dev(eta), dev(0 * u), dev(u), dev(h), dev(0 * u)]
        st = sgn.State(lay, *t)
        st.init()
        st.rk4(0.02, 1, prec=prec)
        assert st.stats()["status"] == 0
        out.append([host(v, -1) for v in t[:3]])
        st.close()
    for a, b in zip(out[1], out[0]):
        assert rel(a, b) < 1e-9
