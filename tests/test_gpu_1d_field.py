"""Derivative and operator on 1d power-of-two grids at the edges of the split: the smallest and
largest sizes, one and several CTAs per instance, mixed batches."""
import numpy as np
import pytest

from oracle import sgn_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def dev(x):
    return torch.as_tensor(np.ascontiguousarray(x, dtype=np.float64).ravel(), device="cuda")


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.fixture(scope="module")
def S():
    from paper_2506_16045_gb300 import sgn
    ctx = sgn.Context(0)
    yield sgn, ctx
    ctx.close()


@pytest.mark.parametrize("sizes", [[8], [128], [256], [512], [1024], [2048], [4096], [8192],
                                   [16384], [16384] * 3 + [256] * 70 + [2048, 64, 8192, 4096],
                                   [1024] * 200])
def test_derivative_and_operator(S, sizes):
    sgn, ctx = S
    rng = np.random.default_rng(sum(sizes))
    grids = [sgn.Grid(1, n, 0.25 * n, g=9.81) for n in sizes]
    lay = sgn.Layout(ctx, grids)
    h = [rng.standard_normal(n) for n in sizes]               # every mode, n/2 too
    eta = [1.0 + 0.3 * rng.random(n) for n in sizes]
    u = [rng.standard_normal(n) for n in sizes]
    P = sum(sizes)
    off = np.concatenate([[0], np.cumsum(sizes)])
    hx = torch.zeros(P, dtype=torch.float64, device="cuda")
    sgn.spectral_grad(lay, dev(np.concatenate(h)), hx)
    alias = dev(np.concatenate(h))
    sgn.spectral_grad(lay, alias, alias)                      # in place
    assert torch.equal(alias, hx)
    Gu = torch.zeros_like(hx)
    ref_hx = [O.grad(f, 0.25 * n) for f, n in zip(h, sizes)]
    sgn.apply_operator(lay, dev(np.concatenate(eta)), dev(np.concatenate(ref_hx)),
                       dev(np.concatenate(u)), Gu)
    torch.cuda.synchronize()
    hx, Gu = hx.cpu().numpy(), Gu.cpu().numpy()
    for i, n in enumerate(sizes):
        s = slice(off[i], off[i + 1])
        grid = O.make_grid(1, n, 0.25 * n, 9.81)
        # a transform and back; two of them in turn
        assert rel(hx[s], ref_hx[i]) < 1e-13
        assert rel(Gu[s], O.apply_G(eta[i], ref_hx[i], u[i], grid)) < 1e-12
