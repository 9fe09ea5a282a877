"""Float64 solves of 1d sizes that are not powers of two at the line between 256 and 512 threads:
against the oracle, and bitwise the same alone and beside larger instances."""
import numpy as np
import pytest

from oracle import sgn_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def dev(x):
    return torch.as_tensor(np.ascontiguousarray(x, dtype=np.float64).ravel(), device="cuda")


@pytest.fixture(scope="module")
def S():
    from paper_2506_16045_gb300 import sgn
    ctx = sgn.Context(0)
    yield sgn, ctx
    ctx.close()


def problem(n):
    x = 2 * np.pi * np.arange(n) / n
    h = 1.0 + 0.2 * np.cos(x)
    eta = h + 0.1 * np.sin(2 * x)
    return h, eta, np.sin(x) + 0.3 * np.cos(3 * x)


def solve(sgn, ctx, sizes):
    lay = sgn.Layout(ctx, [sgn.Grid(1, n, 0.25 * n, g=9.81) for n in sizes])
    p = [problem(n) for n in sizes]
    gh = [O.grad(q[0], 0.25 * n) for q, n in zip(p, sizes)]
    x = torch.zeros(sum(sizes), dtype=torch.float64, device="cuda")
    info = sgn.pcg(lay, dev(np.concatenate([q[1] for q in p])), dev(np.concatenate(gh)),
                   dev(np.concatenate([q[2] for q in p])), x, rtol=1e-12, prec=sgn.PREC_FP64)
    assert all(i["status"] == 0 for i in info)
    return np.split(x.cpu().numpy(), np.cumsum(sizes)[:-1])


@pytest.mark.parametrize("n", [6, 60, 486, 768, 800, 1500])
def test_solve_alone_and_beside_others(S, n):
    sgn, ctx = S
    alone = solve(sgn, ctx, [n])[0]
    h, eta, b = problem(n)
    gh, grid = O.grad(h, 0.25 * n), O.make_grid(1, n, 0.25 * n, 9.81)
    ref = O.solve_G(eta, gh, b, grid, rtol=1e-14, maxit=4000)[0]
    # a residual of 1e-12 times the operator's condition (below 100 here)
    assert np.linalg.norm(alone - ref) <= 1e-10 * np.linalg.norm(ref)
    assert np.array_equal(alone, solve(sgn, ctx, [3000, n, 60, 12288])[1])
