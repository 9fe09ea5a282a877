"""GPU: the 1d kernels that split an instance over the CTAs of a cluster (n = 256 .. 16384).

The number of CTAs per instance follows from the layout's other instances, so the same
instance is computed alone, among a few and in a crowd; every split has to give bitwise the
same numbers, and they have to be the oracle's."""
import numpy as np
import pytest
import torch

from oracle import sgn_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2506_16045_gb300 import sgn
    ctx = sgn.Context(0)
    yield sgn, ctx
    ctx.close()


def fields(n, L):
    x = np.arange(n) * (L / n)
    h = 1.0 - 0.2 * np.exp(-((x - 0.5 * L) / (0.08 * L)) ** 2)
    eta = h + 0.2 * np.exp(-((x - 0.4 * L) / (0.06 * L)) ** 2)
    u = 0.3 * np.sin(2 * np.pi * x / L) + 0.1 * np.cos(4 * np.pi * x / L)
    return h, eta, u


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("log2n", range(8, 15))
def test_every_split_gives_the_same_bits_and_the_oracle(S, log2n, prec):
    """Solve, right-hand side, and two steps of RK4 and of SBDF2 of one instance alone, with
    40 others and with 199 others.  rtol 1e-11 bounds the solution's error by
    sqrt(kappa_ub) 1e-11 < 1e-9 here; two steps carry a few solves."""
    sgn, ctx = S
    n, L, g = 1 << log2n, 50.0, 9.81
    p = sgn.PREC_FP64 if prec == "fp64" else sgn.PREC_MIXED
    h, eta, u = fields(n, L)
    grid = O.make_grid(1, n, L, g)
    ref = O.init_state(eta, u, h, grid)
    b, hx = ref.U.copy(), ref.gradh
    dt = 0.1 * (L / n) / np.sqrt(g * 1.2)
    out = []
    for count in (1, 41, 200):
        lay = sgn.Layout(ctx, [sgn.Grid(1, n, L, g=g)] * count)
        dev = lambda a: torch.as_tensor(np.tile(a, count), dtype=torch.float64, device="cuda")
        zero = lambda: torch.zeros(lay.points, dtype=torch.float64, device="cuda")
        x, fe, fU = zero(), zero(), zero()
        info = sgn.pcg(lay, dev(eta), dev(hx), dev(b), x, rtol=1e-11, prec=p)
        assert all(i["status"] == 0 for i in info)
        sgn.rhs(lay, dev(eta), dev(u), dev(h), dev(hx), fe, fU)
        got = [x, fe, fU]
        for scheme in ("rk4", "linimp"):
            e, v, U, gh = dev(eta), dev(u), zero(), zero()
            st = sgn.State(lay, e, U, v, dev(h), gh)
            st.init()
            getattr(st, scheme)(dt, 2, rtol=1e-11, maxit=4000, prec=p)
            got += [e, U, v]
            torch.cuda.synchronize()
            st.close()
        got = [t.cpu().numpy().reshape(count, n) for t in got]
        assert all(np.array_equal(a[i], a[0]) for a in got for i in range(count))
        out.append([a[0] for a in got])
        lay.close()
    for other in out[1:]:
        assert all(np.array_equal(a, c) for a, c in zip(out[0], other))
    x, fe, fU, e1, U1, u1, e2, U2, u2 = out[0]
    assert rel(x, u) < 1e-9
    re, rU = O.rhs_1d(eta, u, h, hx, L, g)
    # rounding of the fields times the largest wavenumber: (n/2) eps of a first derivative of the
    # lowest modes, k^3 eps eta^3 of the third derivatives against f_U = O(1)
    k = np.pi * n / L
    assert rel(fe, re) < 1e-12 + 1e-15 * n and rel(fU, rU) < 1e-12 + 1e-15 * k ** 3
    a = O.init_state(eta, u, h, grid)
    O.run_rk4(a, dt, 2, 1e-13)
    assert rel(e1, a.eta) < 1e-9 and rel(u1, a.u) < 1e-9
    a = O.init_state(eta, u, h, grid)
    O.run_sbdf2(a, dt, 2, 1e-13)
    assert rel(e2, a.eta) < 1e-9 and rel(u2, a.u) < 1e-9


def test_non_finite_and_huge_inputs_end_with_a_status(S):
    """Inputs that overflow the float32 range, and NaN, in a split instance: the solve ends with
    a breakdown, and another instance of the batch is not touched."""
    sgn, ctx = S
    n, L = 4096, 50.0
    h, eta, u = fields(n, L)
    hx = O.deriv(h, L)
    b = O.apply_G_1d(eta, hx, u, L)
    lay = sgn.Layout(ctx, [sgn.Grid(1, n, L)] * 2)
    dev = lambda *a: torch.as_tensor(np.concatenate(a), dtype=torch.float64, device="cuda")
    for bad in (np.nan, np.inf, 1e30):
        x = torch.zeros(2 * n, dtype=torch.float64, device="cuda")
        info = sgn.pcg(lay, dev(eta, eta), dev(hx, hx), dev(b * bad, b), x, rtol=1e-11,
                       prec=sgn.PREC_MIXED, check=False)
        assert info[0]["status"] == 6 and info[1]["status"] == 0
        assert rel(x[n:].cpu().numpy(), u) < 1e-9
