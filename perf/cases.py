"""Performance cases of the SGN library: the work a user's program has it do, through the
public binding (paper_2506_16045_gb300.sgn).

A case is a dict of plain values with a "kind":

  solve1d  one constraint solve G x = b of one 1d instance (sgn.pcg), from a zero guess, on
           Eq:Testproblem of the paper (eta0 and h0 near 1);
  run1d    one 1d initial-value run: sgn.State.init and `steps` steps of RK4, AB4 or the
           linearly implicit SBDF2 on a solitary wave over a flat bottom or a shelf;
  ens1d    a run of a ragged batch of 1d shelf instances advanced together by RK4;
  solve2d  one call solving `count` 2d instances on one grid (b = G u for a smooth u);
  run2d    a 2d RK4 run of a plane solitary wave over a Gaussian bump;
  serve    a burst of requests (1d and 2d solves, 1d runs, host arrays) to the server.

Precisions and tolerances are the benchmark's: float64 with rtol 1e-12, mixed with 1e-10.
The sizes of a batch come from the case ("mix"); every value (amplitudes, positions, depths)
comes from the seed.
"""
import math
import random
import time

import numpy as np
import torch

from paper_2506_16045_gb300 import sgn

G0 = 9.81
PREC = {"fp64": sgn.PREC_FP64, "mixed": sgn.PREC_MIXED}
RTOL = {"fp64": 1e-12, "mixed": 1e-10}
POW2 = [512, 1024, 2048, 4096, 8192]
GENERIC = [768, 1536, 3072, 6144]


def listed():
    return [
        # the smallest call: one float64 solve at the paper's n = 256, latency only
        dict(name="solve1d-256-fp64", kind="solve1d", n=256, prec="fp64"),
        # the solitary-wave run of §6 (n = 256, L = 100, float64): one instance, many launches
        dict(name="run1d-256-rk4-fp64", kind="run1d", n=256, L=100.0, bed="flat", scheme="rk4",
             prec="fp64", steps=8),
        # the shelf run (n = 4096, L = 200) by the explicit multistep scheme, one instance
        dict(name="run1d-4096-ab4-mixed", kind="run1d", n=4096, L=200.0, bed="shelf",
             scheme="ab4", prec="mixed", steps=24),
        # the same by the linearly implicit scheme: no Krylov iteration, transforms only
        dict(name="run1d-4096-sbdf2-mixed", kind="run1d", n=4096, L=200.0, bed="shelf",
             scheme="sbdf2", prec="mixed", steps=32),
        # the headline: 256 uneven instances, n in {512 .. 8192}, advanced together
        dict(name="ens1d-256-mixed", kind="ens1d", count=256, sizes="pow2", mix=2506,
             prec="mixed", steps=4),
        # the batched float64 form the mixed form is compared with
        dict(name="ens1d-64-fp64", kind="ens1d", count=64, sizes="pow2", mix=2506, prec="fp64",
             steps=2),
        # a batch on grids that are not powers of two
        dict(name="ens1d-128-generic-mixed", kind="ens1d", count=128, sizes="generic", mix=2507,
             prec="mixed", steps=4),
        # the 2d bump run (80 x 80 at 512^2)
        dict(name="run2d-512-mixed", kind="run2d", nx=512, ny=512, prec="mixed", steps=4),
        # a 2d run in float64
        dict(name="run2d-256-fp64", kind="run2d", nx=256, ny=256, prec="fp64", steps=2),
        # a 2d run on a grid whose sides are not powers of two
        dict(name="run2d-384x240-mixed", kind="run2d", nx=384, ny=240, prec="mixed", steps=2),
        # a batch of 2d solves on one grid, past the L2 cache
        dict(name="solve2d-16x512-mixed", kind="solve2d", nx=512, ny=512, count=16,
             prec="mixed"),
        # a burst of uneven requests to the server, host arrays in
        dict(name="serve-24-mixed", kind="serve", requests=24, mix=16045, prec="mixed"),
    ]


def _smooth_sizes(lo, hi):
    """n = 2^a 3^b 5^c, a >= 1, not a power of two, in [lo, hi]."""
    out = []
    for n in range(lo + lo % 2, hi + 1, 2):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1 and n & (n - 1):
            out.append(n)
    return out


def _log_pick(rng, values):
    """One of the sorted values, spread over their logarithm."""
    x = math.exp(rng.uniform(math.log(values[0]), math.log(values[-1])))
    return min(values, key=lambda v: abs(math.log(v / x)))


def draw(rng):
    kind = rng.choice(["solve1d", "run1d", "ens1d", "solve2d", "run2d", "serve"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    odd = rng.random() < 0.4
    if kind == "solve1d":
        sizes = _smooth_sizes(30, 16384) if odd else [2 ** k for k in range(5, 15)]
        return dict(kind=kind, n=_log_pick(rng, sizes), prec=prec)
    if kind == "run1d":
        scheme = rng.choice(["rk4", "ab4"] if odd else ["rk4", "ab4", "sbdf2"])
        sizes = _smooth_sizes(240, 6144) if odd else [2 ** k for k in range(8, 15)]
        n = _log_pick(rng, sizes if prec == "mixed" else [s for s in sizes if s <= 4096])
        return dict(kind=kind, n=n, L=200.0 if n > 512 else 100.0,
                    bed="shelf" if n > 512 else "flat", scheme=scheme, prec=prec,
                    steps=rng.randint(4, 24 if prec == "mixed" else 8))
    if kind == "ens1d":
        fp = prec == "fp64"
        return dict(kind=kind, count=rng.randint(16, 48 if fp else 96 if odd else 256),
                    sizes="generic" if odd else "pow2", mix=rng.randint(1, 1 << 20), prec=prec,
                    steps=rng.randint(1, 2 if fp else 4))
    if kind == "solve2d":
        sides = [64, 128, 256, 512]
        nx, ny = rng.choice(sides), rng.choice(sides)
        most = 16 if prec == "mixed" else max(1, min(8, 131072 // (nx * ny)))
        return dict(kind=kind, nx=nx, ny=ny, count=rng.randint(1, most), prec=prec)
    if kind == "run2d":
        if odd:
            sides = _smooth_sizes(60, 384)
            nx = _log_pick(rng, sides)
            ny = _log_pick(rng, [s for s in sides if nx / 2 <= s <= 2 * nx])
        else:
            nx = 2 ** rng.randint(6, 9 if prec == "mixed" else 8)
            ny = nx * rng.choice([1, 1, 2]) if nx < 512 else nx // rng.choice([1, 2])
        return dict(kind=kind, nx=nx, ny=ny, prec=prec, steps=rng.randint(1, 2))
    return dict(kind="serve", requests=rng.randint(6, 24), mix=rng.randint(1, 1 << 20),
                prec="mixed")


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------

def _grid(n, L):
    return torch.arange(n, dtype=torch.float64, device="cuda") * (L / n)


def _sech2(z):
    return 1.0 / torch.cosh(z.clamp(-300.0, 300.0)) ** 2


def _wave(x, L, a, x0):
    """Surface elevation and velocity of the solitary wave of §6 (h0 = 1), periodic images."""
    gam = math.sqrt(3.0 * a) / (2.0 * math.sqrt(1.0 + a))
    s = sum(_sech2(gam * (x - x0 + m * L)) for m in (-1, 0, 1))
    return a * s, math.sqrt(G0 * (1.0 + a)) * a * s / (1.0 + a * s)


def _shelf(x, L, r, xs, w=5.0):
    W = 0.4 * L
    s = sum(torch.tanh((x - xs + m * L) / w) - torch.tanh((x - xs - W + m * L) / w)
            for m in (-1, 0, 1))
    return 1.0 - 0.5 * (1.0 - r) * s


def _inst1d(n, L, bed, rng, a=None):
    """(h, eta, u, a) of one 1d instance."""
    x = _grid(n, L)
    if bed == "flat":
        a = rng.uniform(0.1, 0.3) if a is None else a
        z, u = _wave(x, L, a, rng.uniform(0.2, 0.3) * L)
        h = torch.ones_like(x)
    else:
        a = rng.uniform(0.05, 0.4) if a is None else a
        xs = rng.uniform(0.3, 0.7) * L
        h = _shelf(x, L, rng.uniform(0.4, 0.8), xs)
        z, u = _wave(x, L, a, xs - 20.0)
    return h, h + z, u, a


def _bump1d(n, L, rng):
    x = _grid(n, L)
    h = 1.0 - rng.uniform(0.1, 0.6) * torch.exp(
        -((x - rng.uniform(0.3, 0.7) * L) / rng.uniform(1.0, 5.0)) ** 2)
    a = rng.uniform(0.05, 0.3)
    z, u = _wave(x, L, a, 0.2 * L)
    return h, h + z, u, a


def _inst2d(nx, ny, Lx, Ly, rng):
    """(h, eta, u, a): a plane wave over a Gaussian bump, fields [ny, nx]."""
    x, y = _grid(nx, Lx)[None, :], _grid(ny, Ly)[:, None]
    H, R = rng.uniform(0.1, 0.6), min(rng.uniform(2.0, 5.0), Ly / 10.0)
    xb, yb = rng.uniform(0.3, 0.7) * Lx, rng.uniform(0.3, 0.7) * Ly
    px = sum(torch.exp(-((x - xb + m * Lx) / R) ** 2) for m in (-1, 0, 1))
    py = sum(torch.exp(-((y - yb + m * Ly) / R) ** 2) for m in (-1, 0, 1))
    h = 1.0 - H * px * py
    a = rng.uniform(0.1, 0.3)
    z, u = _wave(x, Lx, a, 0.25 * Lx)
    u = u.expand(ny, nx)
    return h, h + z, torch.stack([u, torch.zeros_like(u)]), a


def _smooth_u2d(nx, ny, Lx, Ly, rng):
    """A smooth velocity with both components (the answer of a 2d solve)."""
    X = 2 * math.pi * _grid(nx, Lx)[None, :] / Lx
    Y = 2 * math.pi * _grid(ny, Ly)[:, None] / Ly
    k = rng.randint(1, 3)
    return torch.stack([rng.uniform(0.2, 0.4) * torch.sin(k * X) * torch.cos(2 * Y),
                        0.2 * torch.cos(X) + rng.uniform(0.05, 0.15) * torch.sin(k * Y)
                        + 0.0 * X])


def _lengths2d(case):
    return 80.0, 80.0 * case["ny"] / case["nx"]


def _sizes(case):
    rng = random.Random(case["mix"])
    return [rng.choice(POW2 if case["sizes"] == "pow2" else GENERIC) for _ in range(case["count"])]


def _dt(case, a):
    """The time step of one instance: the workloads' Courant numbers."""
    if case["kind"] == "run2d":
        return 0.25 * (80.0 / case["nx"]) / math.sqrt(G0 * (1.0 + a))
    c = {"rk4": 0.25, "ab4": 0.25, "sbdf2": 0.125}[case.get("scheme", "rk4")]
    return c * (case["L"] / case["n"]) / math.sqrt(G0 * (1.0 + a))


def _requests(case):
    """The burst's (kind, dim, side, steps): half 1d, half 2d; a third of the 1d ones runs."""
    rng = random.Random(case["mix"])
    out = []
    for i in range(case["requests"]):
        if i % 2:
            out.append(("solve", 2, 2 ** rng.randint(7, 9), 0))
        elif i % 6 == 4:
            out.append(("run", 1, 2 ** rng.randint(10, 14), rng.randint(4, 16)))
        else:
            out.append(("solve", 1, 2 ** rng.randint(10, 14), 0))
    if case["requests"] >= 20:
        out[1] = ("solve", 2, 1024, 0)
    return out


def _data(case, seed):
    """The inputs: a list of instances, each a dict of tensors and its grid."""
    rng = random.Random(seed * 7919 + 17)
    kind = case["kind"]
    if kind == "solve1d":
        n = case["n"]
        x = _grid(n, 1.0)
        h = 1.0 + rng.uniform(0.5, 1.5) * torch.exp(-((x - 0.5) / 0.05) ** 2)
        eta = 1.0 + rng.uniform(0.5, 1.5) * torch.cos(4 * math.pi * x) ** 2
        b = torch.cos(4 * math.pi * (x - rng.random()))
        return [dict(n=n, L=1.0, h=h, eta=eta, b=b)]
    if kind == "run1d":
        h, eta, u, a = _inst1d(case["n"], case["L"], case["bed"], rng)
        return [dict(n=case["n"], L=case["L"], h=h, eta=eta, u=u, dt=_dt(case, a))]
    if kind == "ens1d":
        out = []
        for n in _sizes(case):
            h, eta, u, a = _inst1d(n, 200.0, "shelf", rng)
            out.append(dict(n=n, L=200.0, h=h, eta=eta, u=u,
                            dt=_dt(dict(kind=kind, L=200.0, n=n), a)))
        return out
    if kind in ("solve2d", "run2d"):
        Lx, Ly = _lengths2d(case)
        out = []
        for _ in range(case.get("count", 1)):
            h, eta, u, a = _inst2d(case["nx"], case["ny"], Lx, Ly, rng)
            if kind == "solve2d":
                u = _smooth_u2d(case["nx"], case["ny"], Lx, Ly, rng)
            out.append(dict(nx=case["nx"], ny=case["ny"], Lx=Lx, Ly=Ly, h=h, eta=eta, u=u,
                            dt=_dt(case, a) if kind == "run2d" else 0.0))
        return out
    out = []
    for what, dim, n, steps in _requests(case):
        if dim == 1:
            h, eta, u, a = _bump1d(n, 200.0, rng)
            out.append(dict(what=what, n=n, L=200.0, h=h, eta=eta, u=u, steps=steps,
                            dt=0.25 * (200.0 / n) / math.sqrt(G0 * (1.0 + a))))
        else:
            h, eta, u, a = _inst2d(n, n, 80.0, 80.0, rng)
            out.append(dict(what=what, nx=n, ny=n, Lx=80.0, Ly=80.0, h=h, eta=eta, u=u))
    return out


# ------------------------------------------------------------------------------------------
# The calls
# ------------------------------------------------------------------------------------------

_CTX = []


def _ctx():
    """The library context a program keeps."""
    if not _CTX:
        _CTX.append(sgn.Context(torch.cuda.current_device()))
    return _CTX[0]


def _sgn_grid(d):
    if "nx" in d:
        return sgn.Grid(2, d["nx"], d["Lx"], g=G0, ny=d["ny"], Ly=d["Ly"])
    return sgn.Grid(1, d["n"], d["L"], g=G0)


def _pack(data, key):
    return torch.cat([d[key].reshape(-1) for d in data]).contiguous()


def _pack_vec(data, key):
    """2d vectors: the x components of every instance, then the y components."""
    if "nx" not in data[0]:
        return _pack(data, key)
    return torch.cat([d[key][c].reshape(-1) for c in (0, 1) for d in data]).contiguous()


def prepare(case, seed):
    data = _data(case, seed)
    s = dict(case=case, data=data)
    if case["kind"] == "serve":
        s["srv"] = sgn.Server(_ctx())
        s["reqs"] = []
        for d in data:
            v = d["u"]
            if d["what"] == "solve":
                lay = sgn.Layout(_ctx(), [_sgn_grid(d)])
                gh, b = (torch.zeros(v.numel(), dtype=torch.float64, device="cuda")
                         for _ in range(2))
                sgn.spectral_grad(lay, d["h"].reshape(-1).contiguous(), gh)
                sgn.apply_operator(lay, d["eta"].reshape(-1).contiguous(), gh,
                                   v.reshape(-1).contiguous(), b)
                v = b
                torch.cuda.synchronize()
                lay.close()
            host = [np.ascontiguousarray(t.reshape(-1).cpu().numpy())
                    for t in (d["eta"], v, d["h"])]
            s["reqs"].append((d, host))
        return s
    lay = s["lay"] = sgn.Layout(_ctx(), [_sgn_grid(d) for d in data])
    s["eta"], s["h"] = _pack(data, "eta"), _pack(data, "h")
    nv = (2 if "nx" in data[0] else 1) * s["eta"].numel()
    s["gh"] = torch.zeros(nv, dtype=torch.float64, device="cuda")
    if case["kind"] in ("solve1d", "solve2d"):
        sgn.spectral_grad(lay, s["h"], s["gh"])
        if case["kind"] == "solve1d":
            s["b"] = _pack(data, "b")
        else:
            s["b"] = torch.zeros(nv, dtype=torch.float64, device="cuda")
            sgn.apply_operator(lay, s["eta"], s["gh"], _pack_vec(data, "u"), s["b"])
        s["x"] = torch.zeros_like(s["b"])
    else:
        s["u"] = _pack_vec(data, "u")
        s["eta0"], s["u0"] = s["eta"].clone(), s["u"].clone()
        s["U"] = torch.zeros_like(s["u"])
        s["dt"] = [d["dt"] for d in data]
        s["st"] = sgn.State(lay, s["eta"], s["U"], s["u"], s["h"], s["gh"])
    del s["data"]
    return s


def run(s):
    case = s["case"]
    prec, rtol = PREC[case["prec"]], RTOL[case["prec"]]
    if case["kind"] in ("solve1d", "solve2d"):
        s["x"].zero_()
        sgn.pcg(s["lay"], s["eta"], s["gh"], s["b"], s["x"], rtol=rtol, maxit=4000, prec=prec,
                info=False)
        return s["x"]
    if case["kind"] == "serve":
        return _serve(s, prec, rtol)
    s["eta"].copy_(s["eta0"])
    s["u"].copy_(s["u0"])
    st = s["st"]
    st.init()
    scheme = case.get("scheme", "rk4")
    args = dict(rtol=rtol, maxit=4000, prec=prec)
    if scheme == "rk4":
        st.rk4(s["dt"], case["steps"], **args)
    elif scheme == "ab4":
        st.abk(4, s["dt"], case["steps"], **args)
    else:
        st.linimp(s["dt"], case["steps"], **args)
    return {"eta": s["eta"], "U": s["U"], "u": s["u"]}


def _serve(s, prec, rtol):
    srv, out, wait = s["srv"], {}, {}
    for i, (d, (eta, v, h)) in enumerate(s["reqs"]):
        solve = d["what"] == "solve"
        status, ticket = srv.submit(sgn.REQ_SOLVE if solve else sgn.REQ_RUN, _sgn_grid(d), eta,
                                    v, h, dt=0.0 if solve else d["dt"],
                                    nsteps=0 if solve else d["steps"], rtol=rtol, prec=prec,
                                    host=True)
        if status != sgn.SGN_OK:
            raise RuntimeError(f"request {i} refused: {status}")
        wait[i] = ticket
    while wait:
        for i in list(wait):
            r = srv.poll(wait[i])
            if r is None:
                continue
            if r["status"] != sgn.SGN_OK:
                raise RuntimeError(f"request {i} failed: {r['status']}")
            n = s["reqs"][i][1][1].size
            out["u%d" % i] = sgn.device_array(r["u"], n)
            if s["reqs"][i][0]["what"] == "run":
                out["eta%d" % i] = sgn.device_array(r["eta"], n)
            srv.release(wait.pop(i))
        if wait:
            time.sleep(0.0001)
    return out


# ------------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------------

#: Solves from a zero guess take about this many PCG iterations at these tolerances, solves
#: warm-started inside a step about half (float64 runs to two more digits).
COLD, WARM = {"fp64": 44, "mixed": 38}, {"fp64": 24, "mixed": 18}


def _iter_flops(n, dim):
    """One PCG iteration: two complex transforms of n points in 1d, three in 2d (six real
    fields), and the pointwise and vector work."""
    lg = math.log2(n)
    return (10.0 * lg + 26.0) * n if dim == 1 else (15.0 * lg + 70.0) * n


def _rhs_flops(n, dim):
    lg = math.log2(n)
    return (30.0 * lg + 40.0) * n if dim == 1 else (60.0 * lg + 120.0) * n


def _step_flops(n, dim, scheme, prec):
    it, rhs = _iter_flops(n, dim), _rhs_flops(n, dim)
    if scheme == "sbdf2":
        return 20.0 * n * math.log2(n) + rhs
    one = WARM[prec] * it + rhs
    return 4.0 * one if scheme == "rk4" else one


def work(case):
    kind, prec = case["kind"], case["prec"]
    if kind == "solve1d":
        n = case["n"]
        return {"bytes": 4 * 8 * n, "flops": COLD[prec] * _iter_flops(n, 1)}
    if kind == "solve2d":
        n = case["nx"] * case["ny"]
        return {"bytes": 7 * 8 * n * case["count"],
                "flops": case["count"] * COLD[prec] * _iter_flops(n, 2)}
    if kind == "serve":
        b = f = 0.0
        for what, dim, side, steps in _requests(case):
            n = side ** dim
            b += 8 * n * (3 if dim == 1 else 6) + (16 * n if what == "run" else 0)
            f += (steps * _step_flops(n, 1, "rk4", prec) if what == "run"
                  else COLD[prec] * _iter_flops(n, dim))
        return {"bytes": b, "flops": f}
    if kind == "run2d":
        n = case["nx"] * case["ny"]
        return {"bytes": 9 * 8 * n, "flops": case["steps"] * _step_flops(n, 2, "rk4", prec)}
    sizes = _sizes(case) if kind == "ens1d" else [case["n"]]
    scheme = case.get("scheme", "rk4")
    return {"bytes": 6 * 8 * sum(sizes),
            "flops": case["steps"] * sum(_step_flops(n, 1, scheme, prec) for n in sizes)}


# ------------------------------------------------------------------------------------------
# The same in 64 bits by torch: spectral derivatives, Def:G, a PCG run to round-off, and the
# time integrators of §5.  Fields are batched: [B, n] in 1d, [B, ny, nx] in 2d; vectors
# carry a component axis after the batch ([B, d, ...]).
# ------------------------------------------------------------------------------------------

class _Exact:
    def __init__(self, lengths, shape, h, eta):
        self.dim = len(shape)
        self.axes = [-1, -2][:self.dim]               # x, then y
        self.k = []
        for ax, L, n in zip(self.axes, lengths, reversed(shape)):
            k = 2 * math.pi / L * torch.fft.fftfreq(n, d=1.0 / n, dtype=torch.float64,
                                                    device="cuda")
            k[n // 2] = 0.0
            self.k.append(k if ax == -1 else k[:, None])
        self.h, self.gh = h, self.grad(h)
        self.set_A(eta)

    def d(self, f, c):
        ax = self.axes[c]
        return torch.fft.ifft(1j * self.k[c] * torch.fft.fft(f, dim=ax), dim=ax).real

    def grad(self, f):
        return torch.stack([self.d(f, c) for c in range(self.dim)], 1)

    def div(self, v):
        return sum(self.d(v[:, c], c) for c in range(self.dim))

    def sum(self, f):
        return f.flatten(1).sum(1).reshape(-1, *([1] * (self.dim + 1)))

    def set_A(self, eta):
        g2 = (self.gh ** 2).sum(1)
        lp, col = (4 + math.sqrt(13.0)) / 6, [-1] + [1] * (self.dim + 1)
        flat = (g2.flatten(1).amax(1) <= 1e-24)
        em = eta.flatten(1).amax(1)
        sig = torch.where(flat, em, (eta + lp * eta * g2).flatten(1).amax(1))
        alp = torch.where(flat, em ** 3 / 3, lp * em ** 3)
        self.sig, self.alp = sig.reshape(col), alp.reshape(col)

    def _spec(self, v, inverse):
        """A v, or A^{-1} v: per Fourier mode sigma I + alpha k k^T and its inverse."""
        dims = self.axes
        V = torch.fft.fftn(v, dim=dims)
        kv = sum(self.k[c] * V[:, c] for c in range(self.dim))
        kk = sum(k * k for k in self.k)
        a = self.alp[:, 0]
        f = -a / (self.sig[:, 0] + a * kk) if inverse else a
        W = V + torch.stack([f * k * kv for k in self.k], 1) if inverse else self.sig * V + \
            torch.stack([f * k * kv for k in self.k], 1)
        return torch.fft.ifftn(W / self.sig if inverse else W, dim=dims).real

    def G(self, eta, u):
        d, s = self.div(u), (self.gh * u).sum(1)
        t = eta ** 3 / 3 * d + eta ** 2 / 2 * s
        e = eta[:, None]
        return e * u - self.grad(t) + self.gh * (eta ** 2 / 2 * d + eta * s)[:, None]

    def solve(self, eta, b, x):
        """PCG twice: the second pass corrects the first with its true residual."""
        for rounds, tol in ((600, 1e-13), (600, 1e-4)):
            r = b - self.G(eta, x)
            ref = b if tol < 1e-8 else r
            stop = tol * tol * self.sum(ref * self._spec(ref, True))
            z = self._spec(r, True)
            rz, p = self.sum(r * z), z
            for _ in range(rounds):
                if bool((rz <= stop).all()):
                    break
                q = self.G(eta, p)
                pq = self.sum(p * q)
                a = torch.where(rz > stop, rz / pq, torch.zeros_like(rz))
                x = x + a * p
                r = r - a * q
                z = self._spec(r, True)
                new = self.sum(r * z)
                p = z + torch.where(rz > stop, new / rz, torch.zeros_like(rz)) * p
                rz = torch.where(rz > stop, new, rz)
        return x

    def rhs(self, eta, u):
        d, m, s = self.div(u), self.div(eta[:, None] * u), (self.gh * u).sum(1)
        S, Q = (u * self.grad(s)).sum(1), (u * self.grad(d)).sum(1) - d * d
        phi = eta ** 3 * Q / 3 + eta ** 2 * m * d + eta ** 2 * S / 2 + eta * m * s
        psi = eta ** 2 * Q / 2 + eta * m * d + eta * S + m * s
        flux = torch.stack([sum(self.d(eta * u[:, c] * u[:, e], e) for e in range(self.dim))
                            for c in range(self.dim)], 1)
        return -m, -G0 * eta[:, None] * self.grad(eta - self.h) - flux + self.grad(phi) \
            - self.gh * psi[:, None]

    def rk4(self, eta, U, u, dt, dv):
        fe, fU = self.rhs(eta, u)
        se, sU, v = fe / 6, fU / 6, u
        for c, w in ((0.5, 1 / 3), (0.5, 1 / 3), (1.0, 1 / 6)):
            ei = eta + c * dt * fe
            v = self.solve(ei, U + c * dv * fU, v)
            fe, fU = self.rhs(ei, v)
            se, sU = se + w * fe, sU + w * fU
        eta, U = eta + dt * se, U + dv * sU
        return eta, U, self.solve(eta, U, v)

    def advance(self, eta, u, dt, steps, scheme):
        """(eta, U, u) after `steps` steps; dt: one value per instance."""
        dt = torch.tensor(dt, dtype=torch.float64, device="cuda")
        dv = dt.reshape([-1] + [1] * (self.dim + 1))
        dt = dt.reshape([-1] + [1] * self.dim)
        U, f, old = self.G(eta, u), [], []
        if scheme == "sbdf2":
            self.set_A(eta)
            A0 = (self.sig, self.alp)
        for i in range(steps):
            if scheme != "rk4":
                f.append(self.rhs(eta, u))
            if scheme == "rk4" or i < (3 if scheme == "ab4" else 1):
                if scheme == "sbdf2":
                    old = [(eta, U, u)]
                eta, U, u = self.rk4(eta, U, u, dt, dv)
            elif scheme == "ab4":
                b = (-9 / 24, 37 / 24, -59 / 24, 55 / 24)
                eta = eta + dt * sum(c * q[0] for c, q in zip(b, f[-4:]))
                U = U + dv * sum(c * q[1] for c, q in zip(b, f[-4:]))
                u = self.solve(eta, U, u)
            else:
                self.sig, self.alp = A0
                e0, U0, u0 = old[-1]
                e2 = (4 * eta - e0 + 2 * dt * (2 * f[-1][0] - f[-2][0])) / 3
                U2 = (4 * U - U0 + 2 * dv * (2 * f[-1][1] - f[-2][1])) / 3
                r1 = self._spec(u, False) - self.G(eta, u) + U
                r0 = self._spec(u0, False) - self.G(e0, u0) + U0
                old = [(eta, U, u)]
                eta, U, u = e2, U2, self._spec(2 * r1 - r0, True)
        return eta, U, u


def _exact_of(group):
    """The _Exact of instances on one grid and their stacked eta and vector of `key`."""
    d0 = group[0]
    two = "nx" in d0
    eta = torch.stack([d["eta"] for d in group])
    E = _Exact((d0["Lx"], d0["Ly"]) if two else (d0["L"],),
               (d0["ny"], d0["nx"]) if two else (d0["n"],),
               torch.stack([d["h"] for d in group]), eta)
    vec = (lambda key: torch.stack([d[key] for d in group])) if two else \
        (lambda key: torch.stack([d[key] for d in group])[:, None])
    return E, eta, vec


def exact(case, seed):
    kind, data = case["kind"], _data(case, seed)
    if kind == "solve1d":
        E, eta, vec = _exact_of(data)
        b = vec("b")
        return E.solve(eta, b, torch.zeros_like(b)).reshape(-1)
    if kind == "solve2d":
        return _pack_vec(data, "u")                   # b = G u
    if kind == "serve":
        out = {}
        for i, d in enumerate(data):
            if d["what"] == "solve":
                out["u%d" % i] = d["u"].reshape(-1)   # b = G u
            else:
                E, eta, vec = _exact_of([d])
                eta, _, u = E.advance(eta, vec("u"), [d["dt"]], d["steps"], "rk4")
                out["u%d" % i], out["eta%d" % i] = u.reshape(-1), eta.reshape(-1)
        return out
    scheme, groups = case.get("scheme", "rk4"), {}
    for i, d in enumerate(data):
        groups.setdefault(d["n"] if "n" in d else 0, []).append(i)
    parts = [None] * len(data)
    for idx in groups.values():
        group = [data[i] for i in idx]
        E, eta, vec = _exact_of(group)
        eta, U, u = E.advance(eta, vec("u"), [d["dt"] for d in group], case["steps"], scheme)
        for j, i in enumerate(idx):
            parts[i] = (eta[j], U[j], u[j])
    cat = lambda c: torch.cat([p[c].reshape(-1) for p in parts])  # noqa: E731
    return {"eta": cat(0), "U": cat(1), "u": cat(2)}
