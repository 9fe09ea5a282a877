"""Serving: what the server keeps between requests (layouts of 2d grids, the arrays' pool) must
not show: the same request gives the same bits on a new and on a kept layout, between other
requests, after a failed one, and under a budget that keeps nothing."""
import time

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


def problem(nx, ny, seed):
    rng = np.random.default_rng(seed)
    x, y = np.arange(nx) / nx, np.arange(ny)[:, None] / ny
    h = 1.0 + 0.2 * np.cos(2 * np.pi * x) * np.cos(2 * np.pi * y)
    eta = h + 0.05 * np.cos(2 * np.pi * (x - y) + rng.random())
    b = np.stack([np.sin(2 * np.pi * (x + y)), np.cos(2 * np.pi * y) + 0 * x])
    return [np.ascontiguousarray(a).ravel() for a in (eta, b, h)]


def serve(sgn, srv, reqs):
    """[(kind, grid, arrays, options)] at once -> their u (None for a failed one)."""
    tickets = []
    for kind, g, arrays, kw in reqs:
        st, t = srv.submit(kind, g, *arrays, host=True, **kw)
        assert st == 0
        tickets.append(t)
    out, t0 = {}, time.time()
    while len(out) < len(tickets):
        assert time.time() - t0 < 120.0
        for i, t in enumerate(tickets):
            if i in out:
                continue
            r = srv.poll(t)
            if r is None:
                continue
            u = sgn.device_array(r["u"], reqs[i][2][1].size)      # read on the client's stream,
            srv.release(t)                                        # given up at once
            out[i] = u if r["status"] == 0 else None
        time.sleep(0.0005)
    # not the whole device: another server may be capturing its solve graph
    torch.cuda.current_stream().synchronize()
    return [None if out[i] is None else out[i].cpu().numpy() for i in range(len(reqs))]


@pytest.mark.parametrize("frac", [0.0, 3e-4])
def test_kept_layouts_and_pool(S, frac):
    sgn, ctx = S
    g = [sgn.Grid(2, 64, 40.0, ny=64, Ly=40.0, g=9.81),
         sgn.Grid(2, 64, 20.0, ny=64, Ly=40.0, g=9.81),       # same sizes, other lengths
         sgn.Grid(2, 48, 40.0, ny=20, Ly=40.0, g=9.81)]
    cases = [(sgn.REQ_SOLVE, g[0], problem(64, 64, 1), {}),
             (sgn.REQ_SOLVE, g[1], problem(64, 64, 2), {}),
             (sgn.REQ_SOLVE, g[2], problem(48, 20, 3), {}),
             (sgn.REQ_RUN, g[0], problem(64, 64, 4), dict(dt=0.01, nsteps=3))]
    # each alone on a server of its own
    ref = []
    for c in cases:
        srv = sgn.Server(ctx)
        ref.append(serve(sgn, srv, [c])[0])
        srv.close()
    srv = sgn.Server(ctx, budget_fraction=frac)
    order = np.random.default_rng(7)
    for rep in range(5):
        pick = [int(i) for i in order.permutation(len(cases))] + [0, 3]
        for i, u in zip(pick, serve(sgn, srv, [cases[i] for i in pick])):
            assert np.array_equal(u, ref[i])
        if rep == 2:                                          # one that cannot converge
            fail = (sgn.REQ_SOLVE, g[0], problem(64, 64, 1), dict(rtol=1e-14, maxit=1))
            assert serve(sgn, srv, [fail]) == [None]
    srv.close()


def test_servers_beside_each_other(S):
    """Three servers take turns, each on grids of its own, so that one builds layouts and solve
    graphs while another cleans up: no request of one may fail by what another does."""
    import threading
    sgn, ctx = S
    sizes = [16, 24, 32, 48, 64, 80, 96, 128]
    failed = []

    def client(k, srv):
        for rep in range(12):
            reqs = []
            for i in range(4):
                n = sizes[(k + 3 * rep + i) % len(sizes)]
                L = 10.0 + k + 0.5 * rep                      # a new grid each time
                reqs.append((sgn.REQ_SOLVE, sgn.Grid(2, n, L, ny=n, Ly=L, g=9.81),
                             problem(n, n, rep), {}))
            for i, u in enumerate(serve(sgn, srv, reqs)):
                if u is None or not np.isfinite(u).all():
                    failed.append((k, rep, i))

    servers = [sgn.Server(ctx) for _ in range(3)]
    threads = [threading.Thread(target=client, args=(k, s)) for k, s in enumerate(servers)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s in servers:
        s.close()
    assert not failed
