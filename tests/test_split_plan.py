"""The number of CTAs per 1d instance (sgn_split_plan.h), compiled with g++: the planned numbers are
ones that the kernels can run on, so what is counted is what is launched."""
import ctypes as C
import os
import random
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2506_16045_gb300", "csrc")
SMS = 152


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text(
        '#include "sgn_split_plan.h"\nusing namespace sgn;\nextern "C" {\n'
        "void plan(const int* n, const int* c, int m, int s, int* o) { split_plan(n, c, m, s, o); }\n"
        "int lo(int L, int m) { return split_min_lcl(L, split_log_e(L, m)); }\n"
        "int hi(int L, int m) { return split_max_lcl(L, split_log_e(L, m)); }\n}\n")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(d / "p.cpp"), "-o",
                    str(d / "p.so")], check=True)
    lib = C.CDLL(str(d / "p.so"))

    def run(num, mixed, two=()):
        A = C.c_int * 16
        n, t, o = A(), A(*[2 if c in two else 1 for c in range(16)]), A()
        for c, v in num.items():
            n[c] = v
        lib.plan(n, t, mixed, SMS, o)
        return list(o)
    return run, lib.lo, lib.hi


@pytest.mark.parametrize("mixed", [0, 1])
def test_kernel_ranges(plan, mixed):
    """256 threads a CTA at most (512 at n = 16384), 32 at least, 8 CTAs at most."""
    _, lo, hi = plan
    for L in range(8, 15):
        e = 4 if mixed or L > 10 else 2
        assert 0 <= lo(L, mixed) <= hi(L, mixed) <= 3
        assert (1 << L) // e >> lo(L, mixed) <= (512 if L == 14 else 256)
        assert (1 << L) // e >> hi(L, mixed) >= 32


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("num", [{8: 1}, {12: 1}, {13: 1, 10: 100}, {12: 60}, {12: 30, 9: 40},
                                 {11: 30, 10: 20, 9: 10}, {14: 3, 13: 4, 0: 5}, {13: 19}, {13: 20}])
def test_what_is_counted_is_launched(plan, num, mixed):
    check(plan, num, mixed)


def test_random_loads(plan):
    rng = random.Random(11)
    for _ in range(3000):
        num = {c: rng.choice([0, 1, 2, 5, 13, 40, 120]) for c in rng.sample(range(16), 5) if c < 15}
        check(plan, num, rng.randrange(2), rng.choice([(), (12,), (13,), (12, 13)]))


def check(plan, num, mixed, two=()):
    run, lo, hi = plan
    p = run(num, mixed, two)
    size = lambda q, c: num.get(c, 0) * (2 if c in two else 1 << q[c])
    split = [c for c in range(8, 15) if num.get(c) and c not in two]
    assert all(p[c] == 0 for c in range(16) if c < 8 or c > 14)
    assert all(lo(c, mixed) <= p[c] <= hi(c, mixed) for c in range(8, 15) if c not in two)
    total = sum(size(p, c) for c in range(16))
    least = [lo(c, mixed) if 8 <= c <= 14 else 0 for c in range(16)]
    # beyond the SMs only where the kernels' own minima are
    assert total <= SMS or all(p[c] == least[c] for c in split)
    # and the largest share that can still be halved does not fit
    left = [c for c in split if p[c] < hi(c, mixed)]
    if left:
        c = max(left, key=lambda c: (c - p[c], c))
        assert total + size(p, c) > SMS
