"""The float-pair arithmetic of the mixed-precision update (csrc/pair_f32.cuh), compiled as host
C++ and held to exact rational arithmetic: relative errors of sums, products, reciprocals within
2^-44 of their operands, and p - ab - cd rounded once."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1702_06359_gb300", "csrc")
EPS = Fraction(1, 2 ** 44)

PROGRAM = r"""
#include <cstdio>
#include "pair_f32.cuh"
using namespace tkf;
int main()
{
    float p;
    pair32 a, b, c, d;
    while (std::scanf("%a %a %a %a %a %a %a %a %a", &p, &a.h, &a.l, &b.h, &b.l, &c.h, &c.l, &d.h, &d.l) == 9) {
        const pair32 s = add(a, b), m = mul(a, b), r = recip(a), f = mul(a, b.h), t = two_prod(a.h, b.h);
        std::printf("%a %a %a %a %a %a %a %a %a %a %a %a\n", s.h, s.l, m.h, m.l, r.h, r.l, f.h, f.l, t.h, t.l,
                    minus_products(p, a, b, c, d), minus_products(p, a, b, c, d.h));
    }
}
"""


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("pair")
    (d / "pair.cpp").write_text(PROGRAM)
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.check_call([gxx, "-O1", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-I", inc, str(d / "pair.cpp"), "-o",
                           str(d / "pair")])
    return str(d / "pair")


@pytest.mark.parametrize("spread", [0, 3, 12])
def test_pairs_against_rational_arithmetic(prog, spread):
    """Operands within 2^+-spread of one another, either sign; p near ab + cd in half the rows, so
    that the difference cancels."""
    rng = np.random.default_rng(spread + 1)
    n = 2000
    h = (rng.uniform(1, 2, (n, 4)) * np.exp2(rng.integers(-spread, spread + 1, (n, 4))) * rng.choice([-1, 1], (n, 4))).astype(np.float32)
    lo = (h * rng.uniform(-1, 1, (n, 4)) * 2.0 ** -25).astype(np.float32)
    w = h.astype(np.float64) + lo
    p = rng.uniform(-4, 4, n).astype(np.float32)
    p[::2] = (w[::2, 0] * w[::2, 1] + w[::2, 2] * w[::2, 3]).astype(np.float32)
    rows = "\n".join(" ".join(float(x).hex() for x in [p[i], *np.stack([h[i], lo[i]], 1).ravel()]) for i in range(n))
    out = subprocess.run([prog], input=rows, capture_output=True, text=True, check=True).stdout.split()
    got = [[Fraction(float.fromhex(x)) for x in out[12 * i:12 * i + 12]] for i in range(n)]
    assert len(out) == 12 * n
    for i, g in enumerate(got):
        a, b, c, d = (Fraction(float(h[i, k])) + Fraction(float(lo[i, k])) for k in range(4))
        bh, dh, q = Fraction(float(h[i, 1])), Fraction(float(h[i, 3])), Fraction(float(p[i]))
        assert abs(g[0] + g[1] - (a + b)) <= EPS * (abs(a) + abs(b))
        assert abs(g[2] + g[3] - a * b) <= EPS * abs(a * b)
        assert abs((g[4] + g[5]) * a - 1) <= EPS
        assert abs(g[6] + g[7] - a * bh) <= EPS * abs(a * bh)
        assert g[8] + g[9] == Fraction(float(h[i, 0])) * bh
        for k, last in ((10, d), (11, dh)):
            exact = q - a * b - c * last
            assert abs(g[k] - exact) <= Fraction(1, 2 ** 24) * abs(exact) + EPS * (abs(q) + abs(a * b) + abs(c * last))
