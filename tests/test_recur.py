"""Sums over tiles and scalars of the BiCGStab recurrence (csrc/recur.cuh), compiled for the host:
never less accurate than the FP64 sums and divisions they stand for."""
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1601_04587_gb300 import build

SRC = r"""
#include <cstdio>
#include <vector>
#include "recur.cuh"
using namespace ddp;
int main(int, char **v) {
    FILE *f = fopen(v[1], "rb");
    int n;
    fread(&n, 4, 1, f);
    std::vector<float> x(n);
    fread(x.data(), 4, n, f);
    // 256 running sums, joined pairwise: the shape of the kernels' sums
    std::vector<Sum3> s(256);
    for (auto &q : s) sum_zero(q);
    for (int i = 0; i < n; i++) sum_add(s[i % 256], x[i]);
    for (int h = 128; h > 0; h /= 2)
        for (int i = 0; i < h; i++) s[i] = sum_join(s[i], s[i + h]);
    printf("%a\n", sum_value(s[0]));
    double w[8], t;
    Cnum r, a, al, inv, om, rc, be;
    fread(w, 8, 8, f);
    fread(&t, 8, 1, f);
    fread(&r, 16, 1, f);
    fread(&a, 16, 1, f);
    printf("%d\n", (int)bicg_alpha(r, a, al, inv));
    printf("%d\n", bicg_omega(w, t, inv, om, rc, be));
    printf("%a %a %a %a %a %a %a %a\n", al.x, al.y, om.x, om.y, rc.x, rc.y, be.x, be.y);
}
"""


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    d = tmp_path_factory.mktemp("recur")
    (d / "r.cu").write_text(SRC)
    exe = str(d / "r")
    subprocess.run([build._nvcc(), "-O2", "-std=c++17", *build.ARCH, "-I", build.CSRC, str(d / "r.cu"), "-o", exe], check=True,
                   capture_output=True)

    def run(x, w=np.ones(8), t=0.0, r=1.0, a=1.0):
        with open(d / "in", "wb") as f:
            f.write(np.int32(len(x)).tobytes() + np.asarray(x, np.float32).tobytes() + np.asarray(w, np.float64).tobytes())
            f.write(np.float64(t).tobytes() + np.complex128(r).tobytes() + np.complex128(a).tobytes())
        out = subprocess.run([exe, str(d / "in")], check=True, capture_output=True, text=True).stdout.split("\n")
        v = [float.fromhex(k) for k in out[3].split()]
        return float.fromhex(out[0]), int(out[1]), int(out[2]), [complex(*v[i:i + 2]) for i in (0, 2, 4, 6)]
    return run


def _cases():
    rng = np.random.default_rng(4)
    n = 30000
    x = (rng.standard_normal(n) * 2.0 ** rng.integers(-40, 20, n)).astype(np.float32)
    yield "mixed sizes", x
    yield "all positive", np.abs(rng.standard_normal(n)).astype(np.float32)
    y = np.concatenate([x, -x[::-1], [np.float32(1e-9)]])
    yield "cancelling", y.astype(np.float32)
    yield "one", np.array([np.float32(0.1)])
    yield "tiny", np.full(1000, 1e-44, np.float32)


@pytest.mark.parametrize("name,x", list(_cases()), ids=lambda v: v if isinstance(v, str) else "")
def test_sums_are_as_good_as_fp64(prog, name, x):
    exact = math.fsum(map(float, x))
    got = prog(x)[0]
    # third float rounded to 2^-24 of 2^-48 of the partial sums (below sum |x|), and the result to FP64
    bound = 2.0 ** -70 * float(np.abs(x.astype(np.float64)).sum()) + 2.0 ** -52 * abs(exact)
    assert abs(got - exact) <= bound


def test_sums_that_are_not_finite(prog):
    assert prog([1.0, math.inf, 2.0])[0] == math.inf
    assert math.isnan(prog([1.0, math.inf, -math.inf])[0])
    assert math.isnan(prog([math.nan] + [1.0] * 300)[0])


def test_recurrence_against_rationals(prog):
    rng = np.random.default_rng(8)

    def frac(z):
        return Fraction(z.real), Fraction(z.imag)

    def mul(a, b):
        return a[0] * b[0] - a[1] * b[1], a[0] * b[1] + a[1] * b[0]

    def div(a, b):
        n = b[0] * b[0] + b[1] * b[1]
        q = mul(a, (b[0], -b[1]))
        return q[0] / n, q[1] / n

    def close(z, want, tol):
        size = math.hypot(*map(float, want))
        assert math.hypot(float(Fraction(z.real) - want[0]), float(Fraction(z.imag) - want[1])) <= tol * size

    for scale in (1.0, 1e-30, 1e30):            # the last two are beyond FP32 in their products
        w = rng.standard_normal(8) * scale
        w[6:] = np.abs(w[6:]) + scale
        w[7] += 2 * (w[0] ** 2 + w[1] ** 2) / w[6]
        r, a = [complex(*rng.standard_normal(2)) * scale for _ in range(2)]
        _, ok, status, (al, om, rc, be) = prog([1.0], w, 0.0, r, a)
        assert ok == 1 and status == 0
        close(al, div(frac(r), frac(a)), 8 * 2.0 ** -53)
        omega = Fraction(w[0]) / Fraction(w[6]), Fraction(w[1]) / Fraction(w[6])
        close(om, omega, 4 * 2.0 ** -53)
        m = mul(omega, (Fraction(w[4]), Fraction(w[5])))
        want = Fraction(w[2]) - m[0], Fraction(w[3]) - m[1]
        assert abs(rc - complex(*map(float, want))) <= 16 * 2.0 ** -53 * (abs(complex(*w[2:4])) + math.hypot(*map(float, m)))
        close(be, div(mul(frac(rc), frac(al)), mul(frac(r), frac(om))), 24 * 2.0 ** -53)


def test_recurrence_breakdown_and_convergence(prog):
    ok = [1.0, 0.5, 0.3, 0.1, 0.2, 0.4, 2.0, 3.0]
    assert prog([1.0], ok, 1e-3)[2] == 0
    assert prog([1.0], ok, 10.0)[2] == 1                                  # (r, r) below the threshold
    assert prog([1.0], [0, 0] + ok[2:], 0.0)[2] == 2                      # omega = 0
    assert prog([1.0], [0, 0, 0, 0, 0, 0, 0, 0], 0.0)[2] == 1             # s = 0: solved
    assert prog([1.0], ok[:7] + [math.nan], 1.0)[2] == 2
    assert prog([1.0], ok, 0.0, 1.0, 0.0)[1] == 0                         # (rh, v) = 0
    assert prog([1.0], ok, 0.0, 1.0, complex(math.inf, 0))[1] == 0
