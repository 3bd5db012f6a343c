"""Host evaluation of the rules that send FP64 interactions to tables and expansions
(the same functions the kernels call, compiled for the CPU): no argument leaves the
table, and every argument that the table serves is within its range."""
import math
import os
import subprocess

import pytest

from paper_1505_07851_gb300 import build

PRELUDE = """
#include <stdio.h>
#include <math.h>
#include "f64.cuh"
using namespace pcm;
"""


def run_host(tmp_path, body, include="f64.cuh"):
    src = tmp_path / "host.cu"
    src.write_text(PRELUDE.replace("f64.cuh", include) + body)
    exe = tmp_path / "host"
    cmd = [build.nvcc(), "-std=c++17", "--expt-relaxed-constexpr", *build.ARCH, "-I", build.CSRC, str(src), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.split()


def test_table_rows(tmp_path):
    """Squared distances and exponents over the whole range of doubles: T < f64_far_T is
    decided as in 64 bits (within 2^-18), so that a row that is read holds T; and the row of
    any double, NaN and infinity among them, is a row of the table."""
    out = run_host(tmp_path, """
int main()
{
    long bad = 0, near = 0;
    for (int L = 0; L <= 5; ++L)
        for (double r = 1e-30; r < 1e307; r *= 1.17)
            for (double rho = 1e-20; rho < 1e30; rho *= 1.31) {
                const double R2 = r, T = rho * R2, top = f64_far_T(L);
                const bool n = f64_below(R2, rho, (float)top);
                near += n;
                if (n && !(T < top * (1 + 0x1p-18))) ++bad;
                if (!n && !(T >= top * (1 - 0x1p-18))) ++bad;
                if (n && abs(f64_row(T + F64_MAGIC) - (int)rint(T * F64_INV_DT)) > 1) ++bad;
            }
    const double odd[] = {0.0, 54.0, 55.0, 1e9, 1e16, 1e30, 1e300, INFINITY, -INFINITY, NAN, -NAN, -1.0, -1e30};
    for (double t : odd)
        for (double u : {t, t + F64_MAGIC}) {
            const int i = f64_row(u);
            if (i < 0 || i >= F64_NROW) ++bad;
        }
    printf("%ld %ld\\n", bad, near);
    return 0;
}
""")
    assert int(out[0]) == 0 and int(out[1]) > 100000


def test_fp32_distance_tests_are_safe(tmp_path):
    """The FP32 tests never miss an interaction whose T, in 64 bits, is below the
    threshold: cavities of 10 to 1e24 bohr, exponents from 1e-3 to 1e36, pairs and points
    close together and far apart, at the same FP32 coordinates as the kernels'."""
    out = run_host(tmp_path, """
static double u() { static unsigned long long s = 42; s = s * 6364136223846793005ull + 1442695040888963407ull;
                    return (double)(s >> 11) * 0x1p-53; }
int main()
{
    long bad = 0, hit = 0;
    for (double ext = 10.0; ext < 1e24; ext *= 7.0) {
        const float slack = ext < 2e18 ? (float)(ext * 0x1p-21) : INFINITY, pad = 2001.f * slack * slack;
        for (int i = 0; i < 20000; ++i) {
            const double p = pow(10.0, u() * (i % 10 ? 6.0 : 39.0) - 3.0), z2 = 1.0 + 60.0 * u(), rho = p * z2 / (p + z2);
            double P[3], C[3], R2 = 0.0;
            const double far = sqrt(50.0 / rho) * 2.0 * u();
            for (int d = 0; d < 3; ++d) {
                P[d] = (u() - 0.5) * ext;
                C[d] = fmin(fmax(P[d] + far * (u() - 0.5) * 2.0, -0.5 * ext), 0.5 * ext);
                R2 += (P[d] - C[d]) * (P[d] - C[d]);
            }
            const float4 b = make_float4((float)P[0], (float)P[1], (float)P[2], (float)fmin(p, 1e30));
            const float4 c = make_float4((float)C[0], (float)C[1], (float)C[2], (float)(1.0 / z2));
            const float4 s = make_float4(c.x, c.y, c.z, slack);
            for (int L = 0; L <= 5; ++L) {
                const float top = (float)f64_far_T(L);
                if (!(rho * R2 < top)) continue;
                ++hit;
                if (!f64_reaches(b, s, (float)z2 * 0.99999f, top, slack)) ++bad;
                if (!f64_is_near(b.x - c.x, b.y - c.y, b.z - c.z, 1.f / b.w + c.w, top, pad)) ++bad;
            }
        }
    }
    printf("%ld %ld\\n", bad, hit);
    return 0;
}
""")
    assert int(out[0]) == 0 and int(out[1]) > 100000


def test_expansion_orders(tmp_path):
    """The order of a cell's expansion: what it leaves out of an n-th derivative of 1/R,
    summed in Python, is below 2n + 1 units of 2^-53 of the leading term, and one order
    less leaves more."""
    out = run_host(tmp_path, """
int main()
{
    for (int n = 0; n <= 5; ++n)
        for (int i = 1; i <= 120; ++i) printf("%d %d %d\\n", n, i, mp_order_for((float)i / 256.f, n));
    printf("%d 0 0\\n", MP_P);
    return 0;
}
""", include="multipole64.cuh")
    v = [int(x) for x in out]
    top = v[-3]

    def left(x, n, p):
        return sum(math.comb(l, n) * x ** (l - n) for l in range(p + 1, p + 400))

    for n, i, p in zip(v[:-3:3], v[1:-3:3], v[2:-3:3]):
        x, eps = i / 256.0, (2 * n + 1) * 2.0 ** -53
        if p:
            assert left(x, n, p) <= eps * 1.0001, (x, n, p)
        if p > max(n, 1):
            assert left(x, n, p - 1) > 0.9 * eps, (x, n, p)
        if p == 0:
            assert left(x, n, top) > 0.9 * eps, (x, n)
    assert any(v[2:-3:3])
