"""The fixed-point arithmetic of the direct kernels (csrc/gq_fix.cuh), compiled
for the host: reciprocal, logarithm, products and the shift that takes a
double's significand to a common format, against long double over random and
extreme significands.  The bounds are the ones stated beside the functions."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "gq_fix.cuh"
#include <stdio.h>
#include <random>
typedef long double L;
static L worst(L w, L e) { e = fabsl(e); return e > w ? e : w; }
static L val(gfx a) { return (L)a.h * 4294967296.0L + a.l; }
int main() {
    std::mt19937_64 g(1);
    static FxLogTable T;
    fx_log_table_host(&T);
    std::uniform_real_distribution<double> U(0, 1);
    L er = 0, el = 0, em = 0, ec = 0, ed = 0, eb = 0;
    for (int i = 0; i < 2000000; ++i) {
        double x = ldexp(1 + U(g), (int)(g() % 40) - 20);
        if (i < 2048) {   // the edges of the tables' cells and of the significand's range
            const uint64_t b = 0x3ff0000000000000ull | ((uint64_t)(i / 4) << 43);
            const uint64_t c = i % 4 == 0 ? b : i % 4 == 1 ? b + 1 : i % 4 == 2 ? b | 0x7ffffffffffull : b | 0x7ffffffull;
            memcpy(&x, &c, 8);
        }
        const uint64_t b = fx_bits(x), m = fx_mant(b);
        er = worst(er, (L)fx_rcp(m) / 0x1p62L * ((L)m / 0x1p52L) - 1);
        el = worst(el, (L)fx_log_half(b, 1020, T.hl, T.t) / 0x1p57L - 0.5L * (logl((L)x) + 3 * logl(2.0L)));
        // products: operands up to 2^62, low words of every pattern (INT_MIN among them)
        long long p = (long long)(g() >> 2) * ((g() & 1) ? 1 : -1), q = (long long)(g() >> 2) * ((g() & 1) ? 1 : -1);
        if (i % 3 == 0) p = (p & ~0xffffffffll) | 0x80000000ll;
        if (i % 5 == 0) q = (q & ~0xffffffffll) | 0x7fffffffll;
        const gfx P = fx_bal(p), Q = fx_bal(q);
        eb = worst(eb, val(P) - (L)p);
        em = worst(em, (L)fx_mul(P, Q) - (L)p * (L)q / 0x1p64L);
        // complex product: |a| < 2^60, |b| < 2^62
        const long long ar = p >> 3, ai = q >> 3, br = (q >> 1) | 1, bi = (p >> 1) | 1;
        const gfx X = fx_bal(br), Y = fx_bal(bi), N = {-Y.h, -Y.l};
        long long re, im;
        fx_cmul30(fx_split30(ar), fx_split30(ai), X, Y, N, re, im);
        ec = worst(ec, (L)re - ((L)ar * br - (L)ai * bi) / 0x1p62L);
        ec = worst(ec, (L)im - ((L)ar * bi + (L)ai * br) / 0x1p62L);
        // a double in the format of an exponent at least its own
        const int e = fx_expo(b) + (int)(g() % 60);
        ed = worst(ed, (L)fx_from_double(i & 1 ? x : -x, e) - ldexpl(i & 1 ? x : -x, 1022 - e + 62));
    }
    printf("%.21Le %.21Le %.21Le %.21Le %.21Le %.21Le %lld %lld\n", er, el, em, ec, ed, eb, fx_from_double(0.0, 1023),
           fx_from_double(0x1p-1030, 1023));
}
"""


def test_host_arithmetic(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(SRC)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1801_04070_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    rcp, log, mul, cmul, dbl, bal = map(float, out[:6])
    assert rcp < 2.0 ** -57
    # r^5 term beyond its mean 2^-53.8, table and constant roundings (20 exponents of 0.33 units of 2^-57)
    assert log < 2.0 ** -52.5
    # rounding 1/2, dropped low product 1/4
    assert mul <= 0.76
    # rounding 1/2, two dropped low products (2^31 2^29 / 2^62 at most each)
    assert cmul <= 1.01
    assert dbl < 1.0 and bal == 0.0
    assert out[6:] == ["0", "0"]
