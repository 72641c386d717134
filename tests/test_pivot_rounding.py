"""The factors' square roots and quotients (csrc/pivot.cuh), compiled for the
host, against the C library's sqrt and division, where rounding is hardest:

- quotients next to the middle between two numbers: numerators V with
  V 2^s - M L = +-1, +-3, ... for the divisor's mantissa L and an odd 54-bit M,
  over random pivots and the divisors closest to the excluded all-ones mantissa;
- roots next to a middle: every d = D 2^-52, D 2^-51 whose D 2^54 or D 2^55 is within
  200 of an odd square, with every y inside its bound;
- divisors whose reciprocal is next to a middle (the factorisations of
  2^106 +- 16), where the stored reciprocal can be the neighbour of RN(1 / l);
- operands on both sides of the tests for the range, subnormals and zeros.

The hardware's approximation of the reciprocal square root is replaced by
1 / sqrt(d) (1 + t), |t| <= 2^-20 (and by every y inside the bound)."""
import math
import shutil
import subprocess
from fractions import Fraction as F
import os

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(HERE, "..", "paper_2510_02156_gb300", "csrc", "pivot.cuh")

SRC = r"""
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
#define __device__
#define __forceinline__ inline
#define __noinline__
struct int2 { int x, y; };
static inline double __fma_rn(double a, double b, double c) { return fma(a, b, c); }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __hiloint2double(int hi, int lo) {
    uint64_t w = (uint64_t)(uint32_t)hi << 32 | (uint32_t)lo;
    double d;
    memcpy(&d, &w, 8);
    return d;
}
#include "%s"
using namespace rorbk;
typedef unsigned __int128 u128;
static uint64_t st = 88172645463325252ull;
static uint64_t rnd() { st ^= st << 13; st ^= st >> 7; st ^= st << 17; return st * 2685821657736338717ull; }
static double uni() { return (double)(rnd() >> 11) * 0x1p-53; }
static long nbad = 0, npairs = 0;
static bool same(double a, double b) { return a == b || (a != a && b != b); }
static void div_check(double v, const Pivot &p, const char *what) {
    const double want = v / p.l, q = pivot_div(v, p);
    ++npairs;
    if (!same(q, want) && nbad++ < 5)
        printf("%%s: v %%a l %%a rl %%a y %%a: %%a, v / l = %%a\n", what, v, p.l, p.rl, p.y, q, want);
}
static Pivot make(double d, double y) {
    const Pivot p = pivot_from(d, y, root_ok(d));
    if (p.l != sqrt(d) && nbad++ < 5) printf("root: d %%a y %%a: %%a, sqrt %%a\n", d, y, p.l, sqrt(d));
    return p;
}
// numerators next to a middle for the divisor l in [1, 2)
static void hard(const Pivot &p, int jmax, const char *what) {
    uint64_t L = (uint64_t)ldexp(p.l, 52);
    const int z = __builtin_ctzll(L);
    const uint64_t Lo = L >> z;
    uint64_t inv = Lo;                                   // 1 / Lo mod 2^64
    for (int i = 0; i < 6; ++i) inv *= 2 - Lo * inv;
    for (int s = 53; s <= 54; ++s)
        for (int j = -jmax; j <= jmax; j += 2) {
            const uint64_t mod = z >= s ? 1 : 1ull << (s - z), m0 = (uint64_t)(-(int64_t)j) * inv;
            uint64_t M = (m0 & (mod - 1)) | ((rnd() << (s - z)) & ((1ull << 53) - 1));
            M = (M & ((1ull << 53) - 1)) | 1ull << 53;
            if (!(M & 1)) continue;
            const u128 n = (u128)M * L + (u128)(__int128)((__int128)j << z);
            if (n & (((u128)1 << s) - 1)) continue;
            const uint64_t V = (uint64_t)(n >> s);
            if (V < 1ull << 52 || V >= 1ull << 53) continue;
            div_check((double)V, p, what);
            div_check(-(double)V, p, what);
        }
}
int main(int argc, char **argv) {
    const long n = atol(argv[1]);
    // every (d, y) given: the root, and quotients by it
    double d, y;
    long given = 0;
    while (scanf("%%lf %%lf", &d, &y) == 2) { hard(make(d, y), 31, "given"); ++given; }
    // random pivots, seeds good to 20 bits; y inside its bound
    for (long i = 0; i < n; ++i) {
        d = 1.0 + 3.0 * uni();
        const double y0 = 1.0 / sqrt(d) * (1.0 + (2.0 * uni() - 1.0) * 0x1p-20);
        y = refine_recip(d, y0);
#if __LDBL_MANT_DIG__ >= 64
        if (fabsl((long double)y * sqrtl((long double)d) - 1.0L) > 1.61L * 0x1p-53L && nbad++ < 5)
            printf("y: d %%a y0 %%a y %%a\n", d, y0, y);
#endif
        hard(make(d, y), 5, "random");
    }
    // divisors at and next to the excluded mantissas; numerators at the top as well
    for (int k = 1; k <= 4096; ++k) {
        const double l = 2.0 - k * 0x1p-52;
        for (int i = -3; i <= 3; ++i) {
            d = l * l + i * 0x1p-51;
            if (sqrt(d) != l) continue;
            y = 1.0 / sqrt(d);
            for (int t = -1; t <= 1; ++t) {
                const Pivot p = make(d, y + t * 0x1p-54);
                hard(p, 63, "top");
                for (int j = 0; j < 64; ++j) div_check(2.0 - j * 0x1p-52, p, "top");
            }
        }
    }
    // both sides of the range tests
    const int es[] = {-1074, -1050, -1023, -1022, -800, -602, -601, -600, -599, -301, -300, -299, 0,
                      299, 300, 301, 599, 600, 601, 602, 800, 1023};
    for (int a : es)
        for (int b : es)
            for (int i = 0; i < 40; ++i) {
                d = ldexp(1.0 + uni(), a);
                if (!(d > 0.0)) continue;
                y = root_ok(d) ? refine_recip(d, 1.0 / sqrt(d) * (1.0 + (2.0 * uni() - 1.0) * 0x1p-20)) : 1.0 / sqrt(d);
                const Pivot p = make(d, y);
                div_check(ldexp(i & 1 ? 1.0 + uni() : 2.0 - 0x1p-52, b), p, "range");
                div_check(0.0, p, "range");
                div_check(INFINITY, p, "range");
                div_check(NAN, p, "range");
            }
    printf("%%ld %%ld %%ld\n", given, npairs, nbad);
    return nbad != 0;
}
"""


def _rn(x):
    """The FP64 number nearest to a positive Fraction in the normal range."""
    e = x.numerator.bit_length() - x.denominator.bit_length()
    if F(2) ** e > x:
        e -= 1
    q = x / F(2) ** (e - 52)
    n = q.numerator // q.denominator
    r = q - n
    if r > F(1, 2) or (r == F(1, 2) and n & 1):
        n += 1
    return float(n * F(2) ** (e - 52))


def _ys(d):
    """Every FP64 y with |y sqrt(d) - 1| <= 1.6 2^-53."""
    b = F(16, 10) / F(2) ** 53
    y = _rn(F(math.isqrt(int(F(2) ** 400 / F(d))), 2 ** 200))
    for _ in range(4):
        y = math.nextafter(y, 0.0)
    for _ in range(9):
        if (1 - b) ** 2 <= F(y) * F(y) * F(d) <= (1 + b) ** 2:
            yield y
        y = math.nextafter(y, 4.0)


def _hard_roots():
    """d in [1, 4) whose root is next to a middle: (M 2^-53)^2 ~ d, M odd."""
    for s, ud in ((54, 52), (55, 51)):
        lo, hi = (2 ** 53, math.isqrt(2 ** 107)) if s == 54 else (math.isqrt(2 ** 107) + 1, 2 ** 54)
        for j in range(-200, 201):
            if (-j) % 8 != 1:                             # odd squares are 1 mod 8
                continue
            x = 1                                         # x^2 = -j mod 2^s, bit by bit
            for b in range(3, s):
                if (x * x + j) >> b & 1:
                    x += 1 << (b - 1)
            for r in {x % 2 ** s, -x % 2 ** s, (x + 2 ** (s - 1)) % 2 ** s, (-x + 2 ** (s - 1)) % 2 ** s}:
                for M in (r, r + 2 ** s):
                    D = (M * M + j) >> s
                    if lo <= M < hi and 2 ** 52 <= D < 2 ** 53:
                        yield math.ldexp(D, -ud)


def _hard_reciprocals():
    """d whose root l has 1 / l next to a middle: L M = 2^106 + j, M odd."""
    sympy = pytest.importorskip("sympy")
    for j in range(-16, 17):
        if not j:
            continue
        divs = [1]
        for p, e in sympy.factorint(2 ** 106 + j).items():
            divs = [q * p ** i for q in divs for i in range(e + 1)]
        for L in divs:
            if 2 ** 52 <= L < 2 ** 53 and (2 ** 106 + j) // L % 2:
                l = math.ldexp(L, -52)
                d = l * l
                for _ in range(6):
                    d = math.nextafter(d, 0.0)
                for _ in range(13):
                    if 1.0 <= d < 4.0 and math.sqrt(d) == l:
                        yield d
                    d = math.nextafter(d, 5.0)


@pytest.mark.skipif(shutil.which("g++") is None, reason="g++ not available")
def test_roots_and_quotients_are_correctly_rounded(tmp_path):
    pairs = [(d, y) for gen in (_hard_roots, _hard_reciprocals) for d in gen() for y in _ys(d)]
    assert len(pairs) > 400
    src, exe = tmp_path / "pivot.cpp", tmp_path / "pivot"
    src.write_text("#include <stdlib.h>\n" + SRC % os.path.abspath(HEADER))
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe), "2000000"], input="\n".join(f"{d.hex()} {y.hex()}" for d, y in pairs),
                         capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:]
    given, npairs, bad = map(int, out.stdout.split()[-3:])
    assert bad == 0 and given == len(pairs) and npairs > 4000000
