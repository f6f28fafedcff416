"""The double-precision root (eik_root64.cuh) compiled for the host: it is the exact root of sum_i max(x - v_i, 0)^2 = r^2
rounded to nearest (down in a tie), whatever the approximate reciprocal square root that its estimate starts from is
within its documented error bound (2^-22.9 relative).

The check needs no other root: x is right exactly when the root lies above the midpoint of x and the double below it and
not above the midpoint of x and the double above it, which 128-bit integers decide where h/F is a quarter of the values
down to 2^-44 of them (the integers' range in the header), in units of half the last place of h/F.
"""
import ctypes as C
import math
import os
import random
import subprocess
from fractions import Fraction

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
using std::fmaxf;
using std::max;
using std::min;
using std::fminf;
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
    return static_cast<unsigned long long>((static_cast<unsigned __int128>(a) * b) >> 64);
}
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline int __float2int_rn(float a) { return static_cast<int>(std::nearbyint(a)); }
static inline int __clzll(long long v) { return __builtin_clzll(static_cast<unsigned long long>(v)); }
static inline int __double2hiint(double v) {
    unsigned long long u;
    std::memcpy(&u, &v, 8);
    return static_cast<int>(u >> 32);
}
static double g_bend = 0.0;            // relative error given to the reciprocal square root
static long g_rare = 0;
namespace eikg {
static inline unsigned long long ubits(double v) {
    unsigned long long u;
    std::memcpy(&u, &v, 8);
    return u;
}
static inline double from_bits(unsigned long long u) {
    double v;
    std::memcpy(&v, &u, 8);
    return v;
}
static inline bool vlt(double a, double b) { return ubits(a) < ubits(b); }
template <typename T> struct BitsOf;
template <> struct BitsOf<double> {
    using U = unsigned long long;
    static constexpr U kInf = 0x7ff0000000000000ull;
};
template <typename T> struct Num;
template <> struct Num<double> {
    static double inf() { return INFINITY; }
};
static inline float rsqrt_approx(float x) {
    return static_cast<float>(1.0 / std::sqrt(static_cast<double>(x)) * (1.0 + g_bend));
}
static inline double root_estimate(double a, double b, double c, double r) {
    ++g_rare;
    return a + r;                      // (it only starts a search)
}
}  // namespace eikg
#include "eik_root64.cuh"
using U = unsigned long long;
using I = __int128;

// Does the root lie at or below the midpoint of x and the next double?  Values in units of half of r's last place.
static bool below_mid(double x, double a, double b, double c, double r) {
    int er;
    std::frexp(r, &er);
    const int unit = er - 54;
    auto q = [&](double v) -> I { return static_cast<I>(std::ldexp(v, -unit)); };
    const double up = eikg::from_bits(eikg::ubits(x) + 1);
    const I m = (q(x) + q(up)) / 2;
    I g = 0;
    for (double v : {a, b, c})
        if (std::isfinite(v) && q(v) < m) {
            const I t = m - q(v);
            if (t > (static_cast<I>(1) << 61)) return true;
            g += t * t;
        }
    return g >= q(r) * q(r);
}
static bool right(double x, double a, double b, double c, double r) {
    return below_mid(x, a, b, c, r) && !below_mid(eikg::from_bits(eikg::ubits(x) - 1), a, b, c, r);
}
static uint64_t g_s;
static uint64_t rnd() {
    g_s += 0x9e3779b97f4a7c15ull;
    uint64_t z = g_s;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}
extern "C" double one(double a, double b, double c, double r, double bend, int* ok, long* rare) {
    g_bend = bend;
    g_rare = 0;
    const double x = eikg::root_fast(a, b, c, r, true);
    *ok = right(x, a, b, c, r);
    *rare = g_rare;
    return x;
}
// n draws with exponent difference sh between a and h/F; kind 0: any mantissas; 1: h/F and the differences end in ones (the
// estimate's integers cut them the most); 2: the same with b, c close to a.  Wrong roots; bad gets the first one's inputs.
extern "C" long wrong(long n, int sh, int kind, double bend, uint64_t seed, double* bad, long* rare) {
    g_s = seed;
    g_bend = bend;
    g_rare = 0;
    long w = 0;
    const U one52 = U(1) << 52;
    for (long i = 0; i < n; ++i) {
        U R = one52 | (rnd() >> 12);
        const U A = one52 | (rnd() >> 12);
        if (kind) R |= 0x3fffffu;
        const U reach = R >> sh;                          // h/F in units of a's last place
        auto diff = [&]() -> U {
            U d = static_cast<U>((static_cast<unsigned __int128>(rnd()) * (reach + 1)) >> 64);
            if (kind == 2) d = static_cast<U>((static_cast<unsigned __int128>(rnd()) * (reach / 64 + 1)) >> 64);
            if (kind) d |= (U(1) << (22 - std::min(sh, 22))) - 1;
            return d;
        };
        U db = diff(), dc = diff();
        if (db > dc) std::swap(db, dc);
        auto val = [&](U m) { return std::ldexp(static_cast<double>(m), -50); };
        // (sums of mantissas beyond 2^53 lose their last bit: the draw is then another, as good)
        const double a = val(A), b = val(A + db), c = rnd() % 8 == 0 ? INFINITY : val(A + dc);
        const double r = std::ldexp(static_cast<double>(R), -50 - sh);
        const double x = eikg::root_fast(a, b, c, r, true);
        if (!right(x, a, b, c, r)) {
            if (w++ == 0) bad[0] = a, bad[1] = b, bad[2] = c, bad[3] = r;
        }
    }
    *rare = g_rare;
    return w;
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("root64")
    src, lib = d / "harness.cpp", d / "harness.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared",
                    "-I" + os.path.join(ROOT, "paper_1811_00009_gb300", "csrc"), str(src), "-o", str(lib)], check=True)
    L = C.CDLL(str(lib))
    dp = C.POINTER(C.c_double)
    L.one.restype = C.c_double
    L.one.argtypes = [C.c_double] * 5 + [C.POINTER(C.c_int), C.POINTER(C.c_long)]
    L.wrong.restype = C.c_long
    L.wrong.argtypes = [C.c_long, C.c_int, C.c_int, C.c_double, C.c_uint64, dp, C.POINTER(C.c_long)]
    return L


BEND = 2.0 ** -22.9


@pytest.mark.parametrize("bend", [0.0, BEND, -BEND])
def test_a_root_two_units_from_its_estimate(host, bend):
    """h/F just above a quarter of psi, differences whose cut-off bits add up: half a last place is then two units of
    the estimate's integers."""
    ok = C.c_int()
    h = float.fromhex
    x = host.one(h("0x1.7c350f80955f7p+2"), h("0x1.c3fe31f2c41a8p+2"), h("0x1.c3fe32638e46p+2"),
                 h("0x1.25da52f7cfdc4p+0"), bend, C.byref(ok), C.byref(C.c_long()))
    assert ok.value, x.hex()


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("sh", [1, 2, 3, 4, 5, 8, 16, 30, 43, 44])
def test_exactly_rounded(host, sh, kind):
    bad, rare = (C.c_double * 4)(), C.c_long()
    for j, bend in enumerate((0.0, BEND, -BEND)):
        n = 1000000 if sh <= 4 else 100000
        w = host.wrong(n, sh, kind, bend, 1000 * sh + 10 * kind + j, bad, C.byref(rare))
        assert rare.value == 0                            # (the integers' path throughout)
        assert w == 0, (w, [v.hex() for v in bad])


def past_mid(x, toward, values, r):
    """G at the midpoint of x and its neighbour, less r^2 (exactly)."""
    m = (Fraction(x) + Fraction(math.nextafter(x, toward))) / 2
    return sum(max(m - Fraction(v), 0) ** 2 for v in values if v < math.inf) - Fraction(r) ** 2


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -1000, 2.0 ** 900])
@pytest.mark.parametrize("sh", [1, 0, -1, -2, -5, -9, -10, -11, -12, -30, -70, None])
def test_exactly_rounded_where_psi_is_small_against_h_over_f(host, sh, scale):
    """Next to a source and at jumps of the speed: psi of any size below h/F (None: zero), values whose last bits lie below
    h/F's, ties.  The search in double-double is left for hardly any of them; there alone a tie may go up."""
    rnd = random.Random(9 if sh is None else sh)
    ok, rare = C.c_int(), C.c_long()
    searched, n = 0, 1500
    for i in range(n):
        r = rnd.uniform(1, 2) if i % 3 else (2 ** 20 + rnd.getrandbits(20)) / 2.0 ** 20
        a = 0.0 if sh is None else rnd.uniform(1, 2) * 2.0 ** sh
        b, c = sorted(a + r * 1.2 * rnd.random() * 2.0 ** -rnd.randrange(0, 40, 3) for _ in range(2))
        if i % 7 == 0:
            b = a
        if i % 5 == 0:
            c = rnd.choice([b, math.inf])
        a, b, c, r = (v * scale for v in (a, b, c, r))
        x = host.one(a, b, c, r, (0.0, BEND, -BEND)[i % 3], C.byref(ok), C.byref(rare))
        searched += rare.value
        assert past_mid(x, math.inf, (a, b, c), r) >= 0, (a, b, c, r)
        below = past_mid(x, 0.0, (a, b, c), r)
        assert below < 0 or (below == 0 and rare.value), (a, b, c, r)
    assert searched <= n // 100
