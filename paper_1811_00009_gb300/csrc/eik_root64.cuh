// Alg. 3 in double precision (see eik_march.cuh for the single-precision root).
#pragma once

// (A host test compiles this file on its own, with the few helpers it needs.)
#ifdef __CUDACC__
#include "eik_march.cuh"
#endif

namespace eikg {

// Alg. 3 in double precision: the exact root of G(x) = sum_i max(x - v_i, 0)^2 =
// r^2 rounded to nearest (down in a tie, but see root_below_mid).  The exact root is monotone in (a, b, c)
// and rounding is monotone, so this root is too, and psi does not depend on the
// order of the work (see eik_march.cuh, whose single-precision root is monotone in
// another way).
//
// It uses no double arithmetic: a double-precision warp instruction occupies its
// scheduler's FP64 pipe for 64 cycles on this part, and the evaluation of the root
// and of G in double took about 80 of them (4600 cycles for 32 nodes by one warp
// alone).  Differences of doubles within a factor of two are integers in units of
// the smaller one's last place, and h/F (53 bits) sets the unit V, its own last
// place, in which all of x - v_i is an integer below 2^54.  The estimate is made in
// single precision and corrected by Newton's method: once on 31-bit values, once on
// the high 64 bits of the squares.  What the 31 bits cut off the inputs moves the
// root by up to (r + t_b + t_c) / (t_a + t_b + t_c) <= 1.25 times 2^22 V (t_i = x -
// v_i); the second step leaves of that the relative error of sqrt(D)'s reciprocal in
// single precision, and adds its own rounding (0.65 V).  With the rounding errors of
// D taken at their bounds and 2^-22.9 for the approximation that is 3.6 V at most
// (where b and c lie close to a + h/F; 2.6 V found).  Half an ulp of x is at least
// 2^(s-1) V, s being the difference of a's and h/F's exponents: enough for s >= 3.
// For s = 1 and 2 (h/F an eighth of a up to a itself: nodes near a source) the second
// step is taken twice, which leaves 0.65 V, out of line: with one step up to 1 root in
// 10^7 was an ulp off at s = 2.  (Twice for s <= 3, inline: 192^3 9.67 -> 10.04 ms.)
// Which of the two neighbouring doubles is nearer is then decided exactly: G at
// their midpoint against r^2, in 128-bit integers.
__device__ __forceinline__ unsigned long long mantissa(double v) {
    return (ubits(v) & 0xfffffffffffffull) | 0x10000000000000ull;
}
struct U128 {
    unsigned long long hi, lo;
};
// t^2 for t < 2^55, from 32-bit halves
__device__ __forceinline__ U128 square(unsigned long long t) {
    const unsigned l = static_cast<unsigned>(t), h = static_cast<unsigned>(t >> 32);
    const unsigned long long ll = static_cast<unsigned long long>(l) * l, m = (static_cast<unsigned long long>(h) * l) << 1;
    U128 p;
    p.lo = ll + (m << 32);
    p.hi = static_cast<unsigned long long>(h) * h + (m >> 32) + (p.lo < ll ? 1ull : 0ull);
    return p;
}
__device__ __forceinline__ void add(U128& s, U128 p) {
    s.lo += p.lo;
    s.hi += p.hi + (s.lo < p.lo ? 1ull : 0ull);
}

// The estimate of T = x - a from the first 31 bits of h/F and, in its units, of b - a
// and c - a (values beyond h/F: not admitted), with the first Newton step, (r^2 - G) /
// (2 sqrt(D)): in units V, and the reciprocal of sqrt(D) in units 2^-52 / V.
__device__ __forceinline__ unsigned long long root_start(unsigned r31, unsigned db, unsigned dc, float& rs) {
    using U = unsigned long long;
    const float rf = static_cast<float>(r31) * 0x1p-30f;
    const float df = fminf(static_cast<float>(db) * 0x1p-30f, rf), ef = fminf(static_cast<float>(dc) * 0x1p-30f, rf);
    const float rf2 = rf * rf, gf = ef - df;
    const float q1 = __fmaf_rn(-df, df, rf2), q2 = rf2 - __fmaf_rn(gf, gf, ef * ef);
    const bool p1 = q1 > 0.0f, p2 = q2 > 0.0f;
    const float D = rf2 + fmaxf(q1, 0.0f) + fmaxf(q2, 0.0f);
    rs = rsqrt_approx(D);
    float sum = p1 ? df : 0.0f;
    sum = p2 ? sum + ef : sum;
    const float inv = p2 ? (1.0f / 3.0f) : (p1 ? 0.5f : 1.0f);
    const unsigned t = static_cast<unsigned>(__fmaf_rn(D, rs, sum) * inv * 0x1p30f);
    const unsigned tb = t > db ? t - db : 0u, tc = t > dc ? t - dc : 0u;
    const U G = static_cast<U>(t) * t + static_cast<U>(tb) * tb + static_cast<U>(tc) * tc;
    const int rho = static_cast<int>(static_cast<long long>(static_cast<U>(r31) * r31 - G) >> 12);
    return (static_cast<U>(t) << 22) + (static_cast<long long>(__float2int_rn(static_cast<float>(rho) * (rs * 0x1p-5f))) << 8);
}

// Ea: a's exponent bits, s: by how much they exceed h/F's, 1 ... 44 (h/F is then below
// a, v - a and x - v integers in V; and h/F squared within the integers).
// TWICE: the second Newton step twice.
template <bool TWICE>
__device__ __forceinline__ double root_int(double a, double b, double c, double r, int Ea, int s) {
    using U = unsigned long long;
    const U A = mantissa(a), R = mantissa(r);
    // (v - a) in units V; a value above a + h/F is not admitted: beyond any T
    auto above_a = [&](double v) -> U {
        const int k = (__double2hiint(v) >> 20) - Ea;
        const U d = (k == 1 ? mantissa(v) << 1 : mantissa(v)) - A;
        return static_cast<unsigned>(k) <= 1u && d <= (R >> s) ? d << s : (U(1) << 54) - 1;
    };
    const U Db = above_a(b), Dc = above_a(c);
    float rs;
    U T = root_start(static_cast<unsigned>(R >> 22), static_cast<unsigned>(Db >> 22), static_cast<unsigned>(Dc >> 22), rs);
    // the second step on the squares' bits from 2^44 up
    auto refine = [&]() {
        const U tb = T > Db ? (T - Db) << 10 : 0ull, tc = T > Dc ? (T - Dc) << 10 : 0ull;
        const U G = __umul64hi(T << 10, T << 10) + __umul64hi(tb, tb) + __umul64hi(tc, tc);
        const int rho = static_cast<int>(static_cast<long long>(__umul64hi(R << 10, R << 10) - G) >> 6);
        T += static_cast<long long>(__float2int_rn(static_cast<float>(rho) * (rs * 0x1p-3f)));
    };
    refine();
    if (TWICE) refine();
    // the double at or below a + T (mantissa X in a's last place, in steps of two from 2^53 up), and the midpoint above it
    U X = A + (T >> s);
    const int two = X >> 53 ? 1 : 0;
    X &= ~static_cast<U>(two);
    const U M = ((X - A) << s) + (U(1) << (s - 1 + two));
    U128 G = square(M);
    add(G, square(M > Db ? M - Db : 0ull));
    add(G, square(M > Dc ? M - Dc : 0ull));
    const U128 Q = square(R);
    if (G.hi < Q.hi || (G.hi == Q.hi && G.lo < Q.lo)) X += 1u + two;
    const int up = X >> 53 ? 1 : 0;
    return from_bits((static_cast<U>(Ea + up) << 52) | ((X >> up) & 0xfffffffffffffull));
}


// Where a is below twice h/F (next to a source, or at a jump of the speed) x - a no
// longer lies within a factor of two of h/F's last place: the same in units W =
// 2^-10 V, with 64-bit values.  What lies below a W of a, b or c is cut off; a Newton
// step more leaves T within 8 W, of the half ulp of x that is at least 256 W, so that
// the fraction of x alone settles all but one root in sixteen, and G at the midpoint
// those (cut values: with its lower bound; false if even that leaves it open).  All
// in double-double, as the rest below, those roots took about 200 FP64 operations:
// 9^3 0.92 -> 0.28 ms, 64^3 1.80 -> 1.71, 48^3 of speeds 0.1 ... 10 drawn per node,
// infinite stride, 16.8 -> 4.9.
__device__ __forceinline__ U128 square64(unsigned long long t) { return U128{__umul64hi(t, t), t * t}; }
__device__ __forceinline__ bool below(U128 p, U128 q) { return p.hi < q.hi || (p.hi == q.hi && p.lo < q.lo); }
__device__ __forceinline__ bool root_wide(double a, double b, double c, double r, double& x) {
    using U = unsigned long long;
    constexpr U kFar = ~0ull;
    const int Er = __double2hiint(r) >> 20;
    const U R = mantissa(r) << 10;
    bool cut = false;
    auto fixed = [&](double v) -> U {
        const int E = __double2hiint(v) >> 20, k = (E > 0 ? E : 1) - Er + 10;
        const U m = (ubits(v) & 0xfffffffffffffull) | (E > 0 ? 0x10000000000000ull : 0ull);
        if (k >= 0) return k <= 11 ? m << k : kFar;              // (beyond 4 h/F: not admitted)
        const U w = k > -53 ? m >> -k : 0ull;
        cut = cut || (k > -53 ? w << -k : 0ull) != m;
        return w;
    };
    const U A = fixed(a), fb = fixed(b), fc = fixed(c);
    const U Db = fb == kFar ? kFar : fb - A, Dc = fc == kFar ? kFar : fc - A;
    float rs;
    U T = root_start(static_cast<unsigned>(R >> 32), static_cast<unsigned>(Db >> 32), static_cast<unsigned>(Dc >> 32), rs) << 10;
    auto residual = [&]() -> long long {                          // r^2 - G, in units 2^64 W^2
        const U tb = T > Db ? T - Db : 0ull, tc = T > Dc ? T - Dc : 0ull;
        return static_cast<long long>(__umul64hi(R, R) - (__umul64hi(T, T) + __umul64hi(tb, tb) + __umul64hi(tc, tc)));
    };
    T += static_cast<long long>(__float2int_rn(static_cast<float>(static_cast<int>(residual() >> 6)) * (rs * 0x1p-3f))) << 10;
    T += static_cast<long long>(__float2int_rn(static_cast<float>(static_cast<int>(residual())) * (rs * 2.0f)));
    const U X = A + T;
    const int n = 11 - __clzll(X);                                // (an ulp of x is 2^n W, n >= 9)
    const U half = U(1) << (n - 1), frac = X & (2 * half - 1);
    U up = frac > half ? 1ull : 0ull;
    if (frac - half + 16 <= 32) {
        const U M = (X - frac + half) - A, mb = M > Db ? M - Db : 0ull, mc = M > Dc ? M - Dc : 0ull;
        const U128 Q = square64(R);
        U128 G = square64(M);
        add(G, square64(mb));
        add(G, square64(mc));
        up = below(G, Q) ? 1ull : 0ull;
        if (up == 0 && cut) {
            G = square64(M - 1);
            add(G, square64(mb > 0 ? mb - 1 : 0ull));
            add(G, square64(mc > 0 ? mc - 1 : 0ull));
            if (below(G, Q)) return false;
        }
    }
    x = from_bits((static_cast<U>(Er + n - 11) << 52) + (X >> n) + up);
    return true;
}

// What is left (h/F below 2^-44 of the values, values or h/F at the ends of the range):
// the predicate "the root lies at or below the midpoint of x and the next value" with
// G - r^2 in double-double arithmetic, searched from the estimate.  (An exact tie may
// go either way here, always the same for the same admitted values.)
__device__ __forceinline__ bool root_below_mid(double x, double a, double b, double c, double r) {
    const double half = 0.5 * __dsub_rn(from_bits(ubits(x) + 1), x);
    const double p = __dmul_rn(r, r);
    double hi = -p, lo = -__fma_rn(r, r, -p);
    const double v[3] = {a, b, c};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (!vlt(v[i], Num<double>::inf())) continue;
        // t = x - v + half as t0 + t1
        const double s = __dsub_rn(x, v[i]), bb = __dsub_rn(s, x);
        const double e = __dsub_rn(__dsub_rn(x, __dsub_rn(s, bb)), __dadd_rn(v[i], bb));
        const double t0 = __dadd_rn(s, half), tb = __dsub_rn(t0, s);
        const double t1 = __dadd_rn(e, __dadd_rn(__dsub_rn(s, __dsub_rn(t0, tb)), __dsub_rn(half, tb)));
        if (!(t0 > 0.0)) continue;
        const double q = __dmul_rn(t0, t0);
        const double qe = __dadd_rn(__fma_rn(t0, t0, -q), __dmul_rn(2.0 * t0, t1));
        const double z = __dadd_rn(hi, q), zb = __dsub_rn(z, hi);
        lo = __dadd_rn(__dadd_rn(lo, qe), __dadd_rn(__dsub_rn(hi, __dsub_rn(z, zb)), __dsub_rn(q, zb)));
        hi = z;
    }
    return __dadd_rn(hi, lo) >= 0.0;
}
static __device__ __noinline__ double root_rare(double a, double b, double c, double r) {
    using U = unsigned long long;
    const int Ea = __double2hiint(a) >> 20, Er = __double2hiint(r) >> 20;
    const int sh = Ea - Er;
    if (static_cast<unsigned>(sh - 1) <= 1u && Er >= 1 && Ea < 2046) return root_int<true>(a, b, c, r, Ea, sh);
    double x;
    if (sh <= 0 && Er >= 2 && Er <= 2040 && root_wide(a, b, c, r, x)) return x;
    if (sh > 54) return a;                                        // (h/F below half an ulp of a)
    // (the squares' exponents stay in range: the larger of a and h/F scaled to 1 ... 2)
    const int E = min(max(max(Ea, Er), 1), 2045);
    const double scale = from_bits(static_cast<U>(2046 - E) << 52);
    a = __dmul_rn(a, scale);
    b = __dmul_rn(b, scale);
    c = __dmul_rn(c, scale);
    r = __dmul_rn(r, scale);
    const U ua = ubits(a), top = BitsOf<double>::kInf - 1;
    U g = ubits(root_estimate(a, b, c, r));
    if (!(g > ua) || g > top) g = ua;
    U lo, hi;                          // root above the midpoint after lo (lo = ua - 1: none), at or below that after hi
    U step = 1;
    if (root_below_mid(from_bits(g), a, b, c, r)) {
        hi = g;
        for (;;) {
            if (hi - ua < step) {
                lo = ua - 1;
                break;
            }
            const U y = hi - step;
            if (!root_below_mid(from_bits(y), a, b, c, r)) {
                lo = y;
                break;
            }
            hi = y;
            step <<= 1;
        }
    } else {
        lo = g;
        for (;;) {
            const U y = top - lo > step ? lo + step : top;
            hi = y;
            if (y == top || root_below_mid(from_bits(y), a, b, c, r)) break;
            lo = y;
            step <<= 1;
        }
    }
    while (hi - lo > 1) {
        const U mid = lo + ((hi - lo) >> 1);
        if (root_below_mid(from_bits(mid), a, b, c, r)) hi = mid;
        else lo = mid;
    }
    return __dmul_rn(from_bits(hi), from_bits(static_cast<U>(E) << 52));
}

__device__ __forceinline__ double root_fast(double a, double b, double c, double r, bool live) {
    const int Ea = __double2hiint(a) >> 20, Er = __double2hiint(r) >> 20, sh = Ea - Er;
    const bool ok = static_cast<unsigned>(sh - 3) <= 41u && Er >= 1 && Ea < 2046;    // (normal numbers)
    double x = root_int<false>(a, b, c, r, Ea, ok ? sh : 3);
    if (live && !ok) x = root_rare(a, b, c, r);
    return x;
}

}  // namespace eikg
