// Device code shared by the restart-loop kernels (one grid, eik_kernels.cu; many
// grids, eik_batch.cu): the upwind root of Alg. 3 and the restart loop's machinery
// -- the ring of work lists, the grid barrier that CTAs arrive at and poll as one,
// and the early marches of the next restart while they wait.  The marches of one
// block (Alg. 4) are in eik_march8.cuh (a warp per 8^3 block), eik_march16.cuh (a
// CTA per 16^3 block) and eik_block32.cu (a CTA per 32^3 block).
#pragma once

#include "eik_internal.cuh"

#include <cfloat>
#include <cstdint>

namespace eikg {
constexpr unsigned kFull = 0xffffffffu;
constexpr int kRoundCap = 1 << 20;

template <typename T>
struct Num;
template <>
struct Num<float> {
    static __device__ __forceinline__ float inf() { return __int_as_float(0x7f800000); }
};
template <>
struct Num<double> {
    static __device__ __forceinline__ double inf() { return __longlong_as_double(0x7ff0000000000000LL); }
};

__device__ __forceinline__ bool sgn(float v) { return (__float_as_uint(v) >> 31) != 0u; }
__device__ __forceinline__ bool sgn(double v) {
    return (static_cast<unsigned long long>(__double_as_longlong(v)) >> 63) != 0ull;
}
__device__ __forceinline__ unsigned ubits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ unsigned long long ubits(double v) {
    return static_cast<unsigned long long>(__double_as_longlong(v));
}
__device__ __forceinline__ float from_bits(unsigned u) { return __uint_as_float(u); }
__device__ __forceinline__ double from_bits(unsigned long long u) {
    return __longlong_as_double(static_cast<long long>(u));
}
__device__ __forceinline__ float vabs(float v) { return fabsf(v); }
// (double precision on the bits: the compiler's negation and absolute value of a
// double are FP64-pipe instructions)
__device__ __forceinline__ double vabs(double v) { return from_bits(ubits(v) & 0x7fffffffffffffffull); }
__device__ __forceinline__ float vneg(float v) { return -v; }
__device__ __forceinline__ double vneg(double v) { return from_bits(ubits(v) ^ 0x8000000000000000ull); }
// Min, max and order of values that are >= 0 or +inf (every use in the march):
// single precision on the FP32 units; double precision as integer operations on
// the bit patterns, which order like such values, keeping them off this part's
// narrow FP64 pipe.
__device__ __forceinline__ float vmin(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double vmin(double a, double b) {
    const unsigned long long x = ubits(a), y = ubits(b);
    return from_bits(x < y ? x : y);
}
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double vmax(double a, double b) {
    const unsigned long long x = ubits(a), y = ubits(b);
    return from_bits(x > y ? x : y);
}
__device__ __forceinline__ bool vlt(float a, float b) { return a < b; }
__device__ __forceinline__ bool vlt(double a, double b) { return ubits(a) < ubits(b); }

__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(unsigned* p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// ---------------------------------------------------------------------------
// Alg. 3: the upwind root for sorted upwind values a <= b <= c (b, c may be
// +inf) and r = h/F.  Alg. 3 solves sum_i (x - v_i)^2 = r^2 (Eq. (2.1)-(2.2))
// for the id smallest values, growing id while the root exceeds the next
// value.  Equivalently the root is the x with G(x) = r^2, where
//   G(x) = sum_i max(x - v_i, 0)^2
// is non-decreasing in x and non-increasing in every v_i: a value v_i >= x
// adds nothing, which is the growth rule of Alg. 3.
//
// In double precision the marches take the exact root rounded to the nearest
// double (root_fast in eik_root64.cuh).  In single precision they take the value x
// at which G_fl(x) comes nearest r^2 from either side (root_search), G_fl being G
// evaluated with round-to-nearest operations in a fixed order (largest term
// first; no contraction); every operation in G_fl is monotone in its operands, so
// G_fl keeps both monotonicities.  Either root is a monotone function of
// (a, b, c): a neighbour that is lower can never give a higher root.  The discrete
// solution is the
// greatest fixed point of psi_p = min(psi_p, root_p(neighbours)) below the
// initial values (+inf off the sources); iterations of a monotone map from
// above reach that one fixed point in any order, so psi does not depend on
// the stride, the schedule, the block edge or the order of the marches, bit
// for bit.
//
// The search in single precision starts from a fast estimate, written without
// cancellation: with k admitted values,
//   x = v_1 + (sum_i (v_i - v_1) + sqrt(D)) / k,
//   D = k r^2 - sum_{i<j} (v_i - v_j)^2          (Lagrange's identity),
// whose differences are exact.  Whenever a value is admitted D > r^2 in
// exact arithmetic, so D < tau*k*r^2 (tau < 1/3) only flags rounding trouble;
// the estimate is then taken in double precision.  The estimate is within an
// ulp or two of the result, so the search usually evaluates G_fl twice (at
// the estimate and one ulp away): it gallops outwards from the estimate until
// the result is bracketed, then bisects on the bit patterns (non-negative
// values order like their bits).
// ---------------------------------------------------------------------------
__device__ __forceinline__ double clamp0(double D) { return (ubits(D) >> 63) ? 0.0 : D; }

__device__ __forceinline__ float gsum(float x, float a, float b, float c) {
    const float ta = fmaxf(__fsub_rn(x, a), 0.0f), tb = fmaxf(__fsub_rn(x, b), 0.0f);
    const float tc = fmaxf(__fsub_rn(x, c), 0.0f);
    return __fadd_rn(__fadd_rn(__fmul_rn(ta, ta), __fmul_rn(tb, tb)), __fmul_rn(tc, tc));
}
// (max with 0 by the sign bit: the FP64 pipe of this part is narrow)
__device__ __forceinline__ double gsum(double x, double a, double b, double c) {
    const double ta = clamp0(__dsub_rn(x, a)), tb = clamp0(__dsub_rn(x, b)), tc = clamp0(__dsub_rn(x, c));
    return __dadd_rn(__dadd_rn(__dmul_rn(ta, ta), __dmul_rn(tb, tb)), __dmul_rn(tc, tc));
}

template <typename T>
struct BitsOf;
template <>
struct BitsOf<float> {
    using U = unsigned;
    static constexpr U kInf = 0x7f800000u;
};
template <>
struct BitsOf<double> {
    using U = unsigned long long;
    static constexpr U kInf = 0x7ff0000000000000ull;
};

// The root: with hi the smallest value of precision T above a with
// gsum(hi) >= r2, and lo the value just below it (gsum(lo) < r2), the one of
// the two whose gsum is nearer r2 (lo on a tie of the distances is not taken).
// Near the root G is linear to far below an ulp of x, so this is the root
// rounded to nearest, without the upward drift that always taking hi would
// add at every step along a characteristic.  It stays monotone: lower values
// (b, c, a) raise gsum everywhere, so hi cannot move up, and if it stays put
// the distance r2 - gsum(lo) can only shrink and gsum(hi) - r2 only grow
// (rounded subtraction is monotone), so lo can only become more likely.
// Searched from the estimate x0 (out of line: the estimate is almost always
// within an ulp of the result, which root_near settles in two evaluations).
template <typename T>
__device__ __noinline__ T root_search(T x0, T a, T b, T c, T r2) {
    using U = typename BitsOf<T>::U;
    const U ua = ubits(a);
    U g = ubits(x0);
    if (!(g > ua) || g > BitsOf<T>::kInf) g = ua + 1;
    U lo, hi;                       // gsum(lo) < r2 <= gsum(hi); lo = a needs no evaluation (G(a) = 0)
    T glo, ghi;
    U step = 1;
    T gg = gsum(from_bits(g), a, b, c);
    if (gg >= r2) {
        hi = g;
        ghi = gg;
        for (;;) {
            const U cand = (hi - ua > step) ? hi - step : ua;
            if (cand == ua) {
                lo = ua;
                glo = 0;
                break;
            }
            const T gc = gsum(from_bits(cand), a, b, c);
            if (!(gc >= r2)) {
                lo = cand;
                glo = gc;
                break;
            }
            hi = cand;
            ghi = gc;
            step <<= 1;
        }
    } else {
        lo = g;
        glo = gg;
        for (;;) {
            const U cand = (BitsOf<T>::kInf - lo > step) ? lo + step : BitsOf<T>::kInf;
            const T gc = gsum(from_bits(cand), a, b, c);
            if (cand == BitsOf<T>::kInf || gc >= r2) {
                hi = cand;
                ghi = gc;
                break;
            }
            lo = cand;
            glo = gc;
            step <<= 1;
        }
    }
    while (hi - lo > 1) {
        const U mid = lo + ((hi - lo) >> 1);
        const T gm = gsum(from_bits(mid), a, b, c);
        if (gm >= r2) {
            hi = mid;
            ghi = gm;
        } else {
            lo = mid;
            glo = gm;
        }
    }
    return (r2 - glo < ghi - r2) ? from_bits(lo) : from_bits(hi);
}

// The same root when it lies within an ulp of the estimate x0, which is the
// usual case: G at x0 says on which side of the crossing x0 lies, G one value
// further that way closes the bracket.  Otherwise the general search.
template <typename T>
__device__ __forceinline__ T root_near(T x0, T a, T b, T c, T r2) {
    using U = typename BitsOf<T>::U;
    const U g = ubits(x0);
    if (g > ubits(a) && g < BitsOf<T>::kInf) {
        const T g0 = gsum(x0, a, b, c);
        const bool up = !(g0 >= r2);                 // x0 below the crossing
        const U g1 = up ? g + 1 : g - 1;
        const T x1 = from_bits(g1);
        const T gx1 = gsum(x1, a, b, c);
        if (up == (gx1 >= r2)) {
            const T glo = up ? g0 : gx1, ghi = up ? gx1 : g0;
            return (r2 - glo < ghi - r2) ? (up ? x0 : x1) : (up ? x1 : x0);
        }
    }
    return root_search<T>(x0, a, b, c, r2);
}

__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The estimate (with the causality clamps: in exact arithmetic the root is not
// below the largest admitted value).  (The division by 3 as a product.)
__device__ __forceinline__ double root_estimate(double a, double b, double c, double r) {
    double x = a + r;
    if (!vlt(b, x)) return x;
    const double d = b - a;
    const double r2 = r * r;
    double D = 2.0 * r2 - d * d;
    x = vmax(a + (d + sqrt(clamp0(D))) * 0.5, b);
    if (!vlt(c, x)) return x;
    const double e = c - a, g = c - b;
    D = 3.0 * r2 - (d * d + e * e + g * g);
    return vmax(a + (d + e + sqrt(clamp0(D))) * (1.0 / 3.0), c);
}

__device__ __forceinline__ double upwind_root(double a, double b, double c, double r) {
    return root_near<double>(root_estimate(a, b, c, r), a, b, c, __dmul_rn(r, r));
}

// FP32: sqrt(D) as D * rsqrt(D) (the hardware reciprocal square root, a few
// ulp) and the division by 3 as a product; D >= tau*k*r^2 > 0 on this path
// (the max guards tau = 0).  When (h/F)^2 underflows single precision the whole
// root is taken in double precision and rounded (rounding is monotone too).
__device__ __forceinline__ float sqrt_f32(float D) { return D * rsqrtf(fmaxf(D, FLT_MIN)); }

// (the double-precision paths out of line: they almost never run, and inlined
// they would crowd the instruction cache around the hot solve loop)
static __device__ __noinline__ float root_in_double(float a, float b, float c, float r) {
    return static_cast<float>(upwind_root(a, b, c, r));
}
static __device__ __noinline__ float estimate_in_double(float a, float b, float c, float r) {
    return static_cast<float>(root_estimate(a, b, c, r));
}

__device__ __forceinline__ float upwind_root_f32(float a, float b, float c, float r, float tau, int& fb) {
    const float r2 = __fmul_rn(r, r);
    if (!(r2 >= FLT_MIN)) {
        ++fb;
        return root_in_double(a, b, c, r);
    }
    float x = a + r;
    if (x > b) {
        const float d = b - a;
        float D = 2.0f * r2 - d * d;
        if (!(D >= tau * 2.0f * r2)) {
            ++fb;
            x = estimate_in_double(a, b, c, r);
        } else {
            x = fmaxf(a + (d + sqrt_f32(D)) * 0.5f, b);
            if (x > c) {
                const float e = c - a, g = c - b;
                D = 3.0f * r2 - (d * d + e * e + g * g);
                if (!(D >= tau * 3.0f * r2)) {
                    ++fb;
                    x = estimate_in_double(a, b, c, r);
                } else {
                    x = fmaxf(a + (d + e + sqrt_f32(D)) * (1.0f / 3.0f), c);
                }
            }
        }
    }
    return root_near<float>(x, a, b, c, r2);
}

// Bounds arrive as doubles; a float node value v satisfies v <= b exactly when
// v <= (the largest float <= b), so the FP32 path compares in float (FP64
// throughput on this part is a small fraction of FP32).
template <typename T>
__device__ __forceinline__ T bound_down(double b);
template <>
__device__ __forceinline__ float bound_down<float>(double b) { return __double2float_rd(b); }
template <>
__device__ __forceinline__ double bound_down<double>(double b) { return b; }

// The value of precision T among a double and its single-precision copy
// (prepared once per restart, so that marches do no double arithmetic).
template <typename T>
__device__ __forceinline__ T pick(double d, float f);
template <>
__device__ __forceinline__ float pick<float>(double, float f) { return f; }
template <>
__device__ __forceinline__ double pick<double>(double d, float) { return d; }

// Bulk prefetch of `bytes` (a multiple of 16, 16-byte aligned) of global memory
// into L2, without a destination or a completion to wait for.
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

template <typename T>
__device__ __forceinline__ void load8_cg(const T* g, T* out);
template <>
__device__ __forceinline__ void load8_cg<float>(const float* g, float* out) {
    const float4 a = __ldcg(reinterpret_cast<const float4*>(g));
    const float4 b = __ldcg(reinterpret_cast<const float4*>(g) + 1);
    out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w;
    out[4] = b.x; out[5] = b.y; out[6] = b.z; out[7] = b.w;
}
template <>
__device__ __forceinline__ void load8_cg<double>(const double* g, double* out) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double2 a = __ldcg(reinterpret_cast<const double2*>(g) + i);
        out[2 * i] = a.x;
        out[2 * i + 1] = a.y;
    }
}
template <typename T>
__device__ __forceinline__ void load8_ro(const T* g, T* out);
template <>
__device__ __forceinline__ void load8_ro<float>(const float* g, float* out) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(g));
    const float4 b = __ldg(reinterpret_cast<const float4*>(g) + 1);
    out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w;
    out[4] = b.x; out[5] = b.y; out[6] = b.z; out[7] = b.w;
}
template <>
__device__ __forceinline__ void load8_ro<double>(const double* g, double* out) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double2 a = __ldg(reinterpret_cast<const double2*>(g) + i);
        out[2 * i] = a.x;
        out[2 * i + 1] = a.y;
    }
}
template <typename T>
__device__ __forceinline__ void store8(T* g, const T* v);
template <>
__device__ __forceinline__ void store8<float>(float* g, const float* v) {
    reinterpret_cast<float4*>(g)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(g)[1] = make_float4(v[4], v[5], v[6], v[7]);
}
template <>
__device__ __forceinline__ void store8<double>(double* g, const double* v) {
#pragma unroll
    for (int i = 0; i < 4; ++i) reinterpret_cast<double2*>(g)[i] = make_double2(v[2 * i], v[2 * i + 1]);
}
// Minimum over the warp of values that are >= 0 (+inf allowed): the bits of
// non-negative IEEE numbers order like unsigned integers, so one integer
// reduction (two for FP64: high words, then low words among the lanes holding
// the smallest high word) replaces the five shuffle-and-min steps.  A NaN sits
// above +inf as an integer and loses to any number, as it does in fmin.
__device__ __forceinline__ float warp_min_nn(float v) {
    return __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(v)));
}
__device__ __forceinline__ double warp_min_nn(double v) {
    const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(v));
    const unsigned hi = static_cast<unsigned>(u >> 32), lo = static_cast<unsigned>(u);
    const unsigned mh = __reduce_min_sync(kFull, hi);
    const unsigned ml = __reduce_min_sync(kFull, hi == mh ? lo : 0xffffffffu);
    return __longlong_as_double(static_cast<long long>((static_cast<unsigned long long>(mh) << 32) | ml));
}
template <typename T>
__device__ __forceinline__ T warp_max(T v) {            // (values >= 0)
    if constexpr (sizeof(T) == 4) {
        return from_bits(__reduce_max_sync(kFull, ubits(v)));
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = vmax(v, __shfl_xor_sync(kFull, v, o));
        return v;
    }
}
struct MarchAcc {
    unsigned accepted;                       // per lane
    unsigned band;                           // counted on lane 0
    int fallbacks;                           // per lane
    unsigned updates;                        // per lane
    unsigned solves, rounds;                 // the same on every lane (one restart of one warp)
    float rmin, rmax;                        // the same on every lane
};

// Where a grid sits in the work space of a launch: its bricks are the global
// indices [boff, boff + BX*BY*BZ), its 2x2x2 groups [goff, goff + GX*GY*GZ).
// One grid per launch has boff = goff = 0.
struct Geo {
    int32_t BX, BY, BZ;
    int32_t boff;
    int32_t GX, GY;
    int32_t goff;
    uint32_t lists;            // bit 0: keep the brick work list; bit 1: keep the group work list
    FastDiv div_x, div_xy;     // by BX and BX*BY
};

// Coordinates of a brick (global index) in its grid.
struct BrickAt {
    int x, y, z;
};
__device__ __forceinline__ BrickAt brick_at(const Geo& G, int32_t b) {
    const int bl = b - G.boff;
    const int z = fast_div(bl, G.div_xy), r = bl - z * (G.BX * G.BY), y = fast_div(r, G.div_x);
    return BrickAt{r - y * G.BX, y, z};
}

// Put brick x (global index; and, if the group work list is kept, its group)
// on restart k+1's work lists, once per restart (the "queued" marks dedupe).
template <typename T>
__device__ __forceinline__ void enqueue_next(const LoopParams<T>& P, const Geo& G, int k, int32_t x) {
    const int s = (k + 1) % kRing;
    if (P.pause) {                       // a sharded grid: ghost bricks belong to another GPU
        const int bz = (x - G.boff) / (G.BX * G.BY);
        if (bz < P.own_bz0 || bz >= P.own_bz1) return;
    }
    if ((G.lists & 1u) && atomicMax(P.queued + s * P.nbricks + x, k + 1) < k + 1) {
        const int pos = atomicAdd(&P.ctrl->count[s], 1);
        P.list[s][pos] = x;
    }
    if (!(G.lists & 2u)) return;
    const int xl = x - G.boff;
    const int bx = xl % G.BX, by = (xl / G.BX) % G.BY, bz = xl / (G.BX * G.BY);
    const int32_t g = G.goff + ((bz >> 1) * G.GY + (by >> 1)) * G.GX + (bx >> 1);
    if (atomicMax(P.qgroup + s * P.ngroups + g, k + 1) < k + 1) {
        const int pos = atomicAdd(&P.ctrl->gcount[s], 1);
        P.glist[s][pos] = g;
    }
}

// At the start of restart k: every thread of the launch clears its share of the
// brick list restart k-1 used (ring slot (k-1) mod kRing, `used` entries),
// coalesced.  The slot is next written in restart k+1 (by early marches of
// restart k+2 while waiting at its barrier) at the earliest, after every warp has
// arrived at the barrier of restart k and so has finished its share.
__device__ __forceinline__ void clear_used_slot(int32_t* list, int used) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < used; i += gridDim.x * blockDim.x) list[i] = -1;
}

// Before an early march of brick b at restart k+1: wait until b and each of its
// six neighbours that is on restart k's work list has finished that march
// (bounded; false on timeout).  After it the march reads what it would read
// after the barrier of restart k.
template <typename T>
__device__ bool wait_ready(const LoopParams<T>& P, const Geo& G, int32_t b, int k, int lane) {
    int32_t x = -1;
    if (lane < 7) {
        const BrickAt at = brick_at(G, b);
        const int bx = at.x, by = at.y, bz = at.z;
        if (lane == 6) x = b;
        else if (lane == 0) x = bx > 0 ? b - 1 : -1;
        else if (lane == 1) x = bx < G.BX - 1 ? b + 1 : -1;
        else if (lane == 2) x = by > 0 ? b - G.BX : -1;
        else if (lane == 3) x = by < G.BY - 1 ? b + G.BX : -1;
        else if (lane == 4) x = bz > 0 ? b - G.BX * G.BY : -1;
        else x = bz < G.BZ - 1 ? b + G.BX * G.BY : -1;
    }
    bool need = x >= 0 && __ldcg(P.queued + (k % kRing) * P.nbricks + x) == k;
    unsigned nap = 128;
    for (long long it = 0;; ++it) {
        if (need && ld_acquire(P.done + x) >= k) need = false;
        if (!__any_sync(0xffffffffu, need)) break;
        if (it > P.wait_limit) return false;
        __nanosleep(nap);
        if (nap < 2048) nap <<= 1;
    }
    __syncwarp();
    return true;
}

// State of the restart loop shared by a CTA's warps.  The control block sits in
// a few cache lines of one L2 slice, which serves about one access a clock: with
// every warp of a full launch (3648) reading, polling and adding there on its own,
// each restart spent 10-15 us in those queues (64^3 in 8^3 blocks: 36 us a restart
// with 3648 warps, 25 us with 608).  So one warp per CTA reads it for the others,
// polls the barrier and claims early work, and the CTA arrives once and adds its
// statistics once.
struct CtaLoop {
    // the restart the CTA is in, as its poller read it
    int k;
    int done;
    int mode;                  // block edge
    int n;                     // length of the brick list
    int used, gused;           // lengths of the lists to clear
    int early;                 // early work allowed while waiting at this restart's barrier
    int grow, grow_next;       // bound, next_bound below width_band (pending nodes re-activate the block)
    double bound, bprev, next_bound;
    float bound_f, bprev_f, next_f;    // the same rounded down to single precision
    unsigned gen;              // barrier generation while in this restart
    // its barrier
    unsigned rel;              // generation last seen by the CTA
    unsigned arrived;          // warps that have arrived
    int stop;                  // a wait ran out: leave
    int token;                 // 1: a warp polls for the CTA
    unsigned long long claim;  // entry of a coming restart's list claimed while waiting: restart << 32 | index
    int drained;               // restart whose list a warp found handed out
    MarchAcc acc;              // the CTA's statistics of the restart
};

// What a warp keeps of its restart once it has arrived at the barrier (the CTA's
// state may then become the next restart's), in shared memory: a march needs its
// registers.
struct WarpLoop {
    double bound, bprev, next_bound;
    float bound_f, bprev_f, next_f;
    int grow, grow_next, early;
};
__device__ __forceinline__ void keep_restart(WarpLoop& L, const CtaLoop& S, int lane) {
    if (lane == 0) {
        L.bound = S.bound;
        L.bprev = S.bprev;
        L.next_bound = S.next_bound;
        L.bound_f = S.bound_f;
        L.bprev_f = S.bprev_f;
        L.next_f = S.next_f;
        L.grow = S.grow;
        L.grow_next = S.grow_next;
        L.early = S.early;
    }
    __syncwarp();
}

template <typename V>
__device__ __forceinline__ V vol(const V& x) {
    return *const_cast<const volatile V*>(&x);
}
template <typename V>
__device__ __forceinline__ void vol_set(V& x, V v) {
    *const_cast<volatile V*>(&x) = v;
}

__device__ __forceinline__ void reset_acc(MarchAcc& A) {
    A = MarchAcc{0u, 0u, 0, 0u, 0u, 0u, __int_as_float(0x7f800000), 0.0f};
}

// One warp arrives at the restart barrier: its statistics (A, if any) go to the
// CTA's; the CTA's last warp adds those to the control block and arrives for the
// CTA.  True for the launch's last arrival, which then runs the restart's
// bookkeeping and releases the others.
__device__ __forceinline__ bool barrier_arrive(Ctrl* C, CtaLoop& S, MarchAcc& A, bool any, int lane) {
    if (any) {
        unsigned* from = reinterpret_cast<unsigned*>(&A);
        unsigned* to = reinterpret_cast<unsigned*>(&S.acc);
        if (lane < 6) atomicAdd(to + lane, from[lane]);
        if (lane == 6) atomicMin(to + 6, from[6]);       // (bits of values >= 0)
        if (lane == 7) atomicMax(to + 7, from[7]);
        __syncwarp();
        if (lane == 0) reset_acc(A);
    }
    __syncwarp();
    int last = 0;
    if (lane == 0) {
        __threadfence();
        last = atomicAdd(&S.arrived, 1u) == (blockDim.x >> 5) - 1;
        if (last) __threadfence();
    }
    if (!__shfl_sync(kFull, last, 0)) return false;
    {
        const unsigned v = lane < 8 ? reinterpret_cast<unsigned*>(&S.acc)[lane] : 0u;
        if (lane < 6 && v != 0u) atomicAdd(&C->r_accepted + lane, static_cast<unsigned long long>(v));
        if (lane == 6) atomicMin(&C->r_rmin_bits, v);
        if (lane == 7) atomicMax(&C->r_rmax_bits, v);
        __syncwarp();
        if (lane == 0) reset_acc(S.acc);
    }
    __syncwarp();
    last = 0;
    if (lane == 0) {
        S.arrived = 0u;                       // (no warp arrives again before this barrier is passed)
        __threadfence();
        last = atomicAdd(&C->bar_count, 1u) == gridDim.x - 1;
        if (last) __threadfence();
    }
    return __shfl_sync(kFull, last, 0) != 0;
}
__device__ __forceinline__ void barrier_release(Ctrl* C, int lane, unsigned gen) {
    __syncwarp();
    if (lane == 0) {
        C->bar_count = 0;
        __threadfence();
        st_release(&C->bar_gen, gen + 1);
    }
}

// A warp that gives up on a wait: the status bit, made visible to every other
// warp of the launch before the warp leaves.
__device__ __forceinline__ void give_up(Ctrl* C, int lane) {
    if (lane == 0) {
        atomicOr(&C->status, kStWaitTimeout);
        __threadfence();
    }
    __syncwarp();
}

// Start of CTA-wide work (16^3 blocks) in a restart: whether the whole CTA may
// go on.  A warp that gives up on a wait (give_up) exits on its own, and an
// exiting thread releases a CTA barrier that waits only for it (the exit rule
// of PTX), so this vote completes whichever warps are still there.  Every
// thread of the CTA gets the same answer: false if a warp is missing, if a
// warp of the CTA brings ok = false, or if any wait of the launch has run out.
// The CTA then leaves as a whole, before its first CTA-wide march, and no
// thread is ever left waiting at a CTA barrier for a warp that has gone.
// s_arrived is a shared counter that starts at zero (and is zero again after).
__device__ __forceinline__ bool cta_go(const Ctrl* C, bool ok, int lane, int* s_arrived) {
    if (lane == 0) atomicAdd(s_arrived, 1);
    const int stop = __syncthreads_or((!ok || (__ldcg(&C->status) & kStWaitTimeout)) ? 1 : 0);
    const bool all = *reinterpret_cast<volatile int*>(s_arrived) == static_cast<int>(blockDim.x >> 5);
    __syncthreads();
    if (threadIdx.x == 0) *s_arrived = 0;
    return stop == 0 && all;
}

// A grid barrier inside a restart (no bookkeeping), by every warp of the launch:
// the CTA's first thread arrives and waits for all.  False if this or another
// wait ran out, or the first warp has left.
__device__ inline bool grid_sync(Ctrl* C, long long limit) {
    __threadfence();
    __syncthreads();
    int ok = 0;
    if (threadIdx.x == 0) {
        const unsigned gen = ld_acquire(&C->sync_gen);
        __threadfence();
        if (atomicAdd(&C->sync_count, 1u) == gridDim.x - 1) {
            C->sync_count = 0;
            __threadfence();
            st_release(&C->sync_gen, gen + 1);
            ok = 1;
        } else {
            unsigned nap = 32;
            for (long long it = 0;; ++it) {
                if (ld_acquire(&C->sync_gen) != gen) {
                    ok = 1;
                    break;
                }
                if (__ldcg(&C->status) & kStWaitTimeout) break;
                if (it > limit) {
                    atomicOr(&C->status, kStWaitTimeout);
                    __threadfence();
                    break;
                }
                __nanosleep(nap);
                if (nap < 1024) nap <<= 1;
            }
        }
    }
    return __syncthreads_or(ok) != 0;
}

// Waiting at the barrier of restart k.  One warp of the CTA at a time holds the
// token: it polls the grid barrier and, if early work is allowed, claims the next
// entry of restart k+1's list (one index at a time, kept in S.claim until the list
// holds it; a claim still open at the release is settled in restart k+1).  The
// others watch shared memory.  Returns 1: released (the CTA's state is the next
// restart's; load(), run by one lane, reads it), 2: leave, 3: *b is a brick of
// restart k+1 to march early.  Every wait is bounded.
template <typename T, typename Load>
__device__ int wait_or_work(const LoopParams<T>& P, CtaLoop& S, int k, unsigned gen, bool early, int lane, int32_t* b,
                            Load load) {
    Ctrl* C = P.ctrl;
    const int s1 = (k + 1) % kRing;
    int st = 0;
    int32_t x = -1;
    if (lane == 0) {
        unsigned nap = 64;
        for (long long it = 0;; ++it) {
            if (vol(S.stop)) st = 2;
            else if (vol(S.rel) != gen) st = 1;
            else if (vol(S.token) == 0 && atomicCAS(&S.token, 0, 1) == 0) st = 3;
            else if (it > kWatchPolls * P.wait_limit) st = 4;
            if (st) break;
            __nanosleep(nap);
            if (nap < kWatchNap) nap <<= 1;
        }
        if (st == 3) {
            nap = 32;
            for (long long it = 0;; ++it) {
                if (vol(S.rel) != gen) {
                    st = 1;
                    break;
                }
                if (ld_acquire(&C->bar_gen) != gen) {
                    load();
                    __threadfence_block();
                    vol_set(S.rel, gen + 1);
                    st = 1;
                    break;
                }
                if (__ldcg(&C->status) & kStWaitTimeout) {
                    vol_set(S.stop, 1);
                    st = 2;
                    break;
                }
                if (early) {
                    const unsigned long long mine = static_cast<unsigned long long>(k + 1) << 32;
                    const unsigned long long open = vol(S.claim);
                    const int c = (open >> 32) == (mine >> 32) ? static_cast<int>(open) : atomicAdd(&C->head[s1], 1);
                    const bool have = c < __ldcg(&C->count[s1]);
                    vol_set(S.claim, have ? 0ull : mine | static_cast<unsigned>(c));
                    if (have) {
                        // (the enqueuer bumps the count, then stores the entry)
                        x = ld_acquire(P.list[s1] + c);
                        for (long long w = 0; x < 0 && w < P.wait_limit; ++w) {
                            __nanosleep(32);
                            x = ld_acquire(P.list[s1] + c);
                        }
                        if (x < 0) st = 4;
                        break;
                    }
                }
                if (it > kBarrierPolls * P.wait_limit) {
                    st = 4;
                    break;
                }
                __nanosleep(nap);
                if (nap < kBarrierNap) nap <<= 1;
            }
            __threadfence_block();
            atomicExch(&S.token, 0);
        }
        if (st == 4) vol_set(S.stop, 1);
    }
    st = __shfl_sync(kFull, st, 0);
    *b = __shfl_sync(kFull, x, 0);
    if (st == 4) {
        give_up(C, lane);
        return 2;
    }
    return st;
}

// The same for a CTA that marches 16^3 blocks, as a whole: its first thread polls,
// claims (open claim: S.claim) and waits until the group and each of its six
// neighbours on restart k's list have finished that march.  1: released, 2:
// leave, 3: *g is a group of restart k+1.
template <typename T, typename Load>
__device__ int wait_or_group(const LoopParams<T>& P, CtaLoop& S, int k, unsigned gen, int* s_answer, int* g, Load load) {
    Ctrl* C = P.ctrl;
    const int s = k % kRing, s1 = (k + 1) % kRing;
    if (threadIdx.x == 0) {
        int st = 0;
        int32_t x = -1;
        unsigned nap = 32;
        for (long long it = 0; st == 0; ++it) {
            if (ld_acquire(&C->bar_gen) != gen) {
                load();
                S.rel = gen + 1;
                st = 1;
                break;
            }
            if (__ldcg(&C->status) & kStWaitTimeout) {
                st = 2;
                break;
            }
            const unsigned long long mine = static_cast<unsigned long long>(k + 1) << 32;
            const int c = (S.claim >> 32) == (mine >> 32) ? static_cast<int>(S.claim) : atomicAdd(&C->ghead[s1], 1);
            const bool have = c < __ldcg(&C->gcount[s1]);
            S.claim = have ? 0ull : mine | static_cast<unsigned>(c);
            if (have) {
                st = 3;
                x = ld_acquire(P.glist[s1] + c);
                for (long long w = 0; x < 0 && w < P.wait_limit; ++w) {
                    __nanosleep(32);
                    x = ld_acquire(P.glist[s1] + c);
                }
                const int gx = x % P.GX, gy = (x / P.GX) % P.GY, gz = x / (P.GX * P.GY);
                const int32_t near[7] = {x, gx > 0 ? x - 1 : -1, gx < P.GX - 1 ? x + 1 : -1, gy > 0 ? x - P.GX : -1,
                                         gy < P.GY - 1 ? x + P.GX : -1, gz > 0 ? x - P.GX * P.GY : -1,
                                         gz < P.GZ - 1 ? x + P.GX * P.GY : -1};
                const long long most = kBarrierPolls * P.wait_limit;
                long long w = x < 0 ? most + 1 : 0;
                for (int j = 0; j < 7 && w <= most; ++j) {
                    if (near[j] < 0 || __ldcg(P.qgroup + static_cast<int64_t>(s) * P.ngroups + near[j]) != k) continue;
                    unsigned d = 64;
                    for (w = 0; ld_acquire(P.gdone + near[j]) < k && w <= most; ++w) {
                        __nanosleep(d);
                        if (d < kBarrierNap) d <<= 1;
                    }
                }
                if (w > most) st = 4;
                break;
            }
            if (it > kBarrierPolls * P.wait_limit) st = 4;
            __nanosleep(nap);
            if (nap < kBarrierNap) nap <<= 1;
        }
        if (st == 4) {
            atomicOr(&C->status, kStWaitTimeout);
            __threadfence();
            st = 2;
        }
        s_answer[0] = st;
        s_answer[1] = x;
    }
    __syncthreads();
    const int st = s_answer[0];
    *g = s_answer[1];
    __syncthreads();                           // (read before the first thread answers again)
    return st;
}

// The next entry of restart k's brick list (ring slot s, S.n entries) for this
// warp, -1 when all are handed out.  `first`: the warp's first call in the
// restart, which settles the claim the CTA left open while waiting.
__device__ __forceinline__ int next_entry(Ctrl* C, CtaLoop& S, int k, int s, bool first, int lane) {
    int i = -1;
    if (lane == 0) {
        if (first) {
            const unsigned long long open = vol(S.claim);
            if (static_cast<int>(open >> 32) == k && atomicCAS(&S.claim, open, 0ull) == open) i = static_cast<int>(open);
        }
        if (i < 0 && vol(S.drained) != k) i = atomicAdd(&C->head[s], 1);
        if (i >= S.n) i = -1;
        if (i < 0) vol_set(S.drained, k);
    }
    return __shfl_sync(kFull, i, 0);
}

}  // namespace eikg
