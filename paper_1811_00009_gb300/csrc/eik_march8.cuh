// March_Narrow_Band (Alg. 4 with Algs. 2, 3 and the ghost exchange of Alg. 5)
// of one 8x8x8 block (a "brick") by one warp.
//
// The brick's psi with its ghost layer and its h/F sit in shared memory in the
// same 10^3 halo layout.  A tentative value (BAND) carries its sign bit set;
// h/F carries its sign bit set while the node must not be queued: always for
// fixed, barrier, padding and ghost nodes (-inf), and for a node that waits in
// the queue.
//
// Stages (Alg. 4): with m the smallest tentative value, everything up to
// thr = min(m + w, bound) is settled before the next stage, w = omega *
// min(h/F) over the brick.  A stage starts by queueing the tentative nodes up
// to thr and the nodes next to such ghosts; then the warp takes 32 queued nodes
// at a time, solves them (Alg. 3) from the accepted neighbours, and a node that
// is now accepted (lowered, or tentative until now, and not above thr) queues
// those of its neighbours that lie above it (Alg. 2: no other can be lowered by
// it).  A node lowered to a value above thr stays tentative for a later stage.
// Every lowered value is passed on, so a march ends in the same state in any
// order (the root is monotone, see eik_march.cuh).
//
// What bounds it: issue slots (shared-memory loads, the root's arithmetic) and,
// on small grids, the chain of dependent steps of one march after another;
// DRAM stays below a tenth of its bandwidth.  The rounds this replaces (accept
// a window, mark all neighbours of the accepted nodes with shifted bit vectors,
// re-solve all of them) solved 506 nodes a march, and 11.2 marches a brick, where
// this solves 383 in 9.6 (1024^3, GRF speeds, stride 1.5h): four in ten of those
// neighbours lay below the accepted node and could not change.  The 383 take 14.3
// passes of 32, five in six of the lanes filled.
#pragma once

#include "eik_root64.cuh"

namespace eikg {

constexpr int kQueue = 512;            // a brick node is in the queue at most once

template <typename T>
struct __align__(16) QueueSmem {
    T psi[1000];                       // index ((z+1)*10 + (y+1))*10 + (x+1); tentative values negative
    T rq[1000];                        // h/F, same index; negative: not to be queued
    uint16_t queue[kQueue];            // ring of halo indices
};

// Bit patterns as signed integers: tentative values (sign set) lie below all
// others and, among themselves, order as their magnitudes.
__device__ __forceinline__ int sbits(float v) { return __float_as_int(v); }
__device__ __forceinline__ long long sbits(double v) { return __double_as_longlong(v); }
template <typename T>
struct SBitsOf;
template <>
struct SBitsOf<float> {
    using S = int;
    static constexpr int kMax = 0x7fffffff;
};
template <>
struct SBitsOf<double> {
    using S = long long;
    static constexpr long long kMax = 0x7fffffffffffffffLL;
};

// A value at the start of a march: tentative (negative) if finite and above the
// previous bound (-1 before the first restart; patterns as signed integers order
// so, and keep the double-precision case off the FP64 pipe).
template <typename T>
__device__ __forceinline__ T band_value(T v, T bprev) {
    return vlt(v, Num<T>::inf()) && sbits(v) > sbits(bprev) ? vneg(v) : v;
}

// 32-bit accesses to the words that hold the signs of shared values.
__device__ __forceinline__ int ld_word(uint32_t a) {
    int v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void st_word(uint32_t a, int v) {
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
// Shared address of the word that holds a value's sign (little-endian).
template <typename T>
__device__ __forceinline__ uint32_t sign_word(const T* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p)) + static_cast<uint32_t>(sizeof(T) - 4);
}

// The ghost positions of h/F are never queued (set once; marches write only the
// brick's own positions).
template <typename T>
__device__ __forceinline__ void init_queue_smem(QueueSmem<T>& S, int lane) {
    const T INF = Num<T>::inf();
    for (int i = lane; i < 1000; i += 32) S.rq[i] = -INF;
    __syncwarp();
}

// Smaller of the accepted values among two neighbours along an axis (+inf if
// neither is accepted): as unsigned bit patterns tentative values lie above +inf.
__device__ __forceinline__ float axis_min(float p, float q) {
    return from_bits(__vimin3_u32(ubits(p), ubits(q), 0x7f800000u));
}
__device__ __forceinline__ double axis_min(double p, double q) {
    const unsigned long long a = ubits(p), b = ubits(q), m = a < b ? a : b;
    return from_bits(m < 0x7ff0000000000000ull ? m : 0x7ff0000000000000ull);
}

// a <= b <= c of three values >= 0 (+inf allowed), on the bit patterns: the
// middle one is what the exclusive or of all three leaves.
__device__ __forceinline__ void sort3(float x, float y, float z, float& a, float& b, float& c) {
    const unsigned u = ubits(x), v = ubits(y), w = ubits(z);
    const unsigned lo = __vimin3_u32(u, v, w), hi = __vimax3_u32(u, v, w);
    a = from_bits(lo);
    c = from_bits(hi);
    b = from_bits(u ^ v ^ w ^ lo ^ hi);
}
__device__ __forceinline__ void sort3(double x, double y, double z, double& a, double& b, double& c) {
    const double lo = vmin(x, y), hi = vmax(x, y), t = vmax(lo, z);
    a = vmin(lo, z);
    b = vmin(hi, t);
    c = vmax(hi, t);
}

// The rare cases of the single-precision root (estimate more than an ulp off,
// (h/F)^2 below the normal range, estimate in double precision): out of line.
// Returned with the count of roots taken in double (by value: a reference would
// keep the march's counters in local memory).
struct RareRoot {
    float x;
    int fb;
};
static __device__ __noinline__ RareRoot root_rare(float a, float b, float c, float r, float tau) {
    RareRoot o{0.0f, 0};
    o.x = upwind_root_f32(a, b, c, r, tau, o.fb);
    return o;
}

// Alg. 3 in single precision for a <= b <= c (see upwind_root_f32, whose result
// this returns): the estimate without branches.  b is admitted when (b - a)^2 <
// r^2, c when (c - a)^2 + (c - b)^2 < r^2, and
//   D = r^2 + max(r^2 - (b-a)^2, 0) + max(r^2 - (c-a)^2 - (c-b)^2, 0)
// is the discriminant of every case.  The estimate only starts the search, so
// it may use fused operations and the approximate reciprocal square root.  (D >= r^2
// but for rounding: below tau = 1/3 an estimate that needs double precision is among
// those that miss the root, which go out of line.)
__device__ __forceinline__ float root_fast(float a, float b, float c, float r, bool live, float tau, int& fb) {
    const float r2 = __fmul_rn(r, r);
    const float d = b - a, e = c - a, g = c - b;
    const float q1 = __fmaf_rn(-d, d, r2), q2 = r2 - __fmaf_rn(g, g, e * e);
    const bool p1 = q1 > 0.0f, p2 = q2 > 0.0f;
    const float D = r2 + fmaxf(q1, 0.0f) + fmaxf(q2, 0.0f);
    float s = p1 ? d : 0.0f;
    s = p2 ? s + e : s;
    const float inv = p2 ? (1.0f / 3.0f) : (p1 ? 0.5f : 1.0f);
    const float x0 = __fmaf_rn(__fmaf_rn(D, rsqrt_approx(D), s), inv, a);
    const float g0 = gsum(x0, a, b, c);
    const bool up = !(g0 >= r2);                     // x0 below the crossing
    const float x1 = from_bits(ubits(x0) + (up ? 1u : 0xffffffffu));
    const float g1 = gsum(x1, a, b, c);
    const float d0 = fabsf(r2 - g0), d1 = fabsf(g1 - r2);
    const bool first = up ? d0 < d1 : d0 <= d1;     // the nearer of the two; a tie takes the upper one
    float x = first ? x0 : x1;
    const bool rare = up != (g1 >= r2) || !(x0 > a) || !(r2 >= FLT_MIN) || (tau > 0.33f && p1);
    if (live && rare) {
        const RareRoot o = root_rare(a, b, c, r, tau);
        x = o.x;
        fb += o.fb;
    }
    return x;
}

template <typename T>
struct QueueRoot;
template <>
struct QueueRoot<float> {
    static __device__ __forceinline__ float go(float a, float b, float c, float r, bool live, float tau, int& fb) {
        return root_fast(a, b, c, r, live, tau, fb);
    }
};
template <>
struct QueueRoot<double> {
    static __device__ __forceinline__ double go(double a, double b, double c, double r, bool live, float, int&) {
        return root_fast(a, b, c, r, live);
    }
};

// (A: the warp's statistics, in shared memory: the march needs its registers)
template <typename T>
__device__ void march8(const LoopParams<T>& P, const Geo& G, QueueSmem<T>& S, MarchAcc& A, int32_t b, int k, T bprev,
                       T bound, bool grow, T window, int lane, bool publish, int32_t pf = -1) {
    using SB = typename SBitsOf<T>::S;
    const T INF = Num<T>::inf();
    const int y = lane & 7, zp = lane >> 3, z0 = 2 * zp;
    const int BX = G.BX, BY = G.BY, BZ = G.BZ;
    const BrickAt at_b = brick_at(G, b);
    const int bx = at_b.x, by = at_b.y, bz = at_b.z;
    const int pbase = (z0 * 8 + y) * 8;                          // brick index of (0, y, z0)
    const int hbase = ((z0 + 1) * 10 + (y + 1)) * 10 + 1;       // halo index of (0, y, z0)
    const unsigned lt = (1u << lane) - 1u;
    // this lane's ghost nodes: face-local u = lane and lane + 32 of every face (x
    // faces: u = z*8 + y, y faces: z*8 + x, z faces: y*8 + x); halo index of u =
    // lane on the faces' low ghost layers, and the step from u to u + 32
    const int gx = (zp + 1) * 100 + (y + 1) * 10, gy = (zp + 1) * 100 + (y + 1), gz = (zp + 1) * 10 + (y + 1);
    auto ghost = [&](int f, int e) { return (f < 2 ? gx + 9 * f : f < 4 ? gy + 90 * (f - 2) : gz + 900 * (f - 4)) +
                                            (f < 4 ? 400 : 40) * e; };
    auto inner = [&](int f, int e) { return ghost(f, e) + (f < 2 ? 1 : f < 4 ? 10 : 100) * ((f & 1) ? -1 : 1); };

    // ---- load phase 1 (independent loads): the stamps -- lane f < 6 that of the
    // neighbour across face f, lane 6 the brick's own, lane 7 that of a brick
    // further down this restart's list (pf >= 0), whose h/F and latest copy are
    // prefetched into L2 below -- and h/F of this lane's two rows
    int32_t mine = -1;
    {
        const int ax = lane >> 1, step = ax == 0 ? 1 : (ax == 1 ? BX : BX * BY);
        const int at = ax == 0 ? bx : (ax == 1 ? by : bz), end = ax == 0 ? BX : (ax == 1 ? BY : BZ);
        if (lane < 6) mine = (lane & 1) ? (at < end - 1 ? b + step : -1) : (at > 0 ? b - step : -1);
        if (lane == 6) mine = b;
        if (lane == 7) mine = pf;
    }
    const unsigned long long ms = mine >= 0 ? __ldcg(P.stamp + mine) : kUntouched;
    using UB = typename BitsOf<T>::U;
    UB rlo = BitsOf<T>::kInf;                                   // patterns: -inf lies above +inf unsigned ...
    SB rhi = 0;                                                  // ... and below 0 signed
    {
        T r8[8];
        const T* rs = P.rr + static_cast<int64_t>(b) * kBrick;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            load8_ro(rs + pbase + 64 * s, r8);
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                S.rq[hbase + 100 * s + x] = r8[x];
                rlo = min(rlo, ubits(r8[x]));
                rhi = max(rhi, sbits(r8[x]));
            }
        }
    }
    // ---- load phase 2: the brick's latest copy, and the ghost layer: the
    // neighbours' faces as of the end of restart k-1 with their Upsilon masks
    // (Alg. 5).  A neighbour that already marched in this restart is read from its
    // other copy.  Lane f works out which copy of its neighbour that is.
    int32_t copy = -1;                        // index of the copy in P.slot (lane 6: the brick's latest; -1: none)
    unsigned long long mups = 0ull;
    if (ms != kUntouched) {
        const bool ahead = lane < 6 && stamp_latest(ms) >= k;
        const int written = ahead ? stamp_other(ms) : stamp_latest(ms);
        if (!ahead || written != static_cast<int>(kNever)) copy = 2 * mine + (stamp_copy(ms) ^ (ahead ? 1 : 0));
        if (lane < 6 && copy >= 0 && written == k - 1) mups = __ldcg(P.ups + static_cast<int64_t>(copy) * 6 + (lane ^ 1));
    }
    const int32_t own = __shfl_sync(kFull, copy, 6);
    T row[16];
    if (own < 0) {
#pragma unroll
        for (int x = 0; x < 16; ++x) row[x] = INF;
    } else {
        const T* src = P.slot + static_cast<int64_t>(own) * kSlot;
        load8_cg(src + pbase, row);
        load8_cg(src + pbase + 64, row + 8);
    }
    T fv[6][2];
#pragma unroll
    for (int f = 0; f < 6; ++f) {
        const int32_t cf = __shfl_sync(kFull, copy, f);
        fv[f][0] = INF;
        fv[f][1] = INF;
        if (cf >= 0) {
            const T* src = P.slot + static_cast<int64_t>(cf) * kSlot;
            int off, step = 32;
            if (f == 0) off = kXF7 + lane;
            else if (f == 1) off = kXF0 + lane;
            else if (f == 2) off = (zp * 8 + 7) * 8 + y, step = 256;
            else if (f == 3) off = zp * 64 + y, step = 256;
            else if (f == 4) off = 7 * 64 + lane;
            else off = lane;
            fv[f][0] = __ldcg(src + off);
            fv[f][1] = __ldcg(src + off + step);
        }
    }
    if (lane == 7 && pf >= 0) {
        prefetch_l2(P.rr + static_cast<int64_t>(pf) * kBrick, kBrick * sizeof(T));
        if (copy >= 0) prefetch_l2(P.slot + static_cast<int64_t>(copy) * kSlot, kSlot * sizeof(T));
    }
    // ---- the band at the start of the march: the brick's finite nodes above the
    // previous bound, and the ghost nodes that are above it or that the neighbour
    // lowered in restart k-1 (Upsilon) -- the heap contents of Alg. 4 after Alg. 5.
    // Ghost nodes up to the bound are accepted at once, whatever their order: what
    // they reach is solved in the first stage and waits for its own stage then.
    SB smin = SBitsOf<T>::kMax;
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const T v = row[8 * s + x];
            const T t = band_value(v, bprev);
            S.psi[hbase + 100 * s + x] = t;
            smin = min(smin, sbits(t));
        }
    unsigned fire = 0;                        // this lane's accepted ghost nodes: bit 2f + e
#pragma unroll
    for (int f = 0; f < 6; ++f)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const T v = fv[f][e];
            const unsigned um = __shfl_sync(kFull, static_cast<unsigned>(mups >> (32 * e)), f);
            const bool tent = vlt(v, INF) && (((um >> lane) & 1u) || sbits(v) > sbits(bprev));
            const bool take = tent && sbits(v) <= sbits(bound);
            S.psi[ghost(f, e)] = tent && !take ? vneg(v) : v;
            if (take) smin = min(smin, sbits(vneg(v)));
            fire |= (take ? 1u : 0u) << (2 * f + e);
        }
    unsigned n_acc = __popc(fire), n_upd = 0u, n_solve = 0u;   // accepted, lowered (per lane), solved (every lane)
    int n_fb = 0;                                              // roots taken in double (per lane)
    __syncwarp();
    // the nodes next to the accepted ghost nodes that lie above them (face-local
    // bit masks by votes; each lane picks its rows')
    unsigned C = 0;
#pragma unroll
    for (int f = 0; f < 6; ++f) {
        unsigned m[2];
#pragma unroll
        for (int e = 0; e < 2; ++e)
            m[e] = __ballot_sync(kFull, ((fire >> (2 * f + e)) & 1u) && vlt(fv[f][e], vabs(S.psi[inner(f, e)])));
        if (f < 2) {
            const unsigned v = (zp < 2 ? m[0] : m[1]) >> (((z0 & 3) << 3) + y);
            C |= (v & 0x101u) << (f ? 7 : 0);
        } else if (f < 4) {
            const unsigned v = (zp < 2 ? m[0] : m[1]) >> ((z0 & 3) << 3);
            if (y == (f == 2 ? 0 : 7)) C |= v & 0xFFFFu;
        } else {
            const unsigned v = ((y < 4 ? m[0] : m[1]) >> ((y & 3) << 3)) & 0xFFu;
            if (zp == (f == 4 ? 0 : 3)) C |= f == 4 ? v : v << 8;
        }
    }
    // (the warp's smallest tentative value, +inf if there is none)
    auto warp_min_tent = [&](SB s) -> T {
        return warp_min_nn(s < 0 ? vabs(from_bits(static_cast<typename BitsOf<T>::U>(s))) : INF);
    };
    T mn = warp_min_tent(smin);
    const T rmin_b = warp_min_nn(from_bits(rlo));
    const T rmax_b = warp_max(from_bits(static_cast<UB>(rhi)));
    if (lane == 0) {
        A.rmin = fminf(A.rmin, static_cast<float>(rmin_b));
        A.rmax = fmaxf(A.rmax, static_cast<float>(rmax_b));
    }
    // a stage spans one and a half windows: fewer stages, and hardly more solves
    const T w = static_cast<T>(1.5f) * window * rmin_b;

    int stages = 0;
    for (;;) {
        if (!(mn < INF) || !(mn <= bound)) break;   // band empty, or its minimum above the bound
        if (++stages > kRoundCap) {
            if (lane == 0) atomicOr(&P.ctrl->status, kStRoundCap);
            break;
        }
        const T thr = vmin(mn + w, bound);
        const SB tk = sbits(vneg(thr));
        // ---- tentative nodes up to thr, and the smallest above it
        SB km = SBitsOf<T>::kMax;
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const SB v = sbits(S.psi[hbase + 100 * s + x]);
                if (v <= tk) C |= 1u << (8 * s + x);
                else km = min(km, v);
            }
        // ---- one list of them all -> the (empty) queue
        int head = 0, tail;
        {
            const int cnt = __popc(C);
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            tail = __shfl_sync(kFull, incl, 31);
            uint16_t* at = S.queue + (incl - cnt);
            const uint32_t rw = sign_word(S.rq + hbase);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const int h = (j >> 3) * 100 + (j & 7);
                const bool in = (C >> j) & 1u;
                const int w0 = ld_word(rw + h * static_cast<int>(sizeof(T)));
                if (in) *at = static_cast<uint16_t>(hbase + h);
                if (in) st_word(rw + h * static_cast<int>(sizeof(T)), w0 | static_cast<int>(0x80000000u));
                at += in ? 1 : 0;
            }
            C = 0;
        }
        __syncwarp();
        // ---- the queue, 32 nodes at a time (reads before writes)
        smin = km;
        while (head < tail) {
            const bool val = head + lane < tail;
            const int n = min(32, tail - head);
            const int hq = val ? S.queue[(head + lane) & (kQueue - 1)] : hbase;
            head += n;
            n_solve += n;
            T* ps = S.psi + hq;
            const T r = vneg(S.rq[hq]);
            const bool live = val && vlt(r, INF);                // (a fixed node only passes its value on)
            const T cur = ps[0], c = vabs(cur);
            const T nv[6] = {ps[-1], ps[1], ps[-10], ps[10], ps[-100], ps[100]};
            if (live) S.rq[hq] = r;                               // may be queued again
            const T mx = axis_min(nv[0], nv[1]), my = axis_min(nv[2], nv[3]), mz = axis_min(nv[4], nv[5]);
            // psi_1 <= psi_2 <= psi_3
            T a0, a1, a2;
            sort3(mx, my, mz, a0, a1, a2);
            const bool go = live && vlt(a0, INF);
            const T xn = QueueRoot<T>::go(a0, a1, a2, r, go, P.tau_f, n_fb);
            const bool imp = go && vlt(xn, c);
            const T v = imp ? xn : c;
            const bool prop = val && (imp || sgn(cur)) && !vlt(thr, v);
            __syncwarp();
            if (imp || prop) ps[0] = prop ? v : vneg(v);
            if (imp && !prop) smin = min(smin, sbits(vneg(v)));
            n_upd += imp ? 1u : 0u;
            n_acc += prop ? 1u : 0u;
            // queue the neighbours above the accepted value, each once: every lane
            // writes its mark on those not queued yet, and the mark that stays wins
            // (two lanes may reach the same neighbour; shared-memory atomics would
            // take 50-60 cycles each, 300 for the six).  The mark is a NaN pattern, so
            // no h/F equals it.
            constexpr int off[6] = {-1, 1, -10, 10, -100, 100};
            const int mark = (sizeof(T) == 4 ? static_cast<int>(0xFFC00000u) : static_cast<int>(0xFFF80000u)) | lane;
            const uint32_t rw = sign_word(S.rq + hq);
            int nw[6];
            bool win[6];
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                nw[d] = ld_word(rw + off[d] * static_cast<int>(sizeof(T)));
                win[d] = prop && vlt(v, vabs(nv[d])) && nw[d] >= 0;
            }
#pragma unroll
            for (int d = 0; d < 6; ++d)
                if (win[d]) st_word(rw + off[d] * static_cast<int>(sizeof(T)), mark);
            __syncwarp();
            unsigned cnt = 0;
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                win[d] = win[d] && ld_word(rw + off[d] * static_cast<int>(sizeof(T))) == mark;
                cnt += win[d] ? 1u : 0u;
            }
            // positions by a prefix sum of the lanes' counts (their three bits by votes)
            const unsigned c0 = __ballot_sync(kFull, cnt & 1u), c1 = __ballot_sync(kFull, cnt & 2u);
            const unsigned c2 = __ballot_sync(kFull, cnt & 4u);
            int at = tail + __popc(c0 & lt) + 2 * __popc(c1 & lt) + 4 * __popc(c2 & lt);
            tail += __popc(c0) + 2 * __popc(c1) + 4 * __popc(c2);
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                if (win[d]) S.queue[at & (kQueue - 1)] = static_cast<uint16_t>(hq + off[d]);
                if (win[d]) st_word(rw + off[d] * static_cast<int>(sizeof(T)), nw[d] | static_cast<int>(0x80000000u));
                at += win[d] ? 1 : 0;
            }
            __syncwarp();
        }
        mn = warp_min_tent(smin);
    }
    // ---- the face nodes of the copy the march started from, read again for the
    // comparison below (an L2 hit; keeping them would cost registers)
    n_upd = __reduce_add_sync(kFull, n_upd);
    T old[6][2];
#pragma unroll
    for (int f = 0; f < 6; ++f)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int u = lane + 32 * e;
            const int o = f == 0 ? kXF0 + u : f == 1 ? kXF7 + u : f == 2 ? (u >> 3) * 64 + (u & 7)
                          : f == 3 ? (u >> 3) * 64 + 56 + (u & 7) : f == 4 ? u : 7 * 64 + u;
            old[f][e] = INF;
            if (n_upd != 0u && own >= 0) old[f][e] = __ldcg(P.slot + static_cast<int64_t>(own) * kSlot + o);
        }
    // ---- the brick's values, and its tentative nodes
    T out[16];
    unsigned nt = 0;
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const T t = S.psi[hbase + 100 * s + x];
            nt += sgn(t) ? 1u : 0u;
            out[8 * s + x] = vabs(t);
        }
    n_acc = __reduce_add_sync(kFull, n_acc);
    n_fb = __reduce_add_sync(kFull, n_fb);
    // ---- Upsilon, per face: the nodes lowered in this march that lie below the neighbour's node beyond the face -- no other can lower
    // anything there, so it neither activates the neighbour nor enters its band.
    // Likewise a tentative ghost node counts as pending only if it lies below the
    // brick's own node.  (Without the two tests one march in five lowered nothing:
    // 11.1 marches a brick against 9.4, GRF speeds, 1.5h.)
    unsigned ulo = 0u, uhi = 0u;              // lane f < 6: face f's mask (face-local bits)
#pragma unroll
    for (int f = 0; f < 6; ++f) {
        unsigned m[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const T g = S.psi[ghost(f, e)], v = vabs(S.psi[inner(f, e)]);
            nt += sgn(g) && vlt(vabs(g), v) ? 1u : 0u;
            m[e] = __ballot_sync(kFull, n_upd != 0u && vlt(v, old[f][e]) && vlt(v, vabs(g)));
        }
        if (lane == f) ulo = m[0], uhi = m[1];
    }
    const unsigned n = __reduce_add_sync(kFull, nt);
    if (lane == 0) {
        A.accepted += n_acc;
        A.band += n;
        A.fallbacks += n_fb;
        A.updates += n_upd;
        A.solves += n_solve;
        A.rounds += stages;
    }
    // A march that lowered no value leaves the brick as its latest copy holds it
    // (which nodes are accepted follows from the bounds), so it writes nothing:
    // readers keep taking that copy, and its Upsilon masks, written in an earlier
    // restart, are not applied again.
    if (n_upd != 0u) {
        // ---- write the other copy, then publish it
        const int ns = own < 0 ? 0 : ((own & 1) ^ 1);
        T* dst = P.slot + (static_cast<int64_t>(b) * 2 + ns) * kSlot;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            store8(dst + pbase + 64 * s, out + 8 * s);
            dst[kXF0 + (z0 + s) * 8 + y] = out[8 * s];
            dst[kXF7 + (z0 + s) * 8 + y] = out[8 * s + 7];
        }
        if (lane < 6)
            P.ups[(static_cast<int64_t>(b) * 2 + ns) * 6 + lane] = (static_cast<unsigned long long>(uhi) << 32) | ulo;
        // No fence: nobody reads this copy before the grid barrier that ends the
        // restart (a reader that sees the new stamp takes the other copy).
        if (lane == 6)
            P.stamp[b] = make_stamp(k, own < 0 ? static_cast<int>(kNever) : stamp_latest(ms), ns);
    }

    // publish: the brick's restart-k march has finished (read by early marches of
    // its neighbours; the release store orders the warp's writes above it).  Before
    // the activation below, whose chain of atomics they need not wait for.
    __syncwarp();
    if (publish && lane == 7) st_release(P.done + b, k);
    // ---- activation for restart k+1 (A of Alg. 4/5, C of Alg. 4)
    // (once the bound has reached width_band, pending nodes above it stay tentative: Alg. 6's A flag)
    if ((lane == 6 && n != 0u && grow) || (lane < 6 && (ulo | uhi) != 0u && mine >= 0)) enqueue_next(P, G, k, mine);
    __syncwarp();
}

}  // namespace eikg
