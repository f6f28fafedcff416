// March_Narrow_Band (Alg. 4 with Algs. 2, 3 and the ghost exchange of Alg. 5) of
// one 16x16x16 block (a group of 2x2x2 bricks) by one CTA of eight warps.
//
// The group's psi with one ghost layer and its h/F sit in shared memory in one
// 18^3 layout; tentative values carry their sign bit, and h/F its sign bit while
// a node must not be queued, as in the 8^3 march (eik_march8.cuh).  The nodes to
// solve are kept in two lists: a wave solves the nodes of one, 32 per warp at a
// time, and queues the neighbours that an accepted node can lower into the other.
//
// A node is in a list at most once, so one thread alone writes its value in a wave.
// A neighbour's value may be read before or after that neighbour's own solve of
// the wave; either is an upper bound of what it ends with, and as the wave starts
// with clearing its nodes' queue marks, a neighbour that is lowered queues them
// again for the next.  So may a listed node's h/F be read while another thread's mark
// (a NaN) stands in its sign word: the node then counts as one that is never solved,
// passes on the value it has, and is solved in the next wave, since a marked node is
// always in the next list.  Either way psi ends the same; the counts of solves and
// accepted nodes depend on the timing.
//
// What bounds it: the chain of waves (two of its three latencies are shared-memory
// round trips) and, with all SMs busy, issue slots.  The march this replaces gave
// each warp a brick of its own and kept the eight in lockstep with four CTA
// barriers a round, most warps idle while the front crossed one brick: 256^3 of
// sines took 21.3 ms with it.
#pragma once

#include "eik_march8.cuh"

namespace eikg {

constexpr int kE16 = 16;
constexpr int kH16 = kE16 + 2;
constexpr int kTile16 = kH16 * kH16 * kH16;
constexpr int kNodes16 = kE16 * kE16 * kE16;

template <typename T>
struct __align__(16) GroupSmem {
    T psi[kTile16];                    // index ((z+1)*18 + (y+1))*18 + (x+1); tentative values negative
    T rq[kTile16];                     // h/F, same index; negative: not to be queued
    uint16_t list[2][kNodes16];        // nodes to solve in this and the next wave (tile indices)
    unsigned long long mask[8][6];     // per brick and face: nodes the neighbour has to see (Upsilon)
    typename SBitsOf<T>::S mn[2];      // smallest tentative value, by stage parity (sbits)
    int count[3];                      // lengths of the lists, by wave number mod 3
    unsigned pend[8];                  // per brick: pending nodes
    T rmin[8];
    T rmax[8];
    int any;                           // the march lowered a value
};

__device__ __forceinline__ int h16(int x, int y, int z) { return ((z + 1) * kH16 + (y + 1)) * kH16 + x + 1; }

// Set the sign bit of a shared value's word where `want` holds; true if it was
// clear.  Predicated, so that several are in flight together (the warps of a CTA
// claim nodes from each other, so this has to be atomic).
__device__ __forceinline__ bool claim_sign(uint32_t word, bool want) {
    unsigned old;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.u32 %0, 0x80000000;\n\t"
                 "@p atom.shared.or.b32 %0, [%1], 0x80000000;\n\t}"
                 : "=r"(old)
                 : "r"(word), "r"(want ? 1u : 0u)
                 : "memory");
    return static_cast<int>(old) >= 0;
}

// Append the lanes' nodes (where `in` holds) to a list: one shared atomic a warp.
__device__ __forceinline__ void append(uint16_t* list, int* count, bool in, int h, int lane) {
    const unsigned m = __ballot_sync(kFull, in);
    if (m == 0u) return;
    int base = 0;
    if (lane == 0) base = atomicAdd(count, __popc(m));
    base = __shfl_sync(kFull, base, 0);
    if (in) list[base + __popc(m & ((1u << lane) - 1u))] = static_cast<uint16_t>(h);
}

// Group (gx, gy, gz) of grid G at restart k; every thread of the CTA.
template <typename T>
__device__ __forceinline__ void march16(const LoopParams<T>& P, const Geo& G, MarchAcc& A, int gx, int gy, int gz, int k,
                                        T bprev, T bound, bool grow, T window) {
    static_assert(kWarps == 8, "a warp per brick of the group");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GroupSmem<T>& S = *reinterpret_cast<GroupSmem<T>*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    using SB = typename SBitsOf<T>::S;
    using UB = typename BitsOf<T>::U;
    const T INF = Num<T>::inf();
    const int BX = G.BX, BY = G.BY, BZ = G.BZ;
    auto brick = [&](int x, int y, int z) -> int32_t {
        return (x >= 0 && x < BX && y >= 0 && y < BY && z >= 0 && z < BZ) ? G.boff + (z * BY + y) * BX + x : -1;
    };
    // this warp's brick, and this lane's two rows of it
    const int wx = warp & 1, wy = (warp >> 1) & 1, wz = warp >> 2;
    const int32_t b = brick(2 * gx + wx, 2 * gy + wy, 2 * gz + wz);
    const int y = lane & 7, zp = lane >> 3, z0 = 2 * zp;
    const int pbase = (z0 * 8 + y) * 8;
    const int hbase = h16(8 * wx, 8 * wy + y, 8 * wz + z0);
    constexpr int kUp = kH16 * kH16;                             // tile index step along z
    // the quadrant (64 nodes) of every outer face this warp's lanes hold half of:
    // face-local index u = 32 * half + lane as in the bricks' own masks
    const int q = warp >> 1, half = warp & 1, u = 32 * half + lane, qa = q & 1, qc = q >> 1;
    const int fa = 8 * qa + (u & 7), fc = 8 * qc + (u >> 3);
    auto ghost = [&](int f) {
        const int w = (f & 1) ? kE16 : -1;
        return f < 2 ? h16(w, fa, fc) : f < 4 ? h16(fa, w, fc) : h16(fa, fc, w);
    };
    auto inner = [&](int f) { return ghost(f) + (f < 2 ? 1 : f < 4 ? kH16 : kUp) * ((f & 1) ? -1 : 1); };
    // brick of the group on face f's side in quadrant (a, c): its number (warp) in the group
    auto side = [&](int f) {
        const int w = f & 1;
        return f < 2 ? w + 2 * qa + 4 * qc : f < 4 ? qa + 2 * w + 4 * qc : qa + 2 * qc + 4 * w;
    };

    // ---- load (as march8): lane f < 6 looks after the neighbour across face f in
    // this warp's quadrant, lane 6 after the warp's own brick
    int32_t mine = -1;
    if (lane < 6) {
        const int n = side(lane), w = (lane & 1) ? 1 : -1, ax = lane >> 1;
        const int nx = 2 * gx + (n & 1), ny = 2 * gy + ((n >> 1) & 1), nz = 2 * gz + (n >> 2);
        if (brick(nx, ny, nz) >= 0)
            mine = brick(nx + (ax == 0 ? w : 0), ny + (ax == 1 ? w : 0), nz + (ax == 2 ? w : 0));
    }
    if (lane == 6) mine = b;
    const unsigned long long ms = mine >= 0 ? __ldcg(P.stamp + mine) : kUntouched;
    UB rlo = BitsOf<T>::kInf;
    SB rhi = 0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        T r8[8];
        if (b >= 0) {
            load8_ro(P.rr + static_cast<int64_t>(b) * kBrick + pbase + 64 * s, r8);
        } else {
#pragma unroll
            for (int x = 0; x < 8; ++x) r8[x] = -INF;
        }
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            S.rq[hbase + kUp * s + x] = r8[x];
            rlo = min(rlo, ubits(r8[x]));
            rhi = max(rhi, sbits(r8[x]));
        }
    }
    int32_t copy = -1;
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
    // nodes on the group's inner faces that the brick lowered in restart k-1 as an
    // 8^3 block (a schedule may mix block edges): its neighbours inside the group
    // have not seen them yet, so they are tentative again (bit per node of the rows)
    unsigned again = 0;
    {
        const unsigned long long mb = __shfl_sync(kFull, ms, 6);
        if (own >= 0 && stamp_latest(mb) == k - 1) {             // (the same on every lane)
            const unsigned long long* um = P.ups + static_cast<int64_t>(own) * 6;
            const unsigned long long ux = __ldcg(um + 1 - wx), uy = __ldcg(um + 3 - wy), uz = __ldcg(um + 5 - wz);
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int z = z0 + s;
                unsigned m = static_cast<unsigned>((ux >> (z * 8 + y)) & 1ull) << (wx ? 0 : 7);
                if (y == (wy ? 0 : 7)) m |= static_cast<unsigned>(uy >> (z * 8)) & 0xFFu;
                if (z == (wz ? 0 : 7)) m |= static_cast<unsigned>(uz >> (y * 8)) & 0xFFu;
                again |= m << (8 * s);
            }
        }
    }
    T fv[6];
#pragma unroll
    for (int f = 0; f < 6; ++f) {
        const int32_t cf = __shfl_sync(kFull, copy, f);
        const int off = f == 0 ? kXF7 + u : f == 1 ? kXF0 + u : f == 2 ? (u >> 3) * 64 + 56 + (u & 7)
                        : f == 3 ? (u >> 3) * 64 + (u & 7) : f == 4 ? 7 * 64 + u : u;
        fv[f] = INF;
        if (cf >= 0) fv[f] = __ldcg(P.slot + static_cast<int64_t>(cf) * kSlot + off);
    }
    if (threadIdx.x == 0) {
        S.count[0] = S.count[1] = S.count[2] = 0;
        S.mn[0] = S.mn[1] = SBitsOf<T>::kMax;
        S.any = 0;
    }
    if (threadIdx.x < 48) S.mask[threadIdx.x / 6][threadIdx.x % 6] = 0ull;
    if (threadIdx.x < 8) S.pend[threadIdx.x] = 0u;
    // ---- the band at the start of the march (as march8; ghost nodes up to the bound accepted at once)
    SB smin = SBitsOf<T>::kMax;
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const T v = row[8 * s + x];
            const T t = ((again >> (8 * s + x)) & 1u) ? vneg(v) : band_value(v, bprev);
            S.psi[hbase + kUp * s + x] = t;
            smin = min(smin, sbits(t));
        }
    unsigned fire = 0;
#pragma unroll
    for (int f = 0; f < 6; ++f) {
        const T v = fv[f];
        const unsigned um = __shfl_sync(kFull, half ? static_cast<unsigned>(mups >> 32) : static_cast<unsigned>(mups), f);
        const bool tent = vlt(v, INF) && (((um >> lane) & 1u) || sbits(v) > sbits(bprev));
        const bool take = tent && sbits(v) <= sbits(bound);
        S.psi[ghost(f)] = tent && !take ? vneg(v) : v;
        S.rq[ghost(f)] = -INF;
        if (take) smin = min(smin, sbits(vneg(v)));
        fire |= (take ? 1u : 0u) << f;
    }
    const T rmin_w = warp_min_nn(from_bits(rlo)), rmax_w = warp_max(from_bits(static_cast<UB>(rhi)));
    if (lane == 0) {
        S.rmin[warp] = rmin_w;
        S.rmax[warp] = rmax_w;
    }
    __syncthreads();
    unsigned n_acc = __popc(fire), n_upd = 0u, n_solve = 0u;
    int n_fb = 0;
    auto warp_min_sb = [&](SB s) -> T {
        return warp_min_nn(s < 0 ? vabs(from_bits(static_cast<UB>(s))) : INF);
    };
    {
        const T m = warp_min_sb(smin);
        if (lane == 0 && m < INF) atomicMin(&S.mn[0], sbits(vneg(m)));
    }
#pragma unroll
    for (int f = 0; f < 6; ++f) {
        const int h = inner(f);
        const bool want = ((fire >> f) & 1u) && vlt(fv[f], vabs(S.psi[h]));
        append(S.list[0], &S.count[0], claim_sign(sign_word(S.rq + h), want), h, lane);
    }
    T rmin_g = S.rmin[0], rmax_g = S.rmax[0];
#pragma unroll
    for (int i = 1; i < kWarps; ++i) rmin_g = vmin(rmin_g, S.rmin[i]), rmax_g = vmax(rmax_g, S.rmax[i]);
    const T w = static_cast<T>(1.5f) * window * rmin_g;           // (a stage spans one and a half windows, as march8)
    int stages = 0, wave = 0;
    __syncthreads();

    for (;;) {
        const SB ms0 = S.mn[stages & 1];
        const T mn = ms0 < 0 ? vabs(from_bits(static_cast<UB>(ms0))) : INF;
        if (!(mn < INF) || !(mn <= bound)) break;   // band empty, or its minimum above the bound
        if (++stages > kRoundCap) {
            if (threadIdx.x == 0) atomicOr(&P.ctrl->status, kStRoundCap);
            break;
        }
        const T thr = vmin(mn + w, bound);
        const SB tk = sbits(vneg(thr));
        // ---- tentative nodes up to thr -> the list, and the smallest above it.  (A
        // node already listed, next to an accepted ghost node, is not listed again; a
        // fixed node is never marked and only passes its value on.)
        smin = SBitsOf<T>::kMax;
        {
            unsigned C = 0;
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    const SB v = sbits(S.psi[hbase + kUp * s + x]);
                    if (v <= tk) C |= 1u << (8 * s + x);
                    else smin = min(smin, v);
                }
            if (__any_sync(kFull, C != 0u)) {                    // (a brick the front is not in has none)
                const uint32_t rw = sign_word(S.rq + hbase);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int h = (j >> 3) * kUp + (j & 7);
                    const int w0 = ld_word(rw + h * static_cast<int>(sizeof(T)));
                    if (w0 < 0 && vlt(vabs(S.rq[hbase + h]), INF)) C &= ~(1u << j);
                    if ((C >> j) & 1u) st_word(rw + h * static_cast<int>(sizeof(T)), w0 | static_cast<int>(0x80000000u));
                }
                const int cnt = __popc(C);
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl += t;
                }
                const int total = __shfl_sync(kFull, incl, 31);
                int base = 0;
                if (lane == 0) base = atomicAdd(&S.count[wave % 3], total);
                uint16_t* at = S.list[wave & 1] + __shfl_sync(kFull, base, 0) + (incl - cnt);
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if ((C >> j) & 1u) *at++ = static_cast<uint16_t>(hbase + (j >> 3) * kUp + (j & 7));
            }
        }
        __syncthreads();
        // ---- waves
        for (;; ++wave) {
            const int n = S.count[wave % 3];
            if (threadIdx.x == 0) {
                S.count[(wave + 2) % 3] = 0;                     // last read in the wave before this one
                if (n == 0) S.mn[stages & 1] = SBitsOf<T>::kMax; // (this stage's was read before the scan's barrier)
            }
            if (n == 0) break;
            const uint16_t* from = S.list[wave & 1];
            uint16_t* to = S.list[(wave + 1) & 1];
            int* fill = &S.count[(wave + 1) % 3];
            // the listed nodes may be queued again from here on
            for (int i = threadIdx.x; i < n; i += 32 * kWarps) {
                T* p = S.rq + from[i];
                const T r = vabs(*p);
                if (vlt(r, INF)) *p = r;
            }
            __syncthreads();
            for (int base = 0; base < n; base += 32 * kWarps) {
                const bool val = base + static_cast<int>(threadIdx.x) < n;
                n_solve += val ? 1u : 0u;
                const int hq = val ? from[base + threadIdx.x] : h16(0, 0, 0);
                T* ps = S.psi + hq;
                volatile const T* pv = ps;
                const T r = vabs(S.rq[hq]);
                // (a fixed node only passes its value on, and so does one that is just
                // being marked for the next wave: r is a NaN)
                const bool live = val && vlt(r, INF);
                const T cur = pv[0], c = vabs(cur);
                const T nv[6] = {pv[-1], pv[1], pv[-kH16], pv[kH16], pv[-kUp], pv[kUp]};
                const T mx = axis_min(nv[0], nv[1]), my = axis_min(nv[2], nv[3]), mz = axis_min(nv[4], nv[5]);
                T a0, a1, a2;
                sort3(mx, my, mz, a0, a1, a2);
                const bool go = live && vlt(a0, INF);
                const T xn = QueueRoot<T>::go(a0, a1, a2, r, go, P.tau_f, n_fb);
                const bool imp = go && vlt(xn, c);
                const T v = imp ? xn : c;
                const bool prop = val && (imp || sgn(cur)) && !vlt(thr, v);
                if (imp || prop) *const_cast<volatile T*>(ps) = prop ? v : vneg(v);
                if (imp && !prop) smin = min(smin, sbits(vneg(v)));
                n_upd += imp ? 1u : 0u;
                n_acc += prop ? 1u : 0u;
                // queue the neighbours above the accepted value, each once, by marks as in
                // march8; marks are negative, so a warp that is a round ahead leaves them be
                constexpr int off[6] = {-1, 1, -kH16, kH16, -kUp, kUp};
                const int mark = (sizeof(T) == 4 ? static_cast<int>(0xFFC00000u) : static_cast<int>(0xFFF80000u)) |
                                 static_cast<int>(threadIdx.x);
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
                __syncthreads();
                unsigned cnt = 0;
#pragma unroll
                for (int d = 0; d < 6; ++d) {
                    win[d] = win[d] && ld_word(rw + off[d] * static_cast<int>(sizeof(T))) == mark;
                    cnt += win[d] ? 1u : 0u;
                }
                const unsigned c0 = __ballot_sync(kFull, cnt & 1u), c1 = __ballot_sync(kFull, cnt & 2u);
                const unsigned c2 = __ballot_sync(kFull, cnt & 4u), lt = (1u << lane) - 1u;
                const int total = __popc(c0) + 2 * __popc(c1) + 4 * __popc(c2);
                if (total > 0) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(fill, total);
                    at = __shfl_sync(kFull, at, 0) + __popc(c0 & lt) + 2 * __popc(c1 & lt) + 4 * __popc(c2 & lt);
#pragma unroll
                    for (int d = 0; d < 6; ++d)
                        if (win[d]) {
                            to[at++] = static_cast<uint16_t>(hq + off[d]);
                            st_word(rw + off[d] * static_cast<int>(sizeof(T)), nw[d] | static_cast<int>(0x80000000u));
                        }
                }
            }
            __syncthreads();
        }
        // (the list of wave `wave` is empty and stays the next stage's)
        {
            const T m = warp_min_sb(smin);
            __syncthreads();                                     // (the other parity's slot is clear)
            if (lane == 0 && m < INF) atomicMin(&S.mn[stages & 1], sbits(vneg(m)));
        }
        __syncthreads();
    }

    // ---- the brick's values and tentative nodes; the copy it started from, to see whether it was lowered
    n_upd = __reduce_add_sync(kFull, n_upd);
    if (lane == 0 && n_upd) S.any = 1;
    __syncthreads();
    const bool any = S.any != 0;
    T out[16];
    unsigned nt = 0;
    bool low = false;
    {
        T old[16];
        T fold[6];
#pragma unroll
        for (int x = 0; x < 16; ++x) old[x] = INF;
        if (any && own >= 0) {
            const T* src = P.slot + static_cast<int64_t>(own) * kSlot;
            load8_cg(src + pbase, old);
            load8_cg(src + pbase + 64, old + 8);
        }
        // the face nodes' old values: their bricks' copies (lane 6 of warp `side` knows which)
        int32_t* copies = reinterpret_cast<int32_t*>(S.list[1]);          // (the lists are done with)
        if (lane == 6) copies[warp] = copy;
        __syncthreads();
#pragma unroll
        for (int f = 0; f < 6; ++f) {
            const int32_t cf = copies[side(f)];
            const int o = f == 0 ? kXF0 + u : f == 1 ? kXF7 + u : f == 2 ? (u >> 3) * 64 + (u & 7)
                          : f == 3 ? (u >> 3) * 64 + 56 + (u & 7) : f == 4 ? u : 7 * 64 + u;
            fold[f] = INF;
            if (any && cf >= 0) fold[f] = __ldcg(P.slot + static_cast<int64_t>(cf) * kSlot + o);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const T t = S.psi[hbase + kUp * s + x];
                nt += sgn(t) ? 1u : 0u;
                out[8 * s + x] = vabs(t);
                low = low || vlt(out[8 * s + x], old[8 * s + x]);
            }
        // Upsilon and pending ghost nodes, per outer face (as march8)
#pragma unroll
        for (int f = 0; f < 6; ++f) {
            const T g = S.psi[ghost(f)], v = vabs(S.psi[inner(f)]);
            const unsigned pg = __ballot_sync(kFull, sgn(g) && vlt(vabs(g), v));
            const unsigned m = __ballot_sync(kFull, any && vlt(v, fold[f]) && vlt(v, vabs(g)));
            if (lane == 0) {
                if (pg) atomicAdd(&S.pend[side(f)], __popc(pg));
                reinterpret_cast<unsigned*>(&S.mask[side(f)][f])[half] = m;
            }
        }
    }
    // A schedule that mixes block edges (it keeps the brick list) may march the next
    // restart brick by brick: a tentative node across an inner face of the group that
    // lies below the brick's own node is then a ghost this brick has to see.  Nothing
    // else would tell it, since the node's brick accepts it without lowering it.  (Not
    // counted in the band: the node's own brick counts it.)
    bool across = false;
    if (G.lists & 1u) {
        auto pending = [&](int h, int d) {
            const T g = S.psi[h + d];
            return sgn(g) && vlt(vabs(g), vabs(S.psi[h]));
        };
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int h = hbase + kUp * s;
            across = across || pending(h + (wx ? 0 : 7), wx ? -1 : 1);
            if (y == (wy ? 0 : 7))
                for (int x = 0; x < 8; ++x) across = across || pending(h + x, wy ? -kH16 : kH16);
            if (z0 + s == (wz ? 0 : 7))
                for (int x = 0; x < 8; ++x) across = across || pending(h + x, wz ? -kUp : kUp);
        }
        across = __any_sync(kFull, across);
    }
    low = __any_sync(kFull, low);
    nt = __reduce_add_sync(kFull, nt);
    if (lane == 0 && nt) atomicAdd(&S.pend[warp], nt);
    n_acc = __reduce_add_sync(kFull, n_acc);
    n_solve = __reduce_add_sync(kFull, n_solve);
    n_fb = __reduce_add_sync(kFull, n_fb);
    __syncthreads();
    if (lane == 0) {
        A.accepted += n_acc;
        A.band += S.pend[warp];
        A.fallbacks += n_fb;
        A.updates += n_upd;
        A.solves += n_solve;
        A.rounds += warp == 0 ? stages : 0;
        A.rmin = fminf(A.rmin, static_cast<float>(rmin_g));
        A.rmax = fmaxf(A.rmax, static_cast<float>(rmax_g));
    }
    if (b < 0) return;
    // ---- a brick that was lowered: write its other copy, then publish it
    if (low) {
        const int ns = own < 0 ? 0 : ((own & 1) ^ 1);
        T* dst = P.slot + (static_cast<int64_t>(b) * 2 + ns) * kSlot;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            store8(dst + pbase + 64 * s, out + 8 * s);
            dst[kXF0 + (z0 + s) * 8 + y] = out[8 * s];
            dst[kXF7 + (z0 + s) * 8 + y] = out[8 * s + 7];
        }
        if (lane < 6) P.ups[(static_cast<int64_t>(b) * 2 + ns) * 6 + lane] = S.mask[warp][lane];
        // No fence: nobody reads this copy before the grid barrier that ends the
        // restart (a reader that sees the new stamp takes the other copy).
        if (lane == 6) P.stamp[b] = make_stamp(k, own < 0 ? static_cast<int>(kNever) : stamp_latest(ms), ns);
    }
    // ---- activation for restart k+1 (A of Alg. 4/5, C of Alg. 4; across the group's own faces, whose masks are 0, only
    // for tentative nodes, see above: the accepted ones have reached the other brick in this march)
    if (lane == 6 && (S.pend[warp] != 0u || across) && grow) enqueue_next(P, G, k, b);
    if (lane < 6 && S.mask[warp][lane] != 0ull) {
        const int ax = lane >> 1, w1 = (lane & 1) ? 1 : -1;
        const int32_t nb = brick(2 * gx + wx + (ax == 0 ? w1 : 0), 2 * gy + wy + (ax == 1 ? w1 : 0),
                                 2 * gz + wz + (ax == 2 ? w1 : 0));
        if (nb >= 0) enqueue_next(P, G, k, nb);
    }
}

}  // namespace eikg
