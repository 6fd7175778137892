// Shared pieces of the packed 16-bit kernels in diagonal coordinates
// (xdrop_diag16.cu): the frame, the per-unit state, code bit planes, live
// masks and window slides.
//
// Frame.  Row i on anti-diagonal d sits at r = i - floor(d' / 2), d' = d + phi
// (phi = 0 or 1, fixed per extension so that the loop's first step has an odd
// d').  A band that follows the main diagonal stays where it is: the window
// slides only when insertions and deletions have moved the band by a good
// part of the window, not once per 16 anti-diagonals as a window of rows
// does.  Only two anti-diagonals are kept, those of even and of odd d', and a
// step replaces the older in place: with e = floor(d' / 2)
//   odd  d' = 2e + 1: up = even[s - 1], left = even[s],    diag = odd[s]
//   even d' = 2e:     up = odd[s],      left = odd[s + 1], diag = even[s]
// (s the window slot of r).  An even step moves the a' codes one slot down,
// an odd step the b' codes one slot up.
//
// Values.  Two slots share a 32-bit register as 16-bit keys
//     v = KS * (S - B_d) + (VR - 1 - k),
// k the slot within its virtual lane of VR = 2 R slots (register h of a
// virtual lane holds slots h and h + R), B_d a base that moves by the gap
// score per anti-diagonal, B_d = B_{d-1} + gap.  So the gap moves add nothing,
// and the diagonal adds KS * (substitution - 2 gap).  With T_d = best_{<d} - X
// a cell is live iff v >= theta_d = KS * (T_d - B_d); theta grows by
// KS * (-gap) per anti-diagonal and by KS per unit of a new best.  Every
// `period` steps theta is brought back to 32768 by one subtraction from
// every register.  A key's low bits are the row's code, so one unsigned 16-bit
// maximum gives the best score and its smallest row.
//
// Pruning without selects.  A pruned cell keeps its value v < theta.  Two rules
// keep the live cells exact: a step along the diagonal adds the substitution
// only when its predecessor is live and the target lies in the evaluated
// range (else it adds 0, i.e. 2 gap in score), and the live mask of a step is
// taken inside the range.  Then
//   * a value below the threshold never climbs back: its moves add gap (<= 0)
//     or 2 gap while the threshold does not fall;
//   * a cell of the matrix outside [lo, hi + 1] has no live neighbour on
//     d - 1, so a live diagonal predecessor D had D + gap < T_{d-1} (both
//     cells between them were evaluated and died), and D + 2 gap < T_d;
//   * slots outside the matrix read none of their values back into it, never
//     exceed the best (they only add gaps), and are masked from the live set.
// So neither values nor ranges are tested per cell: what is left per pair of
// cells is the substitution's mask and multiply-add, the shifted neighbour's
// row code, one 3-input maximum, the threshold's subtraction, half a byte
// permute that collects four slots' signs, and half a maximum for the best.
#pragma once

#include "internal.h"

namespace logan {

namespace {

constexpr uint32_t FULL = 0xffffffffu;
constexpr int NEGU = -(1 << 20);  // -inf of the 32-bit relative records

// G lanes of V virtual lanes of 2 R slots
template <int G, int V, int R>
struct Diag {
    static_assert(R == 16 || (V == 1 && (R == 8 || R == 4 || R == 2)), "registers per virtual lane");
    static constexpr int VR = 2 * R;     // slots of a virtual lane
    static constexpr int C = V * VR;     // slots of a lane
    static constexpr int W = G * C;      // slots of the window
    static constexpr int LOG2W = W == 32    ? 5
                                 : W == 64  ? 6
                                 : W == 128 ? 7
                                 : W == 256 ? 8
                                 : W == 512 ? 9
                                 : W == 1024 ? 10
                                             : 11;
    static_assert((1 << LOG2W) == W, "window must be a power of two");
    // anti-diagonals per loop iteration; with two virtual lanes the body of
    // four costs more in registers than it saves
    static constexpr int UNROLL = V == 1 ? 4 : 2;
    // a slide moves the window by half a virtual lane, or by whole lanes (an
    // eighth of the window) where a virtual lane is short
    static constexpr int SL = R == 16 ? 0 : (G >= 8 ? G / 8 : 1);
    static constexpr int SLIDE = R == 16 ? R : SL * VR;
    static constexpr uint32_t VMASK = VR == 32 ? 0xffffffffu : (1u << VR) - 1u;
};

// Per-unit state, replicated in its lanes except what is marked per lane.
template <int V>
struct DState {
    int dn, mt;         // first slot with a column and slot of row m, minus the lane's first slot
    int theta;
    int best;
    int X;
    int base, e, phi;
    int bd, br;         // per lane: anti-diagonal and r of the last best cell that this lane found
    uint32_t c32;       // per lane: cells since the last fold into `cells`
    unsigned long long cells;   // per lane
    unsigned long long cells0;  // cells of narrower levels (resumed items), in the leader lane
    uint32_t item;
    bool active, done, overflow, migrated;
    uint32_t rb[V];                        // slots of the next step's range (without the matrix's bounds)
    uint32_t LE[V], LO[V];                 // live slots on the last even / odd anti-diagonal
    uint32_t a0[V], a1[V], b0[V], b1[V];   // code bit planes, bit k = slot k
    uint32_t na0, na1, nb0, nb1;           // the codes that enter next (a': low bit first, b': high bit first)
};

// lane masks of a unit of G lanes: the unit's lanes, those below and above
template <int G>
struct Lanes {
    uint32_t all, below, above, prev, next;
    __device__ __forceinline__ explicit Lanes(int lane) {
        const int first = lane / G * G;
        all = G == 32 ? FULL : (((1u << (G & 31)) - 1u) << first);
        const uint32_t me = 1u << lane;
        below = all & (me - 1u);
        above = all & ~(me - 1u) & ~me;
        prev = (me >> 1) & all;
        next = (me << 1) & all;
    }
};

// 16 two-bit codes (code t at bits 2t) -> their low and high bit planes
__device__ __forceinline__ void planes16(uint32_t c, uint32_t& p0, uint32_t& p1) {
    uint32_t x = c & 0x55555555u, y = (c >> 1) & 0x55555555u;
    x = (x | (x >> 1)) & 0x33333333u;
    y = (y | (y >> 1)) & 0x33333333u;
    x = (x | (x >> 2)) & 0x0f0f0f0fu;
    y = (y | (y >> 2)) & 0x0f0f0f0fu;
    x = (x | (x >> 4)) & 0x00ff00ffu;
    y = (y | (y >> 4)) & 0x00ff00ffu;
    p0 = (x | (x >> 8)) & 0xffffu;
    p1 = (y | (y >> 8)) & 0xffffu;
}

// stream codes q..q+15 (code q in the low bits), 0 for indices below 0 and
// outside [0, len) when the whole group is
__device__ __forceinline__ uint32_t codes16z(const uint32_t* __restrict__ w, int64_t pos, int dir,
                                             int len, int q) {
    if (q >= 0) return stream_codes16(w, pos, dir, len, q);
    if (q <= -16) return 0u;
    return stream_codes16(w, pos, dir, len, 0) << (2u * uint32_t(-q));
}

// bit planes of stream codes q..q+31 (code q in bit 0)
__device__ __forceinline__ void planes32(const uint32_t* __restrict__ w, int64_t pos, int dir,
                                         int len, int q, uint32_t& p0, uint32_t& p1) {
    uint32_t l0, l1, h0, h1;
    planes16(codes16z(w, pos, dir, len, q), l0, l1);
    planes16(codes16z(w, pos, dir, len, q + 16), h0, h1);
    p0 = l0 | (h0 << 16);
    p1 = l1 | (h1 << 16);
}

// The codes that enter the lane's slots in the next kPrefetch steps: a' at
// the top of its last virtual lane's 32 planes, b' below its first slot.
template <int G, int V, int R>
__device__ __forceinline__ void load_next(const KernelArgs& ka, const Item& it, DState<V>& u,
                                          int gl) {
    using D = Diag<G, V, R>;
    const int dir = (it.flags & ITEM_LEFT) ? -1 : 1;
    const int s0 = u.base + gl * D::C;  // r of the lane's first slot
    planes32(ka.wa, it.a_pos, dir, int(it.m), s0 + (V - 1) * D::VR + 32 + u.e - 1, u.na0, u.na1);
    planes32(ka.wb, it.b_pos, dir, int(it.n), u.e - u.phi - s0, u.nb0, u.nb1);
    u.nb0 = __brev(u.nb0);
    u.nb1 = __brev(u.nb1);
}

// All planes for a coming odd step of frame e: slot r holds a' index
// r + e - 1 and (one step back) b' index e - 1 - phi - r.
template <int G, int V, int R>
__device__ __forceinline__ void load_planes(const KernelArgs& ka, const Item& it, DState<V>& u,
                                            int gl) {
    using D = Diag<G, V, R>;
    const int dir = (it.flags & ITEM_LEFT) ? -1 : 1;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int s0 = u.base + gl * D::C + v * D::VR;
        planes32(ka.wa, it.a_pos, dir, int(it.m), s0 + u.e - 1, u.a0[v], u.a1[v]);
        uint32_t p0, p1;
        planes32(ka.wb, it.b_pos, dir, int(it.n), u.e - 1 - u.phi - s0 - 31, p0, p1);
        u.b0[v] = __brev(p0);
        u.b1[v] = __brev(p1);
    }
    load_next<G, V, R>(ka, it, u, gl);
}

template <int G>
__device__ __forceinline__ uint32_t unit_max_u32(uint32_t v) {
    if constexpr (G == 32) {
        return __reduce_max_sync(FULL, v);
    } else {
#pragma unroll
        for (int o = G / 2; o >= 1; o >>= 1) v = max(v, __shfl_xor_sync(FULL, v, o, G));
        return v;
    }
}

template <int G>
__device__ __forceinline__ uint32_t unit_max_u16x2(uint32_t v) {
#pragma unroll
    for (int o = G / 2; o >= 1; o >>= 1) v = __vimax3_u16x2(v, __shfl_xor_sync(FULL, v, o, G), 0u);
    return v;
}

// four bytes of sign bits: byte 0 = sign of a's low half, 1 = b's low half,
// 2 = a's high half, 3 = b's high half, each 0xff or 0 (a byte permute in its
// sign-replicating form: a selector nibble's top bit copies the sign of the
// byte; the __byte_perm intrinsic ignores that bit, so this is PTX)
__device__ __forceinline__ uint32_t sign_bytes(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, 0xFBD9;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// Gathers the signs of all half-words of R registers into a mask, bit k = slot
// k, from pairs of registers h and h + R / 2: four slots' sign bytes per
// permute; for R >= 8 they add up by multiply-adds as 255 * mask (each byte 0
// or 255 times its power of two), and 255 * 0xfefefeff = 1 (mod 2^32).
template <int R>
struct SignMask {
    uint32_t acc = 0u;
    __device__ __forceinline__ void add(int h, uint32_t xa, uint32_t xb) {
        const uint32_t w = sign_bytes(xa, xb);
        if constexpr (R == 2) acc = w & 0x08040201u;             // bytes: slots 0, 1, 2, 3
        else if constexpr (R == 4) acc |= w & (h ? 0x80200802u : 0x40100401u);  // byte j: slots 2j, 2j + 1
        else acc = w * (1u << h) + acc;
    }
    __device__ __forceinline__ uint32_t get() const {
        if constexpr (R < 8) return (acc * 0x01010101u) >> 24;
        uint32_t m = acc * 0xfefefeffu;
        if constexpr (R == 8) {  // byte j: slots 4j .. 4j + 3, nibbles to 16 bits
            m = m | (m >> 4);
            m = __byte_perm(m, 0u, 0x4420);
        }
        return m;
    }
};

// bits from the highest set bit of an N-bit mask downwards (0 for 0)
template <int N>
__device__ __forceinline__ uint32_t fill_down(uint32_t m) {
    if constexpr (N <= 8) {  // shifts and ORs: shorter than a find-leading-one
        m = m | (m >> 1) | (m >> 2);
        if constexpr (N == 4) return m | (m >> 3);
        return m | (m >> 3) | (m >> 6);
    } else {
        return __funnelshift_rc(~0u, 0u, __clz(m));
    }
}

// The slots of the next anti-diagonal's range [first live, last live + 1] (rows)
// from the live slots L of this one, without numbers: a slot is in range when
// a live slot lies at or below its row and one at or above the row before.  ODD: L is
// of an odd step, the next one (even) sees rows one slot lower.  Returns the
// warp's vote of lanes with a live slot.
template <int G, int V, int R, bool ODD>
__device__ __forceinline__ uint32_t next_range(const uint32_t (&L)[V], const Lanes<G>& ln,
                                               uint32_t (&rb)[V]) {
    constexpr int VR = Diag<G, V, R>::VR;
    uint32_t anyl = L[0];
    if constexpr (V == 2) anyl |= L[1];
    const uint32_t vote = __ballot_sync(FULL, anyl != 0u);
    bool near_;  // the neighbouring lane's slot next to this lane's first (odd: last) one is live
    if constexpr (G == 1) {
        near_ = false;
    } else if constexpr (ODD) {
        near_ = (__ballot_sync(FULL, (L[0] & 1u) != 0u) & ln.next) != 0u;
    } else {
        near_ = (__ballot_sync(FULL, (L[V - 1] >> (VR - 1)) != 0u) & ln.prev) != 0u;
    }
    const bool below = (vote & ln.below) != 0u, above = (vote & ln.above) != 0u;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        bool bl = below, ab = above;
        if constexpr (V == 2) {
            if (v == 1) bl = bl || L[0] != 0u;
            else ab = ab || L[1] != 0u;
        }
        uint32_t lx, hx;
        if constexpr (ODD) {
            // from one slot below the first live one, to the last live one
            const uint32_t nx = v + 1 < V ? L[v + 1] & 1u : (near_ ? 1u : 0u);
            lx = (L[v] >> 1) | (L[v] & 1u) | (nx << (VR - 1));
            hx = L[v];
        } else {
            // from the first live slot, to one above the last
            const uint32_t pv = v > 0 ? L[v - 1] >> (VR - 1) : (near_ ? 1u : 0u);
            lx = L[v];
            hx = (L[v] << 1) | pv | (L[v] & (1u << (VR - 1)));
            if constexpr (VR < 32) hx &= (1u << VR) - 1u;
        }
        const uint32_t low = bl ? FULL : (lx | (0u - lx));
        const uint32_t high = ab ? Diag<G, V, R>::VMASK : fill_down<VR>(hx);
        rb[v] = low & high;
    }
    return vote;
}

// key of score distance u (>= 0) above a threshold at 32768, slot k of VR
template <int VR>
__device__ __forceinline__ uint32_t live_key(int u, int k) {
    return 32768u + uint32_t(u) * uint32_t(KS) + uint32_t(VR - 1 - k);
}

// Shifts one array's slots by Diag::SLIDE: UP moves the window to larger rows
// (slot s takes what slot s + SLIDE held).  By half a virtual lane, row codes
// move by +R in the low halves and -R in the high ones.
template <int G, int V, int R, bool UP>
__device__ __forceinline__ void shift_slots(uint32_t (&Q)[V * R], bool on, int gl, uint32_t floor2) {
    constexpr int SL = Diag<G, V, R>::SL;
    constexpr uint32_t rebase = uint32_t(R) - (uint32_t(R) << 16);
#pragma unroll
    for (int h = 0; h < R; ++h) {
        if constexpr (SL > 0) {
            uint32_t x = UP ? __shfl_down_sync(FULL, Q[h], SL, G) : __shfl_up_sync(FULL, Q[h], SL, G);
            x = (UP ? gl >= G - SL : gl < SL) ? floor2 : x;
            Q[h] = on ? x : Q[h];
        } else if constexpr (UP) {
            uint32_t nx = __shfl_down_sync(FULL, Q[h], 1, G);  // the upper lane's first virtual lane
            nx = gl == G - 1 ? floor2 : nx;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const uint32_t y = v + 1 < V ? Q[(v + 1) * R + h] : nx;
                const uint32_t x = __byte_perm(Q[v * R + h], y, 0x5432) + rebase;
                Q[v * R + h] = on ? x : Q[v * R + h];
            }
        } else {
            uint32_t pv = __shfl_up_sync(FULL, Q[(V - 1) * R + h], 1, G);
            pv = gl == 0 ? floor2 : pv;
#pragma unroll
            for (int v = V - 1; v >= 0; --v) {
                const uint32_t y = v > 0 ? Q[(v - 1) * R + h] : pv;
                const uint32_t x = __byte_perm(y, Q[v * R + h], 0x5432) + rebase;
                Q[v * R + h] = on ? x : Q[v * R + h];
            }
        }
    }
}

// the same for a live mask
template <int G, int V, int R, bool UP>
__device__ __forceinline__ void shift_mask(uint32_t (&L)[V], bool on, int gl) {
    constexpr int SL = Diag<G, V, R>::SL;
    constexpr uint32_t M = Diag<G, V, R>::VMASK;
    if constexpr (SL > 0) {
        uint32_t x = UP ? __shfl_down_sync(FULL, L[0], SL, G) : __shfl_up_sync(FULL, L[0], SL, G);
        x = (UP ? gl >= G - SL : gl < SL) ? 0u : x;
        L[0] = on ? x : L[0];
    } else if constexpr (UP) {
        uint32_t nx = __shfl_down_sync(FULL, L[0], 1, G);
        nx = gl == G - 1 ? 0u : nx;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const uint32_t y = v + 1 < V ? L[v + 1] : nx;
            const uint32_t x = ((L[v] >> R) | (y << R)) & M;
            L[v] = on ? x : L[v];
        }
    } else {
        uint32_t pv = __shfl_up_sync(FULL, L[V - 1], 1, G);
        pv = gl == 0 ? 0u : pv;
#pragma unroll
        for (int v = V - 1; v >= 0; --v) {
            const uint32_t y = v > 0 ? L[v - 1] : pv;
            const uint32_t x = ((L[v] << R) | (y >> R)) & M;
            L[v] = on ? x : L[v];
        }
    }
}

// Slots inside the matrix, rows <= m and columns <= n: step t of the loop body
// (t odd: an even step) has row m at mt - ceil(t / 2) and the first column at
// dn + floor(t / 2).
template <int G, int V, int R>
__device__ __forceinline__ void matrix_bounds(const DState<V>& u,
                                              uint32_t (&inm)[Diag<G, V, R>::UNROLL][V]) {
    using D = Diag<G, V, R>;
#pragma unroll
    for (int t = 0; t < D::UNROLL; ++t)
#pragma unroll
        for (int v = 0; v < V; ++v) inm[t][v] = FULL;
    if (__any_sync(FULL, u.mt < D::C + D::UNROLL / 2 || u.dn > -D::UNROLL / 2)) {
#pragma unroll
        for (int t = 0; t < D::UNROLL; ++t)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int k0 = __viaddmin_s32_relu(u.dn, t / 2 - v * D::VR, D::VR);
                const int k1 = __viaddmin_s32_relu(u.mt, 1 - (t + 1) / 2 - v * D::VR, D::VR);
                inm[t][v] = __funnelshift_lc(~0u, 0u, k1) & ~__funnelshift_lc(~0u, 0u, k0);
            }
    }
}

}  // namespace

}  // namespace logan
