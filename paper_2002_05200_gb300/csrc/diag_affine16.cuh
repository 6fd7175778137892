// X-drop extension with affine gaps (Gotoh's three states) in the packed 16-bit
// diagonal frame of diag16.cuh: shared by the affine DNA windows
// (xdrop_affine16.cu: bit-plane codes, match / mismatch) and the substitution
// matrix's (xdrop_matrix.cu: letters as bytes, a table in shared memory).
//
// Keys as in diag16.cuh with the base moving by the gap extension,
// B_d = B_{d-1} + ge, so extending a gap adds nothing and opening one adds
// KS * go.  Registers hold, per pair of slots, G = H + KS * go of the last even
// and odd anti-diagonals and E and F of the last one:
//   e = max(E, G)         of the left cell,  f = max(F, G) of the upper one,
//   t = G(d-2) + KS * (sub - 2 ge - go)      where the diagonal predecessor is
//                                            live and the slot in range,
//       G(d-2) or less                       elsewhere,
//   H = max(t, e, f),  G = H + KS * go.
// Nothing is pruned: as for linear gaps, a state below the threshold stays
// below it (every move but the masked diagonal is <= 0), and a slot outside
// the range has a dead cell on both sides, so a live diagonal predecessor D had
// D + go + ge < T_{d-1}: the masked diagonal, D + go + 2 ge, stays dead.  A live
// cell may keep an E or F that came from a dead one; it is below the
// threshold for good and never decides a live H.
// About 11.5 instructions per pair of cells with DNA codes (16.5 in the row-window
// form it replaced, which pruned all three states by selects), 19 and two
// shared loads with letters.
#pragma once

#include <algorithm>

#include "diag16.cuh"

namespace logan {

namespace {

// what a launch needs (by value)
struct DiagAffineArgs {
    const void* pa;        // 2-bit words or letter codes (bytes)
    const void* pb;
    const Item* items;
    ExtRes* ext;
    uint32_t* queues;      // queue q at queues + q * qcap
    uint32_t qcap;
    Counters* counters;
    int level, next_queue; // this launch's queue; where bands that outgrow it go
    int cells_level;       // counters->cells index credited, -1: none
    const int32_t* table;  // letters: K x K scores
    int K, sub_max, sub_min;
    int period;            // anti-diagonals between renormalisations
    int floor;             // smallest H, E, F
    int step;              // theta's growth per anti-diagonal: KS * -ge
    int go;                // KS * gap_open (<= 0)
    uint32_t cb[6], cf[6]; // a mask bit at position p: base, match - mismatch (key units / 2^p)
};

// Bounds (mp the largest substitution or 0, lo the smallest, D the growth of
// theta over `period` steps): live keys below 65536; every value and every
// masked diagonal at or above 0; live keys, also after a worst
// substitution, above the floor.
inline bool diag_affine_plan(int64_t sub_max, int64_t sub_min, int go, int ge, int64_t xmax,
                             DiagAffineArgs* a) {
    const int64_t g = -int64_t(ge), o = -int64_t(go), mp = sub_max > 0 ? sub_max : 0;
    const int64_t am = sub_min < 0 ? -sub_min : 0;
    for (int period = kPrefetch; period >= 4; period >>= 1) {
        const int64_t grow = period * g + mp * (period / 2 + 1);
        const int64_t floor = KS * std::max(grow, o + (sub_max - sub_min) + 1) + 64;
        if (KS * (grow + xmax + mp + 1) + 32 > 32767 ||
            floor + KS * (2 * g + 2 * mp + 2) > 32767 ||
            KS * (am + 2 * g + 2 * mp + 2) + 64 > 32767)
            continue;
        a->period = period;
        a->floor = int(floor);
        a->step = int(KS * g);
        a->go = int(-KS * o);
        return true;
    }
    return false;
}

// letter of stream index q (0 outside [0, len))
__device__ __forceinline__ uint32_t letter_at(const uint8_t* __restrict__ pool, int64_t pos, int dir,
                                              int len, int q) {
    if (q < 0 || q >= len) return 0u;
    return pool[pos + (dir > 0 ? q : -q)];
}

// letters of stream indices q .. q+3 (BACK: q .. q-3), the first in the low byte
template <bool BACK>
__device__ __forceinline__ uint32_t letters4(const uint8_t* __restrict__ pool, int64_t pos, int dir,
                                             int len, int q) {
    uint32_t w = 0u;
#pragma unroll
    for (int t = 0; t < 4; ++t) w |= letter_at(pool, pos, dir, len, BACK ? q - t : q + t) << (8 * t);
    return w;
}

// a lane's letters: a' and b' (doubled, as table byte offsets) of its slots,
// and those that enter in the next 16 steps
template <int R>
struct Letters {
    uint32_t a[R / 2], b[R / 2], na[2], nb[2];
};

template <int G, int R>
__device__ __forceinline__ void load_next_letters(const DiagAffineArgs& x, const Item& it,
                                                  const DState<1>& u, int gl, Letters<R>& l) {
    using D = Diag<G, 1, R>;
    const int dir = (it.flags & ITEM_LEFT) ? -1 : 1;
    const int s0 = u.base + gl * D::C;
    const uint8_t* pa = static_cast<const uint8_t*>(x.pa);
    const uint8_t* pb = static_cast<const uint8_t*>(x.pb);
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        l.na[w] = letters4<false>(pa, it.a_pos, dir, int(it.m), s0 + D::VR + u.e - 1 + 4 * w);
        // the first to enter in the top byte
        l.nb[w] = __byte_perm(letters4<false>(pb, it.b_pos, dir, int(it.n), u.e - u.phi - s0 + 4 * w), 0u,
                              0x0123)
                  << 1;
    }
}

template <int G, int R>
__device__ __forceinline__ void load_letters(const DiagAffineArgs& x, const Item& it,
                                             const DState<1>& u, int gl, Letters<R>& l) {
    using D = Diag<G, 1, R>;
    const int dir = (it.flags & ITEM_LEFT) ? -1 : 1;
    const int s0 = u.base + gl * D::C;
#pragma unroll
    for (int w = 0; w < R / 2; ++w) {
        l.a[w] = letters4<false>(static_cast<const uint8_t*>(x.pa), it.a_pos, dir, int(it.m),
                                 s0 + 4 * w + u.e - 1);
        l.b[w] = letters4<true>(static_cast<const uint8_t*>(x.pb), it.b_pos, dir, int(it.n),
                                u.e - 1 - u.phi - s0 - 4 * w)
                 << 1;
    }
    load_next_letters<G, R>(x, it, u, gl, l);
}

// the 2-bit loaders of diag16.cuh take the pools from KernelArgs
__device__ __forceinline__ KernelArgs word_pools(const DiagAffineArgs& x) {
    KernelArgs ka;
    ka.wa = static_cast<const uint32_t*>(x.pa);
    ka.wb = static_cast<const uint32_t*>(x.pb);
    return ka;
}

template <int G, int R, bool LETTERS>
__device__ __forceinline__ void load_codes(const DiagAffineArgs& x, const Item& it, DState<1>& u, int gl,
                                           Letters<R>& l) {
    if constexpr (LETTERS) load_letters<G, R>(x, it, u, gl, l);
    else load_planes<G, 1, R>(word_pools(x), it, u, gl);
}

template <int G, int R, bool LETTERS>
__device__ __forceinline__ void affine_start(const DiagAffineArgs& x, DState<1>& u, uint32_t id, int gl,
                                             Letters<R>& l, uint32_t (&GE)[R], uint32_t (&GO)[R],
                                             uint32_t (&E)[R], uint32_t (&F)[R]) {
    using D = Diag<G, 1, R>;
    const Item it = x.items[id];
    u.item = id;
    u.X = it.X;
    u.c32 = 0u;
    u.theta = 32768 + x.step;
    u.phi = u.e = 0;
    u.base = -D::W / 2;
    u.best = u.bd = u.br = 0;
    u.cells = u.cells0 = 0ull;
    const uint32_t f2 = uint32_t(x.floor) * 0x10001u, g2 = uint32_t(x.floor + x.go) * 0x10001u;
#pragma unroll
    for (int h = 0; h < R; ++h) {
        GE[h] = GO[h] = g2;
        E[h] = F[h] = f2;
    }
    u.LE[0] = u.LO[0] = 0u;
    if (gl == G / 2) {  // S(0,0) = 0, X above its threshold, no gap state
        GE[0] = (g2 & 0xffff0000u) | uint32_t(int(live_key<D::VR>(it.X, 0)) + x.go);
        u.LE[0] = 1u;
    }
    const int off = u.base + gl * D::C;
    u.dn = 1 - int(it.n) - off;
    u.mt = int(it.m) - off;
    load_codes<G, R, LETTERS>(x, it, u, gl, l);
    u.active = true;
    u.done = u.overflow = u.migrated = false;
}

// One anti-diagonal of every unit of the warp: Q (G of d-2 on entry) receives
// G of d, P holds G of d-1, E and F move from d-1 to d.
template <int G, int R, bool LETTERS, bool ODD>
__device__ __forceinline__ uint32_t affine_step(const DiagAffineArgs& x, const uint16_t* tab,
                                                DState<1>& u, int at, int gl, const Lanes<G>& ln,
                                                uint32_t inm, Letters<R>& l, uint32_t (&Q)[R],
                                                const uint32_t (&P)[R], uint32_t (&E)[R],
                                                uint32_t (&F)[R]) {
    using D = Diag<G, 1, R>;
    constexpr int VR = D::VR, C = D::C, H2 = R / 2;
    const uint32_t f2 = uint32_t(x.floor) * 0x10001u;
    const uint32_t rb = u.rb[0] & inm;
    u.c32 += uint32_t(__popc(rb));
    uint32_t rm = rb & (ODD ? u.LO[0] : u.LE[0]), fm = 0u;
    if constexpr (LETTERS) {
        if constexpr (ODD) {  // b' one slot up
#pragma unroll
            for (int w = R / 2 - 1; w >= 1; --w) l.b[w] = __funnelshift_l(l.b[w - 1], l.b[w], 8);
            l.b[0] = __funnelshift_l(l.nb[0], l.b[0], 8);
            l.nb[0] = __funnelshift_l(l.nb[1], l.nb[0], 8);
            l.nb[1] <<= 8;
        } else {  // a' one slot down
#pragma unroll
            for (int w = 0; w < R / 2 - 1; ++w) l.a[w] = __funnelshift_r(l.a[w], l.a[w + 1], 8);
            l.a[R / 2 - 1] = __funnelshift_r(l.a[R / 2 - 1], l.na[0], 8);
            l.na[0] = __funnelshift_r(l.na[0], l.na[1], 8);
            l.na[1] >>= 8;
        }
    } else {
        if constexpr (ODD) {
            u.b0[0] = __funnelshift_l(u.nb0, u.b0[0], 1);
            u.b1[0] = __funnelshift_l(u.nb1, u.b1[0], 1);
            u.nb0 <<= 1;
            u.nb1 <<= 1;
        } else {
            u.a0[0] = __funnelshift_r(u.a0[0], u.na0, 1);
            u.a1[0] = __funnelshift_r(u.a1[0], u.na1, 1);
            u.na0 >>= 1;
            u.na1 >>= 1;
        }
        fm = rm & ~(u.a0[0] ^ u.b0[0]);
        fm = fm & ~(u.a1[0] ^ u.b1[0]);
    }
    // slot h + R of register h to bit h + 16 (for R < 8 the bits between hold
    // copies that no register's mask picks)
    if constexpr (R == 8) {
        rm = __byte_perm(rm, 0u, 0x4140);
        fm = __byte_perm(fm, 0u, 0x4140);
    } else if constexpr (R < 8) {
        rm *= 1u + (1u << (16 - R));
        fm *= 1u + (1u << (16 - R));
    }
    const uint32_t rm6 = rm >> 6, rm12 = rm >> 12, fm6 = fm >> 6, fm12 = fm >> 12;
    // the shifted gap state (odd: vertical, from the slot below; even: horizontal,
    // from the slot above): the values that the loop overwrites first
    uint32_t (&S)[R] = ODD ? F : E;
    const uint32_t s_mid = ODD ? __vimax3_u16x2(S[H2 - 1], P[H2 - 1], 0u) : __vimax3_u16x2(S[H2], P[H2], 0u);
    const uint32_t s_end = ODD ? __vimax3_u16x2(S[R - 1], P[R - 1], 0u) : __vimax3_u16x2(S[0], P[0], 0u);
    uint32_t edge = f2;
    if constexpr (G > 1) {
        edge = ODD ? __shfl_up_sync(FULL, s_end, 1, G) : __shfl_down_sync(FULL, s_end, 1, G);
        edge = (ODD ? gl == 0 : gl == G - 1) ? f2 : edge;
    }
    const uint32_t thr = uint32_t(32768 - u.theta) * 0x10001u;
    const uint32_t go2 = uint32_t(x.go) * 0x10001u;
    const uint32_t neg2 = uint32_t(-KS * (x.sub_max - x.sub_min)) * 0x10001u;
    uint32_t lk = 0u;
    SignMask<R> live;
#pragma unroll
    for (int jj = 0; jj < H2; ++jj) {
        const int j = ODD ? H2 - 1 - jj : jj;
        uint32_t xs[2], hh[2];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int h = j + half * H2;
            // the gap state whose predecessor sits in the same slot
            uint32_t (&T)[R] = ODD ? E : F;
            T[h] = __vimax3_u16x2(T[h], P[h], 0u);
            uint32_t s;
            if constexpr (ODD) {
                if (h == 0) s = __byte_perm(edge, s_end, 0x5432) - 0x00010001u + uint32_t(VR);
                else s = (h == H2 ? s_mid : __vimax3_u16x2(S[h - 1], P[h - 1], 0u)) - 0x00010001u;
            } else {
                if (h == R - 1) s = __byte_perm(s_end, edge, 0x5432) + 0x00010001u - (uint32_t(VR) << 16);
                else s = (h == H2 - 1 ? s_mid : __vimax3_u16x2(S[h + 1], P[h + 1], 0u)) + 0x00010001u;
            }
            S[h] = s;
            const int p = h % 6;
            const uint32_t wr = h < 6 ? rm : h < 12 ? rm6 : rm12;
            uint32_t t;
            if constexpr (LETTERS) {
                // slots h and h + R: their letters as halves, both table offsets
                // in one multiply-add, two 16-bit loads
                constexpr int B = R / 4 > 0 ? R / 4 : 1;  // words between them (R = 2: the same word)
                const int w0 = h >> 2, w1 = R >= 4 ? w0 + B : 0;
                const uint32_t pick = uint32_t(h & 3) | (uint32_t(((h + R) & 3) + 4) << 4);
                const uint32_t la = __byte_perm(__byte_perm(l.a[w0], l.a[w1], pick), 0u, 0x4140);
                const uint32_t lb = __byte_perm(__byte_perm(l.b[w0], l.b[w1], pick), 0u, 0x4140);
                const uint32_t idx = la * 64u + lb;
                const char* tb = reinterpret_cast<const char*>(tab);
                const uint32_t s0 = *reinterpret_cast<const uint16_t*>(tb + (idx & 0xffffu));
                const uint32_t s1 = *reinterpret_cast<const uint16_t*>(tb + (idx >> 16));
                t = (wr & (0x00010001u << p)) * x.cb[p] + Q[h];
                t = t + (s1 * 65536u + s0) + neg2;
            } else {
                const uint32_t wf = h < 6 ? fm : h < 12 ? fm6 : fm12;
                t = (wf & (0x00010001u << p)) * x.cf[p] + Q[h];
                t = (wr & (0x00010001u << p)) * x.cb[p] + t;
            }
            hh[half] = __vimax3_u16x2(T[h], s, t);
            xs[half] = hh[half] + thr;
            Q[h] = hh[half] + go2;
        }
        lk = __vimax3_u16x2(lk, hh[0], hh[1]);
        live.add(j, xs[0], xs[1]);
    }
    uint32_t L[1] = {live.get() & rb};
    if constexpr (ODD) u.LO[0] = L[0];
    else u.LE[0] = L[0];
    const uint32_t key = max(lk & 0xffffu, lk >> 16);
    // a new best and the first lane that has it
    const int above = int(key) - u.theta;
    const uint32_t mine_u = above >= 0 ? uint32_t(above) >> LOG2KS : 0u;
    const uint32_t top = unit_max_u32<G>(mine_u);
    const int gain = max(int(top) - u.X, 0);
    const bool hit = gain > 0 && mine_u == top;
    const uint32_t vote = __ballot_sync(FULL, hit);
    const bool mine = hit && (vote & ln.below) == 0u;
    u.bd = mine ? 2 * (u.e + at) + (ODD ? 1 : 2) : u.bd;
    u.br = mine ? u.base + gl * C + VR - 1 - int(key & uint32_t(VR - 1)) : u.br;
    u.best += gain;
    u.theta += gain * KS + x.step;
    return next_range<G, 1, R, ODD>(L, ln, u.rb);
}

template <int G, int R, bool LETTERS>
__global__ void __launch_bounds__(128, R >= 8 ? 3 : 4) k_diag_affine(DiagAffineArgs x) {
    using D = Diag<G, 1, R>;
    constexpr int VR = D::VR;
    __shared__ uint16_t tab[LETTERS ? 32 * 32 : 1];
    if constexpr (LETTERS) {
        // KS (M - min M), rows of 32 letters
        for (int t = threadIdx.x; t < 32 * 32; t += blockDim.x) {
            const int a = t >> 5, b = t & 31;
            tab[t] = a < x.K && b < x.K ? uint16_t((x.table[a * x.K + b] - x.sub_min) * KS) : uint16_t(0);
        }
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int gl = lane % G, unit = lane / G;
    const Lanes<G> ln(lane);
    const uint32_t* q = x.queues + size_t(x.level) * x.qcap;
    const uint32_t f2 = uint32_t(x.floor) * 0x10001u, g2 = uint32_t(x.floor + x.go) * 0x10001u;
    uint32_t GE[R], GO[R], E[R], F[R];
#pragma unroll
    for (int h = 0; h < R; ++h) {
        GE[h] = GO[h] = g2;
        E[h] = F[h] = f2;
    }
    Letters<R> l{};
    DState<1> u;
    u.dn = u.mt = 0;
    u.theta = 32768;
    u.best = u.bd = u.br = u.X = 0;
    u.base = u.e = u.phi = 0;
    u.c32 = 0u;
    u.cells = u.cells0 = 0ull;
    u.item = 0u;
    u.active = u.done = u.overflow = u.migrated = false;
    u.rb[0] = u.LE[0] = u.LO[0] = u.a0[0] = u.a1[0] = u.b0[0] = u.b1[0] = 0u;
    u.na0 = u.na1 = u.nb0 = u.nb1 = 0u;
    constexpr uint32_t bot = (1u << (D::UNROLL / 2)) - 1u, tops = bot << (VR - D::UNROLL / 2);
    const uint32_t brink_bot = gl == 0 ? bot : 0u, brink_top = gl == G - 1 ? tops : 0u;
    const int iters = x.period / D::UNROLL;
    int left = iters, fetch = 16 / D::UNROLL;
    bool exhausted = false, first_wave = true;
    uint32_t vote = 0u;
    for (;;) {
        if (u.active && (vote & ln.all) == 0u) {
            u.active = false;
            u.done = true;
        }
        const bool slide = __any_sync(FULL, (u.LE[0] & (brink_top | brink_bot)) != 0u);
        if (__builtin_expect(slide, 0)) {
            const bool at_top = (__ballot_sync(FULL, (u.LE[0] & brink_top) != 0u) & ln.all) != 0u;
            const bool at_bot = (__ballot_sync(FULL, (u.LE[0] & brink_bot) != 0u) & ln.all) != 0u;
            // live slots that the shifted window would lose or have on its brink
            uint32_t low, high;
            if constexpr (D::SL > 0) {
                low = gl < D::SL ? D::VMASK : gl == D::SL ? bot : 0u;
                high = gl >= G - D::SL ? D::VMASK : gl == G - D::SL - 1 ? tops : 0u;
            } else {
                low = brink_bot ? (bot << R) | ((1u << R) - 1u) : 0u;
                high = brink_top ? (tops >> R) | (((1u << R) - 1u) << R) : 0u;
            }
            const bool in_low = (__ballot_sync(FULL, (u.LE[0] & low) != 0u) & ln.all) != 0u;
            const bool in_high = (__ballot_sync(FULL, (u.LE[0] & high) != 0u) & ln.all) != 0u;
            const bool ovf = u.active && ((at_top && in_low) || (at_bot && in_high));
            const bool up = u.active && at_top && !ovf, dn = u.active && at_bot && !ovf;
            if (__any_sync(FULL, up)) {
                shift_slots<G, 1, R, true>(GE, up, gl, g2);
                shift_slots<G, 1, R, true>(GO, up, gl, g2);
                shift_slots<G, 1, R, true>(E, up, gl, f2);
                shift_slots<G, 1, R, true>(F, up, gl, f2);
                shift_mask<G, 1, R, true>(u.LE, up, gl);
                shift_mask<G, 1, R, true>(u.LO, up, gl);
            }
            if (__any_sync(FULL, dn)) {
                shift_slots<G, 1, R, false>(GE, dn, gl, g2);
                shift_slots<G, 1, R, false>(GO, dn, gl, g2);
                shift_slots<G, 1, R, false>(E, dn, gl, f2);
                shift_slots<G, 1, R, false>(F, dn, gl, f2);
                shift_mask<G, 1, R, false>(u.LE, dn, gl);
                shift_mask<G, 1, R, false>(u.LO, dn, gl);
            }
            if (up || dn) {
                const int by = up ? D::SLIDE : -D::SLIDE;
                u.base += by;
                u.dn -= by;
                u.mt -= by;
                load_codes<G, R, LETTERS>(x, x.items[u.item], u, gl, l);
            }
            if (ovf) {  // restarts in the next window
                u.active = false;
                u.done = true;
                u.overflow = true;
                u.LE[0] = u.LO[0] = 0u;
            }
        }
        const bool turn = __any_sync(FULL, u.done || (!u.active && !exhausted));
        if (__builtin_expect(turn, 0)) {
            int bd = u.bd, br = u.br;
            unsigned long long cells = u.cells + u.c32;
#pragma unroll
            for (int o = G / 2; o >= 1; o >>= 1) {
                const int d = __shfl_xor_sync(FULL, bd, o, G), r = __shfl_xor_sync(FULL, br, o, G);
                cells += __shfl_xor_sync(FULL, cells, o, G);
                br = d > bd ? r : br;
                bd = d > bd ? d : bd;
            }
            if (u.done && gl == 0) {
                if (u.overflow) {
                    const unsigned int t = atomicAdd(&x.counters->tail[x.next_queue], 1u);
                    x.queues[size_t(x.next_queue) * x.qcap + t] = u.item;
                } else {
                    ExtRes r;
                    r.best = u.best;
                    r.bi = u.best > 0 ? br + (bd >> 1) : 0;
                    r.bj = u.best > 0 ? bd - r.bi : 0;
                    r.status = 0;
                    r.cells = cells;
                    x.ext[u.item] = r;
                    if (x.cells_level >= 0) atomicAdd(&x.counters->cells[x.cells_level], cells);
                }
            }
            u.done = false;
            const bool need = !u.active && !exhausted;
            uint32_t id = 0xffffffffu;
            const uint32_t want = __ballot_sync(FULL, need && gl == 0);
            if (want) {
                // windows run one after another, so a window's queue is complete
                unsigned int limit = 0u;
                const unsigned int slot = pop_unit_slot<G>(x.counters, x.level, PHASE_WHOLE, want, lane,
                                                           unit, first_wave, limit);
                if (need && slot < limit) id = q[slot];
            }
            if (need) {
                if (id != 0xffffffffu) affine_start<G, R, LETTERS>(x, u, id, gl, l, GE, GO, E, F);
                else exhausted = true;
            }
            if (!__any_sync(FULL, u.active)) break;
        }
        if (__builtin_expect(slide || turn, 0)) next_range<G, 1, R, false>(u.LE, ln, u.rb);
        uint32_t inm[D::UNROLL][1];
        matrix_bounds<G, 1, R>(u, inm);
#pragma unroll
        for (int t = 0; t < D::UNROLL; t += 2) {
            affine_step<G, R, LETTERS, true>(x, tab, u, t / 2, gl, ln, inm[t][0], l, GO, GE, E, F);
            vote = affine_step<G, R, LETTERS, false>(x, tab, u, t / 2, gl, ln, inm[t + 1][0], l, GE, GO, E, F);
        }
        u.e += D::UNROLL / 2;
        u.dn += D::UNROLL / 2;
        u.mt -= D::UNROLL / 2;
        if (LETTERS && --fetch == 0) {
            fetch = 16 / D::UNROLL;
            if (u.active) load_next_letters<G, R>(x, x.items[u.item], u, gl, l);
        }
        if (--left == 0) {
            left = iters;
            u.cells += u.c32;
            u.c32 = 0u;
            if (u.active) {
                // theta back to 32768, states clamped at the floor
                const uint32_t sub = uint32_t(u.theta - 32768) * 0x10001u;
#pragma unroll
                for (int h = 0; h < R; ++h) {
                    GE[h] = __vimax3_u16x2(GE[h], sub + g2, 0u) - sub;
                    GO[h] = __vimax3_u16x2(GO[h], sub + g2, 0u) - sub;
                    E[h] = __vimax3_u16x2(E[h], sub + f2, 0u) - sub;
                    F[h] = __vimax3_u16x2(F[h], sub + f2, 0u) - sub;
                }
                u.theta = 32768;
                if constexpr (!LETTERS) load_next<G, 1, R>(word_pools(x), x.items[u.item], u, gl);
            }
        }
    }
}

}  // namespace

}  // namespace logan
