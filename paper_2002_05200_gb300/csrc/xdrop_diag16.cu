// X-drop extension with linear gaps, G-lane units and the band packed two
// cells to a 32-bit register (16-bit SIMD) in diagonal coordinates, for window
// levels whose score range provably fits 16 bits.
//
// Method: the paper's recurrence and X-drop rule (Sec. III-A), the
// anti-diagonal sweep of Algorithm 1 with the cell update of Algorithm 2,
// and the per-anti-diagonal maximum of Sec. IV-A -- the same computation as
// the 32-bit G-lane kernel (xdrop_group.cu), with the same results.  The
// frame, the keys and why the live cells are exact: diag16.cuh.
//
// A unit is G lanes of V virtual lanes of 2 R slots (32 / G extensions per
// warp).  The host enables a level when, with mp = max(match, 0), some period
// K in {64, 32, 16, 8, 4} and D = K |gap| + mp (K / 2 + 1) (what theta can grow
// by in K steps),
//     KS * (D + X + mp + 1) + 32        <= 32767   (live keys stay below 65536)
//     KS * (D + 2 |gap| + 2 mp + 2) + 64 <= 32767  (live keys stay above the floor)
//     KS * (max(-mismatch, 0) + 2 mp + 2) + 64 <= 32767  (a substitution from a
//                                       live key stays at or above 0)
// (diag_plan.h).
// Then every half-word stays inside [0, 65536) through every addition, and an
// addition of both halves is one 32-bit operation.
//
// Bound by the ALU pipe and issue together: about 7 instructions per pair of
// cells and 90 of bookkeeping per lane and anti-diagonal (level 2: 206 per
// warp and anti-diagonal, 79 % of issue slots, ALU pipe 79 %).  The
// bookkeeping has no numbers to reduce: ranges pass between anti-diagonals as
// masks and two votes, the best as one vote and a note in the lane that has
// it, cells as population counts, all summed when the extension ends.
// 100,000 lognormal pairs, X = 100: level 2 (137e9 cells) 83 ms in the
// row-window form this replaced, 52 with lo / hi / best reduced by shuffles,
// 47 now; level 5 (105e9) 52, 44, 41; the whole call 182, 123, 113 ms.
//
// Latency forms: a lone extension waits for its own chain, so short lanes
// (4 to 16 slots) cut the instructions per anti-diagonal: 112 with 4 slots per
// lane, 140 ns per anti-diagonal on an idle SM (175 ns in the 32-bit one-warp
// form).
#include <algorithm>

#include "diag16.cuh"

namespace logan {

namespace {

// (FRESH: from the extension's start, whatever records exist)
template <int G, int V, int R, bool FRESH = false>
__device__ __forceinline__ void unit_start(const KernelArgs& ka, const DiagArgs& da, DState<V>& u,
                                           uint32_t id, int gl, uint32_t (&QE)[V * R],
                                           uint32_t (&QO)[V * R]) {
    using D = Diag<G, V, R>;
    const Item it = ka.items[id];
    u.item = id;
    u.X = it.X;
    u.c32 = 0u;
    u.theta = 32768;
    bool fits = true;
    const int32_t* rec = nullptr;
    if constexpr (!FRESH) {
        const int32_t slot = ka.mig_slot[id];
        if (slot >= 0) rec = mig_record(ka, slot);
    }
    if (rec && rec[MIG_KIND] == MIG_RELATIVE) {
        // resume a band saved by a narrower level
        const int rows = rec[MIG_ROWS], d = rec[MIG_D], row0 = rec[MIG_BASE];
        const int lo = rec[MIG_LO], hi = rec[MIG_HI];
        u.phi = (d & 1) ? 0 : 1;
        u.e = (d + u.phi - 1) >> 1;
        u.base = ((lo + hi) >> 1) - u.e - D::W / 2;
        u.best = rec[MIG_BEST];
        u.bd = rec[MIG_BI] + rec[MIG_BJ];
        u.br = rec[MIG_BI] - ((u.bd + u.phi) >> 1);
        u.cells0 = (unsigned long long)uint32_t(rec[MIG_CELLS_LO]) |
                   ((unsigned long long)uint32_t(rec[MIG_CELLS_HI]) << 32);
        // d-1 (even) relative to T1, d-2 (odd) relative to T2, onto theta = 32768
        const int c1 = rec[MIG_T1] - rec[MIG_T] + da.gap;
        const int c2 = rec[MIG_T2] - rec[MIG_T] + 2 * da.gap;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            uint32_t le = 0u, lo_ = 0u;
#pragma unroll
            for (int h = 0; h < R; ++h) {
                uint32_t q1 = 0u, q2 = 0u;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const int k = h + R * half;
                    const int r1 = u.base + gl * D::C + v * D::VR + k + u.e - row0;  // d-1: frame e
                    const int r2 = r1 - 1;                                           // d-2: frame e-1
                    const int v1 = (r1 >= 0 && r1 < rows) ? rec[kMigHeader + r1] : NEGU;
                    const int v2 = (r2 >= 0 && r2 < rows) ? rec[kMigHeader + rows + r2] : NEGU;
                    q1 |= (v1 >= 0 ? live_key<D::VR>(v1 + c1, k) : uint32_t(da.floor)) << (16 * half);
                    q2 |= (v2 >= 0 ? live_key<D::VR>(v2 + c2, k) : uint32_t(da.floor)) << (16 * half);
                    le |= (v1 >= 0 ? 1u : 0u) << k;
                    lo_ |= (v2 >= 0 ? 1u : 0u) << k;
                }
                QE[v * R + h] = q1;
                QO[v * R + h] = q2;
            }
            u.LE[v] = le;
            u.LO[v] = lo_;
        }
        // a record as wide as this window (levels whose forms share one) stays
        // as it is for the next level
        const int first = u.base + u.e;
        fits = lo - first >= D::UNROLL / 2 && hi - first < D::W - D::UNROLL / 2;
    } else {
        // S(0,0) = 0 on d = 0 (even), X above its threshold, mid-window
        u.phi = 0;
        u.e = 0;
        u.base = -D::W / 2;
        u.best = u.bd = u.br = 0;
        u.cells0 = 0ull;
        const uint32_t f2 = uint32_t(da.floor) * 0x10001u;
#pragma unroll
        for (int h = 0; h < V * R; ++h) QE[h] = QO[h] = f2;
#pragma unroll
        for (int v = 0; v < V; ++v) u.LE[v] = u.LO[v] = 0u;
        if (gl == G / 2) {  // slot W / 2 is the first of this lane
            static_assert(G > 1, "lanes");
            QE[0] = (f2 & 0xffff0000u) | live_key<D::VR>(it.X, 0);
            u.LE[0] = 1u;
        }
        u.theta += KS * -da.gap;  // theta_1
    }
    u.cells = 0ull;
    const int off = u.base + u.e + gl * D::C;
    u.dn = 2 * u.e + 1 - u.phi - int(it.n) - off;
    u.mt = int(it.m) - off;
    load_planes<G, V, R>(ka, it, u, gl);
    u.active = fits;
    u.done = !fits;
    u.overflow = !fits;
    u.migrated = false;
}

// The unit's last best cell (its lanes' latest) and the cells of this level.
template <int G, int V>
__device__ __forceinline__ void unit_totals(const DState<V>& u, int& bd, int& br,
                                            unsigned long long& cells) {
    bd = u.bd;
    br = u.br;
    cells = u.cells + u.c32;
#pragma unroll
    for (int o = G / 2; o >= 1; o >>= 1) {
        const int d = __shfl_xor_sync(FULL, bd, o, G), r = __shfl_xor_sync(FULL, br, o, G);
        cells += __shfl_xor_sync(FULL, cells, o, G);
        if (d > bd) {  // (equal ones are copies of the cell the unit started with)
            bd = d;
            br = r;
        }
    }
}

// Result or escalation of the finished units (their leader lanes write).
template <int G, int V>
__device__ __forceinline__ void units_end(const KernelArgs& ka, DState<V>& u, int level, int gl,
                                          bool twin) {
    int bd, br;
    unsigned long long cells;
    unit_totals<G, V>(u, bd, br, cells);
    if (!u.done || gl != 0) return;
    if (u.overflow) {
        if (u.migrated) atomicAdd(&ka.counters->cells[level], cells);
        const int nq = escalate_queue(ka, level, twin);
        const unsigned int t = atomicAdd(&ka.counters->tail[nq], 1u);
        ka.queues[size_t(nq) * ka.qcap + t] = u.item;
    } else {
        ExtRes r;
        r.best = u.best;
        r.bi = br + ((bd + u.phi) >> 1);
        r.bj = bd - r.bi;
        r.status = 0;
        r.cells = u.cells0 + cells;
        ka.ext[u.item] = r;
        // (the item's record, if it had one, has been read) the level whose
        // window held the band to the end: the recording sweep of the
        // alignment paths uses the same
        ka.mig_slot[u.item] = int32_t((unsigned(level) << 24) | kMigFinal);
        atomicAdd(&ka.counters->cells[level], cells);
    }
}

// Saves an overflowing band for the next level: rows [row0, row0 + rows) of
// d-1 (even, frame e) and d-2 (odd, frame e-1) as scores above T_d - 2 mp,
// which no live cell of d-2 or d-1 lies below.
template <int G, int V, int R>
__device__ __forceinline__ void save_band(const KernelArgs& ka, const DiagArgs& da, DState<V>& u,
                                          int32_t slot, int level, int gl, int lo, int hi, int bd,
                                          int br, unsigned long long cells,
                                          const uint32_t (&QE)[V * R], const uint32_t (&QO)[V * R]) {
    using D = Diag<G, V, R>;
    int32_t* rec = mig_record(ka, slot);
    const int first = u.base + u.e;       // row of slot 0 on d-1
    const int row0 = max(first, 0);
    const int rows = first + D::W - row0;
    const int ref = 2 * da.mp;
    const int c1 = -da.gap + ref, c2 = -2 * da.gap + ref;
#pragma unroll
    for (int v = 0; v < V; ++v) {
#pragma unroll
        for (int h = 0; h < R; ++h) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int k = h + R * half;
                const int r1 = first + gl * D::C + v * D::VR + k - row0, r2 = r1 - 1;
                const int v1 = int((QE[v * R + h] >> (16 * half)) & 0xffffu);
                const int v2 = int((QO[v * R + h] >> (16 * half)) & 0xffffu);
                if (r1 >= 0)
                    rec[kMigHeader + r1] = ((u.LE[v] >> k) & 1u) ? ((v1 - u.theta) >> LOG2KS) + c1 : NEGU;
                if (r2 >= 0)
                    rec[kMigHeader + rows + r2] =
                        ((u.LO[v] >> k) & 1u) ? ((v2 - u.theta) >> LOG2KS) + c2 : NEGU;
            }
        }
    }
    if (gl == 0) {
        rec[kMigHeader + rows + rows - 1] = NEGU;  // d-2 has no slot for the last row
        const int off = u.base + u.e;
        const int T = u.best - u.X;
        rec[MIG_KIND] = MIG_RELATIVE;
        rec[MIG_ROWS] = rows;
        rec[MIG_D] = 2 * u.e + 1 - u.phi;
        rec[MIG_BASE] = row0;
        rec[MIG_LO] = lo + off;
        rec[MIG_HI] = hi + off;
        rec[MIG_BEST] = u.best;
        rec[MIG_T] = T;
        rec[MIG_T1] = T - ref;
        rec[MIG_T2] = T - ref;
        const int bi = br + ((bd + u.phi) >> 1);
        rec[MIG_BI] = bi;
        rec[MIG_BJ] = bd - bi;
        const unsigned long long c = u.cells0 + cells;
        rec[MIG_CELLS_LO] = int32_t(uint32_t(c));
        rec[MIG_CELLS_HI] = int32_t(uint32_t(c >> 32));
        rec[MIG_LEVEL] = level;
        ka.mig_slot[u.item] = slot;
    }
}

// Loop top, before an odd step, when some unit's band touches its window's
// outermost slots (every two steps reach one slot further): the window slides by half a virtual lane, or overflows when the band does
// not fit.
// (KEEP = false: an overflowing unit keeps no record)
template <int G, int V, int R, bool KEEP = true>
__device__ __forceinline__ void units_slide(const KernelArgs& ka, const DiagArgs& da, DState<V>& u,
                                            int level, int gl, int unit, const Lanes<G>& ln,
                                            uint32_t brink_top, uint32_t brink_bot,
                                            uint32_t (&QE)[V * R], uint32_t (&QO)[V * R]) {
    using D = Diag<G, V, R>;
    constexpr int VR = D::VR;
    const uint32_t f2 = uint32_t(da.floor) * 0x10001u;
    const uint32_t Lf = u.LE[0], Ll = u.LE[V - 1];
    const bool at_top = (__ballot_sync(FULL, (Ll & brink_top) != 0u) & ln.all) != 0u;
    const bool at_bot = (__ballot_sync(FULL, (Lf & brink_bot) != 0u) & ln.all) != 0u;
    // live slots that the shifted window would lose or have on its brink
    uint32_t low, high;
    constexpr uint32_t bot = (1u << (D::UNROLL / 2)) - 1u, top = bot << (VR - D::UNROLL / 2);
    if constexpr (D::SL > 0) {
        low = gl < D::SL ? D::VMASK : gl == D::SL ? bot : 0u;
        high = gl >= G - D::SL ? D::VMASK : gl == G - D::SL - 1 ? top : 0u;
    } else {
        low = brink_bot ? (bot << R) | ((1u << R) - 1u) : 0u;
        high = brink_top ? (top >> R) | (((1u << R) - 1u) << R) : 0u;
    }
    const bool in_low = (__ballot_sync(FULL, (Lf & low) != 0u) & ln.all) != 0u;
    const bool in_high = (__ballot_sync(FULL, (Ll & high) != 0u) & ln.all) != 0u;
    const bool ovf = u.active && ((at_top && in_low) || (at_bot && in_high));
    const bool up = u.active && at_top && !ovf, dn = u.active && at_bot && !ovf;
    if (__any_sync(FULL, up)) {
        shift_slots<G, V, R, true>(QE, up, gl, f2);
        shift_slots<G, V, R, true>(QO, up, gl, f2);
        shift_mask<G, V, R, true>(u.LE, up, gl);
        shift_mask<G, V, R, true>(u.LO, up, gl);
    }
    if (__any_sync(FULL, dn)) {
        shift_slots<G, V, R, false>(QE, dn, gl, f2);
        shift_slots<G, V, R, false>(QO, dn, gl, f2);
        shift_mask<G, V, R, false>(u.LE, dn, gl);
        shift_mask<G, V, R, false>(u.LO, dn, gl);
    }
    if (up || dn) {
        const int by = up ? D::SLIDE : -D::SLIDE;
        u.base += by;
        u.dn -= by;
        u.mt -= by;
        load_planes<G, V, R>(ka, ka.items[u.item], u, gl);
    }
    if constexpr (!KEEP) {
        if (ovf) {
            u.active = false;
            u.done = true;
            u.overflow = true;
#pragma unroll
            for (int v = 0; v < V; ++v) u.LE[v] = u.LO[v] = 0u;
        }
    } else if (__any_sync(FULL, ovf)) {
        int32_t slot = -1;
        if (ovf && gl == 0) {
            if constexpr (R < 16 && D::W == level_window(2)) {
                // the 128-slot latency forms of levels 0-2 share a pool: an extension
                // that moves among them writes over its own record
                constexpr int pool = 2;
                const int32_t own = ka.mig_slot[u.item];
                slot = own >= 0 && (own >> 24) == pool ? own : mig_alloc(ka, pool);
            } else {
                slot = mig_alloc(ka, level);
            }
        }
        slot = __shfl_sync(FULL, slot, unit * G);
        // first and last live slots, the best cell, the cells
        int lo = D::W, hi = -1, bd, br;
        unsigned long long cells;
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (u.LE[v]) {
                lo = min(lo, gl * D::C + v * VR + __ffs(u.LE[v]) - 1);
                hi = gl * D::C + v * VR + 31 - __clz(u.LE[v]);
            }
#pragma unroll
        for (int o = G / 2; o >= 1; o >>= 1) {
            lo = min(lo, __shfl_xor_sync(FULL, lo, o, G));
            hi = max(hi, __shfl_xor_sync(FULL, hi, o, G));
        }
        unit_totals<G, V>(u, bd, br, cells);
        if (ovf) {
            if (slot >= 0)
                save_band<G, V, R>(ka, da, u, slot, level, gl, lo, hi, bd, br, cells, QE, QO);
            u.active = false;
            u.done = true;
            u.overflow = true;
            u.migrated = slot >= 0;
#pragma unroll
            for (int v = 0; v < V; ++v) u.LE[v] = u.LO[v] = 0u;
        }
    }
}

// Every `period` steps: theta back to 32768, values clamped at the floor, the
// next codes prefetched.
template <int G, int V, int R>
__device__ __forceinline__ void unit_maintain(const KernelArgs& ka, const DiagArgs& da,
                                              DState<V>& u, int gl, uint32_t (&QE)[V * R],
                                              uint32_t (&QO)[V * R]) {
    u.cells += u.c32;
    u.c32 = 0u;
    if (!u.active) return;
    const uint32_t sub = uint32_t(u.theta - 32768) * 0x10001u;
    const uint32_t lim = sub + uint32_t(da.floor) * 0x10001u;
#pragma unroll
    for (int h = 0; h < V * R; ++h) {
        QE[h] = __vimax3_u16x2(QE[h], lim, 0u) - sub;
        QO[h] = __vimax3_u16x2(QO[h], lim, 0u) - sub;
    }
    u.theta = 32768;
    load_next<G, V, R>(ka, ka.items[u.item], u, gl);
}

// One anti-diagonal of every unit of the warp: Q (d-2 on entry) receives d,
// P holds d-1; inm: the lane's slots inside the matrix.  Returns the warp's vote of lanes with a live slot.  Units without a
// range compute values without effects.
// REC: rec gets the masks of slots whose value came from the diagonal and, of
// the others, from the vertical predecessor (meaningful for live slots).
template <int G, int V, int R, bool UNIT, bool ODD, bool REC>
__device__ __forceinline__ uint32_t dstep(const DiagArgs& da, DState<V>& u, int at, int gl,
                                          const Lanes<G>& ln, const uint32_t (&inm)[V],
                                          uint32_t (&Q)[V * R], const uint32_t (&P)[V * R],
                                          uint32_t (&rec)[2 * V]) {
    using D = Diag<G, V, R>;
    constexpr int VR = D::VR, C = D::C;
    // the moving operand's codes
    if constexpr (ODD) {
#pragma unroll
        for (int v = V - 1; v >= 1; --v) {
            u.b0[v] = __funnelshift_l(u.b0[v - 1], u.b0[v], 1);
            u.b1[v] = __funnelshift_l(u.b1[v - 1], u.b1[v], 1);
        }
        u.b0[0] = __funnelshift_l(u.nb0, u.b0[0], 1);
        u.b1[0] = __funnelshift_l(u.nb1, u.b1[0], 1);
        u.nb0 <<= 1;
        u.nb1 <<= 1;
    } else {
#pragma unroll
        for (int v = 0; v < V - 1; ++v) {
            u.a0[v] = __funnelshift_r(u.a0[v], u.a0[v + 1], 1);
            u.a1[v] = __funnelshift_r(u.a1[v], u.a1[v + 1], 1);
        }
        u.a0[V - 1] = __funnelshift_r(u.a0[V - 1], u.na0, 1);
        u.a1[V - 1] = __funnelshift_r(u.a1[V - 1], u.na1, 1);
        u.na0 >>= 1;
        u.na1 >>= 1;
    }
    // the neighbour lane's edge register
    const uint32_t f2 = uint32_t(da.floor) * 0x10001u;
    uint32_t edge = f2;
    if constexpr (G > 1) {
        if constexpr (ODD) {
            edge = __shfl_up_sync(FULL, P[V * R - 1], 1, G);
            edge = gl == 0 ? f2 : edge;
        } else {
            edge = __shfl_down_sync(FULL, P[0], 1, G);
            edge = gl == G - 1 ? f2 : edge;
        }
    }
    // v >= theta  <=>  bit 15 of v + (32768 - theta)
    const uint32_t thr = uint32_t(32768 - u.theta) * 0x10001u;
    uint32_t key = 0u;  // the lane's largest key and its slot in the lane
    int key_slot = 0;
    uint32_t L[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        // slots in range, then those whose diagonal predecessor is live (rm),
        // then the matches among them (fm)
        const uint32_t rb = u.rb[v] & inm[v];
        u.c32 += uint32_t(__popc(rb));
        uint32_t rm = rb & (ODD ? u.LO[v] : u.LE[v]);
        uint32_t fm = rm & ~(u.a0[v] ^ u.b0[v]);
        fm = fm & ~(u.a1[v] ^ u.b1[v]);
        // slot h + R of register h to bit h + 16 (for R < 8 the bits between
        // hold copies that no register's mask picks)
        if constexpr (R == 8) {
            rm = __byte_perm(rm, 0u, 0x4140);
            fm = __byte_perm(fm, 0u, 0x4140);
        } else if constexpr (R < 8) {
            rm *= 1u + (1u << (16 - R));
            fm *= 1u + (1u << (16 - R));
        }
        uint32_t wa, wb;
        if constexpr (UNIT) {
            // bits (rm, fm) side by side: the diagonal adds base * (rm + 2 fm)
            wa = (rm & 0x55555555u) | ((fm << 1) & 0xaaaaaaaau);  // even registers
            wb = ((rm >> 1) & 0x55555555u) | (fm & 0xaaaaaaaau);  // odd registers
        } else {
            wa = rm;
            wb = fm;
        }
        const uint32_t wa6 = wa >> 6, wa12 = wa >> 12, wb6 = wb >> 6, wb12 = wb >> 12;
        uint32_t lk = 0u;
        SignMask<R> live, from_diag, from_up;
#pragma unroll
        for (int j = 0; j < R / 2; ++j) {
            uint32_t x[2], yd[2], yu[2];
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int h = j + half * (R / 2);
                const int g = v * R + h;
                // the shifted neighbour, its row code moved by one slot
                uint32_t sh;
                if constexpr (ODD) {
                    if (h) {
                        sh = P[g - 1] - 0x00010001u;
                    } else {
                        const uint32_t lower = v ? P[v * R - 1] : edge;
                        sh = __byte_perm(lower, P[v * R + R - 1], 0x5432) - 0x00010001u + uint32_t(VR);
                    }
                } else {
                    if (h < R - 1) {
                        sh = P[g + 1] + 0x00010001u;
                    } else {
                        const uint32_t upper = v < V - 1 ? P[(v + 1) * R] : edge;
                        sh = __byte_perm(P[v * R], upper, 0x5432) + 0x00010001u - (uint32_t(VR) << 16);
                    }
                }
                uint32_t t;
                if constexpr (UNIT) {
                    const int q = h & ~1, p = q % 6;  // bits (p, p + 1) of word q / 6
                    const uint32_t w = (h & 1) ? (q < 6 ? wb : q < 12 ? wb6 : wb12)
                                               : (q < 6 ? wa : q < 12 ? wa6 : wa12);
                    t = (w & (0x00030003u << p)) * da.cb[p] + Q[g];
                } else {
                    const int p = h % 6;
                    const uint32_t wr = h < 6 ? wa : h < 12 ? wa6 : wa12;
                    const uint32_t wf = h < 6 ? wb : h < 12 ? wb6 : wb12;
                    t = (wf & (0x00010001u << p)) * da.cf[p] + Q[g];
                    t = (wr & (0x00010001u << p)) * da.cb[p] + t;
                }
                if constexpr (REC) {
                    // which predecessor gave the maximum: the diagonal first, then
                    // the vertical one (keys differ by less than 32768 here)
                    const uint32_t gap2 = __vimax3_u16x2(P[g], sh, 0u);
                    yd[half] = t - gap2 + 0x80008000u;
                    yu[half] = (ODD ? sh - P[g] : P[g] - sh) + 0x80008000u;
                    Q[g] = __vimax3_u16x2(gap2, t, 0u);
                } else {
                    Q[g] = __vimax3_u16x2(P[g], sh, t);
                }
                x[half] = Q[g] + thr;
            }
            lk = __vimax3_u16x2(lk, Q[v * R + j], Q[v * R + j + R / 2]);
            live.add(j, x[0], x[1]);
            if constexpr (REC) {
                from_diag.add(j, yd[0], yd[1]);
                from_up.add(j, yu[0], yu[1]);
            }
        }
        L[v] = live.get() & rb;
        if constexpr (REC) {
            rec[2 * v] = from_diag.get();
            rec[2 * v + 1] = from_up.get();
        }
        const uint32_t lkey = max(lk & 0xffffu, lk >> 16);
        // (equal scores: the lower virtual lane's rows come first)
        const bool more = v == 0 || (lkey >> LOG2KS) > (key >> LOG2KS);
        key = more ? lkey : key;
        key_slot = more ? v * VR + VR - 1 - int(lkey & uint32_t(VR - 1)) : key_slot;
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        if constexpr (ODD) u.LO[v] = L[v];
        else u.LE[v] = L[v];
    }
    // a new best (S > best <=> S - T_d > X) and the first lane that has it;
    // slots outside the range never hold one
    int gain;
    bool mine;
    if constexpr (UNIT) {  // one match scores 1, so the best grows by 1 at most
        const bool hit = int(key) >= u.theta + KS * (u.X + 1);
        const uint32_t vote = __ballot_sync(FULL, hit);
        gain = (vote & ln.all) != 0u ? 1 : 0;
        mine = hit && (vote & ln.below) == 0u;
    } else {
        const int above = int(key) - u.theta;
        const uint32_t mine_u = above >= 0 ? uint32_t(above) >> LOG2KS : 0u;
        const uint32_t top = unit_max_u32<G>(mine_u);
        gain = max(int(top) - u.X, 0);
        const bool hit = gain > 0 && mine_u == top;
        const uint32_t vote = __ballot_sync(FULL, hit);
        mine = hit && (vote & ln.below) == 0u;
    }
    u.bd = mine ? 2 * (u.e + at) + (ODD ? 1 : 2) - u.phi : u.bd;
    u.br = mine ? u.base + gl * C + key_slot : u.br;
    u.best += gain;
    u.theta += gain * KS + da.step;
    return next_range<G, V, R, ODD>(L, ln, u.rb);
}

template <int V>
__device__ __forceinline__ void state_clear(DState<V>& u) {
    u.dn = u.mt = 0;
    u.theta = 32768;
    u.best = u.bd = u.br = u.X = 0;
    u.base = u.e = u.phi = 0;
    u.c32 = 0u;
    u.cells = u.cells0 = 0ull;
    u.item = 0u;
    u.active = u.done = u.overflow = u.migrated = false;
#pragma unroll
    for (int v = 0; v < V; ++v)
        u.rb[v] = u.LE[v] = u.LO[v] = u.a0[v] = u.a1[v] = u.b0[v] = u.b1[v] = 0u;
    u.na0 = u.na1 = u.nb0 = u.nb1 = 0u;
}

template <int G, int V, int R, bool UNIT>
__global__ void __launch_bounds__(128, 4)
    k_diag16(KernelArgs ka, DiagArgs da, int level, int queue, int phase) {
    const int lane = threadIdx.x & 31;
    const int gl = lane % G, unit = lane / G;
    using D = Diag<G, V, R>;
    const Lanes<G> ln(lane);
    const bool twin = queue != level;
    const uint32_t* q = ka.queues + size_t(queue) * ka.qcap;
    uint32_t QE[V * R], QO[V * R];
#pragma unroll
    for (int h = 0; h < V * R; ++h) QE[h] = QO[h] = 0u;
    DState<V> u;
    state_clear(u);
    // the outermost slots that the next D::UNROLL steps must find dead
    const uint32_t brink_bot = gl == 0 ? (1u << (D::UNROLL / 2)) - 1u : 0u;
    const uint32_t brink_top = gl == G - 1 ? ((1u << (D::UNROLL / 2)) - 1u) << (D::VR - D::UNROLL / 2) : 0u;
    bool exhausted = false;
    bool first_wave = true;  // the warp's first pop takes static slots
    const int iters = da.period / D::UNROLL;  // between renormalisations
    int left = iters;
    uint32_t vote = 0u;  // lanes with a live slot on the last (even) anti-diagonal
    for (;;) {
        if (u.active && (vote & ln.all) == 0u) {
            u.active = false;
            u.done = true;
        }
        const bool slide = __any_sync(FULL, (u.LE[V - 1] & brink_top) != 0u || (u.LE[0] & brink_bot) != 0u);
        if (__builtin_expect(slide, 0))
            units_slide<G, V, R>(ka, da, u, level, gl, unit, ln, brink_top, brink_bot, QE, QO);
        const bool turn = __any_sync(FULL, u.done || (!u.active && !exhausted));
        if (__builtin_expect(turn, 0)) {
            units_end<G, V>(ka, u, level, gl, twin);
            u.done = false;
            const bool need = !u.active && !exhausted;  // the same in all lanes of a unit
            uint32_t id = 0xffffffffu;
            // one pop per warp for all of its idle units
            const uint32_t want = __ballot_sync(FULL, need && gl == 0);
            if (want) {
                unsigned int limit = 0u;
                const unsigned int slot =
                    pop_unit_slot<G>(ka.counters, queue, phase, want, lane, unit, first_wave, limit);
                if (need && slot < limit) id = q[slot];
            }
            if (need) {
                if (id != 0xffffffffu) unit_start<G, V, R>(ka, da, u, id, gl, QE, QO);
                else exhausted = true;
            }
            if (!__any_sync(FULL, u.active || u.done)) break;
        }
        if (__builtin_expect(slide || turn, 0)) next_range<G, V, R, false>(u.LE, ln, u.rb);
        uint32_t inm[D::UNROLL][V];
        matrix_bounds<G, V, R>(u, inm);
#pragma unroll
        for (int t = 0; t < D::UNROLL; t += 2) {
            uint32_t none[2 * V];
            dstep<G, V, R, UNIT, true, false>(da, u, t / 2, gl, ln, inm[t], QO, QE, none);
            vote = dstep<G, V, R, UNIT, false, false>(da, u, t / 2, gl, ln, inm[t + 1], QE, QO, none);
        }
        u.e += D::UNROLL / 2;
        u.dn += D::UNROLL / 2;
        u.mt -= D::UNROLL / 2;
        if (--left == 0) {
            left = iters;
            unit_maintain<G, V, R>(ka, da, u, gl, QE, QO);
        }
    }
}

// The sweep again, up to each extension's best anti-diagonal, writing for every
// slot which predecessor its value came from: per lane and loop iteration
// (UNROLL anti-diagonals) eight words -- one 32-byte sector -- holding, for a
// virtual lane and anti-diagonal, the mask of slots reached by the diagonal
// and, of the others, by the vertical move; and per iteration the window's
// base.  Five instructions more per pair of cells than the extension's sweep.  A
// band that leaves the window (it fitted one as wide, at other offsets) is
// flagged for the general sweep.
template <int G, int V, bool UNIT>
__global__ void __launch_bounds__(128, V == 1 ? 4 : 3)
    k_diag16_record(KernelArgs ka, DiagArgs da, DiagRecord rc, int cls) {
    constexpr int R = 16;
    using D = Diag<G, V, R>;
    constexpr unsigned int U = 32 / G;
    const int lane = threadIdx.x & 31;
    const int gl = lane % G, unit = lane / G;
    const Lanes<G> ln(lane);
    const uint32_t first_item = rc.class_at[cls], n_items = rc.class_at[cls + 1] - first_item;
    const uint32_t* q = rc.order + first_item;
    uint32_t QE[V * R], QO[V * R];
#pragma unroll
    for (int h = 0; h < V * R; ++h) QE[h] = QO[h] = 0u;
    DState<V> u;
    state_clear(u);
    const uint32_t brink_bot = gl == 0 ? (1u << (D::UNROLL / 2)) - 1u : 0u;
    const uint32_t brink_top = gl == G - 1 ? ((1u << (D::UNROLL / 2)) - 1u) << (D::VR - D::UNROLL / 2) : 0u;
    const int iters = da.period / D::UNROLL;
    int left = iters;
    bool exhausted = false, first_wave = true;
    uint4* codes = nullptr;
    int32_t* bases = nullptr;
    int dstar = 0;
    const unsigned int nwarps = gridDim.x * (blockDim.x >> 5);
    const unsigned int gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    for (;;) {
        if (u.active && 2 * u.e + 1 > dstar) {
            u.active = false;
            u.done = true;
        }
        const bool slide =
            __any_sync(FULL, (u.LE[V - 1] & brink_top) != 0u || (u.LE[0] & brink_bot) != 0u);
        if (__builtin_expect(slide, 0))
            units_slide<G, V, R, false>(ka, da, u, 0, gl, unit, ln, brink_top, brink_bot, QE, QO);
        const bool turn = __any_sync(FULL, u.done || (!u.active && !exhausted));
        if (__builtin_expect(turn, 0)) {
            if (rc.cells) {
                int bd, br;
                unsigned long long cells;
                unit_totals<G, V>(u, bd, br, cells);
                if (u.done && !u.overflow && gl == 0) atomicAdd(rc.cells, cells);
            }
            if (u.done && u.overflow && gl == 0) {
                rc.outgrew[u.item] = 1;
                atomicAdd(rc.n_outgrew, 1u);
            }
            if (u.done) {
#pragma unroll
                for (int v = 0; v < V; ++v) u.LE[v] = u.LO[v] = 0u;
            }
            u.done = false;
            const bool need = !u.active && !exhausted;
            const uint32_t want = __ballot_sync(FULL, need && gl == 0);
            uint32_t id = 0xffffffffu;
            if (want) {
                unsigned int slot;
                if (first_wave) {  // (every unit is idle at the first turn)
                    slot = gw * U + unsigned(unit);
                    first_wave = false;
                } else {
                    const int leader = __ffs(want) - 1;
                    unsigned int f = 0u;
                    if (lane == leader) f = atomicAdd(&rc.next[cls], unsigned(__popc(want)));
                    f = __shfl_sync(FULL, f, leader);
                    slot = U * nwarps + f + unsigned(__popc(want & ((1u << (unit * G)) - 1u)));
                }
                if (need && slot < n_items) id = q[slot];
            }
            if (need) {
                if (id != 0xffffffffu) {
                    unit_start<G, V, R, true>(ka, da, u, id, gl, QE, QO);
                    dstar = rc.dstar[id];
                    codes = rc.codes + rc.code_off[id] + 2 * gl;
                    bases = rc.bases + rc.it_off[id];
                } else {
                    exhausted = true;
                }
            }
            if (!__any_sync(FULL, u.active)) break;
        }
        if (__builtin_expect(slide || turn, 0)) next_range<G, V, R, false>(u.LE, ln, u.rb);
        uint32_t inm[D::UNROLL][V];
        matrix_bounds<G, V, R>(u, inm);
        uint32_t m[D::UNROLL][2 * V];
#pragma unroll
        for (int t = 0; t < D::UNROLL; t += 2) {
            dstep<G, V, R, UNIT, true, true>(da, u, t / 2, gl, ln, inm[t], QO, QE, m[t]);
            dstep<G, V, R, UNIT, false, true>(da, u, t / 2, gl, ln, inm[t + 1], QE, QO, m[t + 1]);
        }
        if (u.active) {
            const int it = u.e / (D::UNROLL / 2);
            uint4* c = codes + size_t(it) * (2 * G);
            if constexpr (V == 1) {
                c[0] = make_uint4(m[0][0], m[0][1], m[1][0], m[1][1]);
                c[1] = make_uint4(m[2][0], m[2][1], m[3][0], m[3][1]);
            } else {
                c[0] = make_uint4(m[0][0], m[0][1], m[1][0], m[1][1]);
                c[1] = make_uint4(m[0][2], m[0][3], m[1][2], m[1][3]);
            }
            if (gl == 0) bases[it] = u.base;
        }
        u.e += D::UNROLL / 2;
        u.dn += D::UNROLL / 2;
        u.mt -= D::UNROLL / 2;
        if (--left == 0) {
            left = iters;
            unit_maintain<G, V, R>(ka, da, u, gl, QE, QO);
        }
    }
}

}  // namespace

// ---- launches ----

// level -> (G, V, R) of its packed form: units of 32-slot lanes, as few as
// the window needs (the 32-row level runs the 64-slot window too: its units
// cost the same).  One extension per warp holds 1024 slots with one virtual
// lane (41.6 ms on the 100,000-pair batch's level 5, against 45 with two lanes' worth of
// rows in 16 lanes), 2048 with two.
#define LOGAN_PACKED_LEVELS(X) \
    X(0, 2, 1, 16) X(1, 2, 1, 16) X(2, 4, 1, 16) X(3, 8, 1, 16) X(4, 16, 1, 16) X(5, 32, 1, 16) \
    X(6, 32, 2, 16)

bool packed_level(int level) { return level <= 6; }

// the latency forms: (G, R) for windows of 128, 256 and 512 slots with 1, 2
// or 4 extensions per warp
#define LOGAN_PACKED_LATENCY(X) \
    X(0, 1, 32, 2) X(0, 2, 16, 4) X(0, 4, 8, 8) X(1, 1, 32, 4) X(1, 2, 16, 8) X(2, 1, 32, 8)

// Levels 0 and 1, four to a warp, with the general substitution: 64 slots, whose
// steps cost half as much (3 kbp at +2/-3/-5, X = 20, 1,000 pairs: 0.87 ms with
// 128 slots, 0.68; lognormal 1.86, 1.41; the 32-bit one-warp form 1.13, 1.55).
// With +1/-1/-1 unrelated pairs drift to bands of 12 X rows, and moving those to the
// next window costs more (X = 10: 1.50 ms with 128 slots, 2.02 with 64).
inline bool half_window(int level, int units, bool unit) { return level <= 1 && units == 4 && !unit; }

// class -> (G, V) of its recording sweep
#define LOGAN_RECORD_CLASSES(X) X(0, 4, 1) X(1, 8, 1) X(2, 16, 1) X(3, 32, 1) X(4, 32, 2)

namespace {

// resident blocks per SM, of the substitution form that needs more registers
template <int G, int V, int R>
int blocks_of() {
    int a = 0, b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_diag16<G, V, R, true>, 128, 0) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_diag16<G, V, R, false>, 128, 0) !=
            cudaSuccess)
        return 1;
    return std::max(1, std::min(a, b));
}

template <int G, int V, int R>
cudaError_t launch(int level, int queue, const KernelArgs& ka, const DiagArgs& da, int grid,
                   int phase, cudaStream_t s) {
    if (da.unit) k_diag16<G, V, R, true><<<grid, 128, 0, s>>>(ka, da, level, queue, phase);
    else k_diag16<G, V, R, false><<<grid, 128, 0, s>>>(ka, da, level, queue, phase);
    return cudaGetLastError();
}

// window and units of a latency form as one number
inline int latency_form(int level, int units) {
    const int w = level <= 2 ? 0 : level - 2;  // levels 0-2 share the 128-slot window
    return 10 * w + (w == 0 ? units : w == 1 ? std::min(units, 2) : 1);
}

}  // namespace

int packed_level_blocks_per_sm(int level) {
    switch (level) {
#define CASE(L, G, V, R) case L: return blocks_of<G, V, R>();
        LOGAN_PACKED_LEVELS(CASE)
#undef CASE
        default: return 0;
    }
}

int packed_latency_blocks_per_sm(int level, int units) {
    switch (latency_form(level, units)) {
#define CASE(K, U, G, R) case 10 * K + U: return blocks_of<G, 1, R>();
        LOGAN_PACKED_LATENCY(CASE)
#undef CASE
        default: return 0;
    }
}

cudaError_t launch_packed_level(int level, const KernelArgs& ka, const DiagArgs& da, int grid,
                                int phase, cudaStream_t s) {
    switch (level) {
#define CASE(L, G, V, R)                                                                   \
    case L:                                                                                \
        static_assert(Diag<G, V, R>::W >= level_window(L) && Diag<G, V, R>::W <= mig_rows(L), \
                      "window and record");                                                \
        return launch<G, V, R>(level, level, ka, da, grid, phase, s);
        LOGAN_PACKED_LEVELS(CASE)
#undef CASE
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_packed_latency(int level, int queue, int units, const KernelArgs& ka,
                                  const DiagArgs& da, int grid, int phase, cudaStream_t s) {
    if (half_window(level, units, da.unit != 0)) {
        static_assert(Diag<8, 1, 4>::W == level_window(1) && Diag<8, 1, 4>::W <= mig_rows(0), "window");
        k_diag16<8, 1, 4, false><<<grid, 128, 0, s>>>(ka, da, level, queue, phase);
        return cudaGetLastError();
    }
    switch (latency_form(level, units)) {
#define CASE(K, U, G, R)                                                                  \
    case 10 * K + U:                                                                      \
        static_assert(Diag<G, 1, R>::W == level_window(K + 2) && 32 / G == U &&          \
                          Diag<G, 1, R>::W <= mig_rows(K + 2), "window and record");      \
        return launch<G, 1, R>(level, queue, ka, da, grid, phase, s);
        LOGAN_PACKED_LATENCY(CASE)
#undef CASE
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_record(int cls, const KernelArgs& ka, const DiagArgs& da, const DiagRecord& rc,
                          int sms, cudaStream_t s) {
    switch (cls) {
#define CASE(K, G, V)                                                                            \
    case K: {                                                                                    \
        using D = Diag<G, V, 16>;                                                                \
        static_assert(D::W == level_window(K + 2) && record_lanes(K) == G &&                    \
                          record_steps(K) == D::UNROLL && (K < 4) == (V == 1),                   \
                      "class");                                                                  \
        int n = 0;                                                                               \
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(                     \
            &n, da.unit ? k_diag16_record<G, V, true> : k_diag16_record<G, V, false>, 128, 0);   \
        if (e != cudaSuccess) return e;                                                          \
        const int grid = sms * std::max(1, n);                                                   \
        if (da.unit) k_diag16_record<G, V, true><<<grid, 128, 0, s>>>(ka, da, rc, K);            \
        else k_diag16_record<G, V, false><<<grid, 128, 0, s>>>(ka, da, rc, K);                   \
        break;                                                                                   \
    }
        LOGAN_RECORD_CLASSES(CASE)
#undef CASE
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace logan
