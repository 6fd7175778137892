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
// Then every half-word stays inside [0, 65536) through every addition, and an
// addition of both halves is one 32-bit operation.
//
// Bound by the ALU pipe and issue together (about 7.5 instructions per pair
// of cells, 3 of them on the ALU pipe, and about 100 of bookkeeping per lane
// and anti-diagonal).  The row-window form it replaced (a prune select, range
// test and re-basing per cell, three rotating arrays, a slide of the window
// every 16 rows) ran 12 per pair of cells and about 140 of bookkeeping.
// 100,000 lognormal pairs, X = 100: level 2 (137e9 cells) 83 -> 52 ms, level 5
// (105e9) 52 -> 44 ms, level 6 19.5 -> 9 ms, the whole call 182 -> 123 ms.
#include "diag16.cuh"

namespace logan {

namespace {

constexpr int kGone = 1 << 20;  // `lo` of a unit without a range

// lo, hi, dn and mt of rows / diagonals given in window coordinates
template <int G, int V, int R>
__device__ __forceinline__ void set_range(DState<V>& u, const Item& it, int lo_row, int hi_row,
                                          int gl) {
    const int off = u.base + u.e + gl * Diag<G, V, R>::C;
    u.lo = lo_row - off;
    u.hi = hi_row - off;
    u.dn = 2 * u.e + 1 - u.phi - int(it.n) - off;
    u.mt = int(it.m) - off;
}

template <int G, int V, int R>
__device__ __forceinline__ void unit_start(const KernelArgs& ka, const DiagArgs& da, DState<V>& u,
                                           uint32_t id, int gl, uint32_t (&QE)[V * R],
                                           uint32_t (&QO)[V * R]) {
    using D = Diag<G, V, R>;
    const Item it = ka.items[id];
    u.item = id;
    u.X = it.X;
    u.c32 = 0u;
    u.theta = 32768;
    const int32_t slot = ka.mig_slot[id];
    const int32_t* rec = slot >= 0 ? mig_record(ka, slot) : nullptr;
    if (rec && rec[MIG_KIND] == MIG_RELATIVE) {
        // resume a band saved by a narrower level
        const int rows = rec[MIG_ROWS], d = rec[MIG_D], row0 = rec[MIG_BASE];
        const int lo = rec[MIG_LO], hi = rec[MIG_HI];
        u.phi = (d & 1) ? 0 : 1;
        u.e = (d + u.phi - 1) >> 1;
        u.base = ((lo + hi) >> 1) - u.e - D::W / 2;
        u.best = rec[MIG_BEST];
        u.bi = rec[MIG_BI];
        u.bd = rec[MIG_BI] + rec[MIG_BJ];
        u.cells = (unsigned long long)uint32_t(rec[MIG_CELLS_LO]) |
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
        set_range<G, V, R>(u, it, lo, hi, gl);
    } else {
        // S(0,0) = 0 on d = 0 (even), X above its threshold, mid-window
        u.phi = 0;
        u.e = 0;
        u.base = -D::W / 2;
        u.best = u.bi = u.bd = 0;
        u.cells = 0ull;
        const uint32_t f2 = uint32_t(da.floor) * 0x10001u;
#pragma unroll
        for (int h = 0; h < V * R; ++h) QE[h] = QO[h] = f2;
#pragma unroll
        for (int v = 0; v < V; ++v) u.LE[v] = u.LO[v] = 0u;
        if (gl == G / 2) {  // slot W / 2 is the first of this lane (G = 1: of virtual lane V / 2)
            constexpr int v0 = G == 1 ? V / 2 : 0;
            QE[v0 * R] = (f2 & 0xffff0000u) | live_key<D::VR>(it.X, 0);
            u.LE[v0] = 1u;
        }
        u.theta += KS * -da.gap;  // theta_1
        set_range<G, V, R>(u, it, 0, 0, gl);
    }
    u.cells0 = u.cells;
    load_planes<G, V, R>(ka, it, u, gl);
    u.active = true;
    u.done = false;
    u.overflow = false;
    u.migrated = false;
}

// Result or escalation of a finished unit (its leader lane writes).
template <int V>
__device__ __forceinline__ void unit_end(const KernelArgs& ka, DState<V>& u, int level, int gl,
                                         bool twin) {
    u.cells += u.c32;
    u.c32 = 0u;
    if (gl != 0) return;
    if (u.overflow) {
        if (u.migrated) atomicAdd(&ka.counters->cells[level], u.cells - u.cells0);
        const int nq = escalate_queue(ka, level, twin);
        const unsigned int t = atomicAdd(&ka.counters->tail[nq], 1u);
        ka.queues[size_t(nq) * ka.qcap + t] = u.item;
    } else {
        ExtRes r;
        r.best = u.best;
        r.bi = u.bi;
        r.bj = u.bd - u.bi;
        r.status = 0;
        r.cells = u.cells;
        ka.ext[u.item] = r;
        atomicAdd(&ka.counters->cells[level], u.cells - u.cells0);
    }
}

// Saves an overflowing band for the next level: rows [row0, row0 + rows) of
// d-1 (even, frame e) and d-2 (odd, frame e-1) as scores above T_d - 2 mp,
// which no live cell of d-2 or d-1 lies below.
template <int G, int V, int R>
__device__ __forceinline__ void save_band(const KernelArgs& ka, const DiagArgs& da, DState<V>& u,
                                          int32_t slot, int level, int gl,
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
        rec[MIG_LO] = u.lo + off;
        rec[MIG_HI] = u.hi + off;
        rec[MIG_BEST] = u.best;
        rec[MIG_T] = T;
        rec[MIG_T1] = T - ref;
        rec[MIG_T2] = T - ref;
        rec[MIG_BI] = u.bi;
        rec[MIG_BJ] = u.bd - u.bi;
        const unsigned long long c = u.cells + u.c32;
        rec[MIG_CELLS_LO] = int32_t(uint32_t(c));
        rec[MIG_CELLS_HI] = int32_t(uint32_t(c >> 32));
        rec[MIG_LEVEL] = level;
        ka.mig_slot[u.item] = slot;
    }
}

// Loop top, before an odd step: units whose range ended are done; windows
// whose band comes within a slot of an edge slide by half virtual lanes, or
// overflow when the band does not fit.
template <int G, int V, int R>
__device__ __forceinline__ void unit_prepare(const KernelArgs& ka, const DiagArgs& da, DState<V>& u,
                                             int level, int gl, int unit, uint32_t (&QE)[V * R],
                                             uint32_t (&QO)[V * R]) {
    using D = Diag<G, V, R>;
    if (u.active && u.lo >= kGone / 2) {
        u.active = false;
        u.done = true;
    }
    // the next two steps reach slots lo - 1 .. hi + 1 (of rows inside the matrix)
    const int off = gl * D::C;
    const int lo_s = max(u.lo, u.dn) + off, hi_s = min(u.hi, u.mt) + off;
    bool up = u.active && hi_s > D::W - 2, dn = u.active && lo_s < 1;
    if (!__any_sync(FULL, up || dn)) return;
    const uint32_t f2 = uint32_t(da.floor) * 0x10001u;
    const bool ovf = (up && lo_s - R < 1) || (dn && hi_s + R > D::W - 2);
    up = up && !ovf;
    dn = dn && !ovf;
    if (__any_sync(FULL, up)) {
        shift_half<G, V, R, true>(QE, up, gl, f2);
        shift_half<G, V, R, true>(QO, up, gl, f2);
        shift_half_mask<G, V, R, true>(u.LE, up, gl);
        shift_half_mask<G, V, R, true>(u.LO, up, gl);
    }
    if (__any_sync(FULL, dn)) {
        shift_half<G, V, R, false>(QE, dn, gl, f2);
        shift_half<G, V, R, false>(QO, dn, gl, f2);
        shift_half_mask<G, V, R, false>(u.LE, dn, gl);
        shift_half_mask<G, V, R, false>(u.LO, dn, gl);
    }
    if (up || dn) {
        const int by = up ? R : -R;
        u.base += by;
        u.lo -= by;
        u.hi -= by;
        u.dn -= by;
        u.mt -= by;
        load_planes<G, V, R>(ka, ka.items[u.item], u, gl);
    }
    if (__any_sync(FULL, ovf)) {
        int32_t slot = -1;
        if (ovf && gl == 0) slot = mig_alloc(ka, level);
        slot = __shfl_sync(FULL, slot, unit * G);
        if (ovf) {
            if (slot >= 0) save_band<G, V, R>(ka, da, u, slot, level, gl, QE, QO);
            u.active = false;
            u.done = true;
            u.overflow = true;
            u.migrated = slot >= 0;
            u.lo = kGone;
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
// P holds d-1.  Units without a range compute values without effects.
template <int G, int V, int R, bool UNIT, bool ODD>
__device__ __forceinline__ void dstep(const KernelArgs& ka, const DiagArgs& da, DState<V>& u,
                                      int gl, uint32_t (&Q)[V * R], const uint32_t (&P)[V * R]) {
    using D = Diag<G, V, R>;
    constexpr int VR = D::VR, C = D::C, W = D::W;
    const int rlo = max(u.lo, u.dn), rhi = min(u.hi + 1, u.mt);
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
    uint32_t fkey = 0u;
    uint32_t L[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        // slots of this virtual lane inside [rlo, rhi], then those whose
        // diagonal predecessor is live (rm), then the matches among them (fm)
        const int k0 = __viaddmin_s32_relu(rlo, -v * VR, VR);
        const int k1 = __viaddmin_s32_relu(rhi, 1 - v * VR, VR);
        const uint32_t s0 = __funnelshift_lc(~0u, 0u, k0), s1 = __funnelshift_lc(~0u, 0u, k1);
        uint32_t rm = s1 & ~s0 & (ODD ? u.LO[v] : u.LE[v]);
        uint32_t fm = rm & ~(u.a0[v] ^ u.b0[v]);
        fm = fm & ~(u.a1[v] ^ u.b1[v]);
        if constexpr (R == 8) {  // slots 8..15 to the upper half-word
            rm = __byte_perm(rm, 0u, 0x4140);
            fm = __byte_perm(fm, 0u, 0x4140);
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
        uint32_t x[R];
#pragma unroll
        for (int h = 0; h < R; ++h) {
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
            const uint32_t val = __vimax3_u16x2(P[g], sh, t);
            Q[g] = val;
            x[h] = val + thr;
            if (h & 1) lk = __vimax3_u16x2(lk, Q[g - 1], val);
        }
        // the signs of four slots per byte permute, gathered as 255 * mask
        uint32_t acc = 0u;
#pragma unroll
        for (int h = 0; h < R / 2; ++h) acc = sign_bytes(x[h], x[h + R / 2]) * (1u << h) + acc;
        uint32_t m = acc * 0xfefefeffu;  // 255 * 0xfefefeff = 1 (mod 2^32)
        if constexpr (R == 8) {          // nibbles in bytes -> 16 bits
            m = m | (m >> 4);
            m = __byte_perm(m, 0u, 0x4420);
        }
        L[v] = m & s1 & ~s0;
        // the virtual lane's best key, widened with its position
        const uint32_t lkey = max(lk & 0xffffu, lk >> 16);
        const int above = int(lkey) - u.theta;
        const uint32_t fk = above >= 0 ? ((uint32_t(above) >> LOG2KS) << D::LOG2W) +
                                             (uint32_t(W - VR - v * VR - gl * C) + (lkey & uint32_t(VR - 1)))
                                       : 0u;
        fkey = max(fkey, fk);
    }
    // the lane's first / last live slots, then the unit's
    int fr, lr;
    bool any;
    if constexpr (V == 1) {
        fr = __ffs(L[0]) - 1;
        lr = 31 - __clz(L[0]);
        any = L[0] != 0u;
    } else {
        const unsigned long long LL = (unsigned long long)L[0] | ((unsigned long long)L[1] << 32);
        fr = __ffsll(LL) - 1;
        lr = 63 - __clzll(LL);
        any = LL != 0ull;
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        if constexpr (ODD) u.LO[v] = L[v];
        else u.LE[v] = L[v];
    }
    const uint32_t flw =
        any ? (uint32_t(W - gl * C - fr) | (uint32_t(gl * C + 1 + lr) << 16)) : 0u;
    const uint32_t wkey = unit_max_u32<G>(fkey);
    uint32_t fl;
    if constexpr (G == 32) {
        const uint32_t vote = __ballot_sync(FULL, any);
        const uint32_t f = __shfl_sync(FULL, flw, __ffs(vote) - 1);
        const uint32_t l = __shfl_sync(FULL, flw, 31 - __clz(vote));
        fl = vote ? __byte_perm(f, l, 0x7610) : 0u;
    } else {
        fl = unit_max_u16x2<G>(flw);
    }
    const bool run = rlo <= rhi;
    u.c32 += run ? uint32_t(rhi - rlo + 1) : 0u;
    // the anti-diagonal's outcome: it advances when it had a live cell (then
    // it had a range), else the extension ends here
    const bool adv = fl != 0u;
    const int umax = int(wkey >> D::LOG2W);
    const bool imp = adv && umax > u.X;  // S > best  <=>  S - T_d > X
    const int d = 2 * u.e + (ODD ? 1 : 2);
    u.bi = imp ? u.base + u.e + (ODD ? 0 : 1) + (W - 1 - int(wkey & uint32_t(W - 1))) : u.bi;
    u.bd = imp ? d - u.phi : u.bd;
    const int gain = imp ? umax - u.X : 0;
    u.best += gain;
    u.theta += gain * KS + da.step;
    // slots of the next step's frame (an even step moves rows one slot down)
    u.lo = adv ? W - int(fl & 0xffffu) - gl * C - (ODD ? 1 : 0) : kGone;
    u.hi = int(fl >> 16) - 1 - gl * C - (ODD ? 1 : 0);
    if constexpr (ODD) u.mt -= 1;
    else u.dn += 1;
}

template <int G, int V, int R, bool UNIT>
__global__ void __launch_bounds__(128, 4)
    k_diag16(KernelArgs ka, DiagArgs da, int level, int queue, int phase) {
    const int lane = threadIdx.x & 31;
    const int gl = lane % G, unit = lane / G;
    const bool twin = queue != level;
    const uint32_t* q = ka.queues + size_t(queue) * ka.qcap;
    uint32_t QE[V * R], QO[V * R];
#pragma unroll
    for (int h = 0; h < V * R; ++h) QE[h] = QO[h] = 0u;
    DState<V> u;
    u.lo = kGone;
    u.hi = -1;
    u.dn = u.mt = 0;
    u.theta = 32768;
    u.best = u.bi = u.bd = u.X = 0;
    u.base = u.e = u.phi = 0;
    u.c32 = 0u;
    u.cells = u.cells0 = 0ull;
    u.item = 0u;
    u.active = u.done = u.overflow = u.migrated = false;
#pragma unroll
    for (int v = 0; v < V; ++v)
        u.LE[v] = u.LO[v] = u.a0[v] = u.a1[v] = u.b0[v] = u.b1[v] = 0u;
    u.na0 = u.na1 = u.nb0 = u.nb1 = 0u;
    bool exhausted = false;
    bool first_wave = true;  // the warp's first pop takes static slots
    int left = da.iters;
    for (;;) {
        unit_prepare<G, V, R>(ka, da, u, level, gl, unit, QE, QO);
        if (__any_sync(FULL, u.done || (!u.active && !exhausted))) {
            if (u.done) {
                unit_end(ka, u, level, gl, twin);
                u.done = false;
            }
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
            if (!__any_sync(FULL, u.active)) break;
        }
        dstep<G, V, R, UNIT, true>(ka, da, u, gl, QO, QE);
        dstep<G, V, R, UNIT, false>(ka, da, u, gl, QE, QO);
        u.e += 1;
        if (--left == 0) {
            left = da.iters;
            unit_maintain<G, V, R>(ka, da, u, gl, QE, QO);
        }
    }
}

}  // namespace

bool packed_plan(Scoring sc, int64_t xmax, DiagArgs* da) {
    const int64_t g = -int64_t(sc.gap), mp = sc.match > 0 ? sc.match : 0;
    for (int period = kPrefetch; period >= 4; period >>= 1) {
        const int64_t grow = period * g + mp * (period / 2 + 1);
        if (KS * (grow + xmax + mp + 1) + 32 > 32767 || KS * (grow + 2 * g + 2 * mp + 2) + 64 > 32767)
            continue;
        const int base = sc.mismatch - 2 * sc.gap, bonus = sc.match - sc.mismatch;
        da->gap = sc.gap;
        da->mp = int(mp);
        da->step = int(KS * g);
        da->floor = int(KS * grow + 64);
        da->iters = period / 2;
        da->unit = bonus == 2 * base ? 1 : 0;
        for (int p = 0; p < 6; ++p) {
            da->cb[p] = uint32_t(base) * uint32_t(KS >> p);
            da->cf[p] = uint32_t(bonus) * uint32_t(KS >> p);
        }
        return true;
    }
    return false;
}

// ---- launches ----

// level -> (G, V, R) of its packed form: 32 slots per lane up to 16 lanes;
// the 1024- and 2048-slot windows share a lane's bookkeeping between two
// virtual lanes.
#define LOGAN_PACKED_LEVELS(X) \
    X(2, 4, 1, 16) X(3, 8, 1, 16) X(4, 16, 1, 16) X(5, 16, 2, 16) X(6, 32, 2, 16)

bool packed_level(int level) {
    switch (level) {
#define CASE(L, G, V, R) case L: return true;
        LOGAN_PACKED_LEVELS(CASE)
#undef CASE
        default: return false;
    }
}

cudaError_t launch_packed_level_persistent(int level, const KernelArgs& ka, const DiagArgs& da,
                                           int grid, int phase, cudaStream_t s) {
    switch (level) {
#define CASE(L, G, V, R)                                                                          \
    case L:                                                                                       \
        static_assert(Diag<G, V, R>::W == level_window(L), "a packed form keeps its level's window"); \
        if (da.unit) k_diag16<G, V, R, true><<<grid, 128, 0, s>>>(ka, da, level, level, phase);   \
        else k_diag16<G, V, R, false><<<grid, 128, 0, s>>>(ka, da, level, level, phase);          \
        break;
        LOGAN_PACKED_LEVELS(CASE)
#undef CASE
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

int packed_level_blocks_per_sm(int level) {
    int n = 0;
    cudaError_t e = cudaErrorInvalidValue;
    switch (level) {
#define CASE(L, G, V, R)                                                                        \
    case L:                                                                                     \
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_diag16<G, V, R, true>, 128, 0); \
        break;
        LOGAN_PACKED_LEVELS(CASE)
#undef CASE
        default: break;
    }
    return e == cudaSuccess ? n : 0;
}

}  // namespace logan
