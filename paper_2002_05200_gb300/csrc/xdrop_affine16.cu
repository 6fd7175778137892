// X-drop extension with affine gaps on DNA, two cells to a 32-bit register
// (16-bit SIMD) in diagonal coordinates, for the affine window levels of 128,
// 256 and 512 rows when the call's scores provably fit 16 bits.
//
// Method: Gotoh's three states per cell under the paper's anti-diagonal
// sweep, X-drop rule and band trimming (Sec. III-A, Algorithms 1 and 2;
// other scoring schemes are the paper's future work, Sec. VIII) -- the
// computation of the 32-bit affine kernel (xdrop_affine.cu), with the same
// results.  Kernel, keys and bounds: diag_affine16.cuh.
//
// A band that outgrows the window restarts at the next level (no band-state
// records), after the widest in the device-memory ring, as in the 32-bit
// affine kernel.
//
// Bound by the ALU pipe and issue (71 % each, 168 registers, 12 warps per SM;
// four blocks per SM at 128 registers 38.2 ms, lanes of 16 slots 47.5 ms).
// 50,000 lognormal pairs, -2 / -1, X = 100: 63.4 ms in the row-window form that
// this replaced, 37.2 now.
#include "diag_affine16.cuh"

namespace logan {

bool affine16_level(int level) { return level >= 1 && level <= 3; }

bool affine16_plan(Scoring sc, int go, int ge, int64_t xmax, DiagAffineArgs16* out) {
    DiagAffineArgs a{};
    if (!diag_affine_plan(sc.match, sc.mismatch, go, ge, xmax, &a)) return false;
    out->period = a.period;
    out->floor = a.floor;
    return true;
}

namespace {

// level -> lanes of 32 slots, and of 16 for batches that cannot fill the GPU's
// warps (shorter steps)
#define LOGAN_AFFINE16_LEVELS(X) X(1, 4, 8) X(2, 8, 16) X(3, 16, 32)

DiagAffineArgs affine16_args(const KernelArgs& ka, const DiagAffineArgs16& plan, int go, int ge,
                             int level, int n_levels) {
    DiagAffineArgs a{};
    a.pa = ka.wa;
    a.pb = ka.wb;
    a.items = ka.items;
    a.ext = ka.ext;
    a.queues = ka.queues;
    a.qcap = ka.qcap;
    a.counters = ka.counters;
    a.level = level;
    a.next_queue = level + 1 < n_levels ? level + 1 : kWarpLevels;
    a.cells_level = -1;
    a.sub_max = ka.sc.match;
    a.sub_min = ka.sc.mismatch;
    a.period = plan.period;
    a.floor = plan.floor;
    a.step = KS * -ge;
    a.go = KS * go;
    const int base = ka.sc.mismatch - 2 * ge - go, bonus = ka.sc.match - ka.sc.mismatch;
    for (int p = 0; p < 6; ++p) {
        a.cb[p] = uint32_t(base) * uint32_t(KS >> p);
        a.cf[p] = uint32_t(bonus) * uint32_t(KS >> p);
    }
    return a;
}

}  // namespace

cudaError_t launch_affine16_level(int level, const KernelArgs& ka, const DiagAffineArgs16& plan,
                                  int go, int ge, int n_levels, bool small, int grid, cudaStream_t s) {
    const DiagAffineArgs a = affine16_args(ka, plan, go, ge, level, n_levels);
    switch (level) {
#define CASE(L, G, GS)                                                      \
    case L:                                                                 \
        if (small) k_diag_affine<GS, 8, false><<<grid, 128, 0, s>>>(a);     \
        else k_diag_affine<G, 16, false><<<grid, 128, 0, s>>>(a);           \
        break;
        LOGAN_AFFINE16_LEVELS(CASE)
#undef CASE
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

int affine16_blocks_per_sm(int level, bool small) {
    int n = 0;
    cudaError_t e = cudaErrorInvalidValue;
    switch (level) {
#define CASE(L, G, GS)                                                                               \
    case L:                                                                                          \
        e = small ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_diag_affine<GS, 8, false>, 128, 0) \
                  : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_diag_affine<G, 16, false>, 128, 0); \
        break;
        LOGAN_AFFINE16_LEVELS(CASE)
#undef CASE
        default: break;
    }
    return e == cudaSuccess ? n : 0;
}

}  // namespace logan
