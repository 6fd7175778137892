// Host side of the packed linear kernels (diag16.cuh, xdrop_diag16.cu): the
// constants of a launch, and the bounds under which every 16-bit key stays
// inside its half-word.  No CUDA here, so that a CPU program can include it.
#pragma once
#include <cstdint>

namespace logan {

constexpr int KS = 32;         // score scale of a key: five bits of row code below it
constexpr int LOG2KS = 5;
constexpr int kPrefetch = 64;  // steps that the prefetched codes last

// Constants of a packed launch (xdrop_diag16.cu), from the scoring and the
// largest X that can reach the level.
struct DiagArgs {
    int gap;     // gap score per base (<= 0)
    int mp;      // max(match, 0)
    int step;    // theta's growth per anti-diagonal: 32 * -gap
    int floor;   // smallest key (a dead one)
    int period;  // anti-diagonals between renormalisations (a power of two, 4 .. 64)
    int unit;    // match 1 and match - mismatch == 2 * (mismatch - 2 gap) (as +1/-1/-1): one
                 // multiply-add per substitution, a best that grows by 1 at most per anti-diagonal
    // multipliers of a mask bit at position p: mismatch - 2 gap and match -
    // mismatch in key units, divided by 2^p
    uint32_t cb[6], cf[6];
};

// The constants for this scoring and X, false when the scores do not fit.  With
// g = -gap, mp = max(match, 0) and D = period g + mp (period / 2 + 1), what theta
// can grow by between renormalisations (the best grows by mp at most in any
// two anti-diagonals):
//   KS (D + X + mp + 1) + 32 <= 32767      live keys stay below 65536;
//   KS (D + 2 g + 2 mp + 2) + 64 <= 32767  live keys stay above the floor,
//                                          which theta does not outgrow;
//   KS (max(-mismatch, 0) + 2 mp + 2) + 64 <= 32767
//       a masked diagonal stays at or above 0: it adds KS (mismatch + 2 g) to a live
//       key two anti-diagonals old, which is at least 32768 - KS (2 g + mp).
//       (Below 0 a half-word wraps to a large live score and borrows from
//       its neighbour.)
inline bool diag_plan(int match, int mismatch, int gap, int64_t xmax, DiagArgs* da) {
    const int64_t g = -int64_t(gap), mp = match > 0 ? match : 0;
    const int64_t am = mismatch < 0 ? -int64_t(mismatch) : 0;
    if (KS * (am + 2 * mp + 2) + 64 > 32767) return false;
    for (int period = kPrefetch; period >= 4; period >>= 1) {
        const int64_t grow = period * g + mp * (period / 2 + 1);
        if (KS * (grow + xmax + mp + 1) + 32 > 32767 || KS * (grow + 2 * g + 2 * mp + 2) + 64 > 32767)
            continue;
        const int base = mismatch - 2 * gap, bonus = match - mismatch;
        da->gap = gap;
        da->mp = int(mp);
        da->step = int(KS * g);
        da->floor = int(KS * grow + 64);
        da->period = period;
        da->unit = bonus == 2 * base && mp == 1 ? 1 : 0;
        for (int p = 0; p < 6; ++p) {
            da->cb[p] = uint32_t(base) * uint32_t(KS >> p);
            da->cf[p] = uint32_t(bonus) * uint32_t(KS >> p);
        }
        return true;
    }
    return false;
}

// The constants for the recording sweep, which also subtracts keys: no two that
// it compares may be 32768 apart.
//   * The two gap moves' keys: the floor is raised so that no key at or above it
//     is 32768 above it (and stays below every live key).
//   * The larger of them, p, against the diagonal's key t.  Where the
//     substitution is masked t is at or above the floor.  Elsewhere
//     p - t <= KS (mp - mismatch): a gap move adds nothing to a key, so the cell
//     above (or left of) a target is at most mp - gap in score above the
//     target's diagonal predecessor.  diag_plan's third bound gives
//     KS (mp - mismatch) <= 32767 - 64 - 2 KS.
inline bool diag_record_plan(int match, int mismatch, int gap, int64_t xmax, DiagArgs* da) {
    if (!diag_plan(match, mismatch, gap, xmax, da)) return false;
    const int64_t g = -int64_t(gap), mp = da->mp;
    const int64_t grow = da->period * g + mp * (da->period / 2 + 1);
    const int64_t floor = KS * (grow + xmax + mp + 1) + 96;
    if (floor + KS * (2 * g + 2 * mp + 2) > 32767) return false;
    da->floor = int(floor);
    return true;
}

}  // namespace logan
