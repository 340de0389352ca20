// Stopping rules of the mixed path's refinement and of its flexible GMRES, per mode.
#pragma once

#include <vector>

namespace pmlbie {

// a mode's refinement is done when, for every rhs, the relative residual
// |B - A x| / |B| <= kTolRel or the normwise backward error
// |B - A x| / (|A|_F |x| + |B|) <= kTolBwd, or at the FP64 floor of ill-conditioned
// modes, whose |A| |x| >> |B|
constexpr double kTolRel = 1e-13;
constexpr double kTolBwd = 1e-16;
// a backward error that no longer halves is at that floor only below kTolFloorIr: above
// it the FP32 factors contract too slowly (a factor near 1 a step looks the same; a stop
// at 1e-14 has hidden an error of 3e-5), and FGMRES takes the mode over, which stops
// below kTolFloor when a cycle gains less than 10 %, and after its last cycle
constexpr double kTolFloor = 1e-14;
constexpr double kTolFloorIr = 4e-16;

enum class RefineStep { kContinue, kDone, kSlow };

// after correction `iters` (>= 1); ok: the tolerances are met for every rhs
inline RefineStep refine_rule(int iters, bool ok, double bwd, double prev) {
    const bool stalled = iters >= 2 && !(bwd < 0.5 * prev);
    if (ok || (stalled && bwd <= kTolFloorIr)) return RefineStep::kDone;
    return stalled ? RefineStep::kSlow : RefineStep::kContinue;      // contraction too slow or divergent
}

// FGMRES starts from zero, not from the refinement's last iterate, when that neither
// improved on the first one nor is at the level that FGMRES itself accepts
inline bool restart_from_zero(double bwd, double first) { return !(bwd <= kTolFloor) && !(bwd < first); }

// before cycle `cyc` of at most max_cycles (cyc = max_cycles: after the last one);
// prev: the backward error before the cycle that just ended
inline bool gmres_rule(bool ok, int cyc, int max_cycles, double bwd, double prev) {
    return ok || (bwd <= kTolFloor && ((cyc > 0 && bwd >= 0.9 * prev) || cyc >= max_cycles));
}

// When there is no memory for FGMRES: the modes whose refinement ended at the level
// that FGMRES accepts keep their iterate; returns how many are left
inline int accept_refined(std::vector<int>& slow, const std::vector<double>& bwd) {
    int left = 0;
    for (size_t m = 0; m < slow.size(); ++m) {
        if (slow[m] && bwd[m] <= kTolFloor) slow[m] = 0;
        left += slow[m] != 0;
    }
    return left;
}

}  // namespace pmlbie
