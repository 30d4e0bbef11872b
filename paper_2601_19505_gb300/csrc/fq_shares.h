// Shares of a batch's segments for the warps of a launch (host code only).
#pragma once

#include <algorithm>
#include <cmath>
#include <vector>

namespace fq {

struct ShareRun {
    unsigned B;   // segments
    double fill;  // expected spawns per segment
};

// cuts[w] is warp w's first segment and cuts[nw] the number of segments.  A
// share lies within one run, and no share's expected work is more than the
// smallest bound for which the nw warps suffice.  A segment costs about as
// much as 32 spawns before its first one (batch of 64 runs with segments of 32
// to 170 spawns: 42.9 ms a chunk with 24, 42.4 with 48, 47.7 with 8, 45.6 with
// 96).  False if the warps cannot hold one share of every run (fewer than
// runs).
inline bool share_cuts(const std::vector<ShareRun>& runs, unsigned nw, std::vector<unsigned>& cuts) {
    auto parts = [](const ShareRun& r, double most) {  // shares of run r: at most `most` each
        const double per = std::max(1.0, std::floor(most / (32.0 + r.fill)));  // segments
        return (unsigned)std::ceil(r.B / per);
    };
    // Twice the largest run's work is one share a run whatever the rounding
    // (the work itself can divide to one segment less, which is two shares).
    double lo = 0.0, hi = 0.0;
    for (const ShareRun& r : runs) hi = std::max(hi, 2.0 * r.B * (32.0 + r.fill));
    for (int i = 0; i < 41; ++i) {
        const double mid = 0.5 * (lo + hi);
        unsigned long long n = 0;
        for (const ShareRun& r : runs) n += parts(r, mid);
        (n <= nw ? hi : lo) = mid;
    }
    cuts.clear();
    unsigned base = 0;
    for (const ShareRun& r : runs) {
        const unsigned k = parts(r, hi);
        for (unsigned i = 0; i < k; ++i)
            cuts.push_back(base + (unsigned)((unsigned long long)r.B * i / k));
        base += r.B;
    }
    if (cuts.size() > nw) return false;
    cuts.resize((size_t)nw + 1, base);  // warps beyond the shares have none
    return true;
}

}  // namespace fq
