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

// The least work that a warp's largest share can have: a share lies within one
// run, and nw warps have a share each or none.  A segment costs about as much
// as 32 spawns before its first one (batch of 64 runs with segments of 32 to
// 170 spawns: 42.9 ms a chunk with 24, 42.4 with 48, 47.7 with 8, 45.6 with 96).
inline unsigned share_parts(const ShareRun& r, double most) {  // shares of at most `most` each
    const double per = std::max(1.0, std::floor(most / (32.0 + r.fill)));  // segments
    return (unsigned)std::ceil(r.B / per);
}
inline double share_bound(const std::vector<ShareRun>& runs, unsigned nw) {
    // Twice the largest run's work is one share a run whatever the rounding
    // (the work itself can divide to one segment less, which is two shares).
    double lo = 0.0, hi = 0.0, one = 0.0;  // one: a share is a segment at least
    for (const ShareRun& r : runs) {
        hi = std::max(hi, 2.0 * r.B * (32.0 + r.fill));
        one = std::max(one, 32.0 + r.fill);
    }
    for (int i = 0; i < 41; ++i) {
        const double mid = 0.5 * (lo + hi);
        unsigned long long n = 0;
        for (const ShareRun& r : runs) n += share_parts(r, mid);
        (n <= nw ? hi : lo) = mid;
    }
    return std::max(hi, one);
}

// Waves of `resident` warps that a batch's shares are cut for.  One, unless the
// shares of so few warps, each within a run, leave many without work: 1024 runs
// of 86 segments are two shares each on 2432 warps (84 % of them busy), 1900
// one (78 %).  In three and four waves of smaller shares they are 93 and 93 %
// (1024 runs of 1e4 walkers 1046 -> 834 us a step, 1900 2239 -> 1499).  A share
// of its own costs its warp a start, taken as 100 spawns: three replicas with
// shares of four segments were 3 % slower in three waves of shares of one.
inline unsigned share_waves(const std::vector<ShareRun>& runs, unsigned resident) {
    double best = (share_bound(runs, resident) + 100.0) / 1.05;
    unsigned waves = 1;
    for (unsigned k = 2; k <= 4; ++k) {
        const double t = k * (share_bound(runs, k * resident) + 100.0);
        if (t < best) {
            best = t;
            waves = k;
        }
    }
    return waves;
}

// cuts[w] is warp w's first segment and cuts[nw] the number of segments.  False
// if the warps cannot hold one share of every run (fewer than runs).
inline bool share_cuts(const std::vector<ShareRun>& runs, unsigned nw, std::vector<unsigned>& cuts) {
    const double hi = share_bound(runs, nw);
    cuts.clear();
    unsigned base = 0;
    for (const ShareRun& r : runs) {
        const unsigned k = share_parts(r, hi);
        for (unsigned i = 0; i < k; ++i)
            cuts.push_back(base + (unsigned)((unsigned long long)r.B * i / k));
        base += r.B;
    }
    if (cuts.size() > nw) return false;
    cuts.resize((size_t)nw + 1, base);  // warps beyond the shares have none
    return true;
}

}  // namespace fq
