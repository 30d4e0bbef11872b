// Sizes of a run's segments and spawn buckets (host code only).
#pragma once

#include <algorithm>
#include <cmath>

namespace fq {

inline unsigned next_pow2(unsigned long long x) {
    unsigned p = 1;
    while (p < x) p <<= 1;
    return p;
}

// segments whose buckets fill a third of a merge warp's table of `slots`
inline double full_segments(double s_ss, unsigned slots) {
    return std::max(1.0, std::ceil(std::min(s_ss / (slots / 3.0), 268000000.0)));
}

// Segments of a run: B of them, in groups of `group` that are one segment of a
// coarser map (segment_of scales the hash, so consecutive segments are).
struct Segments {
    unsigned B, group;
};

// Segments for s_ss spawns a step.  Large runs: full buckets, and a multiple
// of the warps that are resident at once (16 per SM in the default launch
// shape), so that every warp takes the same number: with a power of two, 1e6
// walkers were 8192 buckets on 2432 warps, where some took four and most
// three (now 7296: 8 % off the step), and 1e8 walkers 2^20 of 105 spawns
// instead of 646912 of 170 (2 %).  Below one full bucket per warp, smaller
// buckets on more warps, down to one round of 32 spawns: a step of 1e4
// walkers on 12 sites took 39 us with buckets of 86 spawns and takes 33 with
// 32, 1e5 on 20 sites 42 and 37.  They come in groups that make about a full
// bucket, for batches that fill the warps without them (batch_groups in
// fq_api.cu), of one segment more or fewer where that takes in more of them (1e4
// walkers 344 in fours instead of 340 in fives: 1 % of the step).  Less than 64 such buckets (2000 walkers, in spaces where a few
// addresses draw most of the spawns) stay at 100.
inline Segments segments_for(double s_ss, unsigned slots, int sms) {
    const double warps = sms * 16.0, full = full_segments(s_ss, slots);
    if (full > warps) return {(unsigned)(std::ceil(full / warps) * warps), 1};
    if (s_ss < 64.0 * 32.0) return {(unsigned)std::max(1.0, std::ceil(s_ss / 100.0)), 1};
    const double fine = std::min(warps, std::ceil(s_ss / 32.0));
    const double near = std::max(1.0, std::floor(fine / full + 0.5));
    auto whole = [&](double g) { return std::floor(fine / g) * g; };  // in whole groups
    double group = near;
    if (whole(near) < 0.99 * fine)
        for (double g : {near - 1.0, near + 1.0})
            if (g > 1.0 && whole(g) > whole(group)) group = g;
    return {(unsigned)whole(group), (unsigned)group};
}

// entries per segment for `total` over B segments
inline unsigned vec_slots(double total, unsigned B) {
    const double m = total / B;
    return (unsigned)((m + 4.0 * std::sqrt(m) + 16.0 + 31.0) / 32.0) * 32u;
}

// Spawn slots per bucket for a capacity of `total` spawns a step.  Spawns come
// in clumps of one address (k: the clump of a compound Poisson count), which a
// small bucket feels as much as a full one: where a run has more buckets than
// full ones would be, each has the room of a full one (`rooms` of them hold
// `total`).  The buffers are then B / rooms times as large (5.3 at 7e4 walkers,
// 1.1 at 1e6).  Beyond 16 times the usual capacity, where one bucket holds much
// of a step, what is asked for on top is spread over all B buckets.
struct SpawnRoom {
    double B, rooms, k, most;
    static unsigned per(double total, double buckets, double k) {
        const double m = total / buckets;
        return (unsigned)(std::min(m + 4.0 * std::sqrt(m * k) + k + 16.0 + 31.0, 4.0e9) / 32.0) * 32u;
    }
    unsigned slots(double total) const {
        if (total <= most) return per(total, rooms, k);
        return per(most, rooms, k) + (per(total, B, k) - per(most, B, k));
    }
    // the capacity that `cs` slots per bucket stand for: at least the one they
    // were made for
    double total(unsigned cs) const {
        const unsigned top = per(most, rooms, k);
        return cs <= top ? cs * rooms : top * rooms + (cs - top) * B;
    }
};
inline SpawnRoom spawn_room(unsigned B, double full, double k, double usual) {
    return {(double)B, std::min((double)B, full), k, 16.0 * usual};
}

// Spawn slots per bucket in the dense primary region: the steady-state fill
// plus three standard deviations of its compound-Poisson count (a multiple
// of 32, at most the bucket's capacity), so that nearly every spawn of an
// equilibrated run is stored there.
inline unsigned primary_slots(double s_ss, unsigned B, double k, unsigned Cs) {
    const double m = s_ss / B;
    const unsigned p = (unsigned)((m + 3.0 * std::sqrt(m * k) + 16.0 + 31.0) / 32.0) * 32u;
    return std::min(p, Cs);
}

}  // namespace fq
