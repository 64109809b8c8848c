// hd_route.h -- which calls run their sweeps as one launch (host).
//
// A context that may do so (hd_tile.h) has two orders of its sweeps with the
// same chain: one launch for up to 256 sweeps, or a launch per phase (as strips
// or replica branches inside a captured step).  One launch pays for itself by
// the launch boundaries it saves, and costs more than the phases where it works
// for long on little: a box takes a whole SM for its five dependent phases, a
// tile some eight microseconds beside 2.8 ns per cell, and its start and end
// (staging, waits) are those of a sweep or more.  So it depends on the replicas,
// on how many rounds of boxes or tiles the SMs take, and on the sweeps of the
// call.  Figures: us per call, phases and one launch, on 152 SMs.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace hd {

struct SweepShape {
    bool box;         // whole boxes (else tiles)
    bool fixed;       // number form
    bool crowded;     // more than a disk per cell on average
    int R;            // replicas
    int hm;           // largest half-side
    double rounds;    // boxes or tiles per SM (boxes: rounded up)
    double tile;      // cells per tile on average
    double replica;   // cells per replica on average
};

// Boxes.  Fixed form, 24 sweeps of a step: 608 of N = 36 447 and 450, of N = 1000 800
// and 734; 800 of them 460 and 632, 960 and 1053.  FP64: 760 of N = 400 439 and 450,
// 1000 of N = 1000 2058 and 1835.  A call of hd_sweep makes a launch per phase from
// the host (31 us per sweep at least): 1000 of N = 1000 1352 and 1183.  One sweep:
// 304 of N = 100 45 and 37, 500 49 and 51 (N = 1000 56 and 65).  Crowded, fixed, N = 400
// at cells of 2.5 sigma, 12 sweeps: 304 480 and 402, 608 549 and 783 (from hd_sweep 518 and
// 399, 628 and 773).
inline bool one_launch_boxes(const SweepShape& s, int64_t n, bool step) {
    double most = 1e9;
    if (s.crowded) most = step || n < 3 ? 2 : 3;
    else if (n == 1) most = s.fixed || step ? 2 : 3;
    else if (n == 2) most = step ? 3 : (s.fixed ? 4 : 5);
    else if (step) most = s.fixed ? 4 : (s.hm < 13 ? 5 : 7);
    return s.rounds <= most;
}

// Tiles in a captured step of up to 64 replicas, whose phases run as strips or as a
// branch per replica (about 1.1 us per replica and sweep, or the work).
inline bool one_launch_branched(const SweepShape& s, int64_t n) {
    // Few large replicas whose tiles take about as long as a sweep's work: 16 of
    // 32,768, 20 sweeps 424 and 467; 25 of 50,000, 12 sweeps 483 and 500 (of 25,000 373
    // and 276).  Tiles of 52 x 70 cells: 31 of 40,000 509 and 569 (of 30,000 469 and 396).
    if (s.fixed && s.R > 1 && s.R <= 25 && s.rounds < 2 && s.tile >= 4200 && s.replica > 30000) return false;
    if (s.fixed && s.R > 16 && s.replica > 30000 && s.tile < 4000) return false;
    // FP64 tiles are half as large: eight of 65,536, 12 sweeps 399 and 437, twenty of 25,000
    // 358 and 439; 31 of 10,000 432 and 300.
    if (!s.fixed && s.R > 1 && s.rounds > std::max(1.5, s.R / 18.0)) return false;
    if (n >= 3) return true;
    // One or two sweeps: the tiles' start and end.  N = 4096, fixed, one sweep 22.5 and
    // 26.6; N = 2^20 49 and 63, two 84 and 94; FP64 N = 4096 35 and 31, 524,288 53 and 63;
    // 64 replicas of 16,384 93 and 71, 31 of 40,000 65 and 76, 48 of 65,536 138 and 129; two
    // sweeps of eight of 65,536 56 and 61, crowded (cells of 2.5 sigma) 16 of 16,384 113 and
    // 129, eight 110 and 93.
    const double most = s.R / 24.0;
    if (s.R > 16 && s.tile >= 4500 && s.rounds >= 4) return true;
    if (n == 2) return s.rounds <= std::max(1.0, most) && !(s.R > 1 && s.R <= 16 && s.tile >= (s.fixed && s.crowded ? 1200 : 3500));
    return s.rounds <= std::max(s.fixed && !s.crowded && s.R < 16 ? 0.0 : 1.0, most);
}

inline bool one_launch_pays(const SweepShape& s, int64_t n, bool step) {
    if (s.box) return one_launch_boxes(s, n, step);
    if (step && s.R <= 64) return one_launch_branched(s, n);
    // Beyond: the phases are batched launches (17 to 25 us per sweep, or 28 ns per cell),
    // from hd_sweep 31 to 45 us.  Tiles of 4500 cells and more hold their own in any
    // number: 152 replicas of 65,536, 12 sweeps 5099 and 4154.  Smaller ones up to some
    // rounds; 12 sweeps of a step: 70 of 1300 243 and 200, 90 252 and 252, 114 263 and 314,
    // 1000 (24 sweeps) 1348 and 5696; 76 of 16,384 633 and 636, 200 1635 and 1773; FP64 90 of
    // 1300 347 and 319, 114 of 2000 449 and 467; crowded, cells of 2.5 sigma, 70 of 4096
    // 644 and 707 (FP64 1347 and 1244), 90 of 2000 699 and 820.
    // A single sweep whose last round of tiles is nearly empty: one replica of 800,000
    // (1.05 rounds) 55 and 62, 1,500,000 (2.03) 76 and 82; 2^20 (1.5) 65 and 62.
    if (!step && n == 1 && s.R == 1 && s.rounds > 1.0 && std::ceil(s.rounds) > 1.4 * s.rounds) return false;
    if (s.tile >= 4500) return true;
    const double t = s.tile;
    double most = 0.0;
    if (step) {
        if (n < 4) return false;  // 70 of 1300, two sweeps 46 and 52, four 90 and 87
        most = s.crowded ? (s.fixed ? 1.5 : 2.0) : !s.fixed ? 2.7 : n < 12 ? 2.1 : t < 1500 ? 2.4 : t < 3400 ? 3.0 : 1e9;
    } else if (n == 1) {
        // 90 of 1300 38 and 46, 31 of 4096 43 and 34; one of 2^21 100 and 88
        if (s.fixed && s.R <= 8) return true;
        most = s.crowded ? 1.0 : 1.5;
    } else if (n == 2) {
        // 114 of 1300 74 and 71, 130 74 and 78; 31 of 40,000 144 and 116
        if (s.R <= 64 && !s.crowded) return true;
        most = s.crowded ? 1.0 : !s.fixed ? 2.4 : t < 2000 ? 3.0 : t < 3400 ? 5.0 : 1e9;
    } else {
        // 12 sweeps: 130 of 1300 392 and 367, 152 397 and 429; 200 of 10,000 1154 and 1110, 304 1708
        // and 1771; FP64 130 of 1300 515 and 469, 152 of 2000 612 and 631
        most = s.crowded ? 1.7 : !s.fixed ? 3.5 : t < 1500 ? 3.4 : t < 2900 ? 5.5 : t < 3400 ? 16.0 : 1e9;
    }
    return s.rounds <= most;
}

}  // namespace hd
