// How the tile kernels' work is cut into items (host code without CUDA).
//
// An item is a tile, or one of `parts` parts of its particles where whole tiles are too few, or
// too long, to fill the device evenly. Each part stages the field window and adds its own
// current window, and the parts of a tile take their slots of the next buffer from the tile's
// counters in global memory. The current is an integer sum and its rounding follows the tile's
// population, so the result does not depend on the split.
#pragma once

#include <algorithm>
#include <cmath>

namespace pic {

constexpr int kPartUnit = 256;   // a part holds whole multiples of this: the threads of a CTA
constexpr int kMaxParts = 256;

// Particles per item where `tiles` tiles hold `mean` particles each and the device holds
// `resident` CTAs. The split in p minimises (rounds + 0.4) (mean / p + 500) [x 1.04 if p > 1],
// rounds = tiles x p / resident (1 in all where they fit at once): an item costs its
// particles and its window, worth about 500 of them (8 us of one CTA, measured from 4 to 8
// parts of 2048 x 512 cells); a launch of several rounds ends, on average, in a partly empty
// one; counters in global memory cost 4%. Measured (tile kernel per step, us, one part / the
// chosen split / twice it): 128 x 128 cells, 100 per cell 1046 / 158 (14) / 171; 64 x 64, 8 per
// cell 75 / 21 (32) / 21; 1413 x 247, 50 per cell 989 / 971 (5) / 978; twelve scan simulations
// 1347 / 1176 (3) / 1243; 2048 x 512, 32 per cell 2698 (1, chosen) / 2666 (2) / 2881 (4).
inline double split_size(double tiles, double resident, double mean) {
    double size = mean, best = -1.0;
    for (int p = 1; p <= kMaxParts && (p == 1 || mean / p >= kPartUnit); p++) {
        const double rounds = tiles * p / resident;
        const double cost = (rounds <= 1.0 ? 1.0 : rounds + 0.4) * (mean / p + 500.0) * (p > 1 ? 1.04 : 1.0);
        if (best < 0.0 || cost < best) {
            best = cost;
            size = mean / p;
        }
    }
    return size;
}

// A tile that may hold up to `full` particles before its bins are rebuilt, and holds `mean` on
// average: as many parts of the wanted size, but one up to 1.9 sizes (a split tile's counters
// cost more than its late end). Where a tile holds fewer particles, its last parts find nothing
// to push; where it holds more, all its parts take equal shares. A part that finds nothing
// costs 0.8 us of a CTA, about 50 particles: no more of them than 5% of a mean tile's work.
// (2048 x 512, 8 per cell, 2% of all particles in one tile, whose bins are 20 times the mean's:
// 4122 us per step as whole tiles, 1152 with 256 parts, 984 with 21, 892 with 9.)
struct TileSplit {
    int parts, pchunk;
};
inline TileSplit split_tile(double full, double mean, double size) {
    TileSplit t;
    size = std::max(size, (double)kPartUnit);
    const double most = std::min((double)kMaxParts, mean / size + mean / 1000.0);
    t.parts = full < 1.9 * size ? 1 : std::max(1, (int)std::floor(std::min(full / size, most) + 0.5));
    t.pchunk = ((int)std::min(std::ceil(size), 1e9) + kPartUnit - 1) / kPartUnit * kPartUnit;
    return t;
}

}  // namespace pic
