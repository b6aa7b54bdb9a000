// step_plan.h -- how the steps of a call are launched on a D2Q9 grid: one by one, or several per launch
// (tile_kernels.cu). Host code without CUDA.
#pragma once

#include <algorithm>
#include <cmath>

namespace lbm {

// Costs are microseconds on GB300, measured on square grids of 40 to 304 cells with FP32 storage: a
// launch over regions of 16, 24 or 32 cells squared takes fixed + per_step * steps where all its blocks fit
// the SMs at once, one each; single steps (two launches each in the finite-difference variant) take a
// floor, or a part that grows with the grid's side. Plans of more blocks than SMs are left out, and of the
// others the cheapest for the steps of the call is taken, if single steps are not cheaper still.
//   side       40    64    96    128   184   216   256   304
//   single     1.49  1.49  1.61  1.68  2.18  2.19  2.38  2.71   (difference-free, FP32)
//   chosen     0.91  0.96  1.03  1.54  1.74  1.99  single single
//   single     2.64  2.70  2.76  2.96  3.79  3.88  4.30  5.00   (finite-difference, two launches)
//   chosen     1.10  1.39  1.41  1.86  2.25  2.83  3.40  single
// (single: blocks of whole rows; packed ones are up to 5% faster at sides of 184, 216 and 304)
struct TileCost {
    int region;
    double fixed, per_step;
};
constexpr TileCost kTileDf[] = {{16, 1.52, 0.66}, {24, 3.1, 0.90}};
constexpr TileCost kTileFd[] = {{16, 1.9, 0.45}, {24, 2.6, 0.90}, {32, 3.7, 1.45}};

struct StepPlan {
    int region;   // 0: single steps
    int parts;    // launches over regions, n / parts or one more steps each
    double cost;  // of the call by the figures above
};

// The launches of n steps on an nx x ny grid. The choice depends on n: two steps over 24-cell regions cost
// 4.9 us where two single ones of 184^2 cost 4.0, and 32 of them less than 32 single ones. parity: launches
// even or odd in number as n is, so that the state ends in the buffer that single steps would leave it in.
inline StepPlan plan_steps(int nx, int ny, bool fd, int n, bool parity, int sms) {
    const double side = std::sqrt((double)nx * ny);
    const double single = fd ? std::max(2.65, 1.2 + 0.0125 * side) : std::max(1.48, 0.95 + 0.0058 * side);
    StepPlan best{0, 0, n * single};
    auto consider = [&](const TileCost& k) {
        for (int steps = 2; steps <= 8; ++steps) {
            int parts = n / steps + (n % steps != 0);
            if (parity && ((parts ^ n) & 1)) ++parts;
            if (parts >= n) continue;
            const int most = n / parts + (n % parts != 0), tile = k.region - 2 * most * (fd ? 2 : 1);
            if (tile < 4) continue;
            const long long blocks = (long long)((nx + tile - 1) / tile) * ((ny + tile - 1) / tile);
            const double cost = parts * k.fixed + n * k.per_step;
            if (blocks <= sms && cost < best.cost) best = StepPlan{k.region, parts, cost};
        }
    };
    if (fd)
        for (const TileCost& k : kTileFd) consider(k);
    else
        for (const TileCost& k : kTileDf) consider(k);
    return best;
}

}  // namespace lbm
