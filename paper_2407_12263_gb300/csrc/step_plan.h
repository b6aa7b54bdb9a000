// step_plan.h -- how the steps of a call are launched on a D2Q9 grid: one by one, or several per launch
// (tile_kernels.cu). Host code without CUDA.
#pragma once

#include <algorithm>
#include <cmath>

namespace lbm {

constexpr int kTileSide = 16;  // cells squared of a block's region
constexpr int kTileResident = 3;  // such blocks on an SM at once (256 threads of up to 80 registers)

struct StepPlan {
    int parts;    // launches over regions, n / parts or one more steps each; 0: single steps
    double cost;  // of the call, alone on the GPU, by the figures below
};

// The launches of n steps on an nx x ny grid. Costs are microseconds on GB300, measured on square grids with
// FP32 storage. A launch over regions takes fixed + per_step * steps, a quarter more for every further block
// that an SM has to hold, up to three. Single steps (two launches each in the finite-difference variant) take a
// floor, or a part that grows with the grid's side. The choice depends on n: a plan is taken for the launches
// that the call would make. parity: these are even or odd in number as n is, so that the state ends in the buffer
// that single steps would leave it in.
//
// Regions overlap, so that they occupy more of the chip than single steps do, which other handles may want:
// a plan is taken only where four handles side by side, each on its own stream, are about as fast with it as
// with single steps. Then blocks * their time / (blocks that the SMs hold) of a handle add up (measured
// times are 1.0 to 1.2 of that). Microseconds a step, 32 steps a call:
//   handles              1     2     4     8     16        1     2     4     8     16
//   side                 difference-free                   finite-difference
//   64   single steps    1.55  1.67  1.82  2.11  3.58      2.72  2.83  3.25  3.84  7.06
//        regions         1.01  1.11  1.47  2.15  4.11      1.41  1.40  1.72  2.10  3.60
//   96   single steps    1.63  1.75  2.09  2.41  3.76      2.85  3.20  3.74  4.34  7.49
//        regions         1.05  1.18  1.77  3.19  6.32      1.44  1.68  2.19  3.97  7.89
//   128  single steps    1.69  1.90  2.35  2.86  4.03      3.04  3.60  4.25  5.23  8.12
//        regions         1.56  1.92  2.24  3.58  7.11      1.76  2.33  3.52  6.99  13.97
//   184  single steps    2.00  2.33  2.91  3.95  8.04      3.41  4.33  5.42  7.39  14.43
//        regions         not taken (2.02, 4.61)            2.72  3.39  5.30  10.50 23.58
//   216  single steps    2.14  2.55  3.22  5.27  12.94     3.87  4.85  6.20  9.75  21.13
//        regions         not taken (2.27, 4.71)            not taken (3.29, 6.65)
// (not taken: alone, and four side by side.) Regions of 24 and 32 cells squared hold one block an SM: alone up to
// a quarter faster at sides of 184 to 256 (2.32 us at 184, finite-difference), but four side by side
// twice as slow as single steps (7.67), so there are none.
inline StepPlan plan_steps(int nx, int ny, bool fd, int n, bool parity, int sms) {
    const double side = std::sqrt((double)nx * ny);
    const double fixed = fd ? 1.58 : 1.52, per_step = fd ? 0.62 : 0.66;
    const double single = fd ? std::max(2.65, 1.2 + 0.0125 * side) : std::max(1.48, 0.95 + 0.0058 * side);
    const double single4 = fd ? 1.9 + 0.0195 * side : 1.1 + 0.0105 * side;
    StepPlan best{0, n * single};
    if (n < 2) return best;
    for (int steps = fd ? 1 : 2; steps <= 6; ++steps) {  // one is worth it where it replaces two launches
        int parts = n / steps + (n % steps != 0);
        if (parity && ((parts ^ n) & 1)) ++parts;
        if (parts >= n && !fd) continue;
        const int most = n / parts + (n % parts != 0), tile = kTileSide - 2 * most * (fd ? 2 : 1);
        if (tile < 4) continue;
        const double blocks = (double)((nx - 1) / tile + 1) * ((ny - 1) / tile + 1), held = (double)kTileResident * sms;
        if (blocks > held) continue;
        const double work = parts * fixed + n * per_step;
        if (4 * 1.1 * blocks * work / held > n * single4) continue;
        const double cost = work * (0.75 + 0.25 * std::ceil(blocks / sms));
        if (cost < best.cost) best = StepPlan{parts, cost};
    }
    return best;
}

}  // namespace lbm
