// step_plan.h -- how steps are launched: the blocks of a single step (step_kernels.cu), and on a D2Q9 grid how many
// steps of a call share a launch (tile_kernels.cu). Host code without CUDA.
#pragma once

#include <algorithm>
#include <cmath>

namespace lbm {

constexpr int kStepThreads = 128;  // of a block of a single step, one cell each

// i / nx (nx > 1) for i < 2^31 as a product, the high word of i mul shifted right by `shift`: mul =
// ceil(2^(32 + shift) / nx), 2^shift < nx <= 2^(shift + 1). The excess mul nx - 2^(32 + shift) is below nx <=
// 2^(shift + 1), so i times it stays below 2^(32 + shift).
struct RowDiv {
    unsigned mul;
    int shift;
};

// How a step's blocks lie and address: whole rows or 32 x 4 cells, packed, or whole blocks with 64-bit
// addresses for the 16-bit D3Q19 planes of 4 GiB and more (2^29 cells), where a byte offset does not fit.
enum StepForm { WHOLE = 0, PACKED = 1, WIDE = 2 };

// Blocks of one 128-cell row where rows are at least that long, else 32 x 4 (a warp spans 32 consecutive
// cells of a row either way); where such blocks would stand over the grid's edges, packed ones, which
// leave no lane idle but in a plane's last block. Packed blocks cost a product per cell to find the
// row: 0.4% at 128^3 (59.98 against 60.36 us FP16, 93.16 against 93.39 FP32), so whole blocks stay where
// they fit. Where they do not, packed ones were faster at every size tried (us per step):
//   grid              33^3  33^3   97x96x96  126^3  130^3  130^3   200^3   200^3   94x75x301  600^2  330x270
//                     FP16  FP32*  FP32*     FP16   FP16   FP32    BF16    FP32    BF16*      FP32   FP32
//   whole blocks      3.31  4.30   51.2      61.1   84.6   115.5   266.0   373.6   74.1       6.13   2.87
//   packed            2.42  3.30   44.0      60.0   65.7   99.7    231.2   349.1   72.6       5.85   2.65
// (* walls and a density ratio)
struct StepShape {
    unsigned block[2], grid[3];
    StepForm form;
    RowDiv d;
};

inline StepShape step_shape(int nx, int ny, int nz, bool d3q19_16bit) {
    StepShape h{{nx >= 128 ? 128u : 32u, nx >= 128 ? 1u : 4u}, {0u, 0u, (unsigned)nz}, WHOLE, {0u, 0}};
    h.grid[0] = (nx + h.block[0] - 1) / h.block[0];
    h.grid[1] = (ny + h.block[1] - 1) / h.block[1];
    const unsigned blocks = ((unsigned)nx * (unsigned)ny + kStepThreads - 1) / kStepThreads;
    if (nx > 1 && blocks < h.grid[0] * h.grid[1]) h.form = PACKED;
    if (d3q19_16bit && (long long)nx * ny * nz >= (1ll << 29)) h.form = WIDE;
    if (h.form == PACKED) {
        h.block[0] = kStepThreads;
        h.block[1] = 1;
        h.grid[0] = blocks;
        h.grid[1] = 1;
        while ((2ll << h.d.shift) < nx) ++h.d.shift;
        h.d.mul = (unsigned)(((1ull << (32 + h.d.shift)) + nx - 1) / nx);
    }
    return h;
}

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
