// surrogate_glue.cu -- field transfers between the lattice and the surrogate's coarse grid:
// block means of the macroscopic fields, the restart from trilinearly upsampled coarse fields
// (the same equilibrium-plus-non-equilibrium construction as the initial state, in FP32), and
// the exact correction of sum phi after a restart.
#include <algorithm>

#include "cell.cuh"
#include "surrogate.h"

namespace lbm {

// The fields of one cell that are averaged: the fixed-point phi, u and P = p / cs^2 - w0 (m.P) of
// the propagated state, by the code of the time step: populations stay in storage units until
// the moments, and only warps that hold a wall cell test their links against the walls.
template <int Q, int S, bool GEN>
__device__ __forceinline__ void coarse_cell(const Params& P, const void* __restrict__ fg, int x, int y, int z, Macro& m,
                                            int& phi_fx) {
    const Nbr nb = make_nbr(P, x, y, z);
    const int c = (z * P.ny + y) * P.nx + x;
    const WallSide ws = GEN ? make_wall_side(P, x, y, z) : WallSide{};
    float fb[Q], gb[Q];
    const bool at_wall = GEN && (ws.xlo || ws.xhi || ws.ylo || ws.yhi || ws.zlo || ws.zhi);
    if (GEN && __any_sync(__activemask(), at_wall))
        pull<Q, true, S, true, true>(P, fg, c, nb, fb, gb, phi_fx, ws);
    else
        pull<Q, true, S, false, true>(P, fg, c, nb, fb, gb, phi_fx);
    macro_flow<Q, GEN, S>(P, fb, gb, m);
    macro_interface_df<Q, S>(P, m);
    macro_pressure<GEN>(P, m);
}

// A sum of FP32 values held as an unevaluated pair (Knuth's two-sum: the rounding error of every
// addition goes to lo), about 48 bits. GB300 issues an FP64 instruction per SM and 16 cycles for
// a warp, so FP64 sums of four fields per cell (a conversion and an addition each) alone took as
// long as the cell's bytes; a two-sum is seven FP32 instructions.
struct Sum2 {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float s = __fadd_rn(hi, v), t = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(v, t)));
        hi = s;
    }
    __device__ __forceinline__ void add(const Sum2& o) {
        add(o.hi);
        lo = __fadd_rn(lo, o.lo);
    }
    // the sum rounded once to FP32
    __device__ __forceinline__ float rounded() const { return isfinite(hi) ? __fadd_rn(hi, lo) : hi; }
    // where hi is infinite or NaN, lo is NaN and the sum is hi
    __device__ __forceinline__ double value() const { return isfinite(hi) ? (double)hi + (double)lo : (double)hi; }
};

// The sums of a thread's cells: phi exactly in fixed point, u and P in pairs of FP32.
struct CoarseSums {
    long long phi = 0;
    Sum2 v[4];  // u, P
    __device__ __forceinline__ void add(const Macro& m, int phi_fx) {
        phi += phi_fx;
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a].add(m.u[a]);
        v[3].add(m.P);
    }
};

// Means of n cells from their sums into coarse cell l of nc: p = cs^2 (w0 + mean P).
__device__ __forceinline__ void store_means(const Params& P, long long phi, const double (&s)[4], double n,
                                            float* __restrict__ out, long long nc, long long l) {
    const double inv = 1.0 / n;
    out[l] = (float)((double)phi * (inv / kPhiFx));
#pragma unroll
    for (int a = 0; a < 3; ++a) out[(1 + a) * nc + l] = (float)(s[a] * inv);
    out[4 * nc + l] = (float)((P.w0d + s[3] * inv) / 3.0);
}

constexpr int kCoarseThreads = 128;

// Register budgets as the time step's: the loads of a cell stay in flight at 4 blocks (FP32
// storage, 128 registers) or 5 (16-bit, 96 registers) per SM. The periodic FP32 kernels that also
// hold a thread's sums spill 84 bytes at 4 and take 3.
template <int S, bool GEN, bool SUMS>
constexpr int coarse_min_blocks() {
    return S != STORE_F32 ? 5 : (SUMS && !GEN) ? 3 : 4;
}

// p = cs^2 (w0 + P) rounded to FP32 without an FP64 instruction, w0 = P.w0 + w0_lo: an exact sum,
// and a division by 3 corrected by its remainder, rounds as the FP64 expression does but for ties.
__device__ __forceinline__ float pressure_of(const Params& P, float w0_lo, const Sum2& mean) {
    Sum2 w;
    w.hi = P.w0;
    w.lo = w0_lo;
    w.add(mean);
    constexpr float third = 1.0f / 3.0f;
    const float q = w.hi * third;
    const float r = fmaf(-3.0f, q, w.hi) + w.lo;
    return isfinite(w.hi) ? fmaf(r, third, q) : w.hi;
}

// Factor 1: the fields of every cell. Bound by the state's bytes: 128^3 takes 61 us in FP32 (5.2 TB/s)
// and 41 us in FP16 (4.1 TB/s), where FP64 sums and a division per cell took 203 and 187 us.
template <int Q, int S, bool GEN>
__global__ void __launch_bounds__(kCoarseThreads, (coarse_min_blocks<S, GEN, false>()))
fields_kernel(const Params P, const void* __restrict__ fg, float w0_lo, float* __restrict__ out) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= P.nx || y >= P.ny) return;
    Macro m;
    int phi_fx;
    coarse_cell<Q, S, GEN>(P, fg, x, y, z, m, phi_fx);
    Sum2 dev;
    dev.hi = m.P;
    float* o = out + ((size_t)z * P.ny + y) * P.nx + x;
    const size_t n = (size_t)P.N;
    __stcs(o, __int2float_rn(phi_fx) * kPhiFxInvF);  // one rounding: 2^-30 is exact
    __stcs(o + n, m.u[0]);
    __stcs(o + 2 * n, m.u[1]);
    __stcs(o + 3 * n, m.u[2]);
    __stcs(o + 4 * n, pressure_of(P, w0_lo, dev));
}

// Block means over f^3 cells for factors f > 1 that divide 32: a block takes 32 consecutive fine x
// of one coarse row, its four warps four of the f x f fine rows behind it at a time (neighbouring
// rows together, so that they share their stencils in L1). phi is summed as integers and u in
// pairs, so their order does not matter. The pressures are FP64 sums of rounded thirds, taken row
// by row per lane and then across the f lanes of a coarse cell: their last bit depends on that
// order, and a restart in 16-bit storage amplifies it, so it is fixed. The third of an FP64 value
// is a product corrected by its remainder (the rounding of a division by 3, without its call),
// which leaves six FP64 instructions per cell, fewer cycles than the rest of the cell.
// f^3 is a power of two: the means of phi and u are FP32 roundings of their sums.
// 256^3 at f = 4: 812 -> 380 us (FP16), 937 -> 613 us (FP32), at f = 2 925 -> 471 and 1018 -> 783 us; bound
// by the propagation's instructions (16-bit) and its load latency (FP32).
constexpr int kCoarseWarps = kCoarseThreads / 32;
constexpr int kMaxGridY = 65535;

__device__ __forceinline__ double third_of(double x) {
    constexpr double third = 1.0 / 3.0;
    const double q = __dmul_rn(x, third);
    const double t = fma(fma(-3.0, q, x), third, q);
    return isfinite(t) ? t : q;
}

// TALL: more coarse rows than a grid holds blocks in y go on with the next ncz planes of blocks. A form of its
// own: with it alone 256^3 at f = 2 takes 788 us instead of 782 (FP32) and 513 instead of 498 (BF16).
template <int Q, int S, bool GEN, bool TALL>
__global__ void __launch_bounds__(kCoarseThreads, (coarse_min_blocks<S, GEN, true>()))
coarsen_lanes_kernel(const Params P, const void* __restrict__ fg, int f, int ncy, int ncz, float* __restrict__ out) {
    __shared__ float2 s_u[kCoarseWarps][3][32];
    __shared__ long long s_phi[kCoarseWarps][32];
    __shared__ double s_p[2][kCoarseWarps][32];
    const int lane = threadIdx.x, warp = threadIdx.y;
    int cy = blockIdx.y, cz = blockIdx.z;
    if (TALL) {
        for (; cz >= ncz; cz -= ncz) cy += kMaxGridY;
        if (cy >= ncy) return;  // whole blocks
    } else {
        ncy = gridDim.y;
        ncz = gridDim.z;
    }
    const int x = blockIdx.x * 32 + lane;
    const bool valid = x < P.nx;  // whole groups of f lanes are valid or not: f divides nx and 32
    long long phi = 0;
    Sum2 u[3];
    double p = 0.0;  // in warp 0, of the lane's rows so far
    for (int r0 = 0, k = 0; r0 < f * f; r0 += kCoarseWarps, k ^= 1) {  // f * f is a multiple of 4
        if (valid) {
            Macro m;
            int phi_fx;
            const int r = r0 + warp, dz = r / f;
            coarse_cell<Q, S, GEN>(P, fg, x, cy * f + (r - dz * f), cz * f + dz, m, phi_fx);
            phi += phi_fx;
#pragma unroll
            for (int a = 0; a < 3; ++a) u[a].add(m.u[a]);
            s_p[k][warp][lane] = third_of(P.w0d + (double)m.P);
        }
        __syncthreads();  // the other buffer is written only after every warp has passed the next one
        if (warp == 0 && valid)
            for (int w = 0; w < kCoarseWarps; ++w) p += s_p[k][w][lane];
    }
    s_phi[warp][lane] = phi;
#pragma unroll
    for (int a = 0; a < 3; ++a) s_u[warp][a][lane] = make_float2(u[a].hi, u[a].lo);
    __syncthreads();
    if (warp != 0) return;
    for (int w = 1; w < kCoarseWarps; ++w) {
        phi += s_phi[w][lane];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            Sum2 o;
            o.hi = s_u[w][a][lane].x;
            o.lo = s_u[w][a][lane].y;
            u[a].add(o);
        }
    }
    for (int o = f >> 1; o > 0; o >>= 1) {
        phi += __shfl_xor_sync(0xffffffffu, phi, o);
        p += __shfl_xor_sync(0xffffffffu, p, o);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            Sum2 other;
            other.hi = __shfl_xor_sync(0xffffffffu, u[a].hi, o);
            other.lo = __shfl_xor_sync(0xffffffffu, u[a].lo, o);
            u[a].add(other);
        }
    }
    if (!valid || lane % f) return;
    const float inv = 1.0f / (float)(f * f * f);
    const int ncx = P.nx / f;
    const long long nc = (long long)ncx * ncy * ncz;
    float* o = out + ((long long)cz * ncy + cy) * ncx + x / f;
    o[0] = __ll2float_rn(phi) * (kPhiFxInvF * inv);
#pragma unroll
    for (int a = 0; a < 3; ++a) o[(1 + a) * nc] = u[a].rounded() * inv;
    o[4 * nc] = (float)(p * (double)inv);
}

// Any other factor up to kRowLanes: a block row of kRowLanes threads takes floor(kRowLanes / f)
// whole coarse cells of one coarse row, each thread the f x f cells behind one fine x
// (consecutive threads read consecutive cells), and one thread per coarse cell adds its f columns.
// 192^3 FP32 at f = 3: 261 us, where one thread per coarse cell, which reads f cells apart, took 968 us; that
// form stays for larger factors, whose blocks would hold no whole coarse cell.
constexpr int kRowLanes = 64, kRowRows = kCoarseThreads / kRowLanes;

template <int Q, int S, bool GEN>
__global__ void __launch_bounds__(kCoarseThreads, (coarse_min_blocks<S, GEN, true>()))
coarsen_rows_kernel(const Params P, const void* __restrict__ fg, int f, float* __restrict__ out) {
    __shared__ double s_acc[kRowRows][4][kRowLanes];
    __shared__ long long s_phi[kRowRows][kRowLanes];
    const int t = threadIdx.x, r = threadIdx.y;
    const int per = kRowLanes / f;  // coarse cells of a block row
    const int x = blockIdx.x * per * f + t;
    const int cy = blockIdx.y * kRowRows + r;
    const int cz = blockIdx.z;
    const int ncx = P.nx / f, ncy = P.ny / f, ncz = P.nz / f;
    if (cy < ncy && t < per * f && x < P.nx) {
        CoarseSums sums;
        for (int dz = 0; dz < f; ++dz)
            for (int dy = 0; dy < f; ++dy) {
                Macro m;
                int phi_fx;
                coarse_cell<Q, S, GEN>(P, fg, x, cy * f + dy, cz * f + dz, m, phi_fx);
                sums.add(m, phi_fx);
            }
        s_phi[r][t] = sums.phi;
#pragma unroll
        for (int k = 0; k < 4; ++k) s_acc[r][k][t] = sums.v[k].value();
    }
    __syncthreads();
    const int cx = blockIdx.x * per + t;
    if (cy >= ncy || t >= per || cx >= ncx) return;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    long long phi = 0;
    for (int j = t * f; j < (t + 1) * f; ++j) {
        phi += s_phi[r][j];
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] += s_acc[r][k][j];
    }
    store_means(P, phi, acc, (double)f * f * f, out, (long long)ncx * ncy * ncz, ((long long)cz * ncy + cy) * ncx + cx);
}

template <int Q, int S, bool GEN>
__global__ void __launch_bounds__(kCoarseThreads, (coarse_min_blocks<S, GEN, true>()))
coarsen_cells_kernel(const Params P, const void* __restrict__ fg, int f, float* __restrict__ out) {
    const int cx = blockIdx.x * blockDim.x + threadIdx.x;
    const int cy = blockIdx.y * blockDim.y + threadIdx.y;
    const int cz = blockIdx.z;
    const int ncx = P.nx / f, ncy = P.ny / f, ncz = P.nz / f;
    if (cx >= ncx || cy >= ncy) return;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    long long phi = 0;
    for (int dz = 0; dz < f; ++dz)
        for (int dy = 0; dy < f; ++dy) {
            CoarseSums sums;
            for (int dx = 0; dx < f; ++dx) {
                Macro m;
                int phi_fx;
                coarse_cell<Q, S, GEN>(P, fg, cx * f + dx, cy * f + dy, cz * f + dz, m, phi_fx);
                sums.add(m, phi_fx);
            }
            phi += sums.phi;
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[k] += sums.v[k].value();
        }
    store_means(P, phi, acc, (double)f * f * f, out, (long long)ncx * ncy * ncz, ((long long)cz * ncy + cy) * ncx + cx);
}

template <int Q, int S, bool GEN>
static void coarsen_qsg(const Params& P, const void* fg, int f, float* out, cudaStream_t s) {
    const int ncx = P.nx / f, ncy = P.ny / f, ncz = P.nz / f;
    const float w0_lo = (float)(P.w0d - (double)P.w0);
    if (f == 1) {
        const dim3 block = P.nx >= 128 && P.ny <= kMaxGridY ? dim3(128, 1) : dim3(32, 4);
        const dim3 grid((P.nx + block.x - 1) / block.x, (P.ny + block.y - 1) / block.y, P.nz);
        fields_kernel<Q, S, GEN><<<grid, block, 0, s>>>(P, fg, w0_lo, out);
        return;
    }
    if constexpr (Q == 19) {  // D2Q9 grids have nz = 1, which only factor 1 divides
        if (32 % f == 0) {
            const int chunks = (ncy + kMaxGridY - 1) / kMaxGridY;
            const dim3 block(32, kCoarseWarps), grid((P.nx + 31) / 32, std::min(ncy, kMaxGridY), ncz * chunks);
            if (chunks > 1) coarsen_lanes_kernel<Q, S, GEN, true><<<grid, block, 0, s>>>(P, fg, f, ncy, ncz, out);
            else coarsen_lanes_kernel<Q, S, GEN, false><<<grid, block, 0, s>>>(P, fg, f, ncy, ncz, out);
        } else if (f <= kRowLanes) {
            const int per = kRowLanes / f;
            coarsen_rows_kernel<Q, S, GEN><<<dim3((ncx + per - 1) / per, (ncy + kRowRows - 1) / kRowRows, ncz),
                                             dim3(kRowLanes, kRowRows), 0, s>>>(P, fg, f, out);
        } else {
            coarsen_cells_kernel<Q, S, GEN><<<dim3((ncx + 31) / 32, (ncy + 3) / 4, ncz), dim3(32, 4), 0, s>>>(P, fg, f, out);
        }
    }
}

cudaError_t launch_coarsen(const Params& P, const void* fg, int factor, float* out, cudaStream_t s) {
#define LBM_COARSEN(Q, S) \
    (P.general ? coarsen_qsg<Q, S, true>(P, fg, factor, out, s) : coarsen_qsg<Q, S, false>(P, fg, factor, out, s))
    if (P.Q == 9) {
        if (P.storage == STORE_F16) LBM_COARSEN(9, STORE_F16);
        else if (P.storage == STORE_BF16) LBM_COARSEN(9, STORE_BF16);
        else LBM_COARSEN(9, STORE_F32);
    } else {
        if (P.storage == STORE_F16) LBM_COARSEN(19, STORE_F16);
        else if (P.storage == STORE_BF16) LBM_COARSEN(19, STORE_BF16);
        else LBM_COARSEN(19, STORE_F32);
    }
#undef LBM_COARSEN
    return cudaGetLastError();
}

// What the sum of a restarted state's fixed-point phi must be raised by, cell by cell: every cell by
// q and the first |r| cells by the sign of r more, q N + r = before - the sum of the slots (the sums of
// the restarted blocks). Read by one thread of a block; the others take it from shared memory.
struct Balance {
    const long long* before;  // NULL: nothing to add
    const unsigned long long* slots;
    int n_slots;
    long long N;
};
__device__ __forceinline__ void balance_of(const Balance& B, long long (&s_qr)[2]) {
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        unsigned long long after = 0;
        for (int i = 0; i < B.n_slots; ++i) after += B.slots[i];
        const long long delta = *B.before - (long long)after;
        s_qr[0] = delta / B.N;
        s_qr[1] = delta - s_qr[0] * B.N;
    }
    __syncthreads();
}
__device__ __forceinline__ int balanced(int phi_fx, long long c, const long long (&qr)[2]) {
    const long long ar = qr[1] < 0 ? -qr[1] : qr[1];
    const long long add = qr[0] + (c < ar ? (qr[1] < 0 ? -1 : 1) : 0);
    return (int)((unsigned int)phi_fx + (unsigned int)add);
}

// Block means over F^3 cells of the state's own phi, the fixed-point value of plane 0 (no
// propagation: 8 bytes read per cell), after the balance has been added and stored, if there is one.
// Lane l of a warp takes fine x = 32 b + l; F divides 32, and each aligned group of F lanes is summed
// with shuffles. With the factor known the loads of eight rows are in flight at once: 128^3 at F = 2
// 18 -> 6 us, 9 us with the balance (8.6 us as a pass of its own).
template <int F, bool BALANCE>
__global__ void __launch_bounds__(128) coarse_phi_kernel(float2* plane0, int nx, int ny, int nz, const Balance B,
                                                         float* __restrict__ out) {
    __shared__ long long s_qr[2];
    chain_begin();
    chain_next();
    if (BALANCE) balance_of(B, s_qr);
    const int lane = threadIdx.x;
    const int x = blockIdx.x * 32 + lane;
    const int cy = blockIdx.y * blockDim.y + threadIdx.y;
    const int cz = blockIdx.z;
    const int ncx = nx / F, ncy = ny / F;
    if (cy >= ncy) return;  // whole warps leave together
    const bool valid = x < nx;
    constexpr int kRows = F * F, kStep = kRows < 8 ? kRows : 8;
    long long acc = 0;
    if (valid)
        for (int r0 = 0; r0 < kRows; r0 += kStep) {
            long long c[kStep];
            int v[kStep];
#pragma unroll
            for (int k = 0; k < kStep; ++k) {
                const int r = r0 + k;
                c[k] = ((long long)(cz * F + r / F) * ny + (cy * F + r % F)) * nx + x;
                v[k] = __float_as_int(plane0[c[k]].y);
            }
#pragma unroll
            for (int k = 0; k < kStep; ++k) {
                if (BALANCE) {
                    v[k] = balanced(v[k], c[k], s_qr);
                    plane0[c[k]].y = __int_as_float(v[k]);
                }
                acc += v[k];
            }
        }
#pragma unroll
    for (int o = F >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (!valid || lane % F) return;
    out[((long long)cz * ncy + cy) * ncx + x / F] = (float)((double)acc / (kPhiFx * (double)F * F * F));
}

__global__ void balance_kernel(float2* __restrict__ plane0, const Balance B) {
    __shared__ long long s_qr[2];
    balance_of(B, s_qr);
    if (s_qr[0] == 0 && s_qr[1] == 0) return;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < B.N; c += (long long)gridDim.x * blockDim.x)
        plane0[c].y = __int_as_float(balanced(__float_as_int(plane0[c].y), c, s_qr));
}

static unsigned cell_blocks(long long n) { return (unsigned)std::min<long long>((n + 255) / 256, 4096); }

static Balance balance_of_restart(const Params& P, const RestartSums* sums) {
    return sums ? Balance{sums->before, sums->slots, sums->n_slots, P.N} : Balance{nullptr, nullptr, 0, P.N};
}

cudaError_t launch_balance(const Params& P, void* fg, const RestartSums& sums, cudaStream_t s) {
    balance_kernel<<<cell_blocks(P.N), 256, 0, s>>>(moment_plane(fg), balance_of_restart(P, &sums));
    return cudaGetLastError();
}

template <int F>
static cudaError_t coarse_phi_f(const Params& P, void* fg, const RestartSums* sums, float* out, cudaStream_t s) {
    const dim3 block(32, 4), grid((P.nx + 31) / 32, (P.ny / F + 3) / 4, P.nz / F);
    const Balance B = balance_of_restart(P, sums);
    return launch_chained(sums ? coarse_phi_kernel<F, true> : coarse_phi_kernel<F, false>, grid, block, 0, s, moment_plane(fg), P.nx,
                         P.ny, P.nz, B, out);
}

cudaError_t launch_coarse_phi(const Params& P, void* fg, int factor, const RestartSums* sums, float* out, cudaStream_t s) {
    switch (factor) {
        case 1: return coarse_phi_f<1>(P, fg, sums, out, s);
        case 2: return coarse_phi_f<2>(P, fg, sums, out, s);
        case 4: return coarse_phi_f<4>(P, fg, sums, out, s);
        case 8: return coarse_phi_f<8>(P, fg, sums, out, s);
        case 16: return coarse_phi_f<16>(P, fg, sums, out, s);
        case 32: return coarse_phi_f<32>(P, fg, sums, out, s);
        default: return cudaErrorInvalidValue;
    }
}

// Where fine coordinate i (of n = nc f cells) falls between coarse cell centres: the two coarse
// indices and the weight of the second. Periodic, or clamped to the end centres across a wall.
struct Axis {
    int a, b;
    float t;
};

__device__ __forceinline__ Axis interp_axis(int i, int f, int nc, bool wall) {
    const float xc = ((float)i + 0.5f) / (float)f - 0.5f;
    Axis r;
    r.a = (int)floorf(xc);
    r.t = xc - (float)r.a;
    r.b = r.a + 1;
    if (wall) {
        if (r.a < 0) {
            r.a = 0;
            r.t = 0.f;
        }
        if (r.b > nc - 1) {
            r.b = nc - 1;
            if (r.a == r.b) r.t = 0.f;
        }
    } else {  // r.a is in [-1, nc - 1] and r.b = r.a + 1: one period at most on either side
        if (r.a < 0) r.a += nc;
        if (r.b >= nc) r.b -= nc;
    }
    return r;
}

// The offsets of the eight coarse corners around a fine cell (the coarse grid holds fewer than
// 2^31 cells), computed once for all the fields interpolated there.
struct Corners {
    int o[8];  // (z, y, x) in {a, b}^3, x fastest
    float tx, ty, tz;
};

__device__ __forceinline__ Corners corners(int ncx, int ncy, const Axis& X, const Axis& Y, const Axis& Z) {
    Corners c;
    const int za = Z.a * ncy, zb = Z.b * ncy;
    const int r00 = (za + Y.a) * ncx, r01 = (za + Y.b) * ncx, r10 = (zb + Y.a) * ncx, r11 = (zb + Y.b) * ncx;
    c.o[0] = r00 + X.a;
    c.o[1] = r00 + X.b;
    c.o[2] = r01 + X.a;
    c.o[3] = r01 + X.b;
    c.o[4] = r10 + X.a;
    c.o[5] = r10 + X.b;
    c.o[6] = r11 + X.a;
    c.o[7] = r11 + X.b;
    c.tx = X.t;
    c.ty = Y.t;
    c.tz = Z.t;
    return c;
}

// Trilinear interpolation of q at the corners: along x, then y, then z
__device__ __forceinline__ float trilinear(const float* q, const Corners& c) {
    auto lerp = [](float u, float v, float t) { return fmaf(t, v - u, u); };
    const float c00 = lerp(q[c.o[0]], q[c.o[1]], c.tx);
    const float c01 = lerp(q[c.o[2]], q[c.o[3]], c.tx);
    const float c10 = lerp(q[c.o[4]], q[c.o[5]], c.tx);
    const float c11 = lerp(q[c.o[6]], q[c.o[7]], c.tx);
    return lerp(lerp(c00, c01, c.ty), lerp(c10, c11, c.ty), c.tz);
}

// The upsampled phi of every cell, the first pass of the restart, clamped to [-1, 1.5], the range
// lbm_init_fields accepts, so that its fixed-point value stays in range whatever the prediction holds.
__global__ void phi_fine_kernel(const Params P, const float* coarse, int f, float* __restrict__ phi) {
    chain_begin();
    chain_next();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= P.nx || y >= P.ny) return;
    const int ncx = P.nx / f, ncy = P.ny / f, ncz = P.nz / f;
    const float v = trilinear(coarse, corners(ncx, ncy, interp_axis(x, f, ncx, P.walls & 1),
                                              interp_axis(y, f, ncy, P.walls & 2), interp_axis(z, f, ncz, P.walls & 4)));
    phi[((long long)z * P.ny + y) * P.nx + x] = fminf(fmaxf(v, -1.0f), 1.5f);
}

// The second: the initial-state construction of init_kernel (equilibria of the upsampled phi, u, p plus
// the first-order non-equilibrium part of g, grad phi from the isotropic central difference of the
// upsampled phi) in FP32, directly as deviations from the storage's reference levels. The words of
// opposite pairs are stored whole (a store per population writes half of every sector it touches), and
// the block's sum of the fixed-point phi goes to one of the slots (integer atomics: the same total in
// any order). Bound by instructions: the arithmetic is written with the velocities' zero components,
// and 16-bit restarts, which amplify a last bit, fix its roundings.
template <int Q, int S>
__device__ __forceinline__ int restart_cell(const Params& P, const float* coarse, const float* phi_fine,
                                            int f, float p0, void* __restrict__ fg, int x, int y, int z) {
    const int ncx = P.nx / f, ncy = P.ny / f, ncz = P.nz / f;
    const long long nc = (long long)ncx * ncy * ncz;
    // neighbours: periodic images, or across a wall the cell itself (so that the normal gradient
    // vanishes there); the grid holds fewer than 2^31 cells
    const Nbr nb = mirror_at_walls(make_nbr(P, x, y, z), make_wall_side(P, x, y, z));
    const float* here = phi_fine + ((z * P.ny + y) * P.nx + x);
    const float phi = *here;
    float gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const float v = Lat<Q>::w(i) * here[link_offset<Q>(nb, i, +1)];
        gx += Lat<Q>::cx(i) * v;
        gy += Lat<Q>::cy(i) * v;
        gz += Lat<Q>::cz(i) * v;
    }
    gx *= 3.f;
    gy *= 3.f;
    gz *= 3.f;
    const Corners cc = corners(ncx, ncy, interp_axis(x, f, ncx, P.walls & 1), interp_axis(y, f, ncy, P.walls & 2),
                               interp_axis(z, f, ncz, P.walls & 4));
    const float u[3] = {trilinear(coarse + nc, cc), trilinear(coarse + 2 * nc, cc), trilinear(coarse + 3 * nc, cc)};
    const float pc = trilinear(coarse + 4 * nc, cc);
    const float g2 = gx * gx + gy * gy + gz * gz;
    const float gn = sqrtf(g2);
    const float inv = (g2 > kNormalGuard) ? 1.0f / gn : 0.f;
    const float n[3] = {gx * inv, gy * inv, gz * inv};
    const float smag = P.four_over_delta * phi * (1.f - phi);
    const float Sv[3] = {smag * n[0], smag * n[1], smag * n[2]};
    const float rho = P.rho2 + P.drho * phi;
    const float u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const float sg = P.sigma * gn;
    const float trc3 = ((float)Lat<Q>::D - (n[0] * n[0] + n[1] * n[1] + n[2] * n[2])) * (1.0f / 3.0f);
    const float dP = 3.f * (pc - p0);  // p / cs^2 - w0
    const float Phi = phi - P.phi_ref;
    const float tnq = P.tau_phi - 0.5f;
    const long long c = ((long long)z * P.ny + y) * P.nx + x;
    float fsum = 0.f, fs[Q], gs[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const float t = Lat<Q>::w(i);
        const float eu = Lat<Q>::cx(i) * u[0] + Lat<Q>::cy(i) * u[1] + Lat<Q>::cz(i) * u[2];
        const float en = Lat<Q>::cx(i) * n[0] + Lat<Q>::cy(i) * n[1] + Lat<Q>::cz(i) * n[2];
        const float es = Lat<Q>::cx(i) * Sv[0] + Lat<Q>::cy(i) * Sv[1] + Lat<Q>::cz(i) * Sv[2];
        const float eg = Lat<Q>::cx(i) * gx + Lat<Q>::cy(i) * gy + Lat<Q>::cz(i) * gz;
        const float gam = 3.f * eu + 4.5f * eu * eu - 1.5f * u2;
        const float pis = sg * ((float)Lat<Q>::e2(i) - en * en - trc3);
        const float fdev = t * (dP + rho * gam - 4.5f * pis);                        // f*_i - t_i w0
        const float gdev = t * (Phi + phi * gam + P.tau_phi * es) - t * tnq * eg;  // g*_i - t_i phi_ref
        fsum += fdev;
        fs[i] = fdev * Store<S>::kScaleF;
        gs[i] = gdev * Store<S>::kScaleG;
    }
#pragma unroll
    for (int k = 0; k < Lat<Q>::kPairs; ++k) {
        const int i = Lat<Q>::pair_first(k), j = Lat<Q>::pair_second(k);
        __stcs(pair_plane<S>(fg, P.N, k) + c, Store<S>::word(fs[i], gs[i], fs[j], gs[j]));
    }
    // plane 0: sum_i f*_i - w0, and phi (= sum_i g*_i) as the integer phi * 2^30
    const int phi_fx = __float2int_rn(phi * 1073741824.0f);
    moment_plane(fg)[c] = make_float2(fsum, __int_as_float(phi_fx));
    return phi_fx;
}

template <int Q, int S>
__global__ void __launch_bounds__(128)
restart_kernel(const Params P, const float* coarse, const float* phi_fine, int f, float p0,
               void* __restrict__ fg, unsigned long long* __restrict__ slots, int n_slots) {
    __shared__ long long s_sum[4];
    chain_begin();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    int v = 0;
    if (x < P.nx && y < P.ny) v = restart_cell<Q, S>(P, coarse, phi_fine, f, p0, fg, x, y, blockIdx.z);
    // a warp's sum by halves that cannot overflow
    const long long sum = ((long long)__reduce_add_sync(0xffffffffu, v >> 16) << 16) +
                          (long long)__reduce_add_sync(0xffffffffu, (unsigned)v & 0xffffu);
    if (threadIdx.x == 0) s_sum[threadIdx.y] = sum;
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        const unsigned block = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        atomicAdd(slots + block % (unsigned)n_slots, (unsigned long long)(s_sum[0] + s_sum[1] + s_sum[2] + s_sum[3]));
    }
}

cudaError_t launch_restart(const Params& P, const float* coarse, int factor, double p0, float* phi_fine, void* fg,
                           const RestartSums& sums, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(sums.slots, 0, sums.n_slots * sizeof(*sums.slots), s);
    if (e != cudaSuccess) return e;
    const dim3 block(32, 4), grid((P.nx + 31) / 32, (P.ny + 3) / 4, P.nz);
    if ((e = launch_chained(phi_fine_kernel, grid, block, 0, s, P, coarse, factor, phi_fine)) != cudaSuccess) return e;
#define LBM_RESTART(Q, S) \
    e = launch_chained(restart_kernel<Q, S>, grid, block, 0, s, P, coarse, (const float*)phi_fine, factor, (float)p0, fg, sums.slots, sums.n_slots)
    if (P.Q == 9) {
        if (P.storage == STORE_F16) LBM_RESTART(9, STORE_F16);
        else if (P.storage == STORE_BF16) LBM_RESTART(9, STORE_BF16);
        else LBM_RESTART(9, STORE_F32);
    } else {
        if (P.storage == STORE_F16) LBM_RESTART(19, STORE_F16);
        else if (P.storage == STORE_BF16) LBM_RESTART(19, STORE_BF16);
        else LBM_RESTART(19, STORE_F32);
    }
#undef LBM_RESTART
    return e;
}

__device__ __forceinline__ double warp_sum_jm(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_max_jm(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

constexpr int kJumpThreads = 256;

__global__ void __launch_bounds__(kJumpThreads)
jump_measures_kernel(const float* start, const float* pred, int ncx, int ncy, int ncz,
                     int walls, double* __restrict__ out) {
    chain_begin();
    chain_next();
    const long long nc = (long long)ncx * ncy * ncz;
    double acc[3] = {0.0, 0.0, 0.0}, umax = 0.0;
    for (long long l = (long long)blockIdx.x * kJumpThreads + threadIdx.x; l < nc; l += (long long)gridDim.x * kJumpThreads) {
        const int row = (int)l / ncx, x = (int)l - row * ncx, z = row / ncy, y = row - z * ncy;  // nc < 2^31
        auto idx = [&](int xx, int yy, int zz) { return ((long long)zz * ncy + yy) * ncx + xx; };
        auto nb = [](int i, int d, int n, bool wall) { return wall ? min(max(i + d, 0), n - 1) : (i + d + n) % n; };
        const float ps = start[l], pp = pred[l];
        acc[0] += (double)pp;
        acc[1] += fabs((double)pp - (double)ps);
        const double gx = 0.5 * ((double)start[idx(nb(x, 1, ncx, walls & 1), y, z)] -
                                 (double)start[idx(nb(x, -1, ncx, walls & 1), y, z)]);
        const double gy = 0.5 * ((double)start[idx(x, nb(y, 1, ncy, walls & 2), z)] -
                                 (double)start[idx(x, nb(y, -1, ncy, walls & 2), z)]);
        const double gz = 0.5 * ((double)start[idx(x, y, nb(z, 1, ncz, walls & 4))] -
                                 (double)start[idx(x, y, nb(z, -1, ncz, walls & 4))]);
        acc[2] += sqrt(gx * gx + gy * gy + gz * gz);
        double u2s = 0.0, u2p = 0.0;
#pragma unroll
        for (int a = 1; a <= 3; ++a) {
            const double us = start[a * nc + l], up = pred[a * nc + l];
            u2s += us * us;
            u2p += up * up;
        }
        umax = fmax(umax, fmax(u2s, u2p));
    }
    __shared__ double red[4][kJumpThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3; ++k) acc[k] = warp_sum_jm(acc[k]);
    umax = warp_max_jm(umax);
    if (lane == 0) {
        for (int k = 0; k < 3; ++k) red[k][warp] = acc[k];
        red[3][warp] = umax;
    }
    __syncthreads();
    if (warp == 0) {
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = (lane < kJumpThreads / 32) ? red[k][lane] : 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) v[k] = warp_sum_jm(v[k]);
        v[3] = warp_max_jm(v[3]);
        if (lane == 0) {
            for (int k = 0; k < 3; ++k) atomicAdd(out + k, v[k]);
            // non-negative doubles order like their bit patterns
            atomicMax(reinterpret_cast<unsigned long long*>(out + 3), (unsigned long long)__double_as_longlong(v[3]));
        }
    }
}

cudaError_t launch_jump_measures(const float* start, const float* pred, int ncx, int ncy, int ncz, int walls, double* out,
                                 cudaStream_t s) {
    const long long nc = (long long)ncx * ncy * ncz;
    const long long blocks = (nc + kJumpThreads - 1) / kJumpThreads;
    return launch_chained(jump_measures_kernel, dim3((unsigned)(blocks < 1216 ? blocks : 1216)), dim3(kJumpThreads), 0, s, start, pred,
                          ncx, ncy, ncz, walls, out);
}

__global__ void normalize_kernel(const float* x, float* __restrict__ y, long long n, float m0, float m1,
                                 float m2, float m3, float m4, float s0, float s1, float s2, float s3, float s4, int dir) {
    chain_begin();
    chain_next();
    const float mean[5] = {m0, m1, m2, m3, m4}, sd[5] = {s0, s1, s2, s3, s4};
    const int c = blockIdx.y;
    const float m = mean[c], d = sd[c];
    x += c * n;
    y += c * n;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = dir > 0 ? (x[i] - m) / d : x[i] * d + m;
}

cudaError_t launch_normalize(const float* x, float* y, long long n, const float* ms, int dir, cudaStream_t s) {
    return launch_chained(normalize_kernel, dim3(cell_blocks(n), 5), dim3(256), 0, s, x, y, n, ms[0], ms[1], ms[2], ms[3], ms[4],
                          ms[5], ms[6], ms[7], ms[8], ms[9], dir);
}

// sum |a - b| over n values in FP64: per block, then the blocks by one block, each in a fixed order.
__global__ void __launch_bounds__(kJumpThreads) l1_kernel(const float* a, const float* b, long long n,
                                                         double* __restrict__ out) {
    __shared__ double red[kJumpThreads / 32];
    chain_begin();
    chain_next();
    double acc = 0.0;
    for (long long i = (long long)blockIdx.x * kJumpThreads + threadIdx.x; i < n; i += (long long)gridDim.x * kJumpThreads)
        acc += fabs((double)a[i] - (double)b[i]);
    acc = warp_sum_jm(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        acc = 0.0;
        for (int w = 0; w < kJumpThreads / 32; ++w) acc += red[w];
        out[blockIdx.x] = acc;
    }
}
__global__ void __launch_bounds__(kJumpThreads) l1_finish(const double* part, int n, double* __restrict__ out) {
    __shared__ double red[kJumpThreads / 32];
    chain_begin();
    chain_next();
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += kJumpThreads) acc += part[i];
    acc = warp_sum_jm(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        acc = 0.0;
        for (int w = 0; w < kJumpThreads / 32; ++w) acc += red[w];
        *out = acc;
    }
}

cudaError_t launch_l1_difference(const float* a, const float* b, long long n, double* partials, int n_partials, double* out,
                                 cudaStream_t s) {
    const int blocks = (int)std::min<long long>((n + kJumpThreads - 1) / kJumpThreads, std::min(n_partials, 512));
    const cudaError_t e = launch_chained(l1_kernel, dim3(blocks), dim3(kJumpThreads), 0, s, a, b, n, partials);
    if (e != cudaSuccess) return e;
    return launch_chained(l1_finish, dim3(1), dim3(kJumpThreads), 0, s, (const double*)partials, blocks, out);
}

}  // namespace lbm
