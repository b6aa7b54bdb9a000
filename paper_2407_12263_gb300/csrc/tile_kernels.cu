// tile_kernels.cu -- several time steps of a small D2Q9 grid per launch.
//
// A step of a small grid is over before the next launch can start: a 64 x 64 step takes 1.5 us, of
// which the cells' work is less than half. Here a block loads the state of a region of 16 x 16 cells into
// shared memory and advances it `steps` times by itself, the cells it may still use shrinking by the reach of
// a step (one cell, two in the finite-difference variant: phi, then its gradient) on every side,
// and stores the tile that is left. Cells of the halo are computed by several blocks, each in the
// same way: every value is what launches of single steps give, bit for bit.
//
// What bounds it is the chain of a step's instructions in a block (0.66 us) and 1.5 us to bring a region up
// and down; step_plan.h has the measured rule by which a grid takes this path. 64 x 64 FP32: 1.55 -> 1.01 us per
// step, the finite-difference variant 2.72 -> 1.41, where one launch takes the place of a step's two.
//
// One thread per cell of the region. A step reads the stencil from shared memory, and writes the new
// state back between two barriers, so one copy of the state serves. The arithmetic is that of
// step_cell (cell.cuh); tile_pull is its propagation with the words taken from shared memory.
#include "cell.cuh"
#include "step_plan.h"

namespace lbm {

namespace {

constexpr int Q9 = 9, R = kTileSide;

// pull (cell.cuh) in storage units, from the words and moments of a region of `n` cells in shared memory,
// whose rows lie as nb says.
template <int S, bool WALLS>
__device__ __forceinline__ void tile_pull(const Params& P, const typename Store<S>::Word* words, const float2* moments, int n, int c,
                                          const Nbr& nb, float (&fb)[Q9], float (&gb)[Q9], int& phi_fx, const WallSide& ws) {
    using St = Store<S>;
    float df = 0.f;
    unsigned int dphi = 0u;
    const float fa = P.flux_as, fbk = P.flux_bs;
    const float2 lwm = make_float2(P.lw_m, P.lw_m), lwp = make_float2(P.lw_p, P.lw_p);
    const float2 nfa = make_float2(-fa, -fa), fbk2 = make_float2(fbk, fbk);
#pragma unroll
    for (int k = 0; k < Lat<Q9>::kPairs; ++k) {
        const int i = Lat<Q9>::pair_first(k), j = Lat<Q9>::pair_second(k);
        const typename St::Word* pw = words + k * n + c;
        const typename St::Word vm = pw[link_offset<Q9>(nb, i, -1)], v0 = pw[0], vp = pw[link_offset<Q9>(nb, i, +1)];
        typename St::Raw rmi = St::lo(vm), rpj = St::hi(vm), r0i = St::lo(v0), r0j = St::hi(v0), rpi = St::lo(vp), rmj = St::hi(vp);
        if (WALLS) {  // half-way bounce-back: beyond a wall, the opposite pair of this cell
            if (crosses_wall<Q9>(ws, i, -1)) rmi = r0j;
            if (crosses_wall<Q9>(ws, i, +1)) rpi = r0j;
            if (crosses_wall<Q9>(ws, j, -1)) rmj = r0i;
            if (crosses_wall<Q9>(ws, j, +1)) rpj = r0i;
        }
        const float2 v0i = St::cvt(r0i), v0j = St::cvt(r0j);
        const float2 ei = __ffma2_rn(lwm, St::sub2(rmi, v0i), __fmul2_rn(lwp, St::sub2(rpi, v0i)));
        const float2 ej = __ffma2_rn(lwm, St::sub2(rmj, v0j), __fmul2_rn(lwp, St::sub2(rpj, v0j)));
        const float2 bi = __fadd2_rn(v0i, ei), bj = __fadd2_rn(v0j, ej);
        gb[i] = bi.y;
        gb[j] = bj.y;
        const float2 out = __ffma2_rn(nfa, make_float2(St::sub_g(rmj, v0i.y), St::sub_g(rmi, v0j.y)),
                                      __fmul2_rn(fbk2, make_float2(St::sub_g(rpi, v0j.y), St::sub_g(rpj, v0i.y))));
        dphi -= (unsigned int)__float2int_rn(out.x) + (unsigned int)__float2int_rn(out.y);
        fb[i] = bi.x;
        fb[j] = bj.x;
        df += ei.x + ej.x;
    }
    const float2 m0 = moments[c];
    phi_fx = (int)((unsigned int)__float_as_int(m0.y) + dphi);
    gb[0] = __int2float_rn((int)((unsigned int)phi_fx - (unsigned int)P.phi_ref_fx)) * kPhiFxInvF;
    fb[0] = m0.x + df * St::kInvF;
}

// fd_gradient (cell.cuh) from a plane in shared memory.
__device__ __forceinline__ void tile_gradient(const float* phi, int c, const Nbr& nb, float& gx, float& gy, float& gz) {
    gx = gy = gz = 0.f;
#pragma unroll
    for (int i = 1; i < Q9; ++i) fd_term<Q9>(i, phi[c + link_offset<Q9>(nb, i, +1)], gx, gy, gz);
    gx *= 3.f;
    gy *= 3.f;
    gz *= 3.f;
}

template <int S, int SCHEME>
constexpr size_t tile_smem() {
    return (size_t)R * R * (sizeof(float2) + Lat<Q9>::kPairs * sizeof(typename Store<S>::Word) + (SCHEME == SCHEME_FD ? sizeof(float) : 0));
}

// 65 to 80 registers, three blocks an SM (kTileResident) without asking for them: with the bound the compiler
// takes 80 for the 64 x 64 FP32 step, which then takes 1.06 us instead of 0.98.
template <int SCHEME, bool GEN, int S>
__global__ void __launch_bounds__(R* R)
tile_step_kernel(const Params P, const void* fg_in, void* __restrict__ fg_out, int steps) {
    using Word = typename Store<S>::Word;
    constexpr int n = R * R, kReach = SCHEME == SCHEME_FD ? 2 : 1;
    extern __shared__ __align__(16) unsigned char smem[];
    Word* words = reinterpret_cast<Word*>(smem);
    float2* moments = reinterpret_cast<float2*>(smem + (size_t)Lat<Q9>::kPairs * n * sizeof(Word));
    float* phi = reinterpret_cast<float*>(moments + n);
    const int halo = kReach * steps, tile = R - 2 * halo;
    const int c = threadIdx.x, lx = c % R, ly = c / R;
    const int edge = min(min(lx, R - 1 - lx), min(ly, R - 1 - ly));  // steps reach this cell while it is at least that far in
    // this cell of the grid: its periodic image, or beyond a wall none
    const int gx = (int)blockIdx.x * tile + lx - halo, gy = (int)blockIdx.y * tile + ly - halo;
    const bool beyond = ((P.walls & 1) && (gx < 0 || gx >= P.nx)) || ((P.walls & 2) && (gy < 0 || gy >= P.ny));
    const int x = ((gx % P.nx) + P.nx) % P.nx, y = ((gy % P.ny) + P.ny) % P.ny;
    const long long cell = (long long)y * P.nx + x;
    chain_begin();
    if (!beyond) {
#pragma unroll
        for (int k = 0; k < Lat<Q9>::kPairs; ++k) words[k * n + c] = pair_plane<S>(fg_in, P.N, k)[cell];
        moments[c] = moment_plane(fg_in)[cell];
    }
    const WallSide ws = GEN ? make_wall_side(P, x, y, 0) : WallSide{};
    const bool at_wall = GEN && (ws.xlo || ws.xhi || ws.ylo || ws.yhi);
    const Nbr nb{-1, 1, -R, R, 0, 0};
    __syncthreads();
    for (int t = 1; t <= steps; ++t) {
        float fb[Q9], gb[Q9];
        int phi_fx;
        // the finite-difference variant needs phi one cell farther out than the new state
        const bool pulls = !beyond && edge >= kReach * (t - 1) + 1, active = !beyond && edge >= kReach * t;
        const bool walled = GEN && __any_sync(0xffffffffu, at_wall);
        if (pulls) {
            if (walled) tile_pull<S, true>(P, words, moments, n, c, nb, fb, gb, phi_fx, ws);
            else tile_pull<S, false>(P, words, moments, n, c, nb, fb, gb, phi_fx, ws);
        }
        if (SCHEME == SCHEME_FD) {
            if (pulls) phi[c] = gb[0];
            __syncthreads();
        }
        if (active) {
            Macro m;
            macro_flow<Q9, GEN, S>(P, fb, gb, m);
            if (SCHEME == SCHEME_DF) {
                macro_interface_df<Q9, S>(P, m);
            } else {
                float dx, dy, dz;
                tile_gradient(phi, c, GEN ? mirror_at_walls(nb, ws) : nb, dx, dy, dz);
                macro_interface_fd(P, dx, dy, dz, m);
            }
            macro_pressure<GEN, SCHEME>(P, m);
            collide<Q9, GEN, S>(P, m, fb, gb);
        }
        if (t < steps) {
            __syncthreads();
            if (active) {
                moments[c] = make_float2(fb[0], __int_as_float(phi_fx));
#pragma unroll
                for (int k = 0; k < Lat<Q9>::kPairs; ++k) {
                    const int i = Lat<Q9>::pair_first(k), j = Lat<Q9>::pair_second(k);
                    words[k * n + c] = Store<S>::word(fb[i], gb[i], fb[j], gb[j]);
                }
            }
            __syncthreads();
        } else if (chain_next(); active && gx < P.nx && gy < P.ny) {  // the tile: edge >= halo
            moment_plane(fg_out)[cell] = make_float2(fb[0], __int_as_float(phi_fx));
#pragma unroll
            for (int k = 0; k < Lat<Q9>::kPairs; ++k) {
                const int i = Lat<Q9>::pair_first(k), j = Lat<Q9>::pair_second(k);
                pair_plane<S>(fg_out, P.N, k)[cell] = Store<S>::word(fb[i], gb[i], fb[j], gb[j]);
            }
        }
    }
}

template <int SCHEME, bool GEN, int S>
cudaError_t launch_tile(const Params& P, const void* in, void* out, int steps, cudaStream_t s) {
    constexpr size_t smem = tile_smem<S, SCHEME>();
    const int tile = R - 2 * steps * (SCHEME == SCHEME_FD ? 2 : 1);
    if (steps < 1 || tile < 1) return cudaErrorInvalidValue;
    static_assert(smem <= 48 << 10, "larger needs cudaFuncSetAttribute");
    const dim3 grid((P.nx + tile - 1) / tile, (P.ny + tile - 1) / tile);
    return launch_chained(tile_step_kernel<SCHEME, GEN, S>, grid, dim3(R * R), smem, s, P, in, out, steps);
}

template <int SCHEME>
cudaError_t launch_tile_s(const Params& P, const void* in, void* out, int steps, cudaStream_t s) {
#define LBM_TILE(S) (P.general ? launch_tile<SCHEME, true, S>(P, in, out, steps, s) : launch_tile<SCHEME, false, S>(P, in, out, steps, s))
    if (P.storage == STORE_F16) return LBM_TILE(STORE_F16);
    if (P.storage == STORE_BF16) return LBM_TILE(STORE_BF16);
    return LBM_TILE(STORE_F32);
#undef LBM_TILE
}

}  // namespace

cudaError_t launch_tile_steps(const Params& P, int scheme, const void* in, void* out, int steps, cudaStream_t s) {
    if (P.Q != 9) return cudaErrorInvalidValue;
    return scheme == SCHEME_DF ? launch_tile_s<SCHEME_DF>(P, in, out, steps, s) : launch_tile_s<SCHEME_FD>(P, in, out, steps, s);
}

}  // namespace lbm
