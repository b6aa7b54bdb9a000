// step_kernels.cu -- the fused time step of the difference-free conservative phase-field LBM
// (Zhao, Patel & Lee, arXiv:2407.12263) and its finite-difference twin.
//
// Difference-free step: ONE kernel per time step. Each thread owns one cell; it pulls the
// Lax-Wendroff-propagated f and g (Sec. 2.2: for each opposite pair of populations, three loads
// of the word that holds both (f, g) pairs, at x - e_i, x and x + e_i), computes phi, rho, u,
// the central moment K1, n, S, grad phi and p in registers (Sec. 2.3), collides both sets
// (Eqs. c-n_m and c-n_c) and streams the Q post-collision pairs out, one word per opposite
// pair. The neighbour loads of adjacent threads overlap, so DRAM sees each stored value about
// once per step; everything else is L1/L2 reuse. Interleaving f with g, and a population with
// its opposite, divides the memory instructions per cell by four, and that count (not bytes) is
// what limits a 3-point stencil over 38 planes: with separate planes the same step ran at 74%
// of the HBM copy bandwidth, with (f, g) pairs at 0.98, with opposite pairs interleaved too at
// the copy bandwidth.
//
// Finite-difference variant (the "previous method" of Sec. 3.4): a first kernel propagates g
// and writes the phi plane; the second is the fused step with grad phi taken from the
// isotropic central difference of that plane instead of K1.
#include "cell.cuh"
#include "step_plan.h"

namespace lbm {

// Thread block: 128 threads, one cell per thread, x fastest (step_shape in step_plan.h has the shapes). With FP32 storage the register budget allows 4
// blocks (16 warps) per SM: the difference-free step needs ~122 registers and runs at that
// occupancy with every (f, g) load of a cell in flight. A 16-bit cell moves half the bytes, so
// the same bandwidth needs more cells in flight: the 16-bit steps are held to 96 registers for
// 5 blocks (20 warps), which they fit without spilling.
constexpr int LBM_STEP_MINB = 4;

template <int S>
constexpr int step_min_blocks() {
    return S == STORE_F32 ? LBM_STEP_MINB : 5;
}

// The cell of a thread, false beyond the grid. PACK: blocks of 128 cells that follow one another in
// a plane, whatever its rows, instead of blocks of whole rows or of 32 x 4 cells.
template <bool PACK>
__device__ __forceinline__ bool own_cell(const Params& P, const RowDiv& d, int& x, int& y, int& z) {
    z = blockIdx.z;
    if (PACK) {
        const unsigned i = blockIdx.x * kStepThreads + threadIdx.x;
        y = (int)(__umulhi(i, d.mul) >> d.shift);
        x = (int)i - y * P.nx;
        return y < P.ny;
    }
    x = blockIdx.x * blockDim.x + threadIdx.x;
    y = blockIdx.y * blockDim.y + threadIdx.y;
    return x < P.nx && y < P.ny;
}

template <int Q, int S>
constexpr bool narrow_form(int form) { return Q == 19 && S != STORE_F32 && form != WIDE; }

template <int Q, int SCHEME, bool GEN, int S, int FORM>
__global__ void __launch_bounds__(kStepThreads, (step_min_blocks<S>()))
step_kernel(const Params P, const void* fg_in, void* __restrict__ fg_out, const float* phi_fd, const RowDiv d) {
    chain_begin();
    int x, y, z;
    if (!own_cell<FORM == PACKED>(P, d, x, y, z)) return;
    step_cell<Q, SCHEME, GEN, S, narrow_form<Q, S>(FORM)>(P, fg_in, fg_out, phi_fd, x, y, z);
}

// Finite-difference variant, pass 1: the propagated phi (held as phi - phi_ref), one FP32 plane.
template <int Q, int S, bool WALLS, int FORM>
__global__ void __launch_bounds__(kStepThreads, LBM_STEP_MINB)
fd_phi_kernel(const Params P, const void* fg_in, float* __restrict__ phi, const RowDiv d) {
    chain_begin();
    int x, y, z;
    if (!own_cell<FORM == PACKED>(P, d, x, y, z)) return;
    const Nbr nb = make_nbr(P, x, y, z);
    const int c = (z * P.ny + y) * P.nx + x;
    float fb[Q], gb[Q];
    int phi_fx;
    pull<Q, false, S, WALLS, false, narrow_form<Q, S>(FORM)>(P, fg_in, c, nb, fb, gb, phi_fx, WALLS ? make_wall_side(P, x, y, z) : WallSide{});
    chain_next();
    phi[c] = gb[0];
}

static StepShape step_shape(const Params& P) {
    return step_shape(P.nx, P.ny, P.nz, P.Q == 19 && P.storage != STORE_F32);
}
static dim3 grid_of(const StepShape& h) { return dim3(h.grid[0], h.grid[1], h.grid[2]); }
static dim3 block_of(const StepShape& h) { return dim3(h.block[0], h.block[1]); }

template <int Q, int S, int FORM>
static cudaError_t fd_phi_qs(const Params& P, const StepShape& h, const void* in, float* phi, cudaStream_t s) {
    return launch_chained(P.walls ? fd_phi_kernel<Q, S, true, FORM> : fd_phi_kernel<Q, S, false, FORM>, grid_of(h), block_of(h), 0, s, P, in,
                          phi, h.d);
}

template <int Q, int S, int FORM>
static cudaError_t step_qs(const Params& P, const StepShape& h, int scheme, const void* in, void* out, float* phi, cudaStream_t s,
                           int* launches) {
    if (scheme == SCHEME_DF) {
        *launches += 1;
        return launch_chained(P.general ? step_kernel<Q, SCHEME_DF, true, S, FORM> : step_kernel<Q, SCHEME_DF, false, S, FORM>,
                              grid_of(h), block_of(h), 0, s, P, in, out, (const float*)nullptr, h.d);
    }
    *launches += 2;
    const cudaError_t e = fd_phi_qs<Q, S, FORM>(P, h, in, phi, s);
    if (e != cudaSuccess) return e;
    return launch_chained(P.general ? step_kernel<Q, SCHEME_FD, true, S, FORM> : step_kernel<Q, SCHEME_FD, false, S, FORM>, grid_of(h),
                          block_of(h), 0, s, P, in, out, (const float*)phi, h.d);
}

template <int Q, int S>
static cudaError_t step_s(const Params& P, int scheme, const void* in, void* out, float* phi, cudaStream_t s, int* launches) {
    const StepShape h = step_shape(P);
    if constexpr (narrow_form<Q, S>(WHOLE))
        if (h.form == WIDE) return step_qs<Q, S, WIDE>(P, h, scheme, in, out, phi, s, launches);
    return h.form == PACKED ? step_qs<Q, S, PACKED>(P, h, scheme, in, out, phi, s, launches)
                            : step_qs<Q, S, WHOLE>(P, h, scheme, in, out, phi, s, launches);
}

template <int Q>
static cudaError_t step_q(const Params& P, int scheme, const void* in, void* out, float* phi, cudaStream_t s,
                          int* launches) {
    if (P.storage == STORE_F16) return step_s<Q, STORE_F16>(P, scheme, in, out, phi, s, launches);
    if (P.storage == STORE_BF16) return step_s<Q, STORE_BF16>(P, scheme, in, out, phi, s, launches);
    return step_s<Q, STORE_F32>(P, scheme, in, out, phi, s, launches);
}

cudaError_t launch_step(const Params& P, int scheme, const void* fg_in, void* fg_out, float* phi_fd, cudaStream_t s,
                        int* launches) {
    if (P.Q == 9) return step_q<9>(P, scheme, fg_in, fg_out, phi_fd, s, launches);
    return step_q<19>(P, scheme, fg_in, fg_out, phi_fd, s, launches);
}

template <int Q, int S>
static cudaError_t fd_phi_s(const Params& P, const void* in, float* phi, cudaStream_t s) {
    const StepShape h = step_shape(P);
    if constexpr (narrow_form<Q, S>(WHOLE))
        if (h.form == WIDE) return fd_phi_qs<Q, S, WIDE>(P, h, in, phi, s);
    return h.form == PACKED ? fd_phi_qs<Q, S, PACKED>(P, h, in, phi, s) : fd_phi_qs<Q, S, WHOLE>(P, h, in, phi, s);
}

template <int Q>
static cudaError_t fd_phi_q(const Params& P, const void* in, float* phi, cudaStream_t s) {
    if (P.storage == STORE_F16) return fd_phi_s<Q, STORE_F16>(P, in, phi, s);
    if (P.storage == STORE_BF16) return fd_phi_s<Q, STORE_BF16>(P, in, phi, s);
    return fd_phi_s<Q, STORE_F32>(P, in, phi, s);
}

cudaError_t launch_fd_phi(const Params& P, const void* fg_in, float* phi_fd, cudaStream_t s) {
    return P.Q == 9 ? fd_phi_q<9>(P, fg_in, phi_fd, s) : fd_phi_q<19>(P, fg_in, phi_fd, s);
}

}  // namespace lbm
