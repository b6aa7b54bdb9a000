// surrogate.h -- launchers of the convolutional surrogate's kernels (surrogate_kernels.cu) and
// of the field transfers between the lattice and the coarse grid (surrogate_glue.cu).
// Internal to the library.
#pragma once

#include <cuda_runtime.h>

#include "lbm_internal.h"

namespace lbm {
namespace net {

constexpr int kFieldChannels = 5;  // phi, u, v, w, p
constexpr int kHidden = 32;        // channels of the hidden layers
constexpr int kLayers = 4;

// Periodic 3x3x3 convolution of a batch [B][cin][D][H][W] into [B][cout][D][H][W], FP32 on the
// CUDA cores (cout = 32, or 5 without relu); relu on the output if asked. bias may be NULL.
cudaError_t conv_forward(const float* in, int cin, const float* W, const float* bias, float* out, int cout, int relu, int batch,
                         int D, int H, int Wd, cudaStream_t s);
// gW [cout][cin][27] += correlation of g [B][cout] with h [B][cin]; gb [cout] += sum of g.
cudaError_t conv_wgrad(const float* g, int cout, const float* h, int cin, float* gW, float* gb, int batch, int D, int H, int Wd,
                       cudaStream_t s);
// Wt [cin][cout][27] with the taps reversed: the adjoint convolution's weights.
cudaError_t flip_transpose(const float* W, int cout, int cin, float* Wt, cudaStream_t s);
cudaError_t relu_mask(float* g, const float* h, long long n, cudaStream_t s);
cudaError_t residual(const float* x, const float* d, float* y, long long n, cudaStream_t s);
int loss_blocks(long long n);
// loss sum_i w_c(i) (x + d - target)_i^2 / n and its gradient; w: 5 host weights, vox: cells per channel.
cudaError_t loss_and_grad(const float* x, const float* d, const float* target, float* g, long long n, long long vox,
                          const float* w, double* partials, cudaStream_t s);
cudaError_t adam(float* p, const float* g, float* m, float* v, long long n, float lr, int step, cudaStream_t s);

// The layers on the tensor cores (tcgen05, surrogate_tc.cu): FP16 operands, FP32 accumulation. A
// network's weights and the workspace of a batch, all device memory unless said otherwise.
// Activations and gradients between layers are FP16, channels last; the five field channels are
// padded to eight. *err is set to 1 if a wait gave up: each wait polls its mbarrier at most
// `spin` times, kTcWaitPolls normally or 0 (give up at once, the same in every thread: a test of
// the timeout path); the last wait for MMAs still in flight, before the tensor memory is freed,
// always allows kTcWaitPolls.
constexpr long long kTcWaitPolls = 1ll << 26;
struct TcNet {
    const float* params;
    int cin[kLayers], cout[kLayers];
    long long w_off[kLayers], b_off[kLayers];
    int batch, D, H, W;
    int ctas;                       // SMs of the device (tc_sizes)
    void* x;                        // [B][vox][8]
    void* h[kLayers - 1];           // [B][vox][32], outputs of the hidden layers
    uint32_t* bits[kLayers - 1];    // [B][vox], bit c: channel c of h is positive (gradients only)
    void* gout;                     // [B][vox][8], gradient of the prediction
    void* g[kLayers - 1];           // [B][vox][32], gradients of the hidden layers; g[0] and g[2] may be one buffer
    void* images;                   // tc_sizes().image_bytes: the weights as operands
    float* part;                    // part_floats: the CTAs' weight-gradient sums
    float* bias_part;               // bias_floats
    double* loss_part;              // loss_parts doubles
    float grad_scale;               // power of two that gradients are multiplied by before they are rounded to FP16
    float loss_w[kFieldChannels];
    long long spin;
    int* err;
};
struct TcSizes {
    int ctas, loss_parts;
    size_t image_bytes, part_floats, bias_floats;
};
TcSizes tc_sizes();  // of the current device
// target NULL: y = x + net(x). Otherwise the loss sum w_c (x + net(x) - target)^2 as *loss_parts
// (host) partial sums in loss_part, and its mean's gradients with respect to all parameters in
// grads. Partial sums are added in a fixed order: the same bits on every run.
cudaError_t tc_run(const TcNet& N, const float* x, float* y, const float* target, float* grads, int* loss_parts, cudaStream_t s);

}  // namespace net

// Coarse fields [5][nz/f][ny/f][nx/f] (phi, u, v, w, p; means over f^3 cells of the macroscopic
// fields of the difference-free scheme) of the propagated state fg.
cudaError_t launch_coarsen(const Params& P, const void* fg, int factor, float* out, cudaStream_t s);
// Device sums around a restart: *before is the fixed-point sum of phi that the state must keep,
// slots[0 .. n_slots) receive the restarted state's (their total).
struct RestartSums {
    const long long* before;
    unsigned long long* slots;
    int n_slots;
};
// Block means of the state's own phi (plane 0, before propagation) into out [nz/f][ny/f][nx/f];
// factor must divide 32 (cudaErrorInvalidValue otherwise). With sums the state is balanced first
// (launch_balance), in the same pass.
cudaError_t launch_coarse_phi(const Params& P, void* fg, int factor, const RestartSums* sums, float* out, cudaStream_t s);
// The state launch_init builds (equilibrium plus the first-order non-equilibrium part of g) from
// coarse fields upsampled trilinearly between coarse cell centres (periodic, clamped across
// walls), in FP32 arithmetic: the upsampled phi of every cell into phi_fine (N floats), then the
// populations and sums.slots.
cudaError_t launch_restart(const Params& P, const float* coarse, int factor, double p0, float* phi_fine, void* fg,
                           const RestartSums& sums, cudaStream_t s);
// Adds *before minus the slots' total, in units (2^-30) of phi, spread over the cells of the state so
// that its sum is *before exactly.
cudaError_t launch_balance(const Params& P, void* fg, const RestartSums& sums, cudaStream_t s);
// *out = sum |a - b| over n values, FP64 in a fixed order; partials: n_partials doubles of scratch.
cudaError_t launch_l1_difference(const float* a, const float* b, long long n, double* partials, int n_partials, double* out,
                                 cudaStream_t s);
// What the judge of a jump measures on the coarse grid [5][ncz][ncy][ncx] of the starting fields
// `start` and of the prediction `pred`, accumulated into out[4] (zeroed by the caller):
//   out[0] += sum of the predicted phi;
//   out[1] += sum |phi_pred - phi_start|;
//   out[2] += sum |grad phi_start|, central differences in coarse cells (periodic, or the cell
//             itself beyond a wall, bit 0 x, bit 1 y, bit 2 z of walls);
//   out[3]  = max(out[3], largest |u|^2 of start and prediction) (as non-negative double bits).
cudaError_t launch_jump_measures(const float* start, const float* pred, int ncx, int ncy, int ncz, int walls, double* out,
                                 cudaStream_t s);
constexpr int kProjectLaunches = 8;  // twiddles, three passes, the modes, three passes back
// The divergence-free part of the periodic velocity u [3][nz][ny][nx] in place
// (lbm_project_solenoidal); work holds project_workspace_bytes() bytes, 16-byte aligned.
cudaError_t launch_project_solenoidal(float* u, int nx, int ny, int nz, void* work, cudaStream_t s);
size_t project_workspace_bytes(int nx, int ny, int nz);
bool project_extents_ok(const int grid[3]);  // every extent in 1 .. 512
// (x - mean[c]) / std[c] per channel of [5][n] (dir = +1) or x std[c] + mean[c] (dir = -1).
cudaError_t launch_normalize(const float* x, float* y, long long n, const float* mean_std, int dir, cudaStream_t s);

}  // namespace lbm
