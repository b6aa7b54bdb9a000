// surrogate_tc.cu -- the surrogate's layers on the fifth-generation tensor cores (tcgen05): the
// forward convolutions, their adjoints with the ReLU mask and the bias gradients, the loss, and
// the weight gradients. FP16 operands, FP32 accumulation in tensor memory.
//
// Activations and the gradients between layers are FP16, channels last: [B][D][H][W][8 or 32],
// so that the eight channels of a voxel that an operand row holds are one 16-byte vector, copied
// to shared memory as they are (cp.async) and written by the epilogue as four of them. (With
// [C][vox] arrays a thread loaded 8 x-values of a channel and scattered them as 2-byte stores,
// and gradients were FP32 arrays that both of their readers rounded to FP16: the same bits reach
// the tensor cores, at half the bytes and without the conversion.) The five field channels are
// padded to eight.
//
// Shared-memory operands use the canonical no-swizzle layout, core matrices of 8 rows x 16
// bytes. Measured on GB300, an MMA of M = 128, N columns, K = 16 takes max(N / 2, 32 + N / 4, 39)
// cycles, wherever its operands start: the tensor pipe, or the 4 KB of A and 32 N bytes of B at
// 128 bytes per cycle. With the N = 32 of one tap of a layer it is A that bounds it (40 cycles
// for 16 of work); N = 96 takes 56 for 48.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstdint>

#include "chain.cuh"
#include "surrogate.h"

namespace lbm {
namespace net {

namespace {

constexpr int TX = 8, TY = 16;  // output voxels of a tile of one z plane: the M = 128 rows

// periodic index for any i: in range, one period off, or (a grid smaller than a tile) further
__device__ __forceinline__ int wrap(int i, int n) {
    if (i >= 0 && i < n) return i;
    if (i < 0 && i + n >= 0) return i + n;
    if (i >= n && i < 2 * n) return i - n;
    return ((i % n) + n) % n;
}

// ---------------------------------------------------------------------------------------
// PTX
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Operand descriptor: no swizzle, version 1. Strides between core matrices: lbo along K, sbo along M or N.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// kind::f16 instruction descriptor: FP32 D, FP16 A and B, M = 128, N columns (16 per step)
constexpr uint32_t kIdesc = (1u << 4) | ((128u >> 4) << 24);
constexpr uint32_t kMnMajor = (1u << 15) | (1u << 16);  // both operands with M (N) contiguous
__host__ __device__ constexpr uint32_t idesc_n(uint32_t n) { return (n >> 3) << 17; }

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// this thread's generic-proxy writes to shared memory become visible to the tensor cores
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// Polls `mbar` until phase `parity` completes, at most `limit` times (limit 0 gives up at once
// without polling), or until another thread of the CTA has given up.
__device__ __forceinline__ bool wait_parity(uint32_t mbar, uint32_t parity, long long limit, volatile int* fail) {
    for (long long it = 0; it < limit; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred P1;\n\tmbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\tselp.b32 %0, 1, 0, P1;\n\t}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (fail && *fail) return false;
    }
    return false;
}

// Whether that phase has completed, without waiting for it.
__device__ __forceinline__ bool test_parity(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P1;\n\tmbarrier.test_wait.parity.shared::cta.b64 P1, [%1], %2;\n\tselp.b32 %0, 1, 0, P1;\n\t}\n"
        : "=r"(ok)
        : "r"(mbar), "r"(parity)
        : "memory");
    return ok != 0;
}

// One thread of the (converged) warp. Only under elect.sync does the compiler know that the
// issuing code is uniform and keeps descriptors in uniform registers: 39 cycles per MMA of N <= 32
// against 48 for a branch on the thread index.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.b32 %0, 1, 0, P;\n\t}\n" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void copy16(uint32_t dst, const uint4* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void tmem_load32(uint32_t addr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_load8(uint32_t addr, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
template <int COLS>
__device__ __forceinline__ void tmem_alloc(uint32_t* slot) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "n"(COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
template <int COLS>
__device__ __forceinline__ void tmem_free(uint32_t tmem) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(COLS));
}

// ---------------------------------------------------------------------------------------
// The work of a kernel: the z planes of every (x, y) tile of every sample, in one row, cut into
// equal runs, one per CTA. A CTA walks its run in columns: planes of one tile, at most `most`. (Whole
// columns of 8 planes dealt out to the CTAs left the last round a third full: 4 x 64^3 is 3.4 of
// them per CTA.)
// ---------------------------------------------------------------------------------------
struct Tiling {
    int D, H, W, tiles_x, tiles_y, most;
    int planes;  // fewer than the grid's voxels, whose arrays fit the device
};
struct Column {
    int b, x0, y0, z0, nz;
};
struct Walk {
    int p, end;
    __device__ __forceinline__ explicit Walk(const Tiling& T)
        : p((int)((long long)T.planes * blockIdx.x / gridDim.x)), end((int)((long long)T.planes * (blockIdx.x + 1) / gridDim.x)) {}
    __device__ __forceinline__ bool next(const Tiling& T, Column& c) {
        if (p >= end) return false;
        int tile = p / T.D;
        c.z0 = p - tile * T.D;
        const int n = min(end - p, T.D - c.z0);
        const int parts = (n + T.most - 1) / T.most;
        c.nz = (n + parts - 1) / parts;
        c.x0 = (tile % T.tiles_x) * TX;
        tile /= T.tiles_x;
        c.y0 = (tile % T.tiles_y) * TY;
        c.b = tile / T.tiles_y;
        p += c.nz;
        return true;
    }
};

// ---------------------------------------------------------------------------------------
// Convolution: out[b][o][v] = sum_{c, tap} W[o][c][tap] in[b][c][v + off(tap)] (periodic).
//
// A haloed input plane of a tile (10 x 18 voxels) sits in shared memory in chunk planes: element
// (haloed voxel v, channel k) at (k / 8) * kChunk + 16 v + 2 (k % 8), K-major core matrices whose
// 8 rows are an x-run of voxels; the A operand of tap (dy, dx) is the same descriptor 160 dy + 16 dx
// bytes on. Input plane p contributes to the output planes p - 1, p and p + 1 (taps dz = 2, 1, 0), and
// those have neighbouring accumulators of NB tensor-memory columns: one MMA with the weights of
// the three dz as its N = 3 NB columns does the work of three, for one read of A. Output plane z is
// first touched by plane z - 1 (its block then starts without accumulating, in an MMA of its own)
// and done after plane z + 1; every output still sums its products in the order of the taps
// (dz, dy, dx, channels 16 at a time).
//
// A CTA walks columns of up to 8 output planes (8 blocks of accumulators: two CTAs share an SM's
// tensor memory). Three warps copy planes into a ring of four, one elected thread issues the
// MMAs, four warps drain finished blocks; they meet at mbarriers only. Every wait is bounded: on
// a timeout a thread raises *err and the CTA's fail flag, all roles leave, the issuer waits once
// more, with the full bound, for its MMAs, and the tensor memory is freed.
//
// Bound by shared memory and L1: the MMAs' operands are 1015 cycles per plane of 128 voxels, the rest is
// copies and stores. Batch 4 at 64^3, 32 -> 32 channels: 48 us (1200 TFLOP/s of the layer's own
// multiply-adds; 174 us with N = 32, planes staged through registers and block barriers between
// steps). Asking for the next plane while MMAs are queued, releasing accumulators one by one and
// storing whole rows took it from 53 us; copies through registers, more copying warps and
// announcing copies by their own completion made no difference or cost 3 to 15 us.
// ---------------------------------------------------------------------------------------
constexpr int kHx = TX + 2, kHy = TY + 2, kHaloed = kHx * kHy;
// Bytes between chunk planes: 180 voxels x 16 and on to 32 modulo 128, so that the four 16-byte
// pieces of a voxel, which one 128-byte line of global memory brings, fall into different banks
// (at 2880 a copy of a warp took 16 passes through shared memory instead of 4).
constexpr uint32_t kChunk = 2976;
static_assert(kChunk >= kHaloed * 16 && kChunk % 128 == 32, "chunk planes");
constexpr int kRing = 4;
constexpr int kMaxPlanes = 8;  // output planes of a column
constexpr int kConvThreads = 256, kEpiThreads = 128, kStagers = 96;

template <int KC, int NB>
struct ConvShape {
    static constexpr int kSteps = KC == 4 ? 2 : 1;            // MMAs of K = 16 per tap
    static constexpr uint32_t kSlot = (KC == 4 ? 4 : 2) * kChunk;  // KC = 1: the second chunk is zero
    static constexpr uint32_t kRows = 3 * NB;                 // weight rows of a tap: (dz = 2, 1, 0) x outputs
    static constexpr uint32_t kTap = kSteps * 2 * kRows * 16;
    static constexpr uint32_t kImage = 9 * kTap;
    static constexpr uint32_t kSmem = kRing * kSlot + kImage;
    static constexpr int kCols = kMaxPlanes * NB;
    static constexpr int kPieces = kHaloed * KC;              // 16-byte pieces of a plane
    static constexpr int kPer = (kPieces + kStagers - 1) / kStagers;
};

// What a finished output becomes.
enum ConvMode {
    kHiddenLayer,  // relu(a + bias) as FP16, and a bit per channel of whether it is positive
    kPrediction,   // x + a + bias, FP32 [B][5][vox]
    kLossGrad,     // the gradient of the loss at the prediction, FP16 [B][vox][8], and partial sums
    kAdjoint       // a masked by the layer's bits, FP16, and partial sums for the bias gradients
};

struct ConvArgs {
    const __half* in;
    const __half* image;
    const float* bias;
    __half* out;
    uint32_t* bits;          // hidden layer: written; adjoint: read
    const float* x;          // prediction, loss
    const float* target;
    float* y;
    double* loss_part;       // per CTA
    float* bias_part;        // [CTA][32 or 8]
    float grad_scale;        // of the stored gradients, a power of two
    float loss_scale;        // 2 / elements
    float w[kFieldChannels];
    Tiling t;
    long long spin;
    int* err;
};

// The running sum of w diff^2 of a thread, as an unevaluated pair of FP32 (exact products by FMA,
// two-sums: about 48 bits; an FP64 multiply-add per element would take as long as the layer's
// MMAs). An FP64 sum takes the values whose products, their rounding errors (2^-24 of them) or sums over 2^31
// elements may leave the FP32 range.
struct LossSum {
    float hi = 0.f, lo = 0.f;
    double far = 0.0;
    __device__ __forceinline__ void add(float w, float d) {
        const float m = fabsf(d);
        if (m == 0.f) return;
        if (!(m > 1e-9f && m < 1e9f && w < 1e9f && (w > 1e-9f || w == 0.f))) {
            far += (double)w * (double)d * (double)d;
            return;
        }
        const float a = __fmul_rn(d, d), ea = fmaf(d, d, -a);
        const float p = __fmul_rn(w, a), ep = fmaf(w, a, -p) + w * ea;
        const float s = __fadd_rn(hi, p), t = __fsub_rn(s, hi);
        lo += __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(p, t)) + ep;
        hi = s;
    }
    __device__ __forceinline__ double value() const { return far + ((double)hi + (double)lo); }
};

// The 64 bytes of every voxel of a warp (lane 8 y + x holds voxel (x0 + x, y0 + y)) to a plane of 32
// channels. Lane bits 3 and 4 (y) change places with the 16-byte chunks, so that each store writes 8
// whole voxels of one row, 512 consecutive bytes; a lane storing its own voxel 16 bytes at a time
// took four times the passes through L1, which the copies and operands of the MMAs need.
__device__ __forceinline__ void store_voxels(uint32_t (&v)[16], __half* plane, int x0, int y0, int H, int W) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int bit = 0; bit < 2; ++bit) {
        const bool up = (lane >> (3 + bit)) & 1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if ((k >> bit) & 1) continue;
            const int lo = 4 * k, hi = 4 * (k | 1 << bit);  // chunks k and k + 2^bit
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? v[lo + w] : v[hi + w], 8 << bit);
                if (up) v[lo + w] = got;
                else v[hi + w] = got;
            }
        }
    }
    const int x = x0 + (lane & 7);
    if (x >= W) return;
    uint4* dst = reinterpret_cast<uint4*>(plane) + ((long long)y0 * W + x) * 4 + (lane >> 3);
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (y0 + i < H) dst[(long long)i * W * 4] = make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
}

template <int KC, int NB, int MODE>
__global__ void __launch_bounds__(kConvThreads, 2) conv_tc_kernel(const __grid_constant__ ConvArgs A) {
    using Sh = ConvShape<KC, NB>;
    constexpr int kOut = NB == 32 ? 32 : kFieldChannels;  // channels of an output
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* s_ring = smem;
    unsigned char* s_w = smem + kRing * Sh::kSlot;
    // full[4], empty[4], done[8] (block finished), freed[8] (block read out), weights, drain
    __shared__ __align__(8) unsigned long long s_bar[kRing * 2 + kMaxPlanes * 2 + 2];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_fail;
    const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t / 32, 0);
    const uint32_t bar = smem_u32(s_bar);
    auto full = [&](int s) { return bar + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bar + 8u * (uint32_t)(kRing + s); };
    auto done = [&](int o) { return bar + 8u * (uint32_t)(2 * kRing + o); };
    auto freed = [&](int o) { return bar + 8u * (uint32_t)(2 * kRing + kMaxPlanes + o); };
    const uint32_t bar_w = bar + 8u * (2 * kRing + 2 * kMaxPlanes), bar_drain = bar_w + 8;
    if (t == 0) {
        for (int s = 0; s < kRing; ++s) {
            mbar_init(full(s), kStagers);
            mbar_init(empty(s), 1);
        }
        for (int o = 0; o < kMaxPlanes; ++o) {
            mbar_init(done(o), 1);
            mbar_init(freed(o), kEpiThreads);
        }
        mbar_init(bar_w, 1);
        mbar_init(bar_drain, 1);
        s_fail = 0;
    }
    if (KC == 1)  // the channels 8 .. 15 of the one K step
        for (int i = t; i < kRing * (int)(kChunk / 16); i += kConvThreads)
            *reinterpret_cast<uint4*>(s_ring + (i / (int)(kChunk / 16)) * Sh::kSlot + kChunk + (i % (int)(kChunk / 16)) * 16) =
                make_uint4(0, 0, 0, 0);
    // The kernels of a pass follow one another without gaps (chain.cuh): all CTAs of a launch are resident, so
    // the next one may come up from the start and set its barriers and shared memory up as CTAs here end.
    // Training at 30 x 26 x 45 in batches of 3 251 -> 217 us, a prediction at 64^3 76 -> 67 us.
    chain_begin();
    chain_next();
    if (t < 32) tmem_alloc<Sh::kCols>(&s_tmem);
    fence_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem;
    float sums[MODE == kAdjoint ? 32 : kFieldChannels];  // bias gradients of this thread's voxels
    LossSum loss;
    if (MODE == kAdjoint || MODE == kLossGrad)
        for (float& s : sums) s = 0.f;
    auto give_up = [&]() {
        s_fail = 1;
        atomicExch(A.err, 1);
    };

    if (warp == 7) {
        if (elect_one()) {
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_w), "r"(Sh::kImage) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                             smem_u32(s_w)),
                         "l"(A.image), "r"(Sh::kImage), "r"(bar_w)
                         : "memory");
            const uint32_t ring = smem_u32(s_ring);
            const uint64_t b0 = smem_desc(smem_u32(s_w), Sh::kRows * 16, 128);
            bool ok = wait_parity(bar_w, 0, A.spin, &s_fail);
            uint32_t q = 0, used = 0, phase = 0;  // planes so far; per block: written before, parity of its next release
            bool ready = false;                   // plane q is known to be there
            Walk walk(A.t);
            for (Column c; ok && walk.next(A.t, c);) {
                const int nz = c.nz;
                for (int j = -1; j <= nz; ++j, ++q) {
                    const uint32_t s = q % kRing;
                    ok = ready || wait_parity(full(s), (q / kRing) & 1, A.spin, &s_fail);
                    if (!ok) break;
                    fence_after();
                    // plane j goes to the output planes j - 1 .. j + 1 that the column has
                    const int lo = max(j - 1, 0), hi = min(j + 1, nz - 1);
                    const uint64_t a = smem_desc(ring + s * Sh::kSlot, kChunk, kHx * 16);
                    const uint64_t b = b0 + (uint64_t)((lo - (j - 1)) * NB);  // rows of 16 bytes
                    const uint32_t d = tmem + (uint32_t)(lo * NB), n = (uint32_t)((hi - lo + 1) * NB);
                    const bool fresh = hi == j + 1;
                    if (fresh) {  // block hi starts here: its first product replaces what it held
                        if ((used >> hi) & 1) {  // an output of the column before, which must have been read
                            ok = wait_parity(freed(hi), (phase >> hi) & 1, A.spin, &s_fail);
                            if (!ok) break;
                            phase ^= 1u << hi;
                            fence_after();
                        }
                        used |= 1u << hi;
                        if (lo < hi) mma_f16(d, a, b, kIdesc | idesc_n(n - NB), 1);
                        mma_f16(tmem + (uint32_t)(hi * NB), a, b + (uint64_t)((hi - lo) * NB), kIdesc | idesc_n(NB), 0);
                    } else {
                        mma_f16(d, a, b, kIdesc | idesc_n(n), 1);
                    }
                    const uint32_t id = kIdesc | idesc_n(n);
#pragma unroll
                    for (int tap = 0; tap < 9; ++tap) {
                        // asked while MMAs are queued: the answer's latency leaves no gap between planes
                        if (tap == 6) ready = test_parity(full((q + 1) % kRing), ((q + 1) / kRing) & 1);
#pragma unroll
                        for (int k = 0; k < Sh::kSteps; ++k)
                            if (tap || k)
                                mma_f16(d, a + (uint64_t)((tap / 3) * kHx + tap % 3 + k * (int)(2 * kChunk / 16)),
                                        b + (uint64_t)((tap * (int)Sh::kTap + k * (int)(2 * Sh::kRows * 16)) / 16), id, 1);
                    }
                    commit(empty(s));
                    if (j >= 1) commit(done(j - 1));
                }
            }
            if (!ok) give_up();
            commit(bar_drain);
            (void)wait_parity(bar_drain, 0, kTcWaitPolls, nullptr);
            (void)wait_parity(bar_w, 0, kTcWaitPolls, nullptr);  // the weights' copy, had the first wait given up
        }
        __syncwarp();
    } else if (warp >= 4) {
        // plane q into ring slot q % 4 as 16-byte copies, announced one plane later
        const int st = t - kEpiThreads;
        uint32_t dst[Sh::kPer], off[Sh::kPer];
        uint32_t q = 0;
        bool ok = true;
        const uint32_t ring = smem_u32(s_ring);
        Walk walk(A.t);
        for (Column c; ok && walk.next(A.t, c);) {
#pragma unroll
            for (int i = 0; i < Sh::kPer; ++i) {
                const int p = st + i * kStagers, v = p / KC, k = p % KC;
                dst[i] = (uint32_t)k * kChunk + (uint32_t)v * 16;
                off[i] = (uint32_t)(wrap(c.y0 + v / kHx - 1, A.t.H) * A.t.W + wrap(c.x0 + v % kHx - 1, A.t.W)) * KC + (uint32_t)k;
            }
            const uint4* grid = reinterpret_cast<const uint4*>(A.in) + (long long)c.b * A.t.D * A.t.H * A.t.W * KC;
            for (int j = -1; j <= c.nz; ++j, ++q) {
                const uint32_t s = q % kRing;
                if (q >= kRing && !wait_parity(empty(s), (q / kRing - 1) & 1, A.spin, &s_fail)) {
                    ok = false;
                    break;
                }
                const uint4* plane = grid + (long long)wrap(c.z0 + j, A.t.D) * A.t.H * A.t.W * KC;
#pragma unroll
                for (int i = 0; i < Sh::kPer; ++i)
                    if (st + i * kStagers < Sh::kPieces) copy16(ring + s * Sh::kSlot + dst[i], plane + off[i]);
                copies_commit();
                if (q > 0) {
                    copies_wait<1>();
                    fence_async();
                    mbar_arrive(full((q - 1) % kRing));
                }
            }
        }
        copies_wait<0>();
        if (ok && q > 0) {
            fence_async();
            mbar_arrive(full((q - 1) % kRing));
        }
        if (!ok) give_up();
    } else {
        // rows 32 w .. 32 w + 31 of every finished block belong to warp w: row m is voxel (m % 8, m / 8)
        uint32_t phase = 0;
        bool ok = true;
        const long long vox = (long long)A.t.D * A.t.H * A.t.W;
        float bias[MODE == kAdjoint ? 1 : kOut];
        if (MODE != kAdjoint)
#pragma unroll
            for (int ch = 0; ch < kOut; ++ch) bias[ch] = A.bias[ch];
        Walk walk(A.t);
        for (Column c; ok && walk.next(A.t, c);) {
            const int x = c.x0 + t % TX, y = c.y0 + t / TX;
            const bool inside = x < A.t.W && y < A.t.H;
            // what an output needs besides its sums
            struct Extra {
                uint32_t bits;
                float x[MODE == kPrediction || MODE == kLossGrad ? kFieldChannels : 1], t[MODE == kLossGrad ? kFieldChannels : 1];
            } next;
            auto fetch = [&](long long row, long long e) {
                Extra f{};
                if (!inside) return f;
                if (MODE == kAdjoint) f.bits = A.bits[row];
                if (MODE == kPrediction || MODE == kLossGrad)
#pragma unroll
                    for (int ch = 0; ch < kFieldChannels; ++ch) {
                        f.x[ch] = A.x[e + ch * vox];
                        if (MODE == kLossGrad) f.t[ch] = A.target[e + ch * vox];
                    }
                return f;
            };
            for (int o = 0; o < c.nz; ++o) {
                const long long v = ((long long)(c.z0 + o) * A.t.H + y) * A.t.W + x;  // in its sample
                const long long row = (long long)c.b * vox + v, e = (long long)c.b * kFieldChannels * vox + v;
                if (o == 0) next = fetch(row, e);
                const Extra now = next;
                uint32_t bits = now.bits;
                // read while this output is waited for and finished
                if (o + 1 < c.nz) next = fetch(row + (long long)A.t.H * A.t.W, e + (long long)A.t.H * A.t.W);
                if (!wait_parity(done(o), (phase >> o) & 1, A.spin, &s_fail)) {
                    ok = false;
                    break;
                }
                phase ^= 1u << o;
                fence_after();
                const uint32_t addr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(o * NB);
                if constexpr (NB == 32) {
                    uint32_t r[32];
                    tmem_load32(addr, r);
                    fence_before();
                    mbar_arrive(freed(o));
                    uint32_t packed[16];
                    if (MODE == kHiddenLayer) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const __half2 p = __floats2half2_rn(fmaxf(__uint_as_float(r[2 * i]) + bias[2 * i], 0.f),
                                                                fmaxf(__uint_as_float(r[2 * i + 1]) + bias[2 * i + 1], 0.f));
                            const uint32_t u = *reinterpret_cast<const uint32_t*>(&p);
                            packed[i] = u;  // values are >= 0: positive is not zero
                            bits |= ((u & 0x7fffu) ? 1u : 0u) << (2 * i) | ((u & 0x7fff0000u) ? 1u : 0u) << (2 * i + 1);
                        }
                        if (A.bits && inside) A.bits[row] = bits;
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; ++i) {  // outside the grid every bit is 0
                            const float a = (bits >> (2 * i)) & 1 ? __uint_as_float(r[2 * i]) : 0.f;
                            const float b = (bits >> (2 * i + 1)) & 1 ? __uint_as_float(r[2 * i + 1]) : 0.f;
                            sums[2 * i] += a;
                            sums[2 * i + 1] += b;
                            const __half2 p = __floats2half2_rn(a, b);
                            packed[i] = *reinterpret_cast<const uint32_t*>(&p);
                        }
                    }
                    store_voxels(packed, A.out + ((long long)c.b * vox + (long long)(c.z0 + o) * A.t.H * A.t.W) * 32, c.x0,
                                 c.y0 + 4 * warp, A.t.H, A.t.W);
                } else {
                    uint32_t r[8];
                    tmem_load8(addr, r);
                    fence_before();
                    mbar_arrive(freed(o));
                    if (inside) {
                        float g[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int ch = 0; ch < kFieldChannels; ++ch) {
                            const float d = __uint_as_float(r[ch]) + bias[ch];
                            if (MODE == kPrediction) {
                                A.y[e + ch * vox] = now.x[ch] + d;
                            } else {
                                const float diff = now.x[ch] + d - now.t[ch];
                                g[ch] = A.loss_scale * A.w[ch] * diff;
                                sums[ch] += g[ch];
                                loss.add(A.w[ch], diff);
                            }
                        }
                        if (MODE == kLossGrad) {
                            __half2 p[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                p[i] = __floats2half2_rn(g[2 * i] * A.grad_scale, g[2 * i + 1] * A.grad_scale);
                            reinterpret_cast<uint4*>(A.out)[row] = *reinterpret_cast<const uint4*>(p);
                        }
                    }
                }
                fence_before();
            }
        }
        if (!ok) give_up();
    }
    // every role has left its loop: no copy or MMA of this CTA is in flight
    fence_before();
    __syncthreads();
    fence_after();
    if (t < 32) tmem_free<Sh::kCols>(tmem);
    if (MODE == kAdjoint || MODE == kLossGrad) {
        // this CTA's sums over its 128 rows, in a fixed order
        constexpr int kSums = MODE == kAdjoint ? 32 : kFieldChannels, kLd = kSums + 1;
        float* s_sum = reinterpret_cast<float*>(smem);
        double* s_loss = reinterpret_cast<double*>(smem + 4 * kEpiThreads * 34);
        if (t < kEpiThreads) {
#pragma unroll
            for (int ch = 0; ch < kSums; ++ch) s_sum[t * kLd + ch] = sums[ch];
            if (MODE == kLossGrad) s_loss[t] = loss.value();
        }
        __syncthreads();
        if (t < kSums) {
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            for (int r = 0; r < kEpiThreads; r += 4)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i] += s_sum[(r + i) * kLd + t];
            A.bias_part[blockIdx.x * 32 + t] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
        }
        if (MODE == kLossGrad && t == 32) {
            double s = 0.0;
            for (int r = 0; r < kEpiThreads; ++r) s += s_loss[r];
            A.loss_part[blockIdx.x] = s;
        }
    }
}

// ---------------------------------------------------------------------------------------
// Weight gradients: gW[o][c][dz, dy, dx] = sum over voxels v of g[o][v] h[c][v + off(tap)], as a GEMM
// over the voxels. Both operands are MN-major: a core matrix is 8 voxels of an x-run (K) x 8
// channels (16 bytes of a voxel). The M = 128 rows are (dx, c), three copies of each row of h shifted in
// x, side by side (row pitch 3 chunks of 128 bytes per 8 channels; the rows past dx = 2 read on into
// the next row and belong to nothing). Shifts in y are on the other operand: with w = y + dy - 1 the row
// of h, its products go to the rows w - 1, w, w + 1 of g, which follow one another in shared memory
// with their channel chunks, so the N = 96 columns are (2 - dy, o) and one MMA does three dy. Three
// accumulators, one per dz, stay in tensor memory for all columns of a CTA: 24 MMAs per plane of 128
// voxels (72 of N = 32 when the nine (dz, dy) had accumulators of their own).
//
// Each CTA walks columns of z planes; unit j of a column is plane j of h and plane j - 1 of g, in a
// ring of five; after unit j the MMAs of g's plane j - 1 with h's planes j - 2, j - 1, j run. Its sums
// go to a slice of its own, added in CTA order by grads_finish_kernel.
//
// Bound as the convolution: batch 4 at 64^3, 32 x 32 channels, 58 us against 174 us (45 us against 174
// with the five fields on either side).
// ---------------------------------------------------------------------------------------
constexpr int kWgThreads = 256, kWgStagers = 224, kWgRing = 5;

// KA and KB: chunks of 8 channels of h and g. The five fields (KA = 1) leave room in M for all nine
// (dz, dx): a unit then holds its own copies of the three planes of h, one accumulator serves all
// taps, and a plane takes 8 MMAs instead of 24.
template <int KA, int KB>
struct WgradShape {
    static constexpr bool kStack = KA == 1;
    static constexpr int kAccs = kStack ? 1 : 3, kCopies = kStack ? 9 : 3;
    // core matrices 160 bytes apart where a voxel has four chunks: its pieces fall into different banks
    static constexpr uint32_t kMatA = KA == 4 ? 160 : 128, kMatB = KB == 4 ? 160 : 128;
    static constexpr uint32_t kRowA = kCopies * KA * kMatA, kPlaneA = TY * kRowA;
    static constexpr uint32_t kRowB = KB * kMatB, kPlaneB = (TY + 3) * kRowB;  // 18 rows and one of zeros
    static constexpr uint32_t kN = KB == 4 ? 96 : 32;
    static constexpr uint32_t kUnit = kPlaneA + kPlaneB;
    static constexpr uint32_t kSmem = kWgRing * kUnit;
    static_assert(kRowA * 15 + kMatA * 15 + 128 <= kUnit, "the 16 core matrices read from the last row of A end inside the unit");
    static constexpr int kRowsOut = kCopies * 8 * KA, kColsOut = 3 * 8 * KB;
    static constexpr int kPart = kAccs * kRowsOut * kColsOut;  // floats of a CTA's slice
    static_assert(kPart % 4 == 0);
    static constexpr int kPiecesA = TY * kCopies * TX * KA, kPiecesB = (TY + 2) * TX * KB;
    static constexpr int kPerA = (kPiecesA + kWgStagers - 1) / kWgStagers, kPerB = (kPiecesB + kWgStagers - 1) / kWgStagers;
    static constexpr int kFirst = kStack ? 0 : -1, kPast = kStack ? 0 : 1;  // units of a column: kFirst .. nz - 1 + kPast
};

struct WgradArgs {
    const __half* h;
    const __half* g;
    float* part;
    Tiling t;
    long long spin;
    int* err;
};

template <int KA, int KB>
__global__ void __launch_bounds__(kWgThreads, 1) wgrad_tc_kernel(const __grid_constant__ WgradArgs A) {
    using Sh = WgradShape<KA, KB>;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_bar[2 * kWgRing + 1];  // full, empty, drain
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_fail;
    const int t = threadIdx.x, warp = __shfl_sync(0xffffffffu, t / 32, 0);
    const uint32_t bar = smem_u32(s_bar);
    auto full = [&](uint32_t s) { return bar + 8u * s; };
    auto empty = [&](uint32_t s) { return bar + 8u * (kWgRing + s); };
    const uint32_t bar_drain = bar + 8u * 2 * kWgRing;
    if (t == 0) {
        for (uint32_t s = 0; s < kWgRing; ++s) {
            mbar_init(full(s), kWgStagers);
            mbar_init(empty(s), 1);
        }
        mbar_init(bar_drain, 1);
        s_fail = 0;
    }
    // bytes that nothing writes are read into rows and columns that nothing uses
    for (int i = t; i < (int)(Sh::kSmem / 16); i += kWgThreads) reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
    chain_begin();
    chain_next();
    if (t < 32) tmem_alloc<512>(&s_tmem);
    fence_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem, ring = smem_u32(smem);
    auto give_up = [&]() {
        s_fail = 1;
        atomicExch(A.err, 1);
    };
    if (warp == 7) {
        if (elect_one()) {
            bool ok = true;
            uint32_t q = 0, acc = 0;
            bool ready = false;  // unit q is known to be there
            constexpr uint32_t id = kIdesc | kMnMajor | idesc_n(Sh::kN);
            auto slot = [&](uint32_t back) { return (q + kWgRing - back) % kWgRing; };
            Walk walk(A.t);
            for (Column c; ok && walk.next(A.t, c);) {
                for (int j = Sh::kFirst; j < c.nz + Sh::kPast; ++j, ++q) {
                    ok = ready || wait_parity(full(slot(0)), (q / kWgRing) & 1, A.spin, &s_fail);
                    ready = false;
                    if (!ok) break;
                    fence_after();
                    if (!Sh::kStack && j < 1) continue;
                    const uint64_t b = smem_desc(ring + slot(0) * Sh::kUnit + Sh::kPlaneA, Sh::kRowB, Sh::kMatB);
#pragma unroll
                    for (int dz = 0; dz < Sh::kAccs; ++dz) {
                        const uint64_t a = smem_desc(ring + slot(Sh::kAccs - 1 - dz) * Sh::kUnit, Sh::kRowA, Sh::kMatA);
#pragma unroll
                        for (int k = 0; k < TY / 2; ++k) {  // two rows of 8 voxels per MMA
                            if (dz == Sh::kAccs - 1 && k == 4) ready = test_parity(full((q + 1) % kWgRing), ((q + 1) / kWgRing) & 1);
                            mma_f16(tmem + (uint32_t)(dz * Sh::kN), a + (uint64_t)(2 * k * (int)Sh::kRowA / 16),
                                    b + (uint64_t)(2 * k * (int)Sh::kRowB / 16), id, k ? 1u : acc);
                        }
                    }
                    acc = 1;
                    if (Sh::kStack) {
                        commit(empty(slot(0)));
                    } else {
                        commit(empty(slot(2)));
                        if (j == c.nz) {  // the column's last units serve no further plane
                            commit(empty(slot(1)));
                            commit(empty(slot(0)));
                        }
                    }
                }
            }
            if (!ok) give_up();
            commit(bar_drain);
            (void)wait_parity(bar_drain, 0, kTcWaitPolls, nullptr);
        }
        __syncwarp();
    } else {
        constexpr uint32_t kNone = 0xffffffffu;  // no such piece, or one outside the grid: zero
        uint32_t da[Sh::kPerA], oa[Sh::kPerA], db[Sh::kPerB], ob[Sh::kPerB];
        uint32_t q = 0;
        bool ok = true;
        Walk walk(A.t);
        for (Column c; ok && walk.next(A.t, c);) {
#pragma unroll
            for (int i = 0; i < Sh::kPerA; ++i) {  // (row, copy, voxel, chunk), chunks fastest in global memory
                const int p = t + i * kWgStagers, k = p % KA, v = p / KA % TX, copy = p / (KA * TX) % Sh::kCopies;
                const int r = p / (KA * TX * Sh::kCopies), dx = copy % 3;
                da[i] = p < Sh::kPiecesA ? (uint32_t)r * Sh::kRowA + (uint32_t)(copy * KA + k) * Sh::kMatA + (uint32_t)v * 16 : kNone;
                oa[i] = p < Sh::kPiecesA && c.y0 + r < A.t.H
                            ? (uint32_t)((c.y0 + r) * A.t.W + wrap(c.x0 + v + dx - 1, A.t.W)) * KA + (uint32_t)k
                            : kNone;
            }
#pragma unroll
            for (int i = 0; i < Sh::kPerB; ++i) {
                const int p = t + i * kWgStagers, k = p % KB, v = p / KB % TX, r = p / (KB * TX);
                db[i] = p < Sh::kPiecesB ? Sh::kPlaneA + (uint32_t)r * Sh::kRowB + (uint32_t)k * Sh::kMatB + (uint32_t)v * 16 : kNone;
                ob[i] = p < Sh::kPiecesB && c.x0 + v < A.t.W
                            ? (uint32_t)(wrap(c.y0 + r - 1, A.t.H) * A.t.W + c.x0 + v) * KB + (uint32_t)k
                            : kNone;
            }
            const long long plane = (long long)A.t.H * A.t.W;
            const uint4* hb = reinterpret_cast<const uint4*>(A.h) + (long long)c.b * A.t.D * plane * KA;
            const uint4* gb = reinterpret_cast<const uint4*>(A.g) + (long long)c.b * A.t.D * plane * KB;
            auto put = [&](uint32_t dst, const uint4* src, uint32_t off) {
                if (off != kNone) copy16(dst, src + off);
                else asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "r"(0) : "memory");
            };
            for (int j = Sh::kFirst; j < c.nz + Sh::kPast; ++j, ++q) {
                const uint32_t slot = ring + (q % kWgRing) * Sh::kUnit;
                if (q >= kWgRing && !wait_parity(empty(q % kWgRing), (q / kWgRing - 1) & 1, A.spin, &s_fail)) {
                    ok = false;
                    break;
                }
                const uint4* h0 = hb + (long long)wrap(c.z0 + j - (Sh::kStack ? 1 : 0), A.t.D) * plane * KA;
                const uint4* h1 = Sh::kStack ? hb + (long long)(c.z0 + j) * plane * KA : h0;
                const uint4* h2 = Sh::kStack ? hb + (long long)wrap(c.z0 + j + 1, A.t.D) * plane * KA : h0;
#pragma unroll
                for (int i = 0; i < Sh::kPerA; ++i) {
                    if (da[i] == kNone) continue;
                    const int dz = Sh::kStack ? (t + i * kWgStagers) / (KA * TX * 3) % 3 : 0;
                    put(slot + da[i], dz == 0 ? h0 : dz == 1 ? h1 : h2, oa[i]);
                }
                if (Sh::kStack || j >= 1) {
                    const uint4* gp = gb + (long long)(c.z0 + j - Sh::kPast) * plane * KB;
#pragma unroll
                    for (int i = 0; i < Sh::kPerB; ++i)
                        if (db[i] != kNone) put(slot + db[i], gp, ob[i]);
                }
                copies_commit();
                if (q > 0) {
                    copies_wait<1>();
                    fence_async();
                    mbar_arrive(full((q - 1) % kWgRing));
                }
            }
        }
        copies_wait<0>();
        if (ok && q > 0) {
            fence_async();
            mbar_arrive(full((q - 1) % kWgRing));
        }
        if (!ok) give_up();
    }
    fence_before();
    __syncthreads();
    fence_after();
    // accumulator a, row m, column n = (2 - dy, o) to part[a][n][m]; warp w < 4 holds rows 32 w .. 32 w + 31
    if (!s_fail && t < 128) {
        float* part = A.part + (long long)blockIdx.x * Sh::kPart;
        for (int a = 0; a < Sh::kAccs; ++a)
            for (int n0 = 0; n0 < (int)Sh::kN; n0 += 32) {
                uint32_t r[32];
                tmem_load32(tmem + ((uint32_t)(warp * 32) << 16) + a * Sh::kN + (uint32_t)n0, r);
                if (t < Sh::kRowsOut)
#pragma unroll
                    for (int n = 0; n < 32; ++n)
                        if (n0 + n < Sh::kColsOut)
                            part[(a * Sh::kColsOut + n0 + n) * Sh::kRowsOut + t] = __uint_as_float(r[n]);
            }
    }
    fence_before();
    __syncthreads();
    if (t < 32) tmem_free<512>(tmem);
}

// ---------------------------------------------------------------------------------------
// Small kernels
// ---------------------------------------------------------------------------------------

// FP16 copy of the fields x [B][5][vox], channels last and padded to 8.
__global__ void pack_fields_kernel(const float* x, uint4* __restrict__ out, long long vox, int batch) {
    chain_begin();
    chain_next();
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < vox * batch; i += (long long)gridDim.x * blockDim.x) {
        const long long b = i / vox;
        const float* p = x + b * kFieldChannels * vox + (i - b * vox);
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < kFieldChannels; ++c) v[c] = p[c * vox];
        __half2 h[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) h[c] = __floats2half2_rn(v[2 * c], v[2 * c + 1]);
        out[i] = *reinterpret_cast<const uint4*>(h);
    }
}

// One layer's weights as conv_tc_kernel's B operand: per tap (dy, dx) and K step, two chunks of 8
// input channels, each 3 NB rows (dz = 2, 1, 0; outputs) of 16 bytes. flip: the adjoint's weights,
// Wt[c][o][26 - tap] of a layer W[o][c][tap].
struct ImageArgs {
    struct Layer {
        const float* w;
        __half* image;
        int cout, cin, nb, steps, flip;
    } layer[2 * kLayers - 1];
};
__global__ void weight_images_kernel(const __grid_constant__ ImageArgs A) {
    chain_begin();
    chain_next();
    const ImageArgs::Layer& L = A.layer[blockIdx.y];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int rows = 3 * L.nb, n = 9 * L.steps * 2 * rows * 8;
    if (i >= n) return;
    const int e = i % 8, row = i / 8 % rows, chunk = i / (8 * rows) % (2 * L.steps), tap2 = i / (16 * L.steps * rows);
    const int c = chunk * 8 + e, o = row % L.nb, dz = 2 - row / L.nb;
    const int tap = 9 * dz + tap2;
    float w = 0.f;
    if (!L.flip) {
        if (o < L.cout && c < L.cin) w = L.w[((long long)o * L.cin + c) * 27 + tap];
    } else if (o < L.cin && c < L.cout) {
        w = L.w[((long long)c * L.cin + o) * 27 + (26 - tap)];
    }
    L.image[i] = __float2half_rn(w);
}

// The gradients of every layer from the CTAs' slices: element e of a slice is (accumulator, column
// (2 - dy, o), row). A block takes 64 elements, a thread four of them and a sixteenth of the CTAs in
// order, so that its ten loads of 16 bytes are all in flight; the sixteen sums are then added pairwise.
// The last block of a layer takes the bias gradients, a lane per channel and a warp per eighth of the
// CTAs. 12 us (17 before, when the bias block's loads waited for one another).
constexpr int kFinishElems = 64, kFinishSplit = 16, kFinishThreads = kFinishElems / 4 * kFinishSplit;
struct FinishArgs {
    struct Layer {
        const float* part;
        const float* bias_part;
        float* gw;
        float* gb;
        int cout, cin, stack, rows, cols, n, parts, bias_parts;
        float scale;       // of the slices' sums
        float bias_scale;
    } layer[kLayers];
};
__global__ void __launch_bounds__(kFinishThreads) grads_finish_kernel(const __grid_constant__ FinishArgs A) {
    chain_begin();
    const FinishArgs::Layer& L = A.layer[blockIdx.y];
    __shared__ __align__(16) float s_sum[kFinishSplit][kFinishElems];
    if (blockIdx.x == gridDim.x - 1) {
        constexpr int kWarps = kFinishThreads / 32;
        const int o = threadIdx.x & 31, warp = threadIdx.x >> 5;
        float acc = 0.f;
        const int k0 = L.bias_parts * warp / kWarps, k1 = L.bias_parts * (warp + 1) / kWarps, last = k1 - 1;
        const float* p = L.bias_part + (o < L.cout ? o : 0);
        for (int k = k0; k < k1; k += 20) {
            float v[20];
#pragma unroll
            for (int i = 0; i < 20; ++i) v[i] = p[min(k + i, last) * 32];
#pragma unroll
            for (int i = 0; i < 20; ++i) acc += k + i < k1 ? v[i] : 0.f;
        }
        s_sum[warp][o] = acc;
        __syncthreads();
        if (warp == 0 && o < L.cout) {
            acc = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; w += 2) acc += s_sum[w][o] + s_sum[w + 1][o];
            L.gb[o] = acc * L.bias_scale;
        }
        return;
    }
    if ((int)blockIdx.x * kFinishElems >= L.n) return;
    const int quad = threadIdx.x % (kFinishElems / 4) * 4, part = threadIdx.x / (kFinishElems / 4);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (blockIdx.x * kFinishElems + quad < L.n) {  // slices are multiples of four floats
        const int k0 = L.parts * part / kFinishSplit, k1 = L.parts * (part + 1) / kFinishSplit;
        const float* p = L.part + blockIdx.x * kFinishElems + quad;
        const int last = k1 - 1;
        for (int k = k0; k < k1; k += 10) {
            float4 v[10];
#pragma unroll
            for (int i = 0; i < 10; ++i) v[i] = *reinterpret_cast<const float4*>(p + (long long)min(k + i, last) * L.n);
#pragma unroll
            for (int i = 0; i < 10; ++i)
                if (k + i < k1) {
                    acc.x += v[i].x;
                    acc.y += v[i].y;
                    acc.z += v[i].z;
                    acc.w += v[i].w;
                }
        }
    }
    *reinterpret_cast<float4*>(&s_sum[part][quad]) = acc;
    __syncthreads();
    const int le = threadIdx.x, e = blockIdx.x * kFinishElems + le;
    if (le >= kFinishElems || e >= L.n) return;
    float sum[kFinishSplit];
#pragma unroll
    for (int k = 0; k < kFinishSplit; ++k) sum[k] = s_sum[k][le];
#pragma unroll
    for (int w = kFinishSplit / 2; w > 0; w /= 2)
#pragma unroll
        for (int k = 0; k < w; ++k) sum[k] += sum[k + w];
    const int m = e % L.rows, col = e / L.rows % L.cols;
    const int kc = L.stack ? 8 : L.rows / 3, kb = L.cols / 3, copy = m / kc;
    const int dz = L.stack ? copy / 3 : e / (L.rows * L.cols), dx = copy % 3, c = m % kc, dy = 2 - col / kb, o = col % kb;
    if (o < L.cout && c < L.cin)
        L.gw[((long long)o * L.cin + c) * 27 + 9 * dz + 3 * dy + dx] = sum[0] * L.scale;
}

int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

Tiling tiling(const TcNet& N, int most) {
    Tiling T{N.D, N.H, N.W, (N.W + TX - 1) / TX, (N.H + TY - 1) / TY, most, 0};
    T.planes = T.tiles_x * T.tiles_y * N.batch * N.D;
    return T;
}

// The CTAs launched go to *ctas.
template <int KC, int NB, int MODE>
cudaError_t launch_conv(const TcNet& N, ConvArgs A, int* ctas, cudaStream_t s) {
    using Sh = ConvShape<KC, NB>;
    A.t = tiling(N, kMaxPlanes);
    *ctas = std::min(A.t.planes, 2 * N.ctas);  // two per SM
    cudaError_t e = cudaFuncSetAttribute(conv_tc_kernel<KC, NB, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::kSmem);
    if (e != cudaSuccess) return e;
    return launch_chained(conv_tc_kernel<KC, NB, MODE>, dim3(*ctas), dim3(kConvThreads), Sh::kSmem, s, A);
}

template <int KA, int KB>
cudaError_t launch_wgrad(const TcNet& N, WgradArgs A, int* ctas, cudaStream_t s) {
    using Sh = WgradShape<KA, KB>;
    A.t = tiling(N, N.D);
    *ctas = std::min(A.t.planes, N.ctas);
    cudaError_t e = cudaFuncSetAttribute(wgrad_tc_kernel<KA, KB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::kSmem);
    if (e != cudaSuccess) return e;
    return launch_chained(wgrad_tc_kernel<KA, KB>, dim3(*ctas), dim3(kWgThreads), Sh::kSmem, s, A);
}

constexpr size_t kImageBytes[2 * kLayers - 1] = {
    ConvShape<1, 32>::kImage, ConvShape<4, 32>::kImage, ConvShape<4, 32>::kImage, ConvShape<4, 16>::kImage,  // forward
    ConvShape<1, 32>::kImage, ConvShape<4, 32>::kImage, ConvShape<4, 32>::kImage};                          // adjoints of 3, 2, 1
constexpr int kWgradFloats[kLayers] = {WgradShape<1, 4>::kPart, WgradShape<4, 4>::kPart, WgradShape<4, 4>::kPart,
                                       WgradShape<4, 1>::kPart};

}  // namespace

TcSizes tc_sizes() {
    TcSizes z{};
    for (size_t b : kImageBytes) z.image_bytes += b;
    z.ctas = sm_count();
    for (int f : kWgradFloats) z.part_floats += (size_t)z.ctas * f;
    z.bias_floats = (size_t)kLayers * 2 * z.ctas * 32;
    z.loss_parts = 2 * z.ctas;
    return z;
}

// Layers are numbered 0 .. 3; h[l] is the output of hidden layer l, g[l] the gradient of that
// output before its ReLU, gout that of the prediction.
cudaError_t tc_run(const TcNet& N, const float* x, float* y, const float* target, float* grads, int* loss_parts, cudaStream_t s) {
    cudaError_t e;
    const long long vox = (long long)N.D * N.H * N.W;
    const bool train = target != nullptr;
    int ctas = 0;
    {
        const long long blk = (vox * N.batch + 255) / 256;
        e = launch_chained(pack_fields_kernel, dim3((unsigned)std::min<long long>(blk, 4096)), dim3(256), 0, s, x,
                           static_cast<uint4*>(N.x), vox, N.batch);
        if (e != cudaSuccess) return e;
    }
    const __half* image[2 * kLayers - 1];
    {
        ImageArgs I;
        unsigned char* at = static_cast<unsigned char*>(N.images);
        for (int k = 0; k < 2 * kLayers - 1; ++k) {
            const bool flip = k >= kLayers;  // the adjoints of layers 3, 2, 1
            const int l = flip ? 2 * kLayers - 1 - k : k;
            const int in = flip ? N.cout[l] : N.cin[l], out = flip ? N.cin[l] : N.cout[l];
            I.layer[k] = {N.params + N.w_off[l], reinterpret_cast<__half*>(at), N.cout[l], N.cin[l], out > 8 ? 32 : 16,
                          in > 8 ? 2 : 1, flip};
            image[k] = reinterpret_cast<const __half*>(at);
            at += kImageBytes[k];
        }
        e = launch_chained(weight_images_kernel,
                           dim3((unsigned)(ConvShape<4, 32>::kImage / 2 + 255) / 256, train ? 2 * kLayers - 1 : kLayers), dim3(256), 0, s, I);
        if (e != cudaSuccess) return e;
    }
    ConvArgs A{};
    A.spin = N.spin;
    A.err = N.err;
    for (int l = 0; l < kLayers - 1; ++l) {
        A.in = static_cast<const __half*>(l == 0 ? N.x : N.h[l - 1]);
        A.image = image[l];
        A.bias = N.params + N.b_off[l];
        A.out = static_cast<__half*>(N.h[l]);
        A.bits = train ? N.bits[l] : nullptr;
        e = l == 0 ? launch_conv<1, 32, kHiddenLayer>(N, A, &ctas, s) : launch_conv<4, 32, kHiddenLayer>(N, A, &ctas, s);
        if (e != cudaSuccess) return e;
    }
    A.in = static_cast<const __half*>(N.h[kLayers - 2]);
    A.image = image[kLayers - 1];
    A.bias = N.params + N.b_off[kLayers - 1];
    A.bits = nullptr;
    A.x = x;
    if (!train) {
        A.y = y;
        return launch_conv<4, 16, kPrediction>(N, A, &ctas, s);
    }
    FinishArgs F;
    const size_t bias_layer = (size_t)2 * N.ctas * 32;
    A.target = target;
    A.out = static_cast<__half*>(N.gout);
    A.loss_part = N.loss_part;
    A.bias_part = N.bias_part + (kLayers - 1) * bias_layer;
    A.grad_scale = N.grad_scale;
    A.loss_scale = (float)(2.0 / (double)(vox * N.batch * kFieldChannels));
    for (int c = 0; c < kFieldChannels; ++c) A.w[c] = N.loss_w[c];
    if ((e = launch_conv<4, 16, kLossGrad>(N, A, loss_parts, s)) != cudaSuccess) return e;
    F.layer[kLayers - 1].bias_parts = *loss_parts;
    float* part = N.part;
    for (int l = kLayers - 1; l >= 0; --l) {
        FinishArgs::Layer& L = F.layer[l];
        const void* g = l == kLayers - 1 ? N.gout : N.g[l];
        WgradArgs G{};
        G.h = static_cast<const __half*>(l == 0 ? N.x : N.h[l - 1]);
        G.g = static_cast<const __half*>(g);
        G.part = part;
        G.spin = N.spin;
        G.err = N.err;
        L.part = part;
        L.bias_part = N.bias_part + l * bias_layer;
        L.gw = grads + N.w_off[l];
        L.gb = grads + N.b_off[l];
        L.cout = N.cout[l];
        L.cin = N.cin[l];
        L.stack = N.cin[l] <= 8;
        L.rows = L.stack ? 72 : 96;
        L.cols = N.cout[l] > 8 ? 96 : 24;
        L.n = kWgradFloats[l];
        L.scale = 1.0f / N.grad_scale;
        L.bias_scale = l == kLayers - 1 ? 1.0f : 1.0f / N.grad_scale;
        part += (size_t)N.ctas * kWgradFloats[l];
        if (l == kLayers - 1) e = launch_wgrad<4, 1>(N, G, &L.parts, s);
        else if (l == 0) e = launch_wgrad<1, 4>(N, G, &L.parts, s);
        else e = launch_wgrad<4, 4>(N, G, &L.parts, s);
        if (e != cudaSuccess) return e;
        if (l == 0) break;
        // the gradient of layer l - 1's output, in the same scaled units as this one's
        A.in = static_cast<const __half*>(g);
        A.image = image[2 * kLayers - 1 - l];
        A.bias = nullptr;
        A.out = static_cast<__half*>(N.g[l - 1]);
        A.bits = N.bits[l - 1];
        A.bias_part = N.bias_part + (l - 1) * bias_layer;
        int* parts = &F.layer[l - 1].bias_parts;
        e = l == kLayers - 1 ? launch_conv<1, 32, kAdjoint>(N, A, parts, s) : launch_conv<4, 32, kAdjoint>(N, A, parts, s);
        if (e != cudaSuccess) return e;
    }
    return launch_chained(grads_finish_kernel, dim3((unsigned)(WgradShape<4, 4>::kPart + kFinishElems - 1) / kFinishElems + 1, kLayers),
                          dim3(kFinishThreads), 0, s, F);
}

}  // namespace net
}  // namespace lbm
