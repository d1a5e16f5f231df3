// Warm-start network on the GPU: BF16 tensor-core convolutions with FP32
// accumulation (forward, data gradient, weight gradient), loss, Adam, and the
// feature / target / unpacking kernels.  See include/adr.h (adr_cnn_*).
//
// Network (the same definition as the FP64 reference): a 256 x 256 node grid
// is read as 64 x 64 cells of 4 x 4 nodes, every problem scaled by
// s = max |u0| of its first initial state u0; features NHWC, 40 channels (f
// and u0 / s at the 16 nodes of the cell; cell means of beta1, beta2, mu and
// sigma codes, cell mean of the mask, 3 zeros); eight 3 x 3 convolutions with
// zero padding, channels 40 64 64 128 128 128 64 64 8, bias, ReLU after all
// but the last; output channel 0 = the cell mean of (u - u0) / s, channels
// 1..7 unused; initial state u0 + s * (bilinear interpolation of channel 0).
// Parameters packed as W_0, b_0, W_1, b_1, ...; W_l[(tap * Cin + ci) * Cout + co].
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "adr_internal.cuh"

namespace {

constexpr int kLayers = 8;
constexpr int kCh[kLayers + 1] = {40, 64, 64, 128, 128, 128, 64, 64, 8};
constexpr int kDil[kLayers] = {1, 2, 4, 8, 16, 32, 1, 1};
constexpr int kHW = 64;   // cells per side
constexpr int kSub = 4;   // nodes per cell side
constexpr int kN = kHW * kSub;
constexpr int kCin = 40, kCout = 8;

long param_offset(int l, bool bias)
{
    long off = 0;
    for (int k = 0; k < l; ++k) off += 9L * kCh[k] * kCh[k + 1] + kCh[k + 1];
    return bias ? off + 9L * kCh[l] * kCh[l + 1] : off;
}

typedef __nv_bfloat16 bf16;

// ------------------------------------------------------------ PTX helpers

__device__ __forceinline__ unsigned smem_u32(const void* p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

// ------------------------------------------------------ convolution kernels

// All convolutions run on the 5th-generation tensor cores as implicit GEMMs
// with M = pixels, N = Cout and K = 9 Cin: tcgen05.mma (kind::f16, BF16
// operands, FP32 accumulators in tensor memory), operands staged by TMA.
// Every mbarrier wait is bounded; when a wait gives up the kernel sets *err,
// lets the loads and MMAs it issued finish, skips its output and frees its
// tensor memory.
struct ConvArgs {
    int B, H, W, dil;
    int cblocks;        // 64-channel blocks of the input
    int kc;             // channels per tap of the K-major weights (64 cblocks)
    const float* bias;  // [Cout] or null
    const bf16* mask;   // [B][H][W][Cout] or null: the output is 0 where the mask is not positive
                        // (the ReLU's backward pass)
    bf16* y;            // [B][H][W][Cout] (64 or 128 channels)
    float* y32;         // [B][H][W][8] FP32 (the last layer)
    int relu;
    int stages, tiles;
    long long spin;     // bound of the mbarrier waits in polls (0: the default bound)
};

constexpr long long kWaitLimit = 1LL << 22;  // default bound: blocking polls (about a second)

// Shared-memory matrix descriptors, 128-byte swizzle, 1024-byte aligned
// operands below 256 KB: the low word holds the address (in 16 bytes) and the
// leading offset, the high word the stride offset (8-row groups 1024 bytes
// apart), the version and the swizzle.  An operand `bytes` further is the low
// word plus bytes / 16, which keeps the issuing thread's work per MMA to one
// addition (it sets the pace where N = 64).
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo) { return (addr >> 4) | ((lbo >> 4) << 16); }

// one lane of a converged warp.  The issuing loops below are run by whole warps
// (uniform values, waits included) and only the issue itself is elected: an MMA
// issued from a branch that one thread took by its index cost about 170 cycles
// whatever its shape, as its operands have to reach uniform registers.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

// the warp's index as a value the compiler knows to be the same in all lanes
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0); }

__device__ __forceinline__ void umma(uint32_t d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %5, 0;\n mov.b64 da, {%1, %3};\n mov.b64 db, {%2, "
        "%3};\n tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n}\n" ::"r"(d),
        "r"(a_lo), "r"(b_lo), "n"(kDescHi), "r"(idesc), "r"(acc));
}

// instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, M x N
__device__ __forceinline__ uint32_t umma_idesc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Wait for the phase of parity `parity` of an mbarrier.  spin <= 0: up to
// kWaitLimit blocking polls (try_wait); spin > 0: up to spin non-blocking
// polls (test_wait), a bound a caller sets to exercise the give-up path.
// Gives up by setting *err and returning false.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err, long long spin = 0)
{
    if (spin > 0) {
        for (long long it = 0; it < spin; ++it) {
            uint32_t ok;
            asm volatile(
                "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(ok)
                : "r"(bar), "r"(parity)
                : "memory");
            if (ok) return true;
        }
    } else {
        for (long long it = 0; it < kWaitLimit; ++it) {
            uint32_t ok;
            asm volatile(
                "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(ok)
                : "r"(bar), "r"(parity)
                : "memory");
            if (ok) return true;
        }
    }
    atomicExch(err, 1);
    return false;
}

// a wait of a whole warp: it goes on or gives up together
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, int* err, long long spin)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, err, spin) ? 1 : 0) != 0;
}

// 16 BF16 values set to 0 where the mask's are not positive (sign set, zero or NaN)
__device__ __forceinline__ void relu_mask16(uint32_t (&v)[8], const bf16* mask)
{
    const uint4 a = *reinterpret_cast<const uint4*>(mask), b = *reinterpret_cast<const uint4*>(mask + 8);
    const uint32_t m[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    auto pos = [](uint32_t h) { return h - 1u < 0x7f80u; };  // 1 .. 0x7f80: positive, infinity included
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (!pos(m[j] & 0xffffu)) v[j] &= 0xffff0000u;
        if (!pos(m[j] >> 16)) v[j] &= 0x0000ffffu;
    }
}

// A persistent CTA per SM walks output tiles of 8 MT x 16 pixels of one image
// and all N output channels, its warps specialised: thread 0 issues the TMA
// loads up to S stages ahead ("full" mbarriers, transaction bytes), a thread of
// warp 1 issues a stage's MMAs as it lands and commits them to the stage's
// "empty" mbarrier, and 4 MT warps read finished accumulators back, two sets
// of accumulators in tensor memory so that a tile's output overlaps the next
// tile's MMAs.  A stage is a tap's input window and weights of 64 channels; the
// image border inside a window comes as TMA's zero fill, and a tap whose window
// lies outside the image altogether is left out (of 9 taps 6.25 on average are
// left at dilation 16 and 4 at 32).  The last layer's 8 channels run as N = 16
// with zero-filled weight rows.
// What bounds it is the operands' traffic from L2 (8 to 13 TB/s into all SMs).
// Loading a window once for the three taps above each other (2 KB rows, so the
// taps are 1024-byte aligned offsets of it) was 20 % faster in the layers of
// small dilation, but sums the taps in another order, which flips BF16
// roundings of the stored activations (0.4 % of the output); the order kept
// here is tap by tap.
// Measured, forward of 128 problems (all eight layers): 1.06 ms with two CTAs
// of one tile each per SM and mma.sync for the last layer, 0.83 ms with this
// kernel for all layers but the first, 0.68 ms with the issue elected and
// k_conv_win; the 128 -> 128 layer at dilation 8 runs at 1.1 PFLOP/s and 12.6
// TB/s from L2 (64 problems).
template <int N, int MT>
struct ConvWs {
    static constexpr int WH = 8 * MT, THREADS = 64 + 128 * MT, COLS = 2 * MT * N;
};
constexpr int kConvMaxStages = 8;
constexpr int kWinDil = 2;             // largest dilation of k_conv_win (its windows and weights fit)
constexpr int kFirstSmem = 2 * (128 * 128 + 64 * 128) + 1024;  // k_conv_first's two stages
constexpr int kConvSmem = 224 * 1024;  // stages, without the alignment slack

// one accumulator row (tensor-memory address src, the calling warp's lanes) to
// pixel m of the output: bias, ReLU or ReLU mask, BF16; the last layer (N =
// 16): bias, 8 FP32 channels
template <int N>
__device__ __forceinline__ void conv_output(const ConvArgs& a, uint32_t src, long long m)
{
#pragma unroll
    for (int c0 = 0; c0 < N; c0 += 16) {
        uint32_t v[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
              "=r"(v[15])
            : "r"(src + (uint32_t)c0));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        if constexpr (N == 16) {  // the last layer: 8 FP32 channels
            float f[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) f[j] = __uint_as_float(v[j]) + a.bias[j];
            float4* dst = reinterpret_cast<float4*>(a.y32 + m * kCout);
            dst[0] = make_float4(f[0], f[1], f[2], f[3]);
            dst[1] = make_float4(f[4], f[5], f[6], f[7]);
        } else {
            uint32_t packed[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float f0 = __uint_as_float(v[2 * j]), f1 = __uint_as_float(v[2 * j + 1]);
                if (a.bias) {
                    f0 += a.bias[c0 + 2 * j];
                    f1 += a.bias[c0 + 2 * j + 1];
                }
                if (a.relu) {
                    f0 = fmaxf(f0, 0.f);
                    f1 = fmaxf(f1, 0.f);
                }
                __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
                packed[j] = *reinterpret_cast<uint32_t*>(&h);
            }
            if (a.mask) relu_mask16(packed, a.mask + m * N + c0);
            uint4* dst = reinterpret_cast<uint4*>(a.y + m * N + c0);
            dst[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
            dst[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
        }
    }
}

// the (tap, channel block) steps of a tile in order, both for the loads and for
// the MMAs: f(tap, cb, window y, window x); stops when f returns false
template <int WH, typename F>
__device__ __forceinline__ bool conv_steps(const ConvArgs& a, int y0, int x0, F f)
{
    for (int tap = 0; tap < 9; ++tap) {
        const int y = y0 + (tap / 3 - 1) * a.dil, x = x0 + (tap % 3 - 1) * a.dil;
        if (y >= a.H || y + WH <= 0 || x >= a.W || x + 16 <= 0) continue;
        for (int cb = 0; cb < a.cblocks; ++cb)
            if (!f(tap, cb, y, x)) return false;
    }
    return true;
}

template <int N, int MT>
__global__ void __launch_bounds__(ConvWs<N, MT>::THREADS, 1) k_conv(const __grid_constant__ CUtensorMap ta,
                                                                    const __grid_constant__ CUtensorMap tw,
                                                                    ConvArgs a, int* err)
{
    using C = ConvWs<N, MT>;
    constexpr int WH = C::WH, A_BYTES = WH * 2048, STAGE = A_BYTES + N * 128;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    __shared__ uint64_t full[kConvMaxStages], empty[kConvMaxStages], tfull[2], tempty[2];
    __shared__ uint32_t tmem_base;
    __shared__ int s_issued, s_consumed;
    const int tid = threadIdx.x, warp = warp_index(), S = a.stages;
    const int tiles_x = a.W / 16, per_img = tiles_x * (a.H / WH);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         smem_u32(&tmem_base)),
                     "r"(C::COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&full[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&empty[s])));
        }
        for (int k = 0; k < 2; ++k) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&tfull[k])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(&tempty[k])), "r"(128 * MT));
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n");
        s_issued = s_consumed = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = tmem_base;
    bool ok = true;
    if (warp == 0) {
        // producer
        const uint64_t pa = reinterpret_cast<uint64_t>(&ta), pw = reinterpret_cast<uint64_t>(&tw);
        int k = 0;
        for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x) {
            const int b = t / per_img, r = t - b * per_img;
            const int y0 = (r / tiles_x) * WH, x0 = (r - (r / tiles_x) * tiles_x) * 16;
            ok = conv_steps<WH>(a, y0, x0, [&](int tap, int cb, int y, int x) {
                const int s = k % S;
                // slot s was last read by the MMAs of step k - S
                if (k >= S && !warp_wait(smem_u32(&empty[s]), ((k / S) - 1) & 1, err, a.spin)) return false;
                const uint32_t sa = sbase + s * STAGE, bar = smem_u32(&full[s]);
                ++k;
                if (!elect_one()) return true;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(STAGE)
                             : "memory");
                asm volatile(
                    "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
                    "%4, %5}], [%6];\n" ::"r"(sa),
                    "l"(pa), "r"(cb * 64), "r"(x), "r"(y), "r"(b), "r"(bar)
                    : "memory");
                asm volatile(
                    "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
                    "[%4];\n" ::"r"(sa + A_BYTES),
                    "l"(pw), "r"(tap * a.kc + cb * 64), "r"(0), "r"(bar)
                    : "memory");
                return true;
            });
        }
        if (tid == 0) s_issued = k;
    } else if (warp == 1) {
        // MMA issuer (the whole warp; the same lane is elected throughout)
        const uint32_t idesc = umma_idesc(128, N);
        int k = 0, i = 0;
        for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x, ++i) {
            const int b = t / per_img, r = t - b * per_img;
            const int y0 = (r / tiles_x) * WH, x0 = (r - (r / tiles_x) * tiles_x) * 16;
            const int buf = i & 1;
            if (i >= 2 && !(ok = warp_wait(smem_u32(&tempty[buf]), ((i >> 1) - 1) & 1, err, a.spin))) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            const uint32_t d = tmem + (uint32_t)(buf * MT * N);
            uint32_t acc = 0u;
            ok = conv_steps<WH>(a, y0, x0, [&](int, int, int, int) {
                const int s = k % S;
                if (!warp_wait(smem_u32(&full[s]), (k / S) & 1, err, a.spin)) return false;
                asm volatile("tcgen05.fence::after_thread_sync;\n");
                const uint32_t al = desc_lo(sbase + s * STAGE, 16), bl = al + A_BYTES / 16;
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)  // 16 channels: 32 bytes of the swizzled rows
#pragma unroll
                        for (int m = 0; m < MT; ++m)
                            umma(d + (uint32_t)(m * N), al + m * (128 * 128 / 16) + ks * 2, bl + ks * 2, idesc,
                                 ks > 0 ? 1u : acc);
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                        smem_u32(&empty[s])));
                }
                __syncwarp();
                acc = 1u;
                ++k;
                return true;
            });
            if (ok && elect_one())
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(&tfull[buf])));
            __syncwarp();
        }
        if (tid == 32) s_consumed = k;
    } else if (warp >= 2) {
        // output: warp w reads lanes 32 (w % 4) .. of accumulator (w - 2) / 4;
        // accumulator row r of window q is the pixel (y0 + 8 q + r / 16, x0 + r % 16)
        const int q = (warp - 2) >> 2, r = ((warp & 3) << 5) + (tid & 31);
        const uint32_t lane = ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(q * N);
        int i = 0;
        for (int t = blockIdx.x; t < a.tiles; t += gridDim.x, ++i) {
            const int buf = i & 1;
            // the whole warp goes on or gives up (the loads below are warp-collective)
            const bool w = mbar_wait(smem_u32(&tfull[buf]), (i >> 1) & 1, err, a.spin);
            ok = __all_sync(0xffffffffu, w ? 1 : 0) != 0;
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            const int b = t / per_img, rr = t - b * per_img;
            const int y0 = (rr / tiles_x) * WH, x0 = (rr - (rr / tiles_x) * tiles_x) * 16;
            const long long m = ((long long)b * a.H + y0 + 8 * q + (r >> 4)) * a.W + x0 + (r & 15);
            const uint32_t src = tmem + lane + (uint32_t)(buf * MT * N);
            conv_output<N>(a, src, m);
            asm volatile("tcgen05.fence::before_thread_sync;\n");
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&tempty[buf])) : "memory");
        }
    }
    const bool all_ok = __syncthreads_and(ok ? 1 : 0) != 0;
    if (!all_ok && tid == 0) {
        // a wait gave up: let the loads this CTA issued and no MMA consumed land
        // before the shared memory is released, and the MMAs finish before the
        // tensor memory is (the default bound; commits arrive in issue order)
        for (int k = s_consumed; k < s_issued; ++k) mbar_wait(smem_u32(&full[k % S]), (k / S) & 1, err);
        const int nc = s_consumed;
        if (nc >= 1) mbar_wait(smem_u32(&empty[(nc - 1) % S]), ((nc - 1) / S) & 1, err);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(C::COLS));
}

// The same for 64 input channels and dilations 1 and 2, where a tile of 8 x 16
// pixels shares most of its taps' pixels: the tile's three windows (one per tap
// column, 8 + 2 dil rows of 16 pixels; a row is 2 KB, so the taps of a column
// are 1024-byte aligned offsets of its window) are loaded once, two tiles'
// worth of windows deep, and all nine taps' weights stay in shared memory for
// the whole launch.  A tile then takes 60 or 72 KB from L2 instead of 9 x (16 +
// N / 8) KB.  The taps are summed in k_conv's order.
// Measured, 64 problems, cold: 64 -> 64 channels 46 us and the last layer 43 us
// on k_conv, 32 and 27 here.
template <int N>
__global__ void __launch_bounds__(192, 1) k_conv_win(const __grid_constant__ CUtensorMap ta,
                                                     const __grid_constant__ CUtensorMap tw, ConvArgs a, int* err)
{
    constexpr int WH = 8, SLOTS = 6, B_BYTES = N * 128, COLS = 2 * N;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t wbase = (smem_u32(smem_raw) + 1023u) & ~1023u, sbase = wbase + 9 * B_BYTES;
    __shared__ uint64_t full[SLOTS], empty[SLOTS], tfull[2], tempty[2], wfull, done;
    __shared__ uint32_t tmem_base;
    __shared__ int s_issued, s_landed, s_mma;
    const int tid = threadIdx.x, warp = warp_index();
    const int tiles_x = a.W / 16, per_img = tiles_x * (a.H / WH);
    const int win = (WH + 2 * a.dil) * 2048;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         smem_u32(&tmem_base)),
                     "r"(COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        for (int s = 0; s < SLOTS; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&full[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&empty[s])));
        }
        for (int k = 0; k < 2; ++k) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&tfull[k])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 128;\n" ::"r"(smem_u32(&tempty[k])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&wfull)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&done)));
        asm volatile("fence.mbarrier_init.release.cluster;\n");
        s_issued = s_landed = s_mma = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = tmem_base;
    bool ok = true;
    if (warp == 0) {
        // producer: the weights, then three windows per tile
        const uint64_t pa = reinterpret_cast<uint64_t>(&ta), pw = reinterpret_cast<uint64_t>(&tw);
        if (elect_one()) {
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(&wfull)),
                         "r"(9 * B_BYTES)
                         : "memory");
            for (int tap = 0; tap < 9; ++tap)
                asm volatile(
                    "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
                    "[%4];\n" ::"r"(wbase + tap * B_BYTES),
                    "l"(pw), "r"(tap * 64), "r"(0), "r"(smem_u32(&wfull))
                    : "memory");
        }
        __syncwarp();
        int w = 0;
        for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x) {
            const int b = t / per_img, r = t - b * per_img;
            const int y0 = (r / tiles_x) * WH, x0 = (r - (r / tiles_x) * tiles_x) * 16;
            for (int kx = 0; kx < 3; ++kx, ++w) {
                const int s = w % SLOTS;
                // slot s was last read by the MMAs of window w - SLOTS
                if (w >= SLOTS && !(ok = warp_wait(smem_u32(&empty[s]), ((w / SLOTS) - 1) & 1, err, a.spin))) break;
                const uint32_t bar = smem_u32(&full[s]);
                if (!elect_one()) continue;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(win)
                             : "memory");
                asm volatile(
                    "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
                    "%4, %5}], [%6];\n" ::"r"(sbase + s * win),
                    "l"(pa), "r"(0), "r"(x0 + (kx - 1) * a.dil), "r"(y0 - a.dil), "r"(b), "r"(bar)
                    : "memory");
            }
        }
        __syncwarp();
        if (tid == 0) s_issued = w;
    } else if (warp == 1) {
        // MMA issuer
        const uint32_t idesc = umma_idesc(128, N);
        int w0 = 0, i = 0, landed = 0, mma = 0;
        ok = warp_wait(smem_u32(&wfull), 0, err, a.spin);
        for (int t = blockIdx.x; t < a.tiles && ok; t += gridDim.x, ++i, w0 += 3) {
            const int buf = i & 1;
            if (i >= 2 && !(ok = warp_wait(smem_u32(&tempty[buf]), ((i >> 1) - 1) & 1, err, a.spin))) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            const uint32_t d = tmem + (uint32_t)(buf * N);
            for (int tap = 0; tap < 9 && ok; ++tap) {
                const int ky = tap / 3, kx = tap - 3 * ky, w = w0 + kx, s = w % SLOTS;
                if (ky == 0) {
                    if (!(ok = warp_wait(smem_u32(&full[s]), (w / SLOTS) & 1, err, a.spin))) break;
                    landed = w + 1;
                    asm volatile("tcgen05.fence::after_thread_sync;\n");
                }
                const uint32_t al = desc_lo(sbase + s * win, 16) + ky * a.dil * (2048 / 16);
                const uint32_t bl = desc_lo(wbase + tap * B_BYTES, 16);
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        umma(d, al + ks * 2, bl + ks * 2, idesc, (tap > 0 || ks > 0) ? 1u : 0u);
                    if (ky == 2)
                        asm volatile(
                            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                                smem_u32(&empty[s])));
                }
                __syncwarp();
                mma = 1;
            }
            if (ok && elect_one())
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(&tfull[buf])));
            __syncwarp();
        }
        if (mma && elect_one())
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                smem_u32(&done)));
        __syncwarp();
        if (tid == 32) {
            s_landed = landed;
            s_mma = mma;
        }
    } else if (warp >= 2) {
        const int r = ((warp & 3) << 5) + (tid & 31);
        const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;
        int i = 0;
        for (int t = blockIdx.x; t < a.tiles; t += gridDim.x, ++i) {
            const int buf = i & 1;
            const bool w = mbar_wait(smem_u32(&tfull[buf]), (i >> 1) & 1, err, a.spin);
            ok = __all_sync(0xffffffffu, w ? 1 : 0) != 0;  // the loads below are warp-collective
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            const int b = t / per_img, rr = t - b * per_img;
            const int y0 = (rr / tiles_x) * WH, x0 = (rr - (rr / tiles_x) * tiles_x) * 16;
            conv_output<N>(a, tmem + lane + (uint32_t)(buf * N),
                           ((long long)b * a.H + y0 + (r >> 4)) * a.W + x0 + (r & 15));
            asm volatile("tcgen05.fence::before_thread_sync;\n");
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&tempty[buf])) : "memory");
        }
    }
    const bool all_ok = __syncthreads_and(ok ? 1 : 0) != 0;
    if (!all_ok && tid == 0) {
        // a wait gave up: the loads land and the MMAs finish before the memories
        // are released (the default bound)
        mbar_wait(smem_u32(&wfull), 0, err);
        for (int w = s_landed; w < s_issued; ++w) mbar_wait(smem_u32(&full[w % SLOTS]), (w / SLOTS) & 1, err);
        if (s_mma) mbar_wait(smem_u32(&done), 0, err);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(COLS));
}

// The first layer (40 channels): im2col rows of the 360 features of a pixel
// staged by cp.async in 64-wide K tiles that run across taps, two stages deep,
// one CTA of 128 threads per 128 output pixels.  (On k_conv with the channels
// padded to 64 the K tiles would fall differently and the stored BF16
// activations would round differently.)  Bound by the 16-byte copies, 1536 a K
// tile with their bounds: 60 us for 64 problems, the same with loads two tiles
// ahead of the MMAs.  As in k_conv every wait is bounded; the decision to give
// up is the block's.
__device__ __forceinline__ uint32_t sw128(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }

__global__ void __launch_bounds__(128) k_conv_first(ConvArgs a, const bf16* __restrict__ x,
                                                      const bf16* __restrict__ wk, int* err)
{
    constexpr int N = 64, Cin = kCin, K = 9 * kCin;
    constexpr int BK = 64, A_BYTES = 128 * 128, B_BYTES = N * 128, STAGE = A_BYTES + B_BYTES;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    __shared__ uint64_t mbar[2];
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int HW = a.H * a.W;
    const long long M = (long long)a.B * HW, m0 = (long long)blockIdx.x * 128;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         smem_u32(&tmem_base)),
                     "r"(N));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar[0])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar[1])));
        asm volatile("fence.mbarrier_init.release.cluster;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = tmem_base;
    // this thread stages the 16-byte K chunk c of the rows r = tid/8 + 16 i
    const int c = tid & 7, r0 = tid >> 3;
    int pb[8], py[8], px[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        long long m = m0 + r0 + 16 * i;
        if (m < M) {
            int b = (int)(m / HW), rem = (int)(m - (long long)b * HW);
            pb[i] = b;
            py[i] = rem / a.W;
            px[i] = rem - py[i] * a.W;
        } else {
            pb[i] = -1;
            py[i] = px[i] = 0;
        }
    }
    const int nk = (K + BK - 1) / BK;
    bool ok = true;
    int issued = 0;  // steps whose MMAs were issued and committed
    for (int kt = 0; kt < nk; ++kt) {
        const int st = kt & 1;
        if (kt >= 2) {
            // the stage's previous MMAs (step kt - 2) must be done; the block decides together
            const bool w = mbar_wait(smem_u32(&mbar[st]), ((kt - 2) >> 1) & 1, err, a.spin);
            ok = __syncthreads_and(w ? 1 : 0) != 0;
            if (!ok) break;
        }
        const uint32_t sa = sbase + st * STAGE, sb = sa + A_BYTES;
        const int k = kt * BK + c * 8;
        const bool kin = k < K;
        const int tap = kin ? k / Cin : 0, ci = k - tap * Cin;
        const int dy = (tap / 3 - 1) * a.dil, dx = (tap % 3 - 1) * a.dil;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = r0 + 16 * i;
            const int yy = py[i] + dy, xx = px[i] + dx;
            const bool in = kin && pb[i] >= 0 && yy >= 0 && yy < a.H && xx >= 0 && xx < a.W;
            const bf16* src = in ? x + (((long long)pb[i] * a.H + yy) * a.W + xx) * Cin + ci : x;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa + sw128(r, c)), "l"(src),
                         "r"(in ? 16 : 0));
        }
#pragma unroll
        for (int i = 0; i < N / 16; ++i) {
            const int r = r0 + 16 * i;  // output channel
            const bf16* src = kin ? wk + (long long)r * K + k : wk;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sb + sw128(r, c)), "l"(src),
                         "r"(kin ? 16 : 0));
        }
        asm volatile("cp.async.commit_group;\n");
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            const uint32_t idesc = umma_idesc(128, N), al = desc_lo(sa, 16), bl = desc_lo(sb, 16);
#pragma unroll
            for (int ks = 0; ks < BK / 16; ++ks)
                umma(tmem, al + ks * 2, bl + ks * 2, idesc, (kt > 0 || ks > 0) ? 1u : 0u);
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                smem_u32(&mbar[st])));
        }
        issued = kt + 1;
        __syncthreads();
    }
    // the last commit arrives once every MMA the thread issued is done
    if (issued >= 1) {
        const uint32_t bar = smem_u32(&mbar[(issued - 1) & 1]), par = ((issued - 1) >> 1) & 1;
        bool w = ok && mbar_wait(bar, par, err, a.spin);
        if (!w) mbar_wait(bar, par, err);  // gave up: let the MMAs finish before the memory is freed
        ok = __syncthreads_and((ok && w) ? 1 : 0) != 0;
    }
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    if (ok) {
        const long long m = m0 + tid;  // accumulator row = tensor-memory lane
        const uint32_t lane = (uint32_t)(warp * 32) << 16;
#pragma unroll
        for (int c0 = 0; c0 < N; c0 += 16) {
            uint32_t v[16];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
                : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                  "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                  "=r"(v[15])
                : "r"(tmem + lane + (uint32_t)c0));
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
            if (m < M) {
                uint32_t packed[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    float f0 = __uint_as_float(v[2 * j]), f1 = __uint_as_float(v[2 * j + 1]);
                    if (a.bias) {
                        f0 += a.bias[c0 + 2 * j];
                        f1 += a.bias[c0 + 2 * j + 1];
                    }
                    if (a.relu) {
                        f0 = fmaxf(f0, 0.f);
                        f1 = fmaxf(f1, 0.f);
                    }
                    __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
                    packed[j] = *reinterpret_cast<uint32_t*>(&h);
                }
                uint4* dst = reinterpret_cast<uint4*>(a.y + m * N + c0);
                dst[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
                dst[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(N));
}

// ------------------------------------------------ weight gradient (tcgen05)
// dW[tap][ci][co] = sum over pixels p of x[p + tap][ci] dy[p][co].  The
// reduction runs over pixels, so both operands are MN-major as they lie in
// memory (NHWC: a pixel's channels are contiguous): one TMA load brings 64
// channels of 64 pixels (a 4 x 16 window, shifted by the tap's offset for x;
// the image border and the channels past Cin come as zero fill) as a
// 64-row x 128-byte plane in the 128-byte swizzle, which is the MN-major
// operand layout as it stands: 64 channels along a row, 8 pixels per swizzle
// group (groups 1024 bytes apart: the stride offset), the next 64 channels a
// plane further (the leading offset).
// Two planes make one M = 128 operand: the two channel halves of a tap where
// Cin = 128, two taps where Cin <= 64.  A CTA holds the accumulators of G such
// pairs in tensor memory and walks its share of the pixel windows, each dy tile
// serving all G pairs; partial sums per CTA are reduced in a fixed order
// afterwards, so the gradient is deterministic.  What bounds it is the planes'
// traffic from L2: (2 G + N / 64) 8 KB per 4 G MMAs of 128 x N x 16.
// Measured for a 64-problem batch: 128 -> 128 channels 672 us on mma.sync, 80
// us here at dilation 8 (0.96 PFLOP/s); 64 -> 64 channels 201 -> 38 us.  The
// bias sums came from a pass of their own (176 us per layer); here two idle warps
// add them up from the staged dy tiles.
struct WgradArgs {
    int B, H, W, Cin, Cout, dil;
    float* part;       // [splits][9 Cin][Cout]
    float* bpart;      // [splits][Cout] sums of dy (the bias gradient)
    int G;             // operand pairs of a CTA (blockIdx.y: its first pair / G)
    int npair;         // pairs in all: 9 (Cin = 128) or 5 (Cin <= 64, the tenth plane unused)
    int tiles;         // pixel windows in all
    int per;           // windows of a split (blockIdx.x)
    int stages;
    long long spin;
};

constexpr int kWgPlane = 64 * 128;    // bytes of a plane: 64 pixels x 64 channels
constexpr int kWgThreads = 128;
constexpr int kWgMaxStages = 8;
constexpr int kWgSmem = 216 * 1024;   // stages, without the alignment slack

// the order in which 128-channel inputs' taps are dealt to the CTA groups:
// every three in a row hold one tap of each kernel row and column, so that the
// windows left out at the image's border are spread evenly
__device__ __forceinline__ int wgrad_tap(int i) { return (int)((0x642831750ull >> (4 * i)) & 15u); }

template <int N>
__global__ void __launch_bounds__(kWgThreads, 1) k_wgrad_tc(const __grid_constant__ CUtensorMap tx,
                                                            const __grid_constant__ CUtensorMap ty, WgradArgs a,
                                                            int tmem_cols, int* err)
{
    constexpr int NB = N / 64;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    __shared__ uint64_t full[kWgMaxStages], empty[kWgMaxStages], done;
    __shared__ uint32_t tmem_base;
    __shared__ int consumed, used;
    __shared__ float sbias[128];
    const bool bias = blockIdx.y == 0;  // these CTAs' warps 2 and 3 sum dy from its staged tiles
    const int tid = threadIdx.x, warp = warp_index(), S = a.stages;
    const int g0 = blockIdx.y * a.G, ng = min(a.G, a.npair - g0);
    const int t0 = blockIdx.x * a.per, t1 = min(t0 + a.per, a.tiles), nk = max(t1 - t0, 0);
    const int stage = (2 * a.G + NB) * kWgPlane;
    const int tiles_x = a.W / 16, per_img = tiles_x * (a.H / 4);
    const bool wide = a.Cin > 64;
    // the pairs with a tap whose window meets the image (the others' x is all
    // zero fill): at dilations 16 and 32 a good part of the windows drop out
    auto live = [&](int y0, int x0) -> unsigned {
        // dilations up to 4: only the windows of the image's first and last 4 rows
        // at dilation 4 miss it, 3 taps of 9 each, and zero fill makes them right
        if (!wide) return (1u << ng) - 1u;
        unsigned mk = 0u;
        for (int g = 0; g < ng; ++g) {
            const int tap = wgrad_tap(g0 + g), y = y0 + (tap / 3 - 1) * a.dil, x = x0 + (tap % 3 - 1) * a.dil;
            if (y < a.H && y + 4 > 0 && x < a.W && x + 16 > 0) mk |= 1u << g;
        }
        return mk;
    };
    // the windows of the split in order (y0, x0, image), without divisions
    int b = t0 / per_img, y0 = (t0 - b * per_img) / tiles_x * 4, x0 = (t0 - b * per_img) % tiles_x * 16;
    auto next_window = [&]() {
        if ((x0 += 16) < a.W) return;
        x0 = 0;
        if ((y0 += 4) < a.H) return;
        y0 = 0;
        ++b;
    };
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         smem_u32(&tmem_base)),
                     "r"(tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&full[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(&empty[s])), "r"(bias ? 3 : 1));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&done)));
        asm volatile("fence.mbarrier_init.release.cluster;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = tmem_base;
    bool ok = true;
    int issued = 0;
    if (warp == 0) {
        // producer warp: a lane per plane, so that a stage's loads go out together
        // (one thread issuing all of them kept the MMAs waiting)
        const int q = tid;
        const bool isx = q < 2 * ng, mine = q < 2 * ng + NB;
        int c = (q - 2 * ng) * 64, dx = 0, dy = 0;
        if (isx) {
            const int p = 2 * g0 + q;  // plane: (tap, half) or tap
            const int tap = wide ? wgrad_tap(p >> 1) : min(p, 8);
            c = wide ? (p & 1) * 64 : 0;
            dy = (tap / 3 - 1) * a.dil;
            dx = (tap % 3 - 1) * a.dil;
        }
        const uint64_t map = isx ? reinterpret_cast<uint64_t>(&tx) : reinterpret_cast<uint64_t>(&ty);
        const uint32_t off = (isx ? q : 2 * a.G + q - 2 * ng) * kWgPlane;
        for (int k = 0; k < nk; ++k) {
            const int s = k % S;
            const uint32_t bar = smem_u32(&full[s]);
            const unsigned mk = live(y0, x0);
            if (q == 0) {
                if (k >= S) ok = mbar_wait(smem_u32(&empty[s]), ((k / S) - 1) & 1, err, a.spin);
                if (ok)
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar),
                                 "r"((2 * __popc(mk) + NB) * kWgPlane)
                                 : "memory");
            }
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            if (!ok) break;
            if (mine && (!isx || ((mk >> (q >> 1)) & 1u)))
                asm volatile(
                    "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
                    "%4, %5}], [%6];\n" ::"r"(sbase + s * stage + off),
                    "l"(map), "r"(c), "r"(x0 + dx), "r"(y0 + dy), "r"(b), "r"(bar)
                    : "memory");
            issued = k + 1;
            next_window();
        }
    } else if (warp == 1) {
        // FP32 accumulator, BF16 operands, both MN-major
        const uint32_t idesc = umma_idesc(128, N) | (1u << 15) | (1u << 16);
        unsigned have = 0u;  // pairs accumulated into
        int k = 0;
        for (; k < nk; ++k) {
            const int s = k % S;
            const unsigned mk = live(y0, x0);
            next_window();
            if (!(ok = warp_wait(smem_u32(&full[s]), (k / S) & 1, err, a.spin))) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            const uint32_t al = desc_lo(sbase + s * stage, kWgPlane);
            const uint32_t bl = desc_lo(sbase + s * stage + 2 * a.G * kWgPlane, kWgPlane);
            if (elect_one()) {
                for (int g = 0; g < ng; ++g) {
                    if (!((mk >> g) & 1u)) continue;
                    const uint32_t first = (have >> g) & 1u;
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)  // 16 pixels each
                        umma(tmem + (uint32_t)(g * N), al + (2 * g * kWgPlane + ks * 2048) / 16, bl + ks * (2048 / 16),
                             idesc, ks > 0 ? 1u : first);
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                    smem_u32(&empty[s])));
            }
            __syncwarp();
            have |= mk;
        }
        if (k > 0 && elect_one())
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                smem_u32(&done)));
        __syncwarp();
        if (tid == 32) {
            consumed = k;
            used = (int)have;
        }
    } else if (warp >= 2 && bias) {
        // two channels a lane: warp w takes dy plane w - 2 (N = 128) or half of
        // the rows of the one plane
        constexpr int ROWS = NB == 2 ? 64 : 32;
        const int lane = tid & 31, plane = NB == 2 ? warp - 2 : 0, row0 = NB == 2 ? 0 : (warp - 2) * 32;
        float s0 = 0.f, s1 = 0.f;
        for (int k = 0; k < nk; ++k) {
            const int s = k % S;
            const bool w = mbar_wait(smem_u32(&full[s]), (k / S) & 1, err, a.spin);
            ok = __all_sync(0xffffffffu, w ? 1 : 0) != 0;
            if (!ok) break;
            const uint32_t base = sbase + s * stage + (2 * a.G + plane) * kWgPlane + (lane & 3) * 4;
            float w0 = 0.f, w1 = 0.f;  // a window's sum first: chains of ROWS and of the windows
#pragma unroll 8
            for (int r = row0; r < row0 + ROWS; ++r) {
                uint32_t v;
                asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(base + r * 128 + (((lane >> 2) ^ (r & 7)) << 4)));
                w0 += __uint_as_float(v << 16);
                w1 += __uint_as_float(v & 0xffff0000u);
            }
            s0 += w0;
            s1 += w1;
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&empty[s])) : "memory");
        }
        sbias[(warp - 2) * 64 + 2 * lane] = s0;
        sbias[(warp - 2) * 64 + 2 * lane + 1] = s1;
    }
    const bool all_ok = __syncthreads_and(ok ? 1 : 0) != 0;
    if (!all_ok && tid == 0) {
        // a wait gave up: let the loads this CTA issued and no MMA consumed land
        for (int k = consumed; k < issued; ++k) mbar_wait(smem_u32(&full[k % S]), (k / S) & 1, err);
    }
    ok = all_ok;
    const int nc = consumed;
    if (nc >= 1) {  // every MMA issued has finished
        bool w = ok && mbar_wait(smem_u32(&done), 0, err, a.spin);
        if (!w) mbar_wait(smem_u32(&done), 0, err);
        ok = __syncthreads_and((ok && w) ? 1 : 0) != 0;
    }
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    if (ok) {
        // accumulator row m of pair g: channel m of the tap (Cin = 128), or
        // channel m % 64 of tap 2 g + m / 64
        const int m = tid;
        const uint32_t lane = (uint32_t)(warp * 32) << 16;
        if (bias && tid < N) a.bpart[(size_t)blockIdx.x * N + tid] = sbias[tid] + (NB == 1 ? sbias[tid + 64] : 0.f);
        for (int g = 0; g < ng; ++g) {
            const int p = 2 * (g0 + g) + (m >> 6), tap = wide ? wgrad_tap(g0 + g) : p, ci = wide ? m : m & 63;
            const bool out = tap < 9 && ci < a.Cin;
            float* dst = a.part + ((size_t)blockIdx.x * 9 * a.Cin + (size_t)tap * a.Cin + ci) * N;
#pragma unroll
            for (int c0 = 0; c0 < N; c0 += 16) {
                uint32_t v[16];
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                      "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                      "=r"(v[15])
                    : "r"(tmem + lane + (uint32_t)(g * N + c0)));
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                if (out) {
                    uint4* d4 = reinterpret_cast<uint4*>(dst + c0);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        d4[j] = ((used >> g) & 1) ? make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3])
                                       : make_uint4(0u, 0u, 0u, 0u);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(tmem_cols));
}

// -------------------------------------------- the last layer's backward pass
// Only channel 0 of the output enters the loss, so the output gradient is one
// value per pixel (dy0) and both gradients of the 64 -> 8 layer are sums over
// 9 taps of a scalar times 64 channels: bound by reading and writing the 64
// channels once, not by arithmetic, and no tensor core is needed (161 us for
// the weight gradient on mma.sync and 49 us for the data gradient as a tcgen05
// convolution with 8 input channels, before the ReLU pass; 33 and 30 us here
// with the ReLU mask included, 64 problems).
constexpr int kLastBlocks = 608;

// The 9 neighbours dy0[p + dir * shift] of pixel p = (r, c), 0 outside the image
__device__ __forceinline__ void last_taps(const bf16* __restrict__ dy0, long long p, int r, int c, int H, int W,
                                          int dir, float (&d)[9])
{
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
        const int dr = dir * (tap / 3 - 1), dc = dir * (tap % 3 - 1);
        const bool in = (unsigned)(r + dr) < (unsigned)H && (unsigned)(c + dc) < (unsigned)W;
        d[tap] = in ? __bfloat162float(dy0[p + dr * W + dc]) : 0.f;
    }
}

// dx[p][ci] = sum_tap dy0[p + shift] w[8 - tap][ci] where act > 0, else 0 (w: the
// weights of output channel 0); a thread takes 8 channels of every 32nd pixel
// of the block's run, their 72 weights in registers
__global__ void __launch_bounds__(256) k_last_dgrad(const bf16* __restrict__ dy0, const bf16* __restrict__ w,
                                                    const bf16* __restrict__ act, long long M, int H, int W,
                                                    bf16* __restrict__ dx)
{
    const int cg = (threadIdx.x & 7) * 8, HW = H * W;
    float wr[9][8];
#pragma unroll
    for (int tap = 0; tap < 9; ++tap)
#pragma unroll
        for (int j = 0; j < 8; ++j) wr[tap][j] = __bfloat162float(w[(8 - tap) * 64 + cg + j]);
    const long long chunk = ((M + gridDim.x - 1) / gridDim.x + 31) / 32 * 32;
    const long long p0 = blockIdx.x * chunk, p1 = p0 + chunk < M ? p0 + chunk : M;
    for (long long p = p0 + (threadIdx.x >> 3); p < p1; p += 32) {
        const uint4 av = *reinterpret_cast<const uint4*>(act + p * 64 + cg);
        const int rem = (int)(p % HW), r = rem / W, c = rem - r * W;
        float d[9], acc[8] = {};
        last_taps(dy0, p, r, c, H, W, 1, d);
#pragma unroll
        for (int tap = 0; tap < 9; ++tap)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] = fmaf(d[tap], wr[tap][j], acc[j]);
        const bf16* ab = reinterpret_cast<const bf16*>(&av);
        uint4 ov;
        bf16* ob = reinterpret_cast<bf16*>(&ov);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            ob[j] = __bfloat162float(ab[j]) > 0.f ? __float2bfloat16(acc[j]) : __float2bfloat16(0.f);
        *reinterpret_cast<uint4*>(dx + p * 64 + cg) = ov;
    }
}

// block partials of dW[tap][ci][0] = sum_q x[q][ci] dy0[q - shift] (577 per
// block: the last is the sum of dy0, the bias gradient); a block takes a run of
// pixels, a thread 8 channels of every 32nd pixel
__global__ void __launch_bounds__(256) k_last_wgrad(const bf16* __restrict__ x, const bf16* __restrict__ dy0,
                                                    long long M, int H, int W, float* __restrict__ part)
{
    const int cgi = threadIdx.x & 7, cg = cgi * 8, pl = threadIdx.x >> 3, HW = H * W;
    const long long chunk = ((M + gridDim.x - 1) / gridDim.x + 31) / 32 * 32;
    const long long p0 = blockIdx.x * chunk, p1 = p0 + chunk < M ? p0 + chunk : M;
    float acc[9][8] = {};
    float bs = 0.f;
#pragma unroll 2
    for (long long p = p0 + pl; p < p1; p += 32) {
        const uint4 xv = *reinterpret_cast<const uint4*>(x + p * 64 + cg);
        const int rem = (int)(p % HW), r = rem / W, c = rem - r * W;
        float d[9];
        last_taps(dy0, p, r, c, H, W, -1, d);
        const bf16* xb = reinterpret_cast<const bf16*>(&xv);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float xf = __bfloat162float(xb[j]);
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) acc[tap][j] = fmaf(d[tap], xf, acc[tap][j]);
        }
        bs += d[4];
    }
    // over the warp's 4 pixels, then over the 8 warps
    __shared__ float red[8][577];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int tap = 0; tap < 9; ++tap)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float v = acc[tap][j];
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            if (lane < 8) red[warp][tap * 64 + cg + j] = v;
        }
    bs += __shfl_xor_sync(0xffffffffu, bs, 8);
    bs += __shfl_xor_sync(0xffffffffu, bs, 16);
    if (lane == 0) red[warp][576] = bs;
    __syncthreads();
    for (int i = threadIdx.x; i < 577; i += 256) {
        float v = 0.f;
        for (int q = 0; q < 8; ++q) v += red[q][i];
        part[(size_t)blockIdx.x * 577 + i] = v;
    }
}

// the block partials summed into the layer's gradient (channel 0; the other
// channels' gradients are 0): one warp per entry, a fixed order
__global__ void k_last_sum(const float* __restrict__ part, int blocks, float* __restrict__ gw, float* __restrict__ gb)
{
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= 577) return;
    float v = 0.f;
    for (int b = lane; b < blocks; b += 32) v += part[(size_t)b * 577 + i];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    float* dst = i < 576 ? gw + (size_t)i * kCout : gb;
    if (lane < kCout) dst[lane] = lane == 0 ? v : 0.f;
}

// sums over the splits in a fixed order (deterministic): a layer's n weights
// from part[s][i] and, after them, its nb biases from bpart[s][i].  A block
// takes 32 entries in 8 slices of the splits (one thread per entry took 16 us
// for 152 splits)
__global__ void __launch_bounds__(256) k_sum_splits(const float* __restrict__ part, int splits, int n,
                                                    float* __restrict__ grad, const float* __restrict__ bpart, int nb,
                                                    float* __restrict__ gbias)
{
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    const bool w = blockIdx.x * 32 < n;  // n is a multiple of 32
    const float* src = w ? part + i : bpart + (i - n);
    const int stride = w ? n : nb;
    float s = 0.f;
#pragma unroll 4
    for (int q = sl; q < splits; q += 8) s += src[(size_t)q * stride];
    __shared__ float sh[8][32];
    sh[sl][lane] = s;
    __syncthreads();
    if (sl == 0) {
        for (int q = 1; q < 8; ++q) s += sh[q][lane];
        (w ? grad + i : gbias + (i - n))[0] = s;
    }
}

// loss = 1/2 mean over the M cells of (y[p][0] - t[p])^2, dy0[p] = (y - t) / M
// (the gradient of the other channels is 0); per-block partial sums of the
// loss (FP64)
__global__ void k_loss(const float* y32, int C, const float* t, long long M, bf16* dy0, double* part)
{
    long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    double e2 = 0.0;
    if (p < M) {
        float e = y32[p * C] - t[p];
        e2 = 0.5 * (double)e * (double)e;
        dy0[p] = __float2bfloat16(e / (float)M);
    }
    __shared__ double sh[256];
    sh[threadIdx.x] = e2;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// one block of 256 threads (one thread took 63 us for 1024 partials)
__global__ void k_sum_loss(const double* part, int n, long long count, double* loss)
{
    __shared__ double sh[256];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 256) s += part[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = sh[0] / (double)count;
}

struct LayerTab {
    long woff[kLayers], boff[kLayers];
    int cin[kLayers], cout[kLayers];
};

// BF16 copies of one FP32 parameter, both K-major: the forward's weights
// wk[co][tap * Cin + ci] and the flipped, transposed weights of the data
// gradient wtk[ci][k'], k' = (8 - tap) Cout + co
struct WeightCopies {
    bf16 *wk, *wtk;
};

__device__ __forceinline__ void write_copies(long long i, float p, const LayerTab& T, const WeightCopies& w)
{
    for (int l = 0; l < kLayers; ++l) {
        if (i >= T.woff[l] && i < T.boff[l]) {
            long long q = i - T.woff[l];
            int cin = T.cin[l], cout = T.cout[l];
            int co = (int)(q % cout);
            long long k = q / cout;
            int tap = (int)(k / cin), ci = (int)(k % cin);
            long long kp = (long long)(8 - tap) * cout + co;
            const bf16 pb = __float2bfloat16(p);
            w.wk[T.woff[l] + (long long)co * 9 * cin + k] = pb;
            w.wtk[T.woff[l] + (long long)ci * 9 * cout + kp] = pb;
        }
    }
}

// Adam on the FP32 parameters; refreshes the BF16 weight copies
__global__ void k_adam(float* prm, float* m, float* v, const float* grad, long long n, float lr,
                       float b1, float b2, float eps, float c1, float c2, LayerTab T, WeightCopies w)
{
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    float g = grad[i];
    float mi = b1 * m[i] + (1.f - b1) * g, vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    float p = prm[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    prm[i] = p;
    write_copies(i, p, T, w);
}

// the same refresh without an update (after loading parameters)
__global__ void k_refresh(const float* prm, long long n, LayerTab T, WeightCopies w)
{
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    write_copies(i, prm[i], T, w);
}

// scale of every problem: max |u0| over its grid (1 when u0 is NULL or zero);
// one block per problem, max of non-negative doubles through their bit patterns
__global__ void k_scale(const double* u0, double* scale)
{
    const int b = blockIdx.x;
    unsigned long long m = 0ull;
    if (u0)
        for (long long k = threadIdx.x; k < (long long)kN * kN; k += blockDim.x) {
            unsigned long long v = (unsigned long long)__double_as_longlong(fabs(u0[(size_t)b * kN * kN + k]));
            m = v > m ? v : m;
        }
    __shared__ unsigned long long sh[256];
    sh[threadIdx.x] = m;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w && sh[threadIdx.x + w] > sh[threadIdx.x]) sh[threadIdx.x] = sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double v = __longlong_as_double((long long)sh[0]);
        scale[b] = v > 0.0 ? v : 1.0;
    }
}

// features of a batch of 256 x 256 problems, one thread per cell (u0 nullable)
__global__ void k_features(int batch, const double* f, const double* b1, const double* b2,
                           const uint8_t* mask, const double* mu, const double* sigma,
                           const double* u0, const double* scale, bf16* x)
{
    long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= (long long)batch * kHW * kHW) return;
    int b = (int)(q / (kHW * kHW)), rem = (int)(q % (kHW * kHW)), r = rem / kHW, c = rem % kHW;
    double s1 = 0, s2 = 0, sm = 0;
    size_t base = (size_t)b * kN * kN;
    bf16* o = x + q * kCin;
    for (int i = 0; i < kSub; ++i)
        for (int j = 0; j < kSub; ++j) {
            size_t k = base + (size_t)(r * kSub + i) * kN + (c * kSub + j);
            o[i * kSub + j] = __float2bfloat16((float)f[k]);
            o[16 + i * kSub + j] = __float2bfloat16(u0 ? (float)(u0[k] / scale[b]) : 0.f);
            s1 += b1[k];
            s2 += b2[k];
            sm += mask[k];
        }
    const double inv = 1.0 / (kSub * kSub);
    o[32] = __float2bfloat16((float)(s1 * inv));
    o[33] = __float2bfloat16((float)(s2 * inv));
    o[34] = __float2bfloat16((float)((log10(mu[b]) + 2.5) / 1.5));
    o[35] = __float2bfloat16((float)(sigma[b] - 1.0));
    o[36] = __float2bfloat16((float)(sm * inv));
    o[37] = o[38] = o[39] = __float2bfloat16(0.f);
}

// t[b][cell] = cell mean of (u - u0) / s_b, one thread per cell (u0 nullable)
__global__ void k_targets(int batch, const double* u, const double* u0, const double* scale,
                          float* t)
{
    long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= (long long)batch * kHW * kHW) return;
    int b = (int)(q / (kHW * kHW)), rem = (int)(q % (kHW * kHW)), r = rem / kHW, c = rem % kHW;
    size_t base = (size_t)b * kN * kN;
    double sum = 0.0;
    for (int i = 0; i < kSub; ++i)
        for (int j = 0; j < kSub; ++j) {
            size_t k = base + (size_t)(r * kSub + i) * kN + (c * kSub + j);
            sum += u[k] - (u0 ? u0[k] : 0.0);
        }
    t[q] = (float)(sum / (kSub * kSub) / scale[b]);
}

// u = u0 + s * bilinear(y[..][0]) on the interior nodes, 0 elsewhere; cell
// centres at node 4 k + 1.5, clamped at the outer half cells (u0 nullable)
__global__ void k_upsample(const float* y, const double* u0, const double* scale,
                           const uint8_t* ntype, double* u)
{
    long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= (long long)kN * kN) return;
    int r = (int)(q / kN), c = (int)(q % kN);
    if (ntype[q] != adr::kInterior) {
        u[q] = 0.0;
        return;
    }
    double fy = (r - (kSub - 1) * 0.5) / kSub, fx = (c - (kSub - 1) * 0.5) / kSub;
    fy = fy < 0 ? 0 : (fy > kHW - 1 ? kHW - 1 : fy);
    fx = fx < 0 ? 0 : (fx > kHW - 1 ? kHW - 1 : fx);
    int y0 = (int)fy, x0 = (int)fx;
    if (y0 > kHW - 2) y0 = kHW - 2;
    if (x0 > kHW - 2) x0 = kHW - 2;
    double ly = fy - y0, lx = fx - x0;
    auto Y = [&](int rr, int cc) { return (double)y[((size_t)rr * kHW + cc) * kCout]; };
    double v = (1 - ly) * ((1 - lx) * Y(y0, x0) + lx * Y(y0, x0 + 1)) +
               ly * ((1 - lx) * Y(y0 + 1, x0) + lx * Y(y0 + 1, x0 + 1));
    u[q] = (u0 ? u0[q] : 0.0) + (scale ? *scale : 1.0) * v;
}

}  // namespace

// ------------------------------------------------------------------ handle

struct adr_cnn {
    int max_batch = 0, hw = kHW;
    cudaStream_t stream = nullptr;
    long P = 0;
    LayerTab T{};
    float *prm = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr;
    bf16 *wk = nullptr, *wtk = nullptr;
    int* err = nullptr;  // a bounded wait of a tensor-core kernel gave up
    long long spin = 0;  // bound of those waits (adr_cnn_set_wait_limit; 0: default)
    bf16* act[kLayers] = {};  // post-activation outputs of layers 0..6 (bf16)
    float* y32 = nullptr;     // last layer output (fp32) [M][8]
    bf16 *dA = nullptr, *dB = nullptr, *dy0 = nullptr;
    float* spart = nullptr;   // block partials of the bias and last-layer gradients
    int n_sm = 0;
    float* part = nullptr;
    long long part_size = 0;
    double* lpart = nullptr;
    double* loss = nullptr;
    long step = 0;
    std::vector<void*> owned;
};

namespace {

template <typename T>
adr_status cnn_alloc(adr_cnn* c, T** p, size_t n)
{
    void* q = nullptr;
    cudaError_t e = cudaMalloc(&q, n * sizeof(T) + 16);
    if (e != cudaSuccess) {
        adr::set_error(std::string("cudaMalloc failed: ") + cudaGetErrorString(e));
        return ADR_ENOMEM;
    }
    c->owned.push_back(q);
    *p = static_cast<T*>(q);
    return ADR_OK;
}

// the driver's tensor-map encoder, looked up once through the runtime (the
// first caller looks it up, others wait for it: C++'s rule for local statics);
// null when the driver has none
PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder()
{
    static const PFN_cuTensorMapEncodeTiled_v12000 fn = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
        void* q = nullptr;
        cudaDriverEntryPointQueryResult res = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &q, 12000, cudaEnableDefault, &res) ==
                cudaSuccess &&
            res == cudaDriverEntryPointSuccess)
            return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(q);
        cudaGetLastError();
        return nullptr;
    }();
    return fn;
}

// tensor map of an activation [B][H][W][C] with a box of 64 channels x 16 x
// rows pixels, 128-byte swizzle (channels past C and pixels past the image
// read as zero)
bool act_map(CUtensorMap* m, const bf16* x, int B, int H, int W, int C, int rows)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = tmap_encoder();
    if (!enc) return false;
    cuuint64_t d[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
    cuuint64_t st[3] = {(cuuint64_t)C * 2, (cuuint64_t)C * 2 * W, (cuuint64_t)C * 2 * W * H};
    cuuint32_t box[4] = {64, 16, (cuuint32_t)rows, 1}, e[4] = {1, 1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(x), d, st, box, e,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// tensor map of K-major weights [Cout][K] with a box of 64 x n rows (rows past
// Cout read as zero)
bool weight_map(CUtensorMap* m, const bf16* w, int K, int Cout, int n)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = tmap_encoder();
    if (!enc) return false;
    cuuint64_t d[2] = {(cuuint64_t)K, (cuuint64_t)Cout}, st[1] = {(cuuint64_t)K * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)n}, e[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(w), d, st, box, e,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int N, int MT>
adr_status launch_conv_t(const adr_cnn* c, cudaStream_t st, ConvArgs a, const bf16* x, int cin, const bf16* wk,
                         int cout)
{
    constexpr int WH = 8 * MT;
    a.cblocks = cin / 64;
    a.kc = cin;
    constexpr int stage = WH * 2048 + N * 128;
    a.stages = std::min(kConvMaxStages, kConvSmem / stage);
    a.tiles = a.B * (a.H / WH) * (a.W / 16);
    CUtensorMap ta, tw;
    if (!act_map(&ta, x, a.B, a.H, a.W, cin, WH) || !weight_map(&tw, wk, 9 * a.kc, cout, N)) {
        adr::set_error("the driver refused a tensor map of a convolution");
        return ADR_ECUDA;
    }
    k_conv<N, MT><<<std::min(c->n_sm, a.tiles), ConvWs<N, MT>::THREADS, a.stages * stage + 1024, st>>>(ta, tw, a,
                                                                                                      c->err);
    return ADR_OK;
}

template <int N>
adr_status launch_conv_win(const adr_cnn* c, cudaStream_t st, ConvArgs a, const bf16* x, const bf16* wk, int cout)
{
    const int rows = 8 + 2 * a.dil;
    a.tiles = a.B * (a.H / 8) * (a.W / 16);
    CUtensorMap ta, tw;
    if (!act_map(&ta, x, a.B, a.H, a.W, 64, rows) || !weight_map(&tw, wk, 9 * 64, cout, N)) {
        adr::set_error("the driver refused a tensor map of a convolution");
        return ADR_ECUDA;
    }
    const int smem = 6 * rows * 2048 + 9 * N * 128 + 1024;
    k_conv_win<N><<<std::min(c->n_sm, a.tiles), 192, smem, st>>>(ta, tw, a, c->err);
    return ADR_OK;
}

// tiles of 16 x 16 pixels, or of 8 x 16 where the larger ones would leave SMs
// without one (fewer than about 10 problems)
adr_status launch_conv(const adr_cnn* c, cudaStream_t st, const ConvArgs& a, const bf16* x, int cin, const bf16* wk,
                       int cout)
{
    if (cin == 64 && a.dil <= kWinDil && cout <= 64)  // 64 or 8 output channels
        return cout == 64 ? launch_conv_win<64>(c, st, a, x, wk, cout) : launch_conv_win<16>(c, st, a, x, wk, cout);
    const bool big = a.B * (a.H / 16) * (a.W / 16) >= c->n_sm;
    if (cout == 128)
        return big ? launch_conv_t<128, 2>(c, st, a, x, cin, wk, cout) : launch_conv_t<128, 1>(c, st, a, x, cin, wk, cout);
    if (cout == 64)
        return big ? launch_conv_t<64, 2>(c, st, a, x, cin, wk, cout) : launch_conv_t<64, 1>(c, st, a, x, cin, wk, cout);
    adr::set_error("internal: no convolution kernel for this layer");
    return ADR_EINVAL;
}

// forward of a batch: act[0..6] bf16, y32 of the last layer
adr_status cnn_forward(adr_cnn* c, int batch, const bf16* x)
{
    const bf16* in = x;
    for (int l = 0; l < kLayers; ++l) {
        ConvArgs a{};
        a.B = batch;
        a.H = a.W = c->hw;
        a.dil = kDil[l];
        a.bias = c->prm + c->T.boff[l];
        a.relu = l < kLayers - 1;
        a.spin = c->spin;
        if (l < kLayers - 1) a.y = c->act[l];
        else a.y32 = c->y32;
        const bf16* wk = c->wk + c->T.woff[l];
        if (l == 0)
            k_conv_first<<<(unsigned)(((long long)batch * c->hw * c->hw + 127) / 128), 128, kFirstSmem, c->stream>>>(
                a, in, wk, c->err);
        else TRY_S(launch_conv(c, c->stream, a, in, kCh[l], wk, kCh[l + 1]));
        in = c->act[l];
    }
    ADR_CUDA_TRY(cudaGetLastError());
    return ADR_OK;
}

// weight and bias gradients of a layer of 64 or 128 output channels from its
// input and its pre-activation gradient
adr_status layer_grad(adr_cnn* c, int batch, int l, const bf16* xin, const bf16* dy)
{
    cudaStream_t st = c->stream;
    const int cin = kCh[l], cout = kCh[l + 1];
    const long long M = (long long)batch * c->hw * c->hw;
    CUtensorMap tx, ty;
    if (!act_map(&tx, xin, batch, c->hw, c->hw, cin, 4) || !act_map(&ty, dy, batch, c->hw, c->hw, cout, 4)) {
        adr::set_error("the driver refused a tensor map of the weight gradient");
        return ADR_ECUDA;
    }
    WgradArgs w{};
    w.B = batch;
    w.H = w.W = c->hw;
    w.Cin = cin;
    w.Cout = cout;
    w.dil = kDil[l];
    w.part = c->part;
    w.bpart = c->spart;
    w.spin = c->spin;
    w.npair = cin > 64 ? 9 : 5;
    w.G = cin > 64 || cout == 128 ? 3 : 5;  // accumulators: G x cout of 512 columns of tensor memory
    const int groups = (w.npair + w.G - 1) / w.G;
    const int stage = (2 * w.G + cout / 64) * kWgPlane;
    w.stages = std::min(kWgMaxStages, kWgSmem / stage);
    w.tiles = (int)(M / 64);
    int splits = std::max(1, std::min(c->n_sm / groups, w.tiles));
    splits = (int)std::min<long long>(splits, c->part_size / (9LL * cin * cout));
    w.per = (w.tiles + splits - 1) / splits;
    splits = (w.tiles + w.per - 1) / w.per;
    const int cols = w.G * cout <= 256 ? 256 : 512, smem = w.stages * stage + 1024;
    const dim3 grid((unsigned)splits, (unsigned)groups);
    if (cout == 128) k_wgrad_tc<128><<<grid, kWgThreads, smem, st>>>(tx, ty, w, cols, c->err);
    else k_wgrad_tc<64><<<grid, kWgThreads, smem, st>>>(tx, ty, w, cols, c->err);
    const int nw = 9 * cin * cout;
    k_sum_splits<<<(nw + cout) / 32, 256, 0, st>>>(c->part, splits, nw, c->grad + c->T.woff[l], c->spart, cout,
                                                   c->grad + c->T.boff[l]);
    return ADR_OK;
}

adr_status cnn_backward(adr_cnn* c, int batch, const bf16* x, const float* t)
{
    cudaStream_t st = c->stream;
    const long long M = (long long)batch * c->hw * c->hw;
    const int nb = (int)((M + 255) / 256), last = kLayers - 1;
    k_loss<<<nb, 256, 0, st>>>(c->y32, kCout, t, M, c->dy0, c->lpart);
    k_sum_loss<<<1, 256, 0, st>>>(c->lpart, nb, M, c->loss);
    // the last layer: channel 0 alone
    const int lb = (int)std::min<long long>(kLastBlocks, (M + 31) / 32);
    k_last_wgrad<<<lb, 256, 0, st>>>(c->act[last - 1], c->dy0, M, c->hw, c->hw, c->spart);
    k_last_sum<<<(577 * 32 + 255) / 256, 256, 0, st>>>(c->spart, lb, c->grad + c->T.woff[last],
                                                      c->grad + c->T.boff[last]);
    bf16* dy = c->dA;
    k_last_dgrad<<<lb, 256, 0, st>>>(c->dy0, c->wk + c->T.woff[last], c->act[last - 1], M, c->hw, c->hw, dy);
    for (int l = last - 1; l >= 0; --l) {
        TRY_S(layer_grad(c, batch, l, l == 0 ? x : c->act[l - 1], dy));
        if (l > 0) {
            // data gradient: correlation with the flipped, transposed weights,
            // masked by the ReLU of the layer below
            ConvArgs a{};
            a.B = batch;
            a.H = a.W = c->hw;
            a.dil = kDil[l];
            a.mask = c->act[l - 1];
            a.spin = c->spin;
            a.y = dy == c->dA ? c->dB : c->dA;
            TRY_S(launch_conv(c, st, a, dy, kCh[l + 1], c->wtk + c->T.woff[l], kCh[l]));
            dy = a.y;
        }
    }
    ADR_CUDA_TRY(cudaGetLastError());
    return ADR_OK;
}

// a bounded wait gave up: clear the flag and report it
adr_status report_timeout(adr_cnn* c)
{
    cudaMemsetAsync(c->err, 0, sizeof(int), c->stream);
    cudaStreamSynchronize(c->stream);
    adr::set_error("a tensor-core kernel gave up waiting (bounded mbarrier wait); its outputs are not valid");
    return ADR_ETIMEOUT;
}

}  // namespace

extern "C" {

long adr_cnn_num_params(void) { return param_offset(kLayers, false); }

adr_status adr_cnn_set_wait_limit(adr_cnn* c, long long spins)
{
    if (!c || spins < 0) {
        adr::set_error("adr_cnn_set_wait_limit: NULL handle or negative bound");
        return ADR_EINVAL;
    }
    c->spin = spins;
    return ADR_OK;
}

adr_status adr_cnn_sync(adr_cnn* c)
{
    if (!c) {
        adr::set_error("adr_cnn_sync: NULL handle");
        return ADR_EINVAL;
    }
    int e = 0;
    ADR_CUDA_TRY(cudaMemcpyAsync(&e, c->err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    ADR_CUDA_TRY(cudaStreamSynchronize(c->stream));
    return e ? report_timeout(c) : ADR_OK;
}

void adr_cnn_destroy(adr_cnn* c)
{
    if (!c) return;
    if (c->stream) cudaStreamSynchronize(c->stream);
    else cudaDeviceSynchronize();
    for (void* q : c->owned) cudaFree(q);
    delete c;
}

adr_status adr_cnn_set_params(adr_cnn* c, const float* host)
{
    if (!c || !host) {
        adr::set_error("NULL argument");
        return ADR_EINVAL;
    }
    ADR_CUDA_TRY(cudaMemcpyAsync(c->prm, host, sizeof(float) * c->P, cudaMemcpyHostToDevice, c->stream));
    ADR_CUDA_TRY(cudaMemsetAsync(c->m, 0, sizeof(float) * c->P, c->stream));
    ADR_CUDA_TRY(cudaMemsetAsync(c->v, 0, sizeof(float) * c->P, c->stream));
    c->step = 0;
    k_refresh<<<(int)((c->P + 255) / 256), 256, 0, c->stream>>>(c->prm, c->P, c->T,
                                                                WeightCopies{c->wk, c->wtk});
    ADR_CUDA_TRY(cudaGetLastError());
    ADR_CUDA_TRY(cudaStreamSynchronize(c->stream));
    return ADR_OK;
}

adr_status adr_cnn_get_params(adr_cnn* c, float* host)
{
    if (!c || !host) {
        adr::set_error("NULL argument");
        return ADR_EINVAL;
    }
    ADR_CUDA_TRY(cudaMemcpyAsync(host, c->prm, sizeof(float) * c->P, cudaMemcpyDeviceToHost, c->stream));
    ADR_CUDA_TRY(cudaStreamSynchronize(c->stream));
    return ADR_OK;
}

adr_status adr_cnn_create(int max_batch, const float* params, void* stream, adr_cnn** out)
{
    if (!out || max_batch < 1 || !params) {
        adr::set_error("adr_cnn_create needs max_batch >= 1, initial parameters and an output");
        return ADR_EINVAL;
    }
    *out = nullptr;
    if (!tmap_encoder()) {
        adr::set_error("adr_cnn_create: the driver has no tensor-map encoder (cuTensorMapEncodeTiled)");
        return ADR_ECUDA;
    }
    adr_cnn* c = new (std::nothrow) adr_cnn;
    if (!c) return ADR_ENOMEM;
    c->max_batch = max_batch;
    c->stream = static_cast<cudaStream_t>(stream);
    c->P = param_offset(kLayers, false);
    for (int l = 0; l < kLayers; ++l) {
        c->T.woff[l] = param_offset(l, false);
        c->T.boff[l] = param_offset(l, true);
        c->T.cin[l] = kCh[l];
        c->T.cout[l] = kCh[l + 1];
    }
    const long long M = (long long)max_batch * c->hw * c->hw;
    {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&c->n_sm, cudaDevAttrMultiProcessorCount, dev);
    }
    adr_status s = ADR_OK;
    auto fail = [&](adr_status st) {
        adr_cnn_destroy(c);
        return st;
    };
    if ((s = cnn_alloc(c, &c->prm, c->P)) || (s = cnn_alloc(c, &c->m, c->P)) ||
        (s = cnn_alloc(c, &c->v, c->P)) || (s = cnn_alloc(c, &c->grad, c->P)) ||
        (s = cnn_alloc(c, &c->wk, c->P)) || (s = cnn_alloc(c, &c->wtk, c->P)) ||
        (s = cnn_alloc(c, &c->err, 1)) ||
        (s = cnn_alloc(c, &c->y32, M * kCout)) || (s = cnn_alloc(c, &c->dA, M * 128)) ||
        (s = cnn_alloc(c, &c->dB, M * 128)) || (s = cnn_alloc(c, &c->dy0, M)) ||
        (s = cnn_alloc(c, &c->spart, (size_t)kLastBlocks * 577)) ||
        (s = cnn_alloc(c, &c->lpart, (M + 255) / 256 + 1)) || (s = cnn_alloc(c, &c->loss, 1)))
        return fail(s);
    for (int l = 0; l < kLayers - 1; ++l)
        if ((s = cnn_alloc(c, &c->act[l], M * kCh[l + 1]))) return fail(s);
    c->part_size = 64LL * 9 * 128 * 128;
    if ((s = cnn_alloc(c, &c->part, c->part_size))) return fail(s);
    ADR_CUDA_TRY(cudaMemsetAsync(c->err, 0, sizeof(int), c->stream));
    // the tensor-core kernels use more than 48 KB of shared memory (per device)
    ADR_CUDA_TRY(cudaFuncSetAttribute(k_wgrad_tc<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem + 1024));
    ADR_CUDA_TRY(cudaFuncSetAttribute(k_wgrad_tc<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem + 1024));
    ADR_CUDA_TRY(cudaFuncSetAttribute(k_conv_first, cudaFuncAttributeMaxDynamicSharedMemorySize, kFirstSmem));
    for (const void* f : {(const void*)k_conv_win<16>, (const void*)k_conv_win<64>})
        ADR_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kConvSmem + 1024));
    const void* convs[] = {(const void*)k_conv<64, 1>, (const void*)k_conv<64, 2>, (const void*)k_conv<128, 1>,
                           (const void*)k_conv<128, 2>};
    for (const void* f : convs)
        ADR_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kConvSmem + 1024));
    if ((s = adr_cnn_set_params(c, params))) return fail(s);
    *out = c;
    return ADR_OK;
}

adr_status adr_cnn_features(int batch, int n, const double* f, const double* b1, const double* b2,
                            const uint8_t* mask, const double* mu, const double* sigma,
                            const double* u0, uint16_t* x, double* scale, void* stream)
{
    if (batch < 1 || n != kN || !f || !b1 || !b2 || !mask || !mu || !sigma || !x || !scale) {
        adr::set_error("adr_cnn_features: bad arguments (the network reads 256 x 256 grids)");
        return ADR_EINVAL;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    k_scale<<<batch, 256, 0, st>>>(u0, scale);
    long long q = (long long)batch * kHW * kHW;
    k_features<<<(int)((q + 255) / 256), 256, 0, st>>>(batch, f, b1, b2, mask, mu, sigma, u0, scale,
                                                       reinterpret_cast<bf16*>(x));
    ADR_CUDA_TRY(cudaGetLastError());
    return ADR_OK;
}

adr_status adr_cnn_targets(int batch, int n, const double* u, const double* u0,
                           const double* scale, float* t, void* stream)
{
    if (batch < 1 || n != kN || !u || !scale || !t) {
        adr::set_error("adr_cnn_targets: bad arguments (the network reads 256 x 256 grids)");
        return ADR_EINVAL;
    }
    long long q = (long long)batch * kHW * kHW;
    k_targets<<<(int)((q + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(batch, u, u0,
                                                                                    scale, t);
    ADR_CUDA_TRY(cudaGetLastError());
    return ADR_OK;
}

adr_status adr_cnn_forward(adr_cnn* c, int batch, const uint16_t* x, float* y)
{
    if (!c || batch < 1 || batch > c->max_batch || !x || !y) {
        adr::set_error("adr_cnn_forward: bad arguments");
        return ADR_EINVAL;
    }
    TRY_S(cnn_forward(c, batch, reinterpret_cast<const bf16*>(x)));
    const long long M = (long long)batch * c->hw * c->hw;
    ADR_CUDA_TRY(cudaMemcpyAsync(y, c->y32, sizeof(float) * M * kCout, cudaMemcpyDeviceToDevice,
                                 c->stream));
    return ADR_OK;
}

adr_status adr_cnn_loss_grad(adr_cnn* c, int batch, const uint16_t* x, const float* t, float* grad,
                             double* loss)
{
    if (!c || batch < 1 || batch > c->max_batch || !x || !t) {
        adr::set_error("adr_cnn_loss_grad: bad arguments");
        return ADR_EINVAL;
    }
    const bf16* xb = reinterpret_cast<const bf16*>(x);
    TRY_S(cnn_forward(c, batch, xb));
    TRY_S(cnn_backward(c, batch, xb, t));
    if (grad)
        ADR_CUDA_TRY(cudaMemcpyAsync(grad, c->grad, sizeof(float) * c->P, cudaMemcpyDeviceToDevice,
                                     c->stream));
    if (loss) {
        int e = 0;
        ADR_CUDA_TRY(cudaMemcpyAsync(loss, c->loss, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        ADR_CUDA_TRY(cudaMemcpyAsync(&e, c->err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
        ADR_CUDA_TRY(cudaStreamSynchronize(c->stream));
        if (e) return report_timeout(c);
    }
    return ADR_OK;
}

adr_status adr_cnn_train_step(adr_cnn* c, int batch, const uint16_t* x, const float* t, float lr,
                              double* loss)
{
    if (!c || batch < 1 || batch > c->max_batch || !x || !t || !(lr > 0.f)) {
        adr::set_error("adr_cnn_train_step: bad arguments");
        return ADR_EINVAL;
    }
    const bf16* xb = reinterpret_cast<const bf16*>(x);
    TRY_S(cnn_forward(c, batch, xb));
    TRY_S(cnn_backward(c, batch, xb, t));
    c->step++;
    const float b1 = 0.9f, b2 = 0.999f;
    float c1 = 1.f - powf(b1, (float)c->step), c2 = 1.f - powf(b2, (float)c->step);
    k_adam<<<(int)((c->P + 255) / 256), 256, 0, c->stream>>>(
        c->prm, c->m, c->v, c->grad, c->P, lr, b1, b2, 1e-8f, c1, c2, c->T,
        WeightCopies{c->wk, c->wtk});
    ADR_CUDA_TRY(cudaGetLastError());
    if (loss) {
        int e = 0;
        ADR_CUDA_TRY(cudaMemcpyAsync(loss, c->loss, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        ADR_CUDA_TRY(cudaMemcpyAsync(&e, c->err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
        ADR_CUDA_TRY(cudaStreamSynchronize(c->stream));
        if (e) return report_timeout(c);
    }
    return ADR_OK;
}

}  // extern "C"

namespace adr {
// forward of a batch on stream st (a problem's stream): ordered after the
// network's pending work and before its later work by events both ways
adr_status cnn_forward_on(adr_cnn* c, int batch, const uint16_t* x, float* y, cudaStream_t st)
{
    if (!c || batch < 1 || batch > c->max_batch || !x || !y) {
        set_error("warm start: bad network call");
        return ADR_EINVAL;
    }
    cudaEvent_t ev = nullptr;
    ADR_CUDA_TRY(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    const cudaStream_t own = c->stream;
    adr_status s = ADR_OK;
    cudaError_t e = cudaEventRecord(ev, own);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev, 0);
    if (e != cudaSuccess) s = cuda_fail(e, "warm start: stream order");
    if (s == ADR_OK) {
        c->stream = st;
        s = adr_cnn_forward(c, batch, x, y);
        c->stream = own;
    }
    if (s == ADR_OK) {
        e = cudaEventRecord(ev, st);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(own, ev, 0);
        if (e != cudaSuccess) s = cuda_fail(e, "warm start: stream order");
    }
    cudaEventDestroy(ev);
    return s;
}

// one prediction [64][64][8] around u0 to the handle's 256 x 256 grid
adr_status launch_cnn_upsample(Problem* p, const float* y, const double* u0, const double* scale,
                               double* u)
{
    long long N = p->N;
    k_upsample<<<(int)((N + 255) / 256), 256, 0, p->stream>>>(y, u0, scale, p->ntype, u);
    ADR_CUDA_TRY(cudaGetLastError());
    return ADR_OK;
}
}  // namespace adr
