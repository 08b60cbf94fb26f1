// Tensor-core (tcgen05) 3x3 convolutions for 32 -> 32 channels, stride 1: the
// forward, the data gradient and the weight gradient of the encoder's inner layers.
//
// Activation format between these layers: "padded HWC" BF16 - per image (H+4) x (W+4)
// rows of 32 channels (64 B), the valid pixels at rows (y+2)(W+4) + x+2, zeros
// elsewhere.  On a virtual output grid that keeps the input's row width Wp, output
// pixel q = oy Wp + ox reads input row q + origin(ky, kx), so each of the nine
// taps is the same shared-memory image seen from a shifted start row: the A
// operand of tap (ky, kx) is a descriptor whose start address moves by
// origin(ky, kx) rows, with no im2col copy.  Columns ox >= out_w of the virtual
// grid are computed and discarded.
//
// Shared-memory operand layout: the canonical no-swizzle K-major layout with
// channels split into 4 planes of 8 (16 B per pixel row per plane): element
// (row r, channel c) at (c / 8) * PLANE + r * 16 + (c % 8) * 2.  Any start row is a
// valid descriptor start.  TMA loads each plane of an image box by box.
#include "sq_kernels.cuh"
#include "sq_tc.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>

namespace sq {

namespace {

constexpr long long kWaitCycles = 4000000000ll;   // ~2 s at 2 GHz
constexpr int kCh = 32;                            // channels in and out
constexpr int kWBytes = 9 * kCh * kCh * 2;         // 18432 B: one layer's filter in BF16

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err, int code) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > kWaitCycles) {
            atomicCAS(err, 0, code);
            return false;
        }
    }
    return true;
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
            "r"(dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"((uint64_t)src), "r"(bytes), "r"(bar)
                 : "memory");
}
// No-swizzle shared-memory descriptor (core matrices of 8 rows x 16 B).  K-major operand:
// lbo = stride between core matrices along K, sbo = along M/N.  MN-major operand:
// lbo = stride along K, sbo = along M/N (checked against the oracle's convolution).
__device__ __forceinline__ uint64_t plain_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn, bool b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
            d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols));
}

// ---------------------------------------------------------------- forward / data gradient
struct ConvArgs {
    CUtensorMap tin;                 // input planes: dims {8, 4, nimg * in_rows}
    const __nv_bfloat16* w;          // filter, layout [tap][plane][out ch][8]
    int nimg, in_rows, Wp, out_h, out_w, off0, n_tiles, load_rows, tmem_cols;
    const float* bias;               // forward: bias[out ch]
    int relu;
    const __nv_bfloat16* mask;       // data gradient: padded-HWC activation of the layer below (mask > 0)
    __nv_bfloat16* out_phwc;         // padded-HWC output (grid width out_w + 4), interior written
    float* out_chw;                  // optional CHW FP32 output [nimg, 32, out_h, out_w]
    __nv_bfloat16* out_chw_bf;       // optional CHW BF16 copy
    int* err;
};

// Persistent and warp-specialised: CTA c takes images c, c + gridDim.x, ...  Warp 0 (one
// lane) loads the filter once and each image by TMA into one of two shared-memory
// buffers; warp 1 (one lane) owns the tensor memory and issues each image's MMAs into
// one of two accumulators; warps 2..5 (TMEM lane quarters 2, 3, 0, 1) drain an
// accumulator (bias, ReLU, mask, stores) while the next image is loaded and multiplied.
// Barriers: full/empty per image buffer, tfull/tempty per accumulator; every wait is
// bounded and a wait that gives up records its code in *err and stops that role.
constexpr int kConvThreads = 192;

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void conv32_tc(const ConvArgs& a) {
    SQ_KERNEL_WAIT();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t plane = (uint32_t)a.load_rows * 16;
    const uint32_t ibytes = 4 * plane;
    uint8_t* w_s = smem + 2 * ibytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(w_s + kWBytes);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 10);
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + 2), tfull0 = smem_u32(bars + 4),
                   tempty0 = smem_u32(bars + 6), done_bar = smem_u32(bars + 8);
    const int warp = warp_uniform((int)threadIdx.x / 32), lane = threadIdx.x % 32;
    const int n_local = (int)blockIdx.x < a.nimg ? (a.nimg - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const uint32_t cols = 2 * (uint32_t)a.tmem_cols;

    if (warp == 1) tmem_alloc(smem_u32(tmem_slot), cols);
    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(full0 + 8 * b, 1);
            mbar_init(empty0 + 8 * b, 1);
            mbar_init(tfull0 + 8 * b, 1);
            mbar_init(tempty0 + 8 * b, 4);   // one arrival per epilogue warp
        }
        mbar_init(done_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = warp_uniform(*tmem_slot);
    const uint32_t w_u = smem_u32(w_s);

    if (warp == 0) {
        if (elect_one()) {
            // producer: the filter with the first image, then image i into buffer i % 2 once
            // the MMAs of image i - 2 have read it
            int issued = 0;
            for (int i = 0; i < n_local; ++i) {
                const int b = i & 1;
                if (i >= 2 && !mbar_wait(empty0 + 8 * b, ((i - 2) >> 1) & 1, a.err, 13)) break;
                const int img = (int)blockIdx.x + i * (int)gridDim.x;
                const uint32_t dst = smem_u32(smem) + b * ibytes;
                mbar_expect_tx(full0 + 8 * b, ibytes + (i == 0 ? (uint32_t)kWBytes : 0u));
                for (int c = 0; c < 4; ++c)
                    for (int bb = 0; bb < a.load_rows / 128; ++bb)
                        tma_load_3d(dst + c * plane + bb * 2048, &a.tin, 0, c, img * a.in_rows + bb * 128, full0 + 8 * b);
                if (i == 0) bulk_load(w_u, a.w, kWBytes, full0);
                issued = i + 1;
            }
            // the last loads have landed before the CTA can finish (immediate unless a consumer gave up)
            for (int i = issued - 2 < 0 ? 0 : issued - 2; i < issued; ++i)
                mbar_wait(full0 + 8 * (i & 1), (i >> 1) & 1, a.err, 14);
        }
    } else if (warp == 1) {
        if (elect_one()) {
            constexpr uint32_t idesc = idesc_bf16(128, kCh, false, false);
            for (int i = 0; i < n_local; ++i) {
                const int b = i & 1;
                if (!mbar_wait(full0 + 8 * b, (i >> 1) & 1, a.err, 11)) break;
                if (i >= 2 && !mbar_wait(tempty0 + 8 * b, ((i - 2) >> 1) & 1, a.err, 15)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // descriptors of the first tap; starts move in 16-byte units within the 14-bit field
                const uint64_t a0 = plain_desc(smem_u32(smem) + b * ibytes + a.off0 * 16, plane, 128);
                const uint64_t b0 = plain_desc(w_u, 512, 128);
                const uint32_t acc = tmem + b * (uint32_t)a.tmem_cols;
                for (int t = 0; t < a.n_tiles; ++t)
#pragma unroll
                    for (int tap = 0; tap < 9; ++tap)
#pragma unroll
                        for (int kc = 0; kc < 2; ++kc)
                            mma_bf16(acc + t * kCh, a0 + (uint64_t)(kc * (plane / 8) + t * 128 + (tap / 3) * a.Wp + tap % 3),
                                     b0 + (uint64_t)(tap * 128 + kc * 64), idesc, (tap | kc) ? 1u : 0u);
                mma_commit(empty0 + 8 * b);
                mma_commit(tfull0 + 8 * b);
            }
            // every MMA this CTA issued has completed before the tensor memory is freed
            mma_commit(done_bar);
            mbar_wait(done_bar, 0, a.err, 16);
        }
        __syncwarp();
    } else {
        const int quarter = warp % 4;
        const int wpo = a.out_w + 4;
        const int64_t out_img = (int64_t)(a.out_h + 4) * wpo * kCh;
        // a thread's output pixel in each tile, and the bias, are the same for every image
        int oy_t[4], ox_t[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int q = t * 128 + quarter * 32 + lane;
            oy_t[t] = q / a.Wp;
            ox_t[t] = q - oy_t[t] * a.Wp;
        }
        float bias_r[kCh];
#pragma unroll
        for (int j = 0; j < kCh; ++j) bias_r[j] = a.bias ? a.bias[j] : 0.f;
        for (int i = 0; i < n_local; ++i) {
            const int b = i & 1;
            const bool have = __all_sync(0xffffffffu, mbar_wait(tfull0 + 8 * b, (i >> 1) & 1, a.err, 12));
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int img = (int)blockIdx.x + i * (int)gridDim.x;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if (t >= a.n_tiles || !have) break;
                __syncwarp();   // (the lanes without a pixel in the tile before)
                uint32_t r0[16], r1[16];
                const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + b * (uint32_t)a.tmem_cols + t * kCh;
                tmem_ld16(taddr, r0);
                tmem_ld16(taddr + 16, r1);
                const int oy = oy_t[t], ox = ox_t[t];
                if (oy >= a.out_h || ox >= a.out_w) continue;
                float v[kCh];
#pragma unroll
                for (int j = 0; j < 16; ++j) { v[j] = __uint_as_float(r0[j]); v[16 + j] = __uint_as_float(r1[j]); }
                const int64_t prow = ((int64_t)(oy + 2) * wpo + ox + 2) * kCh;
                if (a.bias) {
#pragma unroll
                    for (int j = 0; j < kCh; ++j) v[j] += bias_r[j];
                }
                if (a.relu) {
#pragma unroll
                    for (int j = 0; j < kCh; ++j) v[j] = fmaxf(v[j], 0.f);
                }
                if (a.mask) {
                    const uint4* mk = reinterpret_cast<const uint4*>(a.mask + (int64_t)img * out_img + prow);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint4 m4 = mk[c];
                        const __nv_bfloat16* mb = reinterpret_cast<const __nv_bfloat16*>(&m4);
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (!(__bfloat162float(mb[j]) > 0.f)) v[c * 8 + j] = 0.f;
                    }
                }
                if (a.out_phwc) {
                    uint4* dst = reinterpret_cast<uint4*>(a.out_phwc + (int64_t)img * out_img + prow);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        __align__(16) __nv_bfloat16 hb[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) hb[j] = __float2bfloat16_rn(v[c * 8 + j]);
                        dst[c] = *reinterpret_cast<const uint4*>(hb);
                    }
                }
                if (a.out_chw || a.out_chw_bf) {
                    const int64_t plane_px = (int64_t)a.out_h * a.out_w;
                    const int64_t base = (int64_t)img * kCh * plane_px + (int64_t)oy * a.out_w + ox;
#pragma unroll
                    for (int j = 0; j < kCh; ++j) {
                        if (a.out_chw) a.out_chw[base + j * plane_px] = v[j];
                        if (a.out_chw_bf) a.out_chw_bf[base + j * plane_px] = __float2bfloat16_rn(v[j]);
                    }
                }
            }
            // this warp's lanes of the accumulator are read: it may take the image after next
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty0 + 8 * b);
            if (!have) break;
        }
    }
    SQ_KERNEL_TRIGGER();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc(tmem, cols);
    }
}

// The two are one kernel compiled twice.  Bounded to two CTAs an SM (what fits), the compiler keeps
// the bias and the pixel places in registers, 136 of them; left to itself it takes 80.  Alone the first is
// the faster: 2,228 images of 11 x 9 16.2 us and 17.7, 4,096 of 9 x 9 24.5 and 27.4, 512 of 15 x 15 (data
// gradient) 9.2 and 9.7.  Beside the kernels of the update's other branches, at 512 images, its registers
// are missed there: 303.1 us an update and 301.8.
__global__ void __launch_bounds__(kConvThreads) conv32_tc_kernel(const __grid_constant__ ConvArgs a) { conv32_tc(a); }
__global__ void __launch_bounds__(kConvThreads, 2) conv32_tc_alone_kernel(const __grid_constant__ ConvArgs a) { conv32_tc(a); }

// ---------------------------------------------------------------- weight gradient
// D_tap[co, ci] += sum_q dy[q, co] x[q + origin(tap), ci] over the virtual grid of
// the input's padded row width (dy = 0 outside the valid outputs), origin(ky, kx) =
// (2 + ky) Wp + 2 + kx.  A = dy^T, MN-major: four warps copy dy's 16-byte pixel chunks
// unchanged into four channel planes of kq pixel rows (no transpose); rows 32..127 of the
// 128-row MMA read whatever follows in shared memory (inside the allocation: the dy
// buffers come first) and land in accumulator rows that are never read.  B stacks the
// three horizontal taps: shared memory holds
// twelve slots (kx, channel plane), slot (kx, p) = rows origin(0, kx) + [0, x_rows)
// of plane p, slot_rows apart, so one MN-major operand of N = 96 (kx, ci) starting ky Wp
// rows into every slot covers taps (ky, 0..2); its accumulator columns ky 96 + kx 32 +
// ci are tap 32 + ci.  Three MMAs per 16 pixels instead of nine.
// What bounds it, for 512 images of 15 x 15, four to a CTA: the products (3,000 cycles an image)
// and the fixed start and end (5,000).  The next image is staged while one is multiplied; four
// more warps copy the input with 16-byte asynchronous copies, where tensor copies of its 16-byte
// plane rows took 4,800 cycles an image to issue; the end reads the accumulators by three
// warps and stores 16 bytes a thread.  20.2 us before, 11.5 now (11 x 11: 17.9 and 9.3).
struct WgradArgs {
    const __nv_bfloat16* x;          // padded-HWC layer input
    const __nv_bfloat16* dy;         // padded-HWC gradient at the layer's pre-activation (grid out_w + 4)
    int nimg, in_rows, Wp, out_h, out_w, kq, slot_rows, x_rows, per_cta;
    float* work;                     // [ctas, 32, 289]: partial dW (co, ci*9 + tap) and db (col 288)
    int* err;
};

constexpr int kDyBytesMax = 32768;
constexpr uint32_t kWgTileBytes = kCh * (kCh * 9 + 1) * 4;   // the partial tile, staged at the end
// bytes from the (1024-aligned) start of shared memory to the barriers: the operand buffers,
// at least as many as the partial tile that reuses them
__host__ __device__ inline uint32_t wgrad_operand_bytes(uint32_t xbytes, uint32_t dybytes) {
    const uint32_t ops = 2 * xbytes + 2 * dybytes;
    return ops > kWgTileBytes ? ops : kWgTileBytes;
}

// Threads 0-127 stage dy, 128-255 the input, warp 8 issues the products.
constexpr int kWgThreads = 288;
__global__ void __launch_bounds__(kWgThreads) wgrad32_tc_kernel(const __grid_constant__ WgradArgs a) {
    SQ_KERNEL_WAIT();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t slot = (uint32_t)a.slot_rows * 16;
    const uint32_t xbytes = 12 * slot;
    const uint32_t dplane = (uint32_t)a.kq * 16;                 // one 8-channel plane of dy
    const uint32_t dybytes = 4 * dplane;
    uint8_t* ds[2] = {smem, smem + dybytes};
    uint8_t* xs[2] = {smem + 2 * dybytes, smem + 2 * dybytes + xbytes};
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + wgrad_operand_bytes(xbytes, dybytes));
    float* red = reinterpret_cast<float*>(bars + 8);             // [128][8] bias partials
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(red + 128 * 8);
    const uint32_t mma_bar[2] = {smem_u32(bars), smem_u32(bars + 1)};
    const uint32_t done_bar = smem_u32(bars + 2);
    const int warp = warp_uniform((int)threadIdx.x / 32), lane = threadIdx.x % 32;
    const int i0 = blockIdx.x * a.per_cta, i1 = min(a.nimg, i0 + a.per_cta);

    if (warp == 0) tmem_alloc(smem_u32(tmem_slot), 512);
    if (threadIdx.x == 32) {
        for (int b = 0; b < 2; ++b) mbar_init(mma_bar[b], 1);
        mbar_init(done_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = warp_uniform(*tmem_slot);
    const int wpo = a.out_w + 4;
    const int64_t dy_img = (int64_t)(a.out_h + 4) * wpo * kCh;
    float bsum[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const int cc = threadIdx.x % 4;         // the 8-channel chunk this thread stages
    bool ok = true;
    constexpr uint32_t idesc = idesc_bf16(128, 3 * kCh, true, true);

    const int64_t x_end = (int64_t)a.nimg * a.in_rows;
    auto stage = [&](int i) {
        const int b = (i - i0) & 1;
        if (warp >= 4) {
            // the input's 16-byte chunks, once per horizontal tap; rows behind the last image read as
            // zero.  (A pixel's four chunks land slot bytes apart, an odd multiple of 32: no bank
            // conflict.  Tensor copies of 16-byte rows would take 1.3 cycles a row, three times this.)
            const int64_t row0 = (int64_t)i * a.in_rows + 2 * a.Wp + 2;
            const uint32_t dst = smem_u32(xs[b]) + cc * slot;
            for (int row = (threadIdx.x - 128) / 4; row < a.x_rows; row += 32) {
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) {
                    const bool in = row0 + kx + row < x_end;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst + kx * 4 * slot + row * 16),
                                 "l"(in ? a.x + (row0 + kx + row) * kCh + cc * 8 : a.x), "r"(in ? 16 : 0) : "memory");
                }
            }
            return;
        }
        // stage dy: the 16-byte chunk of channels 8 cc .. 8 cc + 7 of pixel q at cc PLANE + 16 q
        // (zero outside the valid outputs); a thread's loads for eight pixels are issued
        // before any of them is stored
        uint8_t* d = ds[b];
        for (int j0 = threadIdx.x; j0 < a.kq * 4; j0 += 8 * 128) {
            uint4 v4[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int j = j0 + u * 128;
                const int q = j >> 2;
                const int oy = q / a.Wp, ox = q - (q / a.Wp) * a.Wp;
                v4[u] = make_uint4(0, 0, 0, 0);
                if (j < a.kq * 4 && oy < a.out_h && ox < a.out_w)
                    v4[u] = *reinterpret_cast<const uint4*>(a.dy + (int64_t)i * dy_img +
                                                            ((int64_t)(oy + 2) * wpo + ox + 2) * kCh + cc * 8);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int j = j0 + u * 128;
                if (j >= a.kq * 4) break;
                const int q = j >> 2;
                const __nv_bfloat16* hv = reinterpret_cast<const __nv_bfloat16*>(&v4[u]);
                *reinterpret_cast<uint4*>(d + cc * dplane + q * 16) = v4[u];
#pragma unroll
                for (int k = 0; k < 8; ++k) bsum[k] += __bfloat162float(hv[k]);
            }
        }
    };
    // Every thread runs every iteration (the barriers inside must match); a wait that gives up
    // only records the error and stops this thread's staging.
    if (warp < 8 && i0 < i1) stage(i0);
    for (int i = i0; i < i1; ++i) {
        const int li = i - i0, b = li & 1;
        asm volatile("cp.async.wait_all;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (warp == 8) {
            if (elect_one()) {
                // descriptors built once; each MMA adds its start offset in 16-byte units
                // (shared-memory addresses stay below 2^18: the 14-bit field never carries)
                const uint64_t a0 = plain_desc(smem_u32(ds[b]), 128, dplane);
                const uint64_t b0 = plain_desc(smem_u32(xs[b]), 128, slot);
                for (int k = 0; k < a.kq / 16; ++k)
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky)
                        mma_bf16(tmem + ky * 3 * kCh, a0 + (uint64_t)(k * 16), b0 + (uint64_t)(k * 16 + ky * a.Wp),
                                 idesc, (i > i0 || k > 0) ? 1u : 0u);
                mma_commit(mma_bar[b]);
            }
            __syncwarp();
        } else if (i + 1 < i1) {
            // the next image, into the buffers that the products of the one before have read
            if (li >= 1 && !mbar_wait(mma_bar[b ^ 1], ((li - 1) >> 1) & 1, a.err, 21)) ok = false;
            if (ok) stage(i + 1);
        }
    }
    if (warp == 8 && elect_one()) mma_commit(done_bar);
    __syncwarp();
    SQ_KERNEL_TRIGGER();
    const bool have = mbar_wait(done_bar, 0, a.err, 23) && ok && i1 > i0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // bias partials: reduce the 32 threads of each chunk in a fixed order.  The partial
    // tile [co][ci * 9 + tap | bias] is assembled in shared memory (the operand buffers are
    // idle once the last MMA has completed) and stored by all threads, coalesced.
    if (threadIdx.x < 128) {
#pragma unroll
        for (int k = 0; k < 8; ++k) red[threadIdx.x * 8 + k] = bsum[k];
    }
    __syncthreads();
    constexpr int NW = kCh * 9 + 1;
    float* tile = reinterpret_cast<float*>(smem);   // [kCh][NW]
    if (warp == 1) {
        const int co = lane;
        float s = 0.f;
        for (int t = co / 8; t < 128; t += 4) s += red[t * 8 + (co % 8)];
        tile[co * NW + kCh * 9] = s;
    }
    if (warp % 4 == 0) {   // lanes 0-31 of the accumulators: a row ky of taps each
        const int co = lane;
        for (int tap = 3 * (warp / 4); tap < 3 * (warp / 4) + 3; ++tap) {
            uint32_t r0[16], r1[16];
            tmem_ld16(tmem + tap * kCh, r0);
            tmem_ld16(tmem + tap * kCh + 16, r1);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                tile[co * NW + j * 9 + tap] = have ? __uint_as_float(r0[j]) : 0.f;
                tile[co * NW + (16 + j) * 9 + tap] = have ? __uint_as_float(r1[j]) : 0.f;
            }
        }
    }
    __syncthreads();
    float* out = a.work + (int64_t)blockIdx.x * kCh * NW;
    if (reinterpret_cast<uintptr_t>(out) % 16 == 0) {
        for (int e = threadIdx.x; e < kCh * NW / 4; e += kWgThreads)
            reinterpret_cast<float4*>(out)[e] = reinterpret_cast<const float4*>(tile)[e];
    } else {
        for (int e = threadIdx.x; e < kCh * NW; e += kWgThreads) out[e] = tile[e];
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc(tmem, 512);
    }
}

// 32 elements per block and 8 groups of CTAs: group g adds CTA partials g, g + 8, ... in
// increasing order, then the group sums are added in group order (a fixed order, so
// partials reduced once per whole batch or after chunks give the same bits).
constexpr int kRed32Groups = 8;
__global__ void __launch_bounds__(32 * kRed32Groups) wgrad32_reduce_kernel(const float* __restrict__ work, int splits,
                                                                            float* __restrict__ dw,
                                                                            float* __restrict__ db) {
    SQ_KERNEL_ENTRY();
    constexpr int N = kCh * 9 + 1;
    constexpr int tot = kCh * N;
    __shared__ float part[kRed32Groups][33];
    const int tx = threadIdx.x % 32, g = threadIdx.x / 32;
    const int e = blockIdx.x * 32 + tx;
    float s = 0.f;
    if (e < tot) {
        int z = g;
        for (; z + 3 * kRed32Groups < splits; z += 4 * kRed32Groups) {   // four partials' loads in flight
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = work[(int64_t)(z + u * kRed32Groups) * tot + e];
#pragma unroll
            for (int u = 0; u < 4; ++u) s += v[u];
        }
        for (; z < splits; z += kRed32Groups) s += work[(int64_t)z * tot + e];
    }
    part[g][tx] = s;
    __syncthreads();
    if (g != 0 || e >= tot) return;
    float a = 0.f;
#pragma unroll
    for (int k = 0; k < kRed32Groups; ++k) a += part[k][tx];
    const int co = e / N, col = e - co * N;
    if (col == N - 1) db[co] = a;
    else dw[co * (N - 1) + col] = a;
}

// ---------------------------------------------------------------- first layer straight to padded HWC
// The encoder's first convolution (few input channels, any stride, 32 outputs) for the
// tensor-core path: one thread per output pixel holds its 32 channels, the filter and bias
// are broadcast from shared memory, and the ReLU output goes straight to the padded-HWC
// BF16 image the next (tensor-core) layer reads.  Each output is accumulated over
// k = (ci, ky, kx) in order with fused multiply-adds, then the bias is added: the same
// arithmetic as the CUDA-core implicit GEMM followed by the layout conversion.
__global__ void __launch_bounds__(256) conv0_phwc_kernel(ConvShape sh, const float* __restrict__ x,
                                                         const float* __restrict__ w, const float* __restrict__ bias,
                                                         __nv_bfloat16* __restrict__ out) {
    SQ_KERNEL_ENTRY();
    extern __shared__ float w_s[];   // [K][32] then bias [32]
    const int K = sh.Cin * 9;
    for (int e = threadIdx.x; e < K * kCh; e += blockDim.x) {
        const int k = e / kCh, co = e % kCh;
        w_s[e] = w[(int64_t)co * K + k];
    }
    if (threadIdx.x < kCh) w_s[K * kCh + threadIdx.x] = bias[threadIdx.x];
    __syncthreads();
    // two output pixels per thread (blockDim apart, so each half stays coalesced): every
    // weight read from shared memory feeds both
    const int64_t npix = (int64_t)sh.nimg * sh.OH * sh.OW;
    const int64_t p0 = (int64_t)blockIdx.x * 2 * blockDim.x + threadIdx.x;
    if (p0 >= npix) return;
    const int64_t pp[2] = {p0, p0 + blockDim.x};
    const bool has1 = pp[1] < npix;
    const float* xb[2];
    __nv_bfloat16* dst[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t p = has1 || h == 0 ? pp[h] : pp[0];
        const int img = (int)(p / (sh.OH * sh.OW));
        const int rem = (int)(p - (int64_t)img * sh.OH * sh.OW);
        const int oy = rem / sh.OW, ox = rem - (rem / sh.OW) * sh.OW;
        xb[h] = x + (int64_t)img * sh.x_img_stride + (int64_t)(oy * sh.stride) * sh.W + ox * sh.stride;
        dst[h] = out + ((int64_t)img * (sh.OH + 4) * (sh.OW + 4) + (int64_t)(oy + 2) * (sh.OW + 4) + ox + 2) * kCh;
    }
    float acc0[kCh], acc1[kCh];
#pragma unroll
    for (int co = 0; co < kCh; ++co) { acc0[co] = 0.f; acc1[co] = 0.f; }
    for (int ci = 0; ci < sh.Cin; ++ci)
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int64_t off = (int64_t)ci * sh.H * sh.W + (t / 3) * sh.W + (t % 3);
            const float xv0 = __ldg(xb[0] + off), xv1 = __ldg(xb[1] + off);
            const float* wk = w_s + (ci * 9 + t) * kCh;
#pragma unroll
            for (int co = 0; co < kCh; ++co) {
                const float wv = wk[co];
                acc0[co] = fmaf(xv0, wv, acc0[co]);
                acc1[co] = fmaf(xv1, wv, acc1[co]);
            }
        }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && !has1) break;
        __align__(16) __nv_bfloat16 hb[kCh];
#pragma unroll
        for (int co = 0; co < kCh; ++co) {
            float v = (h == 0 ? acc0[co] : acc1[co]) + w_s[K * kCh + co];
            if (!(v > 0.f)) v = 0.f;
            hb[co] = __float2bfloat16_rn(v);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) reinterpret_cast<uint4*>(dst[h])[c] = reinterpret_cast<const uint4*>(hb)[c];
    }
}


// ---------------------------------------------------------------- first layer on tensor cores
// The first encoder layer (few input channels, any stride, 32 outputs) as an implicit GEMM
// on tcgen05: D[pixel, co] = sum_k A[pixel, k] W[co, k] with k = (ci, ky, kx) in the
// filter's own order, K = 9 Cin zero-padded to 8 PL.  A 128-pixel tile of A is gathered
// by the threads (thread r: pixel r, its K inputs rounded to BF16) into the canonical
// no-swizzle K-major layout, PL planes of 8 k-values (2048 B each); the filter is held as
// the N = 32 operand in the same layout.  One thread issues the PL / 2 MMAs (K = 16) of a
// tile into one of two accumulators; while they run the threads drain the previous tile
// (bias, ReLU, BF16, padded-HWC store) and then gather the next one.  Persistent CTAs.
struct Conv0Args {
    ConvShape sh;
    const float* x;       // NCHW FP32, image stride sh.x_img_stride
    const float* w;       // [32][K] FP32
    const float* bias;    // [32]
    __nv_bfloat16* out;   // padded HWC BF16, grid (OH + 4) x (OW + 4) per image
    int64_t npix;
    int K, n_tiles;
    int* err;
};

// two floats rounded to BF16 (nearest even), the first in the low half
__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

template <int PL>
__global__ void __launch_bounds__(128, PL == 4 ? 5 : 2) conv0_tc_kernel(const __grid_constant__ Conv0Args a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    constexpr uint32_t kTile = PL * 2048;            // one A tile: PL planes of 128 rows x 16 B
    uint8_t* b_s = smem + 2 * kTile;                  // the filter: PL planes of 32 rows x 16 B
    float* bias_s = reinterpret_cast<float*>(b_s + PL * 512);
    uint64_t* bars = reinterpret_cast<uint64_t*>(bias_s + kCh);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2);
    const uint32_t a_u = smem_u32(smem), b_u = smem_u32(b_s), bar0 = smem_u32(bars);
    const int warp = warp_uniform((int)threadIdx.x / 32);
    const ConvShape& sh = a.sh;
    const int opix = sh.OH * sh.OW;

    // inputs are read, and tensor memory taken, only once the previous kernel has finished,
    // as in every tcgen05 kernel of the library: a kernel may let its dependents launch before
    // it allocates, so one that allocated before its wait could hold columns its primary needs
    SQ_KERNEL_ENTRY();
    if (warp == 0) tmem_alloc(smem_u32(tmem_slot), 64);
    if (threadIdx.x == 0) {
        mbar_init(bar0, 1);
        mbar_init(bar0 + 8, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int e = threadIdx.x; e < 32 * PL; e += 128) {   // filter row co, 8 k-values of plane c
        const int co = e / PL, c = e % PL;
        __align__(16) __nv_bfloat16 hb[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = 8 * c + j;
            hb[j] = __float2bfloat16_rn(k < a.K ? a.w[(int64_t)co * a.K + k] : 0.f);
        }
        *reinterpret_cast<uint4*>(b_s + c * 512 + co * 16) = *reinterpret_cast<const uint4*>(hb);
    }
    if (threadIdx.x < kCh) bias_s[threadIdx.x] = a.bias[threadIdx.x];
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = warp_uniform(*tmem_slot);
    const int n_local = (int)blockIdx.x < a.n_tiles ? (a.n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int hw = sh.H * sh.W;
    bool ok = true;

    // this thread's pixel of tile t: its K inputs (loads issued, not yet waited for) ...
    auto load = [&](int t, float (&v)[8 * PL]) {
        const int64_t p = (int64_t)t * 128 + threadIdx.x;
        const bool valid = p < a.npix;
        const float* src = a.x;
        if (valid) {
            const int img = (int)(p / opix);
            const int rem = (int)(p - (int64_t)img * opix);
            const int oy = rem / sh.OW, ox = rem - oy * sh.OW;
            src += (int64_t)img * sh.x_img_stride + (int64_t)(oy * sh.stride) * sh.W + ox * sh.stride;
        }
#pragma unroll
        for (int k = 0; k < 8 * PL; ++k) {
            const int ci = k / 9, tap = k % 9;
            v[k] = (valid && k < a.K) ? __ldg(src + ci * hw + (tap / 3) * sh.W + tap % 3) : 0.f;
        }
    };
    // ... and written as BF16 into its row of A tile buffer b
    auto put = [&](int b, const float (&v)[8 * PL]) {
        uint8_t* dst = smem + b * kTile + threadIdx.x * 16;
#pragma unroll
        for (int c = 0; c < PL; ++c) {
            uint4 w4;
            w4.x = pack2_bf16(v[8 * c], v[8 * c + 1]);
            w4.y = pack2_bf16(v[8 * c + 2], v[8 * c + 3]);
            w4.z = pack2_bf16(v[8 * c + 4], v[8 * c + 5]);
            w4.w = pack2_bf16(v[8 * c + 6], v[8 * c + 7]);
            *reinterpret_cast<uint4*>(dst + c * 2048) = w4;
        }
    };
    // epilogue: this thread's accumulator row of tile t (buffer b) to its output pixel
    auto drain = [&](int t, int b) {
        uint32_t r0[16], r1[16];
        const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)b * kCh;
        tmem_ld16(taddr, r0);
        tmem_ld16(taddr + 16, r1);
        const int64_t p = (int64_t)t * 128 + threadIdx.x;
        if (p >= a.npix) return;
        const int img = (int)(p / opix);
        const int rem = (int)(p - (int64_t)img * opix);
        const int oy = rem / sh.OW, ox = rem - oy * sh.OW;
        uint4* dst = reinterpret_cast<uint4*>(
            a.out + (((int64_t)img * (sh.OH + 4) + oy + 2) * (sh.OW + 4) + ox + 2) * kCh);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float f[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int co = 8 * c + j;
                const float v = __uint_as_float(co < 16 ? r0[co] : r1[co - 16]) + bias_s[co];
                f[j] = v > 0.f ? v : 0.f;
            }
            uint4 w4;
            w4.x = pack2_bf16(f[0], f[1]);
            w4.y = pack2_bf16(f[2], f[3]);
            w4.z = pack2_bf16(f[4], f[5]);
            w4.w = pack2_bf16(f[6], f[7]);
            dst[c] = w4;
        }
    };

    constexpr uint32_t idesc = idesc_bf16(128, kCh, false, false);
    for (int i = 0; i < n_local; ++i) {
        const int t = (int)blockIdx.x + i * (int)gridDim.x, b = i & 1;
        float v[8 * PL];
        load(t, v);   // in flight while the previous tile drains
        if (i > 0 && ok) {
            // the MMAs of tile i - 1 (and so of tile i - 2, which read buffer b) are complete
            const int pb = b ^ 1;
            ok = __all_sync(0xffffffffu, mbar_wait(bar0 + 8 * pb, ((i - 1) >> 1) & 1, a.err, 17));
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (ok) drain(t - (int)gridDim.x, pb);
        }
        put(b, v);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (warp == 0 && elect_one()) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t a0 = plain_desc(a_u + b * kTile, 2048, 128), b0 = plain_desc(b_u, 512, 128);
#pragma unroll
            for (int kc = 0; kc < PL / 2; ++kc)
                mma_bf16(tmem + (uint32_t)b * kCh, a0 + (uint64_t)(kc * 256), b0 + (uint64_t)(kc * 64), idesc, kc > 0 ? 1u : 0u);
            mma_commit(bar0 + 8 * b);
        }
        __syncwarp();
    }
    if (n_local > 0) {
        const int i = n_local - 1, b = i & 1;
        if (__all_sync(0xffffffffu, mbar_wait(bar0 + 8 * b, (i >> 1) & 1, a.err, 18)) && ok) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            drain((int)blockIdx.x + i * (int)gridDim.x, b);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc(tmem, 64);
    }
}

// ---------------------------------------------------------------- the whole encoder forward
// Every layer of a 32-channel encoder (a first layer of at most 3 input channels and any
// stride, then stride-1 layers) in one launch: an image's activations go from layer to layer
// in shared memory, and only what is read later leaves it (the padded-HWC outputs of the first
// n_save images, the features of all).
//
// A CTA runs kEncGroups images at a time, each by a group of four warps with its own two
// activation buffers and tensor-memory columns: the group gathers the first layer's operand,
// and per layer one of its threads issues the layer's MMAs, all wait for them, and each thread
// takes its pixels out of tensor memory (bias, ReLU, BF16) into the other buffer.  The groups
// share nothing but the filters, which stay in shared memory, so one group's MMAs run under
// the others' epilogues.  Between the layers a plane holds its pixels densely, so an output
// grid is as wide as its input (fewer 128-row tiles than the padded rows: the last layer of a
// 32 x 32 input takes one instead of two).  The MMAs of an output and their order are those of
// conv0_tc_kernel and conv32_tc_kernel: the same bits.
//
// Bound by the shared-memory path that the MMAs' operands (5 KB an M = 128, N = 32 MMA, 94 of
// them an image at 32 x 32, 38 cycles each with four groups issuing) share with the gather and
// the epilogues: without the inner MMAs 4,096 images of 3 x 32 x 32 take 51 us, with them 84;
// 8 images 9.4 us, 1,024 with 512 saved 29 us.  The four launches it replaces: 207 us (act of
// 4,096 rows), 59 us (the update's 1,024 images).  Three groups measured 107 us, four 99, six
// (without the staged input) 93, before the issue loops became warp-uniform (103 -> 84).
constexpr int kEncGroups = 4;      // at most
constexpr int kEncMaxInner = 4;
constexpr int kEncTiles = 4;
// A layer's output grid: w columns computed (its input's width), of which ow and oh rows are
// real; 128-pixel tiles; 2^20 / w rounded up, which divides pixel numbers below 512 by w.
struct EncLayer { int w, oh, ow, tiles, inv; };
struct EncArgs {
    ConvShape sh;
    const float* x;
    const float* w0;
    const float* bias[kEncMaxInner + 1];
    const __nv_bfloat16* w[kEncMaxInner];     // layer l + 1, layout [tap][plane][out ch][8]
    EncLayer l[kEncMaxInner + 1];
    __nv_bfloat16* save[kEncMaxInner];        // padded-HWC output of layer l < n_inner (null: not kept)
    float* z;                                 // optional features [nimg, 32 oh ow], FP32 and BF16
    __nv_bfloat16* z_bf;
    int nimg, n_save, n_inner, K, groups, group_cols, cols;   // cols: all groups', a power of two
    uint32_t xbytes, ybytes, ibytes;   // of a group: the two activation buffers, an input image
    int* err;
};

// Inputs k = 16 HALF .. + 15, k = (ci, ky, kx), of first-layer output pixels tg, tg + 128, ... of
// the image at `in`, rounded to BF16, into planes of 8 k-values at `dst`.
template <int HALF>
__device__ __forceinline__ void gather_conv0(const EncArgs& a, const float* in, int tg, int hw, int opix, uint8_t* dst,
                                             uint32_t plane) {
    const ConvShape& sh = a.sh;
    for (int p = tg; p < opix; p += 128) {   // the last tile's other rows read what is there and are dropped
        const int oy = p * a.l[0].inv >> 20, ox = p - oy * sh.OW;
        const float* src = in + (oy * sh.stride) * sh.W + ox * sh.stride;
        float v[16];
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            const int k = 16 * HALF + kk, ci = k / 9, tap = k % 9;
            v[kk] = k < a.K ? src[ci * hw + (tap / 3) * sh.W + tap % 3] : 0.f;
        }
#pragma unroll
        for (int c = 0; c < 2; ++c)
            *reinterpret_cast<uint4*>(dst + (2 * HALF + c) * plane + p * 16) =
                make_uint4(pack2_bf16(v[8 * c], v[8 * c + 1]), pack2_bf16(v[8 * c + 2], v[8 * c + 3]),
                           pack2_bf16(v[8 * c + 4], v[8 * c + 5]), pack2_bf16(v[8 * c + 6], v[8 * c + 7]));
    }
}

__global__ void __launch_bounds__(128 * kEncGroups, 1) encoder_tc_kernel(const __grid_constant__ EncArgs a) {
    SQ_KERNEL_WAIT();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    const uint32_t group_bytes = a.xbytes + a.ybytes + a.ibytes;
    uint8_t* w_s = smem + a.groups * group_bytes;          // inner filters (reads past a buffer's planes end here)
    uint8_t* w0_s = w_s + a.n_inner * kWBytes;               // first filter: 4 planes of 32 rows x 16 B
    float* bias_s = reinterpret_cast<float*>(w0_s + 2048);
    uint64_t* bars = reinterpret_cast<uint64_t*>(bias_s + (kEncMaxInner + 1) * kCh);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + a.groups * (kEncTiles + 1) + 1);
    const int warp = warp_uniform((int)threadIdx.x / 32), g = warp / 4, quarter = warp % 4, tg = threadIdx.x % 128;
    const uint32_t bar = smem_u32(bars + g * (kEncTiles + 1)), ibar = bar + 8 * kEncTiles,
                   wbar = smem_u32(bars + a.groups * (kEncTiles + 1));
    const ConvShape& sh = a.sh;
    const int opix = sh.OH * sh.OW, hw = sh.H * sh.W;

    if (warp == 0) tmem_alloc(smem_u32(tmem_slot), a.cols);
    if (threadIdx.x == 0) {
        for (int b = 0; b <= a.groups * (kEncTiles + 1); ++b) mbar_init(smem_u32(bars + b), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(wbar, a.n_inner * kWBytes);
        for (int l = 0; l < a.n_inner; ++l) bulk_load(smem_u32(w_s) + l * kWBytes, a.w[l], kWBytes, wbar);
    }
    for (int e = threadIdx.x; e < 32 * 4; e += (int)blockDim.x) {
        const int co = e / 4, c = e % 4;
        __align__(16) __nv_bfloat16 hb[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = 8 * c + j;
            hb[j] = __float2bfloat16_rn(k < a.K ? a.w0[(int64_t)co * a.K + k] : 0.f);
        }
        *reinterpret_cast<uint4*>(w0_s + c * 512 + co * 16) = *reinterpret_cast<const uint4*>(hb);
    }
    for (int e = threadIdx.x; e < (a.n_inner + 1) * kCh; e += (int)blockDim.x) bias_s[e] = a.bias[e / kCh][e % kCh];
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t acc = warp_uniform(*tmem_slot) + (uint32_t)(g * a.group_cols);
    uint8_t* const bx = smem + g * group_bytes;
    uint8_t* const by = bx + a.xbytes;
    uint8_t* const bi = by + a.ybytes;
    const uint32_t plane0 = (uint32_t)opix * 16;
    constexpr uint32_t idesc = idesc_bf16(128, kCh, false, false);
    bool ok = mbar_wait(wbar, 0, a.err, 41);
    uint32_t phase = 0;   // bit t: parity of the barrier of tile t

    // the group's shared-memory writes and tensor-memory reads before the next MMAs
    auto group_sync = [&] {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory");
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    // one thread's bulk copy of an image's input, and all threads' first-layer operand from it; nothing
    // is copied or gathered once a wait has given up
    uint32_t iphase = 0;      // parity of the next copy to be waited for
    bool in_flight = false;   // (of the thread that copies)
    auto fetch = [&](int img) {
        if (!ok) return;
        mbar_expect_tx(ibar, a.ibytes);
        bulk_load(smem_u32(bi), a.x + (int64_t)img * sh.x_img_stride, a.ibytes, ibar);
        in_flight = true;
    };
    auto gather = [&] {
        ok = ok && mbar_wait(ibar, iphase, a.err, 44);
        if (ok) {
            iphase ^= 1;
            in_flight = false;
            gather_conv0<0>(a, reinterpret_cast<const float*>(bi), tg, hw, opix, bx, plane0);
            gather_conv0<1>(a, reinterpret_cast<const float*>(bi), tg, hw, opix, bx, plane0);
        }
        __syncwarp();
    };
    // this thread's pixels of a layer's output, tile by tile as the MMAs complete: bias, ReLU,
    // BF16, into `dst` (planes of oh ow pixels; unused for the last layer) and to global memory.
    // A wait that gives up stops this thread's further issue only (the commits go on, so
    // nobody waits for what was not issued).
    auto drain = [&](int img, int layer, uint8_t* dst, bool last) {
        const EncLayer& L = a.l[layer];
        const float4* bias = reinterpret_cast<const float4*>(bias_s + layer * kCh);
        for (int t = 0; t < L.tiles; ++t) {
            if (!mbar_wait(bar + 8 * t, (phase >> t) & 1, a.err, 42)) ok = false;
            phase ^= 1u << t;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int q = t * 128 + tg, y = q * L.inv >> 20, x = q - y * L.w;
#pragma unroll
            for (int half = 0; half < 2; ++half) {   // 16 channels at a time
                uint32_t r[16];
                tmem_ld16(acc + ((uint32_t)(quarter * 32) << 16) + t * kCh + 16 * half, r);
                if (y < L.oh && x < L.ow) {
                    float v[16];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float4 b = bias[4 * half + j];
                        v[4 * j] = fmaxf(__uint_as_float(r[4 * j]) + b.x, 0.f);
                        v[4 * j + 1] = fmaxf(__uint_as_float(r[4 * j + 1]) + b.y, 0.f);
                        v[4 * j + 2] = fmaxf(__uint_as_float(r[4 * j + 2]) + b.z, 0.f);
                        v[4 * j + 3] = fmaxf(__uint_as_float(r[4 * j + 3]) + b.w, 0.f);
                    }
                    const int px = L.oh * L.ow, row = y * L.ow + x;
                    if (!last) {
                        uint4 h[2];
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            h[c] = make_uint4(pack2_bf16(v[8 * c], v[8 * c + 1]), pack2_bf16(v[8 * c + 2], v[8 * c + 3]),
                                              pack2_bf16(v[8 * c + 4], v[8 * c + 5]), pack2_bf16(v[8 * c + 6], v[8 * c + 7]));
                            *reinterpret_cast<uint4*>(dst + ((2 * half + c) * px + row) * 16) = h[c];
                        }
                        if (img < a.n_save && a.save[layer]) {
                            uint4* out = reinterpret_cast<uint4*>(
                                a.save[layer] + (((int64_t)img * (L.oh + 4) + y + 2) * (L.ow + 4) + x + 2) * kCh + 16 * half);
                            out[0] = h[0];
                            out[1] = h[1];
                        }
                    } else {
                        const int64_t base = ((int64_t)img * kCh + 16 * half) * px + row;
                        if (a.z) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) a.z[base + j * px] = v[j];
                        }
                        if (a.z_bf) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) a.z_bf[base + j * px] = __float2bfloat16_rn(v[j]);
                        }
                    }
                }
                __syncwarp();   // tensor memory is read by whole warps: lanes without a pixel wait for the others
            }
        }
    };

    // images in turn over the CTAs, then over a CTA's groups
    const int step = (int)gridDim.x * a.groups;
    int img = (int)blockIdx.x + (int)gridDim.x * g;
    if (img < a.nimg) {
        if (quarter == 0 && elect_one()) fetch(img);
        __syncwarp();
        gather();
    }
    for (; img < a.nimg; img += step) {
        group_sync();   // (the input image has been read)
        if (quarter == 0 && elect_one()) {
            if (img + step < a.nimg) fetch(img + step);
            const uint64_t a0 = plain_desc(smem_u32(bx), plane0, 128), b0 = plain_desc(smem_u32(w0_s), 512, 128);
            for (int t = 0; t < a.l[0].tiles; ++t) {
                if (ok)
#pragma unroll
                    for (int kc = 0; kc < 2; ++kc)
                        mma_bf16(acc + t * kCh, a0 + (uint64_t)(2 * kc * (plane0 / 16) + t * 128), b0 + (uint64_t)(kc * 64),
                                 idesc, kc);
                mma_commit(bar + 8 * t);
            }
        }
        __syncwarp();
        drain(img, 0, by, false);
        for (int l = 1; l <= a.n_inner; ++l) {
            const EncLayer& L = a.l[l];
            const uint32_t plane = (uint32_t)(a.l[l - 1].oh * L.w) * 16;
            const bool last = l == a.n_inner;
            group_sync();
            if (quarter == 0 && elect_one()) {
                // descriptors of the first tap; starts move in 16-byte units within the 14-bit field
                const uint64_t a0 = plain_desc(smem_u32(l % 2 ? by : bx), plane, 128);
                const uint64_t b0 = plain_desc(smem_u32(w_s) + (l - 1) * kWBytes, 512, 128);
                for (int t = 0; t < L.tiles; ++t) {
                    if (ok)
#pragma unroll
                        for (int tap = 0; tap < 9; ++tap)
#pragma unroll
                            for (int kc = 0; kc < 2; ++kc)
                                mma_bf16(acc + t * kCh,
                                         a0 + (uint64_t)(2 * kc * (plane / 16) + t * 128 + (tap / 3) * L.w + tap % 3),
                                         b0 + (uint64_t)(tap * 128 + kc * 64), idesc, (tap | kc) ? 1u : 0u);
                    mma_commit(bar + 8 * t);
                }
            }
            __syncwarp();
            // the next image's operand while the last layer multiplies, where that reads the other buffer
            if (last && l % 2 == 1 && img + step < a.nimg) gather();
            drain(img, l, l % 2 ? bx : by, last);
            if (last && l % 2 == 0 && img + step < a.nimg) gather();
        }
    }
    SQ_KERNEL_TRIGGER();
    if (quarter == 0 && elect_one()) {   // every MMA this group issued has completed before the tensor memory is freed
        mma_commit(bar);
        mbar_wait(bar, phase & 1, a.err, 43);
        if (in_flight) mbar_wait(ibar, iphase, a.err, 45);   // (after a wait that gave up: copies land before the CTA ends)
    }
    if (threadIdx.x == 0 && !ok) mbar_wait(wbar, 0, a.err, 45);
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc(*tmem_slot, a.cols);
    }
}

// ---------------------------------------------------------------- layout conversions
// CHW FP32 (per image stride img_stride) -> padded HWC BF16 interior.
__global__ void to_phwc_kernel(const float* __restrict__ src, int64_t img_stride, int nimg, int H, int W,
                               __nv_bfloat16* __restrict__ dst) {
    SQ_KERNEL_ENTRY();
    const int64_t n = (int64_t)nimg * H * W;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int img = (int)(p / (H * W));
    const int rem = (int)(p - (int64_t)img * H * W);
    const int y = rem / W, x = rem - (rem / W) * W;
    const float* s = src + img * img_stride + rem;
    __nv_bfloat16* d = dst + ((int64_t)img * (H + 4) * (W + 4) + (int64_t)(y + 2) * (W + 4) + x + 2) * kCh;
    __align__(16) __nv_bfloat16 hb[kCh];
#pragma unroll
    for (int c = 0; c < kCh; ++c) hb[c] = __float2bfloat16_rn(s[(int64_t)c * H * W]);
#pragma unroll
    for (int c = 0; c < 4; ++c) reinterpret_cast<uint4*>(d)[c] = reinterpret_cast<const uint4*>(hb)[c];
}

// The same with the zero border and an optional ReLU mask, a thread a padded pixel: one pass
// where filling the buffer, masking and converting were three.
template <bool MASK>
__global__ void __launch_bounds__(128) to_phwc_whole_kernel(const float* __restrict__ src, const float* __restrict__ mask, int nimg,
                                                            int H, int W, __nv_bfloat16* __restrict__ dst) {
    SQ_KERNEL_ENTRY();
    const int wp = W + 4, pix = (H + 4) * wp;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= (int64_t)nimg * pix) return;
    const int img = (int)(p / pix), rem = (int)(p - (int64_t)img * pix);
    const int y = rem / wp - 2, x = rem - (rem / wp) * wp - 2;
    uint4* d = reinterpret_cast<uint4*>(dst + p * kCh);
    if (y < 0 || y >= H || x < 0 || x >= W) {
#pragma unroll
        for (int c = 0; c < 4; ++c) d[c] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    const int64_t at = (int64_t)img * kCh * H * W + y * W + x;
    float v[kCh];
#pragma unroll
    for (int c = 0; c < kCh; ++c) v[c] = src[at + (int64_t)c * H * W];
    if (MASK) {
        float m[kCh];
#pragma unroll
        for (int c = 0; c < kCh; ++c) m[c] = mask[at + (int64_t)c * H * W];
#pragma unroll
        for (int c = 0; c < kCh; ++c) v[c] = m[c] > 0.f ? v[c] : 0.f;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        d[c] = make_uint4(pack2_bf16(v[8 * c], v[8 * c + 1]), pack2_bf16(v[8 * c + 2], v[8 * c + 3]),
                          pack2_bf16(v[8 * c + 4], v[8 * c + 5]), pack2_bf16(v[8 * c + 6], v[8 * c + 7]));
}

// Padded HWC BF16 interior -> NCHW FP32.
__global__ void from_phwc_kernel(const __nv_bfloat16* __restrict__ src, int nimg, int H, int W, float* __restrict__ dst) {
    SQ_KERNEL_ENTRY();
    const int64_t n = (int64_t)nimg * kCh * H * W;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int img = (int)(e / ((int64_t)kCh * H * W));
    const int rem = (int)(e - (int64_t)img * kCh * H * W);
    const int c = rem / (H * W), p = rem - (rem / (H * W)) * (H * W);
    const int y = p / W, x = p - (p / W) * W;
    dst[e] = __bfloat162float(src[((int64_t)img * (H + 4) * (W + 4) + (int64_t)(y + 2) * (W + 4) + x + 2) * kCh + c]);
}

// FP32 filter w[co][ci][ky][kx] -> forward layout [tap][ci/8][co][ci%8] and data-gradient
// layout (tap' = 8 - tap, channels swapped) [tap'][co/8][ci][co%8].
__global__ void conv_weight_cast_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ fwd,
                                        __nv_bfloat16* __restrict__ bwd) {
    SQ_KERNEL_ENTRY();
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= kCh * kCh * 9) return;
    const int co = e / (kCh * 9), rem = e - co * kCh * 9, ci = rem / 9, tap = rem - (rem / 9) * 9;
    const __nv_bfloat16 v = __float2bfloat16_rn(w[e]);
    fwd[tap * kCh * kCh + (ci / 8) * kCh * 8 + co * 8 + (ci % 8)] = v;
    bwd[(8 - tap) * kCh * kCh + (co / 8) * kCh * 8 + ci * 8 + (co % 8)] = v;
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// Planes of a padded-HWC tensor: dims {8 channels, 4 planes, rows}, box {8, 1, 128}.
bool plane_map(CUtensorMap* m, const __nv_bfloat16* base, int64_t rows) {
    auto fn = encode_fn();
    if (!fn || (reinterpret_cast<uintptr_t>(base) & 15)) return false;
    cuuint64_t dims[3] = {8, 4, (cuuint64_t)rows};
    cuuint64_t strides[2] = {16, 64};
    cuuint32_t box[3] = {8, 1, 128};
    cuuint32_t estr[3] = {1, 1, 1};
    std::memset(m, 0, sizeof(*m));
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int round_up(int x, int m) { return (x + m - 1) / m * m; }

size_t conv_smem(int load_rows) { return 1024 + 2 * 4 * (size_t)load_rows * 16 + kWBytes + 10 * 8 + 16; }
constexpr int kEncSmem = 227 * 1024;
constexpr int kConvCtasPerSm = 2;   // resident CTAs per SM of the persistent convolution
int g_num_sms = 152;                 // set by conv_tc_prepare
size_t wgrad_smem(int slot_rows, int kq) {
    return 1024 + wgrad_operand_bytes(12 * (uint32_t)slot_rows * 16, 4 * (uint32_t)kq * 16) + 64 + 128 * 8 * 4 + 16;
}

}  // namespace

// Geometry of one call: the conv reads input rows up to (n_tiles * 128 - 1) + off0 + 2 Wp + 2.
int launch_conv32_tc(const ConvTc& c, int* err, cudaStream_t s) {
    if (c.nimg <= 0) return 0;
    ConvArgs a;
    std::memset(&a, 0, sizeof(a));
    const int mv = c.out_h * c.Wp;
    a.n_tiles = (mv + 127) / 128;
    if (a.n_tiles > 4) return -1;
    a.tmem_cols = a.n_tiles <= 1 ? 32 : (a.n_tiles <= 2 ? 64 : 128);
    const int max_row = a.n_tiles * 128 - 1 + c.off0 + 2 * c.Wp + 2;
    a.load_rows = round_up(max_row + 1, 128);
    if (conv_smem(a.load_rows) > 200 * 1024) return -1;
    if (!plane_map(&a.tin, c.in, (int64_t)c.nimg * c.in_rows)) return -2;
    a.w = c.w; a.nimg = c.nimg; a.in_rows = c.in_rows; a.Wp = c.Wp; a.out_h = c.out_h; a.out_w = c.out_w;
    a.off0 = c.off0; a.bias = c.bias; a.relu = c.relu; a.mask = c.mask; a.out_phwc = c.out_phwc;
    a.out_chw = c.out_chw; a.out_chw_bf = c.out_chw_bf; a.err = err;
    const size_t smem = conv_smem(a.load_rows);
    const int ctas = std::min(c.nimg, g_num_sms * kConvCtasPerSm);
    // more than two images a CTA: the chip is this kernel's
    if (c.nimg > 2 * g_num_sms * kConvCtasPerSm) launch_k(conv32_tc_alone_kernel, dim3(ctas), dim3(kConvThreads), smem, s, a);
    else launch_k(conv32_tc_kernel, dim3(ctas), dim3(kConvThreads), smem, s, a);
    return 0;
}

int64_t wgrad32_tc_workspace(int nimg) { return (int64_t)std::min(nimg, 148) * kCh * (kCh * 9 + 1); }

int wgrad32_per_cta(int nimg) {
    const int ctas = std::max(1, std::min(nimg, 148));
    return (nimg + ctas - 1) / ctas;
}

int launch_wgrad32_tc_partials(const WgradTc& c, int per_cta, float* work, int* err, cudaStream_t s) {
    if (c.nimg <= 0) return 0;
    if (per_cta < 1) return -1;
    WgradArgs a;
    std::memset(&a, 0, sizeof(a));
    a.kq = round_up(c.out_h * c.Wp, 16);
    // a slot covers the rows every K step of every vertical tap reads: kq + 2 Wp
    a.x_rows = a.kq + 2 * c.Wp;
    a.slot_rows = (a.x_rows + 5) / 8 * 8 + 2;
    if (wgrad_smem(a.slot_rows, a.kq) > 220 * 1024) a.slot_rows = a.x_rows;   // the largest images: any pitch that fits
    if (wgrad_smem(a.slot_rows, a.kq) > 220 * 1024 || (a.kq / 8) * 512 + 2048 > kDyBytesMax + 2048) return -1;
    if (reinterpret_cast<uintptr_t>(c.x) & 15) return -2;
    a.x = c.x;
    a.per_cta = per_cta;
    const int grid = (c.nimg + per_cta - 1) / per_cta;
    a.dy = c.dy; a.nimg = c.nimg; a.in_rows = c.in_rows; a.Wp = c.Wp; a.out_h = c.out_h; a.out_w = c.out_w;
    a.work = work; a.err = err;
    launch_k(wgrad32_tc_kernel, dim3(grid), dim3(kWgThreads), wgrad_smem(a.slot_rows, a.kq), s, a);
    return 0;
}

void launch_wgrad32_reduce(const float* work, int ctas, float* dw, float* db, cudaStream_t s) {
    launch_k(wgrad32_reduce_kernel, dim3((kCh * (kCh * 9 + 1) + 31) / 32), dim3(32 * kRed32Groups), 0, s, work, ctas,
             dw, db);
}

int launch_wgrad32_tc(const WgradTc& c, float* work, float* dw, float* db, int* err, cudaStream_t s) {
    if (c.nimg <= 0) return 0;
    const int pc = wgrad32_per_cta(c.nimg);
    const int rc = launch_wgrad32_tc_partials(c, pc, work, err, s);
    if (rc != 0) return rc;
    launch_wgrad32_reduce(work, (c.nimg + pc - 1) / pc, dw, db, s);
    return 0;
}

void conv_tc_prepare() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
        sms > 0)
        g_num_sms = sms;
    cudaFuncSetAttribute(conv32_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    cudaFuncSetAttribute(conv32_tc_alone_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    cudaFuncSetAttribute(wgrad32_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    cudaFuncSetAttribute(encoder_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kEncSmem);
    cudaFuncSetAttribute(conv0_tc_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
    cudaFuncSetAttribute(conv0_tc_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
    cudaFuncSetAttribute(conv0_tc_kernel<18>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
    encode_fn();
}

void launch_conv0_phwc(const ConvShape& sh, const float* x, const float* w, const float* b, __nv_bfloat16* out,
                       cudaStream_t s) {
    const int64_t npix = (int64_t)sh.nimg * sh.OH * sh.OW;
    if (npix <= 0) return;
    const size_t smem = ((size_t)sh.Cin * 9 * kCh + kCh) * sizeof(float);
    launch_k(conv0_phwc_kernel, dim3((unsigned)((npix + 511) / 512)), dim3(256), smem, s, sh, x, w, b, out);
}

namespace {
template <int PL>
size_t conv0_tc_smem() { return 128 + 2 * PL * 2048 + PL * 512 + kCh * 4 + 32; }
// CTAs per SM in the grid (each holds 64 tensor-memory columns, 512 per SM); the
// SQUINT_CONV0_CTAS environment variable (1..8) overrides it
int conv0_ctas_per_sm() {
    static int n = [] {
        const char* e = std::getenv("SQUINT_CONV0_CTAS");
        const int v = e ? std::atoi(e) : 4;
        return v >= 1 && v <= 8 ? v : 4;
    }();
    return n;
}
template <int PL>
void conv0_tc_go(const Conv0Args& a, cudaStream_t s) {
    // at least 28 KB of shared memory per CTA keeps at most 8 of them (8 x 64 columns) on an SM
    const size_t smem = std::max(conv0_tc_smem<PL>(), (size_t)28 * 1024 + 1);
    const int ctas = std::min(a.n_tiles, g_num_sms * conv0_ctas_per_sm());
    launch_k(conv0_tc_kernel<PL>, dim3(ctas), dim3(128), smem, s, a);
}
}  // namespace

int launch_conv0_tc(const ConvShape& sh, const float* x, const float* w, const float* b, __nv_bfloat16* out,
                    int* err, cudaStream_t s) {
    const int K = sh.Cin * 9;
    if (sh.Cout != kCh || K > 144 || sh.nimg < 0 || sh.stride < 1) return -1;
    const int64_t npix = (int64_t)sh.nimg * sh.OH * sh.OW;
    if (npix <= 0) return 0;
    Conv0Args a;
    std::memset(&a, 0, sizeof(a));
    a.sh = sh; a.x = x; a.w = w; a.bias = b; a.out = out; a.npix = npix; a.K = K; a.err = err;
    a.n_tiles = (int)((npix + 127) / 128);
    if (K <= 32) conv0_tc_go<4>(a, s);
    else if (K <= 64) conv0_tc_go<8>(a, s);
    else conv0_tc_go<18>(a, s);
    return 0;
}

namespace {
// The kernel's arguments and shared memory; false outside its range.
bool encoder_plan(const EncoderTc& c, EncArgs& a, size_t& smem) {
    const ConvShape& sh = c.sh;
    const int K = sh.Cin * 9;
    if (sh.Cout != kCh || K > 32 || c.n_inner < 1 || c.n_inner > kEncMaxInner || sh.nimg < 0) return false;
    std::memset(&a, 0, sizeof(a));
    a.sh = sh; a.x = c.x; a.w0 = c.w0; a.nimg = sh.nimg; a.n_save = c.n_save; a.n_inner = c.n_inner; a.K = K;
    a.z = c.z; a.z_bf = c.z_bf;
    auto layer = [](int w, int oh, int ow) { return EncLayer{w, oh, ow, (oh * w + 127) / 128, ((1 << 20) + w - 1) / w}; };
    a.l[0] = layer(sh.OW, sh.OH, sh.OW);
    a.xbytes = a.ybytes = (uint32_t)(sh.OH * sh.OW) * 64;
    a.ibytes = (uint32_t)(sh.Cin * sh.H * sh.W) * 4;
    if (sh.x_img_stride * 4 != (int64_t)a.ibytes || a.ibytes % 16 || (reinterpret_cast<uintptr_t>(c.x) & 15)) return false;
    a.bias[0] = c.bias[0];
    for (int l = 1; l <= c.n_inner; ++l) {
        const EncLayer& p = a.l[l - 1];
        if (p.oh < 3 || p.ow < 3 || (reinterpret_cast<uintptr_t>(c.w[l - 1]) & 15) || (reinterpret_cast<uintptr_t>(c.save[l - 1]) & 15))
            return false;
        a.l[l] = layer(p.ow, p.oh - 2, p.ow - 2);
        if (a.l[l].oh * (p.ow + 4) > 512) return false;   // a layer launch_conv32_tc refuses
        // layer l writes X for odd l, Y for even l; the last one leaves shared memory
        uint32_t& buf = l % 2 ? a.xbytes : a.ybytes;
        if (l < c.n_inner) buf = std::max(buf, (uint32_t)(a.l[l].oh * a.l[l].ow) * 64);
        a.w[l - 1] = c.w[l - 1]; a.bias[l] = c.bias[l]; a.save[l - 1] = c.save[l - 1];
    }
    const int tiles = a.l[0].tiles;   // the most of any layer
    // an MMA reads whole 128-row tiles at every tap: past the last plane it must end inside the filters
    if (tiles > kEncTiles || (tiles * 128 + 2 * sh.OW + 2) * 16 > kWBytes) return false;
    a.group_cols = kCh * tiles;
    const size_t fixed = 128 + (size_t)c.n_inner * kWBytes + 2048 + (kEncMaxInner + 1) * kCh * 4 + 8 + 16;
    const size_t group = a.xbytes + a.ybytes + a.ibytes + (kEncTiles + 1) * 8;
    if (fixed + group > kEncSmem) return false;
    a.groups = (int)std::min<size_t>(kEncGroups, (kEncSmem - fixed) / group);
    a.groups = std::min(a.groups, 512 / a.group_cols);
    // no more groups than the rounds of images need
    const int rounds = (sh.nimg + g_num_sms * a.groups - 1) / (g_num_sms * a.groups);
    while (a.groups > 1 && (sh.nimg + g_num_sms * (a.groups - 1) - 1) / (g_num_sms * (a.groups - 1)) == rounds) --a.groups;
    a.cols = 32;   // a power of two from 32 to 512
    while (a.cols < a.groups * a.group_cols) a.cols *= 2;
    smem = fixed + a.groups * group;
    return true;
}
}  // namespace

bool encoder_tc_fits(const EncoderTc& c) {
    EncArgs a;
    size_t smem;
    return encoder_plan(c, a, smem);
}

int launch_encoder_tc(const EncoderTc& c, int* err, cudaStream_t s) {
    EncArgs a;
    size_t smem;
    if (!encoder_plan(c, a, smem)) return -1;
    if (c.sh.nimg == 0) return 0;
    a.err = err;
    launch_k(encoder_tc_kernel, dim3(std::min(c.sh.nimg, g_num_sms)), dim3(128 * a.groups), smem, s, a);
    return 0;
}

void launch_to_phwc(const float* src, int64_t img_stride, int nimg, int H, int W, __nv_bfloat16* dst, cudaStream_t s) {
    const int64_t n = (int64_t)nimg * H * W;
    if (n) launch_k(to_phwc_kernel, dim3((unsigned)((n + 127) / 128)), dim3(128), 0, s, src, img_stride, nimg, H, W, dst);
}
void launch_to_phwc_whole(const float* src, const float* mask, int nimg, int H, int W, __nv_bfloat16* dst, cudaStream_t s) {
    const int64_t n = (int64_t)nimg * (H + 4) * (W + 4);
    if (n <= 0) return;
    const dim3 grid((unsigned)((n + 127) / 128));
    if (mask) launch_k(to_phwc_whole_kernel<true>, grid, dim3(128), 0, s, src, mask, nimg, H, W, dst);
    else launch_k(to_phwc_whole_kernel<false>, grid, dim3(128), 0, s, src, mask, nimg, H, W, dst);
}
void launch_from_phwc(const __nv_bfloat16* src, int nimg, int H, int W, float* dst, cudaStream_t s) {
    const int64_t n = (int64_t)nimg * kCh * H * W;
    if (n) launch_k(from_phwc_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, s, src, nimg, H, W, dst);
}
void launch_conv_weight_cast(const float* w, __nv_bfloat16* fwd, __nv_bfloat16* bwd, cudaStream_t s) {
    launch_k(conv_weight_cast_kernel, dim3((kCh * kCh * 9 + 255) / 256), dim3(256), 0, s, w, fwd, bwd);
}

}  // namespace sq
