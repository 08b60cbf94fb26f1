// FP32 valid 3x3 convolutions on CUDA cores: forward, data gradient and weight gradient of
// the plain FP32 path's encoder.
//
// What bounds them: the FP32 FMA rate.  The input rows of a tile of output pixels are copied
// once into shared memory, plane by plane (cp.async, in a ring, so that the copies overlap
// the arithmetic), and every tap reads them there: no per-tap index arithmetic, no nine-fold
// gather.  A tile's pixels may cross rows and images: each image it touches brings the rows
// it needs.  Every output is one chain of fused multiply-adds in the order of conv_fwd_kernel,
// conv_dgrad_kernel and conv_wgrad_kernel (sq_gemm.cu), so the results are the same bits.
// 512 images of 32 x 15 x 15 to 32 channels, stride 1 (floor 19.8 us at one FMA per lane and
// cycle; before, there, and now): forward 98 and 53 us, data gradient 190 and 77 us, weight
// gradient 375 and 105 us.
#include "sq_kernels.cuh"

#include <algorithm>

namespace sq {
namespace {

constexpr int kSmemBytes = 48 * 1024;   // no opt-in, on any device
constexpr int kChan = 4;                // planes a stage of conv_f32_kernel
constexpr int kWRow = 36;               // floats a weight row (32 output channels) takes

__device__ __forceinline__ void copy4(float* dst, const float* src, bool valid) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// Output grid of oh x ow pixels an image; output row r reads staged rows r rs .. r rs + 2 of
// a plane pw wide.
struct PixelGrid { int oh, ow, rs, pw; };

// What output pixels [m0, m1) of the flattened (image, row, column) order read: of the first
// image the rows from its first pixel on, of the others the rows from 0.
struct Region {
    int img0, row0, first, full, words;   // first image, its first output row, staged words: first image, a whole image, all
    __device__ __forceinline__ Region(const PixelGrid& g, int m0, int m1) {
        const int px = g.oh * g.ow;
        img0 = m0 / px;
        row0 = (m0 - img0 * px) / g.ow;
        const int img1 = (m1 - 1) / px, row1 = ((m1 - 1) - img1 * px) / g.ow;
        full = ((g.oh - 1) * g.rs + 3) * g.pw;
        if (img1 == img0) {
            first = words = ((row1 - row0) * g.rs + 3) * g.pw;
        } else {
            first = ((g.oh - 1 - row0) * g.rs + 3) * g.pw;
            words = first + (img1 - img0 - 1) * full + (row1 * g.rs + 3) * g.pw;
        }
    }
    __device__ __forceinline__ int pixel(const PixelGrid& g, int img, int oy, int ox) const {
        return (img == img0 ? (oy - row0) * g.rs * g.pw : first + (img - img0 - 1) * full + oy * g.rs * g.pw) + ox * g.rs;
    }
    // image (relative to img0) and staged row of a word
    __device__ __forceinline__ void place(const PixelGrid& g, int w, int& img, int& row, int& col) const {
        const int r = w / g.pw;
        col = w - r * g.pw;
        if (w < first) {
            img = 0;
            row = row0 * g.rs + r;
        } else {
            const int v = w - first, q = v / full;
            img = q + 1;
            row = (v - q * full) / g.pw;
        }
    }
};
// Most words a region of m pixels can take.
int64_t region_words(const PixelGrid& g, int m) {
    const int64_t rows = (m - 1 + g.ow - 1) / g.ow + 1, pieces = (m - 1 + g.oh * g.ow - 1) / (g.oh * g.ow) + 1;
    return (rows * g.rs + std::max(0, 3 - g.rs) * pieces) * g.pw;
}

struct ConvF32Args {
    const float* in;      // forward: x; data gradient: dy
    const float* w;       // [Cout, Cin, 3, 3]
    const float* bias;    // forward
    const float* mask;    // data gradient, optional
    float* out;
    PixelGrid g;
    int M, N, R;          // output pixels, output channels, reduced channels
    int64_t in_img, in_plane, out_img;
    int relu, words, stages;
    // data gradient: dy is oh2 x ow2 and staged with stride - 1 zeros between its elements and
    // two zeros around them
    int stride, oh2, ow2;
};

// 32 P pixels x 32 output channels a CTA, P pixels (32 apart) x 8 channels a thread: at P = 4,
// 6 shared-memory reads (4 inputs, two broadcast 16-byte weights) per 32 FMAs; the FMA pipe is
// 46 % busy, the issue slots 77 %.
template <int P, bool DGRAD>
__global__ void __launch_bounds__(128) conv_f32_kernel(const __grid_constant__ ConvF32Args a) {
    SQ_KERNEL_WAIT();
    extern __shared__ __align__(16) float smem[];
    const int nt = blockDim.x, tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const int m0 = blockIdx.x * 32 * P, m1 = min(a.M, m0 + 32 * P), n0 = blockIdx.y * 32;
    const Region rg(a.g, m0, m1);
    const int xwords = kChan * a.words, stage_words = kChan * 9 * kWRow + (xwords + 3) / 4 * 4;
    int* woff = reinterpret_cast<int*>(smem + a.stages * stage_words);
    for (int w = tid; w < rg.words; w += nt) {
        int img, row, col;
        rg.place(a.g, w, img, row, col);
        int off = -1;
        if (!DGRAD) {
            off = (int)(img * a.in_img) + row * a.g.pw + col;
        } else {
            const int r = row - 2, c = col - 2, oy = r / a.stride, ox = c / a.stride;
            if (r >= 0 && c >= 0 && oy * a.stride == r && ox * a.stride == c && oy < a.oh2 && ox < a.ow2)
                off = (int)(img * a.in_img) + oy * a.ow2 + ox;
        }
        woff[w] = off;
    }
    __syncthreads();
    const float* in0 = a.in + (int64_t)rg.img0 * a.in_img;
    const int steps = (a.R + kChan - 1) / kChan;
    auto stage = [&](int st) {
        if (st < steps) {
            float* sw = smem + (st % a.stages) * stage_words;
            float* sx = sw + kChan * 9 * kWRow;
            const int c0 = st * kChan, nc = min(kChan, a.R - c0);
            for (int e = tid; e < kChan * 9 * 32; e += nt) {
                int n, k;
                const float* src;
                if (!DGRAD) {
                    n = e / (kChan * 9);
                    k = e - n * (kChan * 9);
                    src = a.w + ((int64_t)(n0 + n) * a.R + c0) * 9 + k;
                } else {
                    const int c = e / (32 * 9), nr = e - c * (32 * 9), r = nr % 9;
                    n = nr / 9;
                    k = c * 9 + r;
                    src = a.w + ((int64_t)(c0 + c) * a.N + n0 + n) * 9 + r;
                }
                const bool ok = n0 + n < a.N && k < nc * 9;
                copy4(sw + k * kWRow + n, ok ? src : a.w, ok);
            }
            const float* src0 = in0 + (int64_t)c0 * a.in_plane;
            for (int w = tid; w < rg.words; w += nt) {
                const int off = woff[w];
                const float* src = src0 + (off < 0 ? 0 : off);
#pragma unroll
                for (int c = 0; c < kChan; ++c)
                    if (c < nc) copy4(sx + c * a.words + w, src + c * a.in_plane, off >= 0);
            }
        }
        copies_commit();
    };
    for (int st = 0; st + 1 < a.stages; ++st) stage(st);

    int base[P];
    const int px = a.g.oh * a.g.ow;
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const int m = min(m0 + lane + 32 * i, a.M - 1);
        const int img = m / px, rem = m - img * px, oy = rem / a.g.ow;
        base[i] = m < m1 ? rg.pixel(a.g, img, oy, rem - oy * a.g.ow) : 0;
    }
    float acc[P][8];
#pragma unroll
    for (int i = 0; i < P; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;

    for (int st = 0; st < steps; ++st) {
        if (a.stages == 2) asm volatile("cp.async.wait_group 0;" ::: "memory");
        else asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();   // this stage has landed, the previous one has been read
        stage(st + a.stages - 1);
        const float* sw = smem + (st % a.stages) * stage_words + warp * 8;
        const float* sx = smem + (st % a.stages) * stage_words + kChan * 9 * kWRow;
        const int nc = min(kChan, a.R - st * kChan);
        for (int c = 0; c < nc; ++c, sx += a.words, sw += 9 * kWRow) {
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
                const float* row = sx + (DGRAD ? 2 - ky : ky) * a.g.pw;
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) {
                    const float4 w0 = *reinterpret_cast<const float4*>(sw + (ky * 3 + kx) * kWRow);
                    const float4 w1 = *reinterpret_cast<const float4*>(sw + (ky * 3 + kx) * kWRow + 4);
                    const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
                    for (int i = 0; i < P; ++i) {
                        const float x = row[base[i] + (DGRAD ? 2 - kx : kx)];
#pragma unroll
                        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(x, wv[j], acc[i][j]);
                    }
                }
            }
        }
    }
    SQ_KERNEL_TRIGGER();
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const int m = m0 + lane + 32 * i;
        if (m >= m1) continue;
        const int img = m / px, rem = m - img * px;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int n = n0 + warp * 8 + j;
            if (n >= a.N) continue;
            const int64_t off = (int64_t)img * a.out_img + (int64_t)n * px + rem;
            float v = acc[i][j];
            if (!DGRAD) {
                v += a.bias[n];
                if (a.relu && !(v > 0.f)) v = 0.f;
            } else if (a.mask && !(a.mask[off] > 0.f)) {
                v = 0.f;
            }
            a.out[off] = v;
        }
    }
}

template <bool DGRAD>
bool launch_conv(ConvF32Args a, cudaStream_t s) {
    const int ny = (a.N + 31) / 32, threads = 32 * std::min(4, (a.N + 7) / 8);
    // P: 53 us at 4, 57 at 8, 62 at 2, 88 at 1 for the shape above; fewer pixels a thread where
    // the CTAs would not fill two per SM (32 images of 16 x 7 x 7: 13.2, 9.4 and 8.0 us at 4, 2, 1)
    int p = 4;
    while (p > 1 && (int64_t)((a.M + 32 * p - 1) / (32 * p)) * ny < 2 * 152) p /= 2;
    for (; p >= 1; p /= 2) {
        const int64_t words = region_words(a.g, 32 * p);
        const int64_t pieces = (32 * p - 1 + a.g.oh * a.g.ow - 1) / (a.g.oh * a.g.ow) + 1;
        if (words > kSmemBytes / 4 || pieces * a.in_img >= (1LL << 31)) continue;
        a.words = (int)words;
        const int64_t stage = 4 * (kChan * 9 * kWRow + (kChan * words + 3) / 4 * 4), table = 4 * words;
        a.stages = 3 * stage + table <= kSmemBytes ? 3 : 2;
        const int64_t bytes = a.stages * stage + table;
        if (bytes > kSmemBytes) continue;
        const dim3 grid((a.M + 32 * p - 1) / (32 * p), ny), block(threads);
        switch (p) {
            case 4: launch_k(conv_f32_kernel<4, DGRAD>, grid, block, (size_t)bytes, s, a); break;
            case 2: launch_k(conv_f32_kernel<2, DGRAD>, grid, block, (size_t)bytes, s, a); break;
            default: launch_k(conv_f32_kernel<1, DGRAD>, grid, block, (size_t)bytes, s, a); break;
        }
        return true;
    }
    return false;
}

// ---------------------------------------------------------------- weight gradient
// Split z of the pixels, CI input channels x 32 output channels a CTA: a thread owns CO output
// channels x the nine taps of one input channel and walks the split's pixels in order.  Along
// an output row of a stride-1 layer the taps' inputs slide: three new values a pixel.  Bound by
// issue (half of it staging and row bookkeeping) at 1.6 warps a scheduler: the splits, which fix
// the order of the sums, give 61 chunks x 4 groups of 8 input channels.  8 x 2 channels a thread
// pair measured 105 us, 8 x 4 115, 4 x 2 116 (the shape above).
constexpr int kWTile = 64;   // pixels a stage
struct WgradF32Args {
    const float *x, *dy;
    float* work;
    PixelGrid g;
    int P, Cin, Cout, chunk, words;
    int64_t x_img, x_plane, y_img;
};

// NP consecutive pixels of an output row from pixel u on: all their reads, then their products.
template <int NP, int CO, bool SLIDE, int DROW>
__device__ __forceinline__ void pixels(float (&acc)[CO][9], float (&bacc)[CO], bool bias, float (&edge)[3][2],
                                       const float* row, const float* drow, int u, const PixelGrid& g) {
    float x[NP][9], d[NP][CO];
#pragma unroll
    for (int v = 0; v < NP; ++v) {
        const float* dp = drow + (u + v) * DROW;
        if (CO == 4) {
            const float4 t = *reinterpret_cast<const float4*>(dp);
            d[v][0] = t.x; d[v][1] = t.y; d[v][2 % CO] = t.z; d[v][3 % CO] = t.w;
        } else {
            const float2 t = *reinterpret_cast<const float2*>(dp);
            d[v][0] = t.x; d[v][1] = t.y;
        }
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
            for (int kx = SLIDE ? 2 : 0; kx < 3; ++kx) x[v][ky * 3 + kx] = row[ky * g.pw + (u + v) * g.rs + kx];
    }
    if (SLIDE) {
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
#pragma unroll
            for (int v = 0; v < NP; ++v) {
                x[v][ky * 3] = v >= 2 ? x[v >= 2 ? v - 2 : 0][ky * 3 + 2] : edge[ky][v >= 2 ? 0 : v];
                x[v][ky * 3 + 1] = v >= 1 ? x[v >= 1 ? v - 1 : 0][ky * 3 + 2] : edge[ky][1];
            }
            edge[ky][0] = NP >= 2 ? x[NP >= 2 ? NP - 2 : 0][ky * 3 + 2] : edge[ky][1];
            edge[ky][1] = x[NP - 1][ky * 3 + 2];
        }
    }
#pragma unroll
    for (int v = 0; v < NP; ++v) {
#pragma unroll
        for (int k = 0; k < CO; ++k)
#pragma unroll
            for (int r = 0; r < 9; ++r) acc[k][r] = fmaf(d[v][k], x[v][r], acc[k][r]);
        if (bias)
#pragma unroll
            for (int k = 0; k < CO; ++k) bacc[k] += d[v][k];
    }
}

template <int CI, int CO, bool SLIDE>
__global__ void __launch_bounds__(CI * 32 / CO) wgrad_f32_kernel(const __grid_constant__ WgradF32Args a) {
    static_assert(CI * 32 / CO % kWTile == 0, "whole pixels a pass");
    constexpr int NT = CI * 32 / CO, DROW = CO == 4 ? 36 : 34;
    SQ_KERNEL_WAIT();
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, cg = tid % (32 / CO), ci_l = tid / (32 / CO);
    const int c0 = blockIdx.x * CI, co0 = blockIdx.y * 32, nci = min(CI, a.Cin - c0);
    const int p_begin = blockIdx.z * a.chunk, p_end = min(a.P, p_begin + a.chunk);
    const int px = a.g.oh * a.g.ow;
    const int stage_words = kWTile * DROW + (CI * a.words + 3) / 4 * 4;
    auto stage = [&](int t) {
        const int q0 = p_begin + t * kWTile, q1 = min(p_end, q0 + kWTile);
        if (q0 < q1) {
            float* sd = smem + (t & 1) * stage_words;
            float* sx = sd + kWTile * DROW;
            // a thread copies one pixel's gradients of every NT / kWTile-th channel
            const int pl = tid % kWTile, p = q0 + pl, img = p / px;
            const float* src = a.dy + (int64_t)img * a.y_img + (int64_t)co0 * px + (p - img * px);
            float* dst = sd + pl * DROW;
#pragma unroll 4
            for (int co = tid / kWTile; co < 32; co += NT / kWTile) {
                const bool ok = p < q1 && co0 + co < a.Cout;
                copy4(dst + co, ok ? src + (int64_t)co * px : a.dy, ok);
            }
            const Region rg(a.g, q0, q1);
            const float* x0 = a.x + (int64_t)rg.img0 * a.x_img + (int64_t)c0 * a.x_plane;
            for (int w = tid; w < rg.words; w += NT) {
                int img, row, col;
                rg.place(a.g, w, img, row, col);
                const float* xs = x0 + (int64_t)img * a.x_img + (int64_t)row * a.g.pw + col;
#pragma unroll 4
                for (int c = 0; c < nci; ++c) copy4(sx + c * a.words + w, xs + c * a.x_plane, true);
            }
        }
        copies_commit();
    };
    float acc[CO][9], bacc[CO];
#pragma unroll
    for (int k = 0; k < CO; ++k) {
        bacc[k] = 0.f;
#pragma unroll
        for (int r = 0; r < 9; ++r) acc[k][r] = 0.f;
    }
    const bool bias = blockIdx.x == 0;
    const int tiles = (p_end - p_begin + kWTile - 1) / kWTile;
    stage(0);
    for (int t = 0; t < tiles; ++t) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();   // this stage has landed, the other one has been read
        stage(t + 1);
        const float* sd = smem + (t & 1) * stage_words + cg * CO;
        const float* sx = smem + (t & 1) * stage_words + kWTile * DROW + (ci_l < nci ? ci_l : 0) * a.words;
        const int q0 = p_begin + t * kWTile, q1 = min(p_end, q0 + kWTile);
        const Region rg(a.g, q0, q1);
        int img = rg.img0, oy = rg.row0, ox = (q0 - img * px) - oy * a.g.ow;
        for (int q = q0; q < q1;) {   // one run of pixels of an output row
            const int run = min(a.g.ow - ox, q1 - q);
            const float* row = sx + rg.pixel(a.g, img, oy, ox);
            const float* drow = sd + (q - q0) * DROW;
            float edge[3][2];   // the first two columns of the next pixel's taps
            if (SLIDE) {
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) {
                    edge[ky][0] = row[ky * a.g.pw];
                    edge[ky][1] = row[ky * a.g.pw + 1];
                }
            }
            int u = 0;
            for (; u + 4 <= run; u += 4) pixels<4, CO, SLIDE, DROW>(acc, bacc, bias, edge, row, drow, u, a.g);
            for (; u < run; ++u) pixels<1, CO, SLIDE, DROW>(acc, bacc, bias, edge, row, drow, u, a.g);
            q += run;
            ox = 0;
            if (++oy == a.g.oh) { oy = 0; ++img; }
        }
    }
    SQ_KERNEL_TRIGGER();
    const int N = a.Cin * 9 + 1;
    float* out = a.work + (int64_t)blockIdx.z * a.Cout * N;
#pragma unroll
    for (int k = 0; k < CO; ++k) {
        const int co = co0 + cg * CO + k;
        if (co >= a.Cout) continue;
        if (ci_l < nci) {
#pragma unroll
            for (int r = 0; r < 9; ++r) out[(int64_t)co * N + (c0 + ci_l) * 9 + r] = acc[k][r];
        }
        if (bias && ci_l == 0) out[(int64_t)co * N + N - 1] = bacc[k];
    }
}

template <int CI, int CO, bool SLIDE>
bool launch_wgrad(WgradF32Args a, int splits, cudaStream_t s) {
    constexpr int DROW = CO == 4 ? 36 : 34;
    const int64_t words = region_words(a.g, kWTile);
    const int64_t bytes = 8 * (kWTile * DROW + (CI * words + 3) / 4 * 4);
    if (bytes > kSmemBytes) return false;
    a.words = (int)words;
    launch_with(false, wgrad_f32_kernel<CI, CO, SLIDE>, dim3((a.Cin + CI - 1) / CI, (a.Cout + 31) / 32, splits), dim3(CI * 32 / CO),
             (size_t)bytes, s, a);
    return true;
}

}  // namespace

bool launch_conv_fwd_f32(const ConvShape& sh, const float* x, const float* w, const float* b, float* y, bool relu,
                         cudaStream_t s) {
    ConvF32Args a{};
    a.in = x; a.w = w; a.bias = b; a.out = y;
    a.g = PixelGrid{sh.OH, sh.OW, sh.stride, sh.W};
    a.M = sh.nimg * sh.OH * sh.OW; a.N = sh.Cout; a.R = sh.Cin;
    a.in_img = sh.x_img_stride; a.in_plane = (int64_t)sh.H * sh.W; a.out_img = sh.y_img_stride;
    a.relu = relu ? 1 : 0; a.stride = sh.stride;
    return launch_conv<false>(a, s);
}

bool launch_conv_dgrad_f32(const ConvShape& sh, const float* dy, const float* w, float* dx, const float* mask,
                           cudaStream_t s) {
    ConvF32Args a{};
    a.in = dy; a.w = w; a.mask = mask; a.out = dx;
    a.g = PixelGrid{sh.H, sh.W, 1, sh.W + 2};
    a.M = sh.nimg * sh.H * sh.W; a.N = sh.Cin; a.R = sh.Cout;
    a.in_img = sh.y_img_stride; a.in_plane = (int64_t)sh.OH * sh.OW; a.out_img = sh.x_img_stride;
    a.stride = sh.stride; a.oh2 = sh.OH; a.ow2 = sh.OW;
    return launch_conv<true>(a, s);
}

bool launch_conv_wgrad_partials_f32(const ConvShape& sh, const float* dy, const float* x, float* work, int splits,
                                    int chunk, cudaStream_t s) {
    WgradF32Args a{};
    a.x = x; a.dy = dy; a.work = work;
    a.g = PixelGrid{sh.OH, sh.OW, sh.stride, sh.W};
    a.P = sh.nimg * sh.OH * sh.OW; a.Cin = sh.Cin; a.Cout = sh.Cout; a.chunk = chunk;
    a.x_img = sh.x_img_stride; a.x_plane = (int64_t)sh.H * sh.W; a.y_img = sh.y_img_stride;
    if (sh.stride == 1) return sh.Cin > 4 ? launch_wgrad<8, 2, true>(a, splits, s) : launch_wgrad<4, 2, true>(a, splits, s);
    return sh.Cin > 4 ? launch_wgrad<8, 2, false>(a, splits, s) : launch_wgrad<4, 2, false>(a, splits, s);
}

}  // namespace sq
