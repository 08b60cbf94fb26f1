// FP32 valid 3x3 convolutions on CUDA cores: forward, data gradient and weight gradient of
// the plain FP32 path's encoder.
//
// What bounds them: forward and data gradient the shared-memory read path (60-73 % busy beside an FMA
// pipe at 45-55 %: the two broadcast weight reads and the input reads of a tap take more of its cycles
// than the products take of theirs), the weight gradient the one multiplying warp a scheduler that its
// splits leave.  The FMA rate is the floor.  The input rows of a tile of output pixels are copied
// once into shared memory, plane by plane (cp.async, in a ring, so that the copies overlap
// the arithmetic), and every tap reads them there: no per-tap index arithmetic, no nine-fold
// gather.  A tile's pixels may cross rows and images: each image it touches brings the rows
// it needs.  Every output is one chain of fused multiply-adds in the order of conv_fwd_kernel,
// conv_dgrad_kernel and conv_wgrad_kernel (sq_gemm.cu), so the results are the same bits.
// 512 images of 32 x 15 x 15 to 32 channels, stride 1 (floor 19.8 us at one FMA per lane and
// cycle; before, there, and now): forward 98 and 53 us, data gradient 190 and 72 us, weight
// gradient 375 and 82 us.
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

template <int N>
__device__ __forceinline__ float half_of(const uint64_t (&v)[N], int i) {
    return __uint_as_float((uint32_t)(v[i / 2] >> (32 * (i % 2))));
}

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
// 6 shared-memory reads (4 inputs, two broadcast 16-byte weights) per 32 products, issued in
// pairs (one by one: forward 53.6 us and 53.1 now, data gradient 78 and 72).
// COPY threads stage, as in the weight gradient, beside those that multiply; with none all do both.
// A small grid runs faster with them (32 images of 16 x 7 x 7, P = 1: forward 8.0 and 5.8 us, data
// gradient 10.6 and 7.6), a full one has other warps to issue meanwhile (P = 4: 53 and 58 us).
template <int P, int COPY, bool DGRAD>
__global__ void __launch_bounds__(128 + COPY) conv_f32_kernel(const __grid_constant__ ConvF32Args a) {
    SQ_KERNEL_WAIT();
    extern __shared__ __align__(16) float smem[];
    const int nt = blockDim.x, nm = nt - COPY, tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
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
    const int ct = COPY ? tid - nm : tid, nc_t = COPY ? COPY : nt;   // place among the staging threads, their number
    auto stage = [&](int st) {
        if (st < steps) {
            float* sw = smem + (st % a.stages) * stage_words;
            float* sx = sw + kChan * 9 * kWRow;
            const int c0 = st * kChan, nc = min(kChan, a.R - c0);
            for (int e = ct; e < kChan * 9 * 32; e += nc_t) {
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
            for (int w = ct; w < rg.words; w += nc_t) {
                const int off = woff[w];
                const float* src = src0 + (off < 0 ? 0 : off);
#pragma unroll
                for (int c = 0; c < kChan; ++c)
                    if (c < nc) copy4(sx + c * a.words + w, src + c * a.in_plane, off >= 0);
            }
        }
        copies_commit();
    };
    auto next_stage = [&](int st) {
        if (a.stages == 2) asm volatile("cp.async.wait_group 0;" ::: "memory");
        else asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();   // this stage has landed, the previous one has been read
        stage(st + a.stages - 1);
    };
    if (!COPY || tid >= nm)
        for (int st = 0; st + 1 < a.stages; ++st) stage(st);
    if (COPY && tid >= nm) {
        for (int st = 0; st < steps; ++st) next_stage(st);
        SQ_KERNEL_TRIGGER();
        return;
    }

    int base[P];
    const int px = a.g.oh * a.g.ow;
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const int m = min(m0 + lane + 32 * i, a.M - 1);
        const int img = m / px, rem = m - img * px, oy = rem / a.g.ow;
        base[i] = m < m1 ? rg.pixel(a.g, img, oy, rem - oy * a.g.ow) : 0;
    }
    uint64_t acc[P][4];   // channel pairs
#pragma unroll
    for (int i = 0; i < P; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0;

    for (int st = 0; st < steps; ++st) {
        if (COPY) __syncthreads();
        else next_stage(st);
        const float* sw = smem + (st % a.stages) * stage_words + warp * 8;
        const float* sx = smem + (st % a.stages) * stage_words + kChan * 9 * kWRow;
        const int nc = min(kChan, a.R - st * kChan);
        for (int c = 0; c < nc; ++c, sx += a.words, sw += 9 * kWRow) {
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
                const float* row = sx + (DGRAD ? 2 - ky : ky) * a.g.pw;
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) {
                    const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(sw + (ky * 3 + kx) * kWRow);
                    const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(sw + (ky * 3 + kx) * kWRow + 4);
                    const uint64_t wv[4] = {w0.x, w0.y, w1.x, w1.y};
#pragma unroll
                    for (int i = 0; i < P; ++i) {
                        const uint64_t x = both(row[base[i] + (DGRAD ? 2 - kx : kx)]);
#pragma unroll
                        for (int j = 0; j < 4; ++j) fma_pair(acc[i][j], wv[j], x);
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
            float v = half_of(acc[i], j);
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
    // the CTAs would not fill two per SM (32 images of 16 x 7 x 7: 13.2, 7.2 and 5.8 us at 4, 2, 1)
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
        const dim3 grid((a.M + 32 * p - 1) / (32 * p), ny), block(threads + (p < 4 ? 128 : 0));
        switch (p) {
            case 4: launch_k(conv_f32_kernel<4, 0, DGRAD>, grid, block, (size_t)bytes, s, a); break;
            case 2: launch_k(conv_f32_kernel<2, 128, DGRAD>, grid, block, (size_t)bytes, s, a); break;
            default: launch_k(conv_f32_kernel<1, 128, DGRAD>, grid, block, (size_t)bytes, s, a); break;
        }
        return true;
    }
    return false;
}

// ---------------------------------------------------------------- weight gradient
// Split z of the pixels, CI input channels x 32 output channels a CTA: a thread owns CO output
// channels x the nine taps of one input channel and walks the split's pixels in order, four of an
// output row at a time.  Half of the warps stage: the copies, 4 bytes each because a plane's rows
// have no alignment, then cost the others no issue slots (one kind of warp: 98 us for the shape
// above, so 82).  Input rows are staged so that a group's new columns start at a multiple of four,
// the two before them stay in registers, and the next group is read while one is multiplied; products
// are issued in pairs of output channels (one by one 86 us).
// What bounds it: the splits, which fix the order of the sums, leave one multiplying warp a
// scheduler (61 chunks x 2 groups of 16 input channels), so what a row's ends cost shows; of the
// 82 us the staging is 8.
struct WgradF32Args {
    const float *x, *dy;
    float* work;
    int oh, ow, pw;       // output rows and columns, input columns
    int P, Cin, Cout, chunk;
    int nr, xrows, xp, dp, stages;   // output rows a stage; staged input rows, their pitch, pixels a row
    uint32_t inv_pw;      // ceil(2^32 / pw)
    int64_t x_img, x_plane, y_img;
};

// Four pixels of an output row: the input columns under their taps, and CO channels' gradients.
// Input column c of a row is staged at c + SHIFT, so that the columns new to a group start at a
// multiple of four; the E before them are the previous group's last, or at a row's start read.
template <int CO, int RS>
struct PixelGroup {
    static constexpr int E = 3 - RS, SHIFT = 4 - E, NEW = 4 * RS, DROW = CO == 4 ? 36 : 34;
    float x[3][E + NEW];
    uint64_t d[4][CO / 2];
    __device__ __forceinline__ void load(const float* xs, int pitch, const float* ds, bool start, const PixelGroup& prev) {
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
            const float* r = xs + ky * pitch;
#pragma unroll
            for (int c = 0; c < NEW; c += 4) {
                const float4 v = *reinterpret_cast<const float4*>(r + 4 + c);
                x[ky][E + c] = v.x; x[ky][E + c + 1] = v.y; x[ky][E + c + 2] = v.z; x[ky][E + c + 3] = v.w;
            }
#pragma unroll
            for (int e = 0; e < E; ++e) x[ky][e] = start ? r[SHIFT + e] : prev.x[ky][NEW + e];
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            if (CO == 4) {
                const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(ds + v * DROW);
                d[v][0] = t.x; d[v][CO / 2 - 1] = t.y;
            } else {
                d[v][0] = *reinterpret_cast<const uint64_t*>(ds + v * DROW);
            }
        }
    }
    // pixels LO .. HI - 1 of the group
    template <int LO, int HI>
    __device__ __forceinline__ void multiply(uint64_t (&acc)[CO / 2][9], float (&bacc)[CO], bool bias) const {
        uint64_t xx[3][E + NEW];
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
            for (int c = 0; c < E + NEW; ++c) xx[ky][c] = both(x[ky][c]);
#pragma unroll
        for (int v = LO; v < HI; ++v) {
#pragma unroll
            for (int k = 0; k < CO / 2; ++k)
#pragma unroll
                for (int r = 0; r < 9; ++r) fma_pair(acc[k][r], d[v][k], xx[r / 3][v * RS + r % 3]);
            if (bias)
#pragma unroll
                for (int k = 0; k < CO; ++k) bacc[k] += half_of(d[v], k);
        }
    }
};

template <int CI, int CO, int RS>
__global__ void __launch_bounds__(2 * CI * 32 / CO) wgrad_f32_kernel(const __grid_constant__ WgradF32Args a) {
    using Group = PixelGroup<CO, RS>;
    constexpr int NT = CI * 32 / CO, NW = NT / 32, DROW = Group::DROW;
    SQ_KERNEL_WAIT();
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const int cg = tid % (32 / CO), ci = tid / (32 / CO);
    const int c0 = blockIdx.x * CI, co0 = blockIdx.y * 32, nci = min(CI, a.Cin - c0);
    const int p_begin = blockIdx.z * a.chunk, p_end = min(a.P, p_begin + a.chunk);
    const int px = a.oh * a.ow;
    // rows of the flattened (image, row) order that hold the split's pixels
    const int g_begin = p_begin / a.ow, g_end = p_end > p_begin ? (p_end - 1) / a.ow + 1 : g_begin;
    const int tiles = (g_end - g_begin + a.nr - 1) / a.nr;
    const int full = (a.oh - 1) * RS + 3;
    const int x_words = a.xrows * a.xp, stage_words = CI * x_words + (a.nr * a.dp + 4) * DROW;
    auto stage = [&](int t) {
        if (t < tiles) {
            float* sx = smem + (t % a.stages) * stage_words;
            float* sd = sx + CI * x_words;
            const int r0 = g_begin + t * a.nr, r1 = min(g_end, r0 + a.nr);
            // gradients: a lane's pixels, every NW-th output channel
            for (int l = lane; l < (r1 - r0) * a.ow; l += 32) {
                const int p = r0 * a.ow + l, img = p / px;
                if (p < p_begin || p >= p_end) continue;
                const int row = l / a.ow, col = l - row * a.ow;
                const float* src = a.dy + (int64_t)img * a.y_img + (int64_t)co0 * px + (p - img * px);
                float* dst = sd + (row * a.dp + col) * DROW;
#pragma unroll 4
                for (int co = warp - NW; co < 32; co += NW)
                    if (co0 + co < a.Cout) copy4(dst + co, src + (int64_t)co * px, true);
            }
            // input rows: of the first image from its first output row on, of the others from 0
            const int img0 = r0 / a.oh, oy0 = r0 - img0 * a.oh, n0 = min(r1 - r0, a.oh - oy0), rest = r1 - r0 - n0;
            const int first = (n0 - 1) * RS + 3, last = rest % a.oh;
            const int rows = first + rest / a.oh * full + (last ? (last - 1) * RS + 3 : 0);
            const float* x0 = a.x + (int64_t)img0 * a.x_img + (int64_t)c0 * a.x_plane;
            for (int w = tid - NT; w < rows * a.pw; w += NT) {
                const int r = __umulhi(w, a.inv_pw), col = w - r * a.pw;
                const float* src = x0;
                if (r < first) {
                    src += (oy0 * RS + r) * a.pw + col;
                } else {
                    const int q = (r - first) / full;
                    src += (q + 1) * a.x_img + (r - first - q * full) * a.pw + col;
                }
                float* dst = sx + r * a.xp + col + Group::SHIFT;
#pragma unroll
                for (int c = 0; c < CI; ++c)
                    if (c < nci) copy4(dst + c * x_words, src + c * a.x_plane, true);
            }
        }
        copies_commit();
    };
    if (warp >= NW) {
        for (int st = 0; st + 1 < a.stages; ++st) stage(st);
        for (int t = 0; t < tiles; ++t) {
            if (a.stages == 2) asm volatile("cp.async.wait_group 0;" ::: "memory");
            else asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncthreads();   // this stage has landed, the previous one has been read
            stage(t + a.stages - 1);
        }
        SQ_KERNEL_TRIGGER();
        return;
    }
    uint64_t acc[CO / 2][9];
    float bacc[CO];
    const bool bias = blockIdx.x == 0;
#pragma unroll
    for (int k = 0; k < CO; ++k) {
        bacc[k] = 0.f;
#pragma unroll
        for (int r = 0; r < 9; ++r) acc[k / 2][r] = 0;
    }
    for (int t = 0; t < tiles; ++t) {
        __syncthreads();
        const float* xrow = smem + (t % a.stages) * stage_words + ci * x_words;
        const float* drow = smem + (t % a.stages) * stage_words + CI * x_words + cg * CO;
        const int r1 = min(g_end, g_begin + (t + 1) * a.nr);
        int g = g_begin + t * a.nr, oy = g % a.oh;
        Group ga, gb;
        ga.load(xrow, a.xp, drow, true, ga);
        for (; g < r1; ++g) {
            // pixels [lo, hi) of the row: all but in the split's first and last row
            const int lo = max(0, p_begin - g * a.ow), hi = min(a.ow, p_end - g * a.ow);
            int q = lo / 4;
            const float* xq = xrow + 4 * RS * q;
            const float* dq = drow + 4 * q * DROW;
            if (lo) {
                ga.load(xq, a.xp, dq, true, ga);
                gb.load(xq + 4 * RS, a.xp, dq + 4 * DROW, false, ga);
                const int l = lo - 4 * q, h = hi - 4 * q;
                if (l <= 0 && h > 0) ga.template multiply<0, 1>(acc, bacc, bias);
                if (l <= 1 && h > 1) ga.template multiply<1, 2>(acc, bacc, bias);
                if (l <= 2 && h > 2) ga.template multiply<2, 3>(acc, bacc, bias);
                if (h > 3) ga.template multiply<3, 4>(acc, bacc, bias);
                ga = gb;
                ++q;
                xq += 4 * RS;
                dq += 4 * DROW;
            }
            const int whole = hi / 4;
            for (; q + 1 < whole; q += 2) {
                gb.load(xq + 4 * RS, a.xp, dq + 4 * DROW, false, ga);
                ga.template multiply<0, 4>(acc, bacc, bias);
                xq += 8 * RS;
                dq += 8 * DROW;
                ga.load(xq, a.xp, dq, false, gb);
                gb.template multiply<0, 4>(acc, bacc, bias);
            }
            if (q < whole) {
                gb.load(xq + 4 * RS, a.xp, dq + 4 * DROW, false, ga);
                ga.template multiply<0, 4>(acc, bacc, bias);
                ga = gb;
                ++q;
            }
            oy = oy + 1 == a.oh ? 0 : oy + 1;
            if (g + 1 < r1) {
                xrow += (oy ? RS : 3) * a.xp;
                drow += a.dp * DROW;
            }
            gb.load(xrow, a.xp, drow, true, ga);
            const int left = hi - 4 * q;
            if (left > 0) ga.template multiply<0, 1>(acc, bacc, bias);
            if (left > 1) ga.template multiply<1, 2>(acc, bacc, bias);
            if (left > 2) ga.template multiply<2, 3>(acc, bacc, bias);
            ga = gb;
        }
    }
    SQ_KERNEL_TRIGGER();
    const int N = a.Cin * 9 + 1;
    float* out = a.work + (int64_t)blockIdx.z * a.Cout * N;
#pragma unroll
    for (int k = 0; k < CO; ++k) {
        const int co = co0 + cg * CO + k;
        if (co >= a.Cout) continue;
        if (ci < nci) {
#pragma unroll
            for (int r = 0; r < 9; ++r)
                out[(int64_t)co * N + (c0 + ci) * 9 + r] = __uint_as_float((uint32_t)(acc[k / 2][r] >> (32 * (k % 2))));
        }
        if (bias && ci == 0) out[(int64_t)co * N + N - 1] = bacc[k];
    }
}

template <int CI, int CO, int RS>
bool launch_wgrad(WgradF32Args a, int splits, cudaStream_t s) {
    using Group = PixelGroup<CO, RS>;
    a.dp = (a.ow + 3) / 4 * 4;
    a.xp = std::max(a.dp * RS + 4, (a.pw + Group::SHIFT + 3) / 4 * 4);
    a.inv_pw = (uint32_t)(((1ULL << 32) + a.pw - 1) / a.pw);
    // about 64 pixels a stage
    for (a.nr = std::max(1, std::min(8, 64 / a.ow)); a.nr >= 1; --a.nr) {
        const int pieces = (a.nr - 1 + a.oh - 1) / a.oh + 1;
        a.xrows = a.nr * RS + std::max(0, 3 - RS) * pieces;
        const int64_t stage = 4 * ((int64_t)CI * a.xrows * a.xp + (int64_t)(a.nr * a.dp + 4) * Group::DROW);
        a.stages = 3 * stage <= kSmemBytes ? 3 : 2;
        if (a.stages * stage > kSmemBytes) continue;
        launch_with(false, wgrad_f32_kernel<CI, CO, RS>, dim3((a.Cin + CI - 1) / CI, (a.Cout + 31) / 32, splits), dim3(2 * CI * 32 / CO),
                    (size_t)(a.stages * stage), s, a);
        return true;
    }
    return false;
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
    // Whole planes are staged where a stride reads parts of them, and a stage holds kChan of them: with one
    // input channel, or few and a stride of 3 or more, conv_fwd_kernel's gather is cheaper once its CTAs fill
    // the chip.  1,024 images of 40 x 40, here and there in us: 1 channel to 8, stride 2 32.9 and 25.4, 2 to
    // 8 34 and 39; 3 channels to 32, stride 3 28.9 and 23.6, 9 to 48 102 and 101.
    if ((int64_t)((a.M + 127) / 128) * ((a.N + 31) / 32) >= 800 &&
        ((sh.Cin == 1 && sh.stride >= 2) || (sh.Cin <= 8 && sh.Cout > 8 && sh.stride >= 3)))
        return false;
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
    a.oh = sh.OH; a.ow = sh.OW; a.pw = sh.W;
    a.P = sh.nimg * sh.OH * sh.OW; a.Cin = sh.Cin; a.Cout = sh.Cout; a.chunk = chunk;
    a.x_img = sh.x_img_stride; a.x_plane = (int64_t)sh.H * sh.W; a.y_img = sh.y_img_stride;
    // 512 images of 13 x 13 and 11 x 11, 32 channels: 62 and 47 us by 16 x 4, 66 and 47 by 8 x 2; of
    // 16 channels 7 x 7: 14.6 and 12.6; 70 of 3 x 3, 2 channels: 17.5 by 8 x 2, 16.6 by 4 x 2.
    // Wider strides take conv_wgrad_kernel.
    if (sh.stride == 1) {
        if (sh.Cin > 16) return launch_wgrad<16, 4, 1>(a, splits, s);
        return sh.Cin > 4 ? launch_wgrad<8, 2, 1>(a, splits, s) : launch_wgrad<4, 2, 1>(a, splits, s);
    }
    if (sh.stride == 2) return sh.Cin > 4 ? launch_wgrad<8, 2, 2>(a, splits, s) : launch_wgrad<4, 2, 2>(a, splits, s);
    return false;
}

}  // namespace sq
