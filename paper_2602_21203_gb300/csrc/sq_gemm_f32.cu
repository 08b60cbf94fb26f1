// FP32 GEMM on CUDA cores: the dense contraction of the plain FP32 path (every linear
// layer's forward, data gradient and weight gradient).
//
// What bounds it: at the training shape, shared-memory fragment reads beside the FMAs (8
// 16-byte reads, 4 cycles of the SM's read path each, per 64 FMAs of a scheduler; two warps a
// scheduler, the FMA pipe 32 % busy); at the small ones, the latency of one CTA's pass over K.  Operand tiles come in by cp.async
// into a ring of kStages shared-memory stages, so global latency overlaps the arithmetic;
// both are staged in their memory order (K-contiguous rows, or rows of M / N), so no
// transposing pass is needed, and a thread reads 16-byte fragments: four K steps of a row
// where K is contiguous, four rows of a K step where it is not.  Every output is one
// chain of fused multiply-adds over k ascending (no split of K), so its bits depend neither
// on the tile nor on the rest of the batch, and equal those of gemm_kernel (sq_gemm.cu),
// which stages synchronously: M = N = K = 512 twice 50.4 us there, 22.5 here (floor 6.7 at
// one FMA per lane and cycle), the projections' 2048 x 256 x 2592 244 and 88 us (floor 33.7),
// M 32, N 256, K 412 twice 39.7 and 5.6 us.  Where B's rows are contiguous in n, a read brings
// column pairs and products are issued in pairs: M 512, N 2592, K 256 32.8 us one by one and
// 24.6 in pairs, N = K = 512 twice 22.5 and 20.5 (where they are contiguous in k the pairs would
// have to be put together: 22.5 and 28.8).
#include "sq_kernels.cuh"

#include <algorithm>

namespace sq {
namespace {

constexpr int kMaxGroup = 8;
constexpr int kSmemBytes = 48 * 1024;   // static limit: no opt-in, on any device

struct GemmF32Problem {
    GemmProblem g;
    int va, vb;          // elements per copy of A and B: 4, 2 or 1, by address alignment
    int tile_start, tiles_n;
};
struct GemmF32Batch {
    GemmF32Problem p[kMaxGroup];
    int n;
};

template <int V>
__device__ __forceinline__ void cp_async(uint32_t dst, const float* src, int bytes) {
    if (V == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
    else if (V == 2) asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// One operand tile of R rows x BK steps of k: [R][BK + 4] if k is contiguous, else
// [BK][R + 4].  `src` points at (row0, k0), `rows` and `ks` are what is left of the operand
// there; elements outside arrive as zeros.
template <bool KMAJ, int R, int BK, int NTHR, int V>
__device__ __forceinline__ void stage_tile_v(uint32_t dst, const float* src, int64_t ld, int rows, int ks) {
    constexpr int FAST = KMAJ ? BK : R;          // extent of the contiguous direction
    constexpr int SLOW = KMAJ ? R : BK;
    constexpr int CHUNKS = SLOW * (FAST / V);
    constexpr int STEP = NTHR / (FAST / V);      // slow rows between a thread's chunks
    static_assert(NTHR % (FAST / V) == 0 && CHUNKS % NTHR == 0, "whole rows a pass");
    const int sl = threadIdx.x / (FAST / V), fa = (threadIdx.x % (FAST / V)) * V;
    const int fast_n = KMAJ ? ks : rows, slow_n = KMAJ ? rows : ks;
    const int bytes = 4 * min(V, max(0, fast_n - fa));
    const float* p = src + (int64_t)sl * ld + fa;
    uint32_t d = dst + 4 * (sl * (FAST + 4) + fa);
#pragma unroll
    for (int u = 0; u < CHUNKS / NTHR; ++u) {
        const int b = sl + u * STEP < slow_n ? bytes : 0;
        cp_async<V>(d + 4 * u * STEP * (FAST + 4), b > 0 ? p + (int64_t)u * STEP * ld : src, b);
    }
}
template <bool KMAJ, int R, int BK, int NTHR>
__device__ __forceinline__ void stage_tile(uint32_t dst, const float* src, int64_t ld, int rows, int ks, int vec) {
    if (vec == 4) stage_tile_v<KMAJ, R, BK, NTHR, 4>(dst, src, ld, rows, ks);
    else if (vec == 2) stage_tile_v<KMAJ, R, BK, NTHR, 2>(dst, src, ld, rows, ks);
    else stage_tile_v<KMAJ, R, BK, NTHR, 1>(dst, src, ld, rows, ks);
}

// The same tile by 16-byte copies where all BK steps of k exist: what a thread copies does
// not change over the steps, so its places and sizes are formed once.
template <bool KMAJ, int R, int BK, int NTHR>
struct TileCopy {
    static constexpr int FAST = KMAJ ? BK : R, SLOW = KMAJ ? R : BK, STEP = NTHR / (FAST / 4);
    static constexpr int N = SLOW / STEP;
    static_assert(NTHR % (FAST / 4) == 0 && SLOW % STEP == 0, "whole rows a pass");
    int64_t off;
    uint32_t dst;
    int bytes[N];
    __device__ __forceinline__ TileCopy(int64_t ld, int rows) {
        const int sl = threadIdx.x / (FAST / 4), fa = (threadIdx.x % (FAST / 4)) * 4;
        off = (int64_t)sl * ld + fa;
        dst = 4 * (sl * (FAST + 4) + fa);
#pragma unroll
        for (int u = 0; u < N; ++u)
            bytes[u] = KMAJ ? (sl + u * STEP < rows ? 16 : 0) : 4 * min(4, max(0, rows - fa));
    }
    __device__ __forceinline__ void copy(uint32_t tile, const float* src, int64_t ld) const {
#pragma unroll
        for (int u = 0; u < N; ++u)
            cp_async<4>(tile + dst + 4 * u * STEP * (FAST + 4), bytes[u] > 0 ? src + off + (int64_t)u * STEP * ld : src,
                        bytes[u]);
    }
};

// Row i of thread t's T rows of a tile of R.
template <bool KMAJ, int R, int T>
__device__ __forceinline__ int tile_row(int t, int i) {
    return KMAJ ? t + (R / T) * i : t * T + i;
}

// T fragments of four k steps: f[i][kk].
template <bool KMAJ, int R, int BK, int T>
__device__ __forceinline__ void fragment(float (&f)[T][4], const float* s, int t, int k4) {
    if (KMAJ) {
#pragma unroll
        for (int i = 0; i < T; ++i) {
            const float4 v = *reinterpret_cast<const float4*>(s + tile_row<KMAJ, R, T>(t, i) * (BK + 4) + 4 * k4);
            f[i][0] = v.x; f[i][1] = v.y; f[i][2] = v.z; f[i][3] = v.w;
        }
    } else {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
#pragma unroll
            for (int i = 0; i < T; i += 4) {
                const float* r = s + (4 * k4 + kk) * (R + 4) + tile_row<KMAJ, R, T>(t, i);
                if (T >= 4) {
                    const float4 v = *reinterpret_cast<const float4*>(r);
                    f[i][kk] = v.x; f[i + 1][kk] = v.y; f[(i + 2) % T][kk] = v.z; f[(i + 3) % T][kk] = v.w;
                } else {
                    const float2 v = *reinterpret_cast<const float2*>(r);
                    f[i][kk] = v.x; f[i + 1][kk] = v.y;
                }
            }
        }
    }
}

// BM x BN outputs a CTA, TM x TN a thread (TM, TN in {2, 4}); a warp covers 4 x 8 threads.  Three
// CTAs of the large tile to an SM: left to itself the compiler takes 254 registers where A and B
// are contiguous in m and n, two CTAs, and 328 tiles (M 256, N 2592, K 512) wait for a second
// wave: 30.2 us, 26.7 with three.  (Four: 26.7 too, but the FP32 update 5,167 us against 5,069.)
template <int BM, int BN, int TM, int TN, int BK, bool A_K, bool B_K>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), BN < 64 ? 1 : 3) gemm_f32_kernel(const __grid_constant__ GemmF32Batch gb) {
    constexpr int NTHR = (BM / TM) * (BN / TN);
    constexpr int WN = BN / (8 * TN);
    constexpr int A_FLOATS = A_K ? BM * (BK + 4) : BK * (BM + 4);
    constexpr int B_FLOATS = B_K ? BN * (BK + 4) : BK * (BN + 4);
    constexpr int FIT = kSmemBytes / (4 * (A_FLOATS + B_FLOATS)), kStages = FIT < 8 ? FIT : 8;
    static_assert(kStages >= 3, "operand ring");
    __shared__ __align__(16) float smem[kStages * (A_FLOATS + B_FLOATS)];
    SQ_KERNEL_WAIT();
    int pi = 0;
    while (pi + 1 < gb.n && (int)blockIdx.x >= gb.p[pi + 1].tile_start) ++pi;
    const GemmF32Problem& Q = gb.p[pi];
    const GemmProblem& P = Q.g;
    const int t = blockIdx.x - Q.tile_start;
    const int m0 = (t / Q.tiles_n) * BM, n0 = (t % Q.tiles_n) * BN;
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    const int tx = (warp % WN) * 8 + lane % 8, ty = (warp / WN) * 4 + lane / 8;
    const float* A = static_cast<const float*>(P.A);
    const float* B = static_cast<const float*>(P.B);
    const int64_t lda = A_K ? P.sa_m : P.sa_k, ldb = B_K ? P.sb_n : P.sb_k;
    const int nk = (P.K + BK - 1) / BK, iters = nk * P.n_sum;

    // the tiles at k step `kn` of summed pair `sn`, the next ones to copy
    const float* an = A + (int64_t)m0 * (A_K ? lda : 1);
    const float* bn = B + (int64_t)n0 * (B_K ? ldb : 1);
    int kn = 0, sn = 0;
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem);
    const TileCopy<A_K, BM, BK, NTHR> ca(lda, P.M - m0);
    const TileCopy<B_K, BN, BK, NTHR> cb(ldb, P.N - n0);
    const bool wide = Q.va == 4 && Q.vb == 4;
    auto stage = [&](int slot) {
        if (sn < P.n_sum) {
            const uint32_t sa = ring + 4 * slot * (A_FLOATS + B_FLOATS);
            if (wide && kn + BK <= P.K) {
                ca.copy(sa, an, lda);
                cb.copy(sa + 4 * A_FLOATS, bn, ldb);
            } else {
                stage_tile<A_K, BM, BK, NTHR>(sa, an, lda, P.M - m0, P.K - kn, Q.va);
                stage_tile<B_K, BN, BK, NTHR>(sa + 4 * A_FLOATS, bn, ldb, P.N - n0, P.K - kn, Q.vb);
            }
            kn += BK;
            an += A_K ? BK : BK * lda;
            bn += B_K ? BK : BK * ldb;
            if (kn >= P.K) {
                kn = 0;
                ++sn;
                an = A + (int64_t)sn * P.a_sum + (int64_t)m0 * (A_K ? lda : 1);
                bn = B + (int64_t)sn * P.b_sum + (int64_t)n0 * (B_K ? ldb : 1);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int st = 0; st < kStages; ++st) stage(st);

    float acc[TM][TN];      // B's rows contiguous in k
    uint64_t acc2[TM][TN / 2];   // in n: column pairs
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            acc[i][j] = 0.f;
            acc2[i][j / 2] = 0;
        }

    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 1) : "memory");
    __syncthreads();
    // the fragments of the next four steps are read while the current ones are multiplied
    float a[2][TM][4], b[2][TN][4];
    fragment<A_K, BM, BK, TM>(a[0], smem, ty, 0);
    fragment<B_K, BN, BK, TN>(b[0], smem + A_FLOATS, tx, 0);
    int slot = 0;
    for (int it = 0; it < iters; ++it) {
        const float* cur = smem + slot * (A_FLOATS + B_FLOATS);
        const int next_slot = slot + 1 == kStages ? 0 : slot + 1;
#pragma unroll
        for (int k4 = 0; k4 < BK / 4; ++k4) {
            const float* src = cur;
            if (k4 + 1 == BK / 4) {
                // every thread has read the last of this stage, and the next has landed
                asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
                __syncthreads();
                stage(slot);
                src = smem + next_slot * (A_FLOATS + B_FLOATS);
            }
            const int k4n = (k4 + 1) % (BK / 4);
            fragment<A_K, BM, BK, TM>(a[(k4 + 1) % 2], src, ty, k4n);
            fragment<B_K, BN, BK, TN>(b[(k4 + 1) % 2], src + A_FLOATS, tx, k4n);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) {
                        if (B_K) acc[i][j] = fmaf(a[k4 % 2][i][kk], b[k4 % 2][j][kk], acc[i][j]);
                        else if (j % 2) fma_pair(acc2[i][j / 2], pair(b[k4 % 2][j - 1][kk], b[k4 % 2][j][kk]), both(a[k4 % 2][i][kk]));
                    }
        }
        slot = next_slot;
    }

    SQ_KERNEL_TRIGGER();
    float* C = static_cast<float*>(P.C);
    const float* bias = static_cast<const float*>(P.bias);
    const float* mask = static_cast<const float*>(P.mask);
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + tile_row<A_K, BM, TM>(ty, i);
        if (m >= P.M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int n = n0 + tile_row<B_K, BN, TN>(tx, j);
            if (n >= P.N) continue;
            float v = B_K ? acc[i][j] : __uint_as_float((uint32_t)(acc2[i][j / 2] >> (32 * (j % 2))));
            if (bias) v += bias[n];
            if (mask && !(mask[(int64_t)m * P.sm_m + (int64_t)n * P.sm_n] > 0.f)) v = 0.f;
            float* dst = C + (int64_t)m * P.sc_m + (int64_t)n * P.sc_n;
            *dst = P.accumulate ? *dst + v : v;
        }
    }
}

// The widest copy whose every start address is aligned, given the stride between rows (or
// k steps) and between summed operands.
int copy_width(const void* p, int64_t ld, int64_t sum) {
    const int64_t bits = (int64_t)(reinterpret_cast<uintptr_t>(p) / 4) | ld | sum;
    if (reinterpret_cast<uintptr_t>(p) % 4) return 0;
    return bits % 4 == 0 ? 4 : bits % 2 == 0 ? 2 : 1;
}

template <int BM, int BN, int TM, int TN, int BK, bool A_K, bool B_K>
void launch_tiles(GemmF32Batch& gb, cudaStream_t s) {
    int tiles = 0;
    for (int i = 0; i < gb.n; ++i) {
        gb.p[i].tile_start = tiles;
        gb.p[i].tiles_n = (gb.p[i].g.N + BN - 1) / BN;
        tiles += ((gb.p[i].g.M + BM - 1) / BM) * gb.p[i].tiles_n;
    }
    if (tiles == 0) return;
    // (a full grid of the large tile is not let in early: launch_with)
    launch_with(BN < 64, gemm_f32_kernel<BM, BN, TM, TN, BK, A_K, B_K>, dim3(tiles), dim3((BM / TM) * (BN / TN)), 0, s, gb);
}

int count_tiles(const GemmF32Batch& gb, int bm, int bn) {
    int tiles = 0;
    for (int i = 0; i < gb.n; ++i) tiles += ((gb.p[i].g.M + bm - 1) / bm) * ((gb.p[i].g.N + bn - 1) / bn);
    return tiles;
}

// The tile: the largest that still gives most of the 152 SMs a CTA.  A 32 x 64 tile (128
// threads of 4 x 4) multiplies at the best rate, M = N = K = 512 twice in 20.5 us (64 x 64:
// 21.4, 32 x 32: 26.9, 16 x 32: 27.0); where it leaves SMs idle, one CTA's own pass over K
// is what takes the time, and smaller tiles of smaller fragments are shorter: M 512, N 101,
// K 512 twice 12.5 us by 32 x 64 (64 CTAs) and 9.3 by 32 x 32 (128), M 32, N 256, K 412
// twice 11.1, 8.1 and 5.9 us by 32 x 64, 32 x 32 and 16 x 32.  (The choice was measured with every
// grid let in at its primary's start; as launched now, one such call after another, the chosen tiles
// take 22.5, 11.6 and 5.6.)
template <bool A_K, bool B_K>
void launch_layout(GemmF32Batch& gb, cudaStream_t s) {
    if (count_tiles(gb, 32, 64) >= 100) launch_tiles<32, 64, 4, 4, 32, A_K, B_K>(gb, s);
    else if (count_tiles(gb, 32, 32) >= 100) launch_tiles<32, 32, 2, 4, 32, A_K, B_K>(gb, s);
    else launch_tiles<16, 32, 2, 2, 32, A_K, B_K>(gb, s);
}

// Where gemm_kernel (sq_gemm.cu) is the faster of the two (the bits are the same): grids of more than
// three CTAs an SM whose CTAs have little K to pipeline over.  It pads K to 16 steps, not 32, and more of
// its threads fit an SM; and a stage of the ring costs more where an operand contiguous in K has rows
// that are copied 4 or 8 bytes at a time.  Ring against gemm_kernel in us, M 6000, N 1800 (5,358 tiles of
// 32 x 64): K 16 45 and 31, 48 58 and 54, 52 57 and 66; with both operands' rows of odd length K 33 84 and
// 52, 97 131 and 102, 161 176 and 152, 257 242 and 225 (within 5 % on smaller grids: left to the ring),
// 513 409 and 424; with B's alone K 33 78 and 52, 129 141 and 127, 161 162 and 152.  456 tiles or fewer are
// never slower in the ring (M = N = 512: 6.4 and 11.5); between 641 and 1,000 it fills its second wave
// and gemm_kernel does not, and only the shortest narrow rows lose (K 17: 1.2 times); just above 456 it has
// a nearly empty second wave, and K up to 32, where that is short, stays.
bool general_is_faster(int64_t tiles, int64_t K, bool a_k, bool b_k, int va, int vb) {
    if (tiles <= 456) return false;
    const bool na = a_k && va < 4, nb = b_k && vb < 4;   // K-contiguous rows in narrow copies
    int limit = nb ? (na ? 100 : 70) : na ? 65 : 48;
    if (tiles <= 640) return K > 32 && K <= limit;
    if (tiles <= 1000) return nb && K <= 33;
    if (nb && tiles > 2400) limit = na ? (va == 1 && vb == 1 ? 200 : 130) : vb == 1 ? 140 : 100;
    return K <= limit;
}

}  // namespace

bool launch_gemm_f32(const GemmProblem* probs, int n_probs, cudaStream_t s) {
    GemmF32Batch gb;
    if (n_probs < 1) return false;
    const bool a_k = probs[0].sa_k == 1, b_k = probs[0].sb_k == 1;
    int64_t tiles = 0, steps = 0;   // of the call; the longest chain over K
    int va = 4, vb = 4;             // the narrowest copies
    for (int i = 0; i < n_probs; ++i) {
        const GemmProblem& p = probs[i];
        if ((p.sa_k == 1) != a_k || (p.sb_k == 1) != b_k || (!a_k && p.sa_m != 1) || (!b_k && p.sb_n != 1)) return false;
        if (!copy_width(p.A, 0, 0) || !copy_width(p.B, 0, 0)) return false;
        tiles += (int64_t)((p.M + 31) / 32) * ((p.N + 63) / 64);
        steps = std::max(steps, (int64_t)p.K * std::max(1, p.n_sum));
        va = std::min(va, copy_width(p.A, a_k ? p.sa_m : p.sa_k, p.n_sum > 1 ? p.a_sum : 0));
        vb = std::min(vb, copy_width(p.B, b_k ? p.sb_n : p.sb_k, p.n_sum > 1 ? p.b_sum : 0));
    }
    if (general_is_faster(tiles, steps, a_k, b_k, va, vb)) return false;
    for (int base = 0; base < n_probs; base += kMaxGroup) {
        gb.n = std::min(kMaxGroup, n_probs - base);
        for (int i = 0; i < gb.n; ++i) {
            GemmProblem& g = gb.p[i].g;
            g = probs[base + i];
            if (g.n_sum < 1) g.n_sum = 1;
            gb.p[i].va = copy_width(g.A, a_k ? g.sa_m : g.sa_k, g.n_sum > 1 ? g.a_sum : 0);
            gb.p[i].vb = copy_width(g.B, b_k ? g.sb_n : g.sb_k, g.n_sum > 1 ? g.b_sum : 0);
        }
        if (a_k && b_k) launch_layout<true, true>(gb, s);
        else if (a_k) launch_layout<true, false>(gb, s);
        else if (b_k) launch_layout<false, true>(gb, s);
        else launch_layout<false, false>(gb, s);
    }
    return true;
}

}  // namespace sq
