#pragma once
// omni_fft_level.cuh -- level passes: both axes of one hierarchy level in one kernel.
//
// The hypercube of Eq. ProofEq2 has two axes per level.  A level pass
// transforms axes a = 2k and b = 2k+1 of level k together: per sample the data
// is [outer][n_b][n_a][inner] on input and [outer][L_b][L_a][inner] on output
// (inner = product of the padded lengths of the finer levels, outer = product
// of the sizes of the coarser ones).
//
// Tiling is fixed at compile time:
//  * the finest level (inner == 1): a CTA owns U whole n x n blocks of
//    antennas (Appendix A step 4's per-block 2-D FFT), W = 1, each block
//    contiguous in memory;
//  * a coarser level: a CTA owns W consecutive inner indices (U = 1) so that
//    every global access is a W-wide coalesced row.
// The tile is staged in shared memory as [k_b][k_a][w]; axis a is transformed
// one line per thread (pruned first stage: the upper half of every line is
// zero padding), then axis b, whose outputs go straight to global memory (MID)
// or are squared and summed over the chunk's samples in registers and folded
// into the FP64 accumulator once per chunk (LAST: the |F|^2 time integration).
// In LAST mode the next sample's inputs are loaded into registers while the
// current sample is transformed.
#include "omni_fft_common.cuh"

#include <algorithm>
#include <type_traits>

namespace omni {

// Compile-time tiling of a level pass of L points per axis.
template <int L, bool FINEST, int MODE>
struct LevelTile {
    static constexpr int N = L / 2;
    static constexpr int LPT = (MODE == MODE_LAST) ? (L >= 64 ? 1 : 2) : 1;
    static constexpr int W = FINEST ? 1 : 256 * LPT / L;
    static constexpr int U = FINEST ? ((MODE == MODE_LAST) ? 1 : (L >= 64 ? 2 : 256 / L)) : 1;
    static constexpr int RP = FINEST ? L + 1 : L;          // row pitch, odd for W == 1
    static constexpr int UPL = L * RP * W;                 // shared elements per unit
    static constexpr int IN_PER_UNIT = N * N * W;
    static constexpr int LINES_A = U * N * W;
    static constexpr int LINES_B = U * L * W;
    static constexpr int THREADS = (MODE == MODE_LAST)
        ? (LINES_B / LPT < 32 ? 32 : LINES_B / LPT)
        : (LINES_B > 256 ? 256 : (LINES_B < 32 ? 32 : LINES_B));
    static constexpr int EPT = (U * IN_PER_UNIT + THREADS - 1) / THREADS;  // loads per thread
    static constexpr size_t SMEM = (size_t)U * UPL * sizeof(float2);
};

template <int L, bool FINEST, int MODE, int SRC>
__global__ void __launch_bounds__(LevelTile<L, FINEST, MODE>::THREADS)
level_pass(Pass p, PassArgs a) {
    using T = LevelTile<L, FINEST, MODE>;
    constexpr int N = T::N, W = T::W, U = T::U, RP = T::RP, UPL = T::UPL;
    constexpr int LOG = ilog2(L);
    constexpr int NT = T::THREADS, LPT = T::LPT, EPT = T::EPT;
    extern __shared__ float2 sm[];
    const int64_t inner = p.inner;

    if constexpr (MODE == MODE_MID) {
        __shared__ int64_t unit_src[U];
        __shared__ int64_t unit_dst[U];
        // ---- per-unit base offsets (sample, outer block, inner tile)
        const int64_t tiles = FINEST ? 1 : (inner + W - 1) / W;
        const int64_t units_total = a.S * p.outer * tiles;
        if (threadIdx.x < U) {
            const int64_t ug = (int64_t)blockIdx.x * U + threadIdx.x;
            int64_t sb = -1, db = -1;
            if (ug < units_total) {
                const int64_t tile = FINEST ? 0 : ug % tiles;
                const int64_t so = FINEST ? ug : ug / tiles;
                const int64_t o = so % p.outer, s = so / p.outer;
                sb = src_base(a, s) + o * (int64_t)N * N * inner + tile * W;
                db = s * a.dst_stride + o * (int64_t)L * L * inner + tile * W;
            }
            unit_src[threadIdx.x] = sb;
            unit_dst[threadIdx.x] = db;
        }
        __syncthreads();
        // valid w of this CTA's tile (U == 1 when W > 1)
        const int64_t i_lim = FINEST ? 1 : inner - ((int64_t)blockIdx.x % tiles) * W;
        // ---- load
#pragma unroll
        for (int q = 0; q < EPT; ++q) {
            const int e = threadIdx.x + q * NT;
            if (e < U * T::IN_PER_UNIT) {
                const int u = e / T::IN_PER_UNIT;
                const int r = e - u * T::IN_PER_UNIT;
                const int w = r % W, ja = (r / W) % N, jb = r / (W * N);
                float2 x = make_float2(0.f, 0.f);
                if (unit_src[u] >= 0 && w < i_lim)
                    x = ld_src<SRC>(a.src, unit_src[u] + (int64_t)(jb * N + ja) * inner + w);
                sm[u * UPL + (jb * RP + ja) * W + w] = x;
            }
        }
        __syncthreads();
        // ---- axis a
        for (int l = threadIdx.x; l < T::LINES_A; l += NT) {
            const int u = l / (N * W), r = l - u * (N * W);
            const int jb = r / W, w = r % W;
            float2* row = sm + u * UPL + jb * RP * W + w;
            float2 v[L];
#pragma unroll
            for (int j = 0; j < L; ++j) v[j] = (j < N) ? row[j * W] : make_float2(0.f, 0.f);
            fft_dif<L, true>(v);
#pragma unroll
            for (int k = 0; k < L; ++k) row[k * W] = v[brev(k, LOG)];
        }
        __syncthreads();
        // ---- axis b, straight to global memory
        for (int l = threadIdx.x; l < T::LINES_B; l += NT) {
            const int u = l / (L * W), r = l - u * (L * W);
            const int ka = r / W, w = r % W;
            const float2* col = sm + u * UPL + ka * W + w;
            float2 v[L];
#pragma unroll
            for (int j = 0; j < L; ++j) v[j] = (j < N) ? col[j * RP * W] : make_float2(0.f, 0.f);
            fft_dif<L, true>(v);
            if (unit_dst[u] >= 0 && w < i_lim) {
                float2* d = a.dst + unit_dst[u] + (int64_t)ka * inner + w;
#pragma unroll
                for (int k = 0; k < L; ++k) d[(int64_t)k * L * inner] = v[brev(k, LOG)];
            }
        }
    } else {
        // ---- LAST: CTA = (channel of the chunk, inner tile); loop over samples
        const int64_t tiles = FINEST ? 1 : (inner + W - 1) / W;
        const int64_t cc = blockIdx.x / tiles;
        const int64_t tile = blockIdx.x - cc * tiles;
        const int64_t i0 = tile * W;
        const int64_t i_lim = FINEST ? 1 : inner - i0;
        float acc[LPT][L];
#pragma unroll
        for (int li = 0; li < LPT; ++li)
#pragma unroll
            for (int k = 0; k < L; ++k) acc[li][k] = 0.0f;
        // per-thread load slots: offset within a sample, shared-memory index
        int64_t goff[EPT];
        int sidx[EPT];
        bool live[EPT];
#pragma unroll
        for (int q = 0; q < EPT; ++q) {
            const int e = threadIdx.x + q * NT;  // U == 1
            const int w = e % W, ja = (e / W) % N, jb = e / (W * N);
            live[q] = e < T::IN_PER_UNIT && w < i_lim;
            goff[q] = (int64_t)(jb * N + ja) * inner + i0 + w;
            sidx[q] = e < T::IN_PER_UNIT ? (jb * RP + ja) * W + w : -1;
        }
        float2 pre[EPT];
        auto fetch = [&](int64_t s) {
            const int64_t base = src_base(a, s);
#pragma unroll
            for (int q = 0; q < EPT; ++q)
                pre[q] = live[q] ? ld_src<SRC>(a.src, base + goff[q]) : make_float2(0.f, 0.f);
        };
        int tb, te;
        slice_samples(a, tb, te);
        if (tb < te) fetch(cc * a.tc + tb);
        for (int ts = tb; ts < te; ++ts) {
#pragma unroll
            for (int q = 0; q < EPT; ++q)
                if (sidx[q] >= 0) sm[sidx[q]] = pre[q];
            if (ts + 1 < te) fetch(cc * a.tc + ts + 1);  // in flight during this sample
            __syncthreads();
            for (int l = threadIdx.x; l < T::LINES_A; l += NT) {
                const int jb = l / W, w = l % W;
                float2* row = sm + jb * RP * W + w;
                float2 v[L];
#pragma unroll
                for (int j = 0; j < L; ++j) v[j] = (j < N) ? row[j * W] : make_float2(0.f, 0.f);
                fft_dif<L, true>(v);
#pragma unroll
                for (int k = 0; k < L; ++k) row[k * W] = v[brev(k, LOG)];
            }
            __syncthreads();
#pragma unroll
            for (int li = 0; li < LPT; ++li) {
                const int l = threadIdx.x + li * NT;
                if (l < T::LINES_B) {
                    const int ka = l / W, w = l % W;
                    const float2* col = sm + ka * W + w;
                    float2 v[L];
#pragma unroll
                    for (int j = 0; j < L; ++j) v[j] = (j < N) ? col[j * RP * W] : make_float2(0.f, 0.f);
                    fft_dif<L, true>(v);
#pragma unroll
                    for (int k = 0; k < L; ++k) acc[li][k] += cnorm(v[brev(k, LOG)]);
                }
            }
            __syncthreads();
        }
        const double fs = a.fold_scale != 0.0 ? a.fold_scale : 1.0;
#pragma unroll
        for (int li = 0; li < LPT; ++li) {
            const int l = threadIdx.x + li * NT;
            if (l < T::LINES_B) {
                const int ka = l / W, w = l % W;
                if (w < i_lim) {
#pragma unroll
                    for (int k = 0; k < L; ++k)
                        fold_last(a, cc, ((int64_t)k * L + ka) * inner + i0 + w, acc[li][k], fs);
                }
            }
        }
    }
}

// Both axes of an unpadded square level (beam-space pointings, N x N blocks of
// contiguous antennas, MID): CTA = U blocks, one line per thread and
// axis; what bounds it is HBM (an input read and 8 bytes written per antenna).  One pass per
// axis wrote and read the half-transformed blocks once more, and its contiguous axis
// touched 32 lines of memory per warp access: 16 x 16 blocks on 8 x 8, 64 channels x
// 1024 int8 samples, 5.10 + 2.43 -> 2.25 ms beside the chunk before's last pass.
template <int N, int SRC>
__global__ void __launch_bounds__(N == 32 ? 128 : 256) level_unpadded(Pass p, PassArgs a) {
    constexpr int NT = N == 32 ? 128 : 256, U = NT / N, LOG = ilog2(N), RP = N + 1, BLOCK = N * RP;
    __shared__ float2 sm[U * BLOCK];
    __shared__ int64_t from[U], to[U];
    const int tid = threadIdx.x;
    const int64_t u0 = (int64_t)blockIdx.x * U, units = a.S * p.outer;
    if (tid < U) {
        const int64_t s = (u0 + tid) / p.outer, o = (u0 + tid) - s * p.outer;
        from[tid] = u0 + tid < units ? src_base(a, s) + o * N * N : -1;
        to[tid] = s * a.dst_stride + o * N * N;
    }
    __syncthreads();
    const int u = tid / N, l = tid % N;
    float2 v[N];
    if constexpr (SRC == SRC_CI8 && N >= 8) {
        // int8: the thread's own line (2 N bytes), consecutive threads consecutive lines
        const char2* line = reinterpret_cast<const char2*>(a.src) + from[u] + l * N;
        if (from[u] < 0) {
#pragma unroll
            for (int j = 0; j < N; ++j) v[j] = make_float2(0.f, 0.f);
        } else if ((reinterpret_cast<uintptr_t>(a.src) & 15) == 0) {
#pragma unroll
            for (int q = 0; q < N / 8; ++q) {
                const uint4 x = __ldg(reinterpret_cast<const uint4*>(line) + q);
                const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    v[8 * q + k] = make_float2((float)(int8_t)(w[k >> 1] >> (16 * (k & 1))),
                                               (float)(int8_t)(w[k >> 1] >> (16 * (k & 1) + 8)));
            }
        } else {
#pragma unroll
            for (int j = 0; j < N; ++j) v[j] = ld_src<SRC>(line, j);
        }
    } else {
        // runs of memory through shared memory, all of a thread's loads together
        float2 x[N];
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const int e = tid + NT * q, ub = e / (N * N), r = e % (N * N);
            x[q] = from[ub] >= 0 ? ld_src<SRC>(a.src, from[ub] + r) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const int e = tid + NT * q, ub = e / (N * N), r = e % (N * N);
            sm[ub * BLOCK + (r / N) * RP + r % N] = x[q];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = sm[u * BLOCK + l * RP + j];
        // (the thread writes back to its own line: no barrier in between)
    }
    fft_dif<N, false>(v);
#pragma unroll
    for (int k = 0; k < N; ++k) sm[u * BLOCK + l * RP + k] = v[brev(k, LOG)];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = sm[u * BLOCK + j * RP + l];
    fft_dif<N, false>(v);
    if (from[u] < 0) return;
    float2* d = a.dst + to[u] + l;
#pragma unroll
    for (int k = 0; k < N; ++k) d[k * N] = v[brev(k, LOG)];
}

// Finest-level MID pass, persistent: the CTA walks groups of U contiguous
// blocks (group g, g + gridDim.x, ...), loading the next group two elements
// per thread per load (4-byte int8 or 16-byte float loads, coalesced) into
// registers while the current group is transformed.  Requires every group to
// lie inside one sample (outer % U == 0) and 16-byte aligned group bases.
template <int L, int SRC>
__global__ void __launch_bounds__(LevelTile<L, true, MODE_MID>::THREADS)
level_finest_stream(Pass p, PassArgs a) {
    using T = LevelTile<L, true, MODE_MID>;
    constexpr int N = T::N, U = T::U, RP = T::RP, UPL = T::UPL, NT = T::THREADS;
    constexpr int LOG = ilog2(L);
    constexpr int PER_GROUP = U * N * N;
    constexpr int PAIRS = PER_GROUP / 2 / NT;  // two-element loads per thread per group
    static_assert(PER_GROUP % (2 * NT) == 0, "group must split evenly into pairs");
    using Pair = typename std::conditional<SRC == SRC_CI8, char4, float4>::type;
    extern __shared__ float2 sm[];
    const int64_t groups = a.S * p.outer / U;

    auto group_src = [&](int64_t g) -> const Pair* {
        const int64_t ug = g * U;                    // first unit: (sample, outer block)
        const int64_t s = ug / p.outer, o = ug - s * p.outer;
        return reinterpret_cast<const Pair*>(
            (SRC == SRC_CI8 ? (const char*)a.src + 2 * (src_base(a, s) + o * N * N)
                            : (const char*)a.src + 8 * (src_base(a, s) + o * N * N)));
    };
    Pair pre[PAIRS];
    auto fetch = [&](int64_t g) {
        const Pair* src = group_src(g);
#pragma unroll
        for (int q = 0; q < PAIRS; ++q) pre[q] = src[threadIdx.x + q * NT];
    };
    int64_t g = blockIdx.x;
    if (g < groups) fetch(g);
    for (; g < groups; g += gridDim.x) {
        // registers -> shared memory ([u][j_b][j_a] with odd row pitch)
#pragma unroll
        for (int q = 0; q < PAIRS; ++q) {
            const int e = 2 * (threadIdx.x + q * NT);
            const int u = e / (N * N), r = e - u * N * N;
            const int jb = r / N, ja = r - jb * N;  // ja even: both elements in one row
            float2 x0, x1;
            if constexpr (SRC == SRC_CI8) {
                x0 = make_float2((float)pre[q].x, (float)pre[q].y);
                x1 = make_float2((float)pre[q].z, (float)pre[q].w);
            } else {
                x0 = make_float2(pre[q].x, pre[q].y);
                x1 = make_float2(pre[q].z, pre[q].w);
            }
            float2* d = sm + u * UPL + jb * RP + ja;
            d[0] = x0;
            d[1] = x1;
        }
        if (g + gridDim.x < groups) fetch(g + gridDim.x);  // in flight during this group
        __syncthreads();
        for (int l = threadIdx.x; l < T::LINES_A; l += NT) {
            const int u = l / N, jb = l - u * N;
            float2* row = sm + u * UPL + jb * RP;
            float2 v[L];
#pragma unroll
            for (int j = 0; j < L; ++j) v[j] = (j < N) ? row[j] : make_float2(0.f, 0.f);
            fft_dif<L, true>(v);
#pragma unroll
            for (int k = 0; k < L; ++k) row[k] = v[brev(k, LOG)];
        }
        __syncthreads();
        const int64_t ug0 = g * U;
        const int64_t s = ug0 / p.outer, o0 = ug0 - s * p.outer;
        float2* dst0 = a.dst + s * a.dst_stride + o0 * (int64_t)L * L;
        for (int l = threadIdx.x; l < T::LINES_B; l += NT) {
            const int u = l / L, ka = l - u * L;
            const float2* col = sm + u * UPL + ka;
            float2 v[L];
#pragma unroll
            for (int j = 0; j < L; ++j) v[j] = (j < N) ? col[j * RP] : make_float2(0.f, 0.f);
            fft_dif<L, true>(v);
            float2* d = dst0 + (int64_t)u * L * L + ka;
#pragma unroll
            for (int k = 0; k < L; ++k) d[k * L] = v[brev(k, LOG)];
        }
        __syncthreads();
    }
}

// LAST pass of a coarser level (inner > 1: its source is the scratch buffer), 4 to 32
// points per axis.
//
// What bounds it is FP32 arithmetic and its issue slots (8 points: HBM): axis a is
// transformed straight from the registers that the next sample's inputs were loaded
// into (no staging), and axis b and |F|^2 run two neighbouring columns per instruction
// (f32x2).  The columns between the axes lie in shared memory with real and imaginary
// parts apart, so that a pair of columns is one 8-byte load; two buffers leave one
// barrier per sample.  CTAs are small (128 threads) so that several are in different
// phases on an SM; 16 points with many columns run 3% faster at 256.  Measured, serial:
//   16 points, 1024 columns (64 blocks of 16 x 16, 64 channels x 1024 samples): 13.7 -> 12.0 ms
//   8 points, 262144 columns (three levels, 8 x 64): 4.65 -> 3.86 ms (5.0 TB/s; with two
//     samples loaded ahead and fewer CTAs 4.51)
//   32 points, 64 columns (4 x 4 tiles on 16 x 16, 16 channels x 512): 6.9 -> 5.76 ms
template <int L, int W_>
struct LevelLast {
    static constexpr int N = L / 2;
    static constexpr int W = W_;                // columns per CTA
    static constexpr int NT = N * W;            // lines along axis a, and pairs (L * W / 2) along axis b
    static constexpr int JP = L * W + (W < 32 ? W : 0);  // floats per j_b: a warp's j_b on different banks
    static constexpr int PLANE = N * JP;        // floats of one part of one sample
    static constexpr size_t SMEM = 2 * 2 * (size_t)PLANE * sizeof(float);
    static constexpr int CTAS = 128 * (L >= 32 ? 2 : L == 16 ? 4 : 8) / NT;  // 255, 128 and 64 registers
    static constexpr int AHEAD = L >= 8 ? 1 : 2;  // samples loaded ahead
};

template <int L, int W_>
__global__ void __launch_bounds__(LevelLast<L, W_>::NT, LevelLast<L, W_>::CTAS) level_last(Pass p, PassArgs a) {
    using T = LevelLast<L, W_>;
    constexpr int N = T::N, W = T::W, JP = T::JP, PLANE = T::PLANE, LOG = ilog2(L), D = T::AHEAD;
    extern __shared__ float planes[];  // [2 samples][re, im][j_b][k_a][W]
    const int64_t inner = p.inner;
    const int64_t tiles = (inner + W - 1) / W;
    const int64_t cc = blockIdx.x / tiles;
    const int64_t i0 = (blockIdx.x - cc * tiles) * W;
    // this CTA's samples of the channel
    int tb, te;
    slice_samples(a, tb, te);
    const int wa = threadIdx.x % W, jb = threadIdx.x / W;              // axis a: line (j_b, w)
    const int wb = 2 * (threadIdx.x % (W / 2)), ka = threadIdx.x / (W / 2);  // axis b: columns w, w + 1 of k_a
    const bool live = i0 + wa < inner;
    const float2* src = reinterpret_cast<const float2*>(a.src) + (cc * a.tc + tb) * a.src_stride +
                        (int64_t)jb * N * inner + i0 + wa;
    f2x acc[L];
#pragma unroll
    for (int k = 0; k < L; ++k) acc[k] = dup2(0.f);
    float2 pre[D][N];
    auto fetch = [&](float2 (&d)[N]) {
#pragma unroll
        for (int j = 0; j < N; ++j) d[j] = live ? __ldg(src + (int64_t)j * inner) : make_float2(0.f, 0.f);
        src += a.src_stride;
    };
    auto sample = [&](int ts, float2 (&mine)[N]) {
        float* re = planes + ((ts - tb) & 1) * 2 * PLANE;
        float* im = re + PLANE;
        {
            float2 v[L];
#pragma unroll
            for (int j = 0; j < L; ++j) v[j] = j < N ? mine[j < N ? j : 0] : make_float2(0.f, 0.f);
            if (ts + D < te) fetch(mine);  // in flight during this sample (and the D - 1 after it)
            fft_dif<L, true>(v);
#pragma unroll
            for (int k = 0; k < L; ++k) {
                re[jb * JP + k * W + wa] = v[brev(k, LOG)].x;
                im[jb * JP + k * W + wa] = v[brev(k, LOG)].y;
            }
        }
        __syncthreads();  // this sample's lines are complete, and everyone is done with the other buffer
        f2x x[L], y[L];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            x[j].v = *reinterpret_cast<const unsigned long long*>(re + j * JP + ka * W + wb);
            y[j].v = *reinterpret_cast<const unsigned long long*>(im + j * JP + ka * W + wb);
        }
        fft_dif2<L, true>(x, y);
#pragma unroll
        for (int k = 0; k < L; ++k) {
            const f2x u = x[brev(k, LOG)], v = y[brev(k, LOG)];
            acc[k] = add2(acc[k], fma2(u, u, mul2(v, v)));
        }
    };
#pragma unroll
    for (int d = 0; d < D; ++d)
        if (tb + d < te) fetch(pre[d]);
    for (int ts = tb; ts < te; ts += D) {
#pragma unroll
        for (int d = 0; d < D; ++d)
            if (ts + d < te) sample(ts + d, pre[d]);
    }
    if (i0 + wb >= inner) return;  // inner is even: both columns or neither
    const double fs = a.fold_scale != 0.0 ? a.fold_scale : 1.0;
#pragma unroll
    for (int k = 0; k < L; ++k) {
        const float2 v = unpack2(acc[k]);
        const int64_t e = ((int64_t)k * L + ka) * inner + i0 + wb;
        if (gridDim.y > 1) {  // as fold_last
            *reinterpret_cast<float2*>(a.part + ((int64_t)blockIdx.y * a.S + cc) * a.P_stride + e) = v;
        } else {
            double2* P = reinterpret_cast<double2*>(a.P + (a.c0 + cc) * a.P_stride + e);
            double2 s = *P;
            s.x += fs * (double)v.x;
            s.y += fs * (double)v.y;
            *P = s;
        }
    }
}

// f(LevelLast of this shape), or not supported.
template <int L, class F>
cudaError_t with_level_last(int64_t inner, F&& f) {
    switch (level_last_columns(L, inner)) {
        case 256 / L: return f(LevelLast<L, 256 / L>{});
        case 512 / L:
            if constexpr (L == 16) return f(LevelLast<L, 512 / L>{});
        default: return cudaErrorNotSupported;
    }
}

template <int L, bool FINEST, int MODE, int SRC>
cudaError_t launch_level_t(const Pass& p, const PassArgs& a, cudaStream_t st) {
    using T = LevelTile<L, FINEST, MODE>;
    const int64_t tiles = FINEST ? 1 : (p.inner + T::W - 1) / T::W;
    const int64_t blocks = (MODE == MODE_LAST) ? a.S * tiles
                                               : (a.S * p.outer * tiles + T::U - 1) / T::U;
    if (blocks <= 0) return cudaSuccess;
    if constexpr (FINEST && MODE == MODE_MID && L <= 32) {
        if (p.n == p.L) {  // unpadded: L x L blocks
            constexpr int NT = L == 32 ? 128 : 256, U = NT / L;
            level_unpadded<L, SRC><<<(unsigned)((a.S * p.outer + U - 1) / U), NT, 0, st>>>(p, a);
            return cudaGetLastError();
        }
    }
    if (p.n == p.L) return cudaErrorInvalidValue;
    if constexpr (FINEST && MODE == MODE_MID && SRC != SRC_P64 && L >= 8) {
        constexpr int PER_GROUP = T::U * T::N * T::N;
        const size_t eb = SRC == SRC_CI8 ? 2 : 8;
        const bool contiguous = p.outer % T::U == 0 && PER_GROUP % (2 * T::THREADS) == 0;
        const bool aligned = (((uintptr_t)a.src) % 16 == 0) && ((PER_GROUP * eb) % 16 == 0) &&
                             ((SRC == SRC_BUF ? a.src_stride * eb : a.N * eb) % 16 == 0);
        if (contiguous && aligned && p.grid_cap > 0) {
            const int64_t groups = a.S * p.outer / T::U;
            const int64_t grid = std::min<int64_t>(groups, p.grid_cap);
            auto ks = level_finest_stream<L, SRC>;
            cudaError_t e = smem_limit_once((const void*)ks, T::SMEM);
            if (e != cudaSuccess) return e;
            ks<<<(unsigned)grid, T::THREADS, T::SMEM, st>>>(p, a);
            return cudaGetLastError();
        }
    }
    if constexpr (!FINEST && MODE == MODE_LAST && SRC == SRC_BUF && L <= 32) {
        const cudaError_t e = with_level_last<L>(p.inner, [&](auto t) {
            using LL = decltype(t);
            auto k = level_last<L, LL::W>;
            const cudaError_t e1 = smem_limit_once((const void*)k, LL::SMEM);
            if (e1 != cudaSuccess) return e1;
            k<<<last_grid(a.S * ((p.inner + LL::W - 1) / LL::W), a), LL::NT, LL::SMEM, st>>>(p, a);
            return cudaGetLastError();
        });
        if (e != cudaErrorNotSupported) return e;
    }
    auto k = level_pass<L, FINEST, MODE, SRC>;
    cudaError_t e = smem_limit_once((const void*)k, T::SMEM);
    if (e != cudaSuccess) return e;
    k<<<MODE == MODE_LAST ? last_grid(blocks, a) : dim3((unsigned)blocks), T::THREADS, T::SMEM, st>>>(p, a);
    return cudaGetLastError();
}

// Every forward mode and source of one square level length.
template <int L>
cudaError_t launch_level_len(const Pass& p, const PassArgs& a, cudaStream_t st) {
    return dispatch_mode(p.mode, [&](auto M) -> cudaError_t {
        constexpr int MODE = decltype(M)::value;
        if constexpr (MODE == MODE_MID || MODE == MODE_LAST) {
            return dispatch_src<MODE>(a.src_kind, [&](auto S) {
                return p.inner == 1 ? launch_level_t<L, true, MODE, decltype(S)::value>(p, a, st)
                                    : launch_level_t<L, false, MODE, decltype(S)::value>(p, a, st);
            });
        } else {
            return cudaErrorInvalidValue;
        }
    });
}

// Resident CTAs per SM of the finest-level streaming MID pass (host sizing).
template <int L>
cudaError_t level_stream_blocks_per_sm(int src_kind, int* out) {
    *out = 0;
    if constexpr (L < 8) return cudaSuccess;  // 4-point levels use level_pass
    else return dispatch_src<MODE_MID>(src_kind, [&](auto S) -> cudaError_t {
        using T = LevelTile<L, true, MODE_MID>;
        auto k = level_finest_stream<L, decltype(S)::value>;
        cudaError_t e = smem_limit_once((const void*)k, T::SMEM);
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k, T::THREADS, T::SMEM);
    });
}

// Resident CTAs per SM of the LAST level pass of a given shape (host sizing).
template <int L>
cudaError_t level_last_blocks_per_sm(int64_t inner, int src_kind, int* out) {
    const bool finest = inner == 1;
    if constexpr (L <= 32) {
        cudaError_t e = cudaErrorNotSupported;
        if (src_kind == SRC_BUF)
            e = with_level_last<L>(inner, [&](auto t) {
                using LL = decltype(t);
                auto k = level_last<L, LL::W>;
                const cudaError_t e1 = smem_limit_once((const void*)k, LL::SMEM);
                if (e1 != cudaSuccess) return e1;
                return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k, LL::NT, LL::SMEM);
            });
        if (e != cudaErrorNotSupported) return e;
    }
    return dispatch_src<MODE_LAST>(src_kind, [&](auto S) -> cudaError_t {
        constexpr int SRC = decltype(S)::value;
        if (finest) {
            using T = LevelTile<L, true, MODE_LAST>;
            auto k = level_pass<L, true, MODE_LAST, SRC>;
            cudaError_t e = smem_limit_once((const void*)k, T::SMEM);
            if (e != cudaSuccess) return e;
            return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k, T::THREADS, T::SMEM);
        }
        using T = LevelTile<L, false, MODE_LAST>;
        auto k = level_pass<L, false, MODE_LAST, SRC>;
        cudaError_t e = smem_limit_once((const void*)k, T::SMEM);
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k, T::THREADS, T::SMEM);
    });
}

}  // namespace omni
