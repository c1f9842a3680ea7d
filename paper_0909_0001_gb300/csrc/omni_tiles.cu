// omni_tiles.cu -- tile hybrid (Sec. III): FFT correlation within identical
// tiles placed at arbitrary offsets, brute-force correlation between them.
//
// After the forward passes each sample holds every tile's zero-padded 2-D
// spectrum Y_j(k), k = k1 + L1 k2 (the tile's "synthesized beams").  This pass
// accumulates, for every ordered tile pair (i, j) and frequency k,
//   S_ij(k) += sum over the chunk's samples of Y_i(k) conj(Y_j(k)),
// in FP32 registers over the chunk, then in an FP64 complex accumulator
// [C][n_tiles][n_tiles][K].  S_ji = conj S_ij, so only pairs of tile groups with
// i's group <= j's are summed and both orders are folded.  The inverse 2-D FFT of S_ij gives the visibility
// of every antenna pair (a in tile i, b in tile j) with intra-tile offset
// m_a - m_b = D: the convolution theorem of Sec. II.C applied to two
// different tiles, exact because of the padding.
#include "omni_fft_common.cuh"
#include "omni_tma.cuh"

#include <algorithm>

namespace omni {
namespace {

// What bounds the sum is FP32 arithmetic: 4 fused multiply-adds per tile pair,
// frequency and sample against 8 bytes per tile.  A lane is one frequency and a
// thread holds an 8 x 8 block of pairs (128 sums), so a sample costs 16 shared
// loads (32 cycles of the SM's shared memory per warp) for 256 multiply-adds (64
// cycles of its FP32 lanes): a 2 x 16 block, 18 loads for 128 multiply-adds, kept
// the FP32 pipe at 38%.  Twelve warps of 168 registers fill the register file.
// Half of the pairs are the other half's conjugates and are not summed.
// 64 tiles of 16 x 16 antennas, 8 channels x 1024 samples: 10.3 -> 3.7 ms.
// (Pairs of tiles in packed two-lane multiply-adds, the same block: 6.4 ms.)
constexpr int kXK = 32;       // frequencies per CTA (one per lane)
constexpr int kXG = 8;        // tiles per group; a warp holds one pair of groups
constexpr int kXWarps = 12;   // most warps per CTA
constexpr int kXRows = 64;    // most tiles per CTA
constexpr int kXSamples = 4;  // samples per stage
constexpr int kXStages = 3;
constexpr int kXA = 3, kXB = 4;  // beyond kXRows tiles: groups i x groups j of a CTA (one pair per warp)
constexpr size_t kXBar = 128;    // the stages' barriers, before the stages
static_assert((kXA + kXB) * kXG <= kXRows && kXA * kXB == kXWarps, "rectangular split");
static_assert(kXBar + (size_t)kXStages * kXSamples * kXRows * kXK * 8 <= 227 * 1024, "shared memory of one CTA");

// How the pairs of groups gi <= gj are split over CTAs and warps.  XS_FULL: up to 64
// tiles a CTA reads every tile and its warps take consecutive pairs of the triangle;
// beyond, a CTA takes kXA x kXB groups (24 + 32 tiles) touching the triangle.  XS_QUAD,
// XS_PAIR: rectangles of 2 x 2 groups and single pairs of groups, for grids that would
// leave SMs idle.
enum XForm : int { XS_FULL = 0, XS_QUAD = 1, XS_PAIR = 2 };
struct XSplit {
    int G;      // groups
    int parts;  // CTAs per (channel, frequency tile)
    int warps;  // per CTA
    int A, B;   // rectangle: groups i x groups j
    bool tri;
    __host__ __device__ int first_col(int rb) const { return rb * A / B; }
    // stage rows per sample: tiles i and, apart from them, tiles j (0: the same rows)
    __host__ __device__ int rows_i(int NT) const { return tri ? NT : A * kXG; }
    __host__ __device__ int rows_j() const { return tri ? 0 : B * kXG; }
    __host__ __device__ int rows() const { return tri ? G * kXG : (A + B) * kXG; }
    size_t smem() const { return kXBar + (size_t)kXStages * kXSamples * rows() * kXK * sizeof(float2); }
};
__host__ __device__ inline XSplit xsplit(int NT, int form) {
    XSplit x{};
    x.G = (NT + kXG - 1) / kXG;
    x.tri = form == XS_FULL && NT <= kXRows;
    if (x.tri) {
        const int pairs = x.G * (x.G + 1) / 2;
        x.parts = (pairs + kXWarps - 1) / kXWarps;
        x.warps = (pairs + x.parts - 1) / x.parts;
    } else {
        x.A = form == XS_FULL ? kXA : form == XS_QUAD ? 2 : 1;
        x.B = form == XS_FULL ? kXB : x.A;
        const int rows = (x.G + x.A - 1) / x.A, cols = (x.G + x.B - 1) / x.B;
        for (int rb = 0; rb < rows; ++rb) x.parts += cols - x.first_col(rb);
        x.warps = x.A * x.B;
    }
    return x;
}

// XS_FULL where it gives every SM a CTA; else the form whose busiest SM has the least to
// do: the warps that each of its four schedulers runs, but no less than the 1.5 times as
// long that a warp alone takes, for each set of CTAs that fits (ties: the form that loads
// less).  With XS_FULL alone, its CTAs cut to fewer warps that each still read every tile:
// 64 tiles of 8 x 8, one channel of 64 samples, 172 -> 125 us a pass; 64 of 4 x 4, 4
// channels of 512, 441 -> 266; 90 of 2 x 2, 4 channels of 512, 410 -> 237 (a 2 x 16 block
// of pairs per thread: 127, 319 and 283).
inline int xs_form(int NT, int64_t units) {
    const int64_t sms = 152;
    int best = XS_FULL;
    if (units * xsplit(NT, XS_FULL).parts >= sms) return best;
    double least = 0.0;
    for (int form = XS_FULL; form <= XS_PAIR; ++form) {
        const XSplit x = xsplit(NT, form);
        const int64_t each = (units * x.parts + sms - 1) / sms, resident = (int64_t)(227 * 1024 / x.smem());
        const double t = std::max((double)((each * x.warps + 3) / 4), 1.5 * (double)((each + resident - 1) / resident));
        if (form == XS_FULL || t < least) best = form, least = t;
    }
    return best;
}

// float -> double where the sums are folded: as plain conversions the compiler moved
// all 128 of them above the bounds checks and spilled 700 bytes
__device__ __forceinline__ double widen(float x) {
    double d;
    asm volatile("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(x));
    return d;
}

// 8-byte asynchronous copy global -> shared
__device__ __forceinline__ void cp_async8(float2* dst, const float2* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// CTA = (channel of the chunk, frequency tile, part of the pairs); the parts of one
// frequency tile are adjacent, so that they read its spectra from L2.  TMA: one
// thread brings each stage in with tensor-map boxes two stages ahead (K even: 16-byte
// rows); else every thread copies its share asynchronously, as far ahead (a tile of one
// antenna, K = 1; stages filled and waited for in turn, 64 tiles, 4 channels x 1024
// samples, 0.46 (one sample ahead, 2 x 16 pairs per thread) -> 15.4 ms, so: 0.41).  What a stage has no
// value for (tiles past the last, lanes past K) is whatever shared memory held: those sums
// are not written.
template <bool TMA>
__global__ void __launch_bounds__(kXWarps * 32, 1) xspec(Pass p, PassArgs a, int form, int few,
                                                         const __grid_constant__ CUtensorMap map0,
                                                         const __grid_constant__ CUtensorMap map1) {
    extern __shared__ __align__(128) unsigned char dsm[];
    uint64_t* full = reinterpret_cast<uint64_t*>(dsm);  // [kXStages], then one that nothing arrives on (test hook)
    float2* ring = reinterpret_cast<float2*>(dsm + kXBar);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int NT = (int)p.outer;
    const int64_t K = p.L;
    const int64_t ktiles = (K + kXK - 1) / kXK;
    const XSplit xs = xsplit(NT, form);
    int64_t b = blockIdx.x;
    const int part = (int)(b % xs.parts);
    b /= xs.parts;
    const int64_t kt = b % ktiles, cc = b / ktiles;
    // this warp's groups, and the stage rows that hold their tiles: n0 rows of tiles t0 .. for
    // each of the stage's samples, then n1 rows of tiles t1 .. for each
    int gi, gj, ri, rj, t0 = 0, t1 = 0;
    const int n0 = xs.rows_i(NT), n1 = xs.rows_j();
    bool live;
    if (xs.tri) {
        int q = part * xs.warps + warp;
        gi = 0;
        while (gi < xs.G && q >= xs.G - gi) q -= xs.G - gi++;
        gj = gi + q;
        live = gi < xs.G;
        if (!live) gi = gj = 0;
        ri = gi * kXG;
        rj = gj * kXG;
    } else {
        const int cols = (xs.G + xs.B - 1) / xs.B;
        int rb = 0, q = part;
        while (q >= cols - xs.first_col(rb)) q -= cols - xs.first_col(rb++);
        const int cb = xs.first_col(rb) + q;
        t0 = rb * xs.A * kXG;
        t1 = cb * xs.B * kXG;
        ri = (warp / xs.B) * kXG;
        rj = (warp % xs.B) * kXG;
        gi = rb * xs.A + warp / xs.B;
        gj = cb * xs.B + warp % xs.B;
        live = gi <= gj && gj < xs.G;
    }
    const int jn = n1 ? n1 : n0;  // rows of tiles j per sample, and where they begin
    const int jofs = n1 ? kXSamples * n0 * kXK : 0;
    const int64_t stage_elems = (int64_t)kXSamples * xs.rows() * kXK;
    const int tc = a.tc, stages = (tc + kXSamples - 1) / kXSamples;
    const long long budget = a.force_expire ? kTestWaitCycles : kWaitCycles;
    if (tid == 0) {
        for (int i = 0; i <= kXStages; ++i) mbar_init(full + i, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    __syncthreads();
    auto fill = [&](int n) {  // stage n: samples kXSamples n .. of this channel
        float2* dst = ring + (n % kXStages) * stage_elems;
        if constexpr (TMA) {
            if (tid == 0) {
                uint64_t* bar = full + n % kXStages;
                mbar_expect_tx(bar, (uint32_t)((n0 + n1) * kXK * kXSamples * sizeof(float2)));
                const int x = (int)(2 * kXK * kt), z = (int)(cc * tc + n * kXSamples);
                tma_load3(dst, &map0, x, t0, z, bar);
                if (n1) tma_load3(dst + jofs, &map1, x, t1, z, bar);
            }
        } else {
            const int nk = (int)(K - kt * kXK < kXK ? K - kt * kXK : kXK), nr = n0 + n1;
            const int ns = min(kXSamples, tc - n * kXSamples);
            for (int e = tid; e < nk * nr * ns; e += blockDim.x) {
                const int k = e % nk, r = (e / nk) % nr, s = e / (nk * nr);
                const int tile = r < n0 ? t0 + r : t1 + r - n0;
                float2* d = dst + (r < n0 ? (s * n0 + r) * kXK : jofs + (s * n1 + r - n0) * kXK) + k;
                if (tile < NT)
                    cp_async8(d, reinterpret_cast<const float2*>(a.src) + src_base(a, cc * tc + n * kXSamples + s) +
                                     (int64_t)tile * K + kt * kXK + k);
            }
        }
    };
    float ar[kXG][kXG], ai[kXG][kXG];
#pragma unroll
    for (int u = 0; u < kXG; ++u)
#pragma unroll
        for (int v = 0; v < kXG; ++v) ar[u][v] = ai[u][v] = 0.f;
    bool failed = false;
    int issued = 0;
    for (int i = 0; i < kXStages - 1; ++i) {
        if (issued < stages) fill(issued++);
        if constexpr (!TMA) cp_async_commit();
    }
    for (int n = 0; n < stages; ++n) {
        if constexpr (!TMA) cp_async_wait<kXStages - 2>();  // this thread's copies of stage n
        // every warp is past stage n - 1: its buffer takes stage n + 2
        if (__syncthreads_or(failed)) break;
        if (issued < stages) fill(issued++);
        if constexpr (TMA)
            failed = (a.force_expire && n == 0) ? !wait_bar(full + kXStages, 0, budget)
                                                : !wait_bar(full + n % kXStages, (n / kXStages) & 1, budget);
        else
            cp_async_commit();  // one group per stage, empty past the last
        const float2* st = ring + (n % kXStages) * stage_elems + lane;
        const int ns = min(kXSamples, tc - n * kXSamples);
        if (live && !failed) {
#pragma unroll 1
            for (int s = 0; s < ns; ++s) {
                const float2* yr = st + (s * n0 + ri) * kXK;
                const float2* zr = st + jofs + (s * jn + rj) * kXK;
                float2 y[kXG];
#pragma unroll
                for (int u = 0; u < kXG; ++u) y[u] = yr[u * kXK];
#pragma unroll
                for (int v = 0; v < kXG; ++v) {
                    const float2 z = zr[v * kXK];
#pragma unroll
                    for (int u = 0; u < kXG; ++u) {  // y conj(z)
                        ar[u][v] = fmaf(y[u].x, z.x, fmaf(y[u].y, z.y, ar[u][v]));
                        ai[u][v] = fmaf(y[u].y, z.x, fmaf(-y[u].x, z.y, ai[u][v]));
                    }
                }
            }
        }
        // these loads come before the box that takes the buffer after the next barrier (the
        // asynchronous proxy's writes are not ordered behind them by the barrier alone)
        if constexpr (TMA) fence_async_smem();
    }
    if constexpr (TMA) {
        // no box is in flight when the CTA leaves (each was waited for above unless a wait gave up)
        if (__syncthreads_or(failed)) {
            if (tid == 0) {
                for (int n = max(0, issued - kXStages); n < issued; ++n) wait_bar(full + n % kXStages, (n / kXStages) & 1);
                atomicExch(a.err, 1);
            }
            return;
        }
    }
    const int64_t k = kt * kXK + lane;
    if (!live || k >= K) return;
    double2* S = reinterpret_cast<double2*>(a.P + (a.c0 + cc) * a.P_stride) + k;
    const int i0 = gi * kXG, j0 = gj * kXG;
    if (few) {
        // fewer CTAs than SMs, whose warps would wait for one load after another (9 tiles of
        // 12 x 12, one channel x 8 samples: the pass 35 us, so 13): reductions in L2, one per
        // value of a launch, so that the order of the sums stays that of the launches
#pragma unroll
        for (int u = 0; u < kXG; ++u)
#pragma unroll
            for (int v = 0; v < kXG; ++v) {
                const int i = i0 + u, j = j0 + v;
                if (i < NT && j < NT) {
                    const double re = widen(ar[u][v]), im = widen(ai[u][v]);
                    double* f = reinterpret_cast<double*>(S + (i * NT + j) * K);
                    atomicAdd(f, re);
                    atomicAdd(f + 1, im);
                    if (gi != gj) {
                        double* m = reinterpret_cast<double*>(S + (j * NT + i) * K);
                        atomicAdd(m, re);
                        atomicAdd(m + 1, -im);
                    }
                }
            }
        return;
    }
    // both orders of each pair; kXF of them at a time, their loads together
    constexpr int kXF = 2;
#pragma unroll
    for (int u = 0; u < kXG; ++u) {
        const int i = i0 + u;
#pragma unroll
        for (int v0 = 0; v0 < kXG; v0 += kXF) {
            double2 f[kXF], m[kXF];
#pragma unroll
            for (int v = 0; v < kXF; ++v) {
                const int j = j0 + v0 + v;
                if (i < NT && j < NT) {
                    f[v] = S[(i * NT + j) * K];
                    if (gi != gj) m[v] = S[(j * NT + i) * K];
                }
            }
#pragma unroll
            for (int v = 0; v < kXF; ++v) {
                const int j = j0 + v0 + v;
                if (i < NT && j < NT) {
                    const double re = widen(ar[u][v0 + v]), im = widen(ai[u][v0 + v]);
                    S[(i * NT + j) * K] = make_double2(f[v].x + re, f[v].y + im);
                    if (gi != gj) S[(j * NT + i) * K] = make_double2(m[v].x + re, m[v].y - im);
                }
            }
        }
    }
}

}  // namespace

int64_t xspec_ctas_per_channel(const Pass& p) {
    return ((p.L + kXK - 1) / kXK) * (int64_t)xsplit((int)p.outer, XS_FULL).parts;
}

cudaError_t xspec_occupancy(const Pass& p, int* blocks_per_sm) {
    const XSplit xs = xsplit((int)p.outer, XS_FULL);
    cudaError_t e = smem_limit_once((const void*)xspec<true>, xs.smem());
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, xspec<true>, 32 * xs.warps, xs.smem());
}

cudaError_t launch_xspec(const Pass& p, const PassArgs& a, cudaStream_t st) {
    if (a.src_kind != SRC_BUF || !a.err) return cudaErrorInvalidValue;
    const int64_t ktiles = (p.L + kXK - 1) / kXK;
    if (a.S <= 0 || a.tc <= 0) return cudaSuccess;
    const int NT = (int)p.outer, form = xs_form(NT, a.S * ktiles);
    const XSplit xs = xsplit(NT, form);
    const int64_t blocks = a.S * ktiles * xs.parts;
    // tensor maps want 16-byte aligned rows; an odd K is a tile of one antenna
    const bool tma = p.L % 2 == 0 && reinterpret_cast<uintptr_t>(a.src) % 16 == 0;
    CUtensorMap m0{}, m1{};
    if (tma) {
        const int64_t samples = a.S * a.tc;
        cudaError_t e = encode_spectra_map(a.src, p.L, NT, samples, 2 * kXK, xs.rows_i(NT), kXSamples, &m0);
        if (e == cudaSuccess && !xs.tri)
            e = encode_spectra_map(a.src, p.L, NT, samples, 2 * kXK, xs.rows_j(), kXSamples, &m1);
        if (e != cudaSuccess) return e;
    }
    auto kern = tma ? xspec<true> : xspec<false>;
    cudaError_t e = smem_limit_once((const void*)kern, xs.smem());
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)blocks, 32 * xs.warps, xs.smem(), st>>>(p, a, form, blocks < 152, m0, m1);
    return cudaGetLastError();
}

}  // namespace omni
