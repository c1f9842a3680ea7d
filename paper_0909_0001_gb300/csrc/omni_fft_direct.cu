// omni_fft_direct.cu -- direct-DFT axis transforms.
//
// Axes of any length (non-powers of two, and the degenerate single-antenna
// lattice).  Up to kDftMax points, as shared memory allows, and for enough work: tiles of
// lines in shared memory, sums shared between the outputs of opposite and shifted bins;
// else one thread per output.
#include "omni_fft_common.cuh"

#include <algorithm>
#include <type_traits>

namespace omni {

// ---------------------------------------------------------------- direct DFT passes

// Any length: one thread per output value, X[k] = sum_j x[j] w_L^(jk mod L).
// SLICED (LAST over slices of the samples): four terms' loads together.  Unsliced, one
// plain loop from sample 0: what the compiler makes of it is 1.4 times as fast as that (500
// points, 128 columns, 8 samples: 0.19 against 0.27 ms), and 1.8 times as fast as the same
// loop between two bounds (0.35; in four slices 0.17, four loads together 0.10).  Both in
// one kernel cost the plain loop a quarter.
template <int MODE, int SRC, bool SLICED>
__global__ void __launch_bounds__(256) pass_direct(Pass p, PassArgs a) {
    const int64_t flat = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t inner = p.inner;
    const int L = p.L, n = p.n, Q = p.q_out;
    auto term = [&](float2& sum, float2 x, float2 w) {
        sum.x = fmaf(x.x, w.x, fmaf(-x.y, w.y, sum.x));
        sum.y = fmaf(x.x, w.y, fmaf(x.y, w.x, sum.y));
    };
    if constexpr (MODE == MODE_LAST) {
        const int64_t per = (int64_t)L * inner;
        if (flat >= a.S * per) return;
        const int64_t cc = flat / per;
        const int64_t r = flat - cc * per;
        const int k = (int)(r / inner);
        const int64_t i = r - (int64_t)k * inner;
        float acc = 0.0f;
        if constexpr (!SLICED) {
            for (int tt = 0; tt < a.tc; ++tt) {
                const int64_t base = src_base(a, cc * a.tc + tt) + i;
                float2 sum = make_float2(0.f, 0.f);
                int m = 0;
                for (int j = 0; j < n; ++j) {
                    const float2 x = ld_src<SRC>(a.src, base + (int64_t)j * inner);
                    term(sum, x, __ldg(p.tw + m));
                    m += k;
                    if (m >= L) m -= L;
                }
                acc += cnorm(sum);
            }
        } else {
            constexpr int NB = 4;
            int tb, te;
            slice_samples(a, tb, te);
#pragma unroll 1
            for (int tt = tb; tt < te; ++tt) {
                const int64_t base = src_base(a, cc * a.tc + tt) + i;
                float2 sum = make_float2(0.f, 0.f);
                int m = 0, j = 0;
                for (; j + NB <= n; j += NB) {
                    float2 x[NB], w[NB];
#pragma unroll
                    for (int u = 0; u < NB; ++u) {
                        x[u] = ld_src<SRC>(a.src, base + (int64_t)(j + u) * inner);
                        w[u] = __ldg(p.tw + m);
                        m += k;
                        if (m >= L) m -= L;
                    }
#pragma unroll
                    for (int u = 0; u < NB; ++u) term(sum, x[u], w[u]);
                }
#pragma unroll 1
                for (; j < n; ++j) {
                    term(sum, ld_src<SRC>(a.src, base + (int64_t)j * inner), __ldg(p.tw + m));
                    m += k;
                    if (m >= L) m -= L;
                }
                acc += cnorm(sum);
            }
        }
        fold_last(a, cc, (int64_t)k * inner + i, acc);
    } else {
        const int64_t per = p.outer * (int64_t)Q * inner;
        if (flat >= a.S * per) return;
        const int64_t s = flat / per;
        int64_t r = flat - s * per;
        const int64_t o = r / ((int64_t)Q * inner);
        r -= o * (int64_t)Q * inner;
        const int q = (int)(r / inner);
        const int64_t i = r - (int64_t)q * inner;
        const int k = (MODE == MODE_MID) ? q : inv_bin(q, p.q_shift, L);
        const int64_t base = src_base(a, s) + o * (int64_t)n * inner + i;
        float2 sum = make_float2(0.f, 0.f);
        int m = 0;
        for (int j = 0; j < n; ++j) {
            const float2 x = ld_src<SRC>(a.src, base + (int64_t)j * inner);
            term(sum, x, __ldg(p.tw + m));
            m += k;
            if (m >= L) m -= L;
        }
        const int64_t e = (o * (int64_t)Q + q) * inner + i;
        if constexpr (MODE == MODE_INV_LAST) {
            a.V[(a.c0 + s) * a.V_stride + e] = visibility(sum, a);
        } else {
            a.dst[s * a.dst_stride + e] = sum;
        }
    }
}

// ---------------------------------------------------------------- tiled DFT passes

// One thread per output read every input and a twiddle from L1 for each of its n
// terms (650 GB/s on 24-point axes).  Here a CTA holds a tile of lines in shared
// memory and a thread sums four bins r at once over two lines.  With w^(jr) = c - i s
// the four real sums A = sum xr c, B = sum xi s, C = sum xi c, D = sum xr s give both
//   X[r] = (A + B) + i (C - D)  and  X[-r] = (A - B) + i (C + D),
// and
//  * padded lines (L = 2 n): the sums over even and over odd j apart give X[r + n] too
//    (w^(jn) = (-1)^j): n multiply-adds per output instead of 4 n;
//  * whole lines of even L: inputs j and j + L/2 are added for even r and subtracted
//    for odd r as they are loaded: L instead of 4 L;
//  * whole lines of odd L (beam axes): 2 L.
// Twiddles are read as rows [j][bins 4 g ..] of a table, the same for every lane.  The
// row table bounds the length: kDftMax points, 41 KB.
// 50 tiles of 12 x 12 (24-point axes), 16 channels x 500 samples: 1.62 + 4.23 -> 0.50 + 0.71 ms
// forward, 1.70 + 0.41 -> 0.19 + 0.21 ms inverse (2.7 and 3.9 TB/s; eight loads in flight per
// thread: with one, 0.70 + 1.30 ms).  Padded MID and LAST forms spill 44 and 48 bytes at the
// 80 registers of three CTAs per SM.
constexpr int kDftMax = 192;
constexpr int kDftBins = 4;  // bins r per thread
constexpr size_t kDftSmem = 224 * 1024;  // whole lines reach it at about 160 points

struct DftShape {
    int reps;    // bins r summed: 0 .. n/2 (padded) or 0 .. L/2
    int rows;    // terms j of a sum
    int groups;  // of kDftBins bins
    int kg;      // groups side by side in a CTA
    int lw;      // lines side by side
    int lines;   // lines per CTA
    int held;    // inputs kept per line
    int threads;
    size_t smem;
    bool fold;
};

template <int MODE>
__host__ __device__ constexpr int dft_lines_per_thread() { return MODE == MODE_LAST ? 1 : 2; }

template <int MODE>
__host__ __device__ inline DftShape dft_shape(int L, int n, bool half, bool stage) {
    DftShape d{};
    d.fold = !half && L % 2 == 0;
    d.rows = half ? n : d.fold ? L / 2 : L;
    d.held = half ? n : L;
    d.reps = (half ? n : L) / 2 + 1;
    d.groups = (d.reps + kDftBins - 1) / kDftBins;
    d.kg = d.groups < 8 ? d.groups : 8;
    d.lw = d.groups == 1 ? 128 : d.groups <= 4 ? 64 : 32;
    d.lines = d.lw * dft_lines_per_thread<MODE>();
    d.threads = d.lw * d.kg;
    d.smem = 2 * sizeof(int64_t) * d.lines +
             sizeof(float2) * ((size_t)d.rows * d.groups * kDftBins + (size_t)d.held * (d.lines + 1) +
                               (stage ? (size_t)d.lines * (L + 1 - L % 2) : 0));
    return d;
}

// HALF: padded lines (n = L / 2 inputs); else all L inputs.
template <int MODE, int SRC, bool HALF>
__global__ void __launch_bounds__(256, 3) pass_dft(Pass p, PassArgs a) {
    constexpr int LN = dft_lines_per_thread<MODE>(), KB = kDftBins;
    constexpr int PARTS = HALF ? 2 : 1;   // even and odd j apart
    constexpr int OUTS = HALF ? 4 : 2;    // outputs per bin r
    const int L = p.L, n = p.n;
    const int64_t inner = p.inner;
    const bool rows_out = MODE != MODE_LAST && inner == 1;  // lines contiguous in memory: staged stores
    const DftShape d = dft_shape<MODE>(L, n, HALF, rows_out);
    extern __shared__ __align__(16) unsigned char dft_smem[];
    float2* W = reinterpret_cast<float2*>(dft_smem);                  // [rows][groups * KB]
    const int wp = d.groups * KB;
    float2* in = W + (size_t)d.rows * wp;                             // [held][lines + 1]
    const int ip = d.lines + 1;
    int64_t* sb = reinterpret_cast<int64_t*>(in + (size_t)d.held * ip);
    int64_t* db = sb + d.lines;
    float2* ob = reinterpret_cast<float2*>(db + d.lines);             // rows_out: [lines][op]
    const int op = L + 1 - L % 2;
    const int tid = threadIdx.x;
    for (int e = tid; e < d.rows * wp; e += blockDim.x) {
        const int j = e / wp, r = e - j * wp;
        W[e] = r < d.reps ? __ldg(p.tw + (int)(((int64_t)j * r) % L)) : make_float2(0.f, 0.f);  // (c, -s)
    }
    // this CTA's lines: source and output offsets, -1 past the end
    const int64_t per = MODE == MODE_LAST ? inner : p.outer * inner;
    const int64_t l0 = (int64_t)blockIdx.x * d.lines;
    for (int l = tid; l < d.lines; l += blockDim.x) {
        const int64_t g = l0 + l, s = g / per, r = g - s * per;
        int64_t src = -1, dst = -1;
        if (s < a.S) {
            if constexpr (MODE == MODE_LAST) {
                src = src_base(a, s * a.tc) + r;
                dst = g;  // split into channel and column again at the fold
            } else {
                const int64_t o = r / inner, i = r - o * inner;
                src = src_base(a, s) + o * (int64_t)n * inner + i;
                dst = o * (int64_t)p.q_out * inner + i +
                      (MODE == MODE_INV_LAST ? (a.c0 + s) * a.V_stride : s * a.dst_stride);
            }
        }
        sb[l] = src;
        db[l] = dst;
    }
    __syncthreads();
    const int lx = tid % d.lw, g0 = tid / d.lw;
    const int64_t step = a.src_kind == SRC_BUF ? a.src_stride : a.N;  // LAST: from sample to sample

    float acc[MODE == MODE_LAST ? KB * OUTS : 1];  // LAST: |X|^2 over the samples (LN = 1, one group per pass)
    int tb = 0, te = 1;
    if constexpr (MODE == MODE_LAST) slice_samples(a, tb, te);
    const int passes = (d.groups + d.kg - 1) / d.kg;
    for (int ps = 0; ps < (MODE == MODE_LAST ? passes : 1); ++ps) {
        if constexpr (MODE == MODE_LAST)
#pragma unroll
            for (int e = 0; e < KB * OUTS; ++e) acc[e] = 0.f;
        for (int ts = tb; ts < te; ++ts) {
            // load: terms of one line along memory (contiguous lines), or one term of many lines
            const bool along = inner == 1;
            const int jmax = along ? d.rows : d.lines, dj = blockDim.x % jmax, dl = blockDim.x / jmax;
            int fast = tid % jmax, slow = tid / jmax;
            constexpr int NB = HALF ? 8 : 4;  // loads in flight per thread (twice that, folded)
            const int total = d.rows * d.lines;
            for (int e0 = tid; e0 < total; e0 += NB * (int)blockDim.x) {
                float2 x[NB], y[NB];
                int to[NB];
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    const int j = along ? fast : slow, l = along ? slow : fast;
                    to[u] = e0 + u * (int)blockDim.x < total ? j * ip + l : -1;
                    x[u] = y[u] = make_float2(0.f, 0.f);
                    if (to[u] >= 0 && sb[l] >= 0) {
                        const int64_t at = sb[l] + (int64_t)ts * (MODE == MODE_LAST ? step : 0) + (int64_t)j * inner;
                        x[u] = ld_src<SRC>(a.src, at);
                        if (!HALF && d.fold) y[u] = ld_src<SRC>(a.src, at + (int64_t)d.rows * inner);
                    }
                    fast += dj;
                    slow += dl;
                    if (fast >= jmax) fast -= jmax, ++slow;
                }
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    if (to[u] < 0) continue;
                    if (!HALF && d.fold) {
                        in[to[u]] = cadd(x[u], y[u]);
                        in[to[u] + d.rows * ip] = csub(x[u], y[u]);
                    } else {
                        in[to[u]] = x[u];
                    }
                }
            }
            __syncthreads();
            for (int g = g0 + (MODE == MODE_LAST ? ps * d.kg : 0); g < d.groups;
                 g += MODE == MODE_LAST ? d.groups : d.kg) {
                float s[PARTS][KB][LN][4];  // A, B, C, D with the table's -s: B and D change sign below
#pragma unroll
                for (int h = 0; h < PARTS; ++h)
#pragma unroll
                    for (int b = 0; b < KB; ++b)
#pragma unroll
                        for (int l = 0; l < LN; ++l) s[h][b][l][0] = s[h][b][l][1] = s[h][b][l][2] = s[h][b][l][3] = 0.f;
                auto term = [&](int j, int h) {
                    float2 w[KB], x[LN], y[LN];
                    const float4* w4 = reinterpret_cast<const float4*>(W + (size_t)j * wp + g * KB);
#pragma unroll
                    for (int b = 0; b < KB; b += 2) {
                        const float4 q = w4[b / 2];
                        w[b] = make_float2(q.x, q.y);
                        w[b + 1] = make_float2(q.z, q.w);
                    }
#pragma unroll
                    for (int l = 0; l < LN; ++l) {
                        x[l] = in[j * ip + lx + l * d.lw];
                        y[l] = (!HALF && d.fold) ? in[(d.rows + j) * ip + lx + l * d.lw] : x[l];
                    }
#pragma unroll
                    for (int b = 0; b < KB; ++b)
#pragma unroll
                        for (int l = 0; l < LN; ++l) {
                            const float2 v = (b & 1) ? y[l] : x[l];  // odd bins: the differences
                            s[h][b][l][0] = fmaf(v.x, w[b].x, s[h][b][l][0]);
                            s[h][b][l][1] = fmaf(v.y, w[b].y, s[h][b][l][1]);
                            s[h][b][l][2] = fmaf(v.y, w[b].x, s[h][b][l][2]);
                            s[h][b][l][3] = fmaf(v.x, w[b].y, s[h][b][l][3]);
                        }
                };
                if constexpr (HALF) {
                    int j = 0;
                    for (; j + 1 < d.rows; j += 2) {
                        term(j, 0);
                        term(j + 1, 1);
                    }
                    if (j < d.rows) term(j, 0);
                } else {
#pragma unroll 2
                    for (int j = 0; j < d.rows; ++j) term(j, 0);
                }
                auto emit = [&](int l, int k, float2 v, int slot) {
                    if constexpr (MODE == MODE_LAST) {
                        acc[slot] += cnorm(v);
                    } else {
                        int q = k;
                        if constexpr (MODE != MODE_MID) {
                            q = (k < L - p.q_shift ? k : k - L) + p.q_shift;  // bin k holds lag k or k - L
                            if (q >= p.q_out) return;                        // the padding bin no lag maps to
                        }
                        const int line = lx + l * d.lw;
                        if (rows_out) {
                            ob[line * op + q] = v;
                        } else if (db[line] >= 0) {
                            const int64_t at = db[line] + (int64_t)q * inner;
                            if constexpr (MODE == MODE_INV_LAST)
                                a.V[at] = visibility(v, a);
                            else
                                a.dst[at] = v;
                        }
                    }
                };
#pragma unroll
                for (int b = 0; b < KB; ++b) {
                    const int r = g * KB + b;
                    if (r >= d.reps) continue;
#pragma unroll
                    for (int l = 0; l < LN; ++l)
#pragma unroll
                        for (int h = 0; h < PARTS; ++h) {  // X[+-r], then X[+-r + n]
                            if (h && 2 * r == n) continue;  // r = n / 2: the same two bins again
                            float t[4];
#pragma unroll
                            for (int c = 0; c < 4; ++c)
                                t[c] = !HALF ? s[0][b][l][c]
                                             : (h ? s[0][b][l][c] - s[PARTS - 1][b][l][c]
                                                  : s[0][b][l][c] + s[PARTS - 1][b][l][c]);
                            const int k = h ? r + n : r;
                            const int m = h ? n - r : (r ? L - r : 0);
                            emit(l, k, make_float2(t[0] - t[1], t[2] + t[3]), b * OUTS + 2 * h);
                            if (m != k) emit(l, m, make_float2(t[0] + t[1], t[2] - t[3]), b * OUTS + 2 * h + 1);
                        }
                }
            }
            __syncthreads();
        }
        if constexpr (MODE == MODE_LAST) {
            const int g = g0 + ps * d.kg;
            if (g < d.groups && db[lx] >= 0) {
                const int64_t cc = db[lx] / inner, i = db[lx] - cc * inner;
#pragma unroll
                for (int b = 0; b < KB; ++b) {
                    const int r = g * KB + b;
                    if (r >= d.reps) continue;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h && 2 * r == n) continue;
                        const int k = h ? r + n : r, m = h ? n - r : (r ? L - r : 0);
                        fold_last(a, cc, (int64_t)k * inner + i, acc[b * OUTS + 2 * h]);
                        if (m != k) fold_last(a, cc, (int64_t)m * inner + i, acc[b * OUTS + 2 * h + 1]);
                    }
                }
            }
        }
    }
    if (rows_out) {  // the tile's lines, each contiguous
        const int Q = p.q_out;
        const int dq = blockDim.x % Q, dl = blockDim.x / Q;
        int q = tid % Q, l = tid / Q;
        for (; l < d.lines; q += dq, l += dl) {
            if (q >= Q) {
                q -= Q;
                if (++l >= d.lines) break;
            }
            if (db[l] < 0) continue;
            const float2 v = ob[l * op + q];
            if constexpr (MODE == MODE_INV_LAST)
                a.V[db[l] + q] = visibility(v, a);
            else if constexpr (MODE != MODE_LAST)
                a.dst[db[l] + q] = v;
        }
    }
}

namespace {

// The tiled form of a pass: padded lines (HALF) or whole lines, up to kDftMax points as
// shared memory allows; false: none.
bool dft_form(const Pass& p, DftShape* d, bool* half) {
    if (p.L < 2 || p.L > kDftMax) return false;
    const bool fwd = p.mode == MODE_MID || p.mode == MODE_LAST;
    *half = fwd && 2 * p.n == p.L;
    if (!*half && (p.mode == MODE_LAST || p.n != p.L)) return false;
    const bool stage = p.mode != MODE_LAST && p.inner == 1;
    *d = p.mode == MODE_LAST ? dft_shape<MODE_LAST>(p.L, p.n, *half, stage) : dft_shape<MODE_MID>(p.L, p.n, *half, stage);
    return d->smem <= kDftSmem;
}

// Whether the tiles take S samples (LAST: channels of tc samples), by the terms that the
// pass sums: below, their tables and barriers (2 to 4 us) cost more than they save.  By 530
// passes of 6 to 192 points run in both forms: forward MID passes cross at 2 to 4 M terms
// (24 points, 0.7 M: 13.4 against 8.3 us; 22 M: 18 against 33), inverse MID ones at 1 to 2 M
// (longer lines later), the last at 8 M (14 against 12; 41 M: 18 against 35), LAST passes at
// 2 to 4 M (24 points, 0.9 M: 10.3 against 8.0; 14 M: 13.7 against 22.6).
bool dft_takes(const Pass& p, int64_t S, int64_t tc, DftShape* d, bool* half) {
    const bool last = p.mode == MODE_LAST;
    const double outputs = last ? (double)S * tc * p.L * p.inner : (double)S * p.outer * p.q_out * p.inner;
    const int least = last ? 3 : p.mode == MODE_INV_LAST ? 8 : 4;
    return outputs * p.n >= (double)(least << 20) && dft_form(p, d, half);
}

template <int MODE, int SRC, bool HALF>
cudaError_t launch_dft_t(const Pass& p, const PassArgs& a, const DftShape& d, cudaStream_t st) {
    const int64_t lines = MODE == MODE_LAST ? a.S * p.inner : a.S * p.outer * p.inner;
    auto k = pass_dft<MODE, SRC, HALF>;
    cudaError_t e = smem_limit_once((const void*)k, d.smem);
    if (e != cudaSuccess) return e;
    const int64_t blocks = (lines + d.lines - 1) / d.lines;
    k<<<MODE == MODE_LAST ? last_grid(blocks, a) : dim3((unsigned)blocks), d.threads, d.smem, st>>>(p, a);
    return cudaGetLastError();
}

template <int MODE, int SRC>
cudaError_t launch_direct_t(const Pass& p, const PassArgs& a, cudaStream_t st) {
    const int64_t work = (MODE == MODE_LAST) ? a.S * (int64_t)p.L * p.inner
                                             : a.S * p.outer * (int64_t)p.q_out * p.inner;
    if (work <= 0) return cudaSuccess;
    DftShape d;
    bool half;
    if (dft_takes(p, a.full_S ? a.full_S : a.S, a.tc, &d, &half)) {
        if constexpr (MODE == MODE_MID || MODE == MODE_LAST)
            if (half) return launch_dft_t<MODE, SRC, true>(p, a, d, st);
        if constexpr (MODE != MODE_LAST) return launch_dft_t<MODE, SRC, false>(p, a, d, st);
    }
    const int threads = 256;
    const int64_t blocks = (work + threads - 1) / threads;
    if (MODE == MODE_LAST && a.split > 1)
        pass_direct<MODE, SRC, MODE == MODE_LAST><<<last_grid(blocks, a), threads, 0, st>>>(p, a);
    else
        pass_direct<MODE, SRC, false><<<(unsigned)blocks, threads, 0, st>>>(p, a);
    return cudaGetLastError();
}

}  // namespace

LastShape direct_last_shape(const Pass& p, int64_t cc, int64_t tc) {
    DftShape d;
    bool half;
    // a sample takes the time of its n terms and of about 24 for the index; a slice's sums
    // that of 16 to 24, the kernel that adds them that of 150
    const double sample = p.n + 24;
    if (dft_takes(p, cc, tc, &d, &half))
        return {(cc * p.inner + d.lines - 1) / d.lines, std::min(3, (int)(kDftSmem / d.smem)), 24.0 / sample, 150.0 / sample};
    return {(cc * p.L * p.inner + 255) / 256, 6, 16.0 / sample, 150.0 / sample};
}

double direct_line_flops(const Pass& p, const PassArgs& a) {
    DftShape d;
    bool half;
    // tiles: four real multiply-adds per term and bin r give two or four outputs
    if (dft_takes(p, a.full_S ? a.full_S : a.S, a.tc, &d, &half)) return 8.0 * d.rows * d.reps;
    return 8.0 * p.n * p.q_out;
}

cudaError_t launch_direct(const Pass& p, const PassArgs& a, cudaStream_t st) {
    return dispatch_mode(p.mode, [&](auto M) {
        return dispatch_src<decltype(M)::value>(a.src_kind, [&](auto S) {
            return launch_direct_t<decltype(M)::value, decltype(S)::value>(p, a, st);
        });
    });
}

}  // namespace omni
