#pragma once
// omni_fft_smem.cuh -- four-step shared-memory axis transforms (kernel and launch templates).
//
// Four-step passes for power-of-two axes of 128..4096 points: each line is
// split as L = L1 x L2 and transformed as columns then rows in shared memory.
#include "omni_fft_common.cuh"

#include <type_traits>

namespace omni {

// ---------------------------------------------------------------- four-step passes

// L = L1 * L2 (powers of two, L1 >= L2, both <= 64).  A CTA holds W lines
// (W consecutive inner indices, or, for a non-LAST pass along the innermost axis,
// W consecutive outer lines) in shared memory as [w][j1][j2] (j = j2 + L2 j1,
// i.e. natural order), with odd pitches so that column and row sweeps are
// conflict-free.  Step 1: L1-point FFT down each column j2, times w_L^(j2 k1).
// Step 2: L2-point FFT along each row k1 gives X[k1 + L1 k2].  Lines along the
// innermost axis are read and written as contiguous runs: the threads take the
// points of one line first (j2, or k1, fastest) and the lines second.
// WC: the lines per CTA at compile time (256 / L1, 256 threads; the index splits are
// shifts), or 0 for the fewer lines of a narrow axis.  Each thread's loads are issued
// together, and a LAST pass of WC lines loads the next sample's inputs into registers
// while it transforms the current one.  A batch's 64 x 64 arrays (two
// 128-point axes, 16 channels x 512 samples): divisions by a run-time W and one load at a time, 2.72 +
// 4.07 ms, now 1.94 + 2.03.
template <int L1, int L2, int MODE, int SRC, int WC>
__global__ void __launch_bounds__(256) pass_smem(Pass p, PassArgs a) {
    constexpr bool FWD = (MODE == MODE_MID || MODE == MODE_LAST);
    constexpr int L = L1 * L2;
    constexpr int PITCH = L2 + 1;
    constexpr int PLANE = L1 * PITCH + 1;
    constexpr int LOG1 = ilog2(L1), LOG2 = ilog2(L2);
    constexpr int TWS = kTwiddleN / L;
    extern __shared__ float2 sm[];
    const int W = WC ? WC : p.W;
    const int64_t inner = p.inner;
    constexpr int n = FWD ? L / 2 : L;
    const int NT = WC ? WC * L1 : blockDim.x;
    // lines along the innermost axis: W consecutive outer lines per CTA
    const bool rows = MODE != MODE_LAST && inner == 1;
    const int64_t tiles = rows ? (p.outer + W - 1) / W : (inner + W - 1) / W;

    int64_t b = blockIdx.x;
    const int64_t tile = b % tiles;
    b /= tiles;
    const int64_t i0 = rows ? 0 : tile * W;
    int64_t o = 0, s_first = 0, n_samples = 1, cc = 0;
    if constexpr (MODE == MODE_LAST) {
        cc = b;  // outer == 1
        int tb, te;
        slice_samples(a, tb, te);
        s_first = cc * a.tc + tb;
        n_samples = te - tb;
    } else if (rows) {
        o = tile * W;  // first of the CTA's outer lines
        s_first = b;
    } else {
        o = b % p.outer;
        s_first = b / p.outer;
    }
    auto line_ok = [&](int w) { return rows ? o + w < p.outer : i0 + w < inner; };

    // step-2 ownership (fixed across samples so LAST can keep sums in registers)
    const int u2 = threadIdx.x;
    const int w2 = rows ? u2 / L1 : u2 % W, k1 = rows ? u2 % L1 : u2 / W;
    const bool own2 = u2 < W * L1;
    float acc[L2];
#pragma unroll
    for (int k = 0; k < L2; ++k) acc[k] = 0.0f;

    // inputs per thread of one sample (WC), or the loads in flight at a time
    constexpr int NB = WC ? n / L1 : 8;
    auto at_e = [&](int e, int& j, int& w) {
        j = rows ? e % n : e / W;
        w = rows ? e / n : e % W;
    };
    auto load = [&](float2 (&x)[NB], int64_t base, int e0) {
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            const int e = e0 + r * NT;
            int j, w;
            at_e(e, j, w);
            x[r] = (WC || e < n * W) && line_ok(w)
                       ? ld_src<SRC>(a.src, rows ? base + (int64_t)w * n + j : base + (int64_t)j * inner + w)
                       : make_float2(0.f, 0.f);
        }
    };
    auto store = [&](const float2 (&x)[NB], int e0) {
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            const int e = e0 + r * NT;
            int j, w;
            at_e(e, j, w);
            if (WC || e < n * W) sm[w * PLANE + (j / L2) * PITCH + (j % L2)] = x[r];
        }
    };
    auto base_of = [&](int64_t s) { return src_base(a, s) + o * (int64_t)n * inner + i0; };
    constexpr bool AHEAD = WC > 0 && MODE == MODE_LAST && NB <= 8;
    float2 pre[NB];
    if constexpr (AHEAD)
        if (n_samples > 0) load(pre, base_of(s_first), threadIdx.x);

    for (int64_t ts = 0; ts < n_samples; ++ts) {
        const int64_t s = s_first + ts;
        // n inputs of each of the W lines (coalesced over inner, or along each line)
        if constexpr (AHEAD) {
            store(pre, threadIdx.x);
            if (ts + 1 < n_samples) load(pre, base_of(s + 1), threadIdx.x);  // in flight during this sample
        } else if constexpr (WC > 0) {
            load(pre, base_of(s), threadIdx.x);
            store(pre, threadIdx.x);
        } else {
            for (int e0 = threadIdx.x; e0 < n * W; e0 += NB * NT) {
                load(pre, base_of(s), e0);
                store(pre, e0);
            }
        }
        __syncthreads();
        // step 1: columns
        for (int u = threadIdx.x; u < W * L2; u += NT) {
            const int w = rows ? u / L2 : u % W, j2 = rows ? u % L2 : u / W;
            float2* col = sm + w * PLANE + j2;
            float2 v[L1];
#pragma unroll
            for (int j1 = 0; j1 < L1; ++j1)
                v[j1] = (!FWD || j1 < L1 / 2) ? col[j1 * PITCH] : make_float2(0.f, 0.f);
            fft_dif<L1, FWD>(v);
#pragma unroll
            for (int kk = 0; kk < L1; ++kk) {
                float2 y = v[brev(kk, LOG1)];
                const int e = (j2 * kk) & (L - 1);
                if (e) y = cmul(y, g_tw4096[e * TWS]);
                col[kk * PITCH] = y;
            }
        }
        __syncthreads();
        // step 2: rows
        if (own2) {
            const float2* row = sm + w2 * PLANE + k1 * PITCH;
            float2 v[L2];
#pragma unroll
            for (int j2 = 0; j2 < L2; ++j2) v[j2] = row[j2];
            fft_dif<L2, false>(v);
            const int64_t i = i0 + w2;
            if (line_ok(w2)) {
                // line (outer oo, inner ii) of this thread's outputs
                const int64_t oo = rows ? o + w2 : o, ii = rows ? 0 : i;
                if constexpr (MODE == MODE_LAST) {
#pragma unroll
                    for (int k2 = 0; k2 < L2; ++k2) acc[k2] += cnorm(v[brev(k2, LOG2)]);
                } else if constexpr (MODE == MODE_MID) {
                    float2* d = a.dst + s * a.dst_stride + oo * (int64_t)L * inner + ii;
#pragma unroll
                    for (int k2 = 0; k2 < L2; ++k2) d[(int64_t)(k1 + L1 * k2) * inner] = v[brev(k2, LOG2)];
                } else {
                    constexpr int Q = L - 1, SH = L / 2 - 1;
#pragma unroll
                    for (int k2 = 0; k2 < L2; ++k2) {
                        const int k = k1 + L1 * k2;
                        const int q = (k + SH) % L;  // lag k (k < L/2) or k - L (k > L/2)
                        if (k == L / 2) continue;    // the one padding bin no lag maps to
                        const float2 x = v[brev(k2, LOG2)];
                        if constexpr (MODE == MODE_INV_MID) {
                            a.dst[s * a.dst_stride + (oo * (int64_t)Q + q) * inner + ii] = x;
                        } else {
                            a.V[(a.c0 + s) * a.V_stride + (oo * (int64_t)Q + q) * inner + ii] =
                                visibility(x, a);
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
    if constexpr (MODE == MODE_LAST) {
        const int64_t i = i0 + w2;
        if (own2 && i < inner) {
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) fold_last(a, cc, (int64_t)(k1 + L1 * k2) * inner + i, acc[k2]);
        }
    }
}

// lines per CTA at compile time: the full tile of 256 threads
template <int L1, class F>
cudaError_t with_lines(int W, F&& f) {
    return W == 256 / L1 ? f(std::integral_constant<int, 256 / L1>{}) : f(std::integral_constant<int, 0>{});
}

template <int L1, int L2, int MODE, int SRC>
cudaError_t launch_smem_t(const Pass& p, const PassArgs& a, cudaStream_t st) {
    const bool rows = MODE != MODE_LAST && p.inner == 1;
    const int64_t tiles = rows ? (p.outer + p.W - 1) / p.W : (p.inner + p.W - 1) / p.W;
    const int64_t blocks = (MODE == MODE_LAST) ? a.S * tiles : rows ? a.S * tiles : a.S * p.outer * tiles;
    if (blocks <= 0) return cudaSuccess;
    const int threads = p.W * L1;
    const size_t smem = (size_t)p.W * (L1 * (L2 + 1) + 1) * sizeof(float2);
    return with_lines<L1>(p.W, [&](auto W) {
        auto k = pass_smem<L1, L2, MODE, SRC, decltype(W)::value>;
        cudaError_t e = smem_limit_once((const void*)k, smem);
        if (e != cudaSuccess) return e;
        k<<<MODE == MODE_LAST ? last_grid(blocks, a) : dim3((unsigned)blocks), threads, smem, st>>>(p, a);
        return cudaGetLastError();
    });
}

// Resident CTAs per SM of the LAST-mode kernel of one four-step length.
template <int L1, int L2>
cudaError_t smem_last_occupancy_len(const Pass& p, int src_kind, int* blocks_per_sm) {
    const int threads = p.W * L1;
    const size_t smem = (size_t)p.W * (L1 * (L2 + 1) + 1) * sizeof(float2);
    return dispatch_src<MODE_LAST>(src_kind, [&](auto S) {
        return with_lines<L1>(p.W, [&](auto W) {
            auto k = pass_smem<L1, L2, MODE_LAST, decltype(S)::value, decltype(W)::value>;
            cudaError_t e = smem_limit_once((const void*)k, smem);
            if (e != cudaSuccess) return e;
            return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, threads, smem);
        });
    });
}

// Every mode and source of one four-step length.
template <int L1, int L2>
cudaError_t launch_smem_len(const Pass& p, const PassArgs& a, cudaStream_t st) {
    return dispatch_mode(p.mode, [&](auto M) {
        return dispatch_src<decltype(M)::value>(a.src_kind, [&](auto S) {
            return launch_smem_t<L1, L2, decltype(M)::value, decltype(S)::value>(p, a, st);
        });
    });
}

}  // namespace omni
