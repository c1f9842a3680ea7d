#pragma once
// omni_fft_reg.cuh -- register-resident axis transforms (kernel and launch templates).
//
// Register passes: one thread per line, the whole (power-of-two, <= 64) line
// held in registers.  A forward pass reads the n_d measured values of a line
// and produces all L_d = 2 n_d frequencies (zero padding never stored; the
// first radix-2 stage is twiddles only; a beam-space pointing axis, n_d = L_d,
// is transformed whole).  The last forward pass squares the
// modulus and sums over the chunk's samples before folding into FP64.  An
// inverse pass transforms a full line and keeps the 2 n_d - 1 lag bins.
#include "omni_fft_common.cuh"

#include <type_traits>

namespace omni {

// ---------------------------------------------------------------- register passes

// One thread per line; the whole line lives in registers.
template <int L, int MODE, int SRC>
__global__ void __launch_bounds__(256) pass_reg(Pass p, PassArgs a) {
    constexpr bool FWD = (MODE == MODE_MID || MODE == MODE_LAST);
    constexpr int LOG = ilog2(L);
    const int64_t flat = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t inner = p.inner;
    const void* src = a.src;

    if constexpr (MODE == MODE_LAST) {
        // outer == 1: thread per (channel, inner index); loop over the chunk's samples.
        if (flat >= a.S * inner) return;
        const int64_t cc = flat / inner, i = flat - cc * inner;
        float acc[L];
#pragma unroll
        for (int k = 0; k < L; ++k) acc[k] = 0.0f;
        int tb, te;
        slice_samples(a, tb, te);
        for (int tt = tb; tt < te; ++tt) {
            const int64_t s = cc * a.tc + tt;
            const int64_t base = src_base(a, s) + i;
            float2 v[L];
#pragma unroll
            for (int j = 0; j < L; ++j)
                v[j] = (j < L / 2) ? ld_src<SRC>(src, base + (int64_t)j * inner) : make_float2(0.f, 0.f);
            fft_dif<L, true>(v);
#pragma unroll
            for (int k = 0; k < L; ++k) acc[k] += cnorm(v[brev(k, LOG)]);
        }
#pragma unroll
        for (int k = 0; k < L; ++k) fold_last(a, cc, (int64_t)k * inner + i, acc[k]);
        return;
    } else {
        const int64_t lines = p.outer * inner;
        if (flat >= a.S * lines) return;
        const int64_t s = flat / lines;
        const int64_t r = flat - s * lines;
        const int64_t o = r / inner, i = r - o * inner;
        const int64_t base = src_base(a, s) + o * p.n * inner + i;
        // an unpadded forward line (n == L: a beam-space pointing axis) is a full
        // transform; otherwise the upper half is the zero padding
        const bool full = !FWD || p.n == L;
        float2 v[L];
#pragma unroll
        for (int j = 0; j < L; ++j) {
            const bool live = full || j < L / 2;
            v[j] = live ? ld_src<SRC>(src, base + (int64_t)j * inner) : make_float2(0.f, 0.f);
        }
        if (full) fft_dif<L, false>(v);
        else fft_dif<L, true>(v);
        if constexpr (MODE == MODE_MID) {
            float2* d = a.dst + s * a.dst_stride + o * (int64_t)L * inner + i;
#pragma unroll
            for (int k = 0; k < L; ++k) d[(int64_t)k * inner] = v[brev(k, LOG)];
        } else {
            // keep 2 n_d - 1 = L - 1 bins: lags -(L/2-1) .. L/2-1
            constexpr int Q = L - 1;
            constexpr int SH = L / 2 - 1;
            if constexpr (MODE == MODE_INV_MID) {
                float2* d = a.dst + s * a.dst_stride + o * (int64_t)Q * inner + i;
#pragma unroll
                for (int q = 0; q < Q; ++q) d[(int64_t)q * inner] = v[brev((q - SH + L) % L, LOG)];
            } else {
                double2* d = a.V + (a.c0 + s) * a.V_stride + o * (int64_t)Q * inner + i;
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const float2 x = v[brev((q - SH + L) % L, LOG)];
                    d[(int64_t)q * inner] = visibility(x, a);
                }
            }
        }
    }
}

// Lines along the innermost axis (inner == 1), forward MID and inverse passes: thread
// per line as above, but its points are contiguous in memory, so that a thread reading
// and writing its own line touches 32 lines of memory per warp access (2.3 TB/s, 16-byte
// outputs).  The CTA's lines go through shared memory and memory is read and written in
// runs: one 16 x 16 on 8 x 8 hierarchy, 64 channels, last inverse pass: 149 -> 117 us.
template <int L, int MODE, int SRC>
__global__ void __launch_bounds__(128) pass_reg_rows(Pass p, PassArgs a) {
    constexpr bool FWD = MODE == MODE_MID;
    constexpr int LOG = ilog2(L), LINES = 128, PITCH = L + 1;
    constexpr int Q = FWD ? L : L - 1;
    extern __shared__ float2 rows_sm[];  // [LINES][PITCH]
    __shared__ int64_t from[LINES], to[LINES];
    const int64_t l0 = (int64_t)blockIdx.x * LINES, lines = a.S * p.outer;
    const int count = (int)(lines - l0 < LINES ? lines - l0 : LINES);
    const int tid = threadIdx.x;
    if (tid < count) {
        const int64_t s = (l0 + tid) / p.outer, o = (l0 + tid) - s * p.outer;
        from[tid] = src_base(a, s) + o * p.n;
        to[tid] = o * Q + (MODE == MODE_INV_LAST ? (a.c0 + s) * a.V_stride : s * a.dst_stride);
    }
    __syncthreads();
    const int lg = p.n == L ? LOG : LOG - 1;  // inputs per line: L, or L / 2 (the rest is padding)
    constexpr int NB = 8;                     // loads in flight per thread
    for (int e0 = tid; e0 < count << lg; e0 += NB * LINES) {
        float2 x[NB];
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int e = e0 + u * LINES, l = e >> lg, j = e & ((1 << lg) - 1);
            if (l < count) x[u] = ld_src<SRC>(a.src, from[l] + j);
        }
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int e = e0 + u * LINES, l = e >> lg, j = e & ((1 << lg) - 1);
            if (l < count) rows_sm[l * PITCH + j] = x[u];
        }
    }
    __syncthreads();
    float2* row = rows_sm + tid * PITCH;
    if (tid < count) {
        const bool full = !FWD || p.n == L;
        float2 v[L];
#pragma unroll
        for (int j = 0; j < L; ++j) v[j] = full || j < L / 2 ? row[j] : make_float2(0.f, 0.f);
        if (full) fft_dif<L, false>(v);
        else fft_dif<L, true>(v);
        // inverse: slot q holds lag q - (L/2 - 1)
#pragma unroll
        for (int q = 0; q < Q; ++q) row[q] = v[brev(FWD ? q : (q - (L / 2 - 1) + L) % L, LOG)];
    }
    __syncthreads();
#pragma unroll 8
    for (int e = tid; e < count * Q; e += LINES) {
        const int l = e / Q, q = e - l * Q;
        const float2 x = rows_sm[l * PITCH + q];
        if constexpr (MODE == MODE_INV_LAST)
            a.V[to[l] + q] = visibility(x, a);
        else
            a.dst[to[l] + q] = x;
    }
}

template <int L, int MODE, int SRC>
cudaError_t launch_reg_t(const Pass& p, const PassArgs& a, cudaStream_t st) {
    const int64_t work = (MODE == MODE_LAST) ? a.S * p.inner : a.S * p.outer * p.inner;
    if (work <= 0) return cudaSuccess;
    if constexpr (MODE != MODE_LAST) {
        if (p.inner == 1) {
            constexpr size_t smem = sizeof(float2) * 128 * (L + 1);
            auto k = pass_reg_rows<L, MODE, SRC>;
            cudaError_t e = smem_limit_once((const void*)k, smem);
            if (e != cudaSuccess) return e;
            k<<<(unsigned)((work + 127) / 128), 128, smem, st>>>(p, a);
            return cudaGetLastError();
        }
    }
    const int threads = 256;
    const int64_t blocks = (work + threads - 1) / threads;
    pass_reg<L, MODE, SRC><<<MODE == MODE_LAST ? last_grid(blocks, a) : dim3((unsigned)blocks), threads, 0, st>>>(p, a);
    return cudaGetLastError();
}

// Every mode and source of one register-pass length.
template <int L>
cudaError_t launch_reg_len(const Pass& p, const PassArgs& a, cudaStream_t st) {
    return dispatch_mode(p.mode, [&](auto M) {
        return dispatch_src<decltype(M)::value>(a.src_kind, [&](auto S) {
            return launch_reg_t<L, decltype(M)::value, decltype(S)::value>(p, a, st);
        });
    });
}

}  // namespace omni
