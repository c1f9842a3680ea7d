// omni_fft_common.cuh -- device helpers shared by the transform-pass kernels.
//
// Included by each kernel translation unit; the twiddle tables have internal
// linkage, so every unit owns a copy that upload_twiddles() fills.
#pragma once

#include "omni_internal.h"

#include <cmath>
#include <mutex>
#include <utility>
#include <vector>

namespace omni {

// exp(-2 pi i k / 64): every register-FFT twiddle (spans <= 64) is one of these.
static __constant__ float2 c_tw64[64];
// exp(-2 pi i k / 4096): four-step twiddles w_L^(j2 k1) for L <= 4096.
static __device__ float2 g_tw4096[kTwiddleN];

// Fill this unit's tables on the current device (values from double-precision
// cos/sin, rounded once to float).
[[maybe_unused]] static cudaError_t upload_twiddles() {
    const double two_pi = 6.283185307179586476925286766559;
    std::vector<float2> t64(64), t4096(kTwiddleN);
    for (int k = 0; k < 64; ++k) {
        const double ang = two_pi * k / 64.0;
        t64[k] = make_float2((float)std::cos(ang), (float)-std::sin(ang));
    }
    for (int k = 0; k < kTwiddleN; ++k) {
        const double ang = two_pi * k / (double)kTwiddleN;
        t4096[k] = make_float2((float)std::cos(ang), (float)-std::sin(ang));
    }
    cudaError_t e = cudaMemcpyToSymbol(c_tw64, t64.data(), sizeof(float2) * 64);
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(g_tw4096, t4096.data(), sizeof(float2) * kTwiddleN);
}

// Raise a kernel's dynamic shared-memory limit once per (kernel, device, size):
// later launches (including ones recorded into a CUDA graph) make no attribute call.
inline cudaError_t smem_limit_once(const void* kernel, size_t bytes) {
    static std::mutex mu;
    static std::vector<std::pair<std::pair<const void*, int>, size_t>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    for (auto& d : done)
        if (d.first.first == kernel && d.first.second == dev && d.second >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done.push_back({{kernel, dev}, bytes});
    return e;
}

// ---------------------------------------------------------------- complex helpers

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float cnorm(float2 a) { return fmaf(a.x, a.x, a.y * a.y); }

__host__ __device__ constexpr int ilog2(int x) { return x <= 1 ? 0 : 1 + ilog2(x >> 1); }
__host__ __device__ constexpr int brev(int k, int bits) {
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((k >> b) & 1) << (bits - 1 - b);
    return r;
}

// a * exp(-2 pi i j / M) for 0 <= j < M/2, M <= 64; j and M are compile-time
// constants once the callers are unrolled, so the special angles cost no
// multiplies.
__device__ __forceinline__ float2 twiddle(float2 a, int j, int M) {
    const float h = 0.70710678118654752440f;
    if (j == 0) return a;
    if (4 * j == M) return make_float2(a.y, -a.x);
    if (8 * j == M) return make_float2((a.x + a.y) * h, (a.y - a.x) * h);
    if (8 * j == 3 * M) return make_float2((a.y - a.x) * h, -(a.x + a.y) * h);
    return cmul(a, c_tw64[j * (64 / M)]);
}

// In-place radix-2 decimation-in-frequency DFT of L (power of two <= 64)
// points held in registers: natural-order input, bit-reversed output
// (X[k] = v[brev(k)]).  PRUNED: inputs n >= L/2 are zero, so the first stage
// is twiddles only.
template <int L, bool PRUNED>
__device__ __forceinline__ void fft_dif(float2 (&v)[L]) {
    constexpr int LOG = ilog2(L);
#pragma unroll
    for (int st = 0; st < LOG; ++st) {
        const int half = L >> (st + 1);
#pragma unroll
        for (int base = 0; base < L; base += 2 * half) {
#pragma unroll
            for (int j = 0; j < half; ++j) {
                const float2 a = v[base + j];
                if (PRUNED && st == 0) {
                    v[base + j + half] = twiddle(a, j, 2 * half);
                } else {
                    const float2 b = v[base + j + half];
                    v[base + j] = cadd(a, b);
                    v[base + j + half] = twiddle(csub(a, b), j, 2 * half);
                }
            }
        }
    }
}

// ---------------------------------------------------------------- two lanes per instruction

// Two independent FP32 values per register pair (add/mul/fma.rn.f32x2).  A lane
// rounds as the scalar instruction does; the lane rate is the same (butterflies 37.5
// against 33.9 T operations/s in registers, products by constants 37.6 against 37.2),
// at half the issue slots.  Products with three fresh operands gain nothing (21.8
// against 25.3: register ports).
struct f2x {
    unsigned long long v;
};
__device__ __forceinline__ f2x pack2(float a, float b) {
    f2x r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f2x p) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(p.v));
    return r;
}
__device__ __forceinline__ f2x add2(f2x a, f2x b) {
    f2x r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2x sub2(f2x a, f2x b) {
    f2x r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2x mul2(f2x a, f2x b) {
    f2x r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2x fma2(f2x a, f2x b, f2x c) {
    f2x r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ f2x dup2(float c) { return pack2(c, c); }

// cos(2 pi k / 64), folded to a literal
constexpr float cos64(int k) {
    k &= 63;
    if (k > 32) k = 64 - k;
    if (k > 16) return -cos64(32 - k);
    switch (k) {
        case 0: return 1.0f;
        case 1: return 0.99518472667219688624f;
        case 2: return 0.98078528040323044913f;
        case 3: return 0.95694033573220886494f;
        case 4: return 0.92387953251128675613f;
        case 5: return 0.88192126434835502971f;
        case 6: return 0.83146961230254523708f;
        case 7: return 0.77301045336273696081f;
        case 8: return 0.70710678118654752440f;
        case 9: return 0.63439328416364549822f;
        case 10: return 0.55557023301960222474f;
        case 11: return 0.47139673682599764856f;
        case 12: return 0.38268343236508977173f;
        case 13: return 0.29028467725446236764f;
        case 14: return 0.19509032201612826785f;
        case 15: return 0.09801714032956060199f;
        default: return 0.0f;
    }
}
// ... twice, in constant memory: as literals the pairs were held in registers (24 of them
// in a 16-point transform)
#define OMNI_DUP(k) {cos64(k), cos64(k)}
#define OMNI_DUP8(k) \
    OMNI_DUP(k), OMNI_DUP(k + 1), OMNI_DUP(k + 2), OMNI_DUP(k + 3), OMNI_DUP(k + 4), OMNI_DUP(k + 5), OMNI_DUP(k + 6), \
        OMNI_DUP(k + 7)
static __constant__ float2 c_dup64[64] = {OMNI_DUP8(0),  OMNI_DUP8(8),  OMNI_DUP8(16), OMNI_DUP8(24),
                                          OMNI_DUP8(32), OMNI_DUP8(40), OMNI_DUP8(48), OMNI_DUP8(56)};
#undef OMNI_DUP8
#undef OMNI_DUP
__device__ __forceinline__ f2x dup_cos(int k) {
    f2x r;
    r.v = *reinterpret_cast<const unsigned long long*>(&c_dup64[k & 63]);
    return r;
}

// Two complex values times exp(-2 pi i j / M), 0 <= j < M / 2 compile-time.
__device__ __forceinline__ void twiddle2(f2x& x, f2x& y, int j, int M) {
    const int k = j * (64 / M);  // w = cos64(k) - i cos64(16 - k)
    if (j == 0) return;
    if (4 * j == M) {
        const f2x t = x;
        x = y;
        y = sub2(dup2(0.f), t);
    } else if (8 * j == M) {
        const f2x s = add2(x, y), d = sub2(y, x);
        x = mul2(s, dup_cos(8));
        y = mul2(d, dup_cos(8));
    } else if (8 * j == 3 * M) {
        const f2x s = add2(x, y), d = sub2(y, x);
        x = mul2(d, dup_cos(8));
        y = mul2(s, dup_cos(24));
    } else {
        const f2x t = x;
        x = fma2(t, dup_cos(k), mul2(y, dup_cos(16 - k)));
        y = fma2(y, dup_cos(k), mul2(t, dup_cos(48 - k)));
    }
}

// fft_dif on two lines at once, real and imaginary parts apart.
template <int L, bool PRUNED>
__device__ __forceinline__ void fft_dif2(f2x (&x)[L], f2x (&y)[L]) {
    constexpr int LOG = ilog2(L);
#pragma unroll
    for (int st = 0; st < LOG; ++st) {
        const int half = L >> (st + 1);
#pragma unroll
        for (int base = 0; base < L; base += 2 * half) {
#pragma unroll
            for (int j = 0; j < half; ++j) {
                const int p = base + j, q = p + half;
                if (PRUNED && st == 0) {
                    x[q] = x[p];
                    y[q] = y[p];
                    twiddle2(x[q], y[q], j, 2 * half);
                } else {
                    const f2x ax = x[p], ay = y[p], bx = x[q], by = y[q];
                    x[p] = add2(ax, bx);
                    y[p] = add2(ay, by);
                    if (2 * j == half) {  // times -i: the parts swap, one difference reversed
                        x[q] = sub2(ay, by);
                        y[q] = sub2(bx, ax);
                    } else {
                        x[q] = sub2(ax, bx);
                        y[q] = sub2(ay, by);
                        twiddle2(x[q], y[q], j, 2 * half);
                    }
                }
            }
        }
    }
}

// ---------------------------------------------------------------- sources

// Offset of sample s's first element in the source, in source elements.
// (Kept to one comparison per branch: a second one here raised the tensor-core
// stage-A kernel from 80 to 82 registers, past an allocation step, and cost 9%
// of the mixed path's step time through lost co-residency.)
__device__ __forceinline__ int64_t src_base(const PassArgs& a, int64_t s) {
    if (a.src_kind == SRC_CF32 || a.src_kind == SRC_CI8)
        return ((a.vc0 + s / a.tc) * a.T + a.t0 + s % a.tc) * a.N;
    if (a.src_kind >= SRC_P64) return (a.c0 + s) * a.src_stride;  // P64, PC64: per channel
    return s * a.src_stride;
}

template <int SRC>
__device__ __forceinline__ float2 ld_src(const void* p, int64_t e) {
    if constexpr (SRC == SRC_BUF || SRC == SRC_CF32) {
        return __ldg(reinterpret_cast<const float2*>(p) + e);
    } else if constexpr (SRC == SRC_CI8) {
        const char2 c = reinterpret_cast<const char2*>(p)[e];
        return make_float2((float)c.x, (float)c.y);
    } else if constexpr (SRC == SRC_PC64) {
        // conjugated on load: the inverse passes run forward (e^-) transforms and
        // conjugate at the end, IFFT(S) = conj(FFT(conj(S))) / L; a real |F|^2
        // needs no input conjugate, a complex cross-spectrum does
        const double2 d = __ldg(reinterpret_cast<const double2*>(p) + e);
        return make_float2((float)d.x, -(float)d.y);
    } else {
        return make_float2((float)__ldg(reinterpret_cast<const double*>(p) + e), 0.0f);
    }
}

// INV_LAST: the visibility (x.x scale, -x.y scale) in FP64.  With scale = 2^-k the bits of
// a normal FP32 number are moved into place: the FP64 pipe (conversions and products, 2
// lanes a clock) bound the last inverse pass (262144 antennas, 8 channels, 54 M
// visibilities: 0.64 -> 0.58 ms; 64 x 64 tile pairs, 0.32 -> 0.23).
__device__ __forceinline__ double scaled_double(float x, double scale, int shift) {
    const uint32_t b = __float_as_uint(x);
    if (shift > 0 && ((b >> 23) & 255u) - 1u < 254u)
        return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + ((uint32_t)(896 - shift) << 20))),
                                (int)(b << 29));
    return (double)x * scale;
}
__device__ __forceinline__ double2 visibility(float2 x, const PassArgs& a) {
    return make_double2(scaled_double(x.x, a.scale, a.scale_shift), scaled_double(-x.y, a.scale, a.scale_shift));
}

// LAST passes: grid row y takes slice y of the chunk's samples ([tb, te)) and, when
// there are several, leaves its sums in its own part for launch_fold_parts.
__device__ __forceinline__ void slice_samples(const PassArgs& a, int& tb, int& te) {
    tb = (int)((int64_t)a.tc * blockIdx.y / gridDim.y);
    te = (int)((int64_t)a.tc * (blockIdx.y + 1) / gridDim.y);
}
__device__ __forceinline__ void fold_last(const PassArgs& a, int64_t cc, int64_t e, float v, double fs = 1.0) {
    if (gridDim.y > 1)
        a.part[((int64_t)blockIdx.y * a.S + cc) * a.P_stride + e] = v;
    else
        a.P[(a.c0 + cc) * a.P_stride + e] += fs * (double)v;
}
inline dim3 last_grid(int64_t blocks, const PassArgs& a) { return dim3((unsigned)blocks, a.split > 1 ? (unsigned)a.split : 1u); }

// Inverse passes: output slot q of a line holds lag q - q_shift, which is FFT
// bin (q - q_shift) mod L.
__device__ __forceinline__ int inv_bin(int q, int q_shift, int L) {
    int k = q - q_shift;
    return k < 0 ? k + L : k;
}

// Source kinds a pass mode can read: forward passes read the caller's
// voltages or the scratch buffer, inverse passes the FP64 accumulator (real
// |F|^2, or complex cross-spectra of the tile hybrid) or the scratch buffer.
template <int MODE, class F>
cudaError_t dispatch_src(int src_kind, F&& f) {
    if constexpr (MODE == MODE_MID || MODE == MODE_LAST) {
        switch (src_kind) {
            case SRC_BUF: return f(std::integral_constant<int, SRC_BUF>{});
            case SRC_CF32: return f(std::integral_constant<int, SRC_CF32>{});
            case SRC_CI8: return f(std::integral_constant<int, SRC_CI8>{});
            default: return cudaErrorInvalidValue;
        }
    } else {
        switch (src_kind) {
            case SRC_BUF: return f(std::integral_constant<int, SRC_BUF>{});
            case SRC_P64: return f(std::integral_constant<int, SRC_P64>{});
            case SRC_PC64: return f(std::integral_constant<int, SRC_PC64>{});
            default: return cudaErrorInvalidValue;
        }
    }
}

template <class F>
cudaError_t dispatch_mode(int mode, F&& f) {
    switch (mode) {
        case MODE_MID: return f(std::integral_constant<int, MODE_MID>{});
        case MODE_LAST: return f(std::integral_constant<int, MODE_LAST>{});
        case MODE_INV_MID: return f(std::integral_constant<int, MODE_INV_MID>{});
        default: return f(std::integral_constant<int, MODE_INV_LAST>{});
    }
}

}  // namespace omni
