// omni_fengine.cu -- F-engine (Appendix A, step 2): each antenna's samples are
// Fourier transformed in time into frequency channels and calibrated, and the
// channel voltages are written in the correlator's input layout [F][T][N].
//
// Frame t of antenna a (frame length 2F, P taps):
//   u_t(n) = sum_p w(p 2F + n) r_a((t + p) 2F + n)         (polyphase sum)
//   X_t(f) = sum_n u_t(n) exp(-2 pi i f n / 2F), f < F     (real FFT, Nyquist dropped)
//   y_t(f) = scale g(f, a) X_t(f)                          (calibration)
// The real frame is packed as F complex points z(m) = u(2m) + i u(2m+1), run
// through an F-point FFT and unpacked to the real spectrum, in one pass over the
// samples: fengine64 (F = 64 and 16-byte sample rows), fengine_multi (other F >= 16),
// fengine_fused (F < 16, and few samples of up to 256 channels).  int8 outputs round half to even and clip to +-127.
#include "omni_fft_common.cuh"
#include "omni.h"

#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

namespace omni {
namespace {

constexpr int kFThreads = 256;

// y = scale * g * X with no contraction, so that the float and the int8 output
// modes compute the same float (the quantiser decides on exactly that value)
__device__ __forceinline__ float2 calibrate(float2 x, float2 g, float scale) {
    const float yr = __fsub_rn(__fmul_rn(g.x, x.x), __fmul_rn(g.y, x.y));
    const float yi = __fadd_rn(__fmul_rn(g.x, x.y), __fmul_rn(g.y, x.x));
    return make_float2(__fmul_rn(scale, yr), __fmul_rn(scale, yi));
}

__device__ __forceinline__ int8_t quantize8(float v) {
    const int q = __float2int_rn(v);  // round half to even
    return (int8_t)max(-127, min(127, q));
}

// e^{-2 pi i j / 8192}, j < 4096, built on the host in double: every twiddle of
// an F-point stage (e^{-i pi pos / half} = entry pos * 4096 / half) and of the
// real-spectrum unpacking (e^{-i pi f / F} = entry f * 4096 / F) for F <= 256.
__device__ float2 g_fetw[4096];

constexpr int kFuseAnt = 16;     // antennas per CTA: 32-byte int8 output rows
constexpr int kFusePoints = 4096;  // complex points in shared memory (32 KB)
static_assert(kFuseAnt == 16 && kFusePoints / kFuseAnt == 256, "fused index shifts assume 16 x 256 points");

// Fused F-engine for small F or few samples: CTA = (16 consecutive antennas, FR frames),
// FR = 256 / F; polyphase, FFT, unpacking, calibration and quantisation in
// shared memory, each output row (channel f, frame t) written as the 16
// antennas' values together, so no intermediate spectrum goes through HBM.
template <bool I8, bool VEC>
__global__ void __launch_bounds__(kFThreads) fengine_fused(const int8_t* __restrict__ raw, int64_t N,
                                                           int64_t S, int F, int logF, int P,
                                                           const float* __restrict__ w, int64_t T,
                                                           const float2* __restrict__ gains, float scale,
                                                           void* __restrict__ out) {
    // [antenna][frame][F]: each antenna's 256 points padded to 257 so that the
    // 16 antennas of an output row fall in different banks
    constexpr int kPad = kFusePoints / kFuseAnt + 1;
    __shared__ float2 z[kFuseAnt * kPad];
    // this F's twiddles, from the table into shared memory once per CTA:
    // stw[m] = e^{-2 pi i m / F} (m < F/2, the butterflies), utw[f] = e^{-i pi f / F}
    __shared__ float2 stw[128], utw[256];
    for (int j = threadIdx.x; j < F; j += kFThreads) {
        if (j < F / 2) stw[j] = g_fetw[j << (13 - logF)];
        utw[j] = g_fetw[j << (12 - logF)];
    }
    // per antenna: FR frames x F points = 256 points; all index splits below
    // are shifts and masks (F is a power of two)
    constexpr int per = kFusePoints / kFuseAnt, logPer = 8, n = kFusePoints;
    const int FR = per >> logF;
    const int64_t tchunks = (T + FR - 1) / FR;
    const int64_t a0 = (blockIdx.x / tchunks) * kFuseAnt;
    const int64_t t0 = (blockIdx.x % tchunks) * FR;
    const int64_t M = 2 * (int64_t)F;
    // polyphase sums, packed (even, odd), bit-reversed within each frame.
    // VEC (rows 16-byte aligned, F >= 8): a thread takes 8 packed points, one
    // 16-byte load of samples and four of window weights per tap
    if (VEC) {
        for (int idx = threadIdx.x; idx < n / 8; idx += kFThreads) {
            const int al = idx >> (logPer - 3), rem = idx & (per / 8 - 1), fr = rem >> (logF - 3);
            const int m0 = 8 * (rem & ((F >> 3) - 1));
            const int64_t a = a0 + al, t = t0 + fr;
            float ue[8], uo[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) ue[k] = uo[k] = 0.f;
            if (a < N && t < T) {
                const int8_t* ra = raw + a * S;
                for (int p = 0; p < P; ++p) {
                    const int4 rv = __ldg(reinterpret_cast<const int4*>(ra + (t + p) * M + 2 * m0));
                    const int8_t* r = reinterpret_cast<const int8_t*>(&rv);
                    float wv[16];
                    if (w) {
                        const float4* w4 = reinterpret_cast<const float4*>(w + p * M + 2 * m0);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float4 x = __ldg(w4 + q);
                            wv[4 * q] = x.x;
                            wv[4 * q + 1] = x.y;
                            wv[4 * q + 2] = x.z;
                            wv[4 * q + 3] = x.w;
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < 16; ++q) wv[q] = 1.f;
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        ue[k] = fmaf(wv[2 * k], (float)r[2 * k], ue[k]);
                        uo[k] = fmaf(wv[2 * k + 1], (float)r[2 * k + 1], uo[k]);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                z[al * kPad + fr * F + (int)(__brev((unsigned)(m0 + k)) >> (32 - logF))] = make_float2(ue[k], uo[k]);
        }
    } else
    for (int idx = threadIdx.x; idx < n; idx += kFThreads) {
        const int al = idx >> logPer, rem = idx & (per - 1), fr = rem >> logF, m = rem & (F - 1);
        const int64_t a = a0 + al, t = t0 + fr;
        float ue = 0.f, uo = 0.f;
        if (a < N && t < T) {
            const int8_t* ra = raw + a * S;
            for (int p = 0; p < P; ++p) {
                const int8_t* r = ra + (t + p) * M + 2 * m;
                const float we = w ? __ldg(w + p * M + 2 * m) : 1.f;
                const float wo = w ? __ldg(w + p * M + 2 * m + 1) : 1.f;
                ue = fmaf(we, (float)r[0], ue);
                uo = fmaf(wo, (float)r[1], uo);
            }
        }
        z[al * kPad + fr * F + (int)(__brev((unsigned)m) >> (32 - logF))] = make_float2(ue, uo);
    }
    __syncthreads();
    for (int half = 1, lh = 0; half < F; half <<= 1, ++lh) {
        for (int jt = threadIdx.x; jt < n / 2; jt += kFThreads) {
            const int tr = jt >> (logF - 1), j = jt & (F / 2 - 1);  // transform = (antenna, frame)
            const int pos = j & (half - 1);
            const int base = (tr >> (logPer - logF)) * kPad + (tr & (FR - 1)) * F;
            const int i0 = base + ((j - pos) << 1) + pos, i1 = i0 + half;
            const float2 b = cmul(z[i1], stw[pos << (logF - 1 - lh)]);
            const float2 x0 = z[i0];
            z[i0] = cadd(x0, b);
            z[i1] = csub(x0, b);
        }
        __syncthreads();
    }
    // unpack, calibrate, quantise; thread index: antenna fastest so that each
    // (f, t) row of 16 antennas is one contiguous store
    for (int idx = threadIdx.x; idx < n; idx += kFThreads) {
        const int al = idx & (kFuseAnt - 1), rest = idx >> 4, fr = rest >> logF, f = rest & (F - 1);
        const int64_t a = a0 + al, t = t0 + fr;
        if (a >= N || t >= T) continue;
        const float2* zz = z + al * kPad + fr * F;
        const float2 zf = zz[f], zc = zz[(F - f) & (F - 1)];
        const float2 e = make_float2(0.5f * (zf.x + zc.x), 0.5f * (zf.y - zc.y));
        const float2 o = make_float2(0.5f * (zf.y + zc.y), -0.5f * (zf.x - zc.x));
        const float2 x = cadd(e, cmul(o, utw[f]));
        const float2 g = gains ? __ldg(gains + (int64_t)f * N + a) : make_float2(1.f, 0.f);
        const float2 y = calibrate(x, g, scale);
        const int64_t oi = ((int64_t)f * T + t) * N + a;
        if (I8) reinterpret_cast<char2*>(out)[oi] = make_char2(quantize8(y.x), quantize8(y.y));
        else reinterpret_cast<float2*>(out)[oi] = y;
    }
}

// F = 64 (128-sample frames): eight lanes per (antenna, frame) transform, the
// 64-point FFT as 8 x 8 in registers (m = l + 8 q on lane l, k = k_a + 8 k_b):
//   step 1: lane l: 8-point DFT over q, times w_64^(l k_a)
//   step 2: lane k_a: 8-point DFT over l (the 8 x 8 transpose through a per-warp
//           shared buffer, warp-synchronous: no CTA barrier inside a transform)
// then Z(64 - f) from the partner lane by shuffles, the real-spectrum unpacking and
// calibration.  CTA = 32 consecutive antennas (a warp: 4 of them) x kF64Frames frames.
//
// What bounds it is instruction issue and shared memory (its HBM floor on the shape
// below is 0.63 ms).  Two frames at a time, so that each window weight and each
// converted sample serves both (the frame of tap p + 1 of the first is the frame of tap
// p of the second) and the next pair's first frames are on their way during the transforms;
// the step-1 twiddles sit in registers (as constant-memory reads with a different index
// per lane they serialised the warp, with the 4-way conflicts of the window reads 96%
// of the L1 pipe).  int8 codes are staged so that each (channel, frame) row of 32
// antennas is one 64-byte store; floats go out from the registers (4 antennas = one
// 32-byte sector).  Buffer index of point m: 9 (m / 8) + m % 8 and a transform pitch of
// 72: the half-warps of every step touch 16 different bank pairs.
// 16384 antennas, 4 taps, 1024 frames, int8 out: 6.33 -> 3.59 ms.
// PART (up to 28 antennas): warps without an antenna only meet the barriers (8 antennas, 1
// tap, 2048 frames: 23 -> 12 us; in every group the test costs the large case 6%).
constexpr int kF64Ant = 32;
constexpr int kF64Frames = 16;  // most frames per CTA; fewer (even) while the GPU is not filled
constexpr int kF64MaxTaps = 8;
constexpr int kF64Row = 36;  // char2 per staged row (72 bytes: conflict-free 2-byte stores and 8-byte loads)

template <bool I8, bool GAINS, bool PART>
__global__ void __launch_bounds__(256, 2) fengine64(const int8_t* __restrict__ raw, int64_t N, int64_t S, int P,
                                                    const float* __restrict__ w, int64_t T,
                                                    const float2* __restrict__ gains, float scale,
                                                    void* __restrict__ out, int frames) {
    __shared__ float2 zs[8][4 * 72];                                 // per warp: 4 transforms
    __shared__ __align__(16) char2 yq[2][2][I8 ? 64 : 1][kF64Row];   // [pair parity][frame][channel][antenna]
    __shared__ __align__(16) float wsm[kF64MaxTaps * 128];           // [tap][quarter][lane][4]: w(16 lane + 4 quarter ..)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tr = lane >> 3, l = lane & 7;
    for (int i = tid; i < P * 128; i += 256)
        wsm[i] = w ? w[(i & ~127) + ((i >> 2) & 7) * 16 + ((i >> 5) & 3) * 4 + (i & 3)] : 1.f;
    const int64_t tchunks = (T + frames - 1) / frames;
    const int64_t a0 = (blockIdx.x / tchunks) * kF64Ant, t0 = (blockIdx.x % tchunks) * frames;
    const int al = 4 * warp + tr;  // antenna within the CTA
    const int64_t a = a0 + al;
    const int64_t last = a < N ? T + P - 1 : 0;  // frames of this antenna that exist
    const bool idle = PART && a0 + 4 * warp >= N;  // none of this warp's antennas exists
    float2* buf = zs[warp] + 72 * tr;
    // step-1 twiddles, unpacking twiddles e^{-i pi f / 64} and the gains of this lane's f = l + 8 k_b
    float2 t1[8], ut[8], gl[GAINS ? 8 : 1];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        t1[k] = c_tw64[(l * k) & 63];
        ut[k] = g_fetw[(l + 8 * k) * 64];
        if (GAINS) gl[k] = a < N ? __ldg(gains + (int64_t)(l + 8 * k) * N + a) : make_float2(1.f, 0.f);
    }
    __syncthreads();
    const int8_t* ra = raw + a * S + 16 * l;
    auto fetch = [&](int64_t frame) -> uint4 {
        if (frame >= last) return make_uint4(0, 0, 0, 0);
        return __ldg(reinterpret_cast<const uint4*>(ra + frame * 128));
    };
    auto widen = [](uint4 v, float (&d)[16]) {
        const uint32_t q[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int b = 0; b < 16; ++b) d[b] = (float)(int8_t)(q[b >> 2] >> (8 * (b & 3)));
    };
    uint4 f0 = fetch(t0), f1 = fetch(t0 + 1);
    for (int64_t t = t0; t < t0 + frames && t < T; t += 2) {
        // polyphase sums of samples 16 l .. 16 l + 15 of frames t and t + 1:
        // z(8 l + q) = u(16 l + 2q) + i u(16 l + 2q + 1)
        float u0[16], u1[16];
        if (!idle) {
            float x0[16], x1[16];
#pragma unroll
            for (int b = 0; b < 16; ++b) u0[b] = u1[b] = 0.f;
            uint4 n0 = P > 1 ? fetch(t + 2) : f0, n1 = P > 2 ? fetch(t + 3) : f0;
            widen(f0, x0);
            widen(f1, x1);
            auto tap = [&](int p, float (&xa)[16], float (&xb)[16], uint4& next) {  // then xa takes frame t + p + 2
                const float4* w4 = reinterpret_cast<const float4*>(wsm + p * 128 + 4 * l);
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const float4 ww = w4[8 * h];
                    u0[4 * h] = fmaf(ww.x, xa[4 * h], u0[4 * h]);
                    u0[4 * h + 1] = fmaf(ww.y, xa[4 * h + 1], u0[4 * h + 1]);
                    u0[4 * h + 2] = fmaf(ww.z, xa[4 * h + 2], u0[4 * h + 2]);
                    u0[4 * h + 3] = fmaf(ww.w, xa[4 * h + 3], u0[4 * h + 3]);
                    u1[4 * h] = fmaf(ww.x, xb[4 * h], u1[4 * h]);
                    u1[4 * h + 1] = fmaf(ww.y, xb[4 * h + 1], u1[4 * h + 1]);
                    u1[4 * h + 2] = fmaf(ww.z, xb[4 * h + 2], u1[4 * h + 2]);
                    u1[4 * h + 3] = fmaf(ww.w, xb[4 * h + 3], u1[4 * h + 3]);
                }
                if (p + 1 < P) {
                    widen(next, xa);
                    if (p + 3 < P) next = fetch(t + p + 4);
                }
            };
            for (int p = 0; p < P; p += 2) {
                tap(p, x0, x1, n0);
                if (p + 1 < P) tap(p + 1, x1, x0, n1);
            }
            f0 = fetch(t + 2);
            f1 = fetch(t + 3);
        }
        const int par = (int)((t - t0) >> 1) & 1;
        auto transform = [&](const float (&u)[16], int fr) {
#pragma unroll
            for (int q = 0; q < 8; ++q) buf[9 * l + q] = make_float2(u[2 * q], u[2 * q + 1]);  // point m = 8 l + q
            __syncwarp();
            // step 1: lane l holds z(l + 8 q), q < 8 (buffer index 9 q + l)
            float2 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = buf[9 * q + l];
            fft_dif<8, false>(v);
            __syncwarp();
#pragma unroll
            for (int ka = 0; ka < 8; ++ka) {
                float2 y = v[brev(ka, 3)];
                if (ka) y = cmul(y, t1[ka]);
                buf[9 * ka + l] = y;  // Y[l][k_a]
            }
            __syncwarp();
            // step 2: lane k_a = l holds Y[0..7][k_a] -> Z(k_a + 8 k_b) = v[brev(k_b)]
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = buf[9 * l + j];
            fft_dif<8, false>(v);
            __syncwarp();
            // Z(64 - f) for f = k_a + 8 k_b lives on lane (8 - k_a) mod 8 of this transform
            float2 zp[8];
            const int src = (lane & ~7) | ((8 - l) & 7);
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float2 mine = v[brev(r, 3)];
                zp[r] = make_float2(__shfl_sync(0xffffffffu, mine.x, src), __shfl_sync(0xffffffffu, mine.y, src));
            }
#pragma unroll
            for (int kb = 0; kb < 8; ++kb) {
                const int f = l + 8 * kb;
                const float2 zf = v[brev(kb, 3)];
                // 64 - f = (8 - l) + 8 (7 - k_b) for l > 0, 8 (8 - k_b) for l = 0
                const float2 zc = l ? zp[(7 - kb) & 7] : zp[(8 - kb) & 7];
                const float2 e = make_float2(0.5f * (zf.x + zc.x), 0.5f * (zf.y - zc.y));
                const float2 o = make_float2(0.5f * (zf.y + zc.y), -0.5f * (zf.x - zc.x));
                const float2 x = cadd(e, cmul(o, ut[kb]));
                // gain 1: g x with one rounding less to do, the same value (0 x is exact)
                const float2 y = GAINS ? calibrate(x, gl[kb], scale)
                                       : make_float2(__fmul_rn(scale, __fmaf_rn(-0.f, x.y, x.x)),
                                                     __fmul_rn(scale, __fmaf_rn(0.f, x.x, x.y)));
                if (I8) {
                    yq[par][fr][f][al] = make_char2(quantize8(y.x), quantize8(y.y));
                } else if (a < N && t + fr < T) {
                    reinterpret_cast<float2*>(out)[((int64_t)f * T + t + fr) * N + a] = y;
                }
            }
        };
        if (!idle) {
            transform(u0, 0);
            transform(u1, 1);
        }
        if (I8) {
            // rows (channel f, frame t + fr) of the CTA's 32 antennas, 16 (32 bytes) per thread;
            // the other parity's rows are written next, so one barrier per pair is enough
            __syncthreads();
            const int fr = tid >> 7, f = (tid >> 1) & 63, h = 16 * (tid & 1);
            if (t + fr < T && a0 + h < N) {
                uint2 c[4];
                const uint2* q = reinterpret_cast<const uint2*>(&yq[par][fr][f][h]);
#pragma unroll
                for (int i = 0; i < 4; ++i) c[i] = q[i];
                char2* o = reinterpret_cast<char2*>(out) + ((int64_t)f * T + t + fr) * N + a0 + h;
#pragma unroll
                for (int g = 0; g < 16; g += 8) {
                    if (a0 + h + g + 8 <= N && ((uintptr_t)(o + g) % 16) == 0) {
                        const uint2 u = c[g / 4], v = c[g / 4 + 1];
                        *reinterpret_cast<uint4*>(o + g) = make_uint4(u.x, u.y, v.x, v.y);
                    } else {
                        for (int k = g; k < g + 8 && a0 + h + k < N; ++k) o[k] = yq[par][fr][f][h + k];
                    }
                }
            }
        }
    }
}

// Radix-2 decimation-in-time stages over R points whose index runs in steps of `h`
// elements from `pos`: stage t joins halves of h 2^t elements with
// e^{-i pi (pos + q h) / (h 2^t)}.  The table holds e^{-i pi j / F} at tw_at(j): the
// lanes of a step read it at strides of 16 to 128 entries, which the pads spread over
// the banks.
__device__ __forceinline__ int tw_at(int j) { return j + (j >> 4) + (j >> 7); }
template <int R, int F, bool FIRST = false>
__device__ __forceinline__ void dit(float2 (&v)[R], const float2* tw, int pos, int h) {
#pragma unroll
    for (int half = 1; half < R; half <<= 1)
#pragma unroll
        for (int q = 0; q < half; ++q) {
            const bool one = FIRST && q == 0;  // pos = 0: e^0
            const float2 w = one ? make_float2(1.f, 0.f) : tw[tw_at((pos + q * h) * (F / (h * half)))];
#pragma unroll
            for (int b = q; b < R; b += 2 * half) {
                const float2 x = v[b], y = one ? v[b + half] : cmul(v[b + half], w);
                v[b] = cadd(x, y);
                v[b + half] = csub(x, y);
            }
        }
}

// F >= 16: CTA = A antennas, R frames at a time.
//
// What bounds it is instruction issue and shared memory, not HBM, so: the polyphase sums
// of AT antennas and R frames share each window weight, and those of R frames each
// converted sample (frame t + r of tap p is frame t of tap p + r);
// the transform is three (two up to 256 points) register steps of R1 x R2 x R3 points
// instead of log2 F passes through shared memory; the last step takes columns k and
// R1 R2 - k together, so that f and F - f meet in one thread's registers and the
// unpacked spectrum goes straight to global memory, antennas fastest.
// Point m = j1 (F / R1) + j2 R3 + j3 lies at j1 P1 + j2 P2 + j3 of its transform's
// plane; P1 = 8 (mod 16), P2 odd and the plane's pitch keep every step's half-warps
// on different bank pairs.
// 1000 antennas, 1024 channels, 8 taps, 200 frames, float out: 6.49 (radix-2 passes in shared
// memory, spectra through a scratch buffer) -> 1.94 ms; 2.36 with four frames and one antenna
// per thread, two antennas per CTA, and a table without pads.
// (256 and 4096 channels spill 72 and 88 bytes at the 128 registers of two CTAs per SM.)
template <int LOGF, bool FEW>
struct MGeom {
    static constexpr int F = 1 << LOGF;
    static constexpr int R1 = LOGF <= 5 ? 4 : LOGF == 6 || LOGF == 9 ? 8 : 16;
    static constexpr int R3 = LOGF == 4 ? 4 : LOGF == 8 || LOGF == 12 ? 16 : 8;
    static constexpr int R2 = F / (R1 * R3);
    static constexpr int R = 2;
    static constexpr int TH = 256;
    static constexpr int A0 = 8192 / (R * F) / (FEW ? 4 : 1), A = A0 > 128 ? 128 : A0 < 1 ? 1 : A0;
    static constexpr int AT = A > 1 ? 2 : 1;                                // antennas per thread, polyphase sums
    static constexpr int RT = A * R1 * R2 / 2 >= TH ? R : 1;                // frames per thread, last step
    static constexpr int P2 = R3 + 1;
    static constexpr int P1 = R2 == 1 ? P2 : R2 * P2 + (24 - (R2 * P2) % 16) % 16;
    static constexpr int PG = A >= 16 ? 1 : (16 / A) % 16;  // plane pitch mod 16
    static constexpr int PLANE = R1 * P1 + (16 + PG - (R1 * P1) % 16) % 16;
    static constexpr size_t SMEM = sizeof(float2) * ((size_t)A * R * PLANE + F + F / 16 + F / 128 + 1);
    static_assert(R2 == 1 || P1 % 16 == 8, "pitch");
    static_assert(SMEM <= 113 * 1024, "two CTAs per SM");
};

// FEW: a quarter of the antennas per CTA.
template <int LOGF, bool FEW>
__global__ void __launch_bounds__(MGeom<LOGF, FEW>::TH, 2) fengine_multi(const int8_t* __restrict__ raw, int64_t N,
                                                                      int64_t S, int P, const float* __restrict__ w,
                                                                      int64_t T, const float2* __restrict__ gains,
                                                                      float scale, void* __restrict__ out, int out_i8,
                                                                      int vec, int batches_per_cta) {
    using G = MGeom<LOGF, FEW>;
    constexpr int F = G::F, R1 = G::R1, R2 = G::R2, R3 = G::R3, R = G::R, TH = G::TH, A = G::A, AT = G::AT, RT = G::RT;
    constexpr int P1 = G::P1, P2 = G::P2, PLANE = G::PLANE, H = R1 * R2;
    extern __shared__ float2 sm[];
    float2* tw = sm + A * R * PLANE;  // e^{-i pi j / F}
    const int tid = threadIdx.x;
    for (int j = tid; j < F; j += TH) {
        if constexpr (LOGF <= 8) {
            tw[tw_at(j)] = g_fetw[j << (12 - LOGF)];
        } else {  // no table: its first call needs no upload
            float sn, cs;
            sincospif(-(float)j / (float)F, &sn, &cs);
            tw[tw_at(j)] = make_float2(cs, sn);
        }
    }
    const int64_t groups = (N + A - 1) / A;
    const int64_t a0 = (blockIdx.x % groups) * A;  // neighbouring CTAs complete each other's output lines in L2
    const int64_t M = 2 * (int64_t)F;
    const int64_t t_begin = (blockIdx.x / groups) * (int64_t)batches_per_cta * R;
    const int64_t t_end = min(T, t_begin + (int64_t)batches_per_cta * R);
    auto at = [](int m) { return (m / (R2 * R3)) * P1 + ((m / R3) % R2) * P2 + m % R3; };
    for (int64_t t0 = t_begin; t0 < t_end; t0 += R) {
        // ---- polyphase sums of points m, m + 1 (samples 2m .. 2m + 3), AT antennas x R frames
        for (int item = tid; item < A / AT * (F / 2); item += TH) {
            const int m = 2 * (item & (F / 2 - 1)), al = AT * (item >> (LOGF - 1));
            float u[AT][R][4], x[AT][R][4];
            const int8_t* ra = raw + (a0 + al) * S + 2 * m;
            int64_t last[AT];  // frames of each antenna that exist
#pragma unroll
            for (int i = 0; i < AT; ++i) {
                last[i] = a0 + al + i < N ? T + P - 1 : 0;
#pragma unroll
                for (int r = 0; r < R; ++r) u[i][r][0] = u[i][r][1] = u[i][r][2] = u[i][r][3] = 0.f;
            }
            auto fetch = [&](int i, int64_t frame) -> uint32_t {
                if (frame >= last[i]) return 0;
                const int8_t* q = ra + i * S + frame * M;
                if (vec) return __ldg(reinterpret_cast<const uint32_t*>(q));
                return (uint32_t)(uint8_t)q[0] | (uint32_t)(uint8_t)q[1] << 8 | (uint32_t)(uint8_t)q[2] << 16 |
                       (uint32_t)(uint8_t)q[3] << 24;  // rows of any alignment
            };
            auto window = [&](int p) -> float4 {
                if (!w || p >= P) return make_float4(1.f, 1.f, 1.f, 1.f);
                const float* wp = w + p * M + 2 * m;
                if (vec) return __ldg(reinterpret_cast<const float4*>(wp));
                return make_float4(__ldg(wp), __ldg(wp + 1), __ldg(wp + 2), __ldg(wp + 3));
            };
            auto widen = [](uint32_t v, float (&d)[4]) {
#pragma unroll
                for (int b = 0; b < 4; ++b) d[b] = (float)(int8_t)(v >> (8 * b));
            };
            // x is a ring: frame t0 + p + r sits in x[(p + r) % R].  GP taps at a time, the
            // next GP frames' samples and taps' weights loaded a group ahead
            constexpr int GP = 4;
            static_assert(GP % R == 0, "the ring's place of tap p0 + k is k % R");
            uint32_t nx[AT][GP];
            float4 nw[GP];
            auto ahead = [&](int p0) {  // tap p0 + k's weights, and the frame its successor needs
#pragma unroll
                for (int k = 0; k < GP; ++k) {
                    nw[k] = window(p0 + k);
#pragma unroll
                    for (int i = 0; i < AT; ++i) nx[i][k] = p0 + k + 1 < P ? fetch(i, t0 + p0 + k + R) : 0;
                }
            };
            uint32_t first[AT][R];
#pragma unroll
            for (int i = 0; i < AT; ++i)
#pragma unroll
                for (int r = 0; r < R; ++r) first[i][r] = fetch(i, t0 + r);
            ahead(0);
#pragma unroll
            for (int i = 0; i < AT; ++i)
#pragma unroll
                for (int r = 0; r < R; ++r) widen(first[i][r], x[i][r]);
            for (int p0 = 0; p0 < P; p0 += GP) {
                uint32_t cx[AT][GP];
                float4 cw[GP];
#pragma unroll
                for (int k = 0; k < GP; ++k) {
                    cw[k] = nw[k];
#pragma unroll
                    for (int i = 0; i < AT; ++i) cx[i][k] = nx[i][k];
                }
                if (p0 + GP < P) ahead(p0 + GP);
#pragma unroll
                for (int k = 0; k < GP; ++k) {
                    if (p0 + k < P) {
                        const float wv[4] = {cw[k].x, cw[k].y, cw[k].z, cw[k].w};
#pragma unroll
                        for (int b = 0; b < 4; ++b)
#pragma unroll
                            for (int i = 0; i < AT; ++i)
#pragma unroll
                                for (int r = 0; r < R; ++r) u[i][r][b] = fmaf(wv[b], x[i][(k + r) % R][b], u[i][r][b]);
#pragma unroll
                        for (int i = 0; i < AT; ++i) widen(cx[i][k], x[i][k % R]);  // the oldest frame makes room
                    }
                }
            }
            float2* d = sm + al * PLANE + at(m);
#pragma unroll
            for (int i = 0; i < AT; ++i)
#pragma unroll
                for (int r = 0; r < R; ++r) {  // m is even and R3 too: both points lie in one run
                    d[(r * A + i) * PLANE] = make_float2(u[i][r][0], u[i][r][1]);
                    d[(r * A + i) * PLANE + 1] = make_float2(u[i][r][2], u[i][r][3]);
                }
        }
        __syncthreads();
        // ---- step 1: over j1, for each (j2, j3)
        for (int task = tid; task < A * R * (F / R1); task += TH) {
            const int b = task & (F / R1 - 1);
            float2* z = sm + (task / (F / R1)) * PLANE + (b / R3) * P2 + b % R3;
            float2 v[R1];
#pragma unroll
            for (int j = 0; j < R1; ++j) v[brev(j, ilog2(R1))] = z[j * P1];
            dit<R1, F, true>(v, tw, 0, 1);
#pragma unroll
            for (int q = 0; q < R1; ++q) z[q * P1] = v[q];
        }
        __syncthreads();
        // ---- step 2: over j2, for each (q1, j3)
        if constexpr (R2 > 1) {
            for (int task = tid; task < A * R * R1 * R3; task += TH) {
                const int c = task % R3, q1 = (task / R3) % R1;
                float2* z = sm + (task / (R1 * R3)) * PLANE + q1 * P1 + c;
                float2 v[R2];
#pragma unroll
                for (int j = 0; j < R2; ++j) v[brev(j, ilog2(R2))] = z[j * P2];
                dit<R2, F>(v, tw, q1, R1);
#pragma unroll
                for (int q = 0; q < R2; ++q) z[q * P2] = v[q];
            }
            __syncthreads();
        }
        // ---- step 3: over j3 for the columns k and H - k (k = 0: with H / 2), then
        // X_f = E_f + e^{-i pi f / F} O_f, E_f = (Z_f + conj Z_{F-f}) / 2, O_f = (Z_f - conj Z_{F-f}) / (2i)
        for (int task = tid; task < A * (R / RT) * (H / 2); task += TH) {
            const int al = task % A, tau = (task / A) % (H / 2), r0 = task / (A * (H / 2)) * RT;
            constexpr int HQ = R2 > 1 ? R2 / 2 : 1;  // k = q1 + R1 q2 with q2 fastest over the lanes
            const int k0 = R2 > 1 ? tau / HQ + R1 * (tau % HQ) : tau;
            const int k1 = k0 ? H - k0 : H / 2;
            const int64_t a = a0 + al;
            // gains of f = k0 + H q and k1 + H q, on their way during the transforms (columns of
            // 16 leave no registers for them)
            constexpr bool EARLY = R3 <= 8;
            auto gain = [&](int f) { return gains && a < N ? __ldg(gains + (int64_t)f * N + a) : make_float2(1.f, 0.f); };
            float2 g0[EARLY ? R3 : 1], g1[EARLY ? R3 : 1];
            if constexpr (EARLY) {
#pragma unroll
                for (int q = 0; q < R3; ++q) {
                    g0[q] = gain(k0 + H * q);
                    g1[q] = gain(k1 + H * q);
                }
            }
#pragma unroll 1
            for (int r = r0; r < r0 + RT; ++r) {
                const int64_t t = t0 + r;
                const float2* z = sm + (r * A + al) * PLANE;
                float2 v0[R3], v1[R3];
                const float2 *z0 = z + (k0 % R1) * P1 + (k0 / R1) * P2, *z1 = z + (k1 % R1) * P1 + (k1 / R1) * P2;
#pragma unroll
                for (int j = 0; j < R3; ++j) {
                    v0[brev(j, ilog2(R3))] = z0[j];
                    v1[brev(j, ilog2(R3))] = z1[j];
                }
                dit<R3, F>(v0, tw, k0, H);
                dit<R3, F>(v1, tw, k1, H);
                if (a >= N || t >= T) continue;
                auto put = [&](int c, int q, float2 e, float2 o) {  // f = k + H q of column c
                    const int f = (c ? k1 : k0) + H * q;
                    float2 g;
                    if constexpr (EARLY) g = c ? g1[q] : g0[q];
                    else g = gain(f);
                    const float2 x = cadd(e, cmul(o, tw[tw_at(f)]));
                    const float2 y = calibrate(x, g, scale);
                    const int64_t oi = ((int64_t)f * T + t) * N + a;
                    if (out_i8) reinterpret_cast<char2*>(out)[oi] = make_char2(quantize8(y.x), quantize8(y.y));
                    else reinterpret_cast<float2*>(out)[oi] = y;
                };
                auto unpack = [&](float2 zf, float2 zc, float2& e, float2& o) {
                    e = make_float2(0.5f * (zf.x + zc.x), 0.5f * (zf.y - zc.y));
                    o = make_float2(0.5f * (zf.y + zc.y), -0.5f * (zf.x - zc.x));
                };
                float2 e, o;
                if (k0) {
#pragma unroll
                    for (int q = 0; q < R3; ++q) {
                        unpack(v0[q], v1[R3 - 1 - q], e, o);
                        put(0, q, e, o);
                        put(1, R3 - 1 - q, make_float2(e.x, -e.y), make_float2(o.x, -o.y));  // F - f
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < R3; ++q) {
                        unpack(v0[q], v0[(R3 - q) % R3], e, o);
                        put(0, q, e, o);
                        unpack(v1[q], v1[R3 - 1 - q], e, o);
                        put(1, q, e, o);
                    }
                }
            }
        }
        __syncthreads();
    }
}

template <int LOGF, bool FEW = false>
cudaError_t launch_multi(const int8_t* raw, int64_t N, int64_t S, int P, const float* w, int64_t T, const float2* gains,
                         float scale, void* out, int out_i8, cudaStream_t st) {
    using G = MGeom<LOGF, FEW>;
    // beyond 256 channels (below, the 16-antenna pass takes the small calls), fewer CTAs than
    // a quarter of the SMs: a quarter of the antennas each (512 channels, 8 antennas, 4 frames,
    // 12 taps, odd rows: two CTAs 37.5 us, eight 14; but 1024 channels, 4 antennas, 256 frames,
    // 1 tap: 128 CTAs 15 us, 512 21)
    if constexpr (!FEW && LOGF >= 9 && G::A > 1) {
        if (4 * ((N + G::A - 1) / G::A) * ((T + G::R - 1) / G::R) < 152)
            return launch_multi<LOGF, true>(raw, N, S, P, w, T, gains, scale, out, out_i8, st);
    }
    auto k = fengine_multi<LOGF, FEW>;
    cudaError_t e = smem_limit_once((const void*)k, G::SMEM);
    if (e != cudaSuccess) return e;
    // 4-byte sample loads and 16-byte window loads where the rows allow them
    const int vec = S % 4 == 0 && (uintptr_t)raw % 4 == 0 && (uintptr_t)w % 16 == 0;
    const int64_t groups = (N + G::A - 1) / G::A, batches = (T + G::R - 1) / G::R;
    // several batches per CTA share its twiddle table, as long as eight CTAs per SM remain
    const int64_t per = std::max<int64_t>(1, std::min<int64_t>(8, groups * batches / (8 * 152)));
    const int64_t ctas = groups * ((batches + per - 1) / per);
    k<<<(unsigned)ctas, G::TH, G::SMEM, st>>>(raw, N, S, P, w, T, gains, scale, out, out_i8, vec, (int)per);
    return cudaGetLastError();
}

cudaError_t upload_fengine_twiddles() {
    static float2 h[4096];
    for (int j = 0; j < 4096; ++j) {
        const double ang = -6.283185307179586476925286766559 * j / 8192.0;
        h[j] = make_float2((float)std::cos(ang), (float)std::sin(ang));
    }
    return cudaMemcpyToSymbol(g_fetw, h, sizeof h);
}

}  // namespace

int64_t fengine_frames(int64_t n_samples, int32_t F, int32_t P) {
    const int64_t M = 2 * (int64_t)F;
    return n_samples >= (int64_t)(P - 1) * M ? (n_samples - (int64_t)(P - 1) * M) / M : 0;
}

int64_t fengine_scratch_bytes(int64_t N, int64_t S, int32_t F, int32_t P) {
    if (F <= 256) return 0;
    // larger F staged their spectra here; callers still provide it, no pass uses it
    return (int64_t)sizeof(float2) * N * fengine_frames(S, F, P) * F;
}

int64_t fengine_ctas(int64_t N, int64_t T, int32_t F) {
    if (F <= 256) {
        const int FR = kFusePoints / (kFuseAnt * F);
        return ((N + kFuseAnt - 1) / kFuseAnt) * ((T + FR - 1) / FR);
    }
    // at most one CTA per 32 x 32 channels and antennas of a frame
    return std::max<int64_t>(N * ((T + 31) / 32), ((F + 31) / 32) * ((N + 31) / 32) * T);
}

cudaError_t launch_fengine(const int8_t* raw, int64_t N, int64_t S, int32_t F, int32_t P,
                           const float* window, const float2* gains, float scale, int out_i8,
                           void* out, cudaStream_t st) {
    const int64_t T = fengine_frames(S, F, P);
    if (T <= 0 || N <= 0) return cudaSuccess;
    int logF = 0;
    while ((1 << logF) < F) ++logF;
    if (F <= 256) {  // the tables of the smaller transforms, once per device
        static std::mutex mu;
        static std::vector<int> done;
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        std::lock_guard<std::mutex> lock(mu);
        if (std::find(done.begin(), done.end(), dev) == done.end()) {
            if ((e = upload_fengine_twiddles()) != cudaSuccess) return e;
            if ((e = upload_twiddles()) != cudaSuccess) return e;  // this unit's FFT tables
            done.push_back(dev);
        }
    }
    const bool vec = F >= 8 && S % 16 == 0 && (uintptr_t)raw % 16 == 0 && (uintptr_t)window % 16 == 0;
    if (F == 64 && vec && P <= kF64MaxTaps) {
        int frames = kF64Frames;
        const int64_t groups = (N + kF64Ant - 1) / kF64Ant;
        while (frames > 2 && groups * ((T + frames - 1) / frames) < 152) frames /= 2;
        const unsigned c64 = (unsigned)(groups * ((T + frames - 1) / frames));
        auto pick = [&](auto part) {
            constexpr bool PART = decltype(part)::value;
            return out_i8 ? (gains ? fengine64<true, true, PART> : fengine64<true, false, PART>)
                          : (gains ? fengine64<false, true, PART> : fengine64<false, false, PART>);
        };
        auto k = N <= kF64Ant - 4 ? pick(std::true_type{}) : pick(std::false_type{});
        k<<<c64, 256, 0, st>>>(raw, N, S, P, window, T, gains, scale, out, frames);
        return cudaGetLastError();
    }
    // up to 256 channels the CTA of the pass above takes 4096 / F antennas, twice what the
    // radix-2 pass does in points: with fewer antennas, or too few points for one CTA per SM,
    // the smaller CTAs win (8 antennas, 16 channels, 4 taps, 2048 frames: 14 against 30 us; 64
    // antennas, 256 channels, 16 frames: 21 against 27)
    const bool small = F <= 256 && (N < 4096 / F || N * T * F < (int64_t)152 * 8192);
    switch (small ? 0 : logF) {
#define OMNI_MULTI(n) \
    case n: return launch_multi<n>(raw, N, S, P, window, T, gains, scale, out, out_i8, st)
        OMNI_MULTI(4);
        OMNI_MULTI(5);
        OMNI_MULTI(6);
        OMNI_MULTI(7);
        OMNI_MULTI(8);
        OMNI_MULTI(9);
        OMNI_MULTI(10);
        OMNI_MULTI(11);
        OMNI_MULTI(12);
#undef OMNI_MULTI
        default: break;  // F < 16, or small
    }
    const unsigned ctas = (unsigned)fengine_ctas(N, T, F);
    if (out_i8 && vec)
        fengine_fused<true, true><<<ctas, kFThreads, 0, st>>>(raw, N, S, F, logF, P, window, T, gains, scale, out);
    else if (out_i8)
        fengine_fused<true, false><<<ctas, kFThreads, 0, st>>>(raw, N, S, F, logF, P, window, T, gains, scale, out);
    else if (vec)
        fengine_fused<false, true><<<ctas, kFThreads, 0, st>>>(raw, N, S, F, logF, P, window, T, gains, scale, out);
    else
        fengine_fused<false, false><<<ctas, kFThreads, 0, st>>>(raw, N, S, F, logF, P, window, T, gains, scale, out);
    return cudaGetLastError();
}

}  // namespace omni
