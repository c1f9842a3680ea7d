// omni_fft_smem3.cu -- three-step shared-memory forward transforms of 2048 and
// 4096 points.
//
// L = L1 x L2 x L3 with L1 = L2 = 16 and L3 = 8 or 16, so that no register
// transform is longer than 16 points (a 64-point column held in registers took
// 210-255 registers and left one or two CTAs per SM).  With j = j3 + L3 j2 + M j1
// (M = L2 L3) and k = k1 + L1 (k2 + L2 k3):
//   step 1: L1-point DFTs over j1 for each j' = j3 + L3 j2, times w_L^(j' k1)
//   step 2: L2-point DFTs over j2 for each (k1, j3), times w_M^(j3 k2)
//   step 3: L3-point DFTs over j3 for each (k1, k2)
// (the factorisation of w_L^(j k) into the three DFTs and two twiddle stages).
// The inverse passes use the same transform (the inverse runs as a forward FFT)
// on all L inputs and keep the lag slots, the last one conjugated and scaled.
// A 256-thread CTA, two per SM (one of 512 where four lines of 4096 points go together),
// transforms W lines in pairs: each shared-memory element
// is one point of two lines (re, re, im, im), so that a point is one 16-byte access, the
// butterflies run on both lines per f32x2 instruction and the twiddle powers are formed
// once for both.  A line pair is held as [j1][j2][j3] with a row pitch L3 + 1, so that
// each step's quarter-warps touch 8 different 16-byte banks (j1 pitch
// 1, pair pitch 4, mod 8); each thread reads one
// twiddle w^j through L1 and forms the powers it needs in registers.  LAST, reading the
// scratch buffer, copies the next sample's inputs asynchronously (cp.async) into a staging
// buffer while the current sample runs steps 2 and 3.  Lines are W consecutive inner
// indices (strided axes), or, for an axis that is innermost in memory, W consecutive
// outer lines read and written contiguously: step 1 takes its inputs from memory and step 3,
// whose bins are consecutive across a warp, writes its outputs there.  LAST keeps |X|^2 of
// the chunk's samples in registers and folds them into the FP64 accumulator once.  The
// forward inputs j >= L/2 are zero (padding): step 1 never reads them.
// What bounds it is shared memory (four 8-byte passes per point and line) and FP32.  1024 x
// 1024 antennas (2048-point axes), 64 samples, line by line at 512 (LAST 256) threads against
// pairs, serial: MID 0.48 -> 0.30 ms (5.4 TB/s), LAST 0.65 -> 0.59 ms (inputs and outputs
// through shared memory too, in pairs: MID 0.42).  The 4096-point LAST pass spills 56 bytes
// at the 128 registers of two CTAs per SM.
#include "omni_fft_common.cuh"

namespace omni {
namespace {

// lines per CTA (see smem3_lines)
constexpr int kS3W2048 = 4, kS3W4096 = 2, kS3W4096Strided = 4;

// one step-1 task (16 points of a line pair) per thread
constexpr int s3_threads(int L, int W) { return W / 2 * L / 16; }

template <int L1, int L2, int L3>
struct S3Geom {
    static constexpr int L = L1 * L2 * L3, M = L2 * L3;
    static constexpr int P2 = L3 + 1, P1 = L2 * P2 + 1, PLANE = L1 * P1 + (12 - L1 * P1 % 8) % 8;
    static_assert(P2 % 8 == 1 && P1 % 8 == 1 && PLANE % 8 == 4, "16-byte points on different banks");
};

// 16-byte asynchronous copy global -> shared (zero-filled when !valid; src must
// still be a valid address)
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 16 : 0));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// w^k for k < 16 from w^1 (one shared-memory read per thread instead of a read of
// w^(j k) per k, whose stride k across the lanes conflicted): powers 1..3 and
// 4, 8, 12 by squaring, then w^(4a + b) = w^(4a) w^b (at most six roundings)
struct Pow16 {
    float2 p[4], q[4];  // w^b, w^(4a)
    __device__ __forceinline__ explicit Pow16(float2 w) {
        p[0] = make_float2(1.f, 0.f);
        p[1] = w;
        p[2] = cmul(w, w);
        p[3] = cmul(p[2], w);
        q[0] = p[0];
        q[1] = cmul(p[2], p[2]);
        q[2] = cmul(q[1], q[1]);
        q[3] = cmul(q[2], q[1]);
    }
    __device__ __forceinline__ float2 operator()(int k) const {  // k a compile-time constant after unrolling
        return (k & 3) == 0 ? q[k >> 2] : (k < 4 ? p[k] : cmul(q[k >> 2], p[k & 3]));
    }
};

// one point of two lines, as it lies in shared memory and in registers
__device__ __forceinline__ void get2(const float4* p, f2x& x, f2x& y) {
    const float4 q = *p;
    x = pack2(q.x, q.y);
    y = pack2(q.z, q.w);
}
__device__ __forceinline__ void put2(float4* p, f2x x, f2x y) {
    const float2 a = unpack2(x), b = unpack2(y);
    *p = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void cmul2(f2x& x, f2x& y, float2 w) {
    const f2x c = dup2(w.x), t = x;
    x = fma2(t, c, mul2(y, dup2(-w.y)));
    y = fma2(t, dup2(w.y), mul2(y, c));
}

// PF (LAST from the float2 scratch buffer, 16-byte aligned rows): the next
// sample's W x L/2 inputs are copied asynchronously into a staging buffer
// [j][W] while the current sample runs steps 2 and 3, and step 1 reads them there.
template <int L1, int L2, int L3, int W, bool ROWS, int MODE, int SRC, bool PF>
__global__ void __launch_bounds__(s3_threads(L1 * L2 * L3, W), 512 / s3_threads(L1 * L2 * L3, W)) pass_smem3(Pass p, PassArgs a) {
    using G = S3Geom<L1, L2, L3>;
    static_assert(!PF || (MODE == MODE_LAST && SRC == SRC_BUF && !ROWS), "prefetch form");
    constexpr int L = G::L, M = G::M, P1 = G::P1, P2 = G::P2, PLANE = G::PLANE;
    constexpr bool FWD = MODE == MODE_MID || MODE == MODE_LAST;  // forward: inputs j >= L/2 are zero
    constexpr int LOG1 = ilog2(L1), LOG2 = ilog2(L2), LOG3 = ilog2(L3), H = W / 2;
    constexpr int NT = s3_threads(L, W);
    static_assert(W % 2 == 0 && H * M == NT && H * L1 * L3 == NT, "one task per thread, steps 1 and 2");
    constexpr int T3 = H * L1 * L2 / NT;  // step-3 tasks per thread
    extern __shared__ float4 sm4[];
    float4* lines = sm4;                                            // [H][PLANE]
    float2* stage = reinterpret_cast<float2*>(lines + H * PLANE);   // PF: [L/2][W]
    const int tid = threadIdx.x;
    auto twv = [&](int m) { return __ldg(&g_tw4096[m * (kTwiddleN / L)]); };

    const int n = p.n;  // inputs per line (<= L / 2 forward, <= L inverse)
    const int64_t inner = p.inner;
    int64_t b = blockIdx.x, o0 = 0, i0 = 0, s_first = 0, n_samples = 1, cc = 0;
    if constexpr (ROWS) {  // W consecutive outer lines (inner == 1), one sample
        const int64_t tiles = (p.outer + W - 1) / W;
        o0 = (b % tiles) * W;
        s_first = b / tiles;
    } else {
        const int64_t tiles = (inner + W - 1) / W;
        i0 = (b % tiles) * W;
        b /= tiles;
        if constexpr (MODE == MODE_LAST) {
            cc = b;  // outer == 1
            int tb, te;
            slice_samples(a, tb, te);
            s_first = cc * a.tc + tb;
            n_samples = te - tb;
        } else {
            o0 = b % p.outer;
            s_first = b / p.outer;
        }
    }
    // the lines this CTA has (the last tile may be short)
    auto line_ok = [&](int w) { return ROWS ? o0 + w < p.outer : i0 + w < inner; };

    f2x acc[MODE == MODE_LAST ? T3 : 1][L3];
#pragma unroll
    for (int u = 0; u < (MODE == MODE_LAST ? T3 : 1); ++u)
#pragma unroll
        for (int k = 0; k < L3; ++k) acc[u][k] = dup2(0.f);

    // PF: one sample's inputs, 16 bytes (two lines) per copy; rows j >= n and lines
    // past the axis are zero-filled
    auto prefetch = [&](int64_t s) {
        const float2* row0 = reinterpret_cast<const float2*>(a.src) + s * a.src_stride + i0;
        constexpr int NC = (L / 2) * H / NT;
        static_assert(NC * NT == (L / 2) * H, "copies per thread");
#pragma unroll
        for (int r = 0; r < NC; ++r) {
            const int c = tid + r * NT, j = c / H, h = c % H;
            const bool ok = j < n && i0 + 2 * h < inner;
            cp_async16(stage + j * W + 2 * h, ok ? row0 + (int64_t)j * inner + 2 * h : row0, ok);
        }
        cp_async_commit();
    };
    if constexpr (PF)
        if (n_samples > 0) prefetch(s_first);

    for (int64_t ts = 0; ts < n_samples; ++ts) {
        const int64_t s = s_first + ts;
        const int64_t base = src_base(a, s);
        if constexpr (PF) {
            cp_async_wait_all();  // this sample's staging copies
            __syncthreads();      // ... everyone's, and the lines are free
        }
        // step 1: j' = j3 + L3 j2 fastest across the threads (strided axes: the line pairs), inputs
        // straight from the staging buffer or from memory, all of a thread's loads together
        {
            const int h = ROWS ? tid / M : tid % H, jp = ROWS ? tid - h * M : tid / H, j2 = jp / L3, j3 = jp - j2 * L3;
            float4* col = lines + h * PLANE + j2 * P2 + j3;
            f2x x[L1], y[L1];
            constexpr int NIN = FWD ? L1 / 2 : L1;
            if constexpr (PF) {
#pragma unroll
                for (int j1 = 0; j1 < NIN; ++j1) {
                    const float4 q = *reinterpret_cast<const float4*>(stage + (jp + M * j1) * W + 2 * h);
                    x[j1] = pack2(q.x, q.z);
                    y[j1] = pack2(q.y, q.w);
                }
            } else {
                const bool ok0 = line_ok(2 * h), ok1 = line_ok(2 * h + 1);
                const int64_t first = ROWS ? base + (o0 + 2 * h) * (int64_t)n : base + o0 * (int64_t)n * inner + i0 + 2 * h;
                const int64_t next = ROWS ? n : 1, step = ROWS ? 1 : inner;  // to the second line; to the next input
#pragma unroll
                for (int j1 = 0; j1 < NIN; ++j1) {
                    const int j = jp + M * j1;
                    const float2 zero = make_float2(0.f, 0.f);
                    const float2 u = j < n && ok0 ? ld_src<SRC>(a.src, first + j * step) : zero;
                    const float2 v = j < n && ok1 ? ld_src<SRC>(a.src, first + next + j * step) : zero;
                    x[j1] = pack2(u.x, v.x);
                    y[j1] = pack2(u.y, v.y);
                }
            }
#pragma unroll
            for (int j1 = NIN; j1 < L1; ++j1) x[j1] = y[j1] = dup2(0.f);
            fft_dif2<L1, FWD>(x, y);
            const Pow16 pw(twv(jp));  // w_L^(j' k1)
#pragma unroll
            for (int k1 = 0; k1 < L1; ++k1) {
                f2x &vx = x[brev(k1, LOG1)], &vy = y[brev(k1, LOG1)];
                if (k1) cmul2(vx, vy, pw(k1));
                put2(col + k1 * P1, vx, vy);
            }
        }
        __syncthreads();
        if constexpr (PF)
            if (ts + 1 < n_samples) prefetch(s + 1);  // the staging buffer is free until the next step 1
        // step 2: (k1, j3), j3 fastest
        {
            const int j3 = tid % L3, k1 = (tid / L3) % L1, h = tid / (L3 * L1);
            float4* row = lines + h * PLANE + k1 * P1 + j3;
            f2x x[L2], y[L2];
#pragma unroll
            for (int j2 = 0; j2 < L2; ++j2) get2(row + j2 * P2, x[j2], y[j2]);
            fft_dif2<L2, false>(x, y);
            const Pow16 pw(twv(L1 * j3));  // w_M^(j3 k2) = w_L^(L1 j3 k2)
#pragma unroll
            for (int k2 = 0; k2 < L2; ++k2) {
                f2x &vx = x[brev(k2, LOG2)], &vy = y[brev(k2, LOG2)];
                if (k2) cmul2(vx, vy, pw(k2));
                put2(row + k2 * P2, vx, vy);
            }
        }
        __syncthreads();
        // step 3: (k1, k2), k1 fastest: X[k1 + L1 k2 + L1 L2 k3], so that a warp's outputs of one
        // k3 are consecutive bins and go straight out
#pragma unroll
        for (int u = 0; u < T3; ++u) {
            const int t = tid + u * NT;
            const int h = ROWS ? t / (L1 * L2) : t % H, k12 = ROWS ? t % (L1 * L2) : t / H, k1 = k12 % L1, k2 = k12 / L1;
            const float4* r = lines + h * PLANE + k1 * P1 + k2 * P2;
            f2x x[L3], y[L3];
#pragma unroll
            for (int j3 = 0; j3 < L3; ++j3) get2(r + j3, x[j3], y[j3]);
            fft_dif2<L3, false>(x, y);
            const bool ok0 = line_ok(2 * h), ok1 = line_ok(2 * h + 1);
#pragma unroll
            for (int k3 = 0; k3 < L3; ++k3) {
                const f2x vx = x[brev(k3, LOG3)], vy = y[brev(k3, LOG3)];
                if constexpr (MODE == MODE_LAST) {
                    acc[u][k3] = add2(acc[u][k3], fma2(vx, vx, mul2(vy, vy)));
                } else {
                    // forward: slot k; inverse: the slot of lag k or k - L, if it is kept (the last pass
                    // conjugates and scales: the inverse runs as a forward FFT)
                    const int k = k12 + L1 * L2 * k3, Q = FWD ? L : p.q_out;
                    const int q = FWD ? k : (k < L - p.q_shift ? k : k - L) + p.q_shift;
                    if (!FWD && q >= Q) continue;
                    const float2 re = unpack2(vx), im = unpack2(vy);
                    const int64_t at = ROWS ? (o0 + 2 * h) * (int64_t)Q + q : (o0 * Q + q) * inner + i0 + 2 * h;
                    const int64_t second = at + (ROWS ? Q : 1);
                    if constexpr (MODE == MODE_INV_LAST) {
                        double2* V = a.V + (a.c0 + s) * a.V_stride;
                        if (ok0) V[at] = visibility(make_float2(re.x, im.x), a);
                        if (ok1) V[second] = visibility(make_float2(re.y, im.y), a);
                    } else {
                        float2* d = a.dst + s * a.dst_stride;
                        if (ok0) d[at] = make_float2(re.x, im.x);
                        if (ok1) d[second] = make_float2(re.y, im.y);
                    }
                }
            }
        }
        if (!PF && ts + 1 < n_samples) __syncthreads();  // the lines are free (PF: at the next sample's barrier)
    }
    if constexpr (PF) cp_async_wait_all();  // nothing left in flight at exit
    if constexpr (MODE == MODE_LAST) {
#pragma unroll
        for (int u = 0; u < T3; ++u) {
            const int t = tid + u * NT, h = t % H, k12 = t / H;
            const int64_t e0 = (int64_t)k12 * inner + i0 + 2 * h, step = (int64_t)L1 * L2 * inner;
            if (inner % 2 == 0) {
                // both lines of the pair, or neither: 16 bytes at a time, loads together (value by
                // value, each waited for: 16 x 2048 antennas, 16 channels x 4 samples, the pass
                // 152 us against 56)
                if (!line_ok(2 * h)) continue;
                if (gridDim.y > 1) {  // as fold_last
                    float2* d = reinterpret_cast<float2*>(a.part + ((int64_t)blockIdx.y * a.S + cc) * a.P_stride + e0);
#pragma unroll
                    for (int k3 = 0; k3 < L3; ++k3) d[k3 * step / 2] = unpack2(acc[u][k3]);
                    continue;
                }
                double2* P = reinterpret_cast<double2*>(a.P + (a.c0 + cc) * a.P_stride + e0);
                constexpr int NB = 8;
#pragma unroll
                for (int k0 = 0; k0 < L3; k0 += NB) {
                    double2 s[NB];
#pragma unroll
                    for (int k = 0; k < NB; ++k) s[k] = P[(k0 + k) * step / 2];
#pragma unroll
                    for (int k = 0; k < NB; ++k) {
                        const float2 v = unpack2(acc[u][k0 + k]);
                        P[(k0 + k) * step / 2] = make_double2(s[k].x + (double)v.x, s[k].y + (double)v.y);
                    }
                }
            } else {
#pragma unroll
                for (int k3 = 0; k3 < L3; ++k3) {
                    const float2 v = unpack2(acc[u][k3]);
                    if (line_ok(2 * h)) fold_last(a, cc, e0 + k3 * step, v.x);
                    if (line_ok(2 * h + 1)) fold_last(a, cc, e0 + k3 * step + 1, v.y);
                }
            }
        }
    }
}

template <int L1, int L2, int L3, int W, bool PF>
constexpr size_t s3_smem() {
    return sizeof(float4) * (W / 2) * S3Geom<L1, L2, L3>::PLANE + (PF ? sizeof(float2) * W * (L1 * L2 * L3 / 2) : 0);
}

// the prefetch form: LAST from the scratch buffer with 16-byte aligned input rows
inline bool s3_prefetch(const Pass& p, const PassArgs& a) {
    return p.mode == MODE_LAST && a.src_kind == SRC_BUF && p.inner % 2 == 0 && a.src_stride % 2 == 0 &&
           (reinterpret_cast<uintptr_t>(a.src) & 15) == 0;
}

template <int L1, int L2, int L3, int W, bool ROWS, int MODE, int SRC, bool PF>
cudaError_t launch_s3(const Pass& p, const PassArgs& a, cudaStream_t st) {
    int64_t blocks;
    if (ROWS) blocks = a.S * ((p.outer + W - 1) / W);
    else blocks = (MODE == MODE_LAST ? a.S : a.S * p.outer) * ((p.inner + W - 1) / W);
    if (blocks <= 0) return cudaSuccess;
    constexpr size_t smem = s3_smem<L1, L2, L3, W, PF>();
    auto k = pass_smem3<L1, L2, L3, W, ROWS, MODE, SRC, PF>;
    cudaError_t e = smem_limit_once((const void*)k, smem);
    if (e != cudaSuccess) return e;
    k<<<MODE == MODE_LAST ? last_grid(blocks, a) : dim3((unsigned)blocks), s3_threads(L1 * L2 * L3, W), smem, st>>>(p, a);
    return cudaGetLastError();
}

// one length: W lines in a LAST pass and along the innermost axis, WS in the other passes
// of a strided axis
template <int L1, int L2, int L3, int W, int WS>
cudaError_t launch_s3_len(const Pass& p, const PassArgs& a, cudaStream_t st) {
    const bool fwd = p.mode == MODE_MID || p.mode == MODE_LAST;
    if (p.n > (fwd ? L1 * L2 * L3 / 2 : L1 * L2 * L3) || p.W != smem3_lines(p)) return cudaErrorInvalidValue;
    const bool rows = p.mode != MODE_LAST && p.inner == 1;
    if (p.mode == MODE_LAST) {
        if (s3_prefetch(p, a)) return launch_s3<L1, L2, L3, W, false, MODE_LAST, SRC_BUF, true>(p, a, st);
        return dispatch_src<MODE_LAST>(a.src_kind, [&](auto S) {
            return launch_s3<L1, L2, L3, W, false, MODE_LAST, decltype(S)::value, false>(p, a, st);
        });
    }
    return dispatch_mode(p.mode, [&](auto Mc) {
        constexpr int MO = decltype(Mc)::value;
        if constexpr (MO == MODE_LAST) {
            return cudaErrorInvalidValue;
        } else {
            return dispatch_src<MO>(a.src_kind, [&](auto S) {
                return rows ? launch_s3<L1, L2, L3, W, true, MO, decltype(S)::value, false>(p, a, st)
                            : launch_s3<L1, L2, L3, WS, false, MO, decltype(S)::value, false>(p, a, st);
            });
        }
    });
}

// occupancy of the form a LAST pass reading src_kind launches (the prefetch form
// for the scratch buffer)
template <int L1, int L2, int L3, int W>
cudaError_t s3_last_occupancy_len(const Pass& p, int src_kind, int* blocks_per_sm) {
    return dispatch_src<MODE_LAST>(src_kind, [&](auto S) {
        constexpr int SK = decltype(S)::value;
        constexpr bool PF = SK == SRC_BUF;
        constexpr size_t smem = s3_smem<L1, L2, L3, W, PF>();
        auto k = pass_smem3<L1, L2, L3, W, false, MODE_LAST, SK, PF>;
        cudaError_t e = smem_limit_once((const void*)k, smem);
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, s3_threads(L1 * L2 * L3, W), smem);
    });
}

}  // namespace

// this unit's copies of the twiddle tables (static per translation unit)
cudaError_t upload_twiddles_smem3() { return upload_twiddles(); }

bool smem3_supports(int L) { return L == 2048 || L == 4096; }

// Passes of a strided axis touch memory in runs of 8 W bytes.  4096 points: one line pair,
// two CTAs per SM, where a LAST pass sums in registers and its loads run ahead; the other
// passes write every bin and take two pairs, whole 32-byte sectors (8 x 2048 antennas on
// 2 x 2, 16 channels x 32 samples: MID 1.21 -> 0.89 ms, inverse MID 100 -> 66 us).
int smem3_lines(const Pass& p) {
    return p.L == 2048 ? kS3W2048 : p.mode == MODE_LAST || p.inner == 1 ? kS3W4096 : kS3W4096Strided;
}

cudaError_t launch_smem3(const Pass& p, const PassArgs& a, cudaStream_t st) {
    switch (p.L) {
        case 2048: return launch_s3_len<16, 16, 8, kS3W2048, kS3W2048>(p, a, st);
        case 4096: return launch_s3_len<16, 16, 16, kS3W4096, kS3W4096Strided>(p, a, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t smem3_last_occupancy(const Pass& p, int src_kind, int* blocks_per_sm) {
    switch (p.L) {
        case 2048: return s3_last_occupancy_len<16, 16, 8, kS3W2048>(p, src_kind, blocks_per_sm);
        case 4096: return s3_last_occupancy_len<16, 16, 16, kS3W4096>(p, src_kind, blocks_per_sm);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace omni
