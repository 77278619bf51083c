// Polyphase channeliser (dd_channelise): subband voltages -> finer channels.
//
// The paper's pipeline channelises the received subbands in finer frequency
// before it forms Stokes parameters (Sec. 1) and names the poly-phase filter
// (Sec. 5) without giving the filter or the transform size.  The library's
// reading is the critically sampled polyphase filter bank: per polarisation,
// with x[j] = re + i*im of raw sample j of a subband,
//
//     y_k[n] = sum_{m < M*T} h[m] x[n*M + m] exp(-2 pi i k m / M),   k < M,
//
// for spectra n = 0 .. floor(nraw/M) - T.  Grouping m = t*M + p gives the
// two steps computed here: a T-tap FIR per branch p,
//     z_p[n] = sum_t h[t*M + p] x[(n + t)*M + p],
// then an M-point DFT of z[n] over p.  Channel c = (k + M/2) mod M of subband
// s is written to row s*M + c (the bins of a subband in increasing frequency).
//
// Kernel structure.  A group of max(32, M) threads takes whole segments of
// consecutive spectra and meets no other group: with up to 32 channels it is
// a warp, and no barrier is wider than that.  (One group per CTA of 256
// threads and CTA barriers between FIR, DFT and stores took 838 us on the
// 16-channel workload below against 733: every warp was in the same phase, so
// FMA pipe, ALU and shared memory were busy one after the other.)
//  * FIR: thread (p, g) owns branch p of segment g and slides along its
//    spectra in transposed form: each raw sample (one 32-bit word holding
//    Xre, Xim, Yre, Yim) is loaded and converted once, then added with its T
//    weights into the accumulators of the T spectra it belongs to; a
//    spectrum whose last sample arrived is written to shared memory.  A warp
//    loads 32 consecutive branches (128 contiguous bytes) per spectrum.
//  * DFT, four-step M = 16 x M2: pass 1 does a 16-point FFT in registers
//    over p1 (p = M2*p1 + p2) for each (p2, spectrum, polarisation) and
//    multiplies by W_M^(k1*p2); pass 2 does the M2-point FFT over p2 for each
//    k1, giving y[k1 + 16*k2].  Shared memory holds the FFT index as the
//    fastest dimension, so the 32 lanes of a warp always touch 32 different
//    transforms: every shared-memory access is conflict-free.
//  * Packed FP32: the FIR keeps (re, im) pairs and multiplies them by (h, h)
//    with FFMA2, and the FFT's butterflies a +- t run as FADD2 / FFMA2, so a
//    pair of FP32 operations takes one issue slot.
//  * Output: each transform's values go to a shared-memory staging area laid
//    out as [channel][spectrum] -- int8 codes q = clamp(rint(v*scale), -127,
//    127) with v*scale rounded once (FMA into 1.5*2^23), the two
//    polarisations of a spectrum side by side, or FP32 values -- and the CTA
//    then writes channel rows with 16-byte stores (four int8 elements, or one
//    FP32 element, per thread).
//  * Rounds: each round a segment emits RS spectra; the next round's raw
//    words are loaded before the current round's DFT, so they are in flight
//    while it runs, at constant offsets from one pointer where the whole
//    segment lies in the row (a clamped 64-bit block index per word took 15
//    more instructions per raw word, 77 against 62).
//  * Occupancy: CTAs of 128 threads (256 for 256 channels), so that the
//    register file fills up: 16 warps per SM at 16 channels and int8 codes
//    (112 registers; 20 warps at 96 registers measured 752 us against 720),
//    20 at the other sizes (1082 against 1108 us at 128 channels), 12 above 8
//    taps.  24 warps at 80 registers spill: 885 us.
//
// 64 subbands x 16 channels x 8 taps x 295256 spectra to int8: 714 us (357 us
// of compulsory HBM traffic, 3.4 TB/s), bound by the FMA pipe (FFMA2 and
// FADD2 hold it for two cycles) at 67 % and issue at 66 %; 903 us before.
// Going through shared memory instead of registers for the next round's words
// (cp.async ring of 4 rounds: 887 us) or for the taps (880 us) was slower.
//
// HBM traffic: each raw word is read once by the segment that uses it (plus
// T-1 words of overlap per segment, served from L2), each output element
// written once.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <string>
#include <type_traits>

#include "dd_internal.h"

namespace {

// Threads of a CTA: groups share nothing but the launch.
__host__ __device__ constexpr int threads_of(int M) { return M > 128 ? M : 128; }
__host__ __device__ constexpr int ctas_of(int M, int TI, bool ci8) {
    return M > 128 ? (TI > 8 ? 1 : 2) : TI > 8 ? 3 : M == 16 && ci8 ? 4 : 5;
}
constexpr int kM1 = 16;        // size of the first DFT pass
constexpr int kMaxRounds = 32;  // rounds per CTA (segment length RS * rounds)

struct PfbArgs {
    const uint8_t *in;   // raw words, rows of in_pitch bytes
    int64_t in_pitch;
    int64_t nblk;        // whole blocks of M raw samples per row
    int64_t nspec;       // spectra per row
    const float *h;      // M*T prototype coefficients
    int T;               // taps (<= the kernel's TI; the rest are zero)
    int nr;              // rounds per CTA
    float scale;         // int8 output: codes = rint(v * scale)
    int ci8;             // 1: int8 elements (4 bytes), 0: FP32 elements (16 bytes)
    int vec;             // int8 rows 16-byte aligned: four elements per store
    uint8_t *out;
    int64_t out_pitch;   // bytes
};

__host__ __device__ constexpr int bitrev(int i, int n) {
    int r = 0;
    for (int b = 1; b < n; b <<= 1) {
        r = (r << 1) | (i & 1);
        i >>= 1;
    }
    return r;
}

// b * W_16^j, W_16 = exp(-2 pi i / 16), j < 8 (cos and sin of multiples of
// pi/8: 1, sqrt(2 + sqrt 2)/2, sqrt 2 / 2, sqrt(2 - sqrt 2)/2).
__device__ __forceinline__ float2 mul_w16(float2 b, int j) {
    constexpr float c1 = 0.923879532511286756f, c2 = 0.707106781186547524f,
                    c3 = 0.382683432365089772f;
    float c = 1.f, s = 0.f;
    switch (j) {
    case 0: return b;
    case 4: return make_float2(b.y, -b.x);  // times -i
    case 1: c = c1; s = c3; break;
    case 2: c = c2; s = c2; break;
    case 3: c = c3; s = c1; break;
    case 5: c = -c3; s = c1; break;
    case 6: c = -c2; s = c2; break;
    case 7: c = -c1; s = c3; break;
    }
    // (b.x + i b.y)(c - i s)
    return __ffma2_rn(b, make_float2(c, c), make_float2(b.y * s, -(b.x * s)));
}

__device__ __forceinline__ float2 cmul(float2 b, float2 w) {
    return make_float2(fmaf(b.x, w.x, -(b.y * w.y)), fmaf(b.x, w.y, b.y * w.x));
}

// Packed FP32 pairs (one FADD2 / FFMA2 / FMUL2 per pair): a + b, a - b
// (b * -1 + a, one rounding like a subtraction), h * x + c, h * x.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
}

// In-register forward DFT of N <= 16 points: radix-2 decimation in time.
// Butterflies a +- t run on packed pairs; t = -i*b is a swap and a sign.
template <int N>
__device__ __forceinline__ void fft_reg(float2 (&v)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int j = bitrev(i, N);
        if (j > i) {
            const float2 t = v[i];
            v[i] = v[j];
            v[j] = t;
        }
    }
#pragma unroll
    for (int len = 2; len <= N; len *= 2) {
#pragma unroll
        for (int i0 = 0; i0 < N; i0 += len) {
#pragma unroll
            for (int k = 0; k < len / 2; ++k) {
                const int tj = k * (16 / len);
                const float2 a = v[i0 + k];
                const float2 b = v[i0 + k + len / 2];
                if (tj == 4) {  // t = -i b = (b.y, -b.x)
                    v[i0 + k] = make_float2(a.x + b.y, a.y - b.x);
                    v[i0 + k + len / 2] = make_float2(a.x - b.y, a.y + b.x);
                } else {
                    const float2 t = mul_w16(b, tj);
                    v[i0 + k] = add2(a, t);
                    v[i0 + k + len / 2] = sub2(a, t);
                }
            }
        }
    }
}

// Four signed bytes (Xre, Xim, Yre, Yim) -> FP32 pairs X, Y, exactly: byte
// b + 128 is placed in the mantissa of 2^23 and 2^23 + 128 is subtracted.
__device__ __forceinline__ void s8x4(uint32_t w, float2 &x, float2 &y) {
    const uint32_t u = w ^ 0x80808080u;
    const float2 off = make_float2(-8388736.0f, -8388736.0f);  // -(2^23 + 128)
    x = add2(make_float2(__uint_as_float(__byte_perm(u, 0x4b000000u, 0x7650)),
                         __uint_as_float(__byte_perm(u, 0x4b000000u, 0x7651))), off);
    y = add2(make_float2(__uint_as_float(__byte_perm(u, 0x4b000000u, 0x7652)),
                         __uint_as_float(__byte_perm(u, 0x4b000000u, 0x7653))), off);
}

// Codes (re, im) of v*scale, complemented to t = 127 - code in [0, 254] and
// held in the low 16 bits; byte t ^ 0x7f is the code in two's complement.  The
// FMA into 1.5*2^23 rounds each exact product to the nearest integer (ties to
// even) and leaves it in the low bits.  BOUNDED: |v*scale| < 2^22, so that an
// integer add, minimum and clamp to 0 (one instruction) finish the job; else
// the float is clamped first.
template <bool BOUNDED>
__device__ __forceinline__ uint32_t code16(float2 v, float2 neg_scale2) {
    constexpr float magic = 12582912.0f;   // 1.5 * 2^23
    constexpr int bias = 127 - 0x4b400000;  // 127 - its bits
    float2 u = __ffma2_rn(v, neg_scale2, make_float2(magic, magic));
    if (!BOUNDED) {
        // A code of NaN is -127.
        u.x = fmaxf(fminf(u.x, magic + 127.0f), magic - 127.0f);
        u.y = fmaxf(fminf(u.y, magic + 127.0f), magic - 127.0f);
    }
    const uint32_t x = (uint32_t)__viaddmin_s32_relu(__float_as_int(u.x), bias, 254);
    const uint32_t y = (uint32_t)__viaddmin_s32_relu(__float_as_int(u.y), bias, 254);
    return __byte_perm(x, y, 0x0040);
}

// A group of GT threads (a warp for up to 32 channels) transforms the spectra
// of its own segments and meets no other group.
template <int M, int TI>
struct Shape {
    static constexpr int GT = M > 32 ? M : 32;
    static constexpr int NT = threads_of(M);
    static constexpr int NG = NT / GT;        // groups per CTA
    static constexpr int NSEG = GT / M;             // segments per group
    static constexpr int RS = TI > 8 ? TI : 8;      // spectra per segment per round
    static constexpr int R = NSEG * RS;             // spectra per round
    static constexpr int NF = 2 * R;                // transforms per round
    static constexpr int ZS = NF + 2;               // float2 per branch row (conflict-free STS.128)
    static constexpr int M2 = M / kM1;
    // Per group: z rows and output staging, [channel][spectrum of the round],
    // one 4-byte element (int8) or two float2 (FP32) per cell.
    template <bool CI8>
    static constexpr int GROUP = M * ZS * 8 + M * R * (CI8 ? 4 : 16);
    template <bool CI8>
    static constexpr int SMEM = NG * GROUP<CI8> + M * 8;  // and the twiddle table
};

// Barrier of a group of GT threads (every thread of a group passes each one).
template <int GT, int NT>
__device__ __forceinline__ void group_sync(int group) {
    if constexpr (GT == 32)
        __syncwarp();
    else if constexpr (GT == NT)
        __syncthreads();
    else
        asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(GT) : "memory");
}

template <int M, int TI, bool CI8>
__global__ void __launch_bounds__(threads_of(M), ctas_of(M, TI, CI8)) pfb_kernel(const PfbArgs a) {
    using S = Shape<M, TI>;
    constexpr int GT = S::GT, NSEG = S::NSEG, RS = S::RS, R = S::R, NF = S::NF, ZS = S::ZS,
                  M2 = S::M2;
    extern __shared__ __align__(16) uint8_t smem[];
    const int group = threadIdx.x / GT, tid = threadIdx.x % GT;
    float2 *zsm = reinterpret_cast<float2 *>(smem + group * S::template GROUP<CI8>);
    uint8_t *stg = reinterpret_cast<uint8_t *>(zsm + M * ZS);
    float2 *tw = reinterpret_cast<float2 *>(smem + S::NG * S::template GROUP<CI8>);  // W_M^r

    const int sub = blockIdx.y;
    const int64_t seg_len = (int64_t)a.nr * RS;
    const int64_t n_group = ((int64_t)blockIdx.x * S::NG + group) * NSEG * seg_len;

    for (int r = threadIdx.x; r < M; r += S::NT) {
        float sn, cs;
        sincospif(2.0f * (float)r / (float)M, &sn, &cs);
        tw[r] = make_float2(cs, -sn);
    }

    // ------------------------------ FIR state ------------------------------
    const int p = tid % M;
    const int g = tid / M;
    const int64_t n_first = n_group + g * seg_len;
    const uint8_t *row = a.in + (int64_t)sub * a.in_pitch + 4 * (int64_t)p;
    float2 hr[TI];  // (h, h): one packed multiplier per tap
#pragma unroll
    for (int t = 0; t < TI; ++t) {
        const float h = t < a.T ? __ldg(a.h + t * M + p) : 0.0f;
        hr[t] = make_float2(h, h);
    }
    // Does every possible |v*scale| stay below 2^21 (inputs are below 182 in
    // magnitude)?  NaN and infinite coefficients say no.
    float sum = 0.0f;
#pragma unroll
    for (int t = 0; t < TI; ++t)
        sum += fabsf(hr[t].x);
    const bool bounded =
        __syncthreads_and(!CI8 || sum * a.scale * (182.0f * M) < 2097152.0f) != 0;
    // Raw block j of this segment (blocks past the row repeat the last one:
    // they only meet zero taps or spectra that are not stored).
    auto load = [&](int64_t j) -> uint32_t {
        int64_t b = n_first + j;
        b = b < a.nblk ? b : a.nblk - 1;
        return __ldg(reinterpret_cast<const uint32_t *>(row + 4 * M * b));
    };
    // Segments whose every block lies in the row load without that check, at
    // constant offsets from a pointer that moves on by a round.
    const bool inside = n_first + TI - 1 + seg_len <= a.nblk;
    const uint8_t *ahead = row + 4 * M * (n_first + TI - 1);
    float2 ax[TI], ay[TI];  // per spectrum slot: X and Y partial sums
    // Raw block j (j mod TI = J at compile time) into the spectra j - t.
    auto fir = [&](int J, uint32_t w) {
        float2 x, y;
        s8x4(w, x, y);
#pragma unroll
        for (int t = 0; t < TI; ++t) {
            const int slot = ((J - t) % TI + TI) % TI;
            if (t == 0) {
                ax[slot] = __fmul2_rn(hr[0], x);
                ay[slot] = __fmul2_rn(hr[0], y);
            } else {
                ax[slot] = __ffma2_rn(hr[t], x, ax[slot]);
                ay[slot] = __ffma2_rn(hr[t], y, ay[slot]);
            }
        }
    };
    uint32_t xw[RS];
    {
        uint32_t wu[TI - 1];
#pragma unroll
        for (int j = 0; j < TI - 1; ++j)
            wu[j] = load(j);
#pragma unroll
        for (int i = 0; i < RS; ++i)
            xw[i] = load(TI - 1 + i);
#pragma unroll
        for (int j = 0; j < TI - 1; ++j)
            fir(j % TI, wu[j]);
    }
    const float2 scale2 = make_float2(-a.scale, -a.scale);

    // Value y of transform f (= 2 * spectrum-in-round + polarisation) at bin
    // k, into the staging cell of its channel and spectrum.
    auto stage = [&](auto bnd, int f, int k, float2 y) {
        const int c = (k + M / 2) & (M - 1);
        if constexpr (CI8) {
            reinterpret_cast<uint16_t *>(stg)[(c * R + (f >> 1)) * 2 + (f & 1)] =
                (uint16_t)code16<decltype(bnd)::value>(y, scale2);
        } else {
            reinterpret_cast<float2 *>(stg)[(c * R + (f >> 1)) * 2 + (f & 1)] = y;
        }
    };
    auto last_pass = [&](auto bnd) {
        if constexpr (M2 == 1) {
            for (int f = tid; f < NF; f += GT) {
                float2 v[kM1];
#pragma unroll
                for (int p1 = 0; p1 < kM1; ++p1)
                    v[p1] = zsm[p1 * ZS + f];
                fft_reg<kM1>(v);
#pragma unroll
                for (int k = 0; k < kM1; ++k)
                    stage(bnd, f, k, v[k]);
            }
        } else {
            // Pass 2: M2-point FFT over p2 for each (k1, transform f).
            for (int u = tid; u < kM1 * NF; u += GT) {
                const int f = u % NF;
                const int k1 = u / NF;
                float2 v[M2];
#pragma unroll
                for (int p2 = 0; p2 < M2; ++p2)
                    v[p2] = zsm[(M2 * k1 + p2) * ZS + f];
                fft_reg<M2>(v);
#pragma unroll
                for (int k2 = 0; k2 < M2; ++k2)
                    stage(bnd, f, k1 + kM1 * k2, v[k2]);
            }
        }
    };

    // Stores: a thread has the same spectra of a round in channels kCStep
    // apart, 16 bytes of each.
    constexpr int PER = CI8 ? 4 : 1;  // spectra per 16-byte store
    constexpr int kCStep = GT / (R / PER);
    static_assert(GT % (R / PER) == 0 && M % kCStep == 0, "whole steps of channels");
    const int rho = tid % (R / PER) * PER, c0 = tid / (R / PER);
    const int64_t n0 = n_group + rho / RS * seg_len + rho % RS;
    uint8_t *optr = a.out + ((int64_t)sub * M + c0) * a.out_pitch + (CI8 ? 4 : 16) * n0;
    const int64_t ostep = kCStep * a.out_pitch;
    int left = (int)max((int64_t)-0x40000000, min(a.nspec - n0, (int64_t)0x40000000));

    for (int r = 0; r < a.nr; ++r) {
        // FIR: this round's RS raw blocks per segment; spectrum i of the round
        // completes with block TI-1+i and leaves slot i mod TI.
#pragma unroll
        for (int i = 0; i < RS; ++i) {
            fir((TI - 1 + i) % TI, xw[i]);
            const float4 z = make_float4(ax[i % TI].x, ax[i % TI].y, ay[i % TI].x, ay[i % TI].y);
            *reinterpret_cast<float4 *>(&zsm[p * ZS + 2 * (g * RS + i)]) = z;
        }
        if (r + 1 < a.nr) {
            ahead += 4 * M * RS;
            if (inside) {
#pragma unroll
                for (int i = 0; i < RS; ++i)
                    xw[i] = __ldg(reinterpret_cast<const uint32_t *>(ahead + 4 * M * i));
            } else {
#pragma unroll
                for (int i = 0; i < RS; ++i)
                    xw[i] = load(TI - 1 + (int64_t)(r + 1) * RS + i);
            }
        }
        group_sync<GT, S::NT>(group);

        if constexpr (M2 > 1) {
            // Pass 1: 16-point FFT over p1 for each (p2, transform f).
            for (int u = tid; u < M2 * NF; u += GT) {
                const int f = u % NF;
                const int p2 = u / NF;
                float2 v[kM1];
#pragma unroll
                for (int p1 = 0; p1 < kM1; ++p1)
                    v[p1] = zsm[(M2 * p1 + p2) * ZS + f];
                fft_reg<kM1>(v);
#pragma unroll
                for (int k1 = 0; k1 < kM1; ++k1) {
                    const float2 w = tw[(k1 * p2) & (M - 1)];
                    zsm[(M2 * k1 + p2) * ZS + f] = k1 == 0 ? v[0] : cmul(v[k1], w);
                }
            }
            group_sync<GT, S::NT>(group);
        }
        if (bounded)
            last_pass(std::true_type{});
        else
            last_pass(std::false_type{});
        group_sync<GT, S::NT>(group);

        // Stores: channel rows of the staging area to HBM.  The next round's
        // FIR writes only z, so no barrier is needed after this phase.
#pragma unroll
        for (int i = 0; i < M / kCStep; ++i) {
            const int cell = (c0 + i * kCStep) * R + rho;
            uint8_t *o = optr + i * ostep;
            if constexpr (CI8) {
                uint4 wv = *reinterpret_cast<const uint4 *>(stg + cell * 4);
                wv.x ^= 0x7f7f7f7fu;
                wv.y ^= 0x7f7f7f7fu;
                wv.z ^= 0x7f7f7f7fu;
                wv.w ^= 0x7f7f7f7fu;
                if (a.vec && left >= 4) {
                    __stcs(reinterpret_cast<uint4 *>(o), wv);
                } else {
                    const uint32_t e[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k < left)
                            __stcs(reinterpret_cast<unsigned int *>(o + 4 * k), e[k]);
                }
            } else {
                const float4 el = *reinterpret_cast<const float4 *>(stg + cell * 16);
                if (left > 0)
                    __stcs(reinterpret_cast<float4 *>(o), el);
            }
        }
        optr += (CI8 ? 4 : 16) * RS;
        left -= RS;
    }
}

template <int M, int TI, bool CI8>
cudaError_t launch(const PfbArgs &a, unsigned gx, unsigned gy, cudaStream_t s) {
    constexpr int smem = Shape<M, TI>::template SMEM<CI8>;
    static unsigned long long attr_set = 0;  // per device
    if (smem > 48 * 1024) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess)
            return e;
        if (dev >= 64 || !((attr_set >> dev) & 1ull)) {
            e = cudaFuncSetAttribute(pfb_kernel<M, TI, CI8>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess)
                return e;
            if (dev < 64)
                attr_set |= 1ull << dev;
        }
    }
    pfb_kernel<M, TI, CI8><<<dim3(gx, gy), threads_of(M), smem, s>>>(a);
    return cudaGetLastError();
}

template <int M, bool CI8>
cudaError_t launch_t(int ti, const PfbArgs &a, unsigned gx, unsigned gy, cudaStream_t s) {
    switch (ti) {
    case 2: return launch<M, 2, CI8>(a, gx, gy, s);
    case 4: return launch<M, 4, CI8>(a, gx, gy, s);
    case 8: return launch<M, 8, CI8>(a, gx, gy, s);
    case 16: return launch<M, 16, CI8>(a, gx, gy, s);
    }
    return cudaErrorInvalidValue;
}

template <int M>
cudaError_t launch_m(int ti, const PfbArgs &a, unsigned gx, unsigned gy, cudaStream_t s) {
    return a.ci8 ? launch_t<M, true>(ti, a, gx, gy, s) : launch_t<M, false>(ti, a, gx, gy, s);
}

int taps_instantiated(int T) { return T <= 2 ? 2 : T <= 4 ? 4 : T <= 8 ? 8 : 16; }

// Spectra per round of the kernel for (M, T): NSEG * RS.
int64_t spectra_per_round(int M, int T) {
    const int ti = taps_instantiated(T);
    return (int64_t)(threads_of(M) / M) * (ti > 8 ? ti : 8);
}

bool m_ok(int M) { return M == 16 || M == 32 || M == 64 || M == 128 || M == 256; }

}  // namespace

extern "C" int64_t dd_channelise_nspec(int64_t nraw, int nchan_sub, int ntaps) {
    if (nraw < 0 || !m_ok(nchan_sub) || ntaps < 1 || ntaps > 16)
        return -1;
    const int64_t nblk = nraw / nchan_sub;
    return nblk >= ntaps ? nblk - ntaps + 1 : 0;
}

extern "C" dd_status dd_pfb_prototype(int nchan_sub, int ntaps, float *h) {
    using dd::fail;
    if (nchan_sub < 1 || ntaps < 1 || (int64_t)nchan_sub * ntaps < 2 || !h)
        return fail(DD_ERR_INVALID, "pfb_prototype: need nchan_sub >= 1, ntaps >= 1, "
                                    "nchan_sub*ntaps >= 2 and a host array");
    const int64_t L = (int64_t)nchan_sub * ntaps;
    const double pi = 3.14159265358979323846;
    for (int64_t m = 0; m < L; ++m) {
        // sinc with its first zeros one channel spacing from the centre, times
        // a Hamming window over the L taps.
        const double x = ((double)m - (double)(L - 1) / 2.0) / (double)nchan_sub;
        const double sinc = x == 0.0 ? 1.0 : std::sin(pi * x) / (pi * x);
        const double w = 0.54 - 0.46 * std::cos(2.0 * pi * (double)m / (double)(L - 1));
        h[m] = (float)(sinc * w);
    }
    return DD_OK;
}

extern "C" dd_status dd_channelise(const void *volts, int64_t volts_pitch, int nsub,
                                   int64_t nraw, int nchan_sub, int ntaps, const float *coeffs,
                                   int out_kind, float scale, void *out, int64_t out_pitch,
                                   void *stream) {
    dd::Range nvtx_range("dd_channelise");
    using dd::fail;
    const int M = nchan_sub;
    if (!m_ok(M) || ntaps < 1 || ntaps > 16 || nsub < 1 || nsub > 65535 || nraw < 0)
        return fail(DD_ERR_INVALID, "channelise: need nchan_sub in {16,32,64,128,256}, "
                                    "1 <= ntaps <= 16, 1 <= nsub <= 65535, nraw >= 0");
    if (out_kind != DD_PFB_CF32 && out_kind != DD_PFB_CI8)
        return fail(DD_ERR_INVALID, "channelise: out_kind must be DD_PFB_CF32 or DD_PFB_CI8");
    if (out_kind == DD_PFB_CI8 && !(std::isfinite(scale) && scale > 0.0f))
        return fail(DD_ERR_INVALID, "channelise: scale must be finite and > 0");
    const int64_t elem = out_kind == DD_PFB_CI8 ? 4 : 16;
    const int64_t nspec = dd_channelise_nspec(nraw, M, ntaps);
    if (volts_pitch < 4 * nraw || volts_pitch % 4 != 0 || out_pitch < elem * nspec ||
        out_pitch % elem != 0)
        return fail(DD_ERR_INVALID, "channelise: volts_pitch >= 4*nraw (multiple of 4), "
                                    "out_pitch >= element*nspec (multiple of the element: "
                                    "4 bytes int8, 16 bytes FP32)");
    if (nspec == 0)
        return DD_OK;
    if (!volts || !out || !coeffs || ((uintptr_t)volts & 3u) || ((uintptr_t)coeffs & 3u) ||
        ((uintptr_t)out & (uintptr_t)(elem - 1)))
        return fail(DD_ERR_INVALID, "channelise: NULL or misaligned volts/coeffs/out pointer");
    const int64_t per_round = spectra_per_round(M, ntaps);
    // Rounds per CTA: full waves of equal CTAs, each of at most kMaxRounds (a
    // segment's first T - 1 blocks are read again for every CTA).  With 32
    // rounds always, one subband of 16 channels and 65536 spectra ran 32 CTAs
    // in 37 us; 2 rounds each (512 CTAs) take 5.8 us.
    int64_t nr = (nspec + per_round - 1) / per_round;
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dd::sm_count(dev) > 0) {
        const int64_t slots = (int64_t)dd::sm_count(dev) *
                              ctas_of(M, taps_instantiated(ntaps), out_kind == DD_PFB_CI8);
        const int64_t waves = (nr * nsub + slots * kMaxRounds - 1) / (slots * kMaxRounds);
        nr = (nr * nsub + slots * waves - 1) / (slots * waves);
    }
    if (nr > kMaxRounds)
        nr = kMaxRounds;
    const int64_t per_cta = per_round * nr;
    const int64_t gx = (nspec + per_cta - 1) / per_cta;
    if (gx > 0x7fffffffLL)
        return fail(DD_ERR_INVALID, "channelise: too many spectra");
    PfbArgs a;
    a.in = static_cast<const uint8_t *>(volts);
    a.in_pitch = volts_pitch;
    a.nblk = nraw / M;
    a.nspec = nspec;
    a.h = coeffs;
    a.T = ntaps;
    a.nr = (int)nr;
    a.scale = scale;
    a.ci8 = out_kind == DD_PFB_CI8;
    a.vec = ((uintptr_t)out % 16 == 0) && (out_pitch % 16 == 0);
    a.out = static_cast<uint8_t *>(out);
    a.out_pitch = out_pitch;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int ti = taps_instantiated(ntaps);
    cudaError_t e = cudaErrorInvalidValue;
    switch (M) {
    case 16: e = launch_m<16>(ti, a, (unsigned)gx, (unsigned)nsub, s); break;
    case 32: e = launch_m<32>(ti, a, (unsigned)gx, (unsigned)nsub, s); break;
    case 64: e = launch_m<64>(ti, a, (unsigned)gx, (unsigned)nsub, s); break;
    case 128: e = launch_m<128>(ti, a, (unsigned)gx, (unsigned)nsub, s); break;
    case 256: e = launch_m<256>(ti, a, (unsigned)gx, (unsigned)nsub, s); break;
    }
    if (e != cudaSuccess)
        return fail(DD_ERR_CUDA, std::string("channelise launch: ") + cudaGetErrorString(e));
    dd::count_launch(1);
    return DD_OK;
}
