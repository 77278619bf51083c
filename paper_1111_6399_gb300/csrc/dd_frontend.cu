// Front end (dd_frontend): dual-polarisation voltages -> the uint8 filterbank
// rows dd_execute reads.  The paper's pipeline generates Stokes parameters,
// excises RFI and integrates before the dispersion search (Sec. 1) without
// giving formulas; the library's reading, step by step:
//
//   Stokes I of a raw sample (Xre, Xim, Yre, Yim as int8) = Xre^2 + Xim^2 +
//   Yre^2 + Yim^2 (one dp4a of the sample's word with itself);
//   P[c][t] = sum over raw samples t*nint .. t*nint + nint - 1 (exact);
//   RFI excision by niter passes of sigma clipping: pass i takes the exact
//   count, sum P and sum P^2 over the samples the previous pass kept (all of
//   them for the first), then mean, std and thr = floor(mean + k*std) in
//   FP64; the next pass keeps P <= thr;
//   with the last pass's mean, std and thr: P > thr becomes code 128, else
//   code = clamp(rint(128 + ((float)P - (float)mean) * (float)(16/std)), 0,
//   255) in FP32, one IEEE operation at a time; std == 0 gives 128.
//
// Main path, fused_kernel: one thread-block cluster per channel, its cs CTAs
// (1, 2, 4 or 8) each owning m consecutive output samples.  A CTA streams its
// voltages once (each warp reads 32 samples' bytes in coalesced steps, the
// words of one sample summed over neighbouring lanes), keeps P in shared
// memory, and every clipping pass sums its own P; each CTA reads the partial
// sums of its cluster (distributed shared memory, hardware cluster barriers)
// and derives the statistics.  HBM traffic is the compulsory minimum: 4*nint bytes
// of voltages per output sample in, 1 byte of code out.
//
// Fallback for rows whose P does not fit a cluster's shared memory: P in the
// caller's work array and niter + 1 launches -- power_kernel (P and pass 1's
// sums), clip_kernel for passes 2..niter and quantize_kernel, each block
// deriving its channel's statistics from the exact sums itself.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <string>

#include "dd_internal.h"

namespace {

constexpr int kThreads = 256;
constexpr int64_t kFallbackBlocks = 152 * 8 * 4;

struct Acc {  // exact per-channel sums of one clipping pass
    unsigned long long cnt, s1, s2;
};

struct Stats {
    double mean, sd;
    long long thr;
};

// The FP64 operations of the definition, in order (no contraction).
__device__ __forceinline__ Stats stats_of(const Acc &a, double k) {
    Stats s;
    double var = 0.0;
    s.mean = 0.0;
    if (a.cnt > 0) {
        const double dc = __ull2double_rn(a.cnt);
        s.mean = __ddiv_rn(__ull2double_rn(a.s1), dc);
        var = __dsub_rn(__ddiv_rn(__ull2double_rn(a.s2), dc), __dmul_rn(s.mean, s.mean));
    }
    if (var < 0.0)
        var = 0.0;
    s.sd = __dsqrt_rn(var);
    s.thr = (long long)floor(__dadd_rn(s.mean, __dmul_rn(k, s.sd)));
    return s;
}

// Block sums of (cnt, s1, s2), then one atomic triple per block.  P <= 2^22 and
// a row has at most 2^19 samples, so the P^2 sum stays below 2^64.
__device__ __forceinline__ void block_accumulate(unsigned long long cnt, unsigned long long s1,
                                                 unsigned long long s2, Acc *dst) {
    __shared__ unsigned long long red[3][kThreads / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = cnt;
        red[1][threadIdx.x >> 5] = s1;
        red[2][threadIdx.x >> 5] = s2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        cnt = s1 = s2 = 0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            cnt += red[0][w];
            s1 += red[1][w];
            s2 += red[2][w];
        }
        if (cnt != 0) {
            atomicAdd(&dst->cnt, cnt);
            atomicAdd(&dst->s1, s1);
            atomicAdd(&dst->s2, s2);
        }
    }
}

template <bool VEC>
__global__ void __launch_bounds__(kThreads) power_kernel(const uint8_t *__restrict__ volts,
                                                         int64_t pitch, int64_t n, int64_t prow,
                                                         int nint, uint32_t *__restrict__ p_out,
                                                         Acc *acc) {
    const int c = blockIdx.y;
    unsigned long long cnt = 0, s1 = 0, s2 = 0;
    const int64_t step = (int64_t)gridDim.x * kThreads;
#pragma unroll 4
    for (int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x; t < n; t += step) {
        const uint8_t *src = volts + (int64_t)c * pitch + 4 * t * nint;
        uint32_t p = 0;
        if (VEC) {
            for (int j = 0; j < nint; j += 4) {
                const uint4 v = *reinterpret_cast<const uint4 *>(src + 4 * j);
                p += (uint32_t)(__dp4a((int)v.x, (int)v.x, 0) + __dp4a((int)v.y, (int)v.y, 0) +
                                __dp4a((int)v.z, (int)v.z, 0) + __dp4a((int)v.w, (int)v.w, 0));
            }
        } else {
            for (int j = 0; j < nint; ++j) {
                const int v = *reinterpret_cast<const int *>(src + 4 * j);
                p += (uint32_t)__dp4a(v, v, 0);
            }
        }
        p_out[(int64_t)c * prow + t] = p;
        cnt += 1;
        s1 += p;
        s2 += (unsigned long long)p * p;
    }
    block_accumulate(cnt, s1, s2, &acc[c]);
}

// One clipping pass: sums over the samples at or below the previous pass's
// threshold.
__global__ void __launch_bounds__(kThreads) clip_kernel(const uint32_t *__restrict__ p_in,
                                                        int64_t n, int64_t prow, double k,
                                                        const Acc *prev, Acc *next) {
    const int c = blockIdx.y;
    __shared__ long long sthr;
    if (threadIdx.x == 0)
        sthr = stats_of(prev[c], k).thr;
    __syncthreads();
    const long long thr = sthr;
    const int64_t step = 4 * (int64_t)gridDim.x * kThreads;
    unsigned long long cnt = 0, s1 = 0, s2 = 0;
#pragma unroll 4
    for (int64_t t = 4 * ((int64_t)blockIdx.x * kThreads + threadIdx.x); t < n; t += step) {
        const uint4 q = *reinterpret_cast<const uint4 *>(p_in + (int64_t)c * prow + t);
        const uint32_t v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (t + i < n && (long long)v[i] <= thr) {
                cnt += 1;
                s1 += v[i];
                s2 += (unsigned long long)v[i] * v[i];
            }
        }
    }
    block_accumulate(cnt, s1, s2, &next[c]);
}

// Threshold as a 32-bit value (P is at most 2^22): -1 keeps nothing.
__device__ __forceinline__ int thr32(long long thr) {
    return thr < 0 ? -1 : thr > 0x7fffffff ? 0x7fffffff : (int)thr;
}

// p + 2^23 (exact) less 2^23 is (float)p, and v + 2^23 rounds v in [0, 255] to
// the nearest integer, ties to even, in its low byte: conversions and rintf
// would go through a unit of a quarter of the rate.  A NaN gives code 0.
__device__ __forceinline__ uint32_t code_of(uint32_t p, int thr, float m, float s, bool flat) {
    const float f = __fsub_rn(__uint_as_float(p | 0x4b000000u), 8388608.0f);
    const float v = __fadd_rn(128.0f, __fmul_rn(__fsub_rn(f, m), s));
    const uint32_t q =
        __float_as_uint(__fadd_rn(fminf(fmaxf(v, 0.0f), 255.0f), 8388608.0f)) & 255u;
    return flat || (int)p > thr ? 128u : q;
}

__device__ __forceinline__ uint32_t codes_of(uint4 p, int thr, float m, float s, bool flat) {
    return code_of(p.x, thr, m, s, flat) | code_of(p.y, thr, m, s, flat) << 8 |
           code_of(p.z, thr, m, s, flat) << 16 | code_of(p.w, thr, m, s, flat) << 24;
}

__global__ void __launch_bounds__(kThreads) quantize_kernel(const uint32_t *__restrict__ p_in,
                                                            int64_t n, int64_t prow, double k,
                                                            const Acc *last, uint8_t *out,
                                                            int64_t out_pitch, double *mean,
                                                            double *sd) {
    const int c = blockIdx.y;
    __shared__ float sm, ss;
    __shared__ long long sthr;
    __shared__ int sflat;
    if (threadIdx.x == 0) {
        const Stats st = stats_of(last[c], k);
        sm = (float)st.mean;
        sflat = st.sd > 0.0 ? 0 : 1;
        ss = st.sd > 0.0 ? (float)__ddiv_rn(16.0, st.sd) : 0.0f;
        sthr = st.thr;
        if (blockIdx.x == 0) {
            mean[c] = st.mean;
            sd[c] = st.sd;
        }
    }
    __syncthreads();
    const float m = sm, s = ss;
    const int thr = thr32(sthr);
    const bool flat = sflat != 0;
    const int64_t step = 4 * (int64_t)gridDim.x * kThreads;
#pragma unroll 4
    for (int64_t t = 4 * ((int64_t)blockIdx.x * kThreads + threadIdx.x); t < n; t += step) {
        const uint4 q = *reinterpret_cast<const uint4 *>(p_in + (int64_t)c * prow + t);
        uint8_t *dst = out + (int64_t)c * out_pitch + t;
        if (t + 4 <= n) {
            *reinterpret_cast<uint32_t *>(dst) = codes_of(q, thr, m, s, flat);
        } else {
            const uint32_t v[4] = {q.x, q.y, q.z, q.w};
            for (int i = 0; t + i < n; ++i)
                dst[i] = (uint8_t)code_of(v[i], thr, m, s, flat);
        }
    }
}

// ---------------------------------------------------------------------------
// Fused cluster kernel.
// ---------------------------------------------------------------------------

constexpr int kFusedThreads = 512;
constexpr int kFusedWarps = kFusedThreads / 32;
constexpr int64_t kFusedSmemTarget = 100 * 1024;  // P bytes per CTA aimed for (2 CTAs per SM)
constexpr int64_t kFusedSmemMax = 200 * 1024;     // P bytes per CTA allowed
constexpr int kMaxCluster = 8;

struct Params {
    int thr;
    float m, s;
    int flat;
};

// Block sums of (cnt, s1, s2) for kFusedThreads threads, left in red[][0] for
// thread 0.  Callers separate uses by a barrier.
__device__ __forceinline__ void fused_block_sum(unsigned long long v[3],
                                                unsigned long long (*red)[kFusedWarps]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int i = 0; i < 3; ++i)
            v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    }
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int i = 0; i < 3; ++i)
            red[i][threadIdx.x >> 5] = v[i];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            unsigned long long a = 0;
#pragma unroll
            for (int w = 0; w < kFusedWarps; ++w)
                a += red[i][w];
            v[i] = a;
        }
    }
}

__device__ __forceinline__ uint32_t fused_power_word(uint4 v) {
    return (uint32_t)__dp4a((int)v.x, (int)v.x,
                            __dp4a((int)v.y, (int)v.y,
                                   __dp4a((int)v.z, (int)v.z, __dp4a((int)v.w, (int)v.w, 0))));
}

// Values i of the Q lanes of a group summed over the group; lane l leaves with
// value l % Q (Q - 1 shuffles for Q sums).
template <int Q>
__device__ __forceinline__ uint32_t reduce_scatter(uint32_t (&a)[Q], int lane) {
#pragma unroll
    for (int h = Q / 2; h > 0; h >>= 1) {
        const bool upper = (lane & h) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const uint32_t keep = upper ? a[i + h] : a[i], send = upper ? a[i] : a[i + h];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
    }
    return a[0];
}

// NINT raw samples per output sample; V16: rows on 16 bytes.
//
// HBM-bound at 16 raw samples per output as far as the passes over P overlap
// the other CTA's loads, so those are kept short: 16-byte reads of P, 32-bit
// counts and sums (a thread has at most 100 values of 2^22), codes without
// conversion instructions, and one cluster barrier per pass (every CTA reads
// all partial sums and derives the statistics itself).  256 channels x
// 2362048 raw samples, nint 16, 3 passes: 436 us (363 us of HBM traffic; 450
// with scalar reads and 64-bit sums); 200 x 1048576, nint 64, 5 passes: 145
// (222).  Loads are whole warps of consecutive words, and the words of an
// output sample meet by a reduce-scatter, one output per lane: 77 x 51434,
// nint 32, rows off 16 bytes: 8.7 us (31 with a thread per output); nint 1,
// 135 x 183608: 84 (196).
template <int NINT, bool V16>
__global__ void __launch_bounds__(kFusedThreads, 2) fused_kernel(
    const uint8_t *__restrict__ volts, int64_t pitch, int64_t n, int m, double k,
    int niter, uint8_t *__restrict__ out, int64_t out_pitch, double *mean_out, double *sd_out) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned rank = cluster.block_rank();
    const unsigned cs = cluster.num_blocks();
    const int c = blockIdx.x / cs;
    extern __shared__ uint4 fused_smem[];
    uint32_t *P = reinterpret_cast<uint32_t *>(fused_smem);
    __shared__ unsigned long long red[3][kFusedWarps];
    __shared__ unsigned long long part[2][3];  // of even and odd passes
    __shared__ Params prm;

    const int64_t t0 = (int64_t)rank * m;
    const int len = (int)(n - t0 < 0 ? 0 : (n - t0 < m ? n - t0 : m));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long acc[3] = {0, 0, 0};

    // Pass 1: P = integrated Stokes I, kept in shared memory.
    if constexpr (V16 && NINT >= 4) {
        constexpr int Q = NINT / 4;  // 16-byte words per output sample
        const uint4 *row = reinterpret_cast<const uint4 *>(volts + (int64_t)c * pitch) + t0 * Q;
        constexpr int U = Q >= 8 ? 1 : 8 / Q;  // groups of 32 samples in flight per warp
        constexpr int L = Q > 8 ? 8 : Q;       // words of a group in flight
        for (int g0 = warp * 32; g0 < len; g0 += kFusedWarps * 32 * U) {
            uint32_t a[U][Q];
#pragma unroll
            for (int j0 = 0; j0 < Q; j0 += L) {
                uint4 v[U][L];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int g = g0 + u * kFusedWarps * 32;
                    const uint4 *src = row + (int64_t)g * Q + lane + 32 * j0;
                    if (g + 32 <= len) {
#pragma unroll
                        for (int j = 0; j < L; ++j)
                            v[u][j] = __ldcs(src + 32 * j);
                    } else {
#pragma unroll
                        for (int j = 0; j < L; ++j)
                            v[u][j] = g + (lane + 32 * (j0 + j)) / Q < len ? __ldcs(src + 32 * j)
                                                                           : make_uint4(0, 0, 0, 0);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int j = 0; j < L; ++j)
                        a[u][j0 + j] = fused_power_word(v[u][j]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t p = reduce_scatter<Q>(a[u], lane);
                const int sl = g0 + u * kFusedWarps * 32 + 32 / Q * (lane % Q) + lane / Q;
                if (sl < len) {
                    P[sl] = p;
                    acc[1] += p;
                    acc[2] += (unsigned long long)p * p;
                }
            }
        }
    } else if constexpr (V16) {
        constexpr int W = 4 / NINT;  // output samples of a 16-byte word
        const uint4 *row = reinterpret_cast<const uint4 *>(volts + (int64_t)c * pitch) + t0 / W;
        constexpr int U = 4;
        const int words = (len + W - 1) / W;
        // A row may end within its last word: its samples one by one.
        const int whole = len / W;
        for (int w0 = tid; w0 < words; w0 += U * kFusedThreads) {
            uint4 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int w = w0 + u * kFusedThreads;
                if (w < whole) {
                    v[u] = __ldcs(row + w);
                } else {
                    const int *src = reinterpret_cast<const int *>(row + w);
                    const int in = (len - w * W) * NINT;  // raw samples (< 4, or none)
                    v[u].x = in > 0 ? (uint32_t)__ldcs(src) : 0u;
                    v[u].y = in > 1 ? (uint32_t)__ldcs(src + 1) : 0u;
                    v[u].z = in > 2 ? (uint32_t)__ldcs(src + 2) : 0u;
                    v[u].w = 0u;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int w = w0 + u * kFusedThreads;
                if (w >= words)
                    continue;
                const uint32_t x[4] = {(uint32_t)__dp4a((int)v[u].x, (int)v[u].x, 0),
                                       (uint32_t)__dp4a((int)v[u].y, (int)v[u].y, 0),
                                       (uint32_t)__dp4a((int)v[u].z, (int)v[u].z, 0),
                                       (uint32_t)__dp4a((int)v[u].w, (int)v[u].w, 0)};
                // Samples past the end are 0: they add nothing (P is a whole
                // number of words).
                if constexpr (W == 4) {
                    *reinterpret_cast<uint4 *>(P + 4 * w) = make_uint4(x[0], x[1], x[2], x[3]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        acc[1] += x[i];
                        acc[2] += (unsigned long long)x[i] * x[i];
                    }
                } else {
                    const uint32_t p0 = x[0] + x[1], p1 = x[2] + x[3];
                    *reinterpret_cast<uint2 *>(P + 2 * w) = make_uint2(p0, p1);
                    acc[1] += p0;
                    acc[1] += p1;
                    acc[2] += (unsigned long long)p0 * p0;
                    acc[2] += (unsigned long long)p1 * p1;
                }
            }
        }
    } else {
        // As for 16-byte words, with raw samples: lane l reads words l + 32 j.
        const int *row =
            reinterpret_cast<const int *>(volts + (int64_t)c * pitch) + t0 * NINT;
        constexpr int A = NINT > 32 ? 32 : NINT;   // sums to scatter
        constexpr int U = NINT >= 16 ? 1 : 16 / NINT;
        constexpr int L = NINT > 16 ? 16 : NINT;   // loads of a group in flight
        for (int g0 = warp * 32; g0 < len; g0 += kFusedWarps * 32 * U) {
            uint32_t a[U][A];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int i = 0; i < A; ++i)
                    a[u][i] = 0;
#pragma unroll
            for (int j0 = 0; j0 < NINT; j0 += L) {
                int v[U][L];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int g = g0 + u * kFusedWarps * 32;
                    const int *src = row + (int64_t)g * NINT + lane + 32 * j0;
#pragma unroll
                    for (int j = 0; j < L; ++j)
                        v[u][j] = g + 32 <= len || g + (lane + 32 * (j0 + j)) / NINT < len
                                      ? __ldcs(src + 32 * j)
                                      : 0;
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int j = 0; j < L; ++j)
                        a[u][(j0 + j) / (NINT / A)] = (uint32_t)__dp4a(
                            v[u][j], v[u][j], (int)a[u][(j0 + j) / (NINT / A)]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t p = reduce_scatter<A>(a[u], lane);
                const int sl = g0 + u * kFusedWarps * 32 + 32 / A * (lane % A) + lane / A;
                if (sl < len) {
                    P[sl] = p;
                    acc[1] += p;
                    acc[2] += (unsigned long long)p * p;
                }
            }
        }
    }
    acc[0] = tid == 0 ? (unsigned long long)len : 0ull;

    int thr = 0;
    for (int it = 0; it < niter; ++it) {
        if (it > 0) {
            uint32_t cnt = 0, sum = 0;
            unsigned long long sq = 0;
            auto take = [&](uint32_t p) {
                const bool kept = (int)p <= thr;
                const uint32_t q = kept ? p : 0u;
                cnt += kept ? 1u : 0u;
                sum += q;
                sq += (unsigned long long)q * q;
            };
            for (int sl = 4 * tid; sl < len; sl += 4 * kFusedThreads) {
                if (sl + 4 <= len) {
                    const uint4 p = *reinterpret_cast<const uint4 *>(P + sl);
                    take(p.x);
                    take(p.y);
                    take(p.z);
                    take(p.w);
                } else {
                    for (int i = sl; i < len; ++i)
                        take(P[i]);
                }
            }
            acc[0] = cnt;
            acc[1] = sum;
            acc[2] = sq;
        }
        fused_block_sum(acc, red);  // P is written, too, for every thread
        if (tid == 0) {
            part[it & 1][0] = acc[0];
            part[it & 1][1] = acc[1];
            part[it & 1][2] = acc[2];
        }
        cluster.sync();  // every rank's part is written, and that of two passes ago read
        if (warp == 0) {
            unsigned long long v[3] = {0, 0, 0};
            if ((unsigned)lane < cs) {
                const unsigned long long *rp = cluster.map_shared_rank(part[it & 1], lane);
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    v[i] = rp[i];
            }
#pragma unroll
            for (int o = kMaxCluster / 2; o > 0; o >>= 1)
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
            if (lane == 0) {
                const Acc a = {v[0], v[1], v[2]};
                const Stats st = stats_of(a, k);
                prm.thr = thr32(st.thr);
                if (it == niter - 1) {
                    prm.flat = st.sd > 0.0 ? 0 : 1;
                    prm.m = (float)st.mean;
                    prm.s = st.sd > 0.0 ? (float)__ddiv_rn(16.0, st.sd) : 0.0f;
                    if (rank == 0) {
                        mean_out[c] = st.mean;
                        sd_out[c] = st.sd;
                    }
                }
            }
        }
        __syncthreads();
        thr = prm.thr;
    }
    // A CTA keeps its shared memory until every rank has read its part.
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    const float mean = prm.m, scale = prm.s;
    const bool flat = prm.flat != 0;
    uint8_t *dst = out + (int64_t)c * out_pitch + t0;
    for (int sl = 4 * tid; sl < len; sl += 4 * kFusedThreads) {
        if (sl + 4 <= len) {
            const uint4 q = *reinterpret_cast<const uint4 *>(P + sl);
            *reinterpret_cast<uint32_t *>(dst + sl) = codes_of(q, thr, mean, scale, flat);
        } else {
            for (int i = sl; i < len; ++i)
                dst[i] = (uint8_t)code_of(P[i], thr, mean, scale, flat);
        }
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Samples per CTA for a cluster of cs CTAs: a multiple of 32 (so every CTA's
// first sample starts a warp group and a 4-byte output word).
int64_t fused_m(int64_t n, int cs) { return ((n + cs - 1) / cs + 31) / 32 * 32; }

template <int NINT, bool V16>
cudaError_t launch_fused_q(int cs, int64_t m, const uint8_t *v, int64_t pitch, int64_t n,
                           int nchan, double k, int niter, uint8_t *out,
                           int64_t out_pitch, double *mean, double *sd, cudaStream_t s,
                           bool *fits) {
    static unsigned long long attr_set = 0;  // per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev >= 64 || !((attr_set >> dev) & 1ull)) {
        e = cudaFuncSetAttribute(fused_kernel<NINT, V16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kFusedSmemMax);
        if (e != cudaSuccess)
            return e;
        if (dev < 64)
            attr_set |= 1ull << dev;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nchan * cs));
    cfg.blockDim = dim3(kFusedThreads);
    cfg.dynamicSmemBytes = (size_t)(4 * m);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    e = cudaOccupancyMaxActiveClusters(&clusters, fused_kernel<NINT, V16>, &cfg);
    if (e != cudaSuccess || clusters < 1) {
        (void)cudaGetLastError();  // not an error of the call: leave it to the fallback path
        *fits = false;
        return cudaSuccess;
    }
    *fits = true;
    return cudaLaunchKernelEx(&cfg, fused_kernel<NINT, V16>, v, pitch, n, (int)m, k, niter, out,
                              out_pitch, mean, sd);
}

bool frontend_shape_ok(int nchan, int64_t nsamp_raw, int nint, int niter) {
    return nchan >= 1 && nchan <= 65535 && nsamp_raw >= 0 && nint >= 1 && nint <= 64 &&
           (nint & (nint - 1)) == 0 && niter >= 1 && niter <= 8 &&
           nsamp_raw / nint <= (1LL << 19);
}

// P rows hold a whole number of 16-byte groups.
int64_t p_row(int64_t n) { return (n + 3) / 4 * 4; }

}  // namespace

extern "C" int64_t dd_frontend_work_bytes(int nchan, int64_t nsamp_raw, int nint, int niter) {
    if (!frontend_shape_ok(nchan, nsamp_raw, nint, niter))
        return -1;
    return 4 * (int64_t)nchan * p_row(nsamp_raw / nint) + (int64_t)sizeof(Acc) * niter * nchan;
}

extern "C" dd_status dd_frontend(const void *volts, int64_t volts_pitch, int nchan,
                                 int64_t nsamp_raw, int nint, double k_clip, int niter,
                                 uint8_t *out, int64_t out_pitch, void *work, int64_t work_bytes,
                                 double *mean, double *std_out, void *stream) {
    dd::Range nvtx_range("dd_frontend");
    using dd::fail;
    if (!frontend_shape_ok(nchan, nsamp_raw, nint, niter))
        return fail(DD_ERR_INVALID, "need 1 <= nchan <= 65535, nsamp_raw >= 0, nint a power of "
                                    "two <= 64, 1 <= niter <= 8, nsamp_raw/nint <= 2^19");
    const int64_t n = nsamp_raw / nint;
    if (volts_pitch < 4 * nsamp_raw || volts_pitch % 4 != 0 || out_pitch < n || out_pitch % 16)
        return fail(DD_ERR_INVALID, "volts_pitch >= 4*nsamp_raw (multiple of 4); out_pitch >= "
                                    "nsamp_raw/nint (multiple of 16)");
    // The bound keeps floor(mean + k_clip*std) inside int64 for any P.
    if (!(k_clip > 0.0 && k_clip <= 1e9))
        return fail(DD_ERR_INVALID, "k_clip must be in (0, 1e9]");
    if (!mean || !std_out || ((uintptr_t)mean & 7u) || ((uintptr_t)std_out & 7u))
        return fail(DD_ERR_INVALID, "NULL or misaligned mean/std pointer");
    if (n > 0 && (!volts || !out || !work || ((uintptr_t)volts & 3u) || ((uintptr_t)out & 15u) ||
                  ((uintptr_t)work & 15u)))
        return fail(DD_ERR_INVALID, "NULL or misaligned volts/out/work pointer");
    if (n > 0 && work_bytes < dd_frontend_work_bytes(nchan, nsamp_raw, nint, niter))
        return fail(DD_ERR_INVALID, "work is smaller than dd_frontend_work_bytes");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    if (n == 0) {  // no output samples: mean and std are 0
        e = cudaMemsetAsync(mean, 0, sizeof(double) * nchan, s);
        if (e == cudaSuccess)
            e = cudaMemsetAsync(std_out, 0, sizeof(double) * nchan, s);
        if (e != cudaSuccess)
            return fail(DD_ERR_CUDA, std::string("frontend memset: ") + cudaGetErrorString(e));
        return DD_OK;
    }
    const uint8_t *v = static_cast<const uint8_t *>(volts);
    const bool rows16 = ((uintptr_t)volts & 15u) == 0 && volts_pitch % 16 == 0;
    const bool vec = nint % 4 == 0 && rows16;
    int cs = 1;
    while (cs < kMaxCluster && 4 * fused_m(n, cs) > kFusedSmemTarget)
        cs *= 2;
    if (4 * fused_m(n, cs) <= kFusedSmemMax) {
        const int64_t m = fused_m(n, cs);
        bool fits = false;
        switch (nint) {
#define DD_FE_CASE(NN)                                                                       \
    case NN:                                                                                 \
        e = rows16 ? launch_fused_q<NN, true>(cs, m, v, volts_pitch, n, nchan, k_clip, niter,\
                                              out, out_pitch, mean, std_out, s, &fits)       \
                   : launch_fused_q<NN, false>(cs, m, v, volts_pitch, n, nchan, k_clip,      \
                                               niter, out, out_pitch, mean, std_out, s,      \
                                               &fits);                                       \
        break;
            DD_FE_CASE(1)
            DD_FE_CASE(2)
            DD_FE_CASE(4)
            DD_FE_CASE(8)
            DD_FE_CASE(16)
            DD_FE_CASE(32)
            DD_FE_CASE(64)
#undef DD_FE_CASE
        default:
            return fail(DD_ERR_INVALID, "frontend: no kernel for this nint");
        }
        if (e != cudaSuccess)
            return fail(DD_ERR_CUDA, std::string("frontend launch: ") + cudaGetErrorString(e));
        if (fits) {
            dd::count_launch(1);
            return DD_OK;
        }
    }
    const int64_t prow = p_row(n);
    auto *p = static_cast<uint32_t *>(work);
    auto *acc = reinterpret_cast<Acc *>(static_cast<uint8_t *>(work) + 4 * nchan * prow);
    e = cudaMemsetAsync(acc, 0, sizeof(Acc) * niter * nchan, s);
    if (e != cudaSuccess)
        return fail(DD_ERR_CUDA, std::string("frontend memset: ") + cudaGetErrorString(e));
    // A block ends in three atomics on its channel's sums or begins with the
    // statistics in FP64, so there are no more blocks than fill the device a
    // few times (a block per 256 or 1024 samples took 2.3 ms for 300 channels
    // x 524288 samples against 1.0 ms).
    auto blocks = [&](int64_t per_block) {
        return dim3((unsigned)std::min((n + per_block - 1) / per_block,
                                       (int64_t)(kFallbackBlocks + nchan - 1) / nchan),
                    (unsigned)nchan);
    };
    const dim3 g1 = blocks(kThreads), gc = blocks(4 * kThreads);
    // 16-byte loads need 16-byte aligned rows and whole groups of 4 samples.
    if (vec)
        power_kernel<true><<<g1, kThreads, 0, s>>>(v, volts_pitch, n, prow, nint, p, acc);
    else
        power_kernel<false><<<g1, kThreads, 0, s>>>(v, volts_pitch, n, prow, nint, p, acc);
    e = cudaGetLastError();
    for (int it = 1; it < niter && e == cudaSuccess; ++it) {
        clip_kernel<<<gc, kThreads, 0, s>>>(p, n, prow, k_clip, acc + (int64_t)(it - 1) * nchan,
                                            acc + (int64_t)it * nchan);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        quantize_kernel<<<gc, kThreads, 0, s>>>(p, n, prow, k_clip,
                                                acc + (int64_t)(niter - 1) * nchan, out,
                                                out_pitch, mean, std_out);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess)
        return fail(DD_ERR_CUDA, std::string("frontend launch: ") + cudaGetErrorString(e));
    dd::count_launch(niter + 1);
    return DD_OK;
}
