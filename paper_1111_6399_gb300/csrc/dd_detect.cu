// Detection on the (DM,t) plane (dd_detect): per DM row, the mean and
// standard deviation of the row and, for boxcar widths w = 1, 2, 4, ...,
// 2^(nlevels-1) (at most 256), the highest boxcar sum and the first sample
// where it starts, turned into S/N = (B - w*mean) / (std*sqrt(w)).
//
// Sec. 4 and Fig. 3 of the paper search the plane for a simulated pulse and
// recover it at its DM and time; this is that search as matched boxcar
// filters (the paper gives no formula, so this is the reading the library
// adopts).  Rows where std is 0 report S/N 0; widths longer than the row
// report t = -1 and S/N -inf.
//
// detect_tile_kernel searches the plane in tiles (below): integer-valued planes
// with exact integer boxcars and sums, FP32 planes with FP32 boxcars (summed as
// a tree) and row sums in fixed point.
// finalize_kernel then turns the sums and keys into mean, std, S/N and t with
// the same IEEE FP64 operations, in the same order, as the CPU definition.
// The output arrays double as the accumulators, so no scratch is needed.
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <type_traits>

#include "dd_detect_seg.cuh"
#include "dd_internal.h"

namespace {

using dd::detect_segment;
using dd::kMaxLevels;
using dd::ordered;
using dd::unordered;

constexpr int kWarps = 8;

// A CTA searches tile_own<INT> start positions of one row.  Warp w
// stages regions 31w .. 31w + 31, of 32 samples each, in shared memory of its
// own, and lane l holds the samples of region 31w + l (the last region is the
// next warp's first: its boxcars serve as the reach of the lane before and
// are not the warp's own).  Up to width 32 a boxcar's second half then lies
// in the same lane, w registers on, but for w values of the next lane (31
// shuffles for 32 positions in all); the width-32 boxcars go back to shared
// memory and are read 32 apart, so that the widths above are register adds
// again.  A lane takes only the highest value of each width (half an
// instruction per position); the position is looked for where the warp's
// highest reaches the row's highest so far (tiles of one row run far apart in
// time, so about one time in twelve).  Windows that pass the end of the row,
// or the staged samples, run into zeros (integers): such a sum is no more than that of
// the last whole window, which starts earlier and so wins a tie, or of the
// same window in the next tile.
//
// 1024 rows x 131072 samples: 172 us (79 us to read the plane), bound by
// instruction issue: 34 per sample, 68 % of the slots.  Segments of one warp
// each, with a shuffle per sample and width up to 32 and value and position in
// one key (detect_segment), took 335 us at 68 instructions.  The FP32 plane of
// the same size: 372 us with the final pass, 913 with detect_segment and FP64
// row sums.  There windows past the row run into -infinity instead of zeros.
constexpr int kRegionWords = 36;  // 16-byte reads of 8 lanes meet no bank twice
constexpr int kTileK = 31;        // regions of a warp
constexpr int kTileReach = 7;     // regions beyond, up to width 256
// (FP32 planes: a multiple of the warps, for the tiles that detect_segment takes.)
template <bool INT>
constexpr int tile_own = 32 * (INT ? kWarps * kTileK - kTileReach : kWarps * 30);
constexpr int kTileRows = kWarps * 32 + kTileReach;  // the last ones are zeros

__device__ __forceinline__ void stage_copy(uint32_t dst, const float *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void stage_copy4(uint32_t dst, const float *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ uint32_t max3(uint32_t a, uint32_t b, uint32_t c) {
    return __vimax3_u32(a, b, c);
}
__device__ __forceinline__ float max3(float a, float b, float c) { return fmaxf(fmaxf(a, b), c); }

template <int N, typename T>
__device__ __forceinline__ T highest(const T *z) {
    T a = z[0], b = z[1];  // two chains
#pragma unroll
    for (int k = 2; k + 3 < N; k += 4) {
        a = max3(a, z[k], z[k + 1]);
        b = max3(b, z[k + 2], z[k + 3]);
    }
#pragma unroll
    for (int k = N - (N - 2) % 4; k < N; ++k)
        a = max(a, z[k]);
    return max(a, b);
}

// Boxcars of width 2W from those of width W, a region per lane.
template <int W, typename T>
__device__ __forceinline__ void widen(T *z) {
    T r[W];
#pragma unroll
    for (int k = 0; k < W; ++k)
        r[k] = __shfl_down_sync(0xffffffffu, z[k], 1);
#pragma unroll
    for (int k = 0; k < 32; ++k)
        z[k] += k + W < 32 ? z[(k + W) & 31] : r[(k + W - 32) & (W - 1)];
}

// Values as ordered words, and back.
__device__ __forceinline__ uint32_t word_of(uint32_t v) { return v; }
__device__ __forceinline__ uint32_t word_of(float v) { return ordered(v); }
template <typename T>
__device__ __forceinline__ T value_of(uint32_t w) {
    if constexpr (std::is_same<T, float>::value)
        return unordered(w);
    else
        return w;
}
__device__ __forceinline__ uint32_t bits_of(uint32_t v) { return v; }
__device__ __forceinline__ uint32_t bits_of(float v) { return __float_as_uint(v); }

// FP32 planes: sums of x and x^2 in fixed point below the tile's largest
// magnitude (exponent field e).  x is exact in units of 2^(e - 181), x^2 is
// summed to 2^-32 of a unit of 2^(2 (e - 150) - 10), so only the conversion of
// a tile's sums rounds (FP64 additions round each time, and hold a pipe of two
// lanes per SM: 48 clocks per warp and sample).
struct Fixed {
    unsigned long long s1 = 0, s2 = 0, frac = 0;
    __device__ __forceinline__ void add(float v, int e) {
        const uint32_t b = __float_as_uint(v);
        const int below = e - (int)((b >> 23) & 255u);
        const uint32_t m = below > 31 ? 0u : (b & 0x7fffffu) | 0x800000u;  // 0: v is zero
        const int d = min(below, 31);
        const unsigned long long sign = (unsigned long long)(long long)((int)b >> 31);
        s1 += ((((unsigned long long)m << 31) >> d) ^ sign) - sign;
        const unsigned long long sq = (unsigned long long)(m << 5) * (m << 5);
        s2 += sq >> (2 * d);
        frac += (uint32_t)((sq << (63 - 2 * d)) >> 31);
    }
};
// Tiles whose largest magnitude lies outside [2^-40, 2^100), or with a nonzero
// value 2^-32 of it or less, go the FP64 way (so do infinities and NaN).
constexpr uint32_t kLargeBits = 0x71800000u;  // 2^100
constexpr uint32_t kSmallBits = 0x2b800000u;  // 2^-40

template <bool INT>
__global__ void __launch_bounds__(32 * kWarps, 4)
    detect_tile_kernel(const float *__restrict__ plane, int64_t pitch, int64_t nsamp, int ndm,
                       int nlevels, unsigned long long *s1, unsigned long long *s2,
                       unsigned long long *keys) {
    using T = typename std::conditional<INT, uint32_t, float>::type;
    constexpr uint32_t kNone = INT ? 0u : 0xff800000u;  // past the row: 0, -infinity
    const T none = INT ? (T)0 : (T)__uint_as_float(kNone);
    __shared__ uint32_t limb[8];      // fixed-point sums of the CTA
    __shared__ uint32_t extremes[2];  // largest magnitude, ~(smallest but 0, less 1)
    __shared__ __align__(16) uint32_t stage[kTileRows * kRegionWords];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // Tiles of one row are far apart in launch order: the later ones find the
    // row's highest values so far.
    const int row = blockIdx.x % (unsigned)ndm;
    const int64_t tile0 = (int64_t)(blockIdx.x / (unsigned)ndm) * tile_own<INT>;
    const int64_t s0 = tile0 + 32 * kTileK * warp;  // of the warp
    // Samples of the row from s0 on, as far as it matters.
    const int left = (int)max((int64_t)-4096, min(nsamp - s0, (int64_t)1 << 20));
    const bool busy = left > 0;
    unsigned long long *key_row = keys + (int64_t)row * nlevels;
    uint32_t *mystage = stage + warp * 32 * kRegionWords;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(mystage);
    if (left > -32 * kTileK) {  // else neither this warp nor the one before is busy
        const float *start = plane + (int64_t)row * pitch;
        const float *x = start + s0;
        if (((uintptr_t)x & 15u) == 0) {
            const uint32_t dst = base + 4 * (lane / 8 * kRegionWords + lane % 8 * 4);
            if (left >= 1024) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    stage_copy(dst + 16 * j * kRegionWords, x + 128 * j + 4 * lane, 16);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int at = 128 * j + 4 * lane, in = min(max(left - at, 0), 4);
                    stage_copy(dst + 16 * j * kRegionWords, in ? x + at : start, 4 * in);
                }
            }
        } else {
            const uint32_t dst = base + 4 * lane;
#pragma unroll 8
            for (int j = 0; j < 32; ++j) {
                const bool in = 32 * j + lane < left;
                stage_copy4(dst + 4 * j * kRegionWords, in ? x + 32 * j + lane : start,
                            in ? 4 : 0);
            }
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (warp < kTileReach)
        stage[(kWarps * 32 + warp) * kRegionWords + lane] = kNone;
    if (!INT && threadIdx.x < 8) {
        limb[threadIdx.x] = 0;
        extremes[threadIdx.x & 1] = 0;
    }
    // Highest boxcar of width 2^lane among the tiles done before.
    uint32_t best = 0;
    if (lane < nlevels)
        best = __ldcg(reinterpret_cast<const uint32_t *>(key_row + lane) + 1);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();

    T z[32];
    if (busy) {
        const uint4 *q = reinterpret_cast<const uint4 *>(mystage + lane * kRegionWords);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint4 v = q[k];
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if constexpr (INT)
                    z[4 * k + i] = w[i];
                else
                    z[4 * k + i] = __uint_as_float(w[i]);
            }
        }
    }
    int peak = 0;
    if constexpr (!INT) {
        // The tile's extreme magnitudes (a NaN's bits are above infinity's).
        uint32_t hi = 0, lo = 0xffffffffu;
        if (busy) {
#pragma unroll
            for (int k = 0; k < 32; k += 2) {
                const uint32_t a = __float_as_uint(z[k]) & 0x7fffffffu,
                               b = __float_as_uint(z[k + 1]) & 0x7fffffffu;
                hi = __vimax3_u32(hi, a, b);
                lo = __vimin3_u32(lo, a - 1u, b - 1u);
            }
            hi = __reduce_max_sync(0xffffffffu, hi);
            lo = __reduce_min_sync(0xffffffffu, lo);
        }
        __syncthreads();  // extremes are 0
        if (lane == 0 && hi != 0) {
            atomicMax(&extremes[0], hi);
            atomicMax(&extremes[1], ~lo);
        }
        __syncthreads();
        const uint32_t pb = extremes[0];
        peak = (int)(pb >> 23);
        const int least = (int)((~extremes[1] + 1u) >> 23);
        if (pb >= kLargeBits || (pb != 0 && (pb < kSmallBits || peak - least > 31))) {
            const int64_t seg = tile0 + (int64_t)warp * (tile_own<false> / kWarps);
            if (seg < nsamp)
                detect_segment<false, true, tile_own<false> / kWarps / 32, false>(
                    plane + (int64_t)row * pitch, nsamp, seg, row, nlevels, lane, 1u, s1, s2, keys);
            return;
        }
    }
    if (busy) {
        const bool mine = lane < kTileK;
        const bool own = mine && warp * kTileK + lane < tile_own<INT> / 32;
        uint32_t i1 = 0;
        uint64_t i2 = 0;
        bool bad = false;
        if constexpr (INT) {
#pragma unroll
            for (int k = 0; k < 32; ++k) {
                // x + 2^23 holds x in its low bits; anything but 0, 1, .. 2^21 - 1
                // comes back changed or gives 2^21 or more (as an unsigned value).
                const float v = __uint_as_float(z[k]);
                const float f = v + 8388608.0f;
                bad |= f - 8388608.0f != v;
                z[k] = __float_as_uint(f) - 0x4b000000u;
                i2 += (uint64_t)z[k] * z[k];
            }
        } else {
            Fixed f;
            if (peak != 0) {  // else zeros
#pragma unroll
                for (int k = 0; k < 32; ++k)
                    f.add(z[k], peak);
            }
            // Limbs of 21 bits: the sums of 256 lanes fit 32.  (s1's top one is
            // signed.)
            const uint32_t l[8] = {(uint32_t)(f.s1 & 0x1fffff),
                                   (uint32_t)((f.s1 >> 21) & 0x1fffff),
                                   (uint32_t)((long long)f.s1 >> 42),
                                   (uint32_t)(f.s2 & 0x1fffff),
                                   (uint32_t)((f.s2 >> 21) & 0x1fffff),
                                   (uint32_t)(f.s2 >> 42),
                                   (uint32_t)(f.frac & 0x1fffff),
                                   (uint32_t)(f.frac >> 21)};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t sum = __reduce_add_sync(0xffffffffu, own ? l[i] : 0u);
                if (lane == 0)
                    atomicAdd(&limb[i], sum);
            }
            if (left < 1024) {
#pragma unroll
                for (int k = 0; k < 32; ++k)
                    if (32 * lane + k >= left)
                        z[k] = none;
            }
        }
        // Highest value over the warp's positions, and, where it may be the
        // row's highest, its first position.
        auto track = [&](int lev) {
            const T m = mine ? highest<32>(z) : none;
            const uint32_t top = __reduce_max_sync(0xffffffffu, word_of(m));
            if (top >= __shfl_sync(0xffffffffu, best, lev) && nsamp >= 1 << lev) {
                const uint32_t bits = bits_of(value_of<T>(top));
                const uint32_t who = __ballot_sync(0xffffffffu, mine && word_of(m) == top);
                if (lane == __ffs(who) - 1) {
                    int at = 0;
#pragma unroll
                    for (int k = 31; k >= 0; --k)
                        at = bits_of(z[k]) == bits ? k : at;
                    const uint32_t t = (uint32_t)(s0 + 32 * lane + at);
                    atomicMax(key_row + lev, (unsigned long long)top << 32 | (0xffffffffu - t));
                }
            }
            return top;
        };
        const bool large = track(0) >= 1u << 21;
        if (INT && nlevels <= 5)
#pragma unroll
            for (int k = 0; k < 32; ++k)
                i1 += bits_of(z[k]);
        if (nlevels > 1) {
            widen<1>(z);
            track(1);
        }
        if (nlevels > 2) {
            widen<2>(z);
            track(2);
        }
        if (nlevels > 3) {
            widen<4>(z);
            track(3);
        }
        if (nlevels > 4) {
            widen<8>(z);
            track(4);
        }
        if (nlevels > 5) {
            widen<16>(z);
            i1 = bits_of(z[0]);  // the region's sum
            track(5);
        }
        if (nlevels > 6 && mine) {
            uint4 *w = reinterpret_cast<uint4 *>(mystage + lane * kRegionWords);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                w[k] = make_uint4(bits_of(z[4 * k]), bits_of(z[4 * k + 1]), bits_of(z[4 * k + 2]),
                                  bits_of(z[4 * k + 3]));
        }
        if constexpr (INT) {
            // Row sums: each sample by the one lane that owns its region.
            const bool any_bad = large || __any_sync(0xffffffffu, bad && own);
            uint64_t a = own ? i1 : 0u;
            i2 = own ? i2 : 0u;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a += __shfl_xor_sync(0xffffffffu, a, o);
                i2 += __shfl_xor_sync(0xffffffffu, i2, o);
            }
            if (lane == 0) {
                // The sums stay below 2^63; a row of other values is marked there.
                if (any_bad) {
                    atomicOr(&s2[row], 1ull << 63);
                } else {
                    atomicAdd(&s1[row], (unsigned long long)a);
                    atomicAdd(&s2[row], (unsigned long long)i2);
                }
            }
        }
    } else if (!INT && nlevels > 6 && left > -32 * kTileK) {
        // Past the row, but within the reach of the warp before.
#pragma unroll
        for (int k = 0; k < kTileReach; ++k)
            mystage[k * kRegionWords + lane] = kNone;
    }
    if (INT && nlevels <= 6)
        return;
    __syncthreads();
    if constexpr (!INT) {
        if (threadIdx.x < 2) {
            // l2 2^42 + l1 2^21 + l0 (+ frac 2^-32) units.
            const bool sq = threadIdx.x == 1;
            const uint32_t *l = limb + (sq ? 3 : 0);
            const long long top =
                (long long)((unsigned long long)(long long)(int)l[2] << 21) + l[1];
            double v = (double)l[0];
            if (sq)
                v = __fma_rn((double)((unsigned long long)limb[7] * 2097152 + limb[6]),
                             2.3283064365386963e-10, v);
            v = __fma_rn((double)top, 2097152.0, v);
            atomicAdd(reinterpret_cast<double *>(sq ? &s2[row] : &s1[row]),
                      scalbn(v, sq ? 2 * (peak - 150) - 10 : peak - 181));
        }
        if (nlevels <= 6)
            return;
    }
    if (!busy)
        return;
    T y[kTileK + kTileReach];  // width 32 at s0 + 32 k + lane
#pragma unroll
    for (int k = 0; k < kTileK + kTileReach; ++k)
        y[k] = reinterpret_cast<const T *>(mystage)[(k < kTileK ? k : k + 1) * kRegionWords + lane];
    auto track = [&](int lev) {
        const T m = highest<kTileK>(y);
        const uint32_t top = __reduce_max_sync(0xffffffffu, word_of(m));
        if (top >= __shfl_sync(0xffffffffu, best, lev) && nsamp >= 1 << lev) {
            const uint32_t bits = bits_of(value_of<T>(top));
            int at = 1 << 24;  // none
#pragma unroll
            for (int k = kTileK - 1; k >= 0; --k)
                at = bits_of(y[k]) == bits ? k : at;
            // Relative to the warp's first position, so that the order survives.
            const uint32_t rel = __reduce_min_sync(0xffffffffu, (uint32_t)(32 * at + lane));
            if (lane == 0)
                atomicMax(key_row + lev, (unsigned long long)top << 32 |
                                             (0xffffffffu - ((uint32_t)s0 + rel)));
        }
    };
#pragma unroll
    for (int lev = 6; lev < kMaxLevels; ++lev) {
        if (lev >= nlevels)
            break;
        const int m = 1 << (lev - 6);
#pragma unroll
        for (int k = 0; k + m < kTileK + kTileReach; ++k)
            y[k] += y[k + m];
        track(lev);
    }
}

// Sums and keys -> mean, std, S/N, t (in place): a thread per row and width,
// 28 rows a CTA (the chain of FP64 divisions and roots for all nine widths of
// a row in one thread took 19 us).
constexpr int kFinalRows = 28;
template <bool INT>
__global__ void finalize_kernel(int ndm, int64_t nsamp, int nlevels, double *mean, double *sd,
                                double *snr, int64_t *tpk) {
    const int row = blockIdx.x * kFinalRows + threadIdx.x / nlevels, lev = threadIdx.x % nlevels;
    const bool in = row < ndm && threadIdx.x < kFinalRows * nlevels;
    const double n = (double)nsamp;
    double s1 = 0.0, s2 = 0.0;
    bool bad = false;
    if (in && INT) {
        const unsigned long long a = reinterpret_cast<unsigned long long *>(mean)[row];
        const unsigned long long b = reinterpret_cast<unsigned long long *>(sd)[row];
        bad = (b >> 63) != 0;
        s1 = __ull2double_rn(a);
        s2 = __ull2double_rn(b);
    } else if (in) {
        s1 = mean[row];
        s2 = sd[row];
    }
    __syncthreads();  // the sums are read; mean and sd take their places
    if (!in)
        return;
    const double m = __ddiv_rn(s1, n);
    double var = __dsub_rn(__ddiv_rn(s2, n), __dmul_rn(m, m));
    if (var < 0.0)
        var = 0.0;
    const double s = __dsqrt_rn(var);
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    if (lev == 0) {
        mean[row] = bad ? nan : m;
        sd[row] = bad ? nan : s;
    }
    const int64_t i = (int64_t)row * nlevels + lev;
    const unsigned long long key = reinterpret_cast<unsigned long long *>(snr)[i];
    const double w = (double)(1 << lev);
    if (bad) {
        snr[i] = nan;
        tpk[i] = -1;
    } else if (key == 0) {
        snr[i] = -__longlong_as_double(0x7ff0000000000000ll);  // -inf: no window
        tpk[i] = -1;
    } else {
        const uint32_t v = (uint32_t)(key >> 32);
        const double b = INT ? (double)v : (double)unordered(v);
        tpk[i] = (int64_t)(0xffffffffull - (key & 0xffffffffull));
        snr[i] = s == 0.0 ? 0.0
                          : __ddiv_rn(__dsub_rn(b, __dmul_rn(w, m)), __dmul_rn(s, __dsqrt_rn(w)));
    }
}

// The accumulators in the caller's arrays (one launch; three memsets took 6 us
// longer).
__global__ void clear_kernel(int ndm, int64_t n, double *mean, double *sd, double *snr) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < ndm)
        mean[i] = 0.0;
    else if (i < 2 * (int64_t)ndm)
        sd[i - ndm] = 0.0;
    else if (i < n)
        snr[i - 2 * (int64_t)ndm] = 0.0;
}

template <bool INT>
void launch_finalize(int ndm, int64_t nsamp, int nlevels, double *mean, double *sd, double *snr,
                     int64_t *tpk, cudaStream_t s) {
    finalize_kernel<INT><<<(ndm + kFinalRows - 1) / kFinalRows, kFinalRows * kMaxLevels, 0, s>>>(
        ndm, nsamp, nlevels, mean, sd, snr, tpk);
}

}  // namespace

extern "C" dd_status dd_detect(const float *plane, int64_t pitch, int ndm, int64_t nsamp,
                               int nlevels, int integer_valued, double *mean, double *std_out,
                               double *snr, int64_t *t_peak, void *stream) {
    dd::Range nvtx_range("dd_detect");
    using dd::fail;
    if (ndm < 0 || nsamp < 1 || pitch < nsamp)
        return fail(DD_ERR_INVALID, "need ndm >= 0, nsamp >= 1 and pitch >= nsamp");
    if (nlevels < 1 || nlevels > kMaxLevels)
        return fail(DD_ERR_INVALID, "nlevels must be 1..9 (boxcar widths up to 256)");
    if (nsamp > 0xfffffffeLL || (integer_valued && nsamp > (1LL << 21)))
        return fail(DD_ERR_INVALID, "nsamp too large (2^21 for integer planes)");
    if (ndm == 0)
        return DD_OK;
    if (!plane || !mean || !std_out || !snr || !t_peak || ((uintptr_t)plane & 3u) ||
        ((uintptr_t)mean & 7u) || ((uintptr_t)std_out & 7u) || ((uintptr_t)snr & 7u) ||
        ((uintptr_t)t_peak & 7u))
        return fail(DD_ERR_INVALID, "NULL or misaligned pointer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const dd_status begun = dd::detect_begin(ndm, nlevels, mean, std_out, snr, s);
    if (begun != DD_OK)
        return begun;
    const int64_t own = integer_valued ? tile_own<true> : tile_own<false>;
    const int64_t tiles = (nsamp + own - 1) / own;
    if (tiles * ndm > 0x7fffffffLL)
        return fail(DD_ERR_INVALID, "plane too large for one launch");
    const unsigned grid = (unsigned)(tiles * ndm);
    auto *s1 = reinterpret_cast<unsigned long long *>(mean);
    auto *s2 = reinterpret_cast<unsigned long long *>(std_out);
    auto *keys = reinterpret_cast<unsigned long long *>(snr);
    if (integer_valued)
        detect_tile_kernel<true><<<grid, 32 * kWarps, 0, s>>>(plane, pitch, nsamp, ndm, nlevels,
                                                              s1, s2, keys);
    else
        detect_tile_kernel<false><<<grid, 32 * kWarps, 0, s>>>(plane, pitch, nsamp, ndm, nlevels,
                                                               s1, s2, keys);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) {
        if (integer_valued)
            launch_finalize<true>(ndm, nsamp, nlevels, mean, std_out, snr, t_peak, s);
        else
            launch_finalize<false>(ndm, nsamp, nlevels, mean, std_out, snr, t_peak, s);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess)
        return fail(DD_ERR_CUDA, std::string("detect launch: ") + cudaGetErrorString(e));
    dd::count_launch(2);
    return DD_OK;
}

namespace dd {

dd_status detect_begin(int ndm, int nlevels, double *mean, double *sd, double *snr,
                       cudaStream_t s) {
    const int64_t n = (int64_t)ndm * (nlevels + 2);
    clear_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(ndm, n, mean, sd, snr);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return fail(DD_ERR_CUDA, std::string("detect clear: ") + cudaGetErrorString(e));
    count_launch(1);
    return DD_OK;
}

dd_status detect_finalize_int(int ndm, int64_t nsamp, int nlevels, double *mean, double *sd,
                              double *snr, int64_t *tpk, cudaStream_t s) {
    launch_finalize<true>(ndm, nsamp, nlevels, mean, sd, snr, tpk, s);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return fail(DD_ERR_CUDA, std::string("detect finalize: ") + cudaGetErrorString(e));
    count_launch(1);
    return DD_OK;
}

}  // namespace dd
