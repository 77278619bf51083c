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
// detect_int_kernel searches integer-valued planes (below).
// detect_float_kernel: one warp owns 1024 consecutive start positions of one
// row (a CTA: 8 warps, 8192 positions), searched by detect_segment
// (dd_detect_seg.cuh; the 255-sample halo the widest boxcar needs is re-read
// from L2 by the neighbouring warp).
// finalize_kernel then turns the sums and keys into mean, std, S/N and t with
// the same IEEE FP64 operations, in the same order, as the CPU definition.
// The output arrays double as the accumulators, so no scratch is needed.
#include <cuda_runtime.h>

#include <cstdint>
#include <string>

#include "dd_detect_seg.cuh"
#include "dd_internal.h"

namespace {

using dd::detect_segment;
using dd::kMaxLevels;
using dd::unordered;

constexpr int kOwnK = 32;       // owned positions per lane (1024 per warp)
constexpr int kKH = kOwnK + dd::kReach;
constexpr int kWarps = 8;

__global__ void __launch_bounds__(32 * kWarps, 3)
    detect_float_kernel(const float *__restrict__ plane, int64_t pitch, int64_t nsamp, int groups,
                        int nlevels, unsigned long long *s1, unsigned long long *s2,
                        unsigned long long *keys, uint32_t one) {
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x / groups;
    const int64_t s0 =
        ((int64_t)(blockIdx.x % groups) * kWarps + (threadIdx.x >> 5)) * (32 * kOwnK);
    if (s0 >= nsamp)
        return;
    const float *x = plane + (int64_t)row * pitch;
    if (s0 + 32 * kKH <= nsamp)
        detect_segment<false, false, kOwnK, false>(x, nsamp, s0, row, nlevels, lane, one, s1, s2,
                                                   keys);
    else
        detect_segment<false, true, kOwnK, false>(x, nsamp, s0, row, nlevels, lane, one, s1, s2,
                                                  keys);
}

// Integer planes.  A CTA searches kTileOwn start positions of one row.  Warp w
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
// or the staged samples, run into zeros: such a sum is no more than that of
// the last whole window, which starts earlier and so wins a tie, or of the
// same window in the next tile.
//
// 1024 rows x 131072 samples: 172 us (79 us to read the plane), bound by
// instruction issue: 34 per sample, 68 % of the slots.  Segments of one warp
// each, with a shuffle per sample and width up to 32 and value and position in
// one key (detect_segment), took 335 us at 68 instructions.
constexpr int kRegionWords = 36;  // 16-byte reads of 8 lanes meet no bank twice
constexpr int kTileK = 31;        // regions of a warp
constexpr int kTileReach = 7;     // regions beyond, up to width 256
constexpr int kTileOwn = 32 * (kWarps * kTileK - kTileReach);
constexpr int kTileRows = kWarps * 32 + kTileReach;  // the last ones are zeros

__device__ __forceinline__ void stage_copy(uint32_t dst, const float *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void stage_copy4(uint32_t dst, const float *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}

template <int N>
__device__ __forceinline__ uint32_t highest(const uint32_t *z) {
    uint32_t a = z[0], b = z[1];  // two chains
#pragma unroll
    for (int k = 2; k + 3 < N; k += 4) {
        a = __vimax3_u32(a, z[k], z[k + 1]);
        b = __vimax3_u32(b, z[k + 2], z[k + 3]);
    }
#pragma unroll
    for (int k = N - (N - 2) % 4; k < N; ++k)
        a = max(a, z[k]);
    return max(a, b);
}

// Boxcars of width 2W from those of width W, a region per lane.
template <int W>
__device__ __forceinline__ void widen(uint32_t *z) {
    uint32_t r[W];
#pragma unroll
    for (int k = 0; k < W; ++k)
        r[k] = __shfl_down_sync(0xffffffffu, z[k], 1);
#pragma unroll
    for (int k = 0; k < 32; ++k)
        z[k] += k + W < 32 ? z[(k + W) & 31] : r[(k + W - 32) & (W - 1)];
}

__global__ void __launch_bounds__(32 * kWarps, 4)
    detect_int_kernel(const float *__restrict__ plane, int64_t pitch, int nsamp, int ndm,
                      int nlevels, unsigned long long *s1, unsigned long long *s2,
                      unsigned long long *keys) {
    __shared__ __align__(16) uint32_t stage[kTileRows * kRegionWords];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // Tiles of one row are far apart in launch order: the later ones find the
    // row's highest values so far.
    const int row = blockIdx.x % (unsigned)ndm;
    const int s0 = (int)(blockIdx.x / (unsigned)ndm) * kTileOwn + 32 * kTileK * warp;  // of the warp
    const int left = nsamp - s0;  // samples of the row from s0 on
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
        stage[(kWarps * 32 + warp) * kRegionWords + lane] = 0;
    // Highest boxcar of width 2^lane among the tiles done before.
    uint32_t best = 0;
    if (lane < nlevels)
        best = __ldcg(reinterpret_cast<const uint32_t *>(key_row + lane) + 1);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();

    if (busy) {
        uint32_t z[32];
        const uint4 *q = reinterpret_cast<const uint4 *>(mystage + lane * kRegionWords);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint4 v = q[k];
            z[4 * k] = v.x;
            z[4 * k + 1] = v.y;
            z[4 * k + 2] = v.z;
            z[4 * k + 3] = v.w;
        }
        const bool mine = lane < kTileK;
        uint32_t i1 = 0;
        uint64_t i2 = 0;
        bool bad = false;
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
        // Highest value over the warp's positions, and, where it may be the
        // row's highest, its first position.
        auto track = [&](int lev) {
            const uint32_t m = mine ? highest<32>(z) : 0u;
            const uint32_t top = __reduce_max_sync(0xffffffffu, m);
            if (top >= __shfl_sync(0xffffffffu, best, lev) && nsamp >= 1 << lev) {
                const uint32_t who = __ballot_sync(0xffffffffu, mine && m == top);
                if (lane == __ffs(who) - 1) {
                    int at = 0;
#pragma unroll
                    for (int k = 31; k >= 0; --k)
                        at = z[k] == top ? k : at;
                    const uint32_t t = (uint32_t)(s0 + 32 * lane + at);
                    atomicMax(key_row + lev, (unsigned long long)top << 32 | (0xffffffffu - t));
                }
            }
            return top;
        };
        const bool large = track(0) >= 1u << 21;
        if (nlevels <= 5)
#pragma unroll
            for (int k = 0; k < 32; ++k)
                i1 += z[k];
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
            i1 = z[0];  // the region's sum
            track(5);
        }
        if (nlevels > 6 && mine) {
            uint4 *w = reinterpret_cast<uint4 *>(mystage + lane * kRegionWords);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                w[k] = make_uint4(z[4 * k], z[4 * k + 1], z[4 * k + 2], z[4 * k + 3]);
        }
        // Row sums: each sample by the one lane that owns its region.
        const bool own = mine && warp * kTileK + lane < kTileOwn / 32;
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
    if (nlevels <= 6)
        return;
    __syncthreads();
    if (!busy)
        return;
    uint32_t y[kTileK + kTileReach];  // width 32 at s0 + 32 k + lane
#pragma unroll
    for (int k = 0; k < kTileK + kTileReach; ++k)
        y[k] = mystage[(k < kTileK ? k : k + 1) * kRegionWords + lane];
    auto track = [&](int lev) {
        const uint32_t m = highest<kTileK>(y);
        const uint32_t top = __reduce_max_sync(0xffffffffu, m);
        if (top >= __shfl_sync(0xffffffffu, best, lev) && nsamp >= 1 << lev) {
            int at = 1 << 24;  // none
#pragma unroll
            for (int k = kTileK - 1; k >= 0; --k)
                at = y[k] == top ? k : at;
            const uint32_t t =
                __reduce_min_sync(0xffffffffu, (uint32_t)(s0 + 32 * at + lane));
            if (lane == 0)
                atomicMax(key_row + lev, (unsigned long long)top << 32 | (0xffffffffu - t));
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
    const int64_t per_cta = (int64_t)kWarps * 32 * kOwnK;
    const int64_t groups = (nsamp + per_cta - 1) / per_cta;
    if (groups * ndm > 0x7fffffffLL)
        return fail(DD_ERR_INVALID, "plane too large for one launch");
    const unsigned grid = (unsigned)(groups * ndm);
    auto *s1 = reinterpret_cast<unsigned long long *>(mean);
    auto *s2 = reinterpret_cast<unsigned long long *>(std_out);
    auto *keys = reinterpret_cast<unsigned long long *>(snr);
    if (integer_valued)
        detect_int_kernel<<<(unsigned)((nsamp + kTileOwn - 1) / kTileOwn * ndm), 32 * kWarps, 0,
                            s>>>(plane, pitch, (int)nsamp, ndm, nlevels, s1, s2, keys);
    else
        detect_float_kernel<<<grid, 32 * kWarps, 0, s>>>(plane, pitch, nsamp, (int)groups, nlevels,
                                                         s1, s2, keys, 1u);
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
