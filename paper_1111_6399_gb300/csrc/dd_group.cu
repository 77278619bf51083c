// De-dispersion of uint8 beams with channel-group partial sums (dd_group.h),
// for sm_103a.
//
// What bounds the direct kernel (dd_kernel.cuh) is shared memory: every add
// reads its byte from there.  Here a DM reads one 16-bit sum per group and
// sample, half of the bytes per add with G = 4, and needs no byte unpacking.
//
// CTA: one tile of 64 DMs x 1024 samples; three kinds of warps, with the
// registers split between them (setmaxnreg: 640 x 96 = 256 x 168 + 384 x 48).
//  * One fetch warp copies each pair of groups' channel windows and records
//    into a ring of raw slots, and the DMs' offsets, with TMA bulk copies.
//  * 11 builder warps sum the rows for each pattern, 128 samples a unit, the
//    units of both groups dealt round-robin over the warps.  Arrays are packed
//    16-bit sums, kept twice, one sample apart, so that every shifted read is
//    an aligned 32-bit word.
//  * 8 user warps: a thread owns 8 DMs x 16 words (32 samples), lane-
//    interleaved, so each LDS.32 of a warp covers 32 banks.  It adds the words
//    of both groups for half of a DM's samples (one three-input add) while it
//    loads those of the next half.  16-bit lanes hold 256 channels' sums at
//    most (65280) and are then widened into the FP32 plane, exactly.
// A pair is built while the one before is used, in the other end of the array
// space; mbarriers hand the arrays over, waits are bounded.
//
// Measured on the 4096-channel beam (2000 DMs x 262144 samples): 63.8 ms
// against the direct kernel's 81.4; beams whose DM tiles span fewer samples
// gain more (1024 channels over 64 MHz, 1024 DMs x 65536: 1.82 against 2.77).
// No unit is full: on 16384 samples of that beam, issue slots 62 %, L1 and shared
// memory 73 %, ALU 53 % while CTAs are resident.  Of 8.0 cycles an instruction,
// a warp waits 1.8 for shared-memory loads and their queue, 1.7 on a long
// scoreboard (in the loops only the hand-overs and the fetch warp's records have
// one), 1.6 for the latency of the instruction before.  Measured slower, on the same
// beam: 4 builder warps at 128 registers (217 ms); 16 warps that build and use in
// turn, handing over by mbarriers or a block barrier (68 - 72); 8 builder warps
// that also fetch (68); 15 builders with 768-sample tiles (66.6).  Forms of it
// for FP16/FP32 (one FP32 sum per group) were not kept: 40 - 60 ms against 37 on
// that beam as FP16, 7.6 against 8.05 on the FP32 L-band beam.
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "dd_group.h"
#include "dd_prims.cuh"

namespace dd {
namespace {

constexpr int kDT = kGroupDms;
constexpr int kNW = kGroupWords;
constexpr int kThreads = 32 * (kGroupUsers + kGroupBuilders + 1);

__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(a)
                 : "memory");
    return v;
}
// Two 8-byte stores if a < b, without a branch.
__device__ __forceinline__ void sts64_pair_below(uint32_t a, uint32_t b, uint32_t at0, uint32_t at1,
                                                 uint32_t x0, uint32_t y0, uint32_t x1,
                                                 uint32_t y1) {
    asm volatile("{ .reg .pred q; setp.lt.u32 q, %6, %7; @q st.shared.v2.u32 [%0], {%2, %3}; "
                 "@q st.shared.v2.u32 [%1], {%4, %5}; }" ::"r"(at0),
                 "r"(at1), "r"(x0), "r"(y0), "r"(x1), "r"(y1), "r"(a), "r"(b)
                 : "memory");
}

// Pattern arrays of one group of N channels, unit n: lane l makes samples
// u .. u + 3, u = 128 n + 4 l, of every pattern.
//
// For each channel a lane holds 8 row bytes from the class's smallest offset
// on; a pattern's window F starts 0..3 bytes further (one permute).  Summed
// over the channels with 16-bit lanes: L1 = sum F, O = sum of the odd bytes;
// L1 - 256 O are the even bytes' sums E.  The second copy, one sample on,
// needs the fifth sample's sum X too: a dot product with a one-hot byte (a
// shuffle from the next lane would put a round trip through the busy
// shared-memory queue into every pattern).  The next pattern's record is read
// one pattern ahead, for the same reason.
template <int N>
__device__ __forceinline__ void build_unit(uint32_t rec, uint32_t rows_at, uint32_t arrays, int n,
                                           int lane) {
    const uint32_t u = (uint32_t)(n * kGroupUnit + 4 * lane);
    const uint4 cl = lds128(rec + 16);  // classes, patterns of each
    const uint32_t to = arrays + 2u * u;
    uint32_t cls = rec + (uint32_t)offsetof(GroupRecord, cls);
    uint32_t tp = rec + (uint32_t)offsetof(GroupRecord, tup);
    uint4 d = lds128(tp);
    for (int k = 0; k < (int)cl.x; ++k) {
        uint32_t A[N > 0 ? N : 1][2];
        const uint4 at = lds128(cls), sh = lds128(cls + 16);
        cls += (uint32_t)sizeof(GroupClass);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const uint32_t p = rows_at + u + (i == 0 ? at.x : i == 1 ? at.y : i == 2 ? at.z : at.w);
            const uint32_t q = i == 0 ? sh.x : i == 1 ? sh.y : i == 2 ? sh.z : sh.w;
            const uint32_t w0 = lds32(p), w1 = lds32(p + 4), w2 = lds32(p + 8);
            A[i][0] = prmt(w0, w1, q);
            A[i][1] = prmt(w1, w2, q);
        }
        const uint32_t O0 = N > 0 ? prmt(A[0][0], 0u, 0x4341u) : 0u;
        const uint32_t X0 = N > 0 ? A[0][1] & 0xffu : 0u;
        int left = (int)(((k < 4 ? cl.y : cl.z) >> (8 * (k & 3))) & 255u);
#pragma unroll 1
        do {
            const uint4 c = d;
            tp += (uint32_t)sizeof(GroupTuple);
            d = lds128(tp);  // (past the last: unused)
            const uint32_t lo = c.x & 0xffffu, len = c.x >> 16;
            uint32_t L1 = N > 0 ? A[0][0] : 0u, O = O0, X = X0;
#pragma unroll
            for (int i = 1; i < N; ++i) {
                const uint32_t F = prmt(A[i][0], A[i][1], i == 1 ? c.z : i == 2 ? c.z >> 16 : c.w);
                L1 += F;
                O += prmt(F, 0u, 0x4341u);
                X = __dp4a(A[i][1], __funnelshift_l(0u, 1u, c.w >> (11 + 5 * i)), X);
            }
            const uint32_t E = L1 - (O << 8);
            const uint32_t w = to + c.y;
            sts64_pair_below(u - lo, len, w, w + 2u * len, prmt(E, O, 0x5410u), prmt(E, O, 0x7632u),
                             prmt(E, O, 0x3254u), prmt(O, X, 0x5432u));
        } while (--left > 0);
    }
}

__global__ void __launch_bounds__(kThreads, 1) group_kernel(const __grid_constant__ GroupArgs a) {
    constexpr uint32_t R = kGroupRaw;
    constexpr uint32_t kRec = (uint32_t)sizeof(GroupRecord);
    constexpr uint32_t kRowsAt = 2u * kRec;  // staged rows in a raw slot
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t mb_raw[R], mb_built[R], mb_full[2], mb_empty[2];
    __shared__ __align__(16) int2 offs[kGroupOffs][kGroupDmCta];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // Pair p passes: raw (fetched) -> full (built) -> empty (used); built also
    // frees its raw slot.
    const uint32_t raw = smem_addr(mb_raw), built = smem_addr(mb_built), full = smem_addr(mb_full),
                   empty = smem_addr(mb_empty);
    if (tid == 0) {
        for (uint32_t i = 0; i < R; ++i) {
            mbar_init(raw + 8 * i, 1);
            mbar_init(built + 8 * i, kGroupBuilders);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(full + 8 * i, kGroupBuilders);
            mbar_init(empty + 8 * i, kGroupUsers);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    // The beam and tile.
    int bi = 0;
    for (int hi = a.beams ? a.nbeams - 1 : 0; bi < hi;) {
        const int mid = (bi + hi + 1) >> 1;
        if (a.beams[mid].tile_begin <= (int64_t)blockIdx.x)
            bi = mid;
        else
            hi = mid - 1;
    }
    const GroupBeam &B = a.beams ? a.beams[bi] : a.beam0;
    const int64_t local = (int64_t)blockIdx.x - B.tile_begin;
    const int td = (int)(local % B.ntile_d);
    const int64_t t0 = local / B.ntile_d * kGroupTCta;
    const uint32_t E = (uint32_t)B.npairs;
    const int G = B.G, rowcap = B.rowcap;
    const uint32_t raw_bytes = (uint32_t)group_raw_bytes(G, rowcap);
    const uint32_t raw0 = smem_addr(smem), arrays = raw0 + R * raw_bytes;

    if (warp >= kGroupUsers) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
        bool ok = true;
        const int bw = warp - kGroupUsers;
        if (bw == kGroupBuilders) {
            // ------------------------------- fetch -------------------------------
            // Lane l < 2 G: row l of the pair (its record loaded a pair ahead);
            // lanes 30, 31: the records and the offsets.
            const uint8_t *in = B.in + t0;
            const int64_t rest = (B.nsamp_in - t0 + 15) & ~(int64_t)15;
            const int avail = (int)(rest < 0x7ffffff0 ? rest : 0x7ffffff0);
            const GroupEntry *entry = B.entries + (int64_t)td * E;
            const int rg = lane >= G, rl = lane - rg * G;  // the row's group and place
            GroupRow next = {0, 0, 0, -1};
            if (lane < 2 * G)
                next = entry->g[rg].rows[rl];
            uint32_t s = 0, par = 1;  // f % R; parity of the slot's last build
            for (uint32_t f = 0; f < E; ++f, ++entry) {
                const GroupRow r = next;
                if (lane < 2 * G && f + 1 < E)
                    next = entry[1].g[rg].rows[rl];
                if (f >= R && !mbar_spin(built + 8 * s, par)) {
                    ok = false;
                    break;
                }
                const uint32_t slot = raw0 + s * raw_bytes, bar = raw + 8 * s;
                uint32_t bytes = 0, dst = slot + kRowsAt + (uint32_t)(lane * rowcap);
                const void *src = in + (int64_t)r.chan * B.in_pitch_b + r.first;
                if (r.chan >= 0)
                    bytes = (uint32_t)min(r.bytes, avail - r.first);
                if (lane == 30) {
                    bytes = kRowsAt;
                    src = entry->g;
                    dst = slot;
                } else if (lane == 31) {
                    // Where pair f - 8's were: pair f - 3 is built, so pair f - 5 used.
                    static_assert(kGroupOffs >= (int)R + 3, "offsets outlive their use");
                    bytes = sizeof(entry->offs);
                    src = entry->offs;
                    dst = smem_addr(offs[f % kGroupOffs]);
                }
                const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
                if (lane == 0)
                    mbar_expect_tx_arrive(bar, total);
                __syncwarp();
                if (bytes)
                    bulk_g2s(dst, src, bytes, bar);
                if (++s == R) {
                    s = 0;
                    par ^= 1u;
                }
            }
            // Leave only once the copies in flight have landed (bounded).
            for (uint32_t q = 0; !ok && q < R; ++q)
                mbar_spin(raw + 8 * q, q < s ? par ^ 1u : par);
        } else {
            // ------------------------------ builders ------------------------------
            int uoff = bw;            // this warp's place in the next pair's units
            uint32_t s = 0, par = 0;  // p % R, (p / R) & 1
            for (uint32_t p = 0; p < E; ++p) {
                // Pair p has been fetched and pair p - 2's arrays used.
                if (!mbar_spin(raw + 8 * s, par) ||
                    (p >= 2 && !mbar_spin(empty + 8 * (p & 1), (p / 2 - 1) & 1u))) {
                    ok = false;
                    break;
                }
                const uint32_t slot = raw0 + s * raw_bytes;
                const int n0 = (int)lds32(slot + 4), n1 = n0 + (int)lds32(slot + kRec + 4);
                for (; uoff < n1; uoff += kGroupBuilders) {
                    const bool second = uoff >= n0;
                    const uint32_t rec = slot + (second ? kRec : 0u);
                    const uint32_t rows = slot + kRowsAt + (uint32_t)(second ? G * rowcap : 0);
                    const int n = second ? uoff - n0 : uoff;
                    switch (lds32(rec + 12)) {  // channels: G, or what the last group has
                    case 0: build_unit<0>(rec, rows, arrays, n, lane); break;
                    case 1: build_unit<1>(rec, rows, arrays, n, lane); break;
                    case 2: build_unit<2>(rec, rows, arrays, n, lane); break;
                    case 3: build_unit<3>(rec, rows, arrays, n, lane); break;
                    default: build_unit<4>(rec, rows, arrays, n, lane); break;
                    }
                }
                uoff -= n1;
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(full + 8 * (p & 1));
                    mbar_arrive(built + 8 * s);
                }
                if (++s == R) {
                    s = 0;
                    par ^= 1u;
                }
            }
        }
        if (!ok)
            record(a.status, kDevTimeout);
        return;
    }

    // --------------------------------- users ----------------------------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
    const int close_every = kSwarChannels / G;  // groups between widenings
    const int kthr = td * kGroupDmCta + warp * kDT;
    const uint32_t thr = arrays + 4u * (uint32_t)lane;
    uint32_t acc[kDT][kNW];
#pragma unroll
    for (int j = 0; j < kDT; ++j)
#pragma unroll
        for (int k = 0; k < kNW; ++k)
            acc[j][k] = 0;
    bool fresh = true;  // nothing widened yet

    // Widen the 16-bit sums into the plane: stored first, then added (FP32
    // additions of integers below 2^24 are exact in any order).
    auto widen = [&]() {
        const int64_t n = B.nsamp_out;
#pragma unroll
        for (int j = 0; j < kDT; ++j) {
            const int row = B.perm[kthr + j];
            float *orow = B.out + (int64_t)row * B.out_pitch;
#pragma unroll
            for (int k = 0; k < kNW; ++k) {
                // exact: the bits 0x4b000000 | v are the float 2^23 + v
                const float x = __uint_as_float(0x4b000000u | (acc[j][k] & 0xffffu)) - 8388608.0f;
                const float y = __uint_as_float(0x4b000000u | (acc[j][k] >> 16)) - 8388608.0f;
                acc[j][k] = 0u;
                const int64_t t = t0 + 2 * (lane + 32 * k);
                if (row < 0 || t >= n)
                    continue;
                if (t + 1 < n) {
                    if (fresh)
                        *reinterpret_cast<float2 *>(orow + t) = make_float2(x, y);
                    else
                        asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(orow + t), "f"(x),
                                     "f"(y)
                                     : "memory");
                } else if (fresh) {
                    orow[t] = x;
                } else {
                    atomicAdd(orow + t, x);
                }
            }
        }
        fresh = false;
    };

    // Words of both groups for half h (8 words) of a DM.
    constexpr int HW = kNW / 2;
    uint32_t x[HW], y[HW];
    auto load = [&](int2 off) {
        const uint32_t p = thr + (uint32_t)off.x, q = thr + (uint32_t)off.y;
#pragma unroll
        for (int k = 0; k < HW; ++k) {
            x[k] = lds32(p + 128 * k);
            y[k] = lds32(q + 128 * k);
        }
    };
    // Add the loaded words to half h of DM j and, word by word, load half hn
    // of the DM at `off`.
    auto add_load = [&](int j, int h, bool reload, int hn, int2 off) {
        const uint32_t p = thr + (uint32_t)off.x, q = thr + (uint32_t)off.y;
#pragma unroll
        for (int k = 0; k < HW; k += 2) {
            acc[j][h * HW + k] += x[k] + y[k];
            acc[j][h * HW + k + 1] += x[k + 1] + y[k + 1];
            if (reload) {
                x[k] = lds32(p + 128 * (HW * hn + k));
                y[k] = lds32(q + 128 * (HW * hn + k));
                x[k + 1] = lds32(p + 128 * (HW * hn + k + 1));
                y[k + 1] = lds32(q + 128 * (HW * hn + k + 1));
            }
        }
    };

    int close_in = close_every;
    for (uint32_t p = 0; p < E; ++p) {
        if (!mbar_spin(full + 8 * (p & 1), (p / 2) & 1u)) {
            record(a.status, kDevTimeout);
            return;
        }
        const int4 *op = reinterpret_cast<const int4 *>(&offs[p % kGroupOffs][warp * kDT]);
        int4 o = op[0];  // two DMs
        load(make_int2(o.x, o.y));
#pragma unroll
        for (int j = 0; j < kDT; j += 2) {
            const int2 even = make_int2(o.x, o.y), odd = make_int2(o.z, o.w);
            if (j + 2 < kDT)
                o = op[j / 2 + 1];
            add_load(j, 0, true, 1, even);
            add_load(j, 1, true, 0, odd);
            add_load(j + 1, 0, true, 1, odd);
            add_load(j + 1, 1, j + 2 < kDT, 0, make_int2(o.x, o.y));
        }
        // Every word of this pair has been used: release it.
        __syncwarp();
        if (lane == 0)
            mbar_arrive(empty + 8 * (p & 1));
        if ((close_in -= 2) < 2 || p + 1 == E) {
            close_in = close_every;
            widen();
        }
    }
}

// ---------------------------------------------------------------------------
// The table: one warp per (DM tile, group), in two launches.  A lane has two of
// the tile's DMs, then one of the group's patterns (64 DMs and 24 patterns in
// one thread took 120 us for a table of any size, against 12 us for 1 MB and 26 us
// for 11 MB).
// ---------------------------------------------------------------------------

constexpr int kPrepThreads = 128;
static_assert(kGroupDmCta == 64 && kGroupTuples <= 32, "two DMs, one pattern a lane");

// Channels of one group: reference (smallest delay) first, so that every
// delta_i is >= 0 (the shift rule is monotone in the delay).
struct GroupChans {
    float ds[kGroupMax];
    int chan[kGroupMax];
    int n;
};

__device__ GroupChans chans_of(const GroupPrep &a, int g) {
    GroupChans c;
    c.n = max(0, min(a.G, a.nchan - g * a.G));
    c.ds[0] = 0.0f;
    int ref = 0;
    for (int i = 0; i < c.n; ++i) {
        c.chan[i] = g * a.G + i;
        c.ds[i] = a.dmshift[c.chan[i]];
        if (c.ds[i] < c.ds[ref])
            ref = i;
    }
    if (ref > 0) {
        const float d0 = c.ds[0];
        const int c0 = c.chan[0];
        c.ds[0] = c.ds[ref];
        c.chan[0] = c.chan[ref];
        c.ds[ref] = d0;
        c.chan[ref] = c0;
    }
    return c;
}

// Offsets e_1.. of a DM, four bits a channel; bad if one does not fit.
__device__ uint32_t pattern_key(const GroupChans &c, float dm, int s0, const int *dmin, bool *bad) {
    uint32_t key = 0;
    for (int i = 1; i < c.n; ++i) {
        const int e = shift_of(dm, c.ds[i]) - s0 - dmin[i];
        if (e < 0 || e > 15)
            *bad = true;
        key |= (uint32_t)(e & 15) << (4 * i);
    }
    return key;
}
__device__ uint32_t nibble(uint32_t key, int i) { return (key >> (4 * i)) & 15u; }

// Records and words of each group, as if its arrays came first; sizes: bytes
// of its arrays.
__global__ void __launch_bounds__(kPrepThreads) group_prep_kernel(const GroupPrep a, int *sizes) {
    constexpr uint32_t kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int td = blockIdx.y, g = (blockIdx.x * kPrepThreads + threadIdx.x) / 32;
    const int np = ((a.nchan + a.G - 1) / a.G + 1) / 2, ng = 2 * np;
    if (g >= ng)
        return;
    const float *dm = a.dm_sorted + (int64_t)td * kGroupDmCta;
    GroupEntry *tile = a.entries + (int64_t)td * np;
    GroupRecord &rec = tile[g / 2].g[g & 1];
    const GroupChans c = chans_of(a, g);
    const float dms[2] = {dm[lane], dm[lane + 32]};
    int s0[2], dmin[kGroupMax], smax[kGroupMax];
    for (int h = 0; h < 2; ++h)
        s0[h] = shift_of(dms[h], c.ds[0]);
    for (int i = 0; i < c.n; ++i) {
        const int sa = shift_of(dms[0], c.ds[i]), sb = shift_of(dms[1], c.ds[i]);
        dmin[i] = __reduce_min_sync(kAll, min(sa - s0[0], sb - s0[1]));
        smax[i] = __reduce_max_sync(kAll, max(sa, sb));
    }
    const int ub = __reduce_min_sync(kAll, min(s0[0], s0[1])) & ~3;  // u = 0
    bool bad = false;
    uint32_t key[2];
    for (int h = 0; h < 2; ++h)
        key[h] = pattern_key(c, dms[h], s0[h], dmin, &bad);
    // The patterns, ordered by key, so that neighbours fit a class; lane t has
    // pattern t: key and range of reference shifts.
    uint32_t tkey = 0;
    int lo = 0, hi = 0, nt = 0;
    bool open[2] = {true, true};
    while (__any_sync(kAll, open[0] || open[1])) {
        const uint32_t next =
            __reduce_min_sync(kAll, min(open[0] ? key[0] : kAll, open[1] ? key[1] : kAll));
        int l = 0x7fffffff, m = -1;
        for (int h = 0; h < 2; ++h)
            if (open[h] && key[h] == next) {
                l = min(l, s0[h] - ub);
                m = max(m, s0[h] - ub);
                open[h] = false;
            }
        l = __reduce_min_sync(kAll, l);
        m = __reduce_max_sync(kAll, m);
        if (nt == kGroupTuples) {
            bad = true;
            break;
        }
        if (lane == nt) {
            tkey = next;
            lo = l;
            hi = m;
        }
        ++nt;
    }
    int phase[kGroupMax];  // byte of the staged row that u = 0 of offset 0 reads
    for (int i = 0; i < a.G; ++i) {
        GroupRow r = {0, 0, 0, -1};
        if (i < c.n) {
            const int start = ub + dmin[i];
            r.first = start & ~15;
            r.bytes = (kGroupTCta + smax[i] - r.first + 15) & ~15;
            r.chan = c.chan[i];
            phase[i] = start - r.first;
            if (start < 0 || r.bytes + 16 > a.rowcap)
                bad = true;
        }
        if (lane == 0)
            rec.rows[i] = r;
    }
    const bool mine = lane < nt;
    lo &= ~3;
    hi = mine ? (hi + kGroupTCta + 3) & ~3 : lo;
    if (hi > 0xffff)
        bad = true;
    const int len = hi - lo;
    int size = 4 * len;  // of the arrays up to this lane's
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
        const int v = __shfl_up_sync(kAll, size, o);
        size += lane >= o ? v : 0;
    }
    const int before = size - 4 * len;
    // Classes: each pattern joins the one before it if their offsets differ by
    // at most 3 all told.  cls: this lane's class, base: its smallest offsets.
    int ncls = 0, cls = -1;
    uint32_t base = 0, emin = 0, emax = 0;
    for (int t = 0; t < nt; ++t) {
        const uint32_t k = __shfl_sync(kAll, tkey, t);
        bool fits = t > 0;
        uint32_t lo2 = 0, hi2 = 0;
        for (int i = 1; i < c.n; ++i) {
            const uint32_t e = nibble(k, i);
            const uint32_t l = min(e, nibble(emin, i)), m = max(e, nibble(emax, i));
            fits = fits && m - l <= 3;
            lo2 |= l << (4 * i);
            hi2 |= m << (4 * i);
        }
        if (!fits) {
            ++ncls;
            lo2 = hi2 = k;
        }
        emin = lo2;
        emax = hi2;
        if (lane == t)
            cls = ncls - 1;
        if (cls == ncls - 1)
            base = emin;
    }
    if (ncls > kGroupClasses)
        bad = true;
    bad = __any_sync(kAll, bad);
    if (bad) {
        if (lane == 0) {
            rec.head = GroupHeader{};
            sizes[(int64_t)td * ng + g] = 0;
            atomicExch(a.fail, 1);
        }
        return;
    }
    GroupHeader h = {};
    for (int k = 0; k < ncls; ++k) {
        const uint32_t in = __ballot_sync(kAll, cls == k);
        h.cnt[k / 4] += (uint32_t)__popc(in) << (8 * (k % 4));
        if (lane == __ffs(in) - 1) {
            GroupClass cl = {};
            for (int i = 0; i < c.n; ++i) {
                const int p = phase[i] + (int)nibble(base, i);
                cl.at[i] = i * a.rowcap + (p & ~3);
                cl.sh[i] = 0x3210u + 0x1111u * (uint32_t)(p & 3);
            }
            rec.cls[k] = cl;
        }
    }
    if (mine) {
        uint32_t e[4];
        for (int i = 1; i < 4; ++i)
            e[i] = nibble(tkey, i) - nibble(base, i);
        GroupTuple &v = rec.tup[lane];
        v.lolen = (uint32_t)lo | (uint32_t)len << 16;
        v.at = before - 2 * lo;
        v.a = 0x32103210u + 0x1111u * e[1] + 0x11110000u * e[2];
        v.b = 0x3210u + 0x1111u * e[3] + (e[1] << 19) + (e[2] << 24) + (e[3] << 29);
    }
    const int top = __reduce_max_sync(kAll, mine ? hi : 0);
    size = __shfl_sync(kAll, size, 31);
    if (lane == 0) {
        h.ncls = ncls;
        h.nt = nt;
        h.nunit = (top + kGroupUnit - 1) / kGroupUnit;
        h.nch = c.n;
        rec.head = h;
        sizes[(int64_t)td * ng + g] = size;
    }
    // The DMs' words (from the group's first array; its place is added below).
    int at[2] = {0, 0};
    for (int t = 0; t < nt; ++t) {
        const uint32_t k = __shfl_sync(kAll, tkey, t);
        const int b = __shfl_sync(kAll, before, t), l = __shfl_sync(kAll, lo, t),
                  n = __shfl_sync(kAll, len, t);
        for (int q = 0; q < 2; ++q)
            if (key[q] == k) {
                const int u = s0[q] - ub - l;
                at[q] = b + (u & 1) * 2 * n + (u >> 1) * 4;
            }
    }
    for (int q = 0; q < 2; ++q)
        tile[g / 2].offs[lane + 32 * q][g & 1] = at[q];
}

// The arrays' places: even pairs from the start of the array space, odd pairs
// up to its end; two neighbours are held at once.
__global__ void __launch_bounds__(kPrepThreads) group_place_kernel(const GroupPrep a,
                                                                   const int *sizes) {
    const int lane = threadIdx.x & 31;
    const int td = blockIdx.y, g = (blockIdx.x * kPrepThreads + threadIdx.x) / 32;
    const int np = ((a.nchan + a.G - 1) / a.G + 1) / 2, ng = 2 * np;
    if (g >= ng)
        return;
    const int *size_of = sizes + (int64_t)td * ng;
    const int space = group_array_bytes(a.G, a.rowcap);
    const int first = size_of[g & ~1], pair = first + size_of[g | 1];
    if (pair + ((g | 1) + 2 < ng ? size_of[(g & ~1) + 2] + size_of[(g | 1) + 2] : 0) > space)
        atomicExch(a.fail, 1);
    const int off = ((g & 2) ? space - pair : 0) + ((g & 1) ? first : 0);
    GroupEntry &ent = a.entries[(int64_t)td * np + g / 2];
    ent.offs[lane][g & 1] += off;
    ent.offs[lane + 32][g & 1] += off;
    if (lane < ent.g[g & 1].head.nt)
        ent.g[g & 1].tup[lane].at += off;
}

}  // namespace

namespace {

// Library streams of a device: tables are built outside the caller's streams
// (and their captures), ahead of CTAs that wait for an SM; their failure flags
// are read on another, so that no flag waits for a later table.
struct TableStreams {
    cudaStream_t build = nullptr, read = nullptr;
};
std::mutex g_table_mu;
TableStreams g_table_streams[64];

bool table_streams(int dev, TableStreams **out) {
    TableStreams &t = g_table_streams[dev];
    int least = 0, greatest = 0;
    *out = &t;
    return (t.build || (cudaDeviceGetStreamPriorityRange(&least, &greatest) == cudaSuccess &&
                        cudaStreamCreateWithPriority(&t.build, cudaStreamNonBlocking, greatest) ==
                            cudaSuccess)) &&
           (t.read ||
            cudaStreamCreateWithFlags(&t.read, cudaStreamNonBlocking) == cudaSuccess);
}

// The attribute of group_kernel that its launches need, set once per device.
cudaError_t configure_group_kernel(int dev) {
    static bool configured[64] = {false};
    bool &conf = configured[dev & 63];
    if (!conf) {
        const cudaError_t e = cudaFuncSetAttribute(
            group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGroupSmem);
        if (e != cudaSuccess)
            return e;
        conf = true;
    }
    return cudaSuccess;
}

}  // namespace

bool start_group_table(GroupPrep a, int dev, GroupBuild *b) {
    const size_t pairs = (size_t)a.ntile_d * (size_t)(((a.nchan + a.G - 1) / a.G + 1) / 2);
    std::lock_guard<std::mutex> lk(g_table_mu);
    TableStreams *t = nullptr;
    // The table, the groups' sizes, the failure flag (one allocation; freeing a
    // second one would wait for the device).
    const size_t table = sizeof(GroupEntry) * pairs;
    void *mem = nullptr;
    cudaEvent_t done = nullptr;
    bool ok = table_streams(dev, &t) && configure_group_kernel(dev) == cudaSuccess &&
              cudaEventCreateWithFlags(&done, cudaEventDisableTiming) == cudaSuccess &&
              cudaMalloc(&mem, table + sizeof(int) * (2 * pairs + 1)) == cudaSuccess;
    if (ok) {
        a.entries = static_cast<GroupEntry *>(mem);
        int *sizes = reinterpret_cast<int *>(static_cast<uint8_t *>(mem) + table);
        a.fail = sizes + 2 * pairs;
        const unsigned ng = 2 * (unsigned)(pairs / (size_t)a.ntile_d);
        const dim3 grid((ng + kPrepThreads / 32 - 1) / (kPrepThreads / 32), (unsigned)a.ntile_d);
        ok = cudaMemsetAsync(a.fail, 0, sizeof(int), t->build) == cudaSuccess;
        if (ok) {
            group_prep_kernel<<<grid, kPrepThreads, 0, t->build>>>(a, sizes);
            group_place_kernel<<<grid, kPrepThreads, 0, t->build>>>(a, sizes);
            ok = cudaGetLastError() == cudaSuccess &&
                 cudaEventRecord(done, t->build) == cudaSuccess;
        }
    }
    if (!ok) {
        cudaGetLastError();
        cudaFree(mem);
        if (done)
            cudaEventDestroy(done);
        return false;
    }
    b->entries = a.entries;
    b->fail = a.fail;
    b->done = done;
    return true;
}

TableState finish_group_table(GroupBuild *b, int dev, bool wait) {
    if (!wait && cudaEventQuery(b->done) == cudaErrorNotReady) {
        cudaGetLastError();
        return TableState::kUnderWay;
    }
    int failed = 1;
    cudaStream_t s = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_table_mu);
        s = g_table_streams[dev].read;
    }
    if (cudaEventSynchronize(b->done) != cudaSuccess ||
        cudaMemcpyAsync(&failed, b->fail, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        failed = 1;
    cudaEventDestroy(b->done);
    if (failed) {
        cudaGetLastError();
        cudaFree(b->entries);
    }
    *b = GroupBuild();
    return failed ? TableState::kUnusable : TableState::kComplete;
}

cudaError_t launch_group(const GroupArgs &a, unsigned grid, cudaStream_t s) {
    int dev = 0;
    cudaGetDevice(&dev);
    const cudaError_t e = configure_group_kernel(dev);
    if (e != cudaSuccess)
        return e;
    group_kernel<<<grid, kThreads, kGroupSmem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace dd
