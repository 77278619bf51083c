// Channel groups (uint8): partial sums over adjacent channels shared by trial
// DMs.
//
// Let a group be G adjacent channels with reference channel 0 (the one with
// the smallest delay).  The shift of channel i relative to the reference,
// delta_i(d) = s(c_i,d) - s(c_0,d), grows slowly with the DM, so the DMs of a
// tile have few distinct patterns (delta_1, ..., delta_{G-1}): 4.5 on average
// among 64 DMs for 4 channels of the 4096-channel low-frequency beam.  The sum
// of the group's channels for one pattern,
//     A_p[u] = sum_i in[c_i][u + delta_i],
// is formed once per tile and read by every DM with that pattern at its
// reference shift: out[d][t] += A_{p(d)}[t + s(c_0,d)].  The same integers
// are added in another order, so the sums stay exact.
//
// This header: the tables that describe the patterns of every (DM tile,
// group), built on the device once per plan (they do not depend on time,
// because every tile starts at a multiple of 16 samples; 2 KB per tile and pair of
// groups), and the arguments of the kernel that uses them (dd_group.cu).
#pragma once

#include <cuda_runtime_api.h>

#include <cstdint>
#include <vector>

#include "dd_internal.h"

namespace dd {

constexpr int kGroupUsers = 8;      // warps that own DMs (168 registers a thread)
constexpr int kGroupBuilders = 11;  // warps that build pattern arrays, and one that fetches
                                    // (48 registers a thread)
constexpr int kGroupDms = 8;        // DMs per user thread
constexpr int kGroupWords = 16;     // words per DM and user thread (32 samples)
constexpr int kGroupDmCta = kGroupUsers * kGroupDms;  // DMs of a tile
constexpr int kGroupTCta = 64 * kGroupWords;          // samples of a tile
constexpr int kGroupMax = 4;        // channels per group, at most
constexpr int kGroupRaw = 3;        // pairs of groups whose channel windows are staged at once
constexpr int kGroupOffs = 8;       // pairs whose DM offsets are held at once
constexpr int kGroupUnit = 128;     // samples of a build unit (32 lanes x 4)
constexpr int kGroupClasses = 8;    // classes of patterns of a group, at most
constexpr int kGroupTuples = 24;    // patterns of a group, at most

struct GroupHeader {  // 32 bytes
    int nt;           // patterns
    int nunit;        // build units covering every pattern's array
    int pad0;
    int nch;          // channels (fewer than G in the last group, 0 in an empty one)
    int ncls;         // classes, and the patterns of each, a byte each
    uint32_t cnt[2];
    int pad1;
};
struct GroupRow {     // 16 bytes: one channel's staged window
    int first;        // its first byte relative to the tile's t0 (a multiple of 16)
    int bytes;        // bytes from there, rounded up to 16
    int pad;
    int chan;         // -1: none
};
// Patterns whose offsets e_i = delta_i - min delta_i differ by at most 3 in
// every channel form a class.  A build lane holds each channel's 8 bytes from
// the class's smallest offset on; a pattern's window then starts 0..3 bytes
// further, within a byte permute's reach.
struct GroupClass {   // 32 bytes
    int at[4];        // byte of the group's staged rows that u = 0 reads, word-aligned
    uint32_t sh[4];   // permute selector of the remaining 0..3 bytes
};
// A pattern: its array covers u in [lo, lo + len) (multiples of 4; u = sample
// relative to the tile's smallest reference shift, rounded down to 4).  Two
// copies, one sample apart, of packed 16-bit sums, the second 2 * len bytes
// after the first.
struct GroupTuple {   // 16 bytes
    uint32_t lolen;   // lo | len << 16
    int at;           // byte of the array space that u = 0 would have
    uint32_t a;       // permute selectors of channels 1, 2 << 16
    uint32_t b;       // selector of channel 3; 8 * offset in the class of channels 1, 2,
                      // 3 in the five bits from bit 16, 21, 26
};
// A group's record.
struct GroupRecord {
    GroupHeader head;
    GroupRow rows[kGroupMax];
    GroupClass cls[kGroupClasses];
    GroupTuple tup[kGroupTuples];
};
// One table entry = one (DM tile, pair of groups).  With an odd number of
// groups the last pair's second group is empty: one pattern, all zeros.
struct GroupEntry {
    GroupRecord g[2];
    int offs[kGroupDmCta][2];  // per DM: its words in both groups' arrays (array-space bytes)
};
static_assert(sizeof(GroupRecord) % 16 == 0 && sizeof(GroupEntry) % 16 == 0,
              "records are copied 16 bytes at a time");

// One beam of a grouped launch.
struct GroupBeam {
    const uint8_t *in;
    int64_t in_pitch_b;
    int64_t nsamp_in;
    float *out;
    int64_t out_pitch;
    int64_t nsamp_out;
    const int *perm;            // sorted DM -> output row, -1 for padding
    const GroupEntry *entries;  // [ntile_d][npairs]
    int64_t tile_begin;
    int ntile_d;
    int npairs;
    int G;
    int rowcap;                 // bytes of a staged row
};

struct GroupArgs {
    GroupBeam beam0;
    const GroupBeam *beams;     // NULL: beam0 only
    int nbeams;
    int *status;
};

// A table being built on a library stream.
struct GroupBuild {
    GroupEntry *entries = nullptr;
    int *fail = nullptr;  // 1 on the device when a limit does not hold (table unusable)
    cudaEvent_t done = nullptr;
};

// A complete table, as an execution uses it.
struct GroupTable {
    int G = 0, npairs = 0, ntile_d = 0, rowcap = 0;
    GroupEntry *entries = nullptr;
};

// Grouped execution of a plan on one device.
struct GroupShape {
    int ntile_d = 0, rowcap = 0;
    // Group sizes that may serve, best first: channels, modelled SM clocks per
    // channel and tile.  Once a table is built, its size is the only one.
    struct Size {
        int G;
        double clk;
    };
    std::vector<Size> sizes;
    GroupBuild build;               // of sizes[0], under way if build.entries
    GroupTable table;               // complete if table.entries
};

// Shared memory of a grouped CTA: kGroupRaw raw slots, then the array space.
constexpr int kGroupSmem = kMaxSmem - 5120;  // less the static barriers and offsets
DD_HD constexpr int group_raw_bytes(int G, int rowcap) {
    return (2 * (int)sizeof(GroupRecord) + 2 * G * rowcap + 127) / 128 * 128;
}
// The last 512 bytes are not used: a unit may read that far past a row's end.
DD_HD constexpr int group_array_bytes(int G, int rowcap) {
    return (kGroupSmem - kGroupRaw * group_raw_bytes(G, rowcap) - 512) & ~127;
}

struct GroupPrep {  // arguments of the table builder
    const float *dmshift, *dm_sorted;
    int nchan, ntile_d, G, rowcap;
    GroupEntry *entries;
    int *fail;  // set to 1 when a limit does not hold (table unusable)
};

// Start to build the table described by a (a.entries and a.fail are set here)
// on a library stream of device dev; false, with nothing held, when the device
// memory cannot be had.
bool start_group_table(GroupPrep a, int dev, GroupBuild *b);
// Its state: under way (only if not waited for), complete, or unusable (then
// nothing is held).
enum class TableState { kUnderWay, kComplete, kUnusable };
TableState finish_group_table(GroupBuild *b, int dev, bool wait);

// What an execution of nsamp_out samples takes in the plan's grouped form: the
// time of a tile (microseconds), its tiles and whether the table is there.
struct GroupEstimate {
    double tile_us = 0;
    int64_t tiles = 0;
    bool ready = false;
};
// Whether the plan's patterns have been sampled.
bool group_sampled(dd_plan_s *p, int dev);
// False: no group size serves the plan.  Samples the plan's patterns on first
// use (host work of some 30 us); polls a table under way.
bool group_estimate(dd_plan_s *p, int dev, int64_t nsamp_out, GroupEstimate *e);
// Start the table of the best group size if it is neither there nor under way.
void group_start(dd_plan_s *p, int dev, const DevTables &dt);
// The plan's grouped form, once its table is there: waited for, or started and
// waited for (now), or left if not.
bool group_ready(dd_plan_s *p, int dev, const DevTables &dt, bool now, GroupTable *out);

// Grouped execution is taken when it is expected to gain this much: the model
// is good to about 5 %.
constexpr double kGroupGain = 0.95;
// What a table costs before an execution can use it: sampling, an allocation,
// two launches and a wait (microseconds).
constexpr double kGroupTableUs = 200.0;

// How one execution by dd_execute runs: by the direct kernel, by the direct
// kernel with the table to be started behind it (kGroupLater: the execution
// would gain less than the table costs it), or by the grouped kernel (*out).
// It waits for a table in any case with `now` (the autotuner) or while `stream`
// is being captured (the graph keeps what it captures).
enum class GroupRoute { kDirect, kLater, kGrouped };
GroupRoute group_route(dd_plan_s *p, dd_dtype t, const Geometry &g, const DevTables &dt,
                       int64_t nsamp_out, bool now, cudaStream_t stream, GroupTable *out);
// Whether an execution would take the grouped kernel as things stand (*out).
bool group_taken(dd_plan_s *p, dd_dtype t, const Geometry &g, int64_t nsamp_out,
                 GroupTable *out);
// After a kLater launch: start the table if the plan's next execution of this
// length would take it.
void group_later(dd_plan_s *p, dd_dtype t, const Geometry &g, const DevTables &dt,
                 int64_t nsamp_out);
void group_free(dd_plan_s *p);

GroupBeam group_beam(const GroupTable &g, const DevTables &dt, const void *in, int64_t in_pitch,
                     int64_t nsamp_in, float *out, int64_t out_pitch, int64_t nsamp_out);
inline int64_t group_tiles(int ntile_d, int64_t nsamp_out) {
    return (nsamp_out + kGroupTCta - 1) / kGroupTCta * ntile_d;
}
cudaError_t launch_group(const GroupArgs &a, unsigned grid, cudaStream_t s);

}  // namespace dd
