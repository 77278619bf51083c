// Host side of grouped execution (dd_group.h): whether it pays, its group size
// and its table.
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "dd_group.h"

namespace dd {
namespace {

// Patterns of sampled (DM tile, group) pairs: 3 tiles x 12 groups spread over
// the plan.
struct Sample {
    double nt = 0;      // patterns of a group
    double reach = 0;   // reference shifts a pattern spans (samples)
    double spread = 0;  // reference shifts a tile spans
    double bytes = 0;   // of the arrays of the largest group sampled
    bool fits = true;
};

Sample sample_patterns(const dd_plan_s *p, int G) {
    Sample r;
    const int ntile = (p->ndm + kGroupDmCta - 1) / kGroupDmCta;
    const int ng = (p->nchan + G - 1) / G;
    const int nst = std::min(ntile, 3), nsg = std::min(ng, 12);
    double patterns = 0;
    for (int it = 0; it < nst; ++it) {
        const int td = nst > 1 ? (int)((int64_t)it * (ntile - 1) / (nst - 1)) : 0;
        for (int ig = 0; ig < nsg; ++ig) {
            const int c0 = G * (nsg > 1 ? (int)((int64_t)ig * (ng - 1) / (nsg - 1)) : 0);
            const int n = std::min(G, p->nchan - c0);
            const float *ds = &p->dmshift[(size_t)c0];
            const int ref = (int)(std::min_element(ds, ds + n) - ds);
            int64_t keys[kGroupTuples];
            int lo[kGroupTuples], hi[kGroupTuples], nt = 0, s_lo = 0x7fffffff, s_hi = 0;
            for (int k = 0; k < kGroupDmCta; ++k) {
                const float dm = p->dm_sorted[(size_t)std::min(td * kGroupDmCta + k, p->ndm - 1)];
                const int s0 = trunc_product(dm, ds[ref]);
                int64_t key = 0;
                for (int i = 0; i < n; ++i)
                    key = key << 15 | ((trunc_product(dm, ds[i]) - s0) & 0x7fff);
                int t = nt;
                while (t > 0 && keys[t - 1] != key)
                    --t;
                if (t == 0) {
                    if (nt == kGroupTuples) {
                        r.fits = false;
                        return r;
                    }
                    keys[nt] = key;
                    lo[nt] = hi[nt] = s0;
                    t = ++nt;
                }
                lo[t - 1] = std::min(lo[t - 1], s0);
                hi[t - 1] = std::max(hi[t - 1], s0);
                s_lo = std::min(s_lo, s0);
                s_hi = std::max(s_hi, s0);
            }
            double reach = 0;
            for (int t = 0; t < nt; ++t)
                reach += hi[t] - lo[t];
            r.reach += reach;
            r.bytes = std::max(r.bytes, 4.0 * (nt * kGroupTCta + reach));
            patterns += nt;
            r.spread += s_hi - s_lo;
        }
    }
    r.reach /= patterns;
    r.nt = patterns / (nst * nsg);
    r.spread /= nst * nsg;
    return r;
}

// Clocks per channel and tile.  The users read 2 bytes per DM, sample and
// group; the builders' work, counted in their shared-memory wavefronts, takes
// 3.9 clocks each.  Fitted to nine beams of 256 .. 4096 channels, 493 .. 802
// clocks, within 5 %.
double group_clocks(const Sample &s, int G) {
    const double users = 2.0 * kGroupDmCta * kGroupTCta / 128 / G;
    const double units = (kGroupTCta + s.spread) / 128;
    const double arrays = s.nt * ((kGroupTCta + s.reach) / 128 + 0.5);
    return users + 3.9 * (3 * units + 4.5 * arrays / G + units);
}

// Prologue and epilogue of a tile, clocks.
constexpr double kTileClocks = 10000;
constexpr double kClocksPerUs = 2070;
// Executions shorter than this by the direct kernel stay with it: a table costs
// more than shorter beams gain in many.
constexpr double kLeastUs = 100.0;
// The patterns are sampled before an execution only if it is longer than this;
// behind a shorter one otherwise.
constexpr double kSampleUs = 1000.0;

// The grouped form of the plan on device dev, its patterns sampled.  Caller
// holds p->mu.
GroupShape &shape_of(dd_plan_s *p, int dev) {
    auto it = p->group.find(dev);
    if (it != p->group.end())
        return *it->second;
    auto r = std::make_shared<GroupShape>();
    r->ntile_d = (p->ndm + kGroupDmCta - 1) / kGroupDmCta;
    // A staged window: the tile, its DMs' spread in the most delayed
    // channel, the 16-byte rounding at both ends and the samples by which
    // smallest shifts of channels disagree.
    double spread = 0;
    const double most = *std::max_element(p->dmshift.begin(), p->dmshift.end());
    for (int a = 0; a < p->ndm; a += kGroupDmCta)
        spread = std::max(
            spread, most * ((double)p->dm_sorted[(size_t)std::min(a + kGroupDmCta, p->ndm) - 1] -
                            (double)p->dm_sorted[(size_t)a]));
    if (spread < 8192) {
        r->rowcap = (kGroupTCta + (int)spread + 64 + 15) / 16 * 16;
        for (int G : {4, 3}) {
            const Sample s = sample_patterns(p, G);
            // Four groups' arrays are held at once.
            if (s.fits && kGroupRaw * group_raw_bytes(G, r->rowcap) < kGroupSmem / 2 &&
                4.0 * s.bytes < group_array_bytes(G, r->rowcap))
                r->sizes.push_back({G, group_clocks(s, G)});
        }
        std::sort(r->sizes.begin(), r->sizes.end(),
                  [](const auto &x, const auto &y) { return x.clk < y.clk; });
    }
    return *p->group.emplace(dev, r).first->second;
}

void start(dd_plan_s *p, int dev, const DevTables &dt, GroupShape &r) {
    while (!r.table.entries && !r.build.entries && !r.sizes.empty()) {
        GroupPrep a{};
        a.dmshift = dt.dmshift;
        a.dm_sorted = dt.dm_sorted;
        a.nchan = p->nchan;
        a.ntile_d = r.ntile_d;
        a.G = r.sizes[0].G;
        a.rowcap = r.rowcap;
        // The table is built on a stream of the library's, so a capture of
        // the caller's stream does not see it.
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        cudaThreadExchangeStreamCaptureMode(&mode);
        const bool ok = start_group_table(a, dev, &r.build);
        cudaThreadExchangeStreamCaptureMode(&mode);
        if (!ok)  // no memory for it
            r.sizes.erase(r.sizes.begin());
    }
}

// Take in a table under way; waited for if `wait`.
void poll(dd_plan_s *p, int dev, GroupShape &r, bool wait) {
    if (!r.build.entries)
        return;
    GroupEntry *entries = r.build.entries;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    const TableState st = finish_group_table(&r.build, dev, wait);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (st == TableState::kUnusable) {  // the sampled groups fitted, others do not
        r.sizes.erase(r.sizes.begin());
    } else if (st == TableState::kComplete) {
        const int G = r.sizes[0].G;
        r.table = {G, ((p->nchan + G - 1) / G + 1) / 2, r.ntile_d, r.rowcap, entries};
        r.sizes.resize(1);
    }
}

double tile_us(const dd_plan_s *p, const GroupShape &r) {
    return (p->nchan * r.sizes[0].clk + kTileClocks) / kClocksPerUs;
}

// The preferred tile shape stands for the library's choice; another shape set
// by the caller, or timed by the autotuner, runs as such.
bool may_group(dd_dtype t, const Geometry &g) {
    const dd_tiles pref = default_tiles(DD_U8);
    return t == DD_U8 && (g.chosen || std::memcmp(&pref, &g.tiles, sizeof(pref)) == 0);
}

// Whether an execution alone on the device, of `direct` us by the direct kernel,
// gains enough by groups: *grouped us, in rounds of tiles over the SMs.
bool gains(dd_plan_s *p, int dev, double direct, int64_t nsamp_out, GroupEstimate *e,
           double *grouped) {
    const int sms = sm_count(dev);
    if (!group_estimate(p, dev, nsamp_out, e))
        return false;
    *grouped = (double)((e->tiles + sms - 1) / sms) * e->tile_us;
    return *grouped <= kGroupGain * direct;
}

}  // namespace

bool group_sampled(dd_plan_s *p, int dev) {
    std::lock_guard<std::mutex> lk(p->mu);
    return p->group.count(dev) != 0;
}

bool group_estimate(dd_plan_s *p, int dev, int64_t nsamp_out, GroupEstimate *e) {
    std::lock_guard<std::mutex> lk(p->mu);
    GroupShape &r = shape_of(p, dev);
    poll(p, dev, r, false);
    if (r.sizes.empty())
        return false;
    e->tile_us = tile_us(p, r);
    e->tiles = group_tiles(r.ntile_d, nsamp_out);
    e->ready = r.table.entries != nullptr;
    return true;
}

void group_start(dd_plan_s *p, int dev, const DevTables &dt) {
    std::lock_guard<std::mutex> lk(p->mu);
    start(p, dev, dt, shape_of(p, dev));
}

bool group_ready(dd_plan_s *p, int dev, const DevTables &dt, bool now, GroupTable *out) {
    std::lock_guard<std::mutex> lk(p->mu);
    GroupShape &r = shape_of(p, dev);
    poll(p, dev, r, now);
    while (now && !r.table.entries && !r.sizes.empty()) {
        start(p, dev, dt, r);
        poll(p, dev, r, true);
    }
    *out = r.table;
    return out->entries != nullptr;
}

GroupRoute group_route(dd_plan_s *p, dd_dtype t, const Geometry &g, const DevTables &dt,
                       int64_t nsamp_out, bool now, cudaStream_t stream, GroupTable *out) {
    int dev = 0;
    if (!may_group(t, g) || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return GroupRoute::kDirect;
    const int sms = sm_count(dev);
    const double direct = sms > 0 ? direct_time_us(p, t, g.tiles, nsamp_out, sms) : -1.0;
    if (direct < kLeastUs)
        return GroupRoute::kDirect;
    auto captured = [&]() {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &cap) != cudaSuccess)
            cudaGetLastError();
        return cap != cudaStreamCaptureStatusNone;
    };
    if (!now && direct < kSampleUs && !group_sampled(p, dev) && !(now = captured()))
        return GroupRoute::kLater;
    // (Again if a table turns out unusable: another group size may serve.)
    GroupEstimate e;
    double grouped = 0;
    while (gains(p, dev, direct, nsamp_out, &e, &grouped)) {
        const bool wait = !e.ready && (now || direct - grouped > kGroupTableUs || captured());
        if (!e.ready && !wait)
            return GroupRoute::kLater;
        if (group_ready(p, dev, dt, wait, out))
            return GroupRoute::kGrouped;
    }
    return GroupRoute::kDirect;
}

// Whether it would be grouped if its table were there.
static bool would_group(dd_plan_s *p, dd_dtype t, const Geometry &g, int64_t nsamp_out, int *dev,
                        GroupEstimate *e) {
    if (!may_group(t, g) || cudaGetDevice(dev) != cudaSuccess || *dev < 0 || *dev >= 64)
        return false;
    const int sms = sm_count(*dev);
    const double direct = sms > 0 ? direct_time_us(p, t, g.tiles, nsamp_out, sms) : -1.0;
    double grouped = 0;
    return direct >= kLeastUs && gains(p, *dev, direct, nsamp_out, e, &grouped);
}

void group_later(dd_plan_s *p, dd_dtype t, const Geometry &g, const DevTables &dt,
                 int64_t nsamp_out) {
    int dev = 0;
    GroupEstimate e;
    if (would_group(p, t, g, nsamp_out, &dev, &e) && !e.ready)
        group_start(p, dev, dt);
}

bool group_taken(dd_plan_s *p, dd_dtype t, const Geometry &g, int64_t nsamp_out,
                 GroupTable *out) {
    int dev = 0;
    GroupEstimate e;
    return would_group(p, t, g, nsamp_out, &dev, &e) && e.ready &&
           group_ready(p, dev, DevTables(), false, out);
}

void group_free(dd_plan_s *p) {
    for (auto &kv : p->group) {
        cudaSetDevice(kv.first);
        GroupEntry *building = kv.second->build.entries;
        if (building &&
            finish_group_table(&kv.second->build, kv.first, true) == TableState::kComplete)
            cudaFree(building);
        cudaFree(kv.second->table.entries);
    }
    p->group.clear();
}

GroupBeam group_beam(const GroupTable &g, const DevTables &dt, const void *in, int64_t in_pitch,
                     int64_t nsamp_in, float *out, int64_t out_pitch, int64_t nsamp_out) {
    GroupBeam b{};
    b.in = static_cast<const uint8_t *>(in);
    b.in_pitch_b = in_pitch;
    b.nsamp_in = nsamp_in;
    b.out = out;
    b.out_pitch = out_pitch;
    b.nsamp_out = nsamp_out;
    b.perm = dt.perm;
    b.entries = g.entries;
    b.ntile_d = g.ntile_d;
    b.npairs = g.npairs;
    b.G = g.G;
    b.rowcap = g.rowcap;
    return b;
}

}  // namespace dd

extern "C" int dd_plan_groups(dd_plan_t p, int64_t nsamp_out) {
    int dev = 0;
    dd::Geometry g;
    dd::GroupTable gs;
    if (!p || nsamp_out < 1 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 ||
        !dd::group_sampled(p, dev) ||
        dd::execution_geometry(p, DD_U8, nsamp_out, &g) != DD_OK)
        return 0;
    return dd::group_taken(p, DD_U8, g, nsamp_out, &gs) ? gs.G : 0;
}
