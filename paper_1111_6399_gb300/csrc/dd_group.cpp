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
            for (int t = 0; t < nt; ++t)
                r.reach += hi[t] - lo[t];
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
// Grouped execution is taken when it is expected to gain this much: the model
// is good to about 5 %.
constexpr double kGain = 0.95;

}  // namespace

bool group_shape(dd_plan_s *p, dd_dtype t, const Geometry &g, const DevTables &dt,
                 int64_t nsamp_out, bool alone, GroupShape *out) {
    // The preferred tile shape stands for the library's choice; another shape
    // set by the caller, or timed by the autotuner, runs as such.
    const dd_tiles pref = default_tiles(DD_U8);
    int dev = 0;
    if (t != DD_U8 || (std::memcmp(&pref, &g.tiles, sizeof(pref)) != 0 && !g.chosen) ||
        cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return false;
    const int sms = sm_count(dev);
    const int64_t tiles = (nsamp_out + g.t_cta - 1) / g.t_cta * g.ntile_d;
    if (sms <= 0)
        return false;
    // Time of the direct kernel: in rounds of tiles over the SMs, or, as one of
    // many beams, its share of them (of the time of one tile's round).
    const double direct = alone ? direct_time_us(p, t, g.tiles, nsamp_out, sms)
                                : direct_tile_us(p, t, g.tiles) * (double)tiles / sms;
    // A table costs a plan's first execution about 110 us (35 of them for the
    // samples below), more than shorter beams gain in many.
    if (direct < (alone ? 100.0 : 0.0))
        return false;
    std::lock_guard<std::mutex> lk(p->mu);
    auto it = p->group.find(dev);
    if (it == p->group.end()) {
        auto r = std::make_shared<GroupShape>();
        r->ntile_d = (p->ndm + kGroupDmCta - 1) / kGroupDmCta;
        // A staged window: the tile, its DMs' spread in the most delayed
        // channel, the 16-byte rounding at both ends and the samples by which
        // smallest shifts of channels disagree.
        double spread = 0;
        const double most = *std::max_element(p->dmshift.begin(), p->dmshift.end());
        for (int a = 0; a < p->ndm; a += kGroupDmCta)
            spread = std::max(
                spread,
                most * ((double)p->dm_sorted[(size_t)std::min(a + kGroupDmCta, p->ndm) - 1] -
                        (double)p->dm_sorted[(size_t)a]));
        if (spread < 8192) {
            r->rowcap = (kGroupTCta + (int)spread + 64 + 15) / 16 * 16;
            for (int G : {4, 3}) {
                const Sample s = sample_patterns(p, G);
                // Four groups' arrays are held at once.
                if (s.fits && kGroupRaw * group_raw_bytes(G, r->rowcap) < kGroupSmem / 2 &&
                    16.0 * s.nt * (kGroupTCta + s.reach) < group_array_bytes(G, r->rowcap)) {
                    r->sizes.push_back({G, group_clocks(s, G)});
                }
            }
            std::sort(r->sizes.begin(), r->sizes.end(),
                      [](const auto &x, const auto &y) { return x.clk < y.clk; });
        }
        it = p->group.emplace(dev, r).first;
    }
    GroupShape &r = *it->second;
    const double n = (double)group_tiles(r, nsamp_out) / sms;
    while (!r.sizes.empty() &&
           (alone ? std::ceil(n) : n) * (p->nchan * r.sizes[0].clk + kTileClocks) / kClocksPerUs <=
               kGain * direct) {
        if (!r.entries) {
            GroupPrep a;
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
            r.entries = build_group_table(a, dev);
            cudaThreadExchangeStreamCaptureMode(&mode);
            if (!r.entries) {  // the sampled groups fitted, others do not
                r.sizes.erase(r.sizes.begin());
                continue;
            }
            r.G = a.G;
            r.npairs = ((p->nchan + r.G - 1) / r.G + 1) / 2;
            r.sizes.resize(1);
        }
        *out = r;
        return true;
    }
    return false;
}

void group_free(dd_plan_s *p) {
    for (auto &kv : p->group) {
        cudaSetDevice(kv.first);
        cudaFree(kv.second->entries);
    }
    p->group.clear();
}

GroupBeam group_beam(const GroupShape &g, const DevTables &dt, const void *in, int64_t in_pitch,
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
