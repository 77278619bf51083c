// Which tile shape an execution takes while the caller and the autotuner have
// set none: the listed shape with the least modelled time.
//
// A launch runs in rounds of tiles over the SMs.  Large beams take the shape of
// the least time per output (the preferred one, or one DM column more where
// that saves a round), small ones a shape whose tiles are all resident at once,
// wide windows (coarse DM steps, low frequencies) a shape whose ring still has
// three stages.  With the preferred shape alone, 64 channels x 64 DMs x 8192
// samples took 29 us (16 CTAs on 152 SMs) against 15, and 512 x 200 x 8192 took
// 153 against 71.
//
// A batch or a server has one shape for all its beams: the one in which their
// tiles, largest beams first, are expected to keep the SMs busy for the least
// time.  Eight FP32 beams of 1024 channels x 24 DMs x 16384 samples took 888 us
// in 48-DM tiles, half of them padding, against 575 in 24-DM tiles.
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstring>

#include "dd_internal.h"

namespace dd {
namespace {

// Time of one round of tiles (`resident` CTAs on every SM) at 64 and 512
// channels in microseconds: each shape run for 8 rounds on a 300 MHz band at
// 1.5 GHz with unit DM steps, where its ring has three stages or more.  The
// first of a type is the preferred one.  The wide ones (fewer channels a stage,
// or fewer DMs and more time) stand by for windows of which the preferred
// shape's ring holds less than three stages.
struct ShapeCost {
    dd_tiles tiles;
    int resident;
    double us64, us512;
    bool wide = false;
};
const std::vector<ShapeCost> &shape_costs(dd_dtype t) {
    static const std::vector<ShapeCost> u8 = {
        {{4, 12, 1, 8, 8}, 1, 25.2, 155.0},  {{4, 13, 1, 8, 8}, 1, 26.8, 163.7},
        {{4, 8, 1, 8, 8}, 1, 21.1, 118.8},   {{2, 16, 1, 8, 8}, 1, 19.3, 110.0},
        {{2, 13, 1, 8, 8}, 1, 17.3, 98.0},   {{2, 8, 1, 12, 8}, 1, 15.0, 76.4},
        {{4, 8, 1, 16, 4}, 1, 14.8, 72.8},   {{2, 16, 1, 16, 4}, 1, 14.3, 75.1},
        {{2, 13, 1, 16, 4}, 1, 12.8, 66.3},  {{2, 8, 1, 16, 4}, 1, 11.8, 60.4},
        {{1, 8, 1, 16, 4}, 1, 10.8, 58.0},
        {{4, 12, 1, 4, 8}, 1, 28.7, 185.0, true}, {{4, 6, 2, 4, 8}, 1, 29.1, 189.0, true},
        {{4, 3, 4, 4, 8}, 1, 34.0, 224.0, true},  {{4, 1, 4, 4, 8}, 1, 25.5, 163.0, true}};
    static const std::vector<ShapeCost> f16 = {
        {{4, 12, 1, 12, 8}, 1, 24.0, 133.0}, {{4, 8, 1, 12, 8}, 1, 19.3, 100.6},
        {{2, 8, 1, 16, 8}, 1, 13.9, 75.6},   {{4, 8, 1, 16, 4}, 1, 13.8, 72.4},
        {{2, 16, 1, 16, 4}, 1, 13.8, 80.9},  {{2, 8, 1, 16, 4}, 1, 11.2, 64.6},
        {{1, 8, 1, 16, 4}, 2, 11.5, 69.0},   {{1, 12, 1, 16, 8}, 1, 13.5, 74.7},
        {{4, 6, 2, 8, 8}, 1, 24.4, 147.0, true}, {{4, 6, 2, 4, 8}, 1, 27.7, 177.0, true},
        {{4, 3, 4, 4, 8}, 1, 27.7, 178.0, true}, {{4, 1, 8, 4, 8}, 1, 30.5, 191.5, true},
        {{1, 6, 3, 8, 8}, 1, 18.8, 111.4, true}};
    static const std::vector<ShapeCost> f32 = {
        {{4, 12, 1, 16, 8}, 1, 18.6, 113.4}, {{4, 6, 2, 16, 8}, 1, 18.4, 112.7},
        {{4, 13, 1, 12, 8}, 1, 23.0, 128.8}, {{4, 10, 1, 16, 8}, 1, 16.2, 95.5},
        {{4, 8, 1, 16, 8}, 1, 14.5, 81.6},   {{2, 16, 1, 16, 8}, 1, 14.0, 85.8},
        {{2, 8, 1, 16, 8}, 1, 10.5, 61.5},   {{2, 8, 1, 24, 4}, 1, 9.2, 52.0},
        {{1, 8, 1, 24, 4}, 2, 9.8, 54.0},    {{2, 12, 1, 16, 8}, 1, 12.6, 73.4},
        {{4, 6, 2, 8, 8}, 1, 18.7, 117.3, true}, {{4, 3, 4, 8, 8}, 1, 18.8, 116.9, true},
        {{4, 3, 4, 4, 8}, 1, 22.9, 153.0, true}, {{4, 1, 13, 4, 8}, 1, 23.6, 153.0, true},
        {{2, 1, 16, 4, 8}, 1, 21.5, 142.5, true}};
    return t == DD_U8 ? u8 : t == DD_F16 ? f16 : f32;
}

// A ring of two stages exposes part of every stage's copy and phase building:
// with a stage of `us` otherwise, about this much more.  uint8, 256 channels:
// (4,12,1,8,8) 79 -> 99 us, (2,16,1,8,8) 60 -> 85, (4,1,4,4,8) 81 -> 137; FP16:
// (4,12,1,12,8) 75 -> 86, (4,3,4,4,8) 99 -> 149.  FP32 has no phases to build:
// (4,12,1,16,8) none, (4,1,13,4,8) 83 -> 103.
double two_stages_us(dd_dtype t, double us) {
    return t == DD_F32 ? std::max(0.0, 1.55 - us) : std::max(0.45, 1.3 - 0.3 * us);
}
// A tile of a shape with two CTAs on an SM takes this share of their round where
// its windows leave room for one (FP16 (1,8,1,16,4), 512 channels: 73 us for
// two, 61 alone).
constexpr double kAlone = 0.88;

// Ring stages (0: its windows do not fit) and CTAs on an SM of listed shape i,
// from the DM steps and the largest delay where those decide, else from every
// window.  Caller holds p->mu.
const ShapeFit &shape_fit(dd_plan_s *p, dd_dtype t, int i) {
    std::vector<ShapeFit> &fits = p->shape_fit[t];
    fits.resize(shape_costs(t).size());
    ShapeFit &f = fits[(size_t)i];
    if (f.stages >= 0)
        return f;
    if (p->most_delay < 0.0f)
        p->most_delay = *std::max_element(p->dmshift.begin(), p->dmshift.end());
    const ShapeCost &c = shape_costs(t)[(size_t)i];
    Geometry r = tile_geometry(t, c.tiles);
    double steps = 0;
    for (int d = 0; d < p->ndm; d += r.dm_cta)
        steps = std::max(steps,
                         (double)p->dm_sorted[(size_t)std::min(d + r.dm_cta, p->ndm) - 1] -
                             (double)p->dm_sorted[(size_t)d]);
    // The widest window: its samples less the truncation of both shifts, and
    // with that and the 16-byte rounding at both ends.  (Beyond 2^20 samples it
    // fits in no shape.)
    const int64_t samples =
        r.t_cta + (int64_t)std::min(steps * (double)p->most_delay, 1048576.0);
    auto ring = [&](int64_t widest) {
        int64_t smem = 0;
        ShapeFit x;
        x.stages = 0;
        if (ring_layout(&r, widest, &smem)) {
            x.stages = r.nstages;
            x.resident = std::min(c.resident, resident_ctas(r.smem));
        }
        return x;
    };
    f = ring((r.elem * (samples + 2) + 30) & ~(int64_t)15);
    const ShapeFit room = ring((r.elem * std::max<int64_t>(samples - 2, 0) + 15) & ~(int64_t)15);
    if (room.stages != f.stages || room.resident != f.resident) {
        f.stages = 0;
        if (make_geometry(p, t, c.tiles, &r) == DD_OK) {
            f.stages = r.nstages;
            f.resident = std::min(c.resident, resident_ctas(r.smem));
        }
    }
    return f;
}

// Time of one tile with `resident` CTAs on its SM.
double tile_us(dd_dtype t, const ShapeCost &c, const ShapeFit &f, int nchan, int resident) {
    const double us =
        std::max(0.5 * c.us64, c.us64 + (c.us512 - c.us64) * (nchan - 64) / 448.0) *
        (resident < c.resident ? kAlone : 1.0);
    const int n = (nchan + c.tiles.chan_per_stage - 1) / c.tiles.chan_per_stage;
    return us + (f.stages < 3 ? two_stages_us(t, us / n) * n : 0.0);
}

// Time of nsamp_out samples, ndm DMs.
double shape_time_us(dd_dtype t, const ShapeCost &c, const ShapeFit &f, int nchan, int ndm,
                     int64_t nsamp_out, int sms) {
    const int64_t d = c.tiles.dm_per_thread * c.tiles.dm_warps;
    const int64_t len = (int64_t)warp_span(t, c.tiles.words_per_thread) * c.tiles.time_warps;
    const int64_t nt = (nsamp_out + len - 1) / len, n = (ndm + d - 1) / d * nt;
    const int64_t slots = (int64_t)sms * f.resident;
    // The last of many rounds, partly filled, overlaps the others (their tiles
    // are out of step): 1428 and 1344 tiles of 64 channels took 9.4 and 9.1
    // rounds on 152 SMs, 476 tiles of 1422 channels still 4.
    auto rounds_of = [&](int64_t tiles) {
        const double whole = (double)((tiles + slots - 1) / slots),
                     part = (double)tiles / (double)slots;
        return part + (whole - part) * std::min(1.0, 4.0 / whole);
    };
    double rounds = rounds_of(n);
    // Few DMs left by the preferred FP16 / FP32 shape may run as a launch of
    // their own beside the last round (tail_geometry): 512 channels x 100 DMs
    // x 65536 FP32 take 500 us as 96 + 4 DMs, 522 in 32-DM tiles.  (uint8 beams
    // of that kind go to the channel groups as often as not.)
    const int64_t rem = ndm % d;
    if (t != DD_U8 && &c == &shape_costs(t)[0] && ndm >= d && rem > 0 && 2 * rem <= d) {
        const int64_t full = ndm / d * nt, free = (full + slots - 1) / slots * slots - full,
                      dmw = (rem + c.tiles.dm_per_thread - 1) / c.tiles.dm_per_thread,
                      tl = len * std::max<int64_t>(1, c.tiles.dm_warps / dmw);
        if ((nsamp_out + tl - 1) / tl <= free)
            rounds = std::min(rounds, rounds_of(full) + (double)rem / (double)d);
    }
    return rounds * tile_us(t, c, f, nchan, f.resident);
}

// Place of a shape in the list (-1: not listed).
int place_of(dd_dtype t, const dd_tiles &tl) {
    const std::vector<ShapeCost> &shapes = shape_costs(t);
    for (int i = 0; i < (int)shapes.size(); ++i)
        if (std::memcmp(&shapes[i].tiles, &tl, sizeof(tl)) == 0)
            return i;
    return -1;
}

// The listed shape expected to finish first (-1: none fits), and its time.
// Caller holds p->mu.
int fastest_shape(dd_plan_s *p, dd_dtype t, int64_t nsamp_out, int sms, double *us) {
    ShapeChoice &last = p->shape_choice[t];
    if (last.nsamp_out == nsamp_out && last.sms == sms && last.unfit == p->shape_unfit[t]) {
        *us = last.us;
        return last.place;
    }
    const std::vector<ShapeCost> &shapes = shape_costs(t);
    const bool narrow = shape_fit(p, t, 0).stages >= 3;
    int best = -1;
    for (int i = 0; i < (int)shapes.size(); ++i) {
        if ((shapes[i].wide && narrow) || (p->shape_unfit[t] >> i & 1u) ||
            shape_fit(p, t, i).stages == 0)
            continue;
        // (2 % in favour of the preferred shape, the first.)
        const double u =
            shape_time_us(t, shapes[i], shape_fit(p, t, i), p->nchan, p->ndm, nsamp_out, sms) *
            (i > 0 ? 1.02 : 1.0);
        if (best < 0 || u < *us) {
            best = i;
            *us = u;
        }
    }
    last = {nsamp_out, sms, p->shape_unfit[t], best, *us};
    return best;
}

}  // namespace

void Makespan::run(int64_t tiles, double us) {
    if (tiles > 4 * (int64_t)sms_) {  // whole rounds at once
        const int64_t rounds = tiles / sms_ - 2;
        std::map<double, int> later;
        for (const auto &f : free_)
            later[f.first + (double)rounds * us] += f.second;
        free_.swap(later);
        tiles -= rounds * sms_;
    }
    while (tiles > 0) {
        const auto first = free_.begin();
        const double at = first->first;
        const int n = (int)std::min<int64_t>(tiles, first->second);
        if ((first->second -= n) == 0)
            free_.erase(first);
        free_[at + us] += n;
        end_ = std::max(end_, at + us);
        tiles -= n;
    }
}

namespace {

bool fits_every(const std::vector<BatchLoad> &beams, dd_dtype t, const dd_tiles &tl) {
    Geometry g;
    for (const BatchLoad &b : beams)
        if (make_geometry(b.plan, t, tl, &g) != DD_OK)
            return false;
    return true;
}

// The listed shape in which one persistent launch (a CTA per SM) over the
// beams, largest channel counts first, is expected to finish first (-1: none
// fits all of them).
int fastest_shared_shape(std::vector<BatchLoad> beams, dd_dtype t, int sms) {
    const std::vector<ShapeCost> &shapes = shape_costs(t);
    std::stable_sort(beams.begin(), beams.end(), [](const BatchLoad &x, const BatchLoad &y) {
        return x.plan->nchan > y.plan->nchan;
    });
    // All beams share the ring of the widest windows.
    std::vector<ShapeFit> fits(shapes.size(), ShapeFit{4, 1});
    for (size_t i = 0; i < fits.size(); ++i)
        for (const BatchLoad &b : beams) {
            if (shapes[i].wide && fits[0].stages >= 3)
                break;
            std::lock_guard<std::mutex> lk(b.plan->mu);
            fits[i].stages = std::min(fits[i].stages, shape_fit(b.plan, t, (int)i).stages);
        }
    int best = -1;
    double least = 0;
    for (int i = 0; i < (int)shapes.size(); ++i) {
        if (fits[i].stages == 0 || (shapes[i].wide && fits[0].stages >= 3))
            continue;
        const Geometry g = tile_geometry(t, shapes[i].tiles);
        Makespan m(sms);
        for (const BatchLoad &b : beams)
            m.run((int64_t)((b.plan->ndm + g.dm_cta - 1) / g.dm_cta) *
                      ((b.nsamp_out + g.t_cta - 1) / g.t_cta),
                  tile_us(t, shapes[i], fits[i], b.plan->nchan, 1));
        const double us = m.end() * (i > 0 ? 1.02 : 1.0);
        if (best < 0 || us < least) {
            best = i;
            least = us;
        }
    }
    return best;
}

}  // namespace

bool shared_tiles(const std::vector<BatchLoad> &beams, dd_dtype t, dd_tiles *out) {
    int dev = 0;
    const int sms = cudaGetDevice(&dev) == cudaSuccess ? sm_count(dev) : 0;
    // (uint8 keeps the preferred shape: beams of few DMs gain by the channel
    // groups that stand beside it.)
    if (t != DD_U8 && sms > 0) {
        const int best = fastest_shared_shape(beams, t, sms);
        if (best >= 0 && fits_every(beams, t, shape_costs(t)[(size_t)best].tiles)) {
            *out = shape_costs(t)[(size_t)best].tiles;
            return true;
        }
    }
    for (const dd_tiles &cand : auto_tiles(t))
        if (fits_every(beams, t, cand)) {
            *out = cand;
            return true;
        }
    return false;
}

double direct_time_us(dd_plan_s *p, dd_dtype t, const dd_tiles &tl, int64_t nsamp_out, int sms) {
    const int i = place_of(t, tl);
    std::lock_guard<std::mutex> lk(p->mu);
    if (i < 0 || shape_fit(p, t, i).stages == 0)
        return -1.0;
    return shape_time_us(t, shape_costs(t)[(size_t)i], shape_fit(p, t, i), p->nchan, p->ndm,
                         nsamp_out, sms);
}

double direct_tile_us(dd_plan_s *p, dd_dtype t, const dd_tiles &tl) {
    const int i = place_of(t, tl);
    std::lock_guard<std::mutex> lk(p->mu);
    if (i < 0 || shape_fit(p, t, i).stages == 0)
        return -1.0;
    return tile_us(t, shape_costs(t)[(size_t)i], shape_fit(p, t, i), p->nchan, 1);
}

dd_status execution_geometry(dd_plan_s *p, dd_dtype t, int64_t nsamp_out, Geometry *g) {
    int dev = 0;
    int sms = 0;
    if (valid_dtype(t) && cudaGetDevice(&dev) == cudaSuccess && (sms = sm_count(dev)) > 0) {
        std::lock_guard<std::mutex> lk(p->mu);
        while (p->tiles_open[t]) {
            double us = 0;
            const int best = fastest_shape(p, t, nsamp_out, sms, &us);
            if (best < 0)
                break;
            const dd_tiles &tiles = shape_costs(t)[(size_t)best].tiles;
            const uint64_t key = geo_key(t, tiles);
            auto it = p->geo.find(key);
            Geometry r;
            if (it == p->geo.end() && make_geometry(p, t, tiles, &r) == DD_OK)
                it = p->geo.emplace(key, r).first;
            if (it != p->geo.end()) {
                *g = it->second;
                g->chosen = true;
                return DD_OK;
            }
            // Its windows do not fit shared memory: passed over from now on.
            p->shape_unfit[t] |= 1u << best;
        }
    }
    return plan_geometry(p, t, g);
}

double execution_time(dd_plan_s *p, dd_dtype t, int64_t nsamp_out) {
    int dev = 0;
    const int sms = cudaGetDevice(&dev) == cudaSuccess ? std::max(1, sm_count(dev)) : 1;
    {
        std::lock_guard<std::mutex> lk(p->mu);
        double us = 0;
        if (p->tiles_open[t] && fastest_shape(p, t, nsamp_out, sms, &us) >= 0)
            return us;
    }
    Geometry g;
    if (plan_geometry(p, t, &g) != DD_OK)
        return 1.0;
    const int64_t n = (int64_t)g.ntile_d * ((nsamp_out + g.t_cta - 1) / g.t_cta);
    return (double)((n + sms - 1) / sms);
}

}  // namespace dd
