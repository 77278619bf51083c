// Batches: many uneven beams de-dispersed by one persistent launch, captured
// in a CUDA graph.
//
// Each beam keeps its own plan, buffers and geometry (row width in shared
// memory, number of DM tiles); all beams share one tile shape, so one kernel
// instantiation and one shared-memory layout serve the whole batch.  Beam
// descriptors live in device memory in scheduling order -- largest per-tile
// cost (channel count) first -- and the kernel's producer warps claim global
// tile numbers from an atomic counter, so big beams start first and small
// tiles fill the tail.
//
// Beams that gain by channel groups (dd_group.h) go to a second launch that
// runs beside the persistent one, on a forked stream: its tiles take the SMs
// that the persistent CTAs leave.
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <numeric>
#include <string>
#include <vector>

#include "dd_group.h"
#include "dd_internal.h"
#include "dd_kargs.h"

namespace {

using dd::fail;

struct BatchBeam {
    dd_plan_s *plan = nullptr;
    const void *in = nullptr;
    int64_t in_pitch = 0, nsamp_in = 0;
    float *out = nullptr;
    int64_t out_pitch = 0, nsamp_out = 0;
    bool bound = false;
    dd::Geometry g;
    int64_t ntiles = 0;
};

}  // namespace

struct dd_batch_s {
    dd_dtype dtype = DD_U8;
    std::vector<BatchBeam> beams;
    dd_tiles tiles{};
    bool tiles_set = false;
    int dev = -1;
    dd::BeamArgs *d_beams = nullptr;
    int *d_counter = nullptr;
    int *d_status = nullptr;
    dd::KArgs args{};        // direct launch (args.nbeams == 0: none)
    dd::GroupBeam *d_gbeams = nullptr;
    dd::GroupArgs gargs{};   // grouped launch (gargs.nbeams == 0: none)
    unsigned ggrid = 0;
    cudaStream_t side = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    unsigned grid = 0;
    int threads = 0, smem = 0;
    int64_t total_tiles = 0;
    bool prepared = false;
    int slot = 0;               // of the descriptors in use (two, so that a launch
                                // in flight keeps its own)
    std::vector<int> order;     // beams in launch order
    bool unsampled = false;     // whether beams gain by groups is to be seen behind the launch
    std::vector<int> tables;    // beams whose tables the next preparation waits for
    cudaStream_t capture = nullptr;
    cudaGraphExec_t exec = nullptr;
    std::mutex mu;
};

namespace {

bool fits_all(dd_batch_s *b, const dd_tiles &tl) {
    for (auto &bb : b->beams) {
        dd::Geometry g;
        if (dd::make_geometry(bb.plan, b->dtype, tl, &g) != DD_OK)
            return false;
    }
    return true;
}

void drop_graph(dd_batch_s *b) {
    if (b->exec) {
        cudaGraphExecDestroy(b->exec);
        b->exec = nullptr;
    }
    b->prepared = false;
    b->unsampled = false;
    b->tables.clear();
}

// The shape for the beams as they are bound (beams without buffers count with
// 65536 samples).
bool choose_tiles(dd_batch_s *b, dd_tiles *tiles) {
    std::vector<dd::BatchLoad> load;
    for (const BatchBeam &bb : b->beams)
        load.push_back({bb.plan, bb.bound ? bb.nsamp_out : 65536});
    return dd::shared_tiles(load, b->dtype, tiles);
}

// Beams (in launch order) that run grouped, if the batch is expected to finish
// earlier by it: beside the persistent launch of the others, their tiles take
// the SMs that its CTAs leave.  A beam is a candidate if its tiles are a smaller
// share of the SMs' time; the times compared are those of the whole batch (3
// beams of 1024 channels x 100 DMs x 16384 samples: 144 tiles, one round of
// 306 us; grouped, 96 longer ones, 383 us).
//
// Finding that out samples every plan's patterns, some 30 us of host work each
// once.  Unless `all`, a batch of less than 400 us per plan to be sampled leaves
// it to be done behind its launch (b->unsampled).
std::vector<int> grouped_beams(dd_batch_s *b, bool all, double *gain_us) {
    const dd_tiles pref = dd::default_tiles(DD_U8);
    const int sms = dd::sm_count(b->dev);
    std::vector<int> grouped;
    b->unsampled = false;
    if (b->dtype != DD_U8 || sms <= 0 || std::memcmp(&pref, &b->tiles, sizeof(pref)) != 0)
        return grouped;
    dd::Makespan direct(sms), mixed(sms);
    int unsampled = 0;
    for (int i : b->order) {
        BatchBeam &bb = b->beams[i];
        direct.run(bb.ntiles, dd::direct_tile_us(bb.plan, DD_U8, b->tiles));
        unsampled += dd::group_sampled(bb.plan, b->dev) ? 0 : 1;
    }
    if (!all && direct.end() < 400.0 * unsampled) {
        b->unsampled = true;
        return grouped;
    }
    std::vector<dd::GroupEstimate> est;
    for (int i : b->order) {
        BatchBeam &bb = b->beams[i];
        const double us = dd::direct_tile_us(bb.plan, DD_U8, b->tiles);
        dd::GroupEstimate e;
        if (us > 0 && dd::group_estimate(bb.plan, b->dev, bb.nsamp_out, &e) &&
            (double)e.tiles * e.tile_us <= dd::kGroupGain * (double)bb.ntiles * us) {
            grouped.push_back(i);
            est.push_back(e);
        } else {
            mixed.run(bb.ntiles, us);
        }
    }
    for (const dd::GroupEstimate &e : est)
        mixed.run(e.tiles, e.tile_us);
    *gain_us = direct.end() - mixed.end();
    if (mixed.end() > dd::kGroupGain * direct.end())
        grouped.clear();
    return grouped;
}

// Geometry, descriptors and launch shape for the current tiles.  Tables that
// some beams would need and do not have are built first if `now` or if this
// execution gains more than they cost (started together, 80 us more for each
// after the first); else all beams run directly and
// b->tables names the beams whose tables are to be started behind the launch.
dd_status prepare(dd_batch_s *b, bool now) {
    if (b->prepared)
        return DD_OK;
    for (size_t i = 0; i < b->beams.size(); ++i)
        if (!b->beams[i].bound)
            return fail(DD_ERR_INVALID, "beam " + std::to_string(i) + " has no buffers bound");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess)
        return fail(DD_ERR_CUDA, "cudaGetDevice failed");
    if (b->dev >= 0 && dev != b->dev)
        return fail(DD_ERR_INVALID, "a batch is bound to the device it was first executed on");
    b->dev = dev;
    if (!b->tiles_set && !choose_tiles(b, &b->tiles))
        return fail(DD_ERR_INVALID, "no tile shape fits every beam of the batch");
    const int elem = dd::elem_size(b->dtype);
    int64_t stage_max = 0;
    for (auto &bb : b->beams) {
        dd_status st = dd::make_geometry(bb.plan, b->dtype, b->tiles, &bb.g);
        if (st != DD_OK)
            return st;
        stage_max = std::max<int64_t>(stage_max, bb.g.stage_bytes);
        bb.ntiles = (int64_t)bb.g.ntile_d * ((bb.nsamp_out + bb.g.t_cta - 1) / bb.g.t_cta);
    }
    const dd::Geometry &g0 = b->beams[0].g;
    // Shared-memory layout sized for the widest beam.
    auto smem_for = [&](int64_t n) { return dd::ring_smem(g0, stage_max, (int)n); };
    int nst = 4;
    while (nst > 2 && smem_for(nst) > dd::kMaxSmem)
        --nst;
    if (smem_for(nst) > dd::kMaxSmem)
        return fail(DD_ERR_INVALID, "batch tile shape does not fit shared memory");

    // Scheduling order: larger per-tile cost (channels) first.
    std::vector<int> &order = b->order;
    order.resize(b->beams.size());
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
        return b->beams[x].plan->nchan > b->beams[y].plan->nchan;
    });
    std::vector<dd::DevTables *> tables(b->beams.size());
    for (size_t i = 0; i < b->beams.size(); ++i) {
        const dd_status st = dd::device_tables(b->beams[i].plan, &tables[i]);
        if (st != DD_OK)
            return st;
    }
    const int nsm = dd::sm_count(dev);
    double gain = 0;
    std::vector<int> grouped = grouped_beams(b, now, &gain), missing;
    std::vector<dd::GroupTable> shapes(b->beams.size());
    for (int i : grouped)
        if (!dd::group_ready(b->beams[i].plan, dev, *tables[i], false, &shapes[i]))
            missing.push_back(i);
    b->tables.clear();
    if (!missing.empty() && !now && gain <= dd::kGroupTableUs + 80.0 * (double)(missing.size() - 1)) {
        grouped.clear();
        b->tables = missing;
    } else {
        for (int i : missing)  // all of them under way before the first is waited for
            dd::group_start(b->beams[i].plan, dev, *tables[i]);
    }
    std::vector<dd::BeamArgs> desc;
    std::vector<dd::GroupBeam> gdesc;
    int64_t tile0 = 0, gtile0 = 0;
    for (int i : order) {
        BatchBeam &bb = b->beams[i];
        const dd::DevTables *dt = tables[i];
        if (std::find(grouped.begin(), grouped.end(), i) != grouped.end() &&
            dd::group_ready(bb.plan, dev, *dt, true, &shapes[i])) {
            gdesc.push_back(dd::group_beam(shapes[i], *dt, bb.in, bb.in_pitch, bb.nsamp_in,
                                           bb.out, bb.out_pitch, bb.nsamp_out));
            gdesc.back().tile_begin = gtile0;
            gtile0 += dd::group_tiles(shapes[i].ntile_d, bb.nsamp_out);
            continue;
        }
        desc.emplace_back();
        dd::BeamArgs &d = desc.back();
        d.in = static_cast<const uint8_t *>(bb.in);
        d.in_pitch_b = bb.in_pitch * elem;
        d.nsamp_in = bb.nsamp_in;
        d.out = bb.out;
        d.out_pitch = bb.out_pitch;
        d.nsamp_out = bb.nsamp_out;
        d.dmshift = dt->dmshift;
        d.dm_sorted = dt->dm_sorted;
        d.perm = dt->perm;
        d.tile_begin = tile0;
        d.nchan = bb.plan->nchan;
        d.ntile_d = bb.g.ntile_d;
        d.wp = bb.g.wp;
        d.pad = 0;
        tile0 += bb.ntiles;
    }
    // Each on its own: what an earlier call could not have is asked for again.
    auto have = [](auto **p, size_t bytes) {
        return *p || cudaMalloc((void **)p, bytes) == cudaSuccess;
    };
    const size_t n = b->beams.size();
    const bool fresh = !b->d_status;
    if (!have(&b->d_beams, 2 * sizeof(dd::BeamArgs) * n) ||
        !have(&b->d_gbeams, 2 * sizeof(dd::GroupBeam) * n) ||
        !have(&b->d_counter, sizeof(int)) || !have(&b->d_status, sizeof(int))) {
        cudaGetLastError();
        return fail(DD_ERR_NOMEM, "batch descriptor allocation failed");
    }
    if (fresh)
        cudaMemset(b->d_status, 0, sizeof(int));
    if (!b->capture &&
        cudaStreamCreateWithFlags(&b->capture, cudaStreamNonBlocking) != cudaSuccess)
        return fail(DD_ERR_CUDA, "capture stream creation failed");
    b->slot ^= 1;
    dd::BeamArgs *d_beams = b->d_beams + (size_t)b->slot * n;
    dd::GroupBeam *d_gbeams = b->d_gbeams + (size_t)b->slot * n;
    if (cudaMemcpyAsync(d_beams, desc.data(), sizeof(dd::BeamArgs) * desc.size(),
                        cudaMemcpyHostToDevice, b->capture) != cudaSuccess ||
        cudaMemcpyAsync(d_gbeams, gdesc.data(), sizeof(dd::GroupBeam) * gdesc.size(),
                        cudaMemcpyHostToDevice, b->capture) != cudaSuccess ||
        cudaStreamSynchronize(b->capture) != cudaSuccess)
        return fail(DD_ERR_CUDA, "batch descriptor upload failed");
    auto event = [](cudaEvent_t *e) {
        return *e || cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
    };
    if (!gdesc.empty() && !desc.empty() &&
        ((!b->side &&
          cudaStreamCreateWithFlags(&b->side, cudaStreamNonBlocking) != cudaSuccess) ||
         !event(&b->fork) || !event(&b->join)))
        return fail(DD_ERR_CUDA, "batch stream creation failed");
    if (tile0 > 0x7fffffffLL || gtile0 > 0x7fffffffLL)
        return fail(DD_ERR_INVALID, "too many tiles in one batch");
    b->total_tiles = tile0;
    b->ggrid = (unsigned)gtile0;
    b->gargs = dd::GroupArgs{};
    b->gargs.beams = d_gbeams;
    b->gargs.nbeams = (int)gdesc.size();
    b->gargs.status = b->d_status;
    b->grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(tile0, nsm > 0 ? nsm : 1));
    b->threads = g0.threads;
    b->smem = (int)smem_for(nst);
    dd::KArgs &a = b->args;
    a = dd::KArgs{};
    a.beams = d_beams;
    a.nbeams = (int)desc.size();
    a.total_tiles = tile0;
    a.tile_counter = b->d_counter;
    a.dm_warps = b->tiles.dm_warps;
    a.time_warps = b->tiles.time_warps;
    a.cstage = b->tiles.chan_per_stage;
    a.nstages = nst;
    a.stage_bytes = (int)stage_max;
    a.zero_bytes = g0.zero_bytes;
    a.builders = g0.builders;
    a.one = 1u;
    a.status = b->d_status;
    b->prepared = true;
    return DD_OK;
}

// Between executions: start the tables that the next preparation is to use;
// once all of them have come (or failed) the batch is to be prepared anew.
void look_after_tables(dd_batch_s *b) {
    if (b->unsampled) {
        double gain = 0;
        b->tables = grouped_beams(b, true, &gain);
    }
    if (b->tables.empty())
        return;
    bool waiting = false;
    for (int i : b->tables) {
        BatchBeam &bb = b->beams[i];
        dd::DevTables *dt = nullptr;
        dd::GroupEstimate e;
        if (dd::device_tables(bb.plan, &dt) != DD_OK)
            continue;
        dd::group_start(bb.plan, b->dev, *dt);
        waiting |= dd::group_estimate(bb.plan, b->dev, bb.nsamp_out, &e) && !e.ready;
    }
    if (!waiting)
        drop_graph(b);
}

// De-dispersion kernels of one execution.
int launches(const dd_batch_s *b) {
    return (b->args.nbeams > 0 ? 1 : 0) + (b->gargs.nbeams > 0 ? 1 : 0);
}

// The tile counter reset and the persistent launch of the direct beams; the
// grouped beams' launch beside it.
dd_status enqueue(dd_batch_s *b, cudaStream_t s, bool count = true) {
    const bool direct = b->args.nbeams > 0, grouped = b->gargs.nbeams > 0;
    const bool both = direct && grouped;
    cudaError_t e = cudaSuccess;
    if (both) {
        e = cudaEventRecord(b->fork, s);
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(b->side, b->fork, 0);
        if (e != cudaSuccess)
            return fail(DD_ERR_CUDA, std::string("batch fork: ") + cudaGetErrorString(e));
    }
    if (direct) {
        e = cudaMemsetAsync(b->d_counter, 0, sizeof(int), s);
        if (e != cudaSuccess)
            return fail(DD_ERR_CUDA, std::string("batch counter reset: ") + cudaGetErrorString(e));
        const int dthr = b->tiles.dm_per_thread, nw = b->tiles.words_per_thread;
        switch (b->dtype) {
        case DD_U8: e = dd::launch_kernel_u8(b->args, b->grid, b->threads, b->smem, s, dthr, nw); break;
        case DD_F16: e = dd::launch_kernel_f16(b->args, b->grid, b->threads, b->smem, s, dthr, nw); break;
        case DD_F32: e = dd::launch_kernel_f32(b->args, b->grid, b->threads, b->smem, s, dthr, nw); break;
        }
    }
    if (grouped && e == cudaSuccess)
        e = dd::launch_group(b->gargs, b->ggrid, both ? b->side : s);
    if (both) {
        if (e == cudaSuccess)
            e = cudaEventRecord(b->join, b->side);
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(s, b->join, 0);
    }
    if (e != cudaSuccess)
        return fail(DD_ERR_CUDA, std::string("batch kernel launch: ") + cudaGetErrorString(e));
    if (count)
        dd::count_launch(launches(b));
    return DD_OK;
}

}  // namespace

extern "C" {

dd_status dd_batch_create(const dd_plan_t *plans, int nbeams, dd_dtype dtype, dd_batch_t *out) {
    if (!out)
        return fail(DD_ERR_INVALID, "batch_out is NULL");
    *out = nullptr;
    if (!plans || nbeams < 1)
        return fail(DD_ERR_INVALID, "need at least one plan");
    if (dtype != DD_U8 && dtype != DD_F16 && dtype != DD_F32)
        return fail(DD_ERR_INVALID, "unknown dtype");
    for (int i = 0; i < nbeams; ++i)
        if (!plans[i])
            return fail(DD_ERR_INVALID, "NULL plan in batch");
    dd_batch_s *b = new (std::nothrow) dd_batch_s;
    if (!b)
        return fail(DD_ERR_NOMEM, "out of host memory");
    b->dtype = dtype;
    b->beams.resize(nbeams);
    for (int i = 0; i < nbeams; ++i)
        b->beams[i].plan = plans[i];
    *out = b;
    return DD_OK;
}

void dd_batch_destroy(dd_batch_t b) {
    if (!b)
        return;
    if (b->dev >= 0)
        cudaSetDevice(b->dev);
    cudaDeviceSynchronize();
    drop_graph(b);
    cudaFree(b->d_beams);
    cudaFree(b->d_gbeams);
    cudaFree(b->d_counter);
    cudaFree(b->d_status);
    if (b->fork)
        cudaEventDestroy(b->fork);
    if (b->join)
        cudaEventDestroy(b->join);
    if (b->side)
        cudaStreamDestroy(b->side);
    if (b->capture)
        cudaStreamDestroy(b->capture);
    delete b;
}

dd_status dd_batch_set_io(dd_batch_t b, int beam, const void *in, int64_t in_pitch,
                          int64_t nsamp_in, float *out, int64_t out_pitch, int64_t nsamp_out) {
    if (!b || beam < 0 || beam >= (int)b->beams.size())
        return fail(DD_ERR_INVALID, "bad batch or beam index");
    BatchBeam &bb = b->beams[beam];
    const int64_t elem = dd::elem_size(b->dtype);
    if (nsamp_out < 1 || nsamp_in < nsamp_out + bb.plan->maxshift)
        return fail(DD_ERR_INVALID, "nsamp_out must be >= 1 and nsamp_in >= nsamp_out + maxshift");
    if (in_pitch < nsamp_in || out_pitch < nsamp_out || (in_pitch * elem) % 16 || out_pitch % 4)
        return fail(DD_ERR_INVALID, "pitches must cover a row and be multiples of 16 bytes");
    if (!in || !out || ((uintptr_t)in & 15u) || ((uintptr_t)out & 15u))
        return fail(DD_ERR_INVALID, "in and out must be non-NULL and 16-byte aligned");
    std::lock_guard<std::mutex> lk(b->mu);
    bb.in = in;
    bb.in_pitch = in_pitch;
    bb.nsamp_in = nsamp_in;
    bb.out = out;
    bb.out_pitch = out_pitch;
    bb.nsamp_out = nsamp_out;
    bb.bound = true;
    drop_graph(b);
    return DD_OK;
}

dd_status dd_batch_get_tiles(dd_batch_t b, dd_tiles *t) {
    if (!b || !t)
        return fail(DD_ERR_INVALID, "NULL argument");
    std::lock_guard<std::mutex> lk(b->mu);
    // (A prepared batch has its shape; else the one that its next execution takes.)
    if (!b->tiles_set && !b->prepared && !choose_tiles(b, &b->tiles))
        return fail(DD_ERR_INVALID, "no tile shape fits every beam of the batch");
    *t = b->tiles;
    return DD_OK;
}

dd_status dd_batch_set_tiles(dd_batch_t b, const dd_tiles *t) {
    if (!b || !t)
        return fail(DD_ERR_INVALID, "NULL argument");
    std::lock_guard<std::mutex> lk(b->mu);
    for (auto &bb : b->beams) {
        dd::Geometry g;
        dd_status st = dd::make_geometry(bb.plan, b->dtype, *t, &g);
        if (st != DD_OK)
            return st;
    }
    b->tiles = *t;
    b->tiles_set = true;
    drop_graph(b);
    return DD_OK;
}

dd_status dd_batch_execute(dd_batch_t b, void *stream) {
    dd::Range nvtx_range("dd_batch_execute");
    if (!b)
        return fail(DD_ERR_INVALID, "batch is NULL");
    std::lock_guard<std::mutex> lk(b->mu);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!b->exec) {
        look_after_tables(b);
        dd_status st = prepare(b, false);
        if (st != DD_OK)
            return st;
        // One eager run first: it sets the kernel attributes outside any capture.
        if ((st = enqueue(b, s)) != DD_OK)
            return st;
        look_after_tables(b);
        if (!b->prepared || !b->tables.empty())
            return DD_OK;  // a later execution has the graph
        cudaGraph_t graph = nullptr;
        if (cudaStreamBeginCapture(b->capture, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
            return fail(DD_ERR_CUDA, "stream capture failed to start");
        st = enqueue(b, b->capture, false);
        cudaError_t e = cudaStreamEndCapture(b->capture, &graph);
        if (st != DD_OK)
            return st;
        if (e != cudaSuccess)
            return fail(DD_ERR_CUDA, std::string("stream capture: ") + cudaGetErrorString(e));
        e = cudaGraphInstantiate(&b->exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            b->exec = nullptr;
            return fail(DD_ERR_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
        }
        return DD_OK;  // this call's work was the eager run
    }
    cudaError_t e = cudaGraphLaunch(b->exec, s);
    if (e != cudaSuccess)
        return fail(DD_ERR_CUDA, std::string("graph launch: ") + cudaGetErrorString(e));
    dd::count_launch(launches(b));
    return DD_OK;
}

dd_status dd_batch_sync(dd_batch_t b, void *stream) {
    if (!b)
        return fail(DD_ERR_INVALID, "batch is NULL");
    cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess)
        return fail(DD_ERR_CUDA, std::string("stream synchronize: ") + cudaGetErrorString(e));
    if (!b->d_status)
        return DD_OK;
    int word = 0;
    if (cudaMemcpy(&word, b->d_status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
        return fail(DD_ERR_CUDA, "status read failed");
    if (word != dd::kDevOk) {
        cudaMemset(b->d_status, 0, sizeof(int));
        return word == dd::kDevTimeout ? fail(DD_ERR_TIMEOUT, "a device wait ran out")
                                       : fail(DD_ERR_DEVICE, "kernel recorded a failed check");
    }
    return DD_OK;
}

dd_status dd_batch_autotune(dd_batch_t b, void *stream, int reps, dd_tune_result *results,
                            int max_results, int *n_results) {
    dd::Range nvtx_range("dd_batch_autotune");
    if (!b || reps < 1)
        return fail(DD_ERR_INVALID, "bad batch or reps");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
        return fail(DD_ERR_CUDA, "event creation failed");
    std::vector<dd_tiles> cands;
    for (int nw : {8, 4})
        for (int dthr : {4, 2, 1})
            for (int dw : {6, 8, 10, 12, 16})
                for (int cs : {8, 12, 16}) {
                    const int wt = 1;
                    if (dw * wt > dd::max_consumer_warps(dthr, nw))
                        continue;
                    cands.push_back(dd_tiles{dthr, dw, wt, cs, nw});
                }
    float best = -1.0f;
    dd_tiles best_t{};
    int n = 0;
    dd_status st = DD_OK;
    std::lock_guard<std::mutex> lk(b->mu);
    for (const dd_tiles &c : cands) {
        float ms = -1.0f;
        if (fits_all(b, c)) {
            drop_graph(b);
            b->tiles = c;
            b->tiles_set = true;
            if ((st = prepare(b, true)) != DD_OK)
                break;
            if ((st = enqueue(b, s)) != DD_OK)  // warm-up
                break;
            for (int r = 0; r < reps; ++r) {
                cudaEventRecord(e0, s);
                if ((st = enqueue(b, s)) != DD_OK)
                    break;
                cudaEventRecord(e1, s);
                if (cudaEventSynchronize(e1) != cudaSuccess) {
                    st = fail(DD_ERR_CUDA, "batch autotune synchronize failed");
                    break;
                }
                float t = 0.0f;
                cudaEventElapsedTime(&t, e0, e1);
                ms = (ms < 0.0f || t < ms) ? t : ms;
            }
            if (st != DD_OK)
                break;
            if (ms >= 0.0f && (best < 0.0f || ms < best)) {
                best = ms;
                best_t = c;
            }
        }
        if (results && n < max_results)
            results[n] = dd_tune_result{c, ms};
        ++n;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (n_results)
        *n_results = n;
    if (st != DD_OK)
        return st;
    if (best < 0.0f)
        return fail(DD_ERR_INVALID, "no candidate tile shape fits every beam");
    drop_graph(b);
    b->tiles = best_t;
    b->tiles_set = true;
    return DD_OK;
}

}  // extern "C"
