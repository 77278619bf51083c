// Internal declarations shared by the host plan (dd_plan.cpp) and the CUDA
// translation units of libdd.  Not part of the public ABI (include/dd.h).
#pragma once

#include <cuda_runtime_api.h>

#include <algorithm>
#include <cfloat>
#include <cstdint>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/dd.h"

namespace dd {

// NVTX range over one C-ABI call, named after it, for Nsight timelines (a
// no-op when no tool is attached).
struct Range {
    explicit Range(const char *name) { nvtxRangePushA(name); }
    ~Range() { nvtxRangePop(); }
    Range(const Range &) = delete;
    Range &operator=(const Range &) = delete;
};

// Samples covered by one warp along time: 32 lanes x `words` 4-byte words x
// (4 / element size) samples per word.
inline int elem_size(dd_dtype t) { return t == DD_U8 ? 1 : (t == DD_F16 ? 2 : 4); }
inline int warp_span(dd_dtype t, int words) { return 32 * words * (4 / elem_size(t)); }
inline int phases(dd_dtype t) { return 4 / elem_size(t); }
inline bool valid_dtype(dd_dtype t) { return t == DD_U8 || t == DD_F16 || t == DD_F32; }

// The shift of a channel: one FP32 multiply, rounded to nearest even, then
// truncated.
static_assert(FLT_EVAL_METHOD == 0, "float products are rounded to float");
inline int trunc_product(float dm, float ds) { return (int)(dm * ds); }

// Channels summed into 16-bit SWAR lanes before they are widened (uint8):
// 256 * 255 = 65280 fits a 16-bit lane.
constexpr int kSwarChannels = 256;
// Channels per compensated block for FP16/FP32 input: a multiple of every stage
// size that the library chooses or tunes among (4, 8, 12, 16, 24), so the sums
// have the same bits in all of those shapes, whatever the length of an
// execution, its beam's place in a batch or the blocks of a host buffer.
// (Blocks of 64 channels held 60 with stages of 12 and 48 with stages of 24,
// and the results followed the shape.  Against those, 48 channels cost 1.6 %
// on the 4096-channel FP16 beam, 36.6 -> 37.1 ms, and 0.1 % on the FP32 L-band
// beam, 8.05 -> 8.06 ms.)
constexpr int kFloatBlock = 48;
// Channels per stage, at most.
constexpr int kFloatStage = 64;

constexpr int kMaxSmem = 232448;  // 227 KB dynamic shared memory per CTA
constexpr int kMaxDmPerCta = 64;   // DMs per CTA (offset-table columns, DM padding)
constexpr int kStageMeta = 32;     // bytes of a stage record in shared memory
// Builder warps (8/16-bit input) derive the byte phases 1.. of every staged
// row from phase 0 in shared memory; the producer records the bytes staged
// per row (kRowInfoBytes per stage: one word per row, at most 64 rows).
constexpr int kMaxBuilders = 2;
constexpr int kRowInfoBytes = 256;
// Consumer warps per CTA (plus one producer warp and, for 8/16-bit input, the
// builder warps), from the registers a thread needs: accumulators 2*DT*NW
// (uint8) + two load buffers 4*NW + ~24.  A CTA of at most 16 warps leaves
// 128 registers a thread (at most 4 warps per SM sub-partition), at most 20
// leave 96, at most 24 leave 80, at most 28 leave 72.
#ifdef __CUDACC__
#define DD_HD __host__ __device__
#else
#define DD_HD
#endif
DD_HD constexpr int max_consumer_warps(int dm_per_thread, int words) {
    return words >= 8 ? (dm_per_thread >= 4 ? 13 : dm_per_thread == 2 ? 16 : 20)
                      : (dm_per_thread >= 4 ? 20 : 24);
}

// Device status word values (written by kernels, read by dd_sync).
constexpr int kDevOk = 0;
constexpr int kDevTimeout = 1;
constexpr int kDevCheck = 2;

struct DevTables {
    float *dmshift = nullptr;    // [nchan]
    float *dm_sorted = nullptr;  // [ndm_pad]: DMs in ascending order, padded with the last
    int *perm = nullptr;         // [ndm_pad]: output row of sorted DM k, -1 for padding
    int *status = nullptr;       // device status word
    int ndm_pad = 0;
    int *det_cnt = nullptr;      // tile-boundary counters of fused detection
    int64_t det_cnt_n = 0;
};

// Accumulators of a boxcar search (dd_detect, dd_execute_detect): caller-owned
// output arrays, used as exact sums and keys until the finalize step.
struct DetectTargets {
    int nlevels = 0;
    double *mean = nullptr, *sd = nullptr, *snr = nullptr;
    int64_t *tpk = nullptr;
};

// Launch geometry derived from a tile shape and the plan's tables.
struct Geometry {
    dd_tiles tiles{};
    int elem = 1, nph = 1, span = 0;
    int dm_cta = 0;       // DMs per CTA
    int t_cta = 0;        // samples per CTA
    int ntile_d = 0;      // DM tiles
    int wp = 0;           // bytes of one phase row in shared memory
    int stage_bytes = 0;  // bytes of one ring stage (chan_per_stage rows, every phase)
    int nstages = 0;      // shared-memory stages in the copy ring
    int zero_bytes = 0;   // zero row read by padding channels
    int smem = 0;         // dynamic shared memory per CTA
    int builders = 0;     // phase-builder warps (0 for FP32)
    int threads = 0;      // consumer warps + one producer warp + builder warps
    bool chosen = false;  // by execution_geometry, not set or being measured
};

struct GroupShape;  // dd_group.h

struct ShapeFit {
    int stages = -1;   // of the ring (0: the windows do not fit, -1: not known)
    int resident = 1;  // CTAs on an SM
};

struct ShapeChoice {
    int64_t nsamp_out = -1;
    int sms = 0;
    uint32_t unfit = 0;
    int place = -1;   // in the list of shapes
    double us = 0;
};

}  // namespace dd

struct dd_plan_s {
    int nchan = 0, ndm = 0;
    double fch1 = 0, foff = 0, tsamp = 0;
    int64_t maxshift = 0;
    std::vector<float> dmshift;    // [nchan] FP32 table
    std::vector<float> dm;         // [ndm] caller order
    std::vector<int> order;        // sorted position -> caller index
    std::vector<float> dm_sorted;  // [ndm] ascending
    dd_tiles tiles[3]{};
    bool tiles_auto[3] = {true, true, true};  // resolved by the plan until set
    std::mutex mu;
    std::map<int, dd::DevTables> dev;      // per CUDA device
    bool tiles_open[3] = {true, true, true};  // executions may choose, until set
    std::map<uint64_t, dd::Geometry> geo;  // per (dtype, tiles) key
    std::vector<dd::ShapeFit> shape_fit[3];  // of the listed shapes (dd_shape.cpp), on first use
    dd::ShapeChoice shape_choice[3];         // for the last length asked for
    float most_delay = -1.0f;                // of dmshift, with the first of those
    uint32_t shape_unfit[3] = {0, 0, 0};     // shapes found not to fit, a bit each
    // Remainder-DM launch per (dtype, tiles) key: (found, geometry).
    std::map<uint64_t, std::pair<bool, dd::Geometry>> tail_geo;
    std::map<int, std::shared_ptr<dd::GroupShape>> group;  // grouped execution, per device
};

namespace dd {

// Thread-local error message; returns st for chaining.
dd_status fail(dd_status st, const std::string &msg);

// Dynamic shared memory of a ring of n stages of stage_bytes each for a
// geometry: the stages, the offset table, the stage records, the per-row
// byte counts (with phases to build), the zero row and three mbarriers per
// stage, in the order the kernel lays them out, and 16 bytes for the
// epilogue of fused detection.
int64_t ring_smem(const Geometry &g, int64_t stage_bytes, int n);

// Geometry of a tile shape before its windows are known, and its ring (four
// stages, or as many as fit) for windows of `widest` bytes: false if not even
// two stages of *smem bytes in all fit.
Geometry tile_geometry(dd_dtype t, const dd_tiles &tl);
bool ring_layout(Geometry *r, int64_t widest, int64_t *smem);

// CTAs of `smem` bytes of dynamic shared memory that an SM holds (228 KB, 1 KB
// per CTA reserved by the system).
inline int resident_ctas(int smem) { return std::max(1, 233472 / (smem + 1024)); }

inline uint64_t geo_key(dd_dtype t, const dd_tiles &tl) {
    return ((uint64_t)t << 60) | ((uint64_t)tl.words_per_thread << 48) |
           ((uint64_t)tl.dm_per_thread << 36) | ((uint64_t)tl.dm_warps << 24) |
           ((uint64_t)tl.time_warps << 12) | (uint64_t)tl.chan_per_stage;
}

// Host checks of a beam's layout shared by the entry points that run one
// beam: dtype, sample counts (nsamp_in >= nsamp_out + maxshift), pitches at
// least a row and, for device rows (device_rows), multiples of 16 bytes.
dd_status check_layout(dd_plan_s *p, dd_dtype dtype, int64_t in_pitch, int64_t nsamp_in,
                       int64_t out_pitch, int64_t nsamp_out, bool device_rows);

// Device address of the status word of dd_execute_noalloc's fixed array on
// the current device (looked up once per device; see dd_noalloc.cu).
dd_status noalloc_status_word(int **out);

// Preferred tile shape for a dtype.
dd_tiles default_tiles(dd_dtype t);

// Tile shapes tried, in order, when the plan picks one itself: the preferred
// shape, then fewer channels per stage, then fewer DMs per CTA (more time
// warps), down to one DM per CTA, which always fits.
std::vector<dd_tiles> auto_tiles(dd_dtype t);

// Validate a tile shape for dtype and compute the launch geometry for the
// plan (shared-memory window bound over every DM tile and channel).
dd_status make_geometry(dd_plan_s *p, dd_dtype t, const dd_tiles &tl, Geometry *g);

// The same for the sorted DMs [d0, d0 + nd) only.
dd_status make_geometry_range(dd_plan_s *p, dd_dtype t, const dd_tiles &tl, int d0, int nd,
                              Geometry *g);

// Geometry for the plan's current tile shape, cached.
dd_status plan_geometry(dd_plan_s *p, dd_dtype t, Geometry *g);

// Geometry for one execution of nsamp_out samples: the plan's shape if the
// caller or the autotuner set one, else the shape expected to finish first.
dd_status execution_geometry(dd_plan_s *p, dd_dtype t, int64_t nsamp_out, Geometry *g);

// Modelled time of an execution by the direct kernel, to compare lengths by
// (microseconds, or rounds of tiles where the shape has been set).
double execution_time(dd_plan_s *p, dd_dtype t, int64_t nsamp_out);

// Modelled time of the direct kernel in one of the shapes that
// execution_geometry chooses from (-1 for another shape), and of one of its
// tiles, alone on an SM.
double direct_time_us(dd_plan_s *p, dd_dtype t, const dd_tiles &tl, int64_t nsamp_out, int sms);
double direct_tile_us(dd_plan_s *p, dd_dtype t, const dd_tiles &tl);

// Time to finish tiles that are handed out in order, each to the first free SM.
class Makespan {
  public:
    explicit Makespan(int sms) : sms_(std::max(1, sms)) { free_[0.0] = sms_; }
    void run(int64_t tiles, double us);
    double end() const { return end_; }

  private:
    int sms_;
    double end_ = 0;
    std::map<double, int> free_;  // when free -> SMs
};

// The tile shape that a batch or a server takes for its beams while none has
// been set; false: no shape fits all of them.
struct BatchLoad {
    dd_plan_s *plan;
    int64_t nsamp_out;
};
bool shared_tiles(const std::vector<BatchLoad> &beams, dd_dtype t, dd_tiles *out);

// Launch shape for the DMs of the last, partly filled DM tile of geometry g,
// run as a launch of their own (see dd_plan.cpp); cached per tile shape.
dd_status tail_geometry(dd_plan_s *p, dd_dtype t, const Geometry &g, bool *found,
                        Geometry *tail);

// Device tables for the current device, uploaded on first use.
dd_status device_tables(dd_plan_s *p, DevTables **out);

// Launch the de-dispersion of one beam on stream: the grouped kernel
// (dd_group.cu) where it is expected to be faster, else the direct kernel
// (dd_kernel_*.cu).  kAuto: with a table that the plan does not have yet, the
// first execution runs directly and the table is built behind it, unless this
// execution gains more than the table costs it or a graph captures it; kNow
// waits for the table.
enum class Grouped { kNever, kAuto, kNow };
// With split_tail, the DMs of a last DM tile that is at most half full run
// as a second launch with their own tile shape, on a library stream forked
// from and joined back into `stream`, so its CTAs fill the SMs the first
// launch leaves idle in its last wave instead of padding a whole DM tile --
// when a count of the two launches' waves says that finishes earlier.
dd_status launch_dedisperse(dd_plan_s *p, const Geometry &g, const DevTables &dt,
                            const void *in, dd_dtype dtype, int64_t in_pitch, int64_t nsamp_in,
                            float *out, int64_t out_pitch, int64_t nsamp_out, void *stream,
                            bool split_tail = true, Grouped grouped = Grouped::kAuto);

void count_launch(int n = 1);

// SMs of a device (0 if unknown).
int sm_count(int dev);

// Boxcar search accumulators: clear them (dd_detect.cu), and turn them into
// mean, std, S/N and peak t for an integer-valued plane.
dd_status detect_begin(int ndm, int nlevels, double *mean, double *sd, double *snr,
                       cudaStream_t s);
dd_status detect_finalize_int(int ndm, int64_t nsamp, int nlevels, double *mean, double *sd,
                              double *snr, int64_t *tpk, cudaStream_t s);

// One uint8 de-dispersion launch (no remainder split) with the boxcar search
// fused into its epilogue (dd_launch.cpp): g must have 4 DMs x 8 words per
// thread and one time warp (1024-sample tiles); det_cnt holds
// g.ntile_d * ntile_t zeroed ints.
dd_status launch_dedisperse_detect(dd_plan_s *p, const Geometry &g, const DevTables &dt,
                                   const void *in, int64_t in_pitch, int64_t nsamp_in,
                                   float *out, int64_t out_pitch, int64_t nsamp_out,
                                   const DetectTargets &det, int *det_cnt, void *stream);

}  // namespace dd
