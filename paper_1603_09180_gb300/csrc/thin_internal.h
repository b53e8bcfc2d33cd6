// thin_internal.h -- declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/thin.h"
#include "thin_layout.h"

namespace thin {

// An NVTX range over a C-ABI call, for Nsight Systems timelines.  The NVTX
// header only forwards to a profiler that is attached; otherwise it costs a
// branch.
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// Validated description of one image handed to an engine.
struct JobSpec {
    void *img;
    int w, h;
    size_t pitch;
    int dtype;      // THIN_U8 / THIN_U16
    uint32_t lam;
    int adj;        // THIN_ADJ_8_4 / THIN_ADJ_4_8
    int done_slot = -1;  // resident engine: completion record to post when the image is finished, -1 none
    bool fits_cluster = false;  // tiled engine: the image fits a cluster, so its stats keep the resident engine's rule at a cap
};

// The resident engine's rule at a phase cap: converged if the last three
// phases changed nothing.  `last`: last phase that lowered a point, -1 if none.
// Where a default call takes another engine for images that fit a cluster (or
// the wide mode), its status at a cap stays what this rule says, whenever that
// engine saw its fixed point.
inline bool quiet_at_cap(const thin_options &o, long long last)
{
    return o.max_phases >= 4 && last - o.start_phase < o.max_phases - 3;  // (in this order nothing overflows)
}

inline int elem_size(int dtype) { return dtype == THIN_U16 ? 2 : 1; }

// The point test's mode word for the kernels: bit 0 the F^- reading
// (thin_rule), bit 1 the operator (thin_op); the kernels add bit 2, the
// image's adjacency pair (thin_adj).
inline int test_mode(const thin_options &o) { return (o.rule & 1) | ((o.op & 1) << 1); }

// Naive engine: one launch per subfield phase over the whole image, in place.
int naive_run(const JobSpec &job, const thin_options &opt, cudaStream_t stream, thin_stats *out);

// Tiled engine: TMA-staged tiles, temporal blocking, active-tile worklist,
// one persistent cooperative launch for any number of images.
int tiled_run(const JobSpec *jobs, int n, const thin_options &opt, cudaStream_t stream, thin_stats *out);

// Resident engine: each image held in the shared memory of one thread-block
// cluster of C blocks (kClusterSizes) of 16 warps, one block per SM, for its
// whole run; one launch per cluster size and element size.
// Device-side records of the resident engine (thin_resident.cu).
struct ResJob {
    unsigned long long img;    // the caller's image, thinned in place
    unsigned long long pitch;  // bytes between rows
    int w, h, dtype;
    unsigned lam;
    int rows;   // image rows per block (even)
    int rp;     // shared row pitch in bytes: 16 B pad | w * es | pad to 16 | 16 B pad
    int cw;     // cells per row = ceil(w / 8)
    int wpr;    // bitmap words per cell row = ceil(cw / 32)
    int bulk;   // rows are 16-byte aligned and a multiple of 16 bytes: stage them by bulk copy
    int index;  // position of the job in the caller's list
    int hr;     // halo rows copied from each neighbouring block (even; 0 for a one-block cluster)
    int steph;  // phases between exchanges of halo rows
    int adj;    // thin_adj
    int done_slot;  // completion record of the job (ResArgs::done), -1 none
    unsigned long long ck;  // first word of the job's checkpoint of its dirty bitmaps (ResArgs::ckbits)
};

// Where a job paused at the end of its last time slice (ResArgs::slice).
struct ResRun {
    long long g;     // global phase index to resume at
    long long last;  // last phase that lowered a point, -1 if none
    int resumed;     // 1: the job has a checkpoint to resume from
    int pad;
};

struct ResStat {
    unsigned long long lowered;
    unsigned long long tested;   // point tests on own rows
    long long last_change;  // global phase index, -1 if none
    long long phases;
    int converged;
    int error;
};

// Completion record of one job, in host-mapped memory: the job's stats, then
// `flag` set to 1 (a system-scope release store) once its image is back in
// the caller's memory.  The host resets flag to 0 before the launch.
struct ResDone {
    ResStat st;
    int error;       // the launch's error word when the job finished
    unsigned flag;
};

struct ResCtl {
    unsigned head, tail;  // job ring: entries head .. tail - 1 wait to run (ResArgs::ring)
    int error;
    unsigned bar_count;  // grid barrier of a wide launch
    unsigned bar_gen;
    long long gl_last;   // wide launch: last phase that lowered a point anywhere, -1 if none
};

struct ResArgs {
    const ResJob *jobs;
    ResStat *st;
    ResCtl *ctl;
    int njobs;
    int rule;
    long long start_phase;
    long long max_phases;
    unsigned long long timeout_ns;
    // Wide launch (strips > 0): one image over `strips` clusters, cluster s
    // holding strip s; boundary rows cross between clusters through xbuf.
    int strips;
    int pad;
    unsigned char *xbuf;        // per block: 2 sides x 2 step parities x xslot bytes
    unsigned long long xslot;
    ResDone *done;              // completion records (ResJob::done_slot), nullptr: none
    // Job ring and time slices.  Clusters take jobs from the ring in order.  With
    // slice > 0, a cluster whose job has run `slice` more steps while other jobs
    // wait stores the job's state (its rows to the image, its dirty bitmaps to
    // ckbits, its phase to run[]) and puts it back at the ring's tail.
    int *ring;                  // cap entries: job indices
    unsigned *tag;              // per entry: 1 + the round of the ring it was written in
    ResRun *run;                // per job
    uint32_t *ckbits;           // checkpointed dirty bitmaps
    unsigned cap;
    int slice;                  // steps per time slice (a power of two), 0: jobs run to the end once started
};

// A resident launch prepared on the host (device tables uploaded), ready to
// be enqueued any number of times: see resident_prepare / _enqueue /
// _collect / _release.
struct ResidentPrepared {
    int n = 0, C = 0, grid = 0, strips = 0, es = 1;
    size_t smem = 0;
    bool async_alloc = true;
    char *base = nullptr;         // one device allocation holding everything below
    char *live = nullptr, *pristine = nullptr;  // per-run state (stats, control, job ring) and its initial copy
    size_t live_bytes = 0;
    std::vector<int> order;       // launch position -> index in the prepared job list
    ResArgs P;                    // the kernel's argument block
};
// strips > 0: one image (n == 1) over `strips` clusters of C blocks, one
// cooperative launch (the wide mode for images larger than one cluster).
int resident_prepare(const JobSpec *jobs, int n, int C, const thin_options &opt, cudaStream_t stream,
                     bool async_alloc, ResidentPrepared *R, int strips = 0, ResDone *done = nullptr);
cudaError_t resident_enqueue(const ResidentPrepared &R, cudaStream_t stream);
int resident_collect(const ResidentPrepared &R, const thin_options &opt, cudaStream_t stream, thin_stats *out);
// The public stats of a finished resident job (error: the launch's error word).
void resident_stats(const ResStat &S, int error, const thin_options &opt, thin_stats *o);
void resident_release(ResidentPrepared &R, cudaStream_t stream);
// Smallest cluster whose shared memory holds a w x h image
// of `dtype`, 0 if none.
int resident_cluster_size(int w, int h, int dtype, size_t smem_limit, int *rows_out, int *rp_out);
// Largest resident cluster on the current device: 16 where it can run, else 8.
int resident_max_cluster(size_t smem_limit);
// Shared memory one block may take (one block per SM).
size_t resident_smem_limit();
// Wide mode: the fewest strips (clusters of *c_out blocks, the
// largest cluster size that works) whose shared memory holds the image, all
// clusters resident at once; 0 if none.
int resident_wide_strips(int w, int h, int dtype, size_t smem_limit, int *c_out);

// A tiled launch prepared on the host (opaque; thin_tiled.cu).
struct TiledPrepared;
// max_grid > 0 caps the launch at that many blocks of 8 warps (serving keeps the
// rest of the GPU free for the resident launches of its other lanes).
int tiled_prepare(const JobSpec *jobs, int n, const thin_options &opt, cudaStream_t stream, bool async_alloc,
                  TiledPrepared **out, int max_grid = 0);
cudaError_t tiled_enqueue(const TiledPrepared *T, cudaStream_t stream);
int tiled_collect(const TiledPrepared *T, const thin_options &opt, cudaStream_t stream, thin_stats *out);
void tiled_release(TiledPrepared *T, cudaStream_t stream);

// The shape the tiled engine takes by itself for these images; true if they are
// enough for its large tiles to fill the GPU (nothing to tune then).
bool tiled_fills(const JobSpec *jobs, int n, int *tw, int *th, int *H);

// Defaults of the tiled engine (tile width/height in pixels, halo)
// where the caller sets only some of them.
void tiled_defaults(int *tw, int *th, int *halo);

// Mosaic engine (thin_mosaic.cu): a few images whose tiles all fit in shared
// memory at once, one block to a tile.
// A call of at most this many images (of one element size) goes to the mosaic
// engine where their tiles fit: it spreads an image over far more SMs than a
// cluster has, with no barrier over the grid.  Resident against mosaic (tiles in
// all block slots), one image: 512^2 u8 at lambda = 20 3.9 / 2.3 ms, 1000^2
// 13.1 / 4.6, 2048^2 at lambda = 30 (wide) 21.6 / 10.2, 4096^2 35.1 / 32.0, 64^2
// 0.28 / 0.26; 16 images of 512^2 6.7 / 5.5, of 200^2 1.82 / 1.59; 32 images
// 7.1 / 7.2 and 1.81 / 1.88.
constexpr int kMosaicMax = 16;
// The best tile shape for these images; false if they do not fit.
bool mosaic_shape(const JobSpec *jobs, int n, MosaicShape *out);
struct MosaicPrepared {
    int n = 0, es = 1, grid = 0, smem = 0, halo = 0;
    bool async_alloc = true;
    char *base = nullptr, *live = nullptr;  // one allocation; the part to zero before a run
    size_t live_bytes = 0, o_st = 0, o_err = 0;
    std::vector<char> args;                 // the kernel's argument block
};
int mosaic_prepare(const JobSpec *jobs, int n, const MosaicShape &shape, const thin_options &opt, cudaStream_t stream,
                   bool async_alloc, MosaicPrepared *M);
cudaError_t mosaic_enqueue(const MosaicPrepared &M, cudaStream_t stream);
int mosaic_collect(const MosaicPrepared &M, const thin_options &opt, cudaStream_t stream, thin_stats *out);
void mosaic_release(MosaicPrepared &M, cudaStream_t stream);

int cuda_status(cudaError_t e);

// Cluster sizes of the resident engine.  3 serves images of 430 to 640 KB
// (512^2 u16: 50 clusters of 3 fit the GPU, 36 of 4; 192 such images 23.9 ->
// 22.5 ms).  5 and 6 were tried too: images of 0.9 to 1.3 MB are better off as
// tiles beside larger ones (1024 uneven images 190 ms without, 200 with).
constexpr int kClusterSizes[] = {1, 2, 3, 4, 8, 16};
// Resident launch groups of a batch at most: one per cluster size and element
// size (u8, u16).  Execution::enqueue needs that many helper streams, and one
// event more.
constexpr int kMaxResidentGroups = 2 * int(sizeof kClusterSizes / sizeof kClusterSizes[0]);

// Launch groups of a batch: (cluster size, job indices) for the resident
// engine, job indices for the tiled engine.
struct Grouping {
    std::vector<std::pair<int, std::vector<int>>> resident;
    struct Wide {
        int job, strips, C;
    };
    std::vector<Wide> wide;  // one wide launch each
    std::vector<int> mosaic;  // one launch
    MosaicShape mosaic_tile;
    std::vector<int> tiled;
    std::vector<char> tiled_fits;  // per entry of tiled: it would fit a cluster
    // a grouping made with `spare` needs less scratch
    bool can_spare() const { return !mosaic.empty() || std::count(tiled_fits.begin(), tiled_fits.end(), 1) > 0; }
};
// allow_wide: large images may take the wide resident mode (a cooperative
// launch over the whole GPU); serving turns it off so that its lanes share
// the GPU.  spare: images that fit a cluster or the wide mode stay there, which
// need next to no scratch (the mosaic engine takes twice the images' size and
// the tiled engine once).
int group_jobs(const std::vector<JobSpec> &specs, const thin_options &o, Grouping *G, bool allow_wide = true,
               bool spare = false);

// Every launch group of a batch, prepared; enqueue() is device work only
// (resident groups forked onto up to kMaxResidentGroups side streams with
// events, joined back before the others), so it can be captured in a CUDA graph.
struct Execution {
    std::vector<JobSpec> specs;
    thin_options opt;
    bool async = true;
    ResDone *done = nullptr;  // completion records for the resident groups' jobs (JobSpec::done_slot)
    int tiled_max_grid = 0;   // cap on the tiled launch's blocks, 0 = none
    std::vector<ResidentPrepared> res;
    std::vector<std::vector<int>> res_idx;
    std::vector<ResidentPrepared> wide;
    std::vector<int> wide_idx;
    MosaicPrepared mosaic;
    std::vector<int> mosaic_idx;
    TiledPrepared *tiled = nullptr;
    std::vector<int> tiled_idx;
    int prepare(const std::vector<JobSpec> &specs, const Grouping &G, const thin_options &o, cudaStream_t s,
                bool async_alloc);
    // prepare with stream-ordered scratch; where that runs out, once more by the grouping of options `group`
    // that spares it (G is replaced).
    int prepare_or_spare(const std::vector<JobSpec> &specs, Grouping *G, const thin_options &group, const thin_options &o,
                         cudaStream_t s);
    cudaError_t enqueue(cudaStream_t s, cudaStream_t *side, cudaEvent_t *ev) const;
    int collect(cudaStream_t s, thin_stats *out) const;  // out[k] for specs[k]; waits for s
    void release(cudaStream_t s);
};

// Helper streams and events of the calling host thread for Execution::enqueue
// (created once per thread and device, kept until the process exits or the thread gives them back).
cudaError_t thread_side_streams(cudaStream_t **side, cudaEvent_t **ev);
// For a thread of the library's own that ends (its work has finished): 12 streams take about 6 MiB of device memory.
void release_thread_side_streams();

// Identity of the calling thread's current context, 0 if it cannot be had.
unsigned long long current_context_id();

// Stream-ordered device memory for a call's scratch (freed with cudaFreeAsync).
cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t stream);

// Raises a kernel's dynamic shared-memory cap to the device's opt-in maximum.
// Always the same value, so host threads launching the kernel at once with
// different shared-memory sizes never lower the cap under one another.
cudaError_t allow_max_dynamic_smem(const void *kernel);

}  // namespace thin
