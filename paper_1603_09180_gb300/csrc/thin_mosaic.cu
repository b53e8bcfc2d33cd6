// thin_mosaic.cu -- the mosaic engine: a few images whose tiles all fit on the
// GPU at once.
//
// One cooperative launch, one block to a tile, two blocks to an SM.  A block
// keeps its tile, a halo and their dirty bits in shared memory for the whole
// run and advances in steps of H phases (thin_tile.cuh), as a tile visit of the
// tiled engine does.  Between steps it publishes the rim of its tile (the
// pixels and dirty bits its neighbours hold as halo) in global memory, sets its
// flag, waits for the flags of its eight neighbours and fetches their rims.  No
// barrier spans the grid: a tile that is busy in one step and idle in the next
// delays only its surroundings, and by the difference of the sums, not by the
// sum of the differences.
//
// The halo is one pixel wider than a step has phases, so that every mark a
// neighbour's move makes inside the tile is made by the tile's own block (see
// thin_tiled.cu); a block's own bits are always exact and the halo's are
// replaced by its neighbours' each step.  The published rims lie in a ping-pong
// pair by the step's parity: a block writes the rim of step s + 1 only after its
// neighbours' flags say that they have finished step s - 1, hence have read the
// rim in that slot.
//
// Stop.  A block whose tile has no dirty bit left after step s counts itself in
// the step's counter; the one that completes the count has found the fixed
// point, which is the same for every order of the blocks, and posts it.  The
// others leave at their next look; steps run past that point change nothing.
// Every wait ends with the posted stop, a posted error or a time limit.
//
// What bounds it: in busy steps issue, as in the other engines; in sparse ones
// the latency chain of a phase in the busiest tile (about 2500 cycles) and, per
// step of 15 phases, about 7000 cycles to publish, signal and fetch.  Single
// images against clusters (one strip of rows to a block, two cluster barriers
// per 8 phases) and the wide mode (a grid barrier per 8 phases): 64^2 at
// lambda = 10 224 -> 200 us, 512^2 at lambda = 0 391 -> 257 us, 4096^2 1.31 ->
// 1.02 ms, at lambda = 30 42.5 -> 35.1 ms, 1000^2 at lambda = 30 13.0 -> 4.6 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <vector>

#include "thin_internal.h"
#include "thin_tile.cuh"

namespace thin {

namespace {

constexpr int kCountSlots = 1024;  // step counters of an image, used in turn (blocks are never so far apart)

struct MosImage {
    unsigned long long img, pitch;  // the caller's image
    unsigned long long rim[2];      // published pixels, laid out as the image
    unsigned long long rim_pitch;   // a multiple of 16
    unsigned long long bits[2];     // published dirty bits: a byte per cell, bit p for parity p
    int w, h, adj;
    unsigned lam;
    int tiles_x, tiles_y, tile_base;
    int cells_x;                    // cells of a row of `bits`
    int aligned;                    // the image's rows start at 16-byte boundaries
};

// Zero at the start of a run.
struct MosStat {
    unsigned long long lowered, tested;
    unsigned long long last;        // 1 + last phase that lowered a point, 0 if none
    unsigned stop;                  // steps after which no bit was dirty, 0 while some are
    unsigned pad;
};

// (The images travel as launch arguments: no table to copy before a run.)
struct MosArgs {
    MosImage imgs[kMosaicMax];
    MosStat *st;
    unsigned *count;                // per image: kCountSlots step counters
    unsigned *flag;                 // per tile: steps published
    unsigned *error;
    int n;
    int tw, th, halo, hr, rule;
    long long start_phase, max_phases;
    unsigned long long timeout_ns;
    TileLayout tl;
};

__device__ const DecisionTable d_mos_decisions = kDecisionTable;

__device__ __forceinline__ unsigned ld_relaxed(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Waits until every neighbour has published `steps` steps: 0 then, 1 if the
// image's stop is posted, 2 after an error or the time limit.  All threads call
// it; it ends with a block barrier.
__device__ int wait_neighbours(const MosArgs &P, const MosImage &I, MosStat *S, int tx, int ty, unsigned steps, int *s_out)
{
    if (threadIdx.x < 32) {
        const int d = threadIdx.x + (threadIdx.x >= 4);  // the centre of 3 x 3 left out
        const int nx = tx + d % 3 - 1, ny = ty + d / 3 - 1;
        const bool have = threadIdx.x < 8 && nx >= 0 && nx < I.tiles_x && ny >= 0 && ny < I.tiles_y;
        const unsigned *f = P.flag + I.tile_base + ny * I.tiles_x + nx;
        const unsigned long long t0 = gtimer();
        int out = 0;
        for (;;) {
            const unsigned v = have ? ld_relaxed(f) : steps;
            const unsigned stop = ld_relaxed(&S->stop), err = ld_relaxed(P.error);
            if (__any_sync(0xffffffffu, err != 0)) {
                out = 2;
                break;
            }
            if (__all_sync(0xffffffffu, v >= steps)) {
                out = __any_sync(0xffffffffu, stop != 0) ? 1 : 0;
                break;
            }
            if (__any_sync(0xffffffffu, stop != 0)) {
                out = 1;
                break;
            }
            if (__any_sync(0xffffffffu, gtimer() - t0 > P.timeout_ns)) {
                if (threadIdx.x == 0) atomicCAS(P.error, 0u, unsigned(THIN_ERR_TIMEOUT));
                out = 2;
                break;
            }
        }
        __threadfence();  // what the flags announce is read after them
        if (threadIdx.x == 0) *s_out = out;
    }
    __syncthreads();
    return *s_out;
}

// A block's tile as the exchange of rims sees it, in shared memory: the two
// functions of the exchange are called once a step and kept out of line, so that
// the phases keep their registers.
struct MosTile {
    char *rim[2];
    unsigned char *bits[2];
    unsigned long long rim_pitch;
    int cells_x, x0, y0, th, row_bytes, hr, words, dirty_off;
    int cols, rows;      // cells of the tile
    int inner;           // 16-byte vectors of a row of the tile
    bool left, right, above, below;  // neighbours there
};
constexpr int kOffMosTile = kOffTile - 112;
static_assert(kOffMosTile >= int(kOffBar) && sizeof(MosTile) <= 112, "the tile's record overlaps the control words");

// The rims travel as 16-byte vectors: 2 HR rows of the tile's width (with the
// halo's corners when fetched), then ES vectors a side of every row of the tile
// (2 ES = 1 << ES).
//
// Fetches the neighbours' rims of step `step` and their dirty bits into the
// halo.  All loads are issued before the first is used.
template <int ES>
__device__ __noinline__ void fetch_rims(uint8_t *smem, unsigned step)
{
    const MosTile &t = *reinterpret_cast<const MosTile *>(smem + kOffMosTile);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int es = ES;
    const int HR = t.hr, words = t.words, cols = t.cols, rows = t.rows, inner = t.inner;
    const bool left = t.left, right = t.right, above = t.above, below = t.below;
    uint8_t *tile = smem + kOffTile;
    uint32_t *dirty = reinterpret_cast<uint32_t *>(smem + t.dirty_off);
    const char *rim = t.rim[step & 1];
    const unsigned char *bits = t.bits[step & 1];
    // bits of the halo's cell rows, a lane to a cell (two rows a warp at most: HR <= 16)
    const bool col = lane < cols + 4 && (left || lane >= 2) && (right || lane < cols + 2);
    unsigned hv[2] = {0u, 0u};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int r = warp + q * kWarps;
        if (r < HR && col && (r < HR / 2 ? above : below))
            hv[q] = __ldcg(bits + size_t(t.y0 / 2 + (r < HR / 2 ? r - HR / 2 : rows + r - HR / 2)) * t.cells_x + t.x0 / 8 - 2 + lane);
    }
    // bits of the two cells on either side of the tile's cell rows, a thread to a row
    unsigned side_l = 0, side_r = 0;
    if (tid < rows) {
        const unsigned char *at = bits + size_t(t.y0 / 2 + tid) * t.cells_x + t.x0 / 8;
        if (left) side_l = __ldcg(reinterpret_cast<const unsigned short *>(at - 2));
        if (right) side_r = __ldcg(reinterpret_cast<const unsigned short *>(at + cols));
    }
    // rows above and below, a warp to a row and a lane to a vector (HR <= 16, at most 32 vectors)
    const int v = lane - es;  // the tile's first vector is 0
    const bool in_row = v < inner + es && (left || v >= 0) && (right || v < inner);
    const char *from = rim + (t.x0 * es + 16 * v);
    uint8_t *to = tile + kPadCols * es + 16 * v;
    constexpr int kSide = mosaic_side_turns(ES);
    uint4 row[4], side[kSide];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = warp + q * kWarps, y = r < HR ? r - HR : t.th + r - HR;
        if (r < 2 * HR && in_row && (r < HR ? above : below))
            row[q] = __ldcg(reinterpret_cast<const uint4 *>(from + (long long)(t.y0 + y) * t.rim_pitch));
    }
    // columns left and right: es vectors a side and row, of every row
    const int side_shift = es, side_q = tid & (2 * es - 1);
    const bool side_have = side_q >= es ? right : left;
    const int side_x = side_q >= es ? 16 * (inner + side_q - es) : 16 * (side_q - es);
#pragma unroll
    for (int q = 0; q < kSide; ++q) {
        const int y = (tid + q * kThreads) >> side_shift;
        if (y < t.th && side_have)
            side[q] = __ldcg(reinterpret_cast<const uint4 *>(rim + (size_t(t.y0 + y) * t.rim_pitch + t.x0 * es + side_x)));
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = warp + q * kWarps, y = r < HR ? r - HR : t.th + r - HR;
        if (r < 2 * HR && in_row && (r < HR ? above : below)) *reinterpret_cast<uint4 *>(to + (y + HR) * t.row_bytes) = row[q];
    }
#pragma unroll
    for (int q = 0; q < kSide; ++q) {
        const int y = (tid + q * kThreads) >> side_shift;
        if (y < t.th && side_have)
            *reinterpret_cast<uint4 *>(tile + (y + HR) * t.row_bytes + kPadCols * es + side_x) = side[q];
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int r = warp + q * kWarps;
        const unsigned b0 = __ballot_sync(0xffffffffu, hv[q] & 1u), b1 = __ballot_sync(0xffffffffu, hv[q] & 2u);
        const unsigned b2 = __ballot_sync(0xffffffffu, hv[q] & 4u), b3 = __ballot_sync(0xffffffffu, hv[q] & 8u);
        if (r < HR && lane < 4)
            dirty[lane * words + (r < HR / 2 ? r : rows + r)] = lane == 0 ? b0 : lane == 1 ? b1 : lane == 2 ? b2 : b3;
    }
    if (tid < rows) {
        const uint32_t own = ((1u << cols) - 1u) << 2;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const uint32_t l = ((side_l >> p) & 1u) | (((side_l >> (8 + p)) & 1u) << 1);
            const uint32_t r = ((side_r >> p) & 1u) | (((side_r >> (8 + p)) & 1u) << 1);
            uint32_t &w = dirty[p * words + HR / 2 + tid];
            w = (w & own) | l | (r << (cols + 2));
        }
    }
}

// Publishes the tile's rim after step `step`: its first and last HR rows, its
// first and last 16 columns, and their dirty bits.  Returns nonzero where the
// tile has a dirty bit left.
template <int ES>
__device__ __noinline__ uint32_t publish_rim(uint8_t *smem, unsigned step)
{
    const MosTile &t = *reinterpret_cast<const MosTile *>(smem + kOffMosTile);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int es = ES;
    const int HR = t.hr, words = t.words, cols = t.cols, rows = t.rows, inner = t.inner;
    uint8_t *tile = smem + kOffTile;
    uint32_t *dirty = reinterpret_cast<uint32_t *>(smem + t.dirty_off);
    char *rim = t.rim[step & 1];
    unsigned char *bits = t.bits[step & 1];
    const uint8_t *src = tile + HR * t.row_bytes + kPadCols * es;
    char *dst = rim + size_t(t.y0) * t.rim_pitch + t.x0 * es;
    const int bands = min(t.th, 2 * HR);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = warp + q * kWarps, y = r < HR ? r : t.th - bands + r;
        if (r < bands && lane < inner)
            __stcg(reinterpret_cast<uint4 *>(dst + size_t(y) * t.rim_pitch + 16 * lane),
                   *reinterpret_cast<const uint4 *>(src + y * t.row_bytes + 16 * lane));
    }
    const int q0 = tid & (2 * es - 1), x0 = q0 >= es ? 16 * (inner - 2 * es + q0) : 16 * q0;
#pragma unroll
    for (int q = 0; q < mosaic_side_turns(ES); ++q) {
        const int y = (tid + q * kThreads) >> es;
        if (y >= HR && y < t.th - HR)
            __stcg(reinterpret_cast<uint4 *>(dst + size_t(y) * t.rim_pitch + x0),
                   *reinterpret_cast<const uint4 *>(src + y * t.row_bytes + x0));
    }
    uint32_t any = 0;
    if (tid < rows) {
        const uint32_t *w = dirty + HR / 2 + tid;
        unsigned l = 0, r = 0;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const uint32_t d = (w[p * words] >> 2) & ((1u << cols) - 1u);
            any |= d;
            l |= ((d & 1u) | ((d & 2u) << 7)) << p;
            r |= (((d >> (cols - 2)) & 1u) | (((d >> (cols - 1)) & 1u) << 8)) << p;
        }
        unsigned char *at = bits + size_t(t.y0 / 2 + tid) * t.cells_x + t.x0 / 8;
        __stcg(reinterpret_cast<unsigned short *>(at), static_cast<unsigned short>(l));
        __stcg(reinterpret_cast<unsigned short *>(at + cols - 2), static_cast<unsigned short>(r));
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int i = warp + q * kWarps, r = i < HR / 2 ? i : rows - HR + i;
        if (i < HR && lane < cols) {
            const uint32_t *w = dirty + HR / 2 + r;
            const int c = lane + 2;
            __stcg(bits + size_t(t.y0 / 2 + r) * t.cells_x + t.x0 / 8 + lane,
                   static_cast<unsigned char>(((w[0] >> c) & 1u) | (((w[words] >> c) & 1u) << 1) |
                                              (((w[2 * words] >> c) & 1u) << 2) | (((w[3 * words] >> c) & 1u) << 3)));
        }
    }
    return any;
}

// ES: element size of every image of the launch (1: u8, 2: u16).
template <int ES>
__global__ void __launch_bounds__(kThreads, 2) k_mosaic(MosArgs P)
{
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ int s_go, s_end;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b = blockIdx.x;
    int k = 0;
    while (k + 1 < P.n && P.imgs[k + 1].tile_base <= b) ++k;
    const MosImage I = P.imgs[k];
    MosStat *S = P.st + k;
    const int ty = (b - I.tile_base) / I.tiles_x, tx = (b - I.tile_base) - ty * I.tiles_x;
    constexpr int es = ES;
    TileLayout L = P.tl;
    L.row_bytes = (P.tw + 2 * kPadCols) * es;
    const int words = L.rows / 2, HR = P.hr;
    Visit V;
    V.w = I.w;
    V.h = I.h;
    V.x0 = tx * P.tw;
    V.y0 = ty * P.th;
    V.tw = P.tw;
    V.th = P.th;
    V.hr = HR;
    uint8_t *tile = smem + kOffTile;  // row 0: image row y0 - HR, column 0: image column x0 - kPadCols
    TileCtrl *ctrl = reinterpret_cast<TileCtrl *>(smem + kOffCtrl);
    uint32_t *dirty = reinterpret_cast<uint32_t *>(smem + L.dirty_off);
    const PointRule rule = point_rule(smem, P.rule | (I.adj << 2), I.lam, es, true);

    load_decisions(smem, d_mos_decisions);
    for (int i = tid; i < 4 * words; i += kThreads) dirty[i] = 0xffffffffu;  // every group is tested in the first phase of its parity
    // the tile and its halo as far as they lie in the image
    {
        const int ya = max(0, V.y0 - HR), yb = min(I.h, V.y0 + P.th + HR);
        const int xa = max(0, V.x0 - kPadCols) * es, xb = min(I.w, V.x0 + P.tw + kPadCols) * es;
        const char *img = reinterpret_cast<const char *>(I.img);
        uint8_t *dst = tile - (V.x0 - kPadCols) * es;
        const int vpr = I.aligned ? (xb - xa) / 16 : 0;
        for (int y = ya + warp; y < yb; y += kWarps) {
            const char *g = img + size_t(y) * I.pitch;
            uint8_t *s = dst + (y - V.y0 + HR) * L.row_bytes;
            for (int v = lane; v < vpr; v += 32)
                *reinterpret_cast<uint4 *>(s + xa + 16 * v) = __ldcg(reinterpret_cast<const uint4 *>(g + xa + 16 * v));
            for (int x = xa + 16 * vpr + lane; x < xb; x += 32) s[x] = uint8_t(__ldcg(g + x));
        }
    }
    if (tid == 0) {
        ctrl->qn[0] = 0u;
        ctrl->qn[1] = 0u;
        MosTile &t = *reinterpret_cast<MosTile *>(smem + kOffMosTile);
        t.rim[0] = reinterpret_cast<char *>(I.rim[0]);
        t.rim[1] = reinterpret_cast<char *>(I.rim[1]);
        t.bits[0] = reinterpret_cast<unsigned char *>(I.bits[0]);
        t.bits[1] = reinterpret_cast<unsigned char *>(I.bits[1]);
        t.rim_pitch = I.rim_pitch;
        t.cells_x = I.cells_x;
        t.x0 = V.x0;
        t.y0 = V.y0;
        t.th = P.th;
        t.row_bytes = L.row_bytes;
        t.hr = HR;
        t.words = words;
        t.dirty_off = L.dirty_off;
        t.cols = P.tw / 8;
        t.rows = P.th / 2;
        t.inner = P.tw * es / 16;
        t.left = tx > 0;
        t.right = tx + 1 < I.tiles_x;
        t.above = ty > 0;
        t.below = ty + 1 < I.tiles_y;
    }
    __syncthreads();

    long long g0 = P.start_phase, last = -1;
    unsigned s = 0;  // steps done
    int nlow = 0, ntest = 0;
    for (;;) {
        const long long done = g0 - P.start_phase;
        if (P.max_phases >= 0 && done >= P.max_phases) break;
        V.Hs = (P.max_phases >= 0 && P.max_phases - done < P.halo) ? int(P.max_phases - done) : P.halo;
        V.g0 = g0;
        if (s > 0) {
            if (wait_neighbours(P, I, S, tx, ty, s, &s_go) != 0) break;
            fetch_rims<ES>(smem, s);
            if (tid == 0) {
                ctrl->qn[0] = 0u;
                ctrl->qn[1] = 0u;
            }
            __syncthreads();
        }
        int chg_j = -1;
        visit_phases<typename std::conditional<ES == 1, uint8_t, uint16_t>::type, kThreads>(L, smem, V, rule, nlow, ntest,
                                                                                          chg_j);
        if (chg_j >= 0) last = g0 + chg_j;
        g0 += V.Hs;
        ++s;
        const uint32_t any = publish_rim<ES>(smem, s);
        // (the barrier and the flag's release order every thread's stores before the flag)
        const int busy = __syncthreads_or(any != 0);
        if (tid == 0) {
            unsigned *count = P.count + size_t(k) * kCountSlots;
            const unsigned tiles = unsigned(I.tiles_x) * unsigned(I.tiles_y);
            if (b == I.tile_base) *reinterpret_cast<volatile unsigned *>(&count[(s + kCountSlots / 2) % kCountSlots]) = 0u;
            st_release(P.flag + b, s);
            if (!busy && atomicAdd(&count[s % kCountSlots], 1u) == tiles - 1) atomicCAS(&S->stop, 0u, s);
        }
    }
    // Results.  The neighbours have read this tile's first state out of the image before it is overwritten.
    if (s > 0) wait_neighbours(P, I, S, tx, ty, 1u, &s_end);
    nlow = __reduce_add_sync(0xffffffffu, nlow);
    ntest = __reduce_add_sync(0xffffffffu, ntest);
    if (lane == 0 && nlow) atomicAdd(&S->lowered, (unsigned long long)nlow);
    if (lane == 0 && ntest) atomicAdd(&S->tested, (unsigned long long)ntest);
    if (last >= 0) atomicMax(&S->last, (unsigned long long)(last + 1));
    {
        const int cw = min(P.tw, I.w - V.x0) * es, yb = min(I.h, V.y0 + P.th);
        const int vpr = I.aligned ? cw / 16 : 0;
        for (int y = V.y0 + warp; y < yb; y += kWarps) {
            char *g = reinterpret_cast<char *>(I.img) + size_t(y) * I.pitch + V.x0 * es;
            const uint8_t *d = tile + (y - V.y0 + HR) * L.row_bytes + kPadCols * es;
            for (int v = lane; v < vpr; v += 32)
                *reinterpret_cast<uint4 *>(g + 16 * v) = *reinterpret_cast<const uint4 *>(d + 16 * v);
            for (int x = 16 * vpr + lane; x < cw; x += 32) g[x] = char(d[x]);
        }
    }
}

const void *mosaic_kernel(int es)
{
    return es == 2 ? reinterpret_cast<const void *>(k_mosaic<2>) : reinterpret_cast<const void *>(k_mosaic<1>);
}

}  // namespace

bool mosaic_shape(const JobSpec *jobs, int n, MosaicShape *out)
{
    const bool any16 = jobs[0].dtype == THIN_U16;
    for (int k = 1; k < n; ++k)
        if ((jobs[k].dtype == THIN_U16) != any16) return false;
    int dev = 0, sms = 0, optin = 0, per_sm = 0, reserved = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    return mosaic_search(jobs, n, any16, sms, std::min(optin, per_sm / 2 - reserved) - 256, out);
}

int mosaic_prepare(const JobSpec *jobs, int n, const MosaicShape &shape, const thin_options &opt, cudaStream_t stream,
                   bool async_alloc, MosaicPrepared *M)
{
    *M = MosaicPrepared();
    M->n = n;
    M->async_alloc = async_alloc;
    M->es = elem_size(jobs[0].dtype);
    for (int k = 1; k < n; ++k)
        if (elem_size(jobs[k].dtype) != M->es) return THIN_ERR_ARG;  // one element size per launch
    const bool any16 = M->es == 2;
    if (!mosaic_shape_fits(M->es, shape)) return THIN_ERR_ARG;
    const int tw = shape.tw, th = shape.th, H = shape.halo;
    const TileLayout L = tile_layout(tw, th, halo_rows(H), any16);
    std::vector<MosImage> imgs(n);
    if (n > kMosaicMax) return THIN_ERR_ARG;
    size_t off = 0;
    const size_t o_st = off;
    off = align_up(off + sizeof(MosStat) * n, 256);
    const size_t o_err = off;
    off = align_up(off + sizeof(int), 256);
    const size_t o_count = off;
    off = align_up(off + sizeof(unsigned) * kCountSlots * size_t(n), 256);
    const size_t o_flag = off;
    int tiles = 0;
    for (int k = 0; k < n; ++k) {
        MosImage &I = imgs[k];
        const JobSpec &J = jobs[k];
        std::memset(&I, 0, sizeof I);
        I.img = reinterpret_cast<unsigned long long>(J.img);
        I.pitch = J.pitch;
        I.w = J.w;
        I.h = J.h;
        I.adj = J.adj;
        I.lam = J.lam;
        I.tiles_x = (J.w + tw - 1) / tw;
        I.tiles_y = (J.h + th - 1) / th;
        I.tile_base = tiles;
        I.cells_x = I.tiles_x * tw / 8;
        I.aligned = I.img % 16 == 0 && J.pitch % 16 == 0;
        I.rim_pitch = size_t(I.tiles_x) * tw * elem_size(J.dtype);
        tiles += I.tiles_x * I.tiles_y;
    }
    off = align_up(off + sizeof(unsigned) * tiles, 256);
    M->live_bytes = off;
    std::vector<size_t> o_rim(2 * n), o_bits(2 * n);
    for (int k = 0; k < n; ++k)
        for (int q = 0; q < 2; ++q) {
            o_rim[2 * k + q] = off;
            off = align_up(off + imgs[k].rim_pitch * size_t(imgs[k].tiles_y) * th, 256);
            o_bits[2 * k + q] = off;
            off = align_up(off + size_t(imgs[k].cells_x) * (size_t(imgs[k].tiles_y) * th / 2), 256);
        }
    const void *kernel = mosaic_kernel(M->es);
    cudaError_t e = allow_max_dynamic_smem(kernel);
    int dev = 0, sms = 0, per_sm = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, L.bytes);
    if (e != cudaSuccess) return cuda_status(e);
    if (tiles > per_sm * sms) return THIN_ERR_ARG;  // the blocks wait for one another: all must be resident
    e = async_alloc ? scratch_alloc(reinterpret_cast<void **>(&M->base), off, stream)
                    : cudaMalloc(reinterpret_cast<void **>(&M->base), off);
    if (e != cudaSuccess) {
        cudaGetLastError();
        M->base = nullptr;
        return THIN_ERR_OOM;
    }
    for (int k = 0; k < n; ++k)
        for (int q = 0; q < 2; ++q) {
            imgs[k].rim[q] = reinterpret_cast<unsigned long long>(M->base + o_rim[2 * k + q]);
            imgs[k].bits[q] = reinterpret_cast<unsigned long long>(M->base + o_bits[2 * k + q]);
        }
    M->live = M->base;
    M->o_st = o_st;
    M->o_err = o_err;
    M->grid = tiles;
    M->smem = L.bytes;
    M->halo = H;
    M->args.resize(sizeof(MosArgs));
    MosArgs &P = *reinterpret_cast<MosArgs *>(M->args.data());
    std::memset(&P, 0, sizeof P);
    std::copy(imgs.begin(), imgs.end(), P.imgs);
    P.st = reinterpret_cast<MosStat *>(M->base + o_st);
    P.error = reinterpret_cast<unsigned *>(M->base + o_err);
    P.count = reinterpret_cast<unsigned *>(M->base + o_count);
    P.flag = reinterpret_cast<unsigned *>(M->base + o_flag);
    P.n = n;
    P.tw = tw;
    P.th = th;
    P.halo = H;
    P.hr = halo_rows(H);
    P.rule = test_mode(opt);
    P.start_phase = opt.start_phase;
    P.max_phases = opt.max_phases;
    P.timeout_ns = 2000000000ull;
    if (const char *t = std::getenv("THIN_TIMEOUT_NS")) P.timeout_ns = std::strtoull(t, nullptr, 10);
    P.tl = L;
    return THIN_OK;
}

cudaError_t mosaic_enqueue(const MosaicPrepared &M, cudaStream_t stream)
{
    const cudaError_t e = cudaMemsetAsync(M.live, 0, M.live_bytes, stream);
    if (e != cudaSuccess) return e;
    void *args[] = {const_cast<char *>(M.args.data())};
    return cudaLaunchCooperativeKernel(mosaic_kernel(M.es), dim3(M.grid), dim3(kThreads), args, M.smem, stream);
}

int mosaic_collect(const MosaicPrepared &M, const thin_options &opt, cudaStream_t stream, thin_stats *out)
{
    // (the stats and the error word lie side by side)
    std::vector<char> live(M.o_err - M.o_st + sizeof(int));
    cudaError_t e = cudaMemcpyAsync(live.data(), M.base + M.o_st, live.size(), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return cuda_status(e);
    int error;
    std::memcpy(&error, live.data() + (M.o_err - M.o_st), sizeof error);
    int rc = THIN_OK;
    for (int k = 0; k < M.n; ++k) {
        MosStat S;
        std::memcpy(&S, live.data() + sizeof(MosStat) * k, sizeof S);
        thin_stats &o = out[k];
        std::memset(&o, 0, sizeof o);
        long long phases = S.stop ? (long long)S.stop * M.halo : opt.max_phases;
        if (opt.max_phases >= 0) phases = std::min<long long>(phases, opt.max_phases);
        if (phases < 0) phases = 0;  // (a run that ended with an error)
        const long long last = (long long)S.last - 1;
        o.converged = S.stop != 0 && !error && (opt.max_phases < 0 || quiet_at_cap(opt, last));
        if (S.stop && !error && !o.converged) phases = opt.max_phases;  // (the phases after the stop change nothing)
        o.status = error ? error : (o.converged ? THIN_OK : THIN_ERR_NOT_CONVERGED);
        o.phases = phases;
        o.lowered = (int64_t)S.lowered;
        o.last_change_phase = last;
        o.end_phase = opt.start_phase + phases;
        o.steps = (phases + M.halo - 1) / M.halo;
        o.tested = (int64_t)S.tested;
        if (o.status != THIN_OK && rc == THIN_OK) rc = o.status;
    }
    return rc;
}

void mosaic_release(MosaicPrepared &M, cudaStream_t stream)
{
    if (M.base) {
        if (M.async_alloc) cudaFreeAsync(M.base, stream);
        else cudaFree(M.base);
    }
    M.base = nullptr;
}

}  // namespace thin
