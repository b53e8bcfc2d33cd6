// thin_tiled.cu -- the tiled lambda-thinning engine.
//
// One persistent cooperative launch runs the whole subfield schedule for any
// number of images.  The schedule advances in steps of H phases (temporal
// blocking).  In a step every active tile of every image is visited by one
// block: TMA 2-D tile loads stage the tile with a halo in shared memory, the
// block advances H consecutive phases there (the exact region shrinks by one
// pixel ring per phase) and stores the interior to the other buffer of a
// ping-pong pair.  A grid barrier separates steps.
//
// Which points a phase tests.  As in the resident engine (thin_block.cuh): per
// parity a dirty bit per 4-point group, set by the moves of its neighbours that
// can change its test, consumed by its phase.  Between visits the bits of an
// image lie in global memory, a byte per cell with a bit per parity, in a
// ping-pong pair of their own: a visit reads the bits of its tile and halo from
// one buffer and writes those of its tile to the other.  A tile that no step
// visits keeps, in the buffer it was last read from, bits that its last visit
// consumed: they add tests of points that cannot move and change nothing.  The halo is
// one pixel wider than the step has phases, so that in the last phase too the
// points just outside the tile are exact: every mark a neighbour's move makes
// inside the tile is made by the tile's own visit, and no visit writes another
// tile's bits.
//
// Which tiles a step visits.  A tile that changed at all, which keeps both
// ping-pong buffers equal on every skipped tile; a tile with a dirty bit; and
// its neighbours as far as a move of such a bit's group can come in H phases (a
// move spreads one pixel a phase).  The first step visits every tile, with every
// bit set.  When a step visits no tile the image is at its fixed point and both
// buffers hold it.
//
// What bounds it: issue, as in the resident engine (8192^2 u16 at lambda = 0 is
// read and written once in each of 9 steps: 2.4 GB, 0.4 of 4.8 ms).  Tiles were
// 64 x 32 pixels, one to a warp, with change stamps that re-tested every group
// of the nine cells around a changed one: a ring of 8 around such a tile is a
// third more points, and the stamps' scan took 300 instructions a phase.
// 8192^2 u16 went from 7.1 to 4.8 ms at lambda = 0 and from 22.5 to 13.9 ms at
// lambda = 30; 1024 uneven u8 images from 277 to 239 ms; 48 served requests of
// every size from 91 to 46 ms.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "thin_block.cuh"
#include "thin_common.cuh"
#include "thin_internal.h"
#include "thin_simd.cuh"
#include "thin_tile.cuh"

namespace thin {

namespace {

struct ImgDesc {
    CUtensorMap map[2];          // TMA descriptors of buffer 0 and buffer 1
    unsigned long long buf[2];   // device pointers of the ping-pong pair
    unsigned long long pitch;    // row pitch of both buffers, bytes
    unsigned long long user;     // caller's image
    unsigned long long user_pitch;
    unsigned long long cells[2]; // dirty bits of the ping-pong pair: a byte per cell, bit p for parity p
    int w, h, dtype;
    unsigned lam;
    int tiles_x, tiles_y, tile_base, copy_in;
    int cells_x, cells_y, adj, pad1;
};

struct ImgStat {
    unsigned long long lowered;
    unsigned long long tiles_visited;
    unsigned long long tested;  // point tests on tile interiors
    long long last_change;  // global phase index, -1 if none
    int last_step;          // last step that visited a tile of this image
    int last_listed;        // last step for which a tile of this image was listed
};

struct Ctl {
    unsigned bar_count;
    unsigned bar_gen;
    int error;
    int steps;
    unsigned list_count[3];
    unsigned next_item[3];  // per step (mod 3): items claimed beyond the first one of every block
};

struct EngineArgs {
    const ImgDesc *imgs;
    ImgStat *st;
    int *listed;       // per tile: last step index it was appended for
    unsigned *lists;   // 3 lists of total_tiles entries each
    Ctl *ctl;
    int n_imgs;
    int total_tiles;
    int tw, th, halo, hr, rule;  // halo: phases per step; hr: halo rows staged above and below (even, more than halo)
    long long start_phase;
    long long max_phases;
    unsigned long long timeout_ns;
    TileLayout tl;
    int debug;         // 1: block 0 never arrives at the first barrier (timeout test)
};

__device__ const DecisionTable d_decisions = kDecisionTable;

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for phase `parity` of an mbarrier; false after timeout_ns.
__device__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned long long timeout_ns)
{
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = gtimer();
    for (;;) {
        if (mbar_try(bar, parity)) return true;
        if (gtimer() - t0 > timeout_ns) return false;
    }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(dst),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// Grid barrier with a time limit.  Returns false if the wait ran out or an
// error was posted; then ctl->error is set.
__device__ bool grid_barrier(Ctl *ctl, unsigned nblocks, unsigned long long timeout_ns, bool skip_arrive,
                             int *s_flag)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned *gen = &ctl->bar_gen;
        volatile int *err = &ctl->error;
        const unsigned g = *gen;
        int ok = 1;
        __threadfence();
        asm volatile("fence.proxy.async.global;" ::: "memory");
        bool last = false;
        if (!skip_arrive) last = atomicAdd(&ctl->bar_count, 1u) == nblocks - 1;
        if (last) {
            atomicExch(&ctl->bar_count, 0u);
            __threadfence();
            atomicAdd(&ctl->bar_gen, 1u);
        } else {
            const unsigned long long t0 = gtimer();
            while (*gen == g) {
                if (*err) {
                    ok = 0;
                    break;
                }
                if (gtimer() - t0 > timeout_ns) {
                    atomicCAS(&ctl->error, 0, THIN_ERR_TIMEOUT);
                    ok = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
        asm volatile("fence.proxy.async.global;" ::: "memory");
        if (*err) ok = 0;
        *s_flag = ok;
    }
    __syncthreads();
    return *s_flag != 0;
}

__device__ __forceinline__ int find_image(const ImgDesc *imgs, int n, int gt)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (imgs[mid].tile_base <= gt)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Stores the tile (clipped to the image) to `dst`, a row of which is 16-byte aligned.
template <int THREADS>
__device__ __forceinline__ void tile_store(const uint8_t *tile, int row_bytes, int es, const Visit &V, char *dst, size_t pitch)
{
    const int cw = min(V.tw, V.w - V.x0) * es, ch = min(V.th, V.h - V.y0);
    const int vpr = (cw + 15) / 16;
    const uint32_t M = div_magic(vpr);
    char *base = dst + size_t(V.y0) * pitch + size_t(V.x0) * es;
    const uint8_t *src = tile + V.hr * row_bytes + kPadCols * es;
    for (int v = threadIdx.x; v < ch * vpr; v += THREADS) {
        const int row = div_small(v, vpr, M), col = (v - row * vpr) * 16;
        char *d = base + size_t(row) * pitch + col;
        const uint8_t *s = src + row * row_bytes + col;
        if (col + 16 <= cw) *reinterpret_cast<uint4 *>(d) = *reinterpret_cast<const uint4 *>(s);
        else
            for (int b = 0; col + b < cw; ++b) d[b] = char(s[b]);
    }
}

__device__ __forceinline__ void decode(const EngineArgs &P, bool full, const unsigned *L, unsigned i, int &img,
                                       int &tx, int &ty)
{
    const int gt = full ? int(i) : int(__ldcg(L + i));  // written by other blocks: bypass L1
    img = find_image(P.imgs, P.n_imgs, gt);
    const ImgDesc &D = P.imgs[img];
    const int local = gt - D.tile_base;
    ty = local / D.tiles_x;
    tx = local - ty * D.tiles_x;
}

template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 2 * kWarps / WARPS) k_engine(EngineArgs P)
{
    constexpr int THREADS = 32 * WARPS;
    extern __shared__ __align__(128) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    __shared__ int s_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const TileLayout L = P.tl;
    uint8_t *tile = smem + kOffTile;
    TileCtrl *ctrl = reinterpret_cast<TileCtrl *>(smem + kOffCtrl);
    uint32_t *dirty = reinterpret_cast<uint32_t *>(smem + L.dirty_off);
    const uint32_t bar = smem_u32(smem + kOffBar);
    const int words = L.rows / 2;

    load_decisions(smem, d_decisions);
    if (tid == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    uint32_t parity = 0;
    long long g0 = P.start_phase;
    const int H = P.halo, HR = P.hr;
    for (int s = 0;; ++s) {
        const long long done = g0 - P.start_phase;
        const int Hs = (P.max_phases >= 0 && P.max_phases - done < H) ? int(P.max_phases - done) : H;
        const bool full = s == 0;
        const unsigned count = full ? unsigned(P.total_tiles)
                                    : *reinterpret_cast<volatile unsigned *>(&P.ctl->list_count[s % 3]);
        const unsigned *Lcur = P.lists + size_t(s % 3) * P.total_tiles;
        unsigned *Lnext = P.lists + size_t((s + 1) % 3) * P.total_tiles;
        if (blockIdx.x == 0 && tid == 0) {  // counters of step s + 2, last used in step s - 1
            P.ctl->list_count[(s + 2) % 3] = 0;
            P.ctl->next_item[(s + 2) % 3] = 0;
        }
        const int src = s & 1;
        bool failed = false;
        // A block takes item blockIdx.x first, then claims further items one at a time from the step's
        // counter, so that blocks that drew light tiles take more of them.
        for (unsigned i = blockIdx.x; i < count;) {
            int img, tx, ty;
            decode(P, full, Lcur, i, img, tx, ty);
            const ImgDesc &D = P.imgs[img];
            Visit V;
            V.w = D.w;
            V.h = D.h;
            V.tw = P.tw;
            V.th = P.th;
            V.Hs = Hs;
            V.hr = HR;
            V.g0 = g0;
            V.x0 = tx * P.tw;
            V.y0 = ty * P.th;
            const int u16 = D.dtype == THIN_U16;
            const int es = u16 ? 2 : 1;
            if (tid == 0) {
                const int boxes = L.rows / L.box_rows;
                const uint32_t box_bytes = uint32_t(L.box_rows) * uint32_t((P.tw + 2 * kPadCols) * es);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(box_bytes * boxes)
                             : "memory");
                for (int b = 0; b < boxes; ++b)
                    tma_load_2d(smem_u32(tile) + b * box_bytes, &D.map[src], V.x0 - kPadCols, V.y0 - HR + b * L.box_rows, bar);
                ctrl->qn[0] = 0u;
                ctrl->qn[1] = 0u;
                ctrl->near = 0u;
                ctrl->last = -1;
                ctrl->next = gridDim.x + atomicAdd(&P.ctl->next_item[s % 3], 1u);
            }
            // dirty bits of the tile and its halo (overlaps the load): a warp to a cell row, a lane to a cell
            {
                const unsigned char *bits = reinterpret_cast<const unsigned char *>(D.cells[src]);
                const int gx = (V.x0 - kPadCols) / 8 + lane, gy0 = (V.y0 - HR) / 2;  // (both exact: multiples of 8 and 2)
                const bool col = lane < (P.tw + 2 * kPadCols) / 8 && gx >= 0 && gx < D.cells_x;
#pragma unroll 4
                for (int cr = warp; cr < words; cr += WARPS) {
                    const int gy = gy0 + cr;
                    unsigned v = 0;
                    if (col && gy >= 0 && gy < D.cells_y) v = __ldcg(bits + size_t(gy) * D.cells_x + gx);
                    const unsigned b0 = __ballot_sync(0xffffffffu, v & 1u), b1 = __ballot_sync(0xffffffffu, v & 2u);
                    const unsigned b2 = __ballot_sync(0xffffffffu, v & 4u), b3 = __ballot_sync(0xffffffffu, v & 8u);
                    if (lane < 4) dirty[lane * words + cr] = lane == 0 ? b0 : lane == 1 ? b1 : lane == 2 ? b2 : b3;
                }
            }
            const bool ok = mbar_wait(bar, parity, P.timeout_ns);
            if (!__syncthreads_and(ok)) {
                mbar_wait(bar, parity, P.timeout_ns);  // let copies in flight land (bounded)
                failed = true;
                break;
            }
            parity ^= 1u;
            int nlow = 0, chg_j = -1, ntest = 0;
            const PointRule rule = point_rule(smem, P.rule | (D.adj << 2), D.lam, es, true);  // F^- reading, operator, pair
            TileLayout Li = L;
            Li.row_bytes = (P.tw + 2 * kPadCols) * es;
            if (u16) visit_phases<uint16_t, THREADS>(Li, smem, V, rule, nlow, ntest, chg_j);
            else visit_phases<uint8_t, THREADS>(Li, smem, V, rule, nlow, ntest, chg_j);
            tile_store<THREADS>(tile, Li.row_bytes, es, V, reinterpret_cast<char *>(D.buf[src ^ 1]), D.pitch);
            // the tile's dirty bits, and which neighbours they can reach in the next step
            {
                unsigned char *bits = reinterpret_cast<unsigned char *>(D.cells[src ^ 1]);
                const int gx = V.x0 / 8 + lane, gy0 = V.y0 / 2;
                const int cols = P.tw / 8, rows = P.th / 2;
                const int zx = (H + 2 + 7) / 8, zy = (H + 2 + 1) / 2;  // cells within reach of an edge
                const unsigned left = 0xffffffffu >> (32 - min(zx, 32)), right = left << max(cols - zx, 0);
                unsigned near = 0;
                for (int cr = warp; cr < rows; cr += WARPS) {
                    const int gy = gy0 + cr;
                    const uint32_t *w = dirty + HR / 2 + cr;
                    const int b = lane + kPadCols / 8;
                    unsigned v = 0;
                    if (lane < cols && gx < D.cells_x && gy < D.cells_y) {
                        v = ((w[0] >> b) & 1u) | (((w[words] >> b) & 1u) << 1) | (((w[2 * words] >> b) & 1u) << 2) |
                            (((w[3 * words] >> b) & 1u) << 3);
                        __stcg(bits + size_t(gy) * D.cells_x + gx, static_cast<unsigned char>(v));
                    }
                    const unsigned any = __ballot_sync(0xffffffffu, v != 0);
                    const unsigned xs = (any & left ? 1u : 0u) | (any ? 2u : 0u) | (any & right ? 4u : 0u);
                    near |= (xs << 3) | (cr < zy ? xs : 0u) | (cr >= rows - zy ? xs << 6 : 0u);
                }
                if (lane == 0 && near) atomicOr(&ctrl->near, near);
            }
            nlow = __reduce_add_sync(0xffffffffu, nlow);
            ntest = __reduce_add_sync(0xffffffffu, ntest);
            const int maxj = __reduce_max_sync(0xffffffffu, chg_j);
            if (lane == 0) {
                if (maxj >= 0) atomicMax(&ctrl->last, maxj);
                if (nlow) atomicAdd(&P.st[img].lowered, (unsigned long long)nlow);
                if (ntest) atomicAdd(&P.st[img].tested, (unsigned long long)ntest);
            }
            // order this block's generic shared and global writes before later TMA traffic
            asm volatile("fence.proxy.async;" ::: "memory");
            __syncthreads();
            i = ctrl->next;
            if (tid < 9) {
                const int dx = tid % 3 - 1, dy = tid / 3 - 1;
                const int ntx = tx + dx, nty = ty + dy, last = ctrl->last;
                const bool list = ((ctrl->near >> tid) & 1u) || (tid == 4 && last >= 0);
                if (list && ntx >= 0 && ntx < D.tiles_x && nty >= 0 && nty < D.tiles_y) {
                    const int gt = D.tile_base + nty * D.tiles_x + ntx;
                    if (atomicMax(&P.listed[gt], s + 1) < s + 1) {
                        const unsigned pos = atomicAdd(&P.ctl->list_count[(s + 1) % 3], 1u);
                        Lnext[pos] = unsigned(gt);
                        atomicMax(&P.st[img].last_listed, s + 1);
                    }
                }
                if (tid == 4) {
                    if (last >= 0) atomicMax(&P.st[img].last_change, g0 + last);
                    atomicAdd(&P.st[img].tiles_visited, 1ull);
                    atomicMax(&P.st[img].last_step, s);
                }
            }
            __syncthreads();  // the control words are read before the next visit sets them
        }
        if (__syncthreads_or(failed)) {
            if (tid == 0) atomicCAS(&P.ctl->error, 0, THIN_ERR_TIMEOUT);
            return;
        }
        const bool skip = P.debug == 1 && blockIdx.x == 0 && s == 0;
        if (!grid_barrier(P.ctl, gridDim.x, P.timeout_ns, skip, &s_flag)) return;
        g0 += Hs;
        const long long ran = g0 - P.start_phase;
        const unsigned next = *reinterpret_cast<volatile unsigned *>(&P.ctl->list_count[(s + 1) % 3]);
        const bool stop = (P.max_phases >= 0 && ran >= P.max_phases) || next == 0;
        if (stop) {
            if (blockIdx.x == 0 && tid == 0) P.ctl->steps = s + 1;
            return;
        }
    }
}

// Copies each image's final buffer to the caller's image where they differ.
__global__ void k_copy_out(const ImgDesc *imgs, const ImgStat *st, int n)
{
    const int k = blockIdx.y;
    if (k >= n) return;
    const ImgDesc &D = imgs[k];
    const ImgStat &S = st[k];
    const bool converged = S.last_listed <= S.last_step;
    const int fin = converged ? 0 : ((S.last_step + 1) & 1);
    const char *src = reinterpret_cast<const char *>(D.buf[fin]);
    char *dst = reinterpret_cast<char *>(D.user);
    if (src == dst) return;
    const size_t rowb = size_t(D.w) * (D.dtype == THIN_U16 ? 2 : 1);
    const size_t total = rowb * size_t(D.h);
    for (size_t e = size_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += size_t(gridDim.x) * blockDim.x) {
        const size_t r = e / rowb, c = e - r * rowb;
        dst[r * D.user_pitch + c] = src[r * D.pitch + c];
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// The kernel's builds.  Blocks of fewer warps leave room for more of them on an
// SM (16 warps in all): small tiles, which only a caller or the autotuner sets,
// give a phase too few groups for 8 warps.
struct EngineBuild {
    const void *kernel;
    int warps;
};
const EngineBuild kBuilds[3] = {{reinterpret_cast<const void *>(k_engine<8>), 8},
                                {reinterpret_cast<const void *>(k_engine<4>), 4},
                                {reinterpret_cast<const void *>(k_engine<2>), 2}};

// The build for a launch: with n warps a block where 16 / n blocks fit an SM's
// shared memory and there are tiles enough, one for each of those blocks (4
// warps) or four (2 warps).  4096^2 u8 at lambda = 10 with 8 / 4 / 2 warps: tiles
// of 32 x 32 and 8 phases 165 / 110 / 94 ms, 64 x 32 110 / 79 / 74, 64 x 64 83 /
// 68 / 73, 128 x 64 64 / 57 / 74 (with a warp to a tile of 64 x 32, all points
// tested, 97).  1000^2, 64 x 32 (512 tiles): 9.5 / 9.4 / 11.8 ms, 32 x 32 (1024)
// 11.1 / 10.5 / 12.4.
const EngineBuild &engine_build(int tiles, const TileLayout &L, int smem, int sms)
{
    int dev = 0, per_sm = 0, reserved = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    const auto fits = [&](int warps) {
        return L.rows / 2 <= 32 * warps && smem + 256 + reserved <= per_sm * warps / (2 * kWarps);
    };
    if (tiles >= 32 * sms && fits(2)) return kBuilds[2];
    if (tiles >= 4 * sms && fits(4)) return kBuilds[1];
    return kBuilds[0];
}

// Tile shape and phases per step.  What the caller set is taken as it is (and
// checked); with nothing set the largest of these shapes that still gives every
// SM two tiles: a large tile has less halo (224 x 152 with rings of 1 to 15:
// 17 % more points; 64 x 32 with 1 to 8: 46 %), and two blocks of 113 KB share an
// SM.  Steps of 6 / 8 / 12 / 15 phases: 8192^2 u16 at lambda = 0 4.83 / 4.65 /
// 4.77 / 4.75 ms, at lambda = 30 15.1 / 14.3 / 14.0 / 13.9 ms, the served
// requests 72.7 / 70.5 / 60.8 / 59.3 ms; one block of 16 warps an SM, with
// tiles twice as high: 4.68, 13.9 and 55 ms against 58.9; three of 5 warps:
// 5.6, 15.8 and 73 ms.
int tiled_shape(const JobSpec *jobs, int n, bool any16, const thin_options &opt, int *tw, int *th, int *H)
{
    if (opt.tile_w || opt.tile_h || opt.halo) {
        tiled_defaults(tw, th, H);
        if (opt.tile_w) *tw = opt.tile_w;
        if (opt.tile_h) *th = opt.tile_h;
        if (opt.halo) *H = opt.halo;
        const int max_halo = any16 ? 8 : 16;
        if (*H < kMinHalo || *H > max_halo || *tw < 16 || *tw > 224 || *tw % 16 || *th < 8 || *th % 2 ||
            std::min(*tw, *th) < *H + 1 || *th + 2 * (*H + (*H & 1)) > 256)
            return THIN_ERR_ARG;
        *H = std::min(*H, kMaxStep);
        return THIN_OK;
    }
    static const int shapes[2][5][3] = {{{224, 304, 15}, {224, 160, 15}, {224, 80, 8}, {128, 64, 8}, {64, 32, 8}},
                                        {{224, 152, 15}, {224, 96, 15}, {128, 96, 8}, {96, 48, 8}, {64, 32, 8}}};
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    for (const auto &s : shapes[any16 ? 1 : 0]) {
        *tw = s[0];
        *th = s[1];
        *H = s[2];
        size_t tiles = 0;
        for (int k = 0; k < n; ++k)
            tiles += size_t((jobs[k].w + *tw - 1) / *tw) * size_t((jobs[k].h + *th - 1) / *th);
        if (tiles >= size_t(2 * sms)) break;
    }
    return THIN_OK;
}

}  // namespace

bool tiled_fills(const JobSpec *jobs, int n, int *tw, int *th, int *H)
{
    bool any16 = false;
    for (int k = 0; k < n; ++k) any16 |= jobs[k].dtype == THIN_U16;
    thin_options o;
    std::memset(&o, 0, sizeof o);
    tiled_shape(jobs, n, any16, o, tw, th, H);
    return *H == kMaxStep;  // (the large shapes)
}

void tiled_defaults(int *tw, int *th, int *halo)
{
    *tw = 64;
    *th = 32;
    *halo = 8;
}

// A tiled launch prepared on the host: layout, tensor maps and pristine
// stats/control words uploaded into one device allocation.
struct TiledPrepared {
    int n = 0, H = 0, grid = 0, smem = 0;
    EngineBuild build = {nullptr, 0};
    bool async_alloc = true;
    char *base = nullptr;
    size_t o_stat = 0, o_ctl = 0, o_stat0 = 0, o_ctl0 = 0, o_listed = 0, o_cells = 0, cells_bytes = 0;
    int total_tiles = 0;
    std::vector<JobSpec> jobs;
    std::vector<ImgDesc> descs;
    EngineArgs P;
};

int tiled_prepare(const JobSpec *jobs, int n, const thin_options &opt, cudaStream_t stream, bool async_alloc,
                  TiledPrepared **out, int max_grid)
{
    *out = nullptr;
    bool any16 = false;
    for (int k = 0; k < n; ++k) any16 |= jobs[k].dtype == THIN_U16;
    int tw, th, H;
    const int shape_rc = tiled_shape(jobs, n, any16, opt, &tw, &th, &H);
    if (shape_rc != THIN_OK) return shape_rc;
    const int HR = halo_rows(H);
    const TileLayout TL = tile_layout(tw, th, HR, any16);
    EncodeTiledFn enc = encode_fn();
    if (!enc) return THIN_ERR_CUDA;

    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);

    TiledPrepared *T = new TiledPrepared;
    T->n = n;
    T->H = H;
    T->async_alloc = async_alloc;
    T->jobs.assign(jobs, jobs + n);
    // ---- layout of one scratch allocation
    std::vector<ImgDesc> &descs = T->descs;
    descs.resize(n);
    std::vector<size_t> buf_off(n), cpy_off(n), cell_off(n), cell1_off(n);
    size_t off = 0;
    const size_t o_desc = off;
    off = align_up(off + sizeof(ImgDesc) * n, 256);
    T->o_stat = off;
    off = align_up(off + sizeof(ImgStat) * n, 256);
    T->o_stat0 = off;
    off = align_up(off + sizeof(ImgStat) * n, 256);
    T->o_ctl = off;
    off = align_up(off + sizeof(Ctl), 256);
    T->o_ctl0 = off;
    off = align_up(off + sizeof(Ctl), 256);
    int total_tiles = 0;
    for (int k = 0; k < n; ++k) {
        const JobSpec &J = jobs[k];
        ImgDesc &D = descs[k];
        std::memset(&D, 0, sizeof D);
        D.w = J.w;
        D.h = J.h;
        D.dtype = J.dtype;
        D.lam = J.lam;
        D.adj = J.adj;
        D.tiles_x = (J.w + tw - 1) / tw;
        D.tiles_y = (J.h + th - 1) / th;
        D.tile_base = total_tiles;
        D.cells_x = (J.w + 7) / 8;
        D.cells_y = (J.h + 1) / 2;
        total_tiles += D.tiles_x * D.tiles_y;
        const size_t es = elem_size(J.dtype);
        const bool aligned = (reinterpret_cast<uintptr_t>(J.img) % 16 == 0) && (J.pitch % 16 == 0);
        D.copy_in = aligned ? 0 : 1;
        D.pitch = aligned ? J.pitch : align_up(size_t(J.w) * es, 128);
        D.user = reinterpret_cast<unsigned long long>(J.img);
        D.user_pitch = J.pitch;
        buf_off[k] = off;
        off = align_up(off + D.pitch * J.h, 256);
        cpy_off[k] = 0;
        if (D.copy_in) {
            cpy_off[k] = off;
            off = align_up(off + D.pitch * J.h, 256);
        }
    }
    T->o_cells = off;
    for (int k = 0; k < n; ++k) {
        cell_off[k] = off;
        off = align_up(off + size_t(descs[k].cells_x) * descs[k].cells_y, 256);
    }
    T->cells_bytes = off - T->o_cells;
    for (int k = 0; k < n; ++k) {  // (written by the first step, which visits every tile)
        cell1_off[k] = off;
        off = align_up(off + size_t(descs[k].cells_x) * descs[k].cells_y, 256);
    }
    T->o_listed = off;
    off = align_up(off + sizeof(int) * total_tiles, 256);
    const size_t o_lists = off;
    off = align_up(off + sizeof(unsigned) * 3 * size_t(total_tiles), 256);
    const size_t total_bytes = off;
    T->total_tiles = total_tiles;

    cudaError_t e = async_alloc ? scratch_alloc(reinterpret_cast<void **>(&T->base), total_bytes, stream)
                                : cudaMalloc(reinterpret_cast<void **>(&T->base), total_bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        T->base = nullptr;
        delete T;
        return THIN_ERR_OOM;
    }
    char *base = T->base;
    for (int k = 0; k < n; ++k) {
        ImgDesc &D = descs[k];
        const JobSpec &J = jobs[k];
        void *b0 = D.copy_in ? static_cast<void *>(base + cpy_off[k]) : J.img;
        void *b1 = base + buf_off[k];
        D.buf[0] = reinterpret_cast<unsigned long long>(b0);
        D.buf[1] = reinterpret_cast<unsigned long long>(b1);
        D.cells[0] = reinterpret_cast<unsigned long long>(base + cell_off[k]);
        D.cells[1] = reinterpret_cast<unsigned long long>(base + cell1_off[k]);
        const cuuint64_t gdim[2] = {cuuint64_t(J.w), cuuint64_t(J.h)};
        const cuuint64_t gstr[1] = {cuuint64_t(D.pitch)};
        const cuuint32_t box[2] = {cuuint32_t(tw + 2 * kPadCols), cuuint32_t(TL.box_rows)};
        const cuuint32_t est[2] = {1, 1};
        for (int q = 0; q < 2; ++q) {
            void *bp = q ? b1 : b0;
            CUresult r = enc(&D.map[q], J.dtype == THIN_U16 ? CU_TENSOR_MAP_DATA_TYPE_UINT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8,
                             2, bp, gdim, gstr, box, est, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) {
                tiled_release(T, stream);
                return THIN_ERR_ARG;
            }
        }
    }
    std::vector<ImgStat> st0(n);
    for (auto &x : st0) {
        x.lowered = 0;
        x.tiles_visited = 0;
        x.tested = 0;
        x.last_change = -1;
        x.last_step = -1;
        x.last_listed = 0;
    }
    Ctl ctl0;
    std::memset(&ctl0, 0, sizeof ctl0);
    e = cudaMemcpyAsync(base + o_desc, descs.data(), sizeof(ImgDesc) * n, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(base + T->o_stat0, st0.data(), sizeof(ImgStat) * n, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(base + T->o_ctl0, &ctl0, sizeof ctl0, cudaMemcpyHostToDevice, stream);

    EngineArgs &P = T->P;
    std::memset(&P, 0, sizeof P);
    P.imgs = reinterpret_cast<const ImgDesc *>(base + o_desc);
    P.st = reinterpret_cast<ImgStat *>(base + T->o_stat);
    P.listed = reinterpret_cast<int *>(base + T->o_listed);
    P.lists = reinterpret_cast<unsigned *>(base + o_lists);
    P.ctl = reinterpret_cast<Ctl *>(base + T->o_ctl);
    P.n_imgs = n;
    P.total_tiles = total_tiles;
    P.tw = tw;
    P.th = th;
    P.halo = H;
    P.hr = HR;
    P.rule = test_mode(opt);  // F^- reading and operator
    P.start_phase = opt.start_phase;
    P.max_phases = opt.max_phases;
    P.timeout_ns = 2000000000ull;
    if (const char *t = std::getenv("THIN_TIMEOUT_NS")) P.timeout_ns = std::strtoull(t, nullptr, 10);
    P.debug = opt.reserved;
    P.tl = TL;
    T->smem = 128 + TL.bytes;
    T->build = engine_build(total_tiles, TL, T->smem, sms);
    {
        int optin = 0;
        cudaFuncAttributes fa;
        if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
            cudaFuncGetAttributes(&fa, T->build.kernel) == cudaSuccess &&
            size_t(T->smem) + fa.sharedSizeBytes > size_t(optin)) {
            tiled_release(T, stream);
            return THIN_ERR_ARG;  // this tile shape and halo do not fit one block's shared memory
        }
    }

    if (e == cudaSuccess) e = allow_max_dynamic_smem(T->build.kernel);
    int per_sm = 0;
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, T->build.kernel, 32 * T->build.warps, T->smem);
    if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
    T->grid = std::max(1, std::min(sms * per_sm, total_tiles));
    if (max_grid > 0) T->grid = std::min(T->grid, max_grid * kWarps / T->build.warps);
    if (opt.reserved == 1) T->grid = std::max(T->grid, std::min(2, sms * per_sm));
    if (e != cudaSuccess) {
        tiled_release(T, stream);
        return cuda_status(e);
    }
    *out = T;
    return THIN_OK;
}

// Copies unaligned images in, resets the per-run state, launches the engine
// and the copy-out: device work only, so it can be captured in a CUDA graph.
cudaError_t tiled_enqueue(const TiledPrepared *T, cudaStream_t stream)
{
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < T->n && e == cudaSuccess; ++k) {
        const ImgDesc &D = T->descs[k];
        const JobSpec &J = T->jobs[k];
        if (D.copy_in)
            e = cudaMemcpy2DAsync(reinterpret_cast<void *>(D.buf[0]), D.pitch, J.img, J.pitch,
                                  size_t(J.w) * elem_size(J.dtype), J.h, cudaMemcpyDeviceToDevice, stream);
    }
    char *base = T->base;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(base + T->o_stat, base + T->o_stat0, sizeof(ImgStat) * T->n, cudaMemcpyDeviceToDevice, stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(base + T->o_ctl, base + T->o_ctl0, sizeof(Ctl), cudaMemcpyDeviceToDevice, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(base + T->o_listed, 0xff, sizeof(int) * T->total_tiles, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(base + T->o_cells, 0x0f, T->cells_bytes, stream);  // every group dirty
    if (e == cudaSuccess) {
        void *args[] = {const_cast<EngineArgs *>(&T->P)};
        e = cudaLaunchCooperativeKernel(T->build.kernel, dim3(T->grid), dim3(32 * T->build.warps), args, T->smem, stream);
    }
    if (e == cudaSuccess) {
        k_copy_out<<<dim3(64, T->n), 256, 0, stream>>>(T->P.imgs, T->P.st, T->n);
        e = cudaGetLastError();
    }
    return e;
}

int tiled_collect(const TiledPrepared *T, const thin_options &opt, cudaStream_t stream, thin_stats *out)
{
    const int n = T->n;
    std::vector<ImgStat> st(n);
    Ctl ctl;
    cudaError_t e = cudaMemcpyAsync(st.data(), T->P.st, sizeof(ImgStat) * n, cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&ctl, T->P.ctl, sizeof ctl, cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return cuda_status(e);
    int rc = THIN_OK;
    for (int k = 0; k < n; ++k) {
        const ImgStat &S = st[k];
        thin_stats &o = out[k];
        std::memset(&o, 0, sizeof o);
        const long long steps = S.last_step + 1;
        long long phases = steps * T->H;
        if (opt.max_phases >= 0) phases = std::min<long long>(phases, opt.max_phases);
        o.converged = (S.last_listed <= S.last_step && ctl.error == 0) ? 1 : 0;
        if (T->jobs[k].fits_cluster && opt.max_phases >= 0 && ctl.error == 0) {
            o.converged = quiet_at_cap(opt, S.last_change);
            if (!o.converged) phases = opt.max_phases;
        }
        o.status = ctl.error ? ctl.error : (o.converged ? THIN_OK : THIN_ERR_NOT_CONVERGED);
        o.phases = phases;
        o.lowered = (int64_t)S.lowered;
        o.last_change_phase = S.last_change;
        o.end_phase = opt.start_phase + phases;
        o.tiles_visited = (int64_t)S.tiles_visited;
        o.tested = (int64_t)S.tested;
        o.steps = steps;
        if (o.status != THIN_OK && rc == THIN_OK) rc = o.status;
    }
    return rc;
}

void tiled_release(TiledPrepared *T, cudaStream_t stream)
{
    if (!T) return;
    if (T->base) {
        if (T->async_alloc) cudaFreeAsync(T->base, stream);
        else cudaFree(T->base);
    }
    delete T;
}

int tiled_run(const JobSpec *jobs, int n, const thin_options &opt, cudaStream_t stream, thin_stats *out)
{
    if (n <= 0) return THIN_OK;
    if (opt.max_phases == 0) {  // nothing may run: every image stays as it is, unconverged
        if (out)
            for (int k = 0; k < n; ++k) {
                std::memset(&out[k], 0, sizeof out[k]);
                out[k].status = THIN_ERR_NOT_CONVERGED;
                out[k].last_change_phase = -1;
                out[k].end_phase = opt.start_phase;
            }
        return THIN_ERR_NOT_CONVERGED;
    }
    TiledPrepared *T = nullptr;
    int rc = tiled_prepare(jobs, n, opt, stream, true, &T);
    if (rc != THIN_OK) return rc;
    const cudaError_t e = tiled_enqueue(T, stream);
    if (e != cudaSuccess) rc = cuda_status(e);
    else if (out) rc = tiled_collect(T, opt, stream, out);
    tiled_release(T, stream);
    return rc;
}

}  // namespace thin

// ---------------------------------------------------------------------------
// Allocation-free entry point.
//
// Some callers cannot allocate device memory at the moment they want to thin
// an image: an application that hands all device memory to its own allocator
// at start-up (a further cudaMalloc would fail or eat into that budget), or a
// loop with a fixed time budget that may not call into the allocator, which
// can have to map new memory or wait for the device.  thin_run_noalloc serves
// them with the tiled engine and no allocation at all: its scratch (the
// second ping-pong buffer, the dirty bits, the worklists and the control
// words) lives in one fixed array in device memory that the library declares
// at file scope.  Every GPU that loads the library holds the array until the
// process exits.
static __device__ __align__(256) unsigned char g_thin_noalloc_scratch[THIN_NOALLOC_SCRATCH_BYTES];

namespace thin {
namespace {

struct NoallocSlot {
    unsigned long long ctx_id = 0;  // context the address belongs to (0: unknown)
    void *base = nullptr;
};
std::mutex g_noalloc_mu;
NoallocSlot g_noalloc_slot[256];

// Device address of the scratch array on the current device (in host code the
// array's name is only a host-side stand-in).  Looked up at the first call on
// a device, and again only if the device's context has been created anew
// since (after cudaDeviceReset the array lives at a new address).
cudaError_t noalloc_scratch(void **base)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoallocSlot &S = g_noalloc_slot[dev];
    const unsigned long long id = current_context_id();
    if (!S.base || id == 0 || id != S.ctx_id) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_thin_noalloc_scratch);
        if (e != cudaSuccess) return e;
        S.base = p;
        S.ctx_id = current_context_id();  // the lookup makes the context current if it was not
    }
    *base = S.base;
    return cudaSuccess;
}

// The tiled engine on one image, with every piece of scratch carved from the
// fixed array.  Same kernels, launch and result as tiled_run.
int tiled_run_noalloc(const JobSpec &J, const thin_options &opt, cudaStream_t stream, thin_stats *out)
{
    if (opt.max_phases == 0) {
        if (out) {
            std::memset(out, 0, sizeof *out);
            out->status = THIN_ERR_NOT_CONVERGED;
            out->last_change_phase = -1;
            out->end_phase = opt.start_phase;
        }
        return THIN_ERR_NOT_CONVERGED;
    }
    const bool is16 = J.dtype == THIN_U16;
    int tw, th, H;
    const int shape_rc = tiled_shape(&J, 1, is16, opt, &tw, &th, &H);
    if (shape_rc != THIN_OK) return shape_rc;
    const int HR = halo_rows(H);
    const TileLayout TL = tile_layout(tw, th, HR, is16);
    EncodeTiledFn enc = encode_fn();
    if (!enc) return THIN_ERR_CUDA;

    ImgDesc D;
    std::memset(&D, 0, sizeof D);
    D.w = J.w;
    D.h = J.h;
    D.dtype = J.dtype;
    D.lam = J.lam;
    D.adj = J.adj;
    D.tiles_x = (J.w + tw - 1) / tw;
    D.tiles_y = (J.h + th - 1) / th;
    D.tile_base = 0;
    D.cells_x = (J.w + 7) / 8;
    D.cells_y = (J.h + 1) / 2;
    const int total_tiles = D.tiles_x * D.tiles_y;
    const size_t es = elem_size(J.dtype);
    const bool aligned = (reinterpret_cast<uintptr_t>(J.img) % 16 == 0) && (J.pitch % 16 == 0);
    D.copy_in = aligned ? 0 : 1;
    D.pitch = aligned ? J.pitch : align_up(size_t(J.w) * es, 128);
    D.user = reinterpret_cast<unsigned long long>(J.img);
    D.user_pitch = J.pitch;

    // layout inside the fixed array (same pieces as tiled_run, one image)
    size_t off = 0;
    const size_t o_desc = off;
    off = align_up(off + sizeof(ImgDesc), 256);
    const size_t o_stat = off;
    off = align_up(off + sizeof(ImgStat), 256);
    const size_t o_ctl = off;
    off = align_up(off + sizeof(Ctl), 256);
    const size_t o_buf = off;
    off = align_up(off + D.pitch * J.h, 256);
    const size_t o_cpy = off;
    if (D.copy_in) off = align_up(off + D.pitch * J.h, 256);
    const size_t o_cells = off;
    const size_t cells_bytes = size_t(D.cells_x) * D.cells_y;
    off = align_up(off + cells_bytes, 256);
    const size_t o_cells1 = off;
    off = align_up(off + cells_bytes, 256);
    const size_t o_listed = off;
    off = align_up(off + sizeof(int) * total_tiles, 256);
    const size_t o_lists = off;
    off = align_up(off + sizeof(unsigned) * 3 * size_t(total_tiles), 256);
    if (off > THIN_NOALLOC_SCRATCH_BYTES) return THIN_ERR_TOO_LARGE;

    char *base = nullptr;
    cudaError_t e = noalloc_scratch(reinterpret_cast<void **>(&base));
    if (e != cudaSuccess) return cuda_status(e);

    void *b0 = D.copy_in ? static_cast<void *>(base + o_cpy) : J.img;
    void *b1 = base + o_buf;
    if (D.copy_in)
        e = cudaMemcpy2DAsync(b0, D.pitch, J.img, J.pitch, size_t(J.w) * es, J.h, cudaMemcpyDeviceToDevice, stream);
    D.buf[0] = reinterpret_cast<unsigned long long>(b0);
    D.buf[1] = reinterpret_cast<unsigned long long>(b1);
    D.cells[0] = reinterpret_cast<unsigned long long>(base + o_cells);
    D.cells[1] = reinterpret_cast<unsigned long long>(base + o_cells1);
    {
        const cuuint64_t gdim[2] = {cuuint64_t(J.w), cuuint64_t(J.h)};
        const cuuint64_t gstr[1] = {cuuint64_t(D.pitch)};
        const cuuint32_t box[2] = {cuuint32_t(tw + 2 * kPadCols), cuuint32_t(TL.box_rows)};
        const cuuint32_t est[2] = {1, 1};
        for (int q = 0; q < 2; ++q) {
            CUresult r = enc(&D.map[q], is16 ? CU_TENSOR_MAP_DATA_TYPE_UINT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 2,
                             q ? b1 : b0, gdim, gstr, box, est, CU_TENSOR_MAP_INTERLEAVE_NONE,
                             CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) return THIN_ERR_ARG;
        }
    }
    // the array keeps the previous call's contents: set everything the engine reads
    ImgStat st0;
    st0.lowered = 0;
    st0.tiles_visited = 0;
    st0.tested = 0;
    st0.last_change = -1;
    st0.last_step = -1;
    st0.last_listed = 0;
    Ctl ctl0;
    std::memset(&ctl0, 0, sizeof ctl0);
    if (e == cudaSuccess) e = cudaMemcpyAsync(base + o_desc, &D, sizeof D, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(base + o_stat, &st0, sizeof st0, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(base + o_ctl, &ctl0, sizeof ctl0, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(base + o_listed, 0xff, sizeof(int) * total_tiles, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(base + o_cells, 0x0f, cells_bytes, stream);

    EngineArgs P;
    std::memset(&P, 0, sizeof P);
    P.imgs = reinterpret_cast<const ImgDesc *>(base + o_desc);
    P.st = reinterpret_cast<ImgStat *>(base + o_stat);
    P.listed = reinterpret_cast<int *>(base + o_listed);
    P.lists = reinterpret_cast<unsigned *>(base + o_lists);
    P.ctl = reinterpret_cast<Ctl *>(base + o_ctl);
    P.n_imgs = 1;
    P.total_tiles = total_tiles;
    P.tw = tw;
    P.th = th;
    P.halo = H;
    P.hr = HR;
    P.rule = test_mode(opt);  // F^- reading and operator
    P.start_phase = opt.start_phase;
    P.max_phases = opt.max_phases;
    P.timeout_ns = 2000000000ull;
    if (const char *t = std::getenv("THIN_TIMEOUT_NS")) P.timeout_ns = std::strtoull(t, nullptr, 10);
    P.debug = 0;
    P.tl = TL;
    const int smem = 128 + TL.bytes;

    int dev = 0, sms = 0, per_sm = 0, optin = 0;
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const EngineBuild build = engine_build(total_tiles, TL, smem, sms);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, build.kernel);
    if (e == cudaSuccess && size_t(smem) + fa.sharedSizeBytes > size_t(optin)) return THIN_ERR_ARG;
    // (every build, so that the first call loads them all and a later one of another size maps nothing)
    for (const EngineBuild &b : kBuilds)
        if (e == cudaSuccess) e = allow_max_dynamic_smem(b.kernel);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, build.kernel, 32 * build.warps, smem);
    if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
    const int grid = std::max(1, std::min(sms * per_sm, total_tiles));
    if (e == cudaSuccess) {
        void *args[] = {&P};
        e = cudaLaunchCooperativeKernel(build.kernel, dim3(grid), dim3(32 * build.warps), args, smem, stream);
    }
    if (e == cudaSuccess) {
        k_copy_out<<<dim3(64, 1), 256, 0, stream>>>(P.imgs, P.st, 1);
        e = cudaGetLastError();
    }
    int rc = THIN_OK;
    if (e == cudaSuccess && out) {
        ImgStat S;
        Ctl ctl;
        e = cudaMemcpyAsync(&S, P.st, sizeof S, cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&ctl, P.ctl, sizeof ctl, cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        if (e == cudaSuccess) {
            std::memset(out, 0, sizeof *out);
            const long long steps = S.last_step + 1;
            long long phases = steps * H;
            if (opt.max_phases >= 0) phases = std::min<long long>(phases, opt.max_phases);
            out->converged = (S.last_listed <= S.last_step && ctl.error == 0) ? 1 : 0;
            out->status = ctl.error ? ctl.error : (out->converged ? THIN_OK : THIN_ERR_NOT_CONVERGED);
            out->phases = phases;
            out->lowered = (int64_t)S.lowered;
            out->last_change_phase = S.last_change;
            out->end_phase = opt.start_phase + phases;
            out->tiles_visited = (int64_t)S.tiles_visited;
            out->tested = (int64_t)S.tested;
            out->steps = steps;
            rc = out->status;
        }
    }
    if (e != cudaSuccess) return cuda_status(e);
    return rc;
}

}  // namespace
}  // namespace thin

extern "C" int thin_run_noalloc(void *img_dev, int w, int h, size_t pitch_bytes, thin_dtype dt, uint32_t lambda,
                                thin_adj adj, void *stream, const thin_options *opt, thin_stats *out)
{
    thin_options o;
    thin_default_options(&o);
    if (opt) o = *opt;
    if (adj != THIN_ADJ_8_4 && adj != THIN_ADJ_4_8) return THIN_ERR_ARG;
    if (o.rule != THIN_RULE_MAX && o.rule != THIN_RULE_MIN) return THIN_ERR_ARG;
    if (o.op != THIN_OP_THINNING && o.op != THIN_OP_SKELETON) return THIN_ERR_ARG;
    if (o.start_phase < 0 || o.tile_w < 0 || o.tile_h < 0 || o.halo < 0) return THIN_ERR_ARG;
    if (w < 0 || h < 0 || (dt != THIN_U8 && dt != THIN_U16)) return THIN_ERR_ARG;
    const size_t es = dt == THIN_U16 ? 2 : 1;
    if (w > 0 && h > 0) {
        if (!img_dev || pitch_bytes < size_t(w) * es) return THIN_ERR_ARG;
        if (es == 2 && ((reinterpret_cast<uintptr_t>(img_dev) & 1) || (pitch_bytes & 1))) return THIN_ERR_ARG;
    }
    if (w < 3 || h < 3) {  // empty, or no interior point: nothing to do
        if (out) {
            std::memset(out, 0, sizeof *out);
            out->converged = 1;
            out->last_change_phase = -1;
            out->end_phase = o.start_phase;
        }
        return THIN_OK;
    }
    thin::JobSpec j{img_dev, w, h, pitch_bytes, int(dt), lambda, int(adj)};
    return thin::tiled_run_noalloc(j, o, static_cast<cudaStream_t>(stream), out);
}
