// thin_tile.cuh -- a tile of an image and its halo in a block's shared memory,
// and the phases of a step on it: shared by the tiled engine, whose blocks load
// and store a tile every step, and the mosaic engine, whose blocks keep theirs.
#pragma once

#include <cstddef>
#include <cstdint>

#include "thin_block.cuh"
#include "thin_common.cuh"
#include "thin_layout.h"
#include "thin_simd.cuh"

namespace thin {

__device__ __forceinline__ unsigned long long gtimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Exact n / d for n, d < 2^16 with M = floor(2^32 / d) + 1 (M unused when d == 1).
__device__ __forceinline__ int div_small(int n, int d, uint32_t M)
{
    return d == 1 ? n : int(__umulhi(uint32_t(n), M));
}

__device__ __forceinline__ uint32_t div_magic(int d)
{
    return d > 1 ? 0xffffffffu / uint32_t(d) + 1u : 0u;
}

// One visit of a block: the tile, its place in the image and the step.
struct Visit {
    int w, h;           // image size
    int x0, y0;         // tile origin in the image
    int tw, th;         // tile size
    int Hs, hr;         // phases to run, halo rows staged
    long long g0;       // global index of the first phase of the step
};

// The block's control words.
struct TileCtrl {
    unsigned qn[2];     // fill counters of the queue, alternating by phase
    unsigned next;      // the next list entry to visit
    unsigned near;      // bit 3 (dy + 1) + dx + 1: the tile at (dx, dy) may change next step
    int last;           // last phase of the step that moved a point of the tile, -1 none
};
static_assert(sizeof(TileCtrl) <= kOffBar - kOffCtrl, "control words overlap the mbarrier");

// Hs phases of the subfield schedule on a staged tile.  Staged column 0 is
// image column x0 - kPadCols, staged row 0 image row y0 - hr.  Phase j updates
// the points of its parity within distance Hs - j of the tile and off the image
// border; after Hs phases the tile and its dirty bits are exact.  A bitmap has at
// most a word per thread.
template <typename T, int THREADS>
__device__ __forceinline__ void visit_phases(const TileLayout &L, uint8_t *smem, const Visit &V, const PointRule &rule,
                                             int &nlow, int &ntest, int &chg_j)
{
    TileCtrl *ctrl = reinterpret_cast<TileCtrl *>(smem + kOffCtrl);
    uint32_t *dirty = reinterpret_cast<uint32_t *>(smem + L.dirty_off);
    uint16_t *queue = reinterpret_cast<uint16_t *>(smem + L.queue_off);
    const int words = L.rows / 2;
    PieceMap map;
    map.rows = smem + kOffTile;
    map.dirty = smem_u32(dirty);
    map.pitch = L.row_bytes;
    map.cell_words = 1;
    map.bitmap_words = words;
    map.cbits = 5;
    map.own_row = V.hr / 2;
    map.own_rows = V.th / 2;
    map.own_col = kPadCols / 8;
    map.own_cols = V.tw / 8;
    // this thread's piece of a bitmap: a byte, or 16 or 32 bits where there are more of them than threads
    const int unit = words * 4 <= THREADS ? 0 : words * 2 <= THREADS ? 1 : 2;
    const int pword = int(threadIdx.x) >> (2 - unit), pshift = (int(threadIdx.x) << (3 + unit)) & 31;
    const uint32_t pones = unit == 0 ? 0xffu : unit == 1 ? 0xffffu : 0xffffffffu;
    for (int j = 0; j < V.Hs; ++j) {
        const int p = int((V.g0 + j) & 3), px = p & 1, py = p >> 1;
        const int r = V.Hs - j;
        const int xlo = max(V.x0 - r, 1) - V.x0 + kPadCols, xhi = min(V.x0 + V.tw - 1 + r, V.w - 2) - V.x0 + kPadCols;
        if (pword < words) {
            uint32_t *dp = dirty + p * words;
            uint32_t d = (dp[pword] >> pshift) & pones;
            if (d) {
                if (unit == 0) reinterpret_cast<uint8_t *>(dp)[threadIdx.x] = 0;
                else if (unit == 1) reinterpret_cast<uint16_t *>(dp)[threadIdx.x] = 0;
                else dp[threadIdx.x] = 0;
                const int y = V.y0 - V.hr + 2 * pword + py;
                const uint32_t cols = (0xffffffffu << (xlo >> 3)) & (0xffffffffu >> (31 - (xhi >> 3)));
                d &= cols >> pshift;
                if (d && y >= max(V.y0 - r, 1) && y <= min(V.y0 + V.th - 1 + r, V.h - 2)) {
                    uint16_t *q = queue + atomicAdd(&ctrl->qn[j & 1], unsigned(__popc(d)));
                    int code = (pword << 5) | pshift;
                    do {
#pragma unroll
                        for (int b = 0; b < 8; ++b)
                            if ((d >> b) & 1u) *q++ = uint16_t(code + b);
                        code += 8;
                        d >>= 8;
                    } while (d);
                }
            }
        }
        __syncthreads();
        const int N = int(*reinterpret_cast<volatile unsigned *>(&ctrl->qn[j & 1]));
        if (threadIdx.x == 0) ctrl->qn[(j + 1) & 1] = 0u;  // last read in the previous phase
        if (work_queue<T, THREADS>(map, rule, queue, N, px, py, xlo, xhi, nlow, ntest)) chg_j = j;
        __syncthreads();
    }
}

}  // namespace thin
