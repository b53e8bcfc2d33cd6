// thin_layout.h -- sizes of a tile in a block's shared memory and the mosaic
// engine's choice of a tile shape.  Host arithmetic only: a host compiler can
// build it without CUDA.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>

#include "thin_common.cuh"

namespace thin {

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
constexpr int kMinHalo = 3;
constexpr int kPadCols = 16;   // halo columns staged on each side of a tile (two cells)
constexpr int kMaxStep = 15;   // phases a step can have: one halo column more than that is needed

// Shared memory of a block: decision table, control words, tile rows, dirty
// bitmaps (a word per cell row and parity: a tile and its halo are at most 32
// cells wide), queue of groups.
struct TileLayout {
    int row_bytes;   // bytes of a staged row (tile and halo columns)
    int rows;        // staged rows
    int box_rows;    // rows of one TMA box (one or two boxes to a tile)
    int dirty_off, queue_off, bytes;
};
constexpr int kOffCtrl = (kDecisionBytes + 15) / 16 * 16;  // control words, then the mbarrier
constexpr int kOffBar = kOffCtrl + 32;
constexpr int kOffTile = (kOffBar + 8 + 127) / 128 * 128 + 128;  // TMA destinations are 128-byte aligned

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Shared memory of a block for tiles tw x th with hr halo rows.  A tile of more
// than 256 staged rows takes two TMA boxes, each starting at a multiple of 128 bytes.
inline TileLayout tile_layout(int tw, int th, int hr, bool any16)
{
    TileLayout L;
    L.row_bytes = (tw + 2 * kPadCols) * (any16 ? 2 : 1);
    L.rows = th + 2 * hr;
    L.box_rows = L.rows;
    if (L.rows > 256) {
        L.box_rows = int(align_up(size_t(L.rows + 1) / 2, 8));
        L.rows = 2 * L.box_rows;
    }
    L.dirty_off = int(align_up(size_t(kOffTile) + size_t(L.row_bytes) * L.rows + 16, 16));
    L.queue_off = L.dirty_off + 4 * 4 * (L.rows / 2);
    L.bytes = L.queue_off + 2 * 32 * (L.rows / 2);
    return L;
}

// Halo rows for steps of H phases: one pixel more than phases, even.
inline int halo_rows(int H) { return (H + 2) / 2 * 2; }

// ---- mosaic engine (thin_mosaic.cu)

struct MosaicShape {
    int tw, th, halo;  // tile, phases per step
};
constexpr int kMosMaxRows = 304;  // the highest tile

// The turns of the block's threads in which the rims' side columns go to and
// from global memory, es 16-byte vectors a side and row: enough for the highest tile.
constexpr int mosaic_side_turns(int es) { return (2 * es * kMosMaxRows + kThreads - 1) / kThreads; }

// What the exchange of rims and the phases rest on (es: element size).
constexpr bool mosaic_shape_fits(int es, const MosaicShape &s)
{
    const int hr = (s.halo + 2) / 2 * 2;  // halo_rows
    return s.tw % 16 == 0 && s.th % 2 == 0 &&              // cells of 8 x 2, vectors of 16 bytes
           s.halo >= 1 && s.halo < kPadCols &&             // a halo column more than a step has phases
           s.tw >= kPadCols && s.th >= hr &&               // a halo reaches into the next tile only
           s.tw / 8 + 4 <= 32 && s.tw * es / 16 + 2 * es <= 32 &&  // a lane to a cell, a lane to a vector of a row
           hr <= 2 * kWarps &&                             // the halo's rows in four turns of the warps, its cell rows in two
           s.th <= kMosMaxRows && 2 * es * s.th <= mosaic_side_turns(es) * kThreads &&  // the side columns
           (s.th + 2 * hr + 16) / 2 <= kThreads;           // a thread to a cell row (two TMA boxes round the rows up)
}

template <typename Job>
int mosaic_tiles(const Job *jobs, int n, int tw, int th)
{
    long long t = 0;
    for (int k = 0; k < n; ++k) t += (long long)((jobs[k].w + tw - 1) / tw) * ((jobs[k].h + th - 1) / th);
    return int(std::min<long long>(t, 1 << 30));
}

// How many tiles: about one for every 10 pixels of an image's side (the root of
// its area), so that a whole number of such calls fill the block slots.  Small
// tiles gain little, since each also tests its ring, and calls on other streams
// run beside this one only if their blocks all fit.  One call, and 16 calls on
// 16 streams, in ms, on the clusters and the wide mode / with tiles in all slots /
// by this rule (u8): 512^2 at lambda = 0 0.56 / 0.22 / 0.22 and 1.54 / 2.95 /
// 0.91, at lambda = 20 6.9 / 2.7 / 2.9 and 10.6 / 39.2 / 8.9; 256^2 3.1 / 1.4 /
// 1.55 and 5.9 / 11.4 / 3.6; 1000^2 17.4 / 5.0 / 5.3 and 33.9 / 79.6 / 33.3;
// 2048^2 at lambda = 30 30.0 / 11.7 / 13.2 and 173 / 188 / 122; 4 batches of 4
// 512^2 images on 4 streams 10.3 / 13.8 / 7.8.  A tile every 8 or 12 pixels: one
// call 4 % less or 6 % more, 16 at once 30 % more or 8 % less.  (Long strips need
// more tiles than that: all slots.)  limit: shared memory a block may take, two
// blocks to an SM.  False if the images do not fit.
template <typename Job>
bool mosaic_search(const Job *jobs, int n, bool any16, int sms, int limit, MosaicShape *out)
{
    const int slots = 2 * sms;
    double want = 0;
    for (int k = 0; k < n; ++k) want += std::max(std::sqrt(double(jobs[k].w) * jobs[k].h) / 10, 8.0);
    for (int most : {slots / std::max(int(slots / want + 0.6), 1), slots}) {
        // for every width the lowest tile that gives few enough tiles; of these the smallest with its halo
        double best = 0;
        for (int tw = 32; tw <= 224; tw += 16) {
            int lo = 16, hi = kMosMaxRows;
            if (mosaic_tiles(jobs, n, tw, hi) > most) continue;
            while (lo < hi) {
                const int mid = (lo + hi) / 16 * 8;  // a multiple of 8 below hi
                if (mosaic_tiles(jobs, n, tw, mid) <= most) hi = mid;
                else lo = mid + 8;
            }
            const double cost = double(tw + 16) * (hi + 16);
            if ((best == 0 || cost < best) && tile_layout(tw, hi, halo_rows(kMaxStep), any16).bytes <= limit) {
                best = cost;
                out->tw = tw;
                out->th = hi;
                out->halo = kMaxStep;
            }
        }
        if (best > 0) return true;
    }
    return false;
}

}  // namespace thin
