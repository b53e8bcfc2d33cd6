// thin_block.cuh -- the work of one phase on a piece of an image that a thread
// block holds in shared memory, shared by the resident and the tiled engine.
//
// The piece is rows of pixels (a cell is 8 columns x 2 rows, aligned to the
// image) and four dirty bitmaps, one per parity 2 (y & 1) + (x & 1), with a bit
// per cell: "a neighbour of one of the cell's four points of this parity moved
// since their last test".  A phase takes its parity's bits, queues their cells
// as groups of four points, tests and lowers them, and marks the groups whose
// test a move can change.
#pragma once

#include <cstdint>

#include "thin_common.cuh"
#include "thin_simd.cuh"

namespace thin {

// Where the piece lies and which of its points count.
struct PieceMap {
    uint8_t *rows;       // row 0, column 0 (shared memory; the words just left and right of a cell are readable)
    uint32_t dirty;      // shared address of the four bitmaps
    int pitch;           // bytes between rows
    int cell_words;      // bitmap words per cell row
    int bitmap_words;    // words of one bitmap
    int cbits;           // a group's code is (cell row << cbits) | cell column
    int own_row, own_rows;  // cell rows and columns whose points count
    int own_col, own_cols;
};

// ORs m into a word of shared memory; nothing where m is 0 (a predicate, not a branch).
__device__ __forceinline__ void smem_or(uint32_t addr, uint32_t m)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %1, 0;\n @p red.shared.or.b32 [%0], %1;\n}\n" ::"r"(addr), "r"(m) : "memory");
}

// The groups of the other three parities holding a neighbour to test again
// become dirty.  A: byte k holds the ring directions (bit 0 E, 1 NE, 2 N, 3 NW,
// 4 W, 5 SW, 6 S, 7 SE) of point k's neighbours to mark.  E and W neighbours
// are in the row's other column parity, N and S in the other row parity, the
// diagonals in the fourth.  For px == 0 the W side of point 0 is in the cell to
// the left; for px == 1 the E side of point 3 is in the cell to the right.
// Rows y - 1 and y + 1 of a tested point are held, and so are the cells beside it.
__device__ __forceinline__ void mark_neighbours(const PieceMap &m, int cr, int cc, uint32_t A, int px, int py)
{
    const uint32_t bytes = 4u * uint32_t(m.bitmap_words), below = 4u * uint32_t(m.cell_words), up = py ? 0u : 0u - below;
    const uint32_t beside = px ? 0x83000000u : 0x00000038u;  // towards the cell beside
    const uint32_t X = A & beside, x = px ? X >> 24 : X;
    uint32_t f = A ^ X;  // the rest, folded into one set of directions
    f |= f >> 16;
    f |= f >> 8;
    const uint32_t mc = 1u << (cc & 31);
    const uint32_t mx = px ? mc << 1 : mc >> 1;  // 0: the cell beside is in the next word
    const uint32_t mrow = (f & 0x11u ? mc : 0u) | (x & 0x11u ? mx : 0u);
    const uint32_t ma = (f & 0x0au ? mc : 0u) | (x & 0x0au ? mx : 0u);
    const uint32_t mb = (f & 0xa0u ? mc : 0u) | (x & 0xa0u ? mx : 0u);
    // word of the group's own cell in the bitmap of each parity; for the last two of the cell row of y - 1
    const uint32_t o = m.dirty + 4u * uint32_t(cr * m.cell_words + (cc >> 5));
    const uint32_t drow = o + bytes * uint32_t(2 * py + (px ^ 1));
    const uint32_t dcol = o + (bytes * uint32_t(2 * (py ^ 1) + px) + up);
    const uint32_t ddiag = o + (bytes * uint32_t(2 * (py ^ 1) + (px ^ 1)) + up);
    smem_or(drow, mrow);
    smem_or(dcol, f & 0x04u ? mc : 0u);
    smem_or(ddiag, ma);
    smem_or(dcol + below, f & 0x40u ? mc : 0u);
    smem_or(ddiag + below, mb);
    if (mx == 0u && x) {  // the group across a word boundary (rare)
        const uint32_t ws = px ? 4u : ~3u, ms = px ? 1u : 0x80000000u;
        smem_or(drow + ws, x & 0x11u ? ms : 0u);
        smem_or(ddiag + ws, x & 0x0au ? ms : 0u);
        smem_or(ddiag + below + ws, x & 0xa0u ? ms : 0u);
    }
}

// Tests and lowers the N queued groups of parity (px, py) with the THREADS
// threads of the block.  Only the points in columns lo .. hi are tested.  With
// few groups a lane goes to a point; otherwise a thread to a group, the chunks
// of 32 groups going to the warps in turn (every chunk but the last is full, and
// the schedulers' shares differ by one chunk at most: against even shares for
// all warps 192 512^2 u8 images went from 16.4 to 15.2 ms).  Adds the steps and
// tests of points that count to nlow and ntest; returns whether one of them moved.
template <typename T, int THREADS>
__device__ __forceinline__ bool work_queue(const PieceMap &m, const PointRule &rule, const uint16_t *queue, int N, int px,
                                           int py, int lo, int hi, int &nlow, int &ntest)
{
    // Phases with at most this many groups take a lane to a point (four to a
    // group): 64^2 at lambda = 10 245 -> 220 us, 192 512^2 u16 images
    // 24.1 -> 23.9 ms; with twice as many a block's lanes take two turns, and the
    // u8 batch lost 3 %.
    constexpr int kLaneItems = THREADS / 4;
    bool moved = false;
    const int rest = N % THREADS, quads = rest <= kLaneItems ? N - rest : N;
    if (quads < N) {
        const int k = quads + (int(threadIdx.x) >> 2), j4 = threadIdx.x & 3;
        if (k < N) {
            const int code = queue[k];
            const int cr = code >> m.cbits, cc = code - (cr << m.cbits);
            const int x = 8 * cc + px + 2 * j4;
            if (x >= lo && x <= hi) {
                T *rb = reinterpret_cast<T *>(m.rows + (2 * cr + py) * m.pitch) + x;
                const T *ra = reinterpret_cast<const T *>(reinterpret_cast<const uint8_t *>(rb) - m.pitch);
                const T *rc = reinterpret_cast<const T *>(reinterpret_cast<const uint8_t *>(rb) + m.pitch);
                uint32_t A;
                const int n = lower_one<T>(ra, rb, rc, rule, A);
                if (unsigned(cr - m.own_row) < unsigned(m.own_rows) && unsigned(cc - m.own_col) < unsigned(m.own_cols)) {
                    ++ntest;
                    nlow += n;
                    moved = n > 0;
                }
                if (A) mark_neighbours(m, cr, cc, A << (8 * j4), px, py);
            }
        }
    }
    {
        for (int k = threadIdx.x; k < quads; k += THREADS) {
            const int code = queue[k];
            const int cr = code >> m.cbits, cc = code - (cr << m.cbits);
            const int first = (lo - px - 8 * cc + 1) >> 1, last = (hi - px - 8 * cc) >> 1;  // of the points 0 .. 3
            uint32_t vm = last >= 3 ? kLsb8 : last >= 0 ? kLsb8 >> (8 * (3 - last)) : 0u;
            if (first > 0) vm = first < 4 ? vm & (kLsb8 << (8 * first)) : 0u;
            const bool own = unsigned(cr - m.own_row) < unsigned(m.own_rows) && unsigned(cc - m.own_col) < unsigned(m.own_cols);
            const uint32_t in = own ? vm : 0u;
            ntest += int((in * kLsb8) >> 24);
            T *rb = reinterpret_cast<T *>(m.rows + (2 * cr + py) * m.pitch) + 8 * cc;
            const T *ra = reinterpret_cast<const T *>(reinterpret_cast<const uint8_t *>(rb) - m.pitch);
            const T *rc = reinterpret_cast<const T *>(reinterpret_cast<const uint8_t *>(rb) + m.pitch);
            uint32_t aff;
            moved |= (lower_item(ra, rb, rc, px, vm, in, rule, nlow, aff) & in) != 0;
            if (aff) mark_neighbours(m, cr, cc, aff, px, py);
        }
    }
    return moved;
}

}  // namespace thin
