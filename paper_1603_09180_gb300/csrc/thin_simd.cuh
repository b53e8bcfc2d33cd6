// thin_simd.cuh -- the point test of Sec. 2.1 and the lowering loop of
// Sec. 2.2 on four points of one parity at once, shared by the engines.
//
// A work item is the four points (x0 + px + 2k, y), k = 0..3, of one parity in
// an 8-pixel aligned block of row y.  The callers pass pointers to that block
// in rows y - 1, y and y + 1; the rows must hold readable pixels from 1 pixel
// left to 1 pixel right of the block (u8: the aligned words just left and
// right of it).
//
// What bounds it.  A work item is a few hundred instructions on values that
// are in registers, so it runs at the rate of the pipe that takes most of
// them.  Compares and mask merges on integer lanes all go to the ALU pipe (one
// warp instruction per two cycles and scheduler: measured 0.50 SM cycles a
// LOP3, PRMT or shift), while the FMA pipes idle.  Here the comparisons are
// floating-point subtractions with saturation: for integers a, b held exactly,
// sat(a - b) is 1 where a > b and 0 where not, and one FMA adds the result,
// times its weight, to a sum.  u8 pixels are taken as the halves 1024 + v, two
// points to a register (HADD2.SAT / HFMA2: 0.50 SM cycles for two points); u16
// pixels as the floats 2^23 + v (FADD.SAT / FFMA: 0.26 and 0.25).  With these
// biases a value's bits are the bias's bits plus v, so pixels enter by one
// byte permute and sums leave as integers without a conversion.  The sums with
// weights 3^d index the decision table, so the test itself is one byte load a
// point in every mode (the adjacency pair (4,8) and the skeleton too).  Against
// the same steps on integer lanes (about 1000 ALU instructions per 32 items):
// 192 512^2 images 20.6 -> 16.4 ms (u8), 37.9 -> 27.7 ms (u16), 24.1 -> 16.0 ms
// (skeleton); 64 under (4,8), which went through a table point by point,
// 16.4 -> 4.0 ms; 8192^2 u16 at lambda = 30 36.9 -> 25.4 ms.
#pragma once

#include <cstdint>

#include "thin_common.cuh"

namespace thin {

constexpr uint32_t kLsb8 = 0x01010101u;

// a - b clamped to [0, 1], and a * b + c, on two halves.
__device__ __forceinline__ uint32_t h2_subsat(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("sub.sat.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t h2_sub(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t h2_add(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("add.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t h2_fma(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t r;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

__device__ __forceinline__ uint32_t lds_u8(uint32_t addr)
{
    uint32_t v;
    asm("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// The half of a small non-negative integer, in both lanes.
__device__ constexpr uint32_t h2_of(int n)
{
    if (n == 0) return 0;
    int e = 0;
    while ((n >> (e + 1)) != 0) ++e;
    const uint32_t h = uint32_t((e + 15) << 10) | ((uint32_t(n) << (10 - e)) & 0x3ffu);
    return h | (h << 16);
}

// The same for a run-time n < 1024: 1024 + n has the bits 0x6400 + n.
__device__ __forceinline__ uint32_t h2_from(uint32_t n) { return h2_sub((0x6400u + n) * 0x10001u, 0x64006400u); }

// What the test of a job needs besides the pixels.
struct PointRule {
    uint32_t tab;   // shared address of the decision table
    uint32_t mode;  // the decision's bit in a table entry
    uint32_t lam;   // lambda, capped at the largest difference of two pixels
    uint32_t lamh;  // lambda as two halves (u8 images)
    float lamf;
    bool cap;       // bound the marks by the old value + lambda (lower_item)
};

__device__ __forceinline__ PointRule point_rule(const void *table_smem, int mode, uint32_t lam, int es, bool cap)
{
    PointRule r;
    r.tab = static_cast<uint32_t>(__cvta_generic_to_shared(table_smem));
    r.mode = uint32_t(mode);
    r.lam = min(lam, es == 1 ? 255u : 65535u);
    r.lamh = h2_from(min(r.lam, 255u));
    r.lamf = float(r.lam);
    r.cap = cap;
    return r;
}

// Copies the decision table to shared memory (16-byte aligned); the caller synchronises.
__device__ __forceinline__ void load_decisions(void *smem, const DecisionTable &t)
{
    for (int i = threadIdx.x; i < kDecisionBytes / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(smem)[i] = reinterpret_cast<const uint4 *>(t.v)[i];
}

// The work item of a u8 image.  Points 0 and 1 are the halves of the words A,
// points 2 and 3 those of B.
struct Quad8 {
    uint32_t nA[8], nB[8];  // neighbours in ring order E, NE, N, NW, W, SW, S, SE
    uint32_t cA, cB;        // centre values
    uint2 wb;               // row y's block as loaded

    static constexpr uint32_t kBias = 0x64006400u;

    // Bytes 0 and 2 (odd: 1 and 3) of w as biased halves.
    static __device__ __forceinline__ uint32_t even(uint32_t w) { return __byte_perm(w, 0x64646464u, 0x4240); }
    static __device__ __forceinline__ uint32_t odd(uint32_t w) { return __byte_perm(w, 0x64646464u, 0x4341); }

    __device__ __forceinline__ void gather(const uint8_t *ra, const uint8_t *rb, const uint8_t *rc, int px)
    {
        const uint2 wa = *reinterpret_cast<const uint2 *>(ra);
        wb = *reinterpret_cast<const uint2 *>(rb);
        const uint2 wc = *reinterpret_cast<const uint2 *>(rc);
        if (px == 0) {  // points at pixels 0, 2, 4, 6: E is odd(), W the pixel before
            const uint32_t la = *reinterpret_cast<const uint32_t *>(ra - 4);
            const uint32_t lb = *reinterpret_cast<const uint32_t *>(rb - 4);
            const uint32_t lc = *reinterpret_cast<const uint32_t *>(rc - 4);
            cA = even(wb.x);
            cB = even(wb.y);
            nA[0] = odd(wb.x);
            nB[0] = odd(wb.y);
            nA[1] = odd(wa.x);
            nB[1] = odd(wa.y);
            nA[2] = even(wa.x);
            nB[2] = even(wa.y);
            nA[3] = even(__byte_perm(la, wa.x, 0x6543));
            nB[3] = even(__byte_perm(wa.x, wa.y, 0x6543));
            nA[4] = even(__byte_perm(lb, wb.x, 0x6543));
            nB[4] = even(__byte_perm(wb.x, wb.y, 0x6543));
            nA[5] = even(__byte_perm(lc, wc.x, 0x6543));
            nB[5] = even(__byte_perm(wc.x, wc.y, 0x6543));
            nA[6] = even(wc.x);
            nB[6] = even(wc.y);
            nA[7] = odd(wc.x);
            nB[7] = odd(wc.y);
        } else {  // points at pixels 1, 3, 5, 7: W is even(), E the pixel after
            const uint32_t la = *reinterpret_cast<const uint32_t *>(ra + 8);
            const uint32_t lb = *reinterpret_cast<const uint32_t *>(rb + 8);
            const uint32_t lc = *reinterpret_cast<const uint32_t *>(rc + 8);
            cA = odd(wb.x);
            cB = odd(wb.y);
            nA[0] = odd(__byte_perm(wb.x, wb.y, 0x4321));
            nB[0] = odd(__byte_perm(wb.y, lb, 0x4321));
            nA[1] = odd(__byte_perm(wa.x, wa.y, 0x4321));
            nB[1] = odd(__byte_perm(wa.y, la, 0x4321));
            nA[2] = odd(wa.x);
            nB[2] = odd(wa.y);
            nA[3] = even(wa.x);
            nB[3] = even(wa.y);
            nA[4] = even(wb.x);
            nB[4] = even(wb.y);
            nA[5] = even(wc.x);
            nB[5] = even(wc.y);
            nA[6] = odd(wc.x);
            nB[6] = odd(wc.y);
            nA[7] = odd(__byte_perm(wc.x, wc.y, 0x4321));
            nB[7] = odd(__byte_perm(wc.y, lc, 0x4321));
        }
    }

    // Adds to each sum the weights w[d % 4] of the neighbours below c: directions
    // 0..3 to lo, 4..7 to hi (so that every sum stays below 1024, exact and with
    // its integer in the low bits).
    static __device__ __forceinline__ void add_below(const uint32_t n[8], uint32_t c, uint32_t &lo, uint32_t &hi)
    {
        constexpr uint32_t w[4] = {h2_of(1), h2_of(3), h2_of(9), h2_of(27)};
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            lo = h2_fma(h2_subsat(c, n[d]), w[d], lo);
            hi = h2_fma(h2_subsat(c, n[d + 4]), w[d], hi);
        }
    }

    // 0x01 in the bytes of the points that may be lowered at the current values (vm: the points that exist).
    __device__ __forceinline__ uint32_t decide(const PointRule &R, uint32_t vm) const
    {
        uint32_t loA = kBias, hiA = kBias, loB = kBias, hiB = kBias;
        add_below(nA, cA, loA, hiA);
        add_below(nB, cB, loB, hiB);
        uint32_t base = R.tab - 0x6400u;
        if (R.lam != 0) {
            add_below(nA, h2_sub(cA, R.lamh), loA, hiA);
            add_below(nB, h2_sub(cB, R.lamh), loB, hiB);
        }
        // state index per lane, biased by 0x6400: lo + 81 hi
        uint32_t iA = (hiA & 0x00ff00ffu) * 81u + loA, iB = (hiB & 0x00ff00ffu) * 81u + loB;
        if (R.lam == 0) {  // every lower neighbour is deep: twice the index (and the bias), within the lane
            iA <<= 1;
            iB <<= 1;
            base -= 0x6400u;
        }
        const uint32_t t0 = lds_u8(base + (iA & 0xffffu)), t1 = lds_u8(base + (iA >> 16));
        const uint32_t t2 = lds_u8(base + (iB & 0xffffu)), t3 = lds_u8(base + (iB >> 16));
        const uint32_t t = __byte_perm(__byte_perm(t0, t1, 0x0040), __byte_perm(t2, t3, 0x0040), 0x5410);
        return (t >> R.mode) & vm;
    }

    // alpha^- at the points of ok.  n - c mod 2^16 is largest for the largest n below c.
    __device__ __forceinline__ void lower(uint32_t ok)
    {
        const uint32_t mA = ~cA + 0x00010001u, mB = ~cB + 0x00010001u;  // -c per lane (c is never 0)
        uint32_t dA = 0, dB = 0;
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            dA = __viaddmax_u16x2(nA[d], mA, dA);
            dB = __viaddmax_u16x2(nB[d], mB, dB);
        }
        const uint32_t okm = ok * 0xffu;
        const uint32_t kA = __byte_perm(okm, 0, 0x1100), kB = __byte_perm(okm, 0, 0x3322);
        cA = (__viaddmax_u16x2(cA, dA, 0) & kA) | (cA & ~kA);
        cB = (__viaddmax_u16x2(cB, dB, 0) & kB) | (cB & ~kB);
    }

    struct Centre {
        uint32_t A, B;
    };
    __device__ __forceinline__ Centre centre() const { return {cA, cB}; }

    // Neighbours above the centre value c1 and, with R.cap, at most the old value c0 + lambda:
    // bit d of byte k for direction d of point k.
    __device__ __forceinline__ uint32_t above(const PointRule &R, Centre c0) const
    {
        uint32_t sA = kBias, sB = kBias;
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            sA = h2_fma(h2_subsat(nA[d], cA), h2_of(1 << d), sA);
            sB = h2_fma(h2_subsat(nB[d], cB), h2_of(1 << d), sB);
        }
        if (R.cap) {
            const uint32_t tA = h2_add(c0.A, R.lamh), tB = h2_add(c0.B, R.lamh);
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                sA = h2_fma(h2_subsat(nA[d], tA), h2_of(1 << d) | 0x80008000u, sA);
                sB = h2_fma(h2_subsat(nB[d], tB), h2_of(1 << d) | 0x80008000u, sB);
            }
        }
        return __byte_perm(sA, sB, 0x6420);
    }

    // Writes the four points' values back into row y's block.
    __device__ __forceinline__ void store(uint8_t *rb, int px) const
    {
        const uint32_t sel = px == 0 ? 0x3614u : 0x6240u;
        *reinterpret_cast<uint2 *>(rb) = make_uint2(__byte_perm(wb.x, cA, sel), __byte_perm(wb.y, cB, sel));
    }
};

// The work item of a u16 image: one float to a point.
struct Quad16 {
    float p[3][9];  // rows y - 1, y, y + 1: pixels px - 1 .. px + 7 of the block; point k is p[1][2 k + 1]
    float c[4];     // centre values
    uint4 wb;       // row y's block as loaded

    static constexpr uint32_t kBias = 0x4b000000u;  // 2^23

    static __device__ __forceinline__ float lo16(uint32_t w) { return __uint_as_float(__byte_perm(w, kBias, 0x7610)); }
    static __device__ __forceinline__ float hi16(uint32_t w) { return __uint_as_float(__byte_perm(w, kBias, 0x7632)); }

    __device__ __forceinline__ void gather(const uint16_t *ra, const uint16_t *rb, const uint16_t *rc, int px)
    {
        const uint16_t *rows[3] = {ra, rb, rc};
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const uint4 w = *reinterpret_cast<const uint4 *>(rows[r]);
            if (r == 1) wb = w;
            if (px == 0) {
                p[r][0] = hi16(*reinterpret_cast<const uint32_t *>(rows[r] - 2));
                p[r][1] = lo16(w.x);
                p[r][2] = hi16(w.x);
                p[r][3] = lo16(w.y);
                p[r][4] = hi16(w.y);
                p[r][5] = lo16(w.z);
                p[r][6] = hi16(w.z);
                p[r][7] = lo16(w.w);
                p[r][8] = hi16(w.w);
            } else {
                p[r][0] = lo16(w.x);
                p[r][1] = hi16(w.x);
                p[r][2] = lo16(w.y);
                p[r][3] = hi16(w.y);
                p[r][4] = lo16(w.z);
                p[r][5] = hi16(w.z);
                p[r][6] = lo16(w.w);
                p[r][7] = hi16(w.w);
                p[r][8] = lo16(*reinterpret_cast<const uint32_t *>(rows[r] + 8));
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) c[k] = p[1][2 * k + 1];
    }

    // Neighbour d of point k, ring order E, NE, N, NW, W, SW, S, SE.
    __device__ __forceinline__ float nb(int k, int d) const
    {
        constexpr int dx[8] = {1, 1, 0, -1, -1, -1, 0, 1}, dy[8] = {0, -1, -1, -1, 0, 1, 1, 1};
        return p[1 + dy[d]][2 * k + 1 + dx[d]];
    }

    __device__ __forceinline__ uint32_t decide(const PointRule &R, uint32_t vm) const
    {
        constexpr float w[8] = {1, 3, 9, 27, 81, 243, 729, 2187};
        float s[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = __uint_as_float(kBias);
#pragma unroll
        for (int d = 0; d < 8; ++d)
#pragma unroll
            for (int k = 0; k < 4; ++k) s[k] = __fmaf_rn(__saturatef(__fsub_rn(c[k], nb(k, d))), w[d], s[k]);
        if (R.lam != 0) {
#pragma unroll
            for (int d = 0; d < 8; ++d)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    s[k] = __fmaf_rn(__saturatef(__fsub_rn(__fsub_rn(c[k], R.lamf), nb(k, d))), w[d], s[k]);
        }
        uint32_t t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t i = __float_as_uint(s[k]) - kBias;
            t[k] = lds_u8(R.tab + (R.lam != 0 ? i : 2u * i));  // lambda = 0: every lower neighbour is deep
        }
        const uint32_t b = __byte_perm(__byte_perm(t[0], t[1], 0x0040), __byte_perm(t[2], t[3], 0x0040), 0x5410);
        return (b >> R.mode) & vm;
    }

    __device__ __forceinline__ void lower(uint32_t ok)
    {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t m = 0u - __float_as_uint(c[k]);
            uint32_t best = 0;
#pragma unroll
            for (int d = 0; d < 8; ++d) best = __viaddmax_u32(__float_as_uint(nb(k, d)), m, best);
            const uint32_t v = __float_as_uint(c[k]) + best;
            c[k] = ((ok >> (8 * k)) & 1u) ? __uint_as_float(v) : c[k];
        }
    }

    struct Centre {
        float v[4];
    };
    // (the values before the loop are the block's own pixels)
    __device__ __forceinline__ Centre centre() const { return {{p[1][1], p[1][3], p[1][5], p[1][7]}}; }

    __device__ __forceinline__ uint32_t above(const PointRule &R, Centre c0) const
    {
        float s[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = __uint_as_float(kBias);
#pragma unroll
        for (int d = 0; d < 8; ++d)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                s[k] = __fmaf_rn(__saturatef(__fsub_rn(nb(k, d), c[k])), float(1 << d), s[k]);
        if (R.cap) {
#pragma unroll
            for (int d = 0; d < 8; ++d)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    s[k] = __fmaf_rn(__saturatef(__fsub_rn(nb(k, d), __fadd_rn(c0.v[k], R.lamf))), -float(1 << d), s[k]);
        }
        const uint32_t a = __byte_perm(__float_as_uint(s[0]), __float_as_uint(s[1]), 0x0040);
        const uint32_t b = __byte_perm(__float_as_uint(s[2]), __float_as_uint(s[3]), 0x0040);
        return __byte_perm(a, b, 0x5410);
    }

    __device__ __forceinline__ void store(uint16_t *rb, int px) const
    {
        const uint32_t a = __byte_perm(__float_as_uint(c[0]), __float_as_uint(c[1]), 0x5410);
        const uint32_t b = __byte_perm(__float_as_uint(c[2]), __float_as_uint(c[3]), 0x5410);
        uint4 w = wb;
        if (px == 0) {
            w.x = __byte_perm(a, w.x, 0x7610);
            w.y = __byte_perm(a, w.y, 0x7632);
            w.z = __byte_perm(b, w.z, 0x7610);
            w.w = __byte_perm(b, w.w, 0x7632);
        } else {
            w.x = __byte_perm(w.x, a, 0x5410);
            w.y = __byte_perm(w.y, a, 0x7610);
            w.z = __byte_perm(w.z, b, 0x5410);
            w.w = __byte_perm(w.w, b, 0x7610);
        }
        *reinterpret_cast<uint4 *>(rb) = w;
    }
};

template <typename T>
struct QuadOf;
template <>
struct QuadOf<uint8_t> {
    using type = Quad8;
};
template <>
struct QuadOf<uint16_t> {
    using type = Quad16;
};

// One work item: the lowering loop of Sec. 2.2 on its four points (while a
// point may be lowered, F(x) := alpha^-(x, F), its neighbours fixed; each step
// lands on another neighbour value, so at most eight succeed), the block
// written back if a point moved.  vm: 0x01 in the bytes of the points that
// exist, `in`: of those whose steps are added to nin.  Returns the bytes lowered.
//
// aff receives the neighbours to test again, bit d of byte k for direction d
// of point k.  The test of a neighbour q sees the point only through two bits:
// is it below F(q), and is it below F(q) - lambda.  The point went from c0 down
// to c1, and no neighbour lies strictly between two successive values of its
// loop (each step goes to the largest lower neighbour), so neither bit can
// change for a neighbour with F(q) <= c1 (the point stays >= F(q)), nor for one
// with F(q) > c0 + lambda (the point was already below F(q) - lambda).  The
// second bound is taken where R.cap is set: it costs another set of compares,
// which saves more tests than it costs in a batch but not in the wide mode's
// tail.  This holds in every mode, since the decision depends on the
// neighbour values through those two masks only.
template <typename T>
__device__ __forceinline__ uint32_t lower_item(const T *ra, T *rb, const T *rc, int px, uint32_t vm, uint32_t in,
                                               const PointRule &R, int &nin, uint32_t &aff)
{
    typename QuadOf<T>::type q;
    q.gather(ra, rb, rc, px);
    const auto c0 = q.centre();
    uint32_t moved = 0, count = 0;
#pragma unroll 1
    for (int it = 0; it < 9; ++it) {
        const uint32_t ok = q.decide(R, vm);
        if (!ok) break;
        q.lower(ok);
        moved |= ok;
        count += ok & in;  // per byte, at most eight
    }
    nin += int((count * kLsb8) >> 24);
    aff = 0;
    if (moved) {
        q.store(rb, px);
        aff = q.above(R, c0) & (moved * 0xffu);
    }
    return moved;
}

// One point on one lane: the same loop with the pixels as floats (either
// element size), for phases with too few work items to fill the warps with
// four points a lane.  A work item is then four lanes, and each of them issues
// about a quarter of the instructions (a chain of one warp runs at the rate it
// can issue: two cycles for each half-rate instruction).  ra, rb, rc point at
// the point's column in rows y - 1, y and y + 1.  Returns the number of steps;
// aff: the neighbours to test again, bit d for direction d.
template <typename T>
__device__ __forceinline__ int lower_one(const T *ra, T *rb, const T *rc, const PointRule &R, uint32_t &aff)
{
    constexpr uint32_t kBias = 0x4b000000u;  // 2^23
    const float n[8] = {__uint_as_float(kBias | rb[1]),  __uint_as_float(kBias | ra[1]),  __uint_as_float(kBias | ra[0]),
                        __uint_as_float(kBias | ra[-1]), __uint_as_float(kBias | rb[-1]), __uint_as_float(kBias | rc[-1]),
                        __uint_as_float(kBias | rc[0]),  __uint_as_float(kBias | rc[1])};
    const float c0 = __uint_as_float(kBias | rb[0]);
    float c = c0;
    constexpr float w[8] = {1, 3, 9, 27, 81, 243, 729, 2187};
    int steps = 0;
#pragma unroll 1
    for (; steps < 9; ++steps) {
        float s = __uint_as_float(kBias), t = 0.0f;
        const float cl = __fsub_rn(c, R.lamf);
        const uint32_t m = 0u - __float_as_uint(c);
        uint32_t best = 0;
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            s = __fmaf_rn(__saturatef(__fsub_rn(c, n[d])), w[d], s);
            t = __fmaf_rn(__saturatef(__fsub_rn(cl, n[d])), w[d], t);  // lambda = 0: all of them once more
        }
        const uint32_t e = lds_u8(R.tab + __float_as_uint(__fadd_rn(s, t)) - kBias);
#pragma unroll
        for (int d = 0; d < 8; ++d) best = __viaddmax_u32(__float_as_uint(n[d]), m, best);
        if (!((e >> R.mode) & 1u)) break;
        c = __uint_as_float(__float_as_uint(c) + best);
    }
    aff = 0;
    if (steps) {
        rb[0] = static_cast<T>(__float_as_uint(c));
        const float top = R.cap ? __fadd_rn(c0, R.lamf) : __uint_as_float(0x4b800000u);  // above every pixel
#pragma unroll
        for (int d = 0; d < 8; ++d) aff |= n[d] > c && n[d] <= top ? 1u << d : 0u;
    }
    return steps;
}

}  // namespace thin
