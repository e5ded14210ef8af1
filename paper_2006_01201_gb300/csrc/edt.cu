// edt.cu -- the global blending coefficient of Eq. (1) (Section III-C-2) on
// a labelled canvas of any shape, through an exact Euclidean distance
// transform.
//
// Eq. (1): Blend = 0 in Area1, 1 in Area2 and Lmin / (Lmin + Rmin) in
// Area3, where Lmin / Rmin are the distances from the pixel to the nearest
// Area1 / Area2 pixel (Euclidean, between pixel centres). Pixels in none of
// the areas get 0.5. A canvas without any Area1 pixel gives Blend = 1 in
// Area3 (the limit as Lmin grows without bound), without Area2 0, with
// neither 0.5.
//
// Distances are computed exactly, as integers, in two separable passes:
//   columns: g(x, y) = |y - y'| to the nearest feature pixel (x, y') of the
//            same column, or "none";
//   rows:    d2(x, y) = min over columns x' of (x - x')^2 + g(x', y)^2. The
//            leftmost column that attains the minimum never moves left as x
//            grows, so the columns of a few pixels bound those of the pixels
//            between them (edt_near_kernel). Canvases with a diagonal above
//            kNearMaxDiagonal, whose squared distances leave 32 bits, take the
//            lower envelope of one parabola per column instead
//            (edt_row.cuh: banded envelopes merged in a tree).
// Only the final ratio is rounded (FP32 square roots and one division).
#include <stdio.h>
#include <string.h>

#include <climits>
#include <type_traits>

#include "bounds.cuh"
#include "common.cuh"
#include "ctx.h"
#include "edt_row.cuh"
#include "pano_flow.h"

namespace pano {

namespace {

// ---------------------------------------------------------------------------
// Column pass. A CTA of 32 x 16 threads owns 32 columns and walks down them
// in blocks of 512 rows; thread (tx, ty) holds rows ty*32 .. ty*32+31 of a
// block of column tx as two 32-bit masks (Area1, Area2 pixels). A first pass
// over the labels finds, per column and block, the first feature row; a
// suffix minimum gives the first feature row at or after each block. The
// second pass finds the nearest features above and below the thread's rows
// from the masks of the other threads of its block (shared memory), the last
// feature row of the blocks above and the first of the blocks below, and counts
// the distance from row to row, down and up, both areas in the halves of a word.
// Where a warp's 32 columns can be read as aligned words, a lane reads eight
// rows of four columns, and the masks are put together by shuffles. The masks
// of the first kKeptBlocks blocks stay in shared memory between the two passes,
// so canvases of up to 4096 rows are read once.
// kPacked: g of both areas in one 32-bit element (Area1 low, Area2 high), one
// coalesced 4-byte store a pixel; otherwise a plane of 16-bit values each.
// 78 us on a 4000 x 9000 canvas (0.18 GB: 27 us at the memory's rate): 17 us
// without reads and distances, 14 for the reads, 20 for the distances and 26
// for the stores, one after the other in all CTAs. With a byte per load and a
// row number per area and pixel instead 99 us (67 M warp instructions, now
// 36 M). Without the barriers between the blocks of the second pass 82 us.
// kNearNone (packed) or edt::kNoSite where the column has no feature pixel. gp:
// elements per row.
// ---------------------------------------------------------------------------
// The row pass's 32-bit distances: the largest diagonal, and the g of a column
// without a site there.
constexpr int kNearMaxDiagonal = 46340;
constexpr unsigned kNearNone = kNearMaxDiagonal;

constexpr int kColW = 32;                     // columns per CTA
constexpr int kColTY = 16;                    // threads along y, 32 rows each
constexpr int kColBlock = 32 * kColTY;        // rows per block
constexpr int kMaxBlocks = (65535 + kColBlock - 1) / kColBlock;
constexpr int kKeptBlocks = 8;
constexpr int kAboveNone = -(1 << 20);        // y - kAboveNone > any distance
constexpr int kBelowNone = INT_MAX;

struct ColSmem {
    uint32_t mask[kKeptBlocks][2][kColTY][kColW];
    int next[2][kMaxBlocks + 1][kColW];       // first feature row at or after block rb's first row
    int above[2][kColW];                      // last feature row above the current block
    uint32_t some[kKeptBlocks][2][kColW];     // bit k: thread row k of the block has a feature pixel
};

// Bit 7 of every byte of c that equals k, shifted in from above: after eight
// rows a byte holds their bits in order.
__device__ __forceinline__ uint32_t shift_in_equal(uint32_t acc, uint32_t c, uint32_t k) {
    const uint32_t v = c ^ k * 0x01010101u, z = ~(((v & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | v) & 0x80808080u;
    return (acc >> 1 & 0x7F7F7F7Fu) | z;
}

// Masks of rows y0 .. y0 + 31 (< h) of column x, by a whole warp on columns
// x - lane .. x - lane + 31. words: these are all in the canvas and 4-byte
// aligned on every row; a lane then reads eight rows of four columns.
__device__ __forceinline__ void col_masks(const unsigned char* label, long long pitch, long long nl, int h, int w, int x,
                                          int y0, bool words, uint32_t* m1, uint32_t* m2) {
    const int n = min(32, h - y0), lane = threadIdx.x;
    uint32_t a = 0, b = 0;
    if (words) {
        const int yq = 8 * (lane >> 3);
        const long long o = (long long)(y0 + yq) * pitch + (x - lane) + 4 * (lane & 7);
        uint32_t qa = 0, qb = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t c = yq + i < n ? PANO_VEC(const uint32_t, label, o + i * pitch, 4, nl, 500) : 0u;
            qa = shift_in_equal(qa, c, 1);
            qb = shift_in_equal(qb, c, 2);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t va = __shfl_sync(0xffffffffu, qa, 8 * q + (lane >> 2));
            const uint32_t vb = __shfl_sync(0xffffffffu, qb, 8 * q + (lane >> 2));
            a |= (va >> 8 * (lane & 3) & 0xFFu) << 8 * q;
            b |= (vb >> 8 * (lane & 3) & 0xFFu) << 8 * q;
        }
    } else if (x < w) {
        const unsigned char* p = label + (long long)y0 * pitch + x;
#pragma unroll 8
        for (int i = 0; i < 32; ++i) {
            if (i < n) {
                const unsigned char c = PANO_AT(p, (long long)i * pitch, nl - ((long long)y0 * pitch + x), 501);
                a |= (uint32_t)(c == 1) << i;
                b |= (uint32_t)(c == 2) << i;
            }
        }
    }
    *m1 = a;
    *m2 = b;
}

template <bool kPacked>
__global__ void __launch_bounds__(kColW * kColTY, 2) edt_cols_kernel(const unsigned char* label, int h,
                                                                    int w, long long pitch, uint32_t* gb,
                                                                    uint16_t* g1,
                                                                    uint16_t* g2, int gp) {
    extern __shared__ __align__(16) unsigned char s_col[];
    grid_begin();
    ColSmem& S = *reinterpret_cast<ColSmem*>(s_col);
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kColW + tx;
    const int x = blockIdx.x * kColW + tx;
    const bool col_in = x < w;
    const bool words = (((uintptr_t)label | (uintptr_t)pitch) & 3) == 0 && (blockIdx.x + 1) * kColW <= w;
    const int nblk = (h + kColBlock - 1) / kColBlock;
    const long long nl = (long long)(h - 1) * pitch + w, ng = (long long)h * gp;  // label and g elements
    (void)nl;
    (void)ng;
    const int nn = 2 * (kMaxBlocks + 1) * kColW;
    for (int i = tid; i < nn; i += kColW * kColTY) PANO_AT(&S.next[0][0][0], i, nn, 502) = kBelowNone;
    if (tid < 2 * kColW) PANO_AT(&S.above[0][0], tid, 2 * kColW, 503) = kAboveNone;
    for (int i = tid; i < kKeptBlocks * 2 * kColW; i += kColW * kColTY) (&S.some[0][0][0])[i] = 0;
    __syncthreads();
    for (int rb = 0; rb < nblk; ++rb) {
        const int y0 = rb * kColBlock + ty * 32;
        uint32_t m1 = 0, m2 = 0;
        if (y0 < h) col_masks(label, pitch, nl, h, w, x, y0, words, &m1, &m2);
        if (m1) atomicMin(&S.next[0][rb][tx], y0 + __ffs(m1) - 1);
        if (m2) atomicMin(&S.next[1][rb][tx], y0 + __ffs(m2) - 1);
        if (rb < kKeptBlocks) {
            S.mask[rb][0][ty][tx] = m1, S.mask[rb][1][ty][tx] = m2;
            if (m1) atomicOr(&S.some[rb][0][tx], 1u << ty);
            if (m2) atomicOr(&S.some[rb][1][tx], 1u << ty);
        }
    }
    __syncthreads();
    if (ty < 2)
        for (int rb = nblk - 1; rb >= 0; --rb) S.next[ty][rb][tx] = min(S.next[ty][rb][tx], S.next[ty][rb + 1][tx]);
    __syncthreads();
    for (int rb = 0; rb < nblk; ++rb) {
        const int yb = rb * kColBlock, y0 = yb + ty * 32;
        const int slot = rb < kKeptBlocks ? rb : 0;
        uint32_t m[2] = {0, 0};
        if (rb < kKeptBlocks) {
            m[0] = S.mask[slot][0][ty][tx];
            m[1] = S.mask[slot][1][ty][tx];
        } else {
            if (y0 < h) col_masks(label, pitch, nl, h, w, x, y0, words, &m[0], &m[1]);
            if (tid < 2 * kColW) (&S.some[slot][0][0])[tid] = 0;
            S.mask[slot][0][ty][tx] = m[0];
            S.mask[slot][1][ty][tx] = m[1];
            __syncthreads();
            if (m[0]) atomicOr(&S.some[slot][0][tx], 1u << ty);
            if (m[1]) atomicOr(&S.some[slot][1][tx], 1u << ty);
            __syncthreads();
        }
        int above[2], below[2];  // nearest feature rows above and below this thread's 32 rows
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const uint32_t some = S.some[slot][a][tx], lo = some & ((1u << ty) - 1u), hi = some & ~((2u << ty) - 1u);
            int p = S.above[a][tx], n = S.next[a][rb + 1][tx];
            if (lo) {
                const int k = 31 - __clz(lo);
                p = yb + k * 32 + 31 - __clz(S.mask[slot][a][k][tx]);
            }
            if (hi) {
                const int k = __ffs(hi) - 1;
                n = yb + k * 32 + __ffs(S.mask[slot][a][k][tx]) - 1;
            }
            above[a] = p;
            below[a] = n;
        }
        if (col_in && y0 < h) {
            // Distances of both areas in the halves of a word, counted up from row
            // to row: nothing leaves 16 bits, kCap + 1 included.
            constexpr uint32_t kCap = kPacked ? kNearNone : edt::kNoSite - 1, kCap2 = kCap | kCap << 16;
            auto both = [](unsigned d1, unsigned d2) { return min(d1, kCap) | min(d2, kCap) << 16; };
            // a distance of 65534 is that of the last row of the highest canvas
            // from the first, so the columns without a site are set apart
            uint32_t none = 0;
            if (!kPacked) {
                if (!m[0] && above[0] == kAboveNone && below[0] == kBelowNone) none |= 0xFFFFu;
                if (!m[1] && above[1] == kAboveNone && below[1] == kBelowNone) none |= 0xFFFF0000u;
            }
            auto at = [](uint32_t bits, int i) { return (bits >> i & 0x00010001u) * 0xFFFFu; };  // 0xFFFF where a site lies
            const int n = min(32, h - y0);
#pragma unroll 1
            for (int i0 = 0; i0 < n; i0 += 16) {
                // 16 rows at a time (their distances upwards stay in registers)
                const uint32_t before[2] = {m[0] & ((1u << i0) - 1u), m[1] & ((1u << i0) - 1u)};
                const uint32_t after[2] = {i0 ? 0u : m[0] & 0xFFFF0000u, i0 ? 0u : m[1] & 0xFFFF0000u};
                const uint32_t bits = (m[0] >> i0 & 0xFFFFu) | m[1] >> i0 << 16;
                const int ya = y0 + i0 - 1, yb1 = y0 + i0 + 16;  // the rows before and after
                const int p1 = before[0] ? y0 + 31 - __clz(before[0]) : above[0], p2 = before[1] ? y0 + 31 - __clz(before[1]) : above[1];
                const int q1 = after[0] ? y0 + __ffs(after[0]) - 1 : below[0], q2 = after[1] ? y0 + __ffs(after[1]) - 1 : below[1];
                uint32_t d[16];  // distance to the last site above
                uint32_t v = both((unsigned)(ya - p1), (unsigned)(ya - p2));
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    v = __viaddmin_u16x2(v, 0x00010001u, kCap2) & ~at(bits, i);
                    d[i] = v;
                }
                // the sums stay below 2^31 with kBelowNone too
                v = both((unsigned)(q1 - yb1), (unsigned)(q2 - yb1));
                const long long o = (long long)(y0 + i0) * gp + x;
                auto up = [&](auto whole) {
#pragma unroll
                    for (int i = 15; i >= 0; --i) {
                        v = __viaddmin_u16x2(v, 0x00010001u, kCap2) & ~at(bits, i);
                        const uint32_t g = __vminu2(d[i], v) | none;
                        if (decltype(whole)::value || i0 + i < n) {
                            if constexpr (kPacked) {
                                PANO_AT(gb, o + i * gp, ng, 504) = g;
                            } else {
                                PANO_AT(g1, o + i * gp, ng, 504) = (uint16_t)(g & 0xFFFFu);
                                PANO_AT(g2, o + i * gp, ng, 504) = (uint16_t)(g >> 16);
                            }
                        }
                    }
                };
                if (i0 + 16 <= n) up(std::true_type{});
                else up(std::false_type{});
            }
        }
        __syncthreads();  // the masks and S.above are read
        if (ty == kColTY - 1) {
            S.above[0][tx] = m[0] ? y0 + 31 - __clz(m[0]) : above[0];
            S.above[1][tx] = m[1] ? y0 + 31 - __clz(m[1]) : above[1];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Row pass, diagonals up to kNearMaxDiagonal: one CTA per row, both areas. The row's
// columns are cut into groups of 64; only groups with an Area3 pixel matter.
//   1  g of both areas to shared memory, with the least g of every block of 32
//      columns; pixels of the other groups are written at once;
//   2  the nearest column (leftmost of equals) for the first pixel of every
//      group and the last pixel of every run of groups, by bisection over
//      these points: a warp searches between the columns of the two neighbours
//      already known. A long range is searched by blocks: the least g bounds every
//      distance to a block from both sides, and only the blocks whose lower
//      bound does not exceed the least upper bound are looked through;
//   3  a lane per two pixels: the least distance over the columns between those of
//      its group's point and of the next one, and Eq. (1). Where that range is
//      long (the nearest column jumps from one seam to another), the bisection
//      goes on over the group's lanes.
// Distances are 32-bit integers. In shared memory a column without a site has
// g = kNearNone, the largest diagonal: no pixel is that far from a site, and its
// square plus that of any distance within the row stays below 2^32.
// What bounds it: the instructions of steps 2 and 3 (177 M warp instructions on
// a 4000 x 9000 canvas, 65% of the issue rate); the g plane is read once.
// 224 us there, against 457 + 505 us of the envelopes' two launches; 254 us
// with points at first pixels only, whose ranges span the gaps between runs,
// and with a test for the missing site at every column. Groups of
// 32: 284 us; steps 2 and 3 alone without the bisection in step 3: a row whose
// overlaps lie far apart looks through the columns between them, 935 us.
// ---------------------------------------------------------------------------
constexpr int kNearThreads = 256;
constexpr int kNearWarps = kNearThreads / 32;
constexpr int kNearScan = 64;  // columns that a lane looks through one by one
constexpr int kNearFew = 4;    // a shorter range is left for step 3

struct NearSmem {
    int w4, nb, ng;  // columns rounded up to 4, blocks of 32 columns, groups of 64
    __host__ __device__ explicit NearSmem(int w) : w4((w + 3) / 4 * 4), nb((w + 31) / 32), ng((w + 63) / 64) {}
    __host__ __device__ size_t bytes() const { return 4 * ((size_t)w4 + nb) + 2 * 5 * ((size_t)ng + 2); }
};

__device__ __forceinline__ unsigned near_cost(unsigned g, int dx) { return (unsigned)dx * (unsigned)dx + g * g; }

// Leftmost nearest column of pixel x among [lo, hi], by one warp; some column
// of [lo, hi] is a nearest one of the whole row. gs and bm hold both areas'
// values, sh (0 or 16) selects the area.
__device__ __forceinline__ int near_search(const uint32_t* gs, const uint32_t* bm, int sh, int w,
                                           int nb, int x, int lo, int hi) {
    (void)w, (void)nb;
    const int lane = threadIdx.x & 31;
    constexpr unsigned kAll = 0xffffffffu;
    unsigned best = 0xFFFFFFFFu;
    int bq = hi;
    if (hi - lo < 128) {
        for (int q = lo + lane; q <= hi; q += 32) {
            const unsigned c = near_cost(PANO_AT(gs, q, w, 516) >> sh & 0xFFFFu, x - q);
            if (c < best) best = c, bq = q;
        }
        const unsigned m = __reduce_min_sync(kAll, best);
        return (int)__reduce_min_sync(kAll, best == m ? (unsigned)bq : 0xFFFFFFFFu);
    }
    const int b0 = lo >> 5, b1 = hi >> 5;
    unsigned ub = 0xFFFFFFFFu;
    for (int b = b0 + lane; b <= b1; b += 32) {
        const unsigned g = PANO_AT(bm, b, nb, 517) >> sh & 0xFFFFu;
        if (g != kNearNone) ub = min(ub, near_cost(g, max(abs(x - 32 * b), abs(x - 32 * b - 31))));
    }
    ub = __reduce_min_sync(kAll, ub);
    for (int base = b0; base <= b1; base += 32) {
        const int b = base + lane;
        unsigned lb = 0xFFFFFFFFu;
        if (b <= b1) {
            const unsigned g = PANO_AT(bm, b, nb, 518) >> sh & 0xFFFFu;
            if (g != kNearNone) lb = near_cost(g, max(0, max(32 * b - x, x - 32 * b - 31)));
        }
        unsigned todo = __ballot_sync(kAll, lb <= ub && lb != 0xFFFFFFFFu);
        while (todo) {
            const int k = __ffs(todo) - 1;
            const int q = 32 * (base + k) + lane;
            unsigned c = 0xFFFFFFFFu;
            if (q >= lo && q <= hi) c = near_cost(PANO_AT(gs, q, w, 519) >> sh & 0xFFFFu, x - q);
            const unsigned m = __reduce_min_sync(kAll, c);
            if (m < best) {
                best = m;
                bq = 32 * (base + k) + __ffs(__ballot_sync(kAll, c == m)) - 1;
                ub = min(ub, m);
            }
            todo &= __ballot_sync(kAll, lb <= ub && lb != 0xFFFFFFFFu) & ~((2u << k) - 1u);
        }
    }
    return bq;
}

__global__ void __launch_bounds__(kNearThreads) edt_near_kernel(const unsigned char* label, int h, int w,
                                                               long long pitch, const uint32_t* gb, int gp, float* blend,
                                                               int blend_pitch) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ int s_n;
    __shared__ unsigned s_any[2];
    grid_begin();
    const NearSmem L(w);
    const int w4 = L.w4, nb = L.nb, ng = L.ng;
    uint32_t* gs = reinterpret_cast<uint32_t*>(s_dyn);      // [w4] g of both areas
    uint32_t* bm = gs + w4;                                  // [nb] least g of a block, both areas
    uint16_t* ql = reinterpret_cast<uint16_t*>(bm + nb);     // [2][ng + 2] the nearest column of point i lies
    uint16_t* qh = ql + 2 * (ng + 2);                        // [2][ng + 2] between these two
    uint16_t* list = qh + 2 * (ng + 2);                      // [ng + 2] points: 2 group (+ 1 for a run's last pixel)
    uint16_t* flag = qh;                                     // [ng + 1] group with an Area3 pixel, before step 2
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, y = blockIdx.x;
    constexpr unsigned kAll = 0xffffffffu;
    const unsigned char* lab = label + (long long)y * pitch;
    float* out = blend + (long long)y * blend_pitch;

    // ---- 1: g, and the least g of each block (eight threads of four columns)
    if (tid < 2) s_any[tid] = 0;
    __syncthreads();
    {
        const uint32_t* row = gb + (long long)y * gp;
        const bool vec = (((uintptr_t)row) & 15) == 0;
        constexpr unsigned kNone2 = kNearNone | kNearNone << 16;
        unsigned all = kNone2;
        for (int v0 = 0; v0 < w4 / 4; v0 += kNearThreads) {
            const int v = v0 + tid;
            uint4 k = make_uint4(kNone2, kNone2, kNone2, kNone2);
            if (v < w4 / 4) {
                if (vec && 4 * v + 4 <= w) {
                    k = PANO_VEC(const uint4, row, 4 * v, 4, w, 505);
                } else {
                    uint32_t e[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) e[i] = 4 * v + i < w ? PANO_AT(row, 4 * v + i, w, 506) : kNone2;
                    k = make_uint4(e[0], e[1], e[2], e[3]);
                }
                PANO_VEC(uint4, gs, 4 * v, 4, w4, 507) = k;
            }
            unsigned m = __vminu2(__vminu2(k.x, k.y), __vminu2(k.z, k.w));
            m = __vminu2(m, __shfl_xor_sync(kAll, m, 1));
            m = __vminu2(m, __shfl_xor_sync(kAll, m, 2));
            m = __vminu2(m, __shfl_xor_sync(kAll, m, 4));
            if (v < w4 / 4 && (v & 7) == 0) PANO_AT(bm, v / 8, nb, 508) = m;
            all = __vminu2(all, m);
        }
        if ((all & 0xFFFFu) != kNearNone) s_any[0] = 1;
        if (all >> 16 != kNearNone) s_any[1] = 1;
    }
    // groups without an Area3 pixel are written now; the others are listed
    const bool lvec = (((uintptr_t)lab) & 3) == 0, ovec = (((uintptr_t)out) & 15) == 0;
    for (int x0 = 128 * wid; x0 < w; x0 += 128 * kNearWarps) {
        // two groups, four columns a lane
        const int x = x0 + 4 * lane;
        unsigned c = 0;
        if (lvec && x + 4 <= w) {
            c = PANO_VEC(const unsigned, lab, x, 4, w, 509);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (x + i < w) c |= (unsigned)PANO_AT(lab, x + i, w, 509) << (8 * i);
        }
        const unsigned three = __ballot_sync(kAll, __vcmpeq4(c, 0x03030303u) != 0u);
        const bool act = (lane < 16 ? three & 0xFFFFu : three >> 16) != 0u;
        if ((lane & 15) == 0 && x < w) PANO_AT(flag, x / 64, ng + 1, 510) = act;
        if (act || x >= w) continue;
        float b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned e = c >> (8 * i) & 0xFFu;
            b[i] = e == 1 ? 0.f : e == 2 ? 1.f : 0.5f;
        }
        if (ovec && x + 4 <= w) {
            PANO_VEC(float4, out, x, 4, w, 511) = make_float4(b[0], b[1], b[2], b[3]);
        } else {
            for (int i = 0; i < 4 && x + i < w; ++i) PANO_AT(out, x + i, w, 511) = b[i];
        }
    }
    if (tid == 0) flag[ng] = 0;
    __syncthreads();
    if (wid == 0) {
        // the points: the first pixel of every such group, the last one of every
        // run of neighbouring groups
        int n = 0;
        for (int g0 = 0; g0 < ng; g0 += 32) {
            const int g = g0 + lane;
            const bool act = g < ng && PANO_AT(flag, g, ng + 1, 512), end = act && !PANO_AT(flag, g + 1, ng + 1, 512);
            const unsigned ma = __ballot_sync(kAll, act), me = __ballot_sync(kAll, end), lt = (1u << lane) - 1u;
            const int o = n + __popc(ma & lt) + __popc(me & lt);
            if (act) PANO_AT(list, o, ng + 2, 512) = (uint16_t)(2 * g);
            if (end) PANO_AT(list, o + 1, ng + 2, 512) = (uint16_t)(2 * g + 1);
            n += __popc(ma) + __popc(me);
        }
        if (lane == 0) s_n = n;
    }
    __syncthreads();
    if (s_n == 0) return;
    const int n = s_n - 1;  // the last point
    const bool any0 = s_any[0] != 0, any1 = s_any[1] != 0;

    // ---- 2: nearest columns of points 0 .. n
    auto point_x = [&](int i) { return list[i] & 1 ? min(w - 1, 32 * (int)list[i] + 31) : 32 * (int)list[i]; };
    if (wid < 4) {
        const int a = wid & 1, i = wid < 2 ? 0 : n;
        const int q = (a ? any1 : any0) ? near_search(gs, bm, 16 * a, w, nb, point_x(i), 0, w - 1) : 0;
        if (lane == 0) PANO_AT(ql, a * (ng + 2) + i, 2 * (ng + 2), 513) = PANO_AT(qh, a * (ng + 2) + i, 2 * (ng + 2), 513) = (uint16_t)q;
    }
    __syncthreads();
    int s = 1;
    while (2 * s < n) s *= 2;
    for (; s >= 1; s >>= 1) {
        const int cnt = (n - 1 + s) / (2 * s);  // odd multiples of s below n
        // a lane per point and area; the warp searches the long ranges together
        for (int t0 = 0; t0 < 2 * cnt; t0 += kNearThreads) {
            const int t = t0 + wid + kNearWarps * lane;
            const int a = t & 1, i = s * (2 * (t >> 1) + 1), o = a * (ng + 2);
            int lo = 0, hi = 0;
            if (t < 2 * cnt) {
                lo = PANO_AT(ql, o + i - s, 2 * (ng + 2), 514);
                hi = PANO_AT(qh, o + min(i + s, n), 2 * (ng + 2), 515);
            }
            for (unsigned todo = __ballot_sync(kAll, hi - lo > kNearFew); todo; todo &= todo - 1) {
                const int k = __ffs(todo) - 1;
                const int l = __shfl_sync(kAll, lo, k), u = __shfl_sync(kAll, hi, k), j = __shfl_sync(kAll, i, k);
                const int q = near_search(gs, bm, 16 * __shfl_sync(kAll, a, k), w, nb, point_x(j), l, u);
                if (lane == k) lo = hi = q;
            }
            if (t < 2 * cnt) ql[o + i] = (uint16_t)lo, qh[o + i] = (uint16_t)hi;
        }
        __syncthreads();
    }

    // ---- 3: distances and Eq. (1)
    for (int i = wid; i < n; i += kNearWarps) {
        if (list[i] & 1) continue;
        const int X = 32 * (int)list[i], x = X + 2 * lane;
        const unsigned c0 = x < w ? PANO_AT(lab, x, w, 548) : 0, c1 = x + 1 < w ? PANO_AT(lab, x + 1, w, 548) : 0;
        unsigned d0[2], d1[2];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            unsigned b0 = 0xFFFFFFFFu, b1 = 0xFFFFFFFFu;
            if (a ? any1 : any0) {
                int lo = ql[a * (ng + 2) + i], hi = qh[a * (ng + 2) + i + 1];
                if (hi - lo > kNearScan) {
                    // the nearest column jumps in this group: bisect on, over the
                    // lanes, where the range is long
                    for (int st = 16; st >= 1; st >>= 1)
                        for (int b = 0; b < 32; b += 2 * st) {
                            const int l = __shfl_sync(kAll, lo, b), u = __shfl_sync(kAll, hi, b), xm = X + 2 * (b + st);
                            if (u - l <= kNearScan || xm >= w) continue;
                            const int m = near_search(gs, bm, 16 * a, w, nb, xm, l, u);
                            if (lane >= b && lane < b + st) hi = m;
                            if (lane >= b + st && lane < b + 2 * st) lo = m;
                        }
                }
                const uint16_t* ga = reinterpret_cast<const uint16_t*>(gs) + a;
#pragma unroll 2
                for (int q = lo; q <= hi; ++q) {
                    const unsigned g = PANO_AT(ga, 2 * q, 2 * w - a, 546), g2 = g * g;
                    const unsigned dx = (unsigned)(x - q);
                    b0 = min(b0, g2 + dx * dx);
                    b1 = min(b1, g2 + (dx + 1) * (dx + 1));
                }
            }
            d0[a] = b0, d1[a] = b1;
        }
        auto eq1 = [&](unsigned c, unsigned e0, unsigned e1) {
            if (c != 3) return c == 1 ? 0.f : c == 2 ? 1.f : 0.5f;
            if (!any0 || !any1) return any1 ? 1.f : any0 ? 0.f : 0.5f;
            const float dl = sqrtf((float)e0), dr = sqrtf((float)e1);
            return dl / (dl + dr);
        };
        const float v0 = eq1(c0, d0[0], d0[1]), v1 = eq1(c1, d1[0], d1[1]);
        if (ovec && x + 2 <= w) {
            PANO_VEC(float2, out, x, 2, w, 547) = make_float2(v0, v1);
        } else {
            if (x < w) PANO_AT(out, x, w, 547) = v0;
            if (x + 1 < w) PANO_AT(out, x + 1, w, 547) = v1;
        }
    }
}

// ---------------------------------------------------------------------------
// Row pass of larger canvases: one CTA of kRowThreads per row and area, one band of
// ceil(w / kRowThreads) columns per thread (edt_row.cuh for the steps).
// The Area1 launch writes the distances to Area1 (FP32 square roots of the
// exact squared distances, +inf with no Area1 pixel on the canvas) of the
// Area3 pixels to a plane; the Area2 launch reads them there and writes
// Eq. (1).
// Shared memory, all dynamic (the kernel's limit is set to the device
// maximum): the row's g (2 B per column), the kept sites (2 B per column),
// five ints per band and 33 ints for the scans; five CTAs fit on an SM at
// 9000 columns.
// ---------------------------------------------------------------------------
constexpr int kRowThreads = 256;
constexpr int kRowWarps = kRowThreads / 32;
constexpr int kRowCtas = 5;

// inclusive prefix maximum over the threads of the block
__device__ __forceinline__ int block_prefix_max(int v, int* s_warp) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v = max(v, t);
    }
    if (lane == 31) s_warp[wid] = v;
    __syncthreads();
    if (wid == 0) {
        int t = lane < kRowWarps ? s_warp[lane] : INT_MIN;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t = max(t, u);
        }
        if (lane < kRowWarps) s_warp[lane] = t;
    }
    __syncthreads();
    if (wid > 0) v = max(v, s_warp[wid - 1]);
    __syncthreads();
    return v;
}

// inclusive suffix minimum over the threads of the block
__device__ __forceinline__ int block_suffix_min(int v, int* s_warp) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_down_sync(0xffffffffu, v, o);
        if (lane + o < 32) v = min(v, t);
    }
    if (lane == 0) s_warp[wid] = v;
    __syncthreads();
    if (wid == 0) {
        int t = lane < kRowWarps ? s_warp[lane] : INT_MAX;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_down_sync(0xffffffffu, t, o);
            if (lane + o < 32) t = min(t, u);
        }
        if (lane < kRowWarps) s_warp[lane] = t;
    }
    __syncthreads();
    if (wid + 1 < kRowWarps) v = min(v, s_warp[wid + 1]);
    __syncthreads();
    return v;
}

// kFinal false: Area1 (g = g1), writes dist1; true: Area2, writes Blend
template <bool kFinal>
__global__ void __launch_bounds__(kRowThreads, kRowCtas) edt_row_kernel(const unsigned char* __restrict__ label,
                                                                        int h, int w, long long pitch,
                                                                        const uint16_t* __restrict__ gplane,
                                                                        float* __restrict__ dist1,
                                                                        float* __restrict__ blend, int blend_pitch) {
    using namespace edt;
    constexpr int NB = kRowThreads;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    uint16_t* gs = reinterpret_cast<uint16_t*>(s_dyn);                  // [w]
    uint16_t* st = gs + w;                                              // [w]
    int* lo = reinterpret_cast<int*>(s_dyn + 4 * (size_t)w);            // [NB]
    int* hi = lo + NB;                                                  // [NB]
    int* gfirst = hi + NB;   // [NB] first band of a group; then the last band <= b with a site
    int* glast = gfirst + NB;  // [NB] last band of a group; then the first band >= b with a site
    int* zs = glast + NB;      // [NB] start of the region of band b's first site
    int* s_warp = zs + NB;     // [32] warp totals of the scans
    int* s_any = s_warp + 32;  // [1] the row has a site
    const int tid = threadIdx.x, y = blockIdx.x;
    const int bw = (w + NB - 1) / NB;
    const long long ng = (long long)h * w;
    (void)ng;
    for (int i = tid; i < w; i += NB) PANO_AT(gs, i, w, 505) = PANO_AT(gplane, (long long)y * w + i, ng, 506);
    __syncthreads();
    const int x0 = min(w, tid * bw), x1 = min(w, x0 + bw);
    {
        // step 0: the runs of equal g at the band's edges, against the
        // columns before and after them (found by scans over the bands)
        int ls, fe;
        band_run_edges(gs, w, x0, x1, &ls, &fe);
        const int ps = block_prefix_max(ls, s_warp);
        const int sf = block_suffix_min(fe, s_warp);
        zs[tid] = ps;
        glast[tid] = sf;
        __syncthreads();
        int L = -1, R = w;
        if (x0 < x1) {
            const int u = (x0 == 0 || gs[x0] != gs[x0 - 1]) ? x0 : (tid > 0 ? zs[tid - 1] : 0);
            const int v = (x1 == w || gs[x1 - 1] != gs[x1]) ? x1 - 1 : (tid + 1 < NB ? glast[tid + 1] : w - 1);
            L = u - 1;
            R = v + 1;
        }
        edge_runs_hidden(gs, st, w, x0, x1, L, R);
        __syncthreads();
        for (int q = x0; q < x1; ++q)
            if (st[q]) gs[q] = (uint16_t)kNoSite;
        __syncthreads();
    }
    {
        const int k = band_envelope(gs, st, w, x0, x1);
        PANO_AT(lo, tid, NB, 507) = x0;
        PANO_AT(hi, tid, NB, 507) = x0 + k;
        PANO_AT(gfirst, tid, NB, 507) = k ? tid : -1;
        PANO_AT(glast, tid, NB, 507) = k ? tid : -1;
    }
    __syncthreads();
    // merge tree: in the round of stride s, thread lg (a multiple of 2 s)
    // merges the groups lg and lg + s
    for (int s = 1; s < NB; s <<= 1) {
        const int lg = tid;
        if ((lg & (2 * s - 1)) == 0 && lg + s < NB) {
            const int lf = PANO_AT(gfirst, lg, NB, 508), ll = PANO_AT(glast, lg, NB, 508);
            const int rf = PANO_AT(gfirst, lg + s, NB, 508), rl = PANO_AT(glast, lg + s, NB, 508);
            if (rf >= 0) {
                if (lf < 0) {
                    gfirst[lg] = rf;
                } else {
                    const bool ok = merge_groups(gs, st, lo, hi, w, NB, lf, ll, rf, rl);
                    PANO_FLAG(!ok, 509);  // the merge reached its iteration limit
                    (void)ok;
                }
                glast[lg] = rl;
            }
        }
        __syncthreads();
    }
    if (tid == 0) s_any[0] = gfirst[0] >= 0;
    // the last band <= b and the first band >= b that keep a site
    {
        const bool kept = hi[tid] > lo[tid];
        const int pv = block_prefix_max(kept ? tid : -1, s_warp);
        const int nx = block_suffix_min(kept ? tid : NB, s_warp);
        gfirst[tid] = pv;
        glast[tid] = nx;
    }
    __syncthreads();
    if (hi[tid] > lo[tid]) {
        const int pb = tid > 0 ? gfirst[tid - 1] : -1;
        int z = -1;
        if (pb >= 0) {
            const int p = PANO_AT(st, hi[pb] - 1, w, 510), q = PANO_AT(st, lo[tid], w, 510);
            z = region_start(f_of(gs, w, p), p, f_of(gs, w, q), q, w);
        }
        zs[tid] = z;
    }
    __syncthreads();
    if (hi[tid] <= lo[tid]) {
        const int n = glast[tid];
        zs[tid] = n < NB ? PANO_AT(zs, n, NB, 511) : w;
    }
    __syncthreads();
    if (x0 >= x1) return;
    const bool any = s_any[0] != 0;
    Walker k = {0, 0, 0, 0, 0};
    if (any) k = walk_start(gs, st, lo, hi, zs, w, NB, x0);
    const long long ro = (long long)y * w;
    const unsigned char* lab = label + (long long)y * pitch;
    if constexpr (!kFinal) {
        // only Area3 pixels read the distances to Area1
        for (int x = x0; x < x1; ++x)
            if (PANO_AT(lab, x, w, 512) == 3)
                PANO_AT(dist1, ro + x, ng, 512) =
                    any ? sqrtf((float)walk_to(gs, st, lo, hi, glast, w, NB, x, &k)) : INFINITY;
    } else {
        float* out = blend + (long long)y * blend_pitch;
        for (int x = x0; x < x1; ++x) {
            const unsigned char c = PANO_AT(lab, x, w, 513);
            float b;
            if (c == 1) {
                b = 0.f;
            } else if (c == 2) {
                b = 1.f;
            } else if (c == 3) {
                const float dl = PANO_AT(dist1, ro + x, ng, 514);
                const float dr = any ? sqrtf((float)walk_to(gs, st, lo, hi, glast, w, NB, x, &k)) : INFINITY;
                const bool no1 = isinf(dl), no2 = !any;
                if (no1 && no2) b = 0.5f;
                else if (no1) b = 1.f;
                else if (no2) b = 0.f;
                else b = dl / (dl + dr);
            } else {
                b = 0.5f;
            }
            PANO_AT(out, x, w, 515) = b;
        }
    }
}

}  // namespace

PANO_BOUNDS_READER(bounds_read_edt)

size_t blend_coeff_scratch_bytes(int h, int w) {
    return (size_t)h * w * (2 * sizeof(uint16_t) + sizeof(float));  // g of both areas, distances to Area1
}

size_t blend_coeff_row_smem(int w) { return (size_t)4 * w + (size_t)(5 * kRowThreads + 33) * sizeof(int); }

cudaError_t blend_coeff_prepare(int max_smem_bytes) {
    cudaError_t e = cudaFuncSetAttribute(edt_near_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)NearSmem(kNearMaxDiagonal).bytes());
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(edt_cols_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ColSmem));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(edt_cols_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ColSmem));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(edt_row_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem_bytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(edt_row_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem_bytes);
}

cudaError_t launch_blend_coeff(const unsigned char* label, int h, int w, long long pitch, float* blend,
                               int blend_pitch, void* scratch, cudaStream_t s) {
    const bool near = (long long)h * h + (long long)w * w <= (long long)kNearMaxDiagonal * kNearMaxDiagonal;
    const dim3 grid((w + kColW - 1) / kColW), block(kColW, kColTY);
    cudaError_t e;
    if (near) {
        // rows of whole 16 bytes where the scratch (8 bytes a pixel) has the room for it
        const int gp = w >= 4 ? (w + 3) / 4 * 4 : w;
        uint32_t* gb = static_cast<uint32_t*>(scratch);
        e = launch_dependent(edt_cols_kernel<true>, grid, block, sizeof(ColSmem), s, 0, label, h, w, pitch, gb, (uint16_t*)nullptr,
                             (uint16_t*)nullptr, gp);
        if (e != cudaSuccess) return e;
        return launch_dependent(edt_near_kernel, dim3(h), dim3(kNearThreads), NearSmem(w).bytes(), s, 0, label, h, w, pitch,
                                (const uint32_t*)gb, gp, blend, blend_pitch);
    }
    uint16_t* g1 = static_cast<uint16_t*>(scratch);
    uint16_t* g2 = g1 + (size_t)h * w;
    edt_cols_kernel<false><<<grid, block, sizeof(ColSmem), s>>>(label, h, w, pitch, nullptr, g1, g2, w);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    float* dist1 = reinterpret_cast<float*>(g2 + (size_t)h * w);
    const size_t smem = blend_coeff_row_smem(w);
    edt_row_kernel<false><<<h, kRowThreads, smem, s>>>(label, h, w, pitch, g1, dist1, blend, blend_pitch);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    edt_row_kernel<true><<<h, kRowThreads, smem, s>>>(label, h, w, pitch, g2, dist1, blend, blend_pitch);
    return cudaGetLastError();
}

}  // namespace pano

using namespace pano;

extern "C" {

size_t pano_blend_coeff_scratch_bytes(int h, int w) {
    if (h < 1 || w < 1) return 0;
    return blend_coeff_scratch_bytes(h, w);
}

pano_status pano_blend_coeff(const unsigned char* label, int h, int w, size_t label_pitch, float* blend,
                             int blend_pitch, void* scratch, size_t scratch_bytes, void* cuda_stream) {
    if (!label || !blend || !scratch) return fail(PANO_ERR_INVALID_ARG, "label, blend or scratch is NULL");
    if (h < 1 || w < 1) return fail(PANO_ERR_INVALID_ARG, "canvas size %dx%d", h, w);
    if (h > 65535 || w > 65535)
        return fail(PANO_ERR_UNSUPPORTED, "canvas %dx%d: sides above 65535 (16-bit distances and columns)", h, w);
    if (label_pitch < (size_t)w) return fail(PANO_ERR_INVALID_ARG, "label_pitch %zu < w %d", label_pitch, w);
    if (blend_pitch < w) return fail(PANO_ERR_INVALID_ARG, "blend_pitch %d < w %d", blend_pitch, w);
    if (((uintptr_t)blend) % 4 || ((uintptr_t)scratch) % 4)
        return fail(PANO_ERR_INVALID_ARG, "blend or scratch not 4-byte aligned");
    const size_t need = blend_coeff_scratch_bytes(h, w);
    if (scratch_bytes < need) return fail(PANO_ERR_INVALID_ARG, "scratch of %zu bytes < %zu", scratch_bytes, need);
    if ((double)h * (double)w > (double)INT_MAX * 8.0) return fail(PANO_ERR_UNSUPPORTED, "canvas too large");
    const size_t bb = (size_t)h * blend_pitch * sizeof(float), lb = (size_t)h * label_pitch;
    if (overlaps(blend, bb, label, lb) || overlaps(scratch, need, label, lb) || overlaps(scratch, need, blend, bb))
        return fail(PANO_ERR_INVALID_ARG, "label, blend and scratch must not overlap");
    int max_smem = 0;
    pano_status st;
    if ((st = ensure_lk_ready(&max_smem)) != PANO_OK) return st;
    if (blend_coeff_row_smem(w) > (size_t)max_smem)
        return fail(PANO_ERR_UNSUPPORTED, "canvas width %d needs %zu bytes of shared memory per row (device: %d)", w,
                    blend_coeff_row_smem(w), max_smem);
    cudaError_t e = launch_blend_coeff(label, h, w, (long long)label_pitch, blend, blend_pitch, scratch,
                                       static_cast<cudaStream_t>(cuda_stream));
    return e == cudaSuccess ? PANO_OK : cuda_fail(e, "blend coefficient launch");
}

}  // extern "C"
