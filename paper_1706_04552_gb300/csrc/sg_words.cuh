// sg_words.cuh -- k B3/S23 steps of up to 32 64-tiles at once, one bit per
// tile: the core of the fused CA kernels (sg_fused.cu, sg_batch.cu).
//
// Layout.  Every non-empty 64-tile holds the same 729 gasket cells, so 32
// tiles are held as 729 words in shared memory, one word per cell, one bit
// per tile ("lane" t of the unit is bit t).  A step is then the same short
// sequence of bitwise adders on every word, and nothing is spent on the
// off-gasket 82 % of a tile.
//
// Triples.  A cell (x, y) is a gasket cell iff (x & y) == 0, so the cells come
// in threes A = (X, Y), B = (X+1, Y), C = (X, Y+1) with X, Y even and
// (X & Y) == 0: a tile is 243 triples, one per thread, whose states stay in
// the thread's registers for all k steps.  A triple's cells are neighbours of
// one another.  Outside, a triple -- and in the same way a tile, or any
// triangle of the gasket -- touches others only at its three corners, and at
// each corner at most one other:
//   corner A: the triangle to the left (its corner B), beside our A and C, or
//             the one above (its corner C), beside our A and B;
//   corner B: the triangle to the right (its A and C cells of the corner
//             triple), or the one above to the right (its corner C);
//   corner C: the triangle below (its A and B), or the one below to the left
//             (its corner B).
// So a step reads at most 5 words per triple and counts at most 5 neighbours
// per cell: 15 bitwise operations for the three cells of 32 tiles.
//
// Units.  The tiles of a unit are the 3^l 64-tiles (l <= 3) of one block of
// side 64 * 2^l, plus the three tiles that touch its corners (3^l + 3 <= 30
// bits), of which only the cells a 16-step light cone reaches are read.  Each
// step the warp that owns the corner triples of the tile passes the corner
// words between the bits: for each bit the source bit is known, so a word is
// one shift per lane and a ballot.
//
// Bound.  A step costs a unit about 320 warp instructions (12 per tile, against
// 128 for the dense bit rows, which also step a 16-cell halo all round), so a
// launch is bound by moving the tiles' sectors and by the chain of load, steps
// and store within a CTA (figures at the kernels).
#pragma once

#include "sg_stencil.cuh"
#include "sg_write_sector.cuh"

namespace sg {

constexpr int kWordThreads = 256;
constexpr int kWordCtas = 3;                    // resident per SM (80 registers a thread)
constexpr int kTriples = 243;
// Words per plane (A, B, C cells): 11 banks apart.  The threads of a warp read
// their corners in all three planes near their own index; with the planes 256
// words apart those reads met on the same banks.
constexpr int kPlane = 267;
constexpr int kWordZero = 3 * kPlane;           // a word that stays 0
constexpr int kWordBuf = 3 * kPlane + 8;
constexpr uint32_t kCornerB = 121, kCornerC = 242;   // digits all 1, all 2 (corner A is 0)

// The warp's index, by a shuffle: the compiler then knows it for uniform, and
// the branches on it around shuffles and ballots cost no reconvergence (16 steps
// at level 11, 7.6 us against 7.2).
__device__ __forceinline__ int uniform_warp()
{
    return __shfl_sync(~0u, (int)(threadIdx.x >> 5), 0);
}

// Index of the gasket cell (x, y) of a level-`levels` gasket: base-3 digit j
// is 0, 1 or 2 for the bits (x_j, y_j) = (0,0), (1,0), (0,1).
__host__ __device__ constexpr uint32_t gasket_digits(uint32_t x, uint32_t y, int levels)
{
    uint32_t d = 0;
    for (int j = levels - 1; j >= 0; --j) d = 3u * d + ((x >> j) & 1u) + 2u * ((y >> j) & 1u);
    return d;
}
__device__ __forceinline__ uint2 gasket_coords(uint32_t p, int levels)
{
    uint32_t x = 0, y = 0;
    for (int j = 0; j < levels; ++j) {
        const uint32_t q = p / 3u, d = p - 3u * q;
        x |= (d & 1u) << j;
        y |= (d >> 1) << j;
        p = q;
    }
    return make_uint2(x, y);
}

// The triangle touching corner C (0: A, 1: B, 2: C) of triangle (x, y) in an
// n x n arrangement: 0 if none, 1 for left / right / below, 2 for above /
// above to the right / below to the left.
template <int C>
__host__ __device__ constexpr uint32_t corner_neighbour(uint32_t x, uint32_t y, uint32_t n,
                                                        uint32_t &nx, uint32_t &ny)
{
    nx = x;
    ny = y;
    if (C == 0) {
        if (x > 0u && ((x - 1u) & y) == 0u) { nx = x - 1u; return 1u; }
        if (y > 0u && (x & (y - 1u)) == 0u) { ny = y - 1u; return 2u; }
    } else if (C == 1) {
        if (x + 1u >= n) return 0u;
        if (((x + 1u) & y) == 0u) { nx = x + 1u; return 1u; }
        if (y > 0u && ((x + 1u) & (y - 1u)) == 0u) { nx = x + 1u; ny = y - 1u; return 2u; }
    } else {
        if (y + 1u >= n) return 0u;
        if ((x & (y + 1u)) == 0u) { ny = y + 1u; return 1u; }
        if (x > 0u && ((x - 1u) & (y + 1u)) == 0u) { nx = x - 1u; ny = y + 1u; return 2u; }
    }
    return 0u;
}

// What a thread keeps about its triple: its index (its words are p, kPlane + p
// and 2 kPlane + p) and where the words at its corners sit.  One table entry
// per thread; the three corner triples of the tile are in the last warp.
struct TripleRefs {
    uint16_t p, rp, rq1, rq2, rr1, rr2;
    uint8_t side;                  // bit 0: rp is to the left, bit 1: above
    uint8_t px, py, pad;
};
struct TripleTable {
    TripleRefs t[kWordThreads];
};

constexpr TripleTable make_triple_table()
{
    TripleTable T{};
    for (uint32_t tid = 0; tid < (uint32_t)kWordThreads; ++tid) {
        TripleRefs &e = T.t[tid];
        const uint32_t p = tid == 0u ? 240u : tid == 240u ? 0u : tid == kCornerB ? 241u
                         : tid == 241u ? kCornerB : tid;
        e.p = (uint16_t)p;
        e.rp = e.rq1 = e.rq2 = e.rr1 = e.rr2 = (uint16_t)kWordZero;
        if (p >= (uint32_t)kTriples) continue;         // the last 13 threads: no triple
        uint32_t px = 0, py = 0, q = p;
        for (int j = 0; j < 5; ++j, q /= 3u) {
            px |= (q % 3u & 1u) << j;
            py |= (q % 3u >> 1) << j;
        }
        e.px = (uint8_t)px;
        e.py = (uint8_t)py;
        uint32_t nx = 0, ny = 0;
        const uint32_t ka = corner_neighbour<0>(px, py, 32u, nx, ny);
        const uint32_t ia = gasket_digits(nx, ny, 5);
        if (ka != 0u) e.rp = (uint16_t)((ka == 1u ? kPlane : 2 * kPlane) + ia);
        e.side = (uint8_t)ka;
        const uint32_t kb = corner_neighbour<1>(px, py, 32u, nx, ny);
        const uint32_t ib = gasket_digits(nx, ny, 5);
        if (kb == 1u) { e.rq1 = (uint16_t)ib; e.rq2 = (uint16_t)(2 * kPlane + ib); }
        if (kb == 2u) e.rq1 = (uint16_t)(2 * kPlane + ib);
        const uint32_t kc = corner_neighbour<2>(px, py, 32u, nx, ny);
        const uint32_t ic = gasket_digits(nx, ny, 5);
        if (kc == 1u) { e.rr1 = (uint16_t)ic; e.rr2 = (uint16_t)(kPlane + ic); }
        if (kc == 2u) e.rr1 = (uint16_t)(kPlane + ic);
    }
    return T;
}
__device__ const TripleTable kTripleTable = make_triple_table();

// What a lane keeps about its tile (the same in every warp).
struct WordLane {
    const uint8_t *in;      // the tile's first cell
    uint8_t *out;
    int r;                  // level of its grid
    uint32_t blocks;        // its 16 x 16 blocks to read (bit = block index, 9 blocks)
    uint32_t own;           // written back (a tile of the unit, not a halo tile)
    uint32_t x, y, nb;      // the tile among the nb x nb of its grid
    uint32_t ox, oy, l;     // the block of 2^l x 2^l tiles around it, and the
    uint32_t base;          //   lane of that block's first tile
};

// Blocks of a tile that lie in its grid (levels below 6 fill part of a tile).
__device__ __forceinline__ uint32_t tile_blocks(int r)
{
    return r >= 6 ? 0x1FFu : r == 5 ? 0x7u : 0x1u;
}

// Lanes of the unit (ux, uy) of a level-r grid (r >= 6 + l): 3^l tiles in digit order, then
// the tiles at its corners A, B, C.  Of a corner tile only the blocks a
// 16-step light cone reaches are read: the 16-block at the touching corner,
// and where that corner is an A, the block past its far end as well (its
// first cells are 16 steps from ours by the C or B cell).
__device__ __forceinline__ WordLane unit_lane(const uint8_t *in, uint8_t *out, int r, int l,
                                              uint32_t ux, uint32_t uy, uint32_t lane)
{
    const uint32_t nt = (uint32_t)pow3i(l), far = (1u << l) - 1u;
    WordLane w;
    w.r = r;
    w.nb = 1u << (r - 6);
    w.ox = ux << l;
    w.oy = uy << l;
    w.l = (uint32_t)l;
    w.base = 0u;
    w.own = lane < nt;
    w.blocks = 0u;
    w.x = w.ox;
    w.y = w.oy;
    if (lane < nt) {
        const uint2 c = gasket_coords(lane, l);
        w.x += c.x;
        w.y += c.y;
        w.blocks = 0x1FFu;
    } else if (lane < nt + 3u) {
        uint32_t nx = 0, ny = 0, k = 0;
        if (lane == nt) {                      // its corner B, or its C
            k = corner_neighbour<0>(w.ox, w.oy, w.nb, nx, ny);
            w.blocks = k == 1u ? 1u << 4 : 1u << 8;
        } else if (lane == nt + 1u) {          // its corner A, or its C
            k = corner_neighbour<1>(w.ox + far, w.oy, w.nb, nx, ny);
            w.blocks = k == 1u ? (1u << 0) | (1u << 2) : 1u << 8;
        } else {                               // its corner A, or its B
            k = corner_neighbour<2>(w.ox, w.oy + far, w.nb, nx, ny);
            w.blocks = k == 1u ? (1u << 0) | (1u << 1) : 1u << 4;
        }
        if (k == 0u) w.blocks = 0u;
        w.x = nx;
        w.y = ny;
    }
    const uint64_t at = ((uint64_t)(w.y << 6) << r) + (w.x << 6);
    w.in = in + at;
    w.out = out + at;
    return w;
}

// Per corner of the lane's tile 8 bits: kind (2 bits, 0 none) << 5 | the lane
// of the tile it touches.  Warp-collective.
__device__ __forceinline__ uint32_t corner_links(const WordLane &w, int lane)
{
    const uint32_t side = 1u << w.l, nt = (uint32_t)pow3i((int)w.l);
    // the corner tiles of a unit follow its own (packed gaskets have none)
    const uint32_t h0 = min(nt, 29u), h1 = min(nt + 1u, 30u), h2 = min(nt + 2u, 31u);
    const uint32_t xy = (w.y << 16) | w.x;
    const uint32_t c0 = __shfl_sync(~0u, xy, h0), c1 = __shfl_sync(~0u, xy, h1);
    const uint32_t c2 = __shfl_sync(~0u, xy, h2);
    auto find = [&](uint32_t k, uint32_t nx, uint32_t ny) -> uint32_t {
        if (k == 0u || w.blocks == 0u) return 0u;
        const uint32_t dx = nx - w.ox, dy = ny - w.oy;       // wraps when outside
        if (dx < side && dy < side) return (k << 5) | (w.base + gasket_digits(dx, dy, (int)w.l));
        const uint32_t at = (ny << 16) | nx;
        return at == c0 ? (k << 5) | h0 : at == c1 ? (k << 5) | h1 : at == c2 ? (k << 5) | h2 : 0u;
    };
    uint32_t nx, ny;
    uint32_t k = corner_neighbour<0>(w.x, w.y, w.nb, nx, ny);
    uint32_t link = find(k, nx, ny);
    k = corner_neighbour<1>(w.x, w.y, w.nb, nx, ny);
    link |= find(k, nx, ny) << 8;
    k = corner_neighbour<2>(w.x, w.y, w.nb, nx, ny);
    link |= find(k, nx, ny) << 16;
    return link;
}

// ---------------------------------------------------------------------------
// Bytes <-> words.  A 16-block's rows come in groups of four, q = row / 4, and
// a group's gasket cells lie in some of its 4-cell nibbles only:
//   q = 0: all four nibbles of each row    (two words: rows 0, 1 and 2, 3)
//   q = 1: columns 0..3 and 8..11          (one word)
//   q = 2: columns 0..7                    (one word)
//   q = 3: columns 0..3                    (half a word; two blocks share one)
// A lane packs the nibbles of its own tile into such words (one multiply and
// one funnel shift each), and a 32 x 32 bit transpose across the warp turns
// "32 cells of my tile" into "my cell of 32 tiles".  The same in reverse on
// the way out.  A ballot per cell took twice the instructions and, being
// straight-line code that a launch fetches once, much longer (level 15, 2
// steps: 50.8 us against 38.6; level 6: 7.1 us against 4.6).
// ---------------------------------------------------------------------------

// Word (within a plane block) of bit position `pos` of word kind m (0, 1: q =
// 0; 2: q = 1; 3: q = 2; 4: q = 3, the upper half that of the next block);
// kNoWord where the position holds no gasket cell.
constexpr uint16_t kNoWord = 0xFFFFu;
struct ChunkTable {
    uint16_t at[5][32];
};
constexpr ChunkTable make_chunk_table()
{
    ChunkTable t{};
    for (int m = 0; m < 5; ++m)
        for (uint32_t pos = 0; pos < 32u; ++pos) {
            uint32_t row = 0, col = 0, next = 0;
            if (m < 2) { row = 2u * m + (pos >> 4); col = pos & 15u; }
            if (m == 2) { row = 4u + (pos >> 3); col = (pos & 3u) + ((pos & 4u) << 1); }
            if (m == 3) { row = 8u + (pos >> 3); col = pos & 7u; }
            if (m == 4) { row = 12u + ((pos >> 2) & 3u); col = pos & 3u; next = pos >> 4; }
            const uint32_t plane = (row & 1u) ? 2u : (col & 1u);
            t.at[m][pos] = (row & col) != 0u
                               ? kNoWord
                               : (uint16_t)(plane * kPlane + 27u * next +
                                            gasket_digits(col >> 1, row >> 1, 3));
        }
    return t;
}
__device__ const ChunkTable kChunkTable = make_chunk_table();

// 32 x 32 bit transpose across the warp: bit j of lane i <-> bit i of lane j.
struct Transpose {
    uint32_t sel16, sel8, r4, r2, r1, m4, m2, m1;
    __device__ __forceinline__ void init(int lane)
    {
        // a lane with bit j set keeps its upper halves and takes the other
        // lane's upper halves into its lower ones, and the reverse
        sel16 = (lane & 16) ? 0x3276u : 0x5410u;
        sel8 = (lane & 8) ? 0x3715u : 0x6240u;
        r4 = (lane & 4) ? 4u : 28u;
        r2 = (lane & 2) ? 2u : 30u;
        r1 = (lane & 1) ? 1u : 31u;
        m4 = (lane & 4) ? 0xF0F0F0F0u : 0x0F0F0F0Fu;
        m2 = (lane & 2) ? 0xCCCCCCCCu : 0x33333333u;
        m1 = (lane & 1) ? 0xAAAAAAAAu : 0x55555555u;
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const
    {
        uint32_t y = __shfl_xor_sync(~0u, x, 16);
        x = __byte_perm(x, y, sel16);
        y = __shfl_xor_sync(~0u, x, 8);
        x = __byte_perm(x, y, sel8);
        y = __shfl_xor_sync(~0u, x, 4);
        x = (x & m4) | (__funnelshift_r(y, y, r4) & ~m4);
        y = __shfl_xor_sync(~0u, x, 2);
        x = (x & m2) | (__funnelshift_r(y, y, r2) & ~m2);
        y = __shfl_xor_sync(~0u, x, 1);
        return (x & m1) | (__funnelshift_r(y, y, r1) & ~m1);
    }
};

// acc << 4 | the four 0/1 bytes of w as a nibble: the product has byte i's bit
// at bit 28 + i (and at distinct lower bits), so no carry disturbs it.
__device__ __forceinline__ uint32_t add_nibble(uint32_t acc, uint32_t w)
{
    return __funnelshift_l(w * 0x10204080u, acc, 4);
}
// Nibble i of b as four 0/1 bytes.
__device__ __forceinline__ uint32_t nibble_bytes(uint32_t b, int i)
{
    return (((b >> (4 * i)) & 0xFu) * 0x00204081u) & 0x01010101u;
}

// Nibbles of a row of group Q; nibble k is its 4-byte word word_of(k).
template <int Q> struct RowGroup {
    static constexpr int NIB = Q == 0 ? 4 : Q == 3 ? 1 : 2;
    __host__ __device__ static constexpr int word_of(int k) { return Q == 1 ? 2 * k : k; }
};

// The nibbles of one block's row group as 4-byte words in registers.
template <int Q>
__device__ __forceinline__ void load_rows(uint32_t (&v)[4][RowGroup<Q>::NIB], const uint8_t *p,
                                          int r, bool on)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint8_t *row = p + ((uint64_t)(4 * Q + i) << r);
#pragma unroll
        for (int k = 0; k < RowGroup<Q>::NIB; ++k) v[i][k] = 0u;
        if (!on) continue;
        if constexpr (Q == 0) {
            const uint4 c = __ldg(reinterpret_cast<const uint4 *>(row));
            v[i][0] = c.x; v[i][1] = c.y; v[i][2] = c.z; v[i][3] = c.w;
        } else if constexpr (Q == 1) {
            v[i][0] = __ldg(reinterpret_cast<const uint32_t *>(row));
            v[i][1] = __ldg(reinterpret_cast<const uint32_t *>(row + 8));
        } else if constexpr (Q == 2) {
            const uint2 c = __ldg(reinterpret_cast<const uint2 *>(row));
            v[i][0] = c.x; v[i][1] = c.y;
        } else {
            v[i][0] = __ldg(reinterpret_cast<const uint32_t *>(row));
        }
    }
}

// Rows first .. of a block's group packed: two rows of group 0, all four rows
// of the others (group 3: the low half).
template <int Q>
__device__ __forceinline__ uint32_t pack_rows(const uint32_t (&v)[4][RowGroup<Q>::NIB], int first)
{
    constexpr int ROWS = Q == 0 ? 2 : 4;
    uint32_t acc = 0u;
#pragma unroll
    for (int i = ROWS - 1; i >= 0; --i)
#pragma unroll
        for (int k = RowGroup<Q>::NIB - 1; k >= 0; --k) acc = add_nibble(acc, v[first + i][k]);
    return acc;
}

// Row group Q of 32-block u: the tiles' bytes -> words.
template <int Q>
__device__ __forceinline__ void group_to_words(uint32_t *s, const WordLane &w, uint32_t u,
                                               const Transpose &tr, int lane)
{
    const uint8_t *src = w.in + ((u == 2u ? 32ull << w.r : 0ull) + (u == 1u ? 32u : 0u));
    const uint32_t on = w.blocks >> (3u * u);
    uint32_t *b = s + 81u * u;
    if constexpr (Q == 0) {
        // two blocks in flight, then the third: 32 registers of loads, not 48
        const uint32_t a0 = kChunkTable.at[0][lane], a1 = kChunkTable.at[1][lane];
        auto words = [&](const uint32_t (&v)[4][4], int j) {
            const uint32_t x0 = tr(pack_rows<Q>(v, 0)), x1 = tr(pack_rows<Q>(v, 2));
            if (a0 != kNoWord) b[27 * j + a0] = x0;
            if (a1 != kNoWord) b[27 * j + a1] = x1;
        };
        uint32_t v[2][4][4];
        load_rows<Q>(v[0], src, w.r, on & 1u);
        load_rows<Q>(v[1], src + 16, w.r, on & 2u);
        words(v[0], 0);
        load_rows<Q>(v[0], src + (16ull << w.r), w.r, on & 4u);
        words(v[1], 1);
        words(v[0], 2);
        return;
    }
    uint32_t v[3][4][RowGroup<Q>::NIB];
    load_rows<Q>(v[0], src, w.r, on & 1u);
    load_rows<Q>(v[1], src + 16, w.r, on & 2u);
    load_rows<Q>(v[2], src + (16ull << w.r), w.r, on & 4u);
    if constexpr (Q < 3) {
        const uint32_t a = kChunkTable.at[Q + 1][lane];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const uint32_t x = tr(pack_rows<Q>(v[j], 0));
            if (a != kNoWord) b[27 * j + a] = x;
        }
    } else {
        const uint32_t a = kChunkTable.at[4][lane];
        const uint32_t x = tr(pack_rows<Q>(v[0], 0) | (pack_rows<Q>(v[1], 0) << 16));
        const uint32_t y = tr(pack_rows<Q>(v[2], 0));
        if (a != kNoWord) {
            b[a] = x;
            if (lane < 16) b[54 + a] = y;
        }
    }
}

// Row group Q of 32-block u: words -> the tiles' bytes.  Each row's sector is
// written whole (block 2's partner on the lower rows holds no gasket cell), so
// the L2 has nothing to fill.
template <int Q>
__device__ __forceinline__ void words_to_group(const uint32_t *s, const WordLane &w, uint32_t u,
                                               bool wide, const Transpose &tr, int lane)
{
    constexpr int NIB = RowGroup<Q>::NIB;
    const uint32_t *b = s + 81u * u;
    uint32_t x[3], y[3] = {0u, 0u, 0u};       // y: rows 2 and 3 of group 0
    if constexpr (Q == 3) {
        const uint32_t a = kChunkTable.at[4][lane];
        x[0] = tr(a != kNoWord ? b[a] : 0u);
        x[1] = x[0] >> 16;
        x[2] = tr(a != kNoWord && lane < 16 ? b[54 + a] : 0u);
    } else {
        const uint32_t a = kChunkTable.at[Q == 0 ? 0 : Q + 1][lane];
#pragma unroll
        for (int j = 0; j < 3; ++j) x[j] = tr(a != kNoWord ? b[27 * j + a] : 0u);
        if constexpr (Q == 0) {
            const uint32_t a1 = kChunkTable.at[1][lane];
#pragma unroll
            for (int j = 0; j < 3; ++j) y[j] = tr(a1 != kNoWord ? b[27 * j + a1] : 0u);
        }
    }
    if (!w.own || !((w.blocks >> (3u * u)) & 1u)) return;
    uint8_t *p = w.out + ((u == 2u ? 32ull << w.r : 0ull) + (u == 1u ? 32u : 0u)) +
                 ((uint64_t)(4 * Q) << w.r);
#pragma unroll 1
    for (int i = 0; i < 4; ++i, p += 1ull << w.r) {
        uint4 o[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            uint32_t v[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int k = 0; k < NIB; ++k) v[RowGroup<Q>::word_of(k)] = nibble_bytes(x[j], k);
            o[j] = make_uint4(v[0], v[1], v[2], v[3]);
            x[j] >>= 4 * NIB;
            if (Q == 0 && i == 1) x[j] = y[j];
        }
        uint8_t *q = p + (16ull << w.r);
        if (wide) {
            const uint32_t hi[8] = {o[0].x, o[0].y, o[0].z, o[0].w, o[1].x, o[1].y, o[1].z, o[1].w};
            const uint32_t lo[8] = {o[2].x, o[2].y, o[2].z, o[2].w, 0u, 0u, 0u, 0u};
            st_global_v8(p, hi);
            st_global_v8(q, lo);
        } else {
            *reinterpret_cast<uint4 *>(p) = o[0];
            if (w.r > 4) {
                *reinterpret_cast<uint4 *>(p + 16) = o[1];
                *reinterpret_cast<uint4 *>(q) = o[2];
                *reinterpret_cast<uint4 *>(q + 16) = make_uint4(0u, 0u, 0u, 0u);
            }
        }
    }
}

// The 12 (row group, 32-block) pieces over the eight warps, by their words:
// group 0 has 6, groups 1 and 2 have 3, group 3 has 2.
#define SG_WORD_PIECES(F)                                                        \
    do {                                                                         \
        const int warp_ = uniform_warp();                                        \
        if (warp_ < 3) {                                                         \
            F(0, (uint32_t)warp_);                                               \
        } else if (warp_ < 6) {                                                  \
            F(1, (uint32_t)warp_ - 3u);                                          \
            F(3, (uint32_t)warp_ - 3u);                                          \
        } else {                                                                 \
            _Pragma("unroll 1") for (uint32_t u_ = warp_ == 6 ? 0u : 2u;         \
                                     u_ < (warp_ == 6 ? 2u : 3u); ++u_)          \
                F(2, u_);                                                        \
        }                                                                        \
    } while (0)

__device__ __forceinline__ uint32_t maj3w(uint32_t a, uint32_t b, uint32_t c)
{
    return (a & b) | (c & (a ^ b));
}

// k steps on the words in st[k & 1], written by the CTA's warps just before
// (the call begins with a barrier); the result is in st[0], behind a barrier.
// Every thread of the CTA (kWordThreads) calls it with its lane's tile.  st:
// two buffers whose words kWordZero are 0.  kk: this lane's step count, k the
// largest; mixed: some lane's count differs or some lane's grid fills only
// part of its tile (its other cells stay 0).
__device__ __forceinline__ void words_steps(uint32_t (&st)[2][kWordBuf], const WordLane &w,
                                            const TripleRefs &t, int kk, int k, bool mixed)
{
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    // the last warp's lanes pass the corner words between the bits: the bit
    // they take from a corner's B or C cell, or A cell, and their own kinds
    uint32_t fa1 = 0u, fa2 = 0u, fb1 = 0u, fb2 = 0u, fc1 = 0u, fc2 = 0u, ml = 0u, mu = 0u;
    if (warp == kWordThreads / 32 - 1) {
        const uint32_t link = corner_links(w, lane);
        const uint32_t ka = (link >> 5) & 3u, kb = (link >> 13) & 3u, kc = (link >> 21) & 3u;
        fa1 = ka == 1u ? 1u << (link & 31u) : 0u;
        fa2 = ka == 2u ? 1u << (link & 31u) : 0u;
        fb1 = kb == 1u ? 1u << ((link >> 8) & 31u) : 0u;
        fb2 = kb == 2u ? 1u << ((link >> 8) & 31u) : 0u;
        fc1 = kc == 1u ? 1u << ((link >> 16) & 31u) : 0u;
        fc2 = kc == 2u ? 1u << ((link >> 16) & 31u) : 0u;
        ml = __ballot_sync(~0u, ka == 1u);
        mu = __ballot_sync(~0u, ka == 2u);
    }
    uint32_t part = 0u;
    if (mixed) {
        const uint32_t m4 = __ballot_sync(~0u, w.r == 4), m5 = __ballot_sync(~0u, w.r == 5);
        part = (max(t.px, t.py) >= 8u ? m4 : 0u) | (max(t.px, t.py) >= 16u ? m5 : 0u);
    }
    const uint32_t left = (t.side & 1u) ? ~0u : 0u, up = (t.side & 2u) ? ~0u : 0u;
    __syncthreads();
    uint32_t a = 0u, b = 0u, c = 0u;
    if (t.p < kTriples) {
        a = st[k & 1][t.p];
        b = st[k & 1][kPlane + t.p];
        c = st[k & 1][2 * kPlane + t.p];
    }
    auto step = [&](const uint32_t *cur, uint32_t *nxt, int s) {
        uint32_t P = cur[t.rp], q1 = cur[t.rq1], q2 = cur[t.rq2], r1 = cur[t.rr1], r2 = cur[t.rr2];
        uint32_t pl = P & left, pu = P & up;
        if (warp == kWordThreads / 32 - 1) {
            const uint32_t wa = cur[0], wab = cur[kPlane], wac = cur[2 * kPlane];
            const uint32_t wb = cur[kPlane + kCornerB], wc = cur[2 * kPlane + kCornerC];
            const uint32_t xp = __ballot_sync(~0u, ((wb & fa1) | (wc & fa2)) != 0u);
            const uint32_t x1 = __ballot_sync(~0u, ((wa & fb1) | (wc & fb2)) != 0u);
            const uint32_t x2 = __ballot_sync(~0u, (wac & fb1) != 0u);
            const uint32_t y1 = __ballot_sync(~0u, ((wa & fc1) | (wb & fc2)) != 0u);
            const uint32_t y2 = __ballot_sync(~0u, (wab & fc1) != 0u);
            if (t.p == 0u) { P = xp; pl = xp & ml; pu = xp & mu; }
            if (t.p == kCornerB) { q1 = x1; q2 = x2; }
            if (t.p == kCornerC) { r1 = y1; r2 = y2; }
        }
        // alive next iff 3 neighbours, or 2 and alive.  A has at most three
        // neighbours (B, C and P); B and C at most five: two full adders, and
        // the count is 2 or 3 iff exactly one of their carries is set
        const uint32_t na = maj3w(b, c, P) & ((b ^ c ^ P) | a);
        const uint32_t s1 = a ^ c ^ pu, c1 = maj3w(a, c, pu);
        const uint32_t nb = ((s1 ^ q1 ^ q2) | b) & (c1 ^ maj3w(s1, q1, q2));
        const uint32_t s2 = a ^ b ^ pl, c2 = maj3w(a, b, pl);
        const uint32_t nc = ((s2 ^ r1 ^ r2) | c) & (c2 ^ maj3w(s2, r1, r2));
        if (mixed) {
            const uint32_t act = __ballot_sync(~0u, s < kk) & ~part;
            a = (na & act) | (a & ~act);
            b = (nb & act) | (b & ~act);
            c = (nc & act) | (c & ~act);
        } else {
            a = na;
            b = nb;
            c = nc;
        }
        nxt[t.p] = a;
        nxt[kPlane + t.p] = b;
        nxt[2 * kPlane + t.p] = c;
        __syncthreads();
    };
    // two steps a round (the buffers' addresses are then constants); an odd
    // count starts in the second buffer, so the last step ends in the first
#pragma unroll 1
    for (int s = -(k & 1); s < k; s += 2) {
        if (s >= 0) step(st[0], st[1], s);
        step(st[1], st[0], s + 1);
    }
}

// k steps of a unit of embedded tiles: rows to words, steps, words to rows.
__device__ __forceinline__ void words_unit_steps(uint32_t (&st)[2][kWordBuf], const WordLane &w,
                                                 const TripleRefs &t, int kk, int k, bool mixed)
{
    const int lane = threadIdx.x & 31;
    Transpose tr;
    tr.init(lane);
#define CALL(Q, U) group_to_words<Q>(st[k & 1], w, U, tr, lane)
    SG_WORD_PIECES(CALL);
#undef CALL
    words_steps(st, w, t, kk, k, mixed);
    // 32-byte stores where every tile's address allows them (16-byte ones halve
    // the sectors a request carries: 38.7 against 42.8 us at level 15, k = 2)
    const bool wide = __all_sync(~0u, !w.own || (w.r > 4 && ((uintptr_t)w.out & 31u) == 0u));
    tr.init(lane);
#define CALL(Q, U) words_to_group<Q>(st[0], w, U, wide, tr, lane)
    SG_WORD_PIECES(CALL);
#undef CALL
    __syncthreads();                     // the words are read before the next unit's are written
}

}  // namespace sg
