// sg_compact_fused.cu -- B3/S23 steps on a compact array of 64-tiles (layout in
// sg_compact.cuh), k <= SG_FUSE_MAX per launch, on words of 32 tiles.
//
// The steps are those of sg_words.cuh: a unit is up to 27 64-tiles of one block
// and the three tiles at its corners, one bit per tile, whatever order the
// tiles have in memory (lambda_index gives each lane its tile's place).  What
// differs is the way in and out.  A tile is a run of 729 bytes at any byte
// address; lane t reads its own tile's run in aligned 16-byte pieces, packs
// each to 16 bits, shifts the bits to the run's start, and a 32 x 32 bit
// transpose across the warp turns "32 cells of my tile" into "my cell of 32
// tiles".  On the way out the bits are shifted to the alignment of the output
// run, and only its first and last pieces, shared with the neighbouring runs,
// are stored byte by byte.
//
// Bound: latency and issue, half and half (14.3 MB read and written at level 15).
// Level 15, 16 steps, dense rows of bits with a 16-cell halo and here: over several
// inputs in turn 183.4 and 20.3 us, one input again and again (the state stays in
// the L2) 180.0 and 18.1; level 10, 26.4 and 8.6.
#include "sg_compact.cuh"
#include "sg_words.cuh"

namespace sg {

namespace {

// Word of the e-th element of a 64-tile's run of 729; the positions past the
// last cell have none.  Tile side 64: rows top to bottom, each left to right.
// Tile sides 16 and 32 in the interleaved order: the 64-tile is a run of 9 or 3
// whole tiles, in the order of their digits (finest first: 0 the lower, 1 the
// upper left, 2 the right third).
struct CellTable {
    uint16_t at[736];
};
constexpr CellTable make_cell_table(int s)
{
    CellTable t{};
    const uint32_t rho = 1u << s;
    int e = 0;
    for (uint32_t q = 0; q < (uint32_t)pow3i(6 - s); ++q) {
        uint32_t x0 = 0, y0 = 0, v = q;
        for (int j = s; j < 6; ++j, v /= 3u) {
            x0 |= (v % 3u == 2u ? 1u : 0u) << j;
            y0 |= (v % 3u == 0u ? 1u : 0u) << j;
        }
        for (uint32_t y = y0; y < y0 + rho; ++y)
            for (uint32_t x = x0; x < x0 + rho; ++x)
                if ((x & y) == 0u)
                    t.at[e++] = (uint16_t)(((y & 1u) ? 2u : (x & 1u)) * kPlane +
                                           gasket_digits(x >> 1, y >> 1, 5));
    }
    for (; e < 736; ++e) t.at[e] = kNoWord;
    return t;
}
__device__ const CellTable kCellTables[3] = {make_cell_table(4), make_cell_table(5),
                                             make_cell_table(6)};

__device__ __forceinline__ uint32_t piece_bits(uint4 c)
{
    return add_nibble(add_nibble(add_nibble(add_nibble(0u, c.w), c.z), c.y), c.x);
}

// 16 bytes at p as 16 bits where some lie outside [lo, hi), the whole array:
// those are not read and give 0.
__device__ __noinline__ uint32_t edge_piece_bits(const uint8_t *p, const uint8_t *lo,
                                                 const uint8_t *hi)
{
    uint32_t v = 0u;
#pragma unroll
    for (int i = 0; i < 16; ++i) {         // (unrolled: one memory latency, not sixteen)
        const uint32_t b = p + i >= lo && p + i < hi ? __ldg(p + i) : 0u;
        v |= (b & 1u) << i;
    }
    return v;
}

// Cells 96 W .. 96 W + 95 of every lane's tile -> words (warp W).
__device__ __forceinline__ void run_to_words(uint32_t *s, const uint8_t *run, bool on,
                                             const uint8_t *lo, const uint8_t *hi,
                                             const Transpose &tr, const CellTable &ct, int warp,
                                             int lane)
{
    const uint32_t off = (uint32_t)((uintptr_t)run & 15u);
    const uint8_t *p = run - off + 96 * warp;
    const int last = (int)off + kUnit - 96 * warp;    // the run ends here (bytes from p)
    uint32_t b[4] = {0u, 0u, 0u, 0u};                 // 7 pieces: 112 bits from the aligned start
    // all pieces in the array (every unit but the one with its first or last
    // tile): the loads go out together
    if (__all_sync(~0u, !on || (run - off >= lo && run - off + 752 <= hi))) {
        uint4 c[7];
#pragma unroll
        for (int i = 0; i < 7; ++i) {
            c[i] = make_uint4(0u, 0u, 0u, 0u);
            if (on && 16 * i < last) c[i] = __ldg(reinterpret_cast<const uint4 *>(p + 16 * i));
        }
#pragma unroll
        for (int i = 0; i < 7; ++i) b[i >> 1] |= piece_bits(c[i]) << (16 * (i & 1));
    } else {
#pragma unroll
        for (int i = 0; i < 7; ++i)
            if (on && 16 * i < last) {
                const uint8_t *q = p + 16 * i;
                const uint32_t v = q >= lo && q + 16 <= hi
                                       ? piece_bits(__ldg(reinterpret_cast<const uint4 *>(q)))
                                       : edge_piece_bits(q, lo, hi);
                b[i >> 1] |= v << (16 * (i & 1));
            }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int g = 3 * warp + i;
        if (g > 22) break;
        const uint32_t x = tr(__funnelshift_r(b[i], b[i + 1], off));
        const uint32_t a = ct.at[32 * g + lane];
        if (a != kNoWord) s[a] = x;
    }
}

// The pieces 6 W .. 6 W + 5 of every own tile's output run.
__device__ __forceinline__ void words_to_run(const uint32_t *s, uint8_t *run, bool own,
                                             const Transpose &tr, const CellTable &ct, int warp,
                                             int lane)
{
    uint32_t g[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int e = 96 * warp - 32 + 32 * i + lane;
        const uint32_t a = e >= 0 && e < 736 ? ct.at[e] : kNoWord;
        g[i] = tr(a != kNoWord ? s[a] : 0u);
    }
    if (!own) return;
    const uint32_t off = (uint32_t)((uintptr_t)run & 15u);
    uint8_t *p = run - off + 96 * warp;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        uint32_t v = __funnelshift_l(g[i], g[i + 1], off);
#pragma unroll
        for (int h = 0; h < 2; ++h, v >>= 16) {
            const int e = 96 * warp + 32 * i + 16 * h - (int)off;      // first cell of the piece
            uint8_t *q = p + 32 * i + 16 * h;
            if (e >= 0 && e + 16 <= kUnit) {
                *reinterpret_cast<uint4 *>(q) = make_uint4(nibble_bytes(v, 0), nibble_bytes(v, 1),
                                                           nibble_bytes(v, 2), nibble_bytes(v, 3));
            } else {
#pragma unroll 4
                for (int j = 0; j < 16; ++j)
                    if (e + j >= 0 && e + j < kUnit) q[j] = (uint8_t)((v >> j) & 1u);
            }
        }
    }
}

// Where the tiles across the corners of unit q lie, as launch indices of the
// interleaved order (digits finest first: 0 the lower, 1 the upper left, 2 the
// right third).  At corner A, B, C (digit at = 1, 2, 0) the unit's finest digits
// that equal `at` are skipped; if the next one is d, the triangle across is the
// one with d replaced by `at` and the finer digits, down to the tiles, by d.
// ~0u: none.
__device__ __forceinline__ uint32_t corner_tile_index(uint32_t q, uint32_t at, int rbu, int l)
{
    uint32_t pw = 1u, rest = q, d = at;
    int j = 0;
    for (; j < rbu; ++j, pw *= 3u) {
        const uint32_t n = rest / 3u;
        d = rest - 3u * n;
        rest = n;
        if (d != at) break;
    }
    if (j == rbu) return ~0u;
    const uint32_t per = (uint32_t)pow3i(l);
    const uint32_t unit = q + (at - d) * (pw - (pw - 1u) / 2u);
    return unit * per + d * ((per - 1u) / 2u);
}

template <int CTAS>
__global__ void __launch_bounds__(kWordThreads, CTAS)
compact_words_kernel(const uint8_t *__restrict__ in, uint8_t *__restrict__ out, int r, int order,
                     int l, uint32_t units, uint32_t total, int k, int s)
{
    const CellTable &ct = kCellTables[s - 4];
    __shared__ uint32_t st[2][kWordBuf];
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    if (threadIdx.x < 16) st[threadIdx.x >> 3][kWordZero + (threadIdx.x & 7)] = 0u;
    const TripleRefs t = kTripleTable.t[threadIdx.x];
    Transpose tr;
    const int rbu = r - 6 - l;
    LambdaLane ll;
    ll.init(lane, rbu, order);
    const uint32_t W = pi_word(order, rbu);
    // the lane's tile within a unit: base-3 digits 0, 1, 2 of the lane (upper
    // left, right, lower) are the order's digits 1, 2, 0
    const uint32_t per = (uint32_t)pow3i(l);
    uint32_t within = 0u;
    {
        uint32_t v = (uint32_t)lane, pw = 1u;
        for (int j = 0; j < l; ++j, pw *= 3u, v /= 3u) within += (v % 3u + 1u) % 3u * pw;
    }
    const uint32_t corner = (uint32_t)lane - per;                 // lanes per .. per + 2
    const uint32_t at_digit = corner == 0u ? 1u : corner == 1u ? 2u : 0u;
    for (uint32_t q = blockIdx.x; q < units; q += gridDim.x) {
        const uint2 c = decode_tile<kMapLambda>(q, units, rbu, W, ll);
        const WordLane w = unit_lane(nullptr, nullptr, r, l, c.x, c.y, (uint32_t)lane);
        const bool on = w.blocks != 0u;
        uint32_t tile;
        if (order == kOrderInterleaved)
            tile = (uint32_t)lane < per ? q * per + within : corner_tile_index(q, at_digit, rbu, l);
        else
            tile = lambda_index(w.x, w.y, r - 6, order);
        const uint64_t at = (uint64_t)(on ? tile : 0u) * kUnit;
        tr.init(lane);
        run_to_words(st[k & 1], in + at, on, in, in + total, tr, ct, warp, lane);
        words_steps(st, w, t, k, k, false);
        tr.init(lane);
        words_to_run(st[0], out + at, w.own, tr, ct, warp, lane);
        __syncthreads();                 // the words are read before the next unit's are written
    }
}

}  // namespace

cudaError_t launch_compact_ca_words(int r, int s, int order, const uint8_t *in, uint8_t *out, int k,
                                    cudaStream_t st, const LaunchCfg &cfg)
{
    // unit depth as for the embedded kernel (one input again and again, 16 steps, 9
    // against 27 tiles: level 12, 8.5 and 9.3 us; level 13, 9.7 and 9.3; level 14,
    // 15.6 and 11.2)
    const int l = min(r >= 13 ? 3 : 2, r - 6);
    const uint32_t units = (uint32_t)pow3i(r - 6 - l);
    int err = 0;
    const int sms = sm_count(&err);
    if (err) return (cudaError_t)err;
    // Units for more than a round of three CTAs an SM: five (48 registers) keep
    // level 15 to one round (16 steps, 19.5 us against 23.1); below, more
    // registers are the shorter chain (level 10: 8.9 against 9.5).
    static std::atomic<int> occ3{0}, occ5{0};
    unsigned grid = 1;
    if (units > 3u * (uint32_t)sms) {
        auto k5 = compact_words_kernel<5>;
        cudaError_t e = persistent_grid(k5, kWordThreads, 0, units, cfg, &grid, &occ5);
        if (e != cudaSuccess) return e;
        k5<<<grid, kWordThreads, 0, st>>>(in, out, r, order, l, units, (uint32_t)pow3i(r), k, s);
    } else {
        auto k3 = compact_words_kernel<3>;
        cudaError_t e = persistent_grid(k3, kWordThreads, 0, units, cfg, &grid, &occ3);
        if (e != cudaSuccess) return e;
        k3<<<grid, kWordThreads, 0, st>>>(in, out, r, order, l, units, (uint32_t)pow3i(r), k, s);
    }
    return cudaGetLastError();
}

}  // namespace sg
