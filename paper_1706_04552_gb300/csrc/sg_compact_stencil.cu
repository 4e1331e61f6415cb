// sg_compact_stencil.cu -- the B3/S23 CA step and the diffusion step on
// compact arrays (layout in sg_compact.cuh).
//
// Diffusion at rho >= 16 runs on triples of cells, the CA at rho = 64 on rows of
// bits and, from level 14 on (rho 16, 32: in the interleaved order always), on
// words of 32 tiles (sg_compact_fused.cu); all below or there.  The rest runs the
// gather form:
//
// Each warp of a persistent grid takes units of 729 elements (G whole tiles)
// on its own, with a staging region of its own in shared memory:
//   1. it decodes the unit's tiles (lambda reduction of Theorem 1) and copies
//      the unit's values in (32 consecutive elements per load: whole
//      sectors);
//   2. it fetches each tile's halo: the 8 (CA) or 4 (diffusion) cells of
//      neighbouring tiles that touch it.  A neighbouring block exists when it
//      lies in the block grid and (bx & by) == 0; its launch index comes from
//      lambda_index, the inverse of the decode.  Missing neighbours read 0;
//   3. it updates the unit's elements from shared memory and stores them in
//      whole sectors.  Where each neighbour of position c sits among the
//      staged values is read from a per-CTA table expanded from the
//      compile-time tables, so a cell costs one table load and 8 (4) value
//      loads from shared memory.
// Warps never wait for one another after the table is built: the latency of
// one warp's loads is covered by the other warps of the SM.  Only gasket
// cells exist here: nothing is spent on the off-gasket 82 % of a 64-tile, and
// the state of a level-15 CA (14.3 MB) stays in L2.
//
// The CA on 64-tiles up to level 13 runs bit-sliced instead (compact_ca_bits_kernel
// below):
// the gather above spends 9 shared loads per cell and is bound by the L1 /
// shared-memory pipe, while rows of bits take the rule 64 cells at a time.
//
// The cell arithmetic is the embedded kernels' own (life rule on (count |
// self) == 3; diffusion through diffuse_update with the same grouping of the
// neighbour sum), so a compact step equals the embedded step cell for cell.
#include "sg_compact.cuh"
#include "sg_stencil.cuh"

namespace sg {

namespace {

// Staged values of a unit: its 729 elements, then G * H halo cells, then one
// zero that neighbours off the gasket point at.
template <int S, int H> struct UnitStage {
    static constexpr int G = CompactPattern<S>::G;
    static constexpr int HALO = kUnit, ZERO = kUnit + G * H, SIZE = ZERO + 1;
};

// Resolve a table entry (index in the tile / kHaloBit | h / kNoCell) of a
// cell of tile g into an index of the staged values.
template <int S, int H>
__device__ __forceinline__ uint32_t stage_slot(uint16_t v, int g)
{
    using U = UnitStage<S, H>;
    if (v == kNoCell) return (uint32_t)U::ZERO;
    if (v & kHaloBit) return (uint32_t)(U::HALO + g * H + (v & (kHaloBit - 1)));
    return (uint32_t)(g * CompactPattern<S>::C + v);
}

// The halo cell h of tile g: value of the neighbouring tile's cell, or 0
// (and *present = false) when that tile is outside the grid or empty.
template <typename T, int S>
__device__ __forceinline__ T halo_value(const T *__restrict__ in, uint2 b, int dbx, int dby,
                                        uint32_t rank, int rb, int order, bool *present)
{
    *present = false;
    if (b.x == 0xFFFFFFFFu) return T(0);
    const uint32_t nbx = b.x + (uint32_t)dbx, nby = b.y + (uint32_t)dby;   // wraps when < 0
    if ((nbx >> rb) != 0u || (nby >> rb) != 0u || (nbx & nby) != 0u) return T(0);
    *present = true;
    const uint64_t q = lambda_index(nbx, nby, rb, order);
    return in[q * (uint64_t)CompactPattern<S>::C + rank];
}

// Shared memory of a CTA: the unit table (per position, where its
// neighbours sit among the staged values), then one region per warp with the
// unit's tile coordinates, halo presence bytes and staged values.
template <typename T, int S, int H, int TABLE_BYTES> struct StencilSmem {
    static constexpr int G = CompactPattern<S>::G;
    using U = UnitStage<S, H>;
    static constexpr int COORD = 0, PRES = G * 8, VALS = ((G * 8 + G * 4) + 15) / 16 * 16;
    static constexpr int WARP = (VALS + U::SIZE * (int)sizeof(T) + 15) / 16 * 16;
    static constexpr int TABLE = TABLE_BYTES;
    static constexpr int BYTES = TABLE + kUnitWarps * WARP;
    static_assert(TABLE % 16 == 0 && WARP % 16 == 0 && VALS % 16 == 0 && PRES % 8 == 0,
                  "every region aligned for its widest element");
};

// Stage unit u into the warp's region: its values, then the halo cells of
// each of its tiles (with presence bytes when `pres` is given).  Called by
// all lanes of the warp; returns the number of elements in the unit.
template <typename T, int S, int H>
__device__ __forceinline__ uint32_t stage_unit(T *sv, uint2 *coord, uint8_t *pres,
                                               const T *__restrict__ in, uint32_t u,
                                               uint32_t total, uint32_t ntiles, uint32_t W,
                                               const LambdaLane &ll, const int8_t (*hl)[4],
                                               const uint16_t *hrank, int rb, int order)
{
    using U = UnitStage<S, H>;
    constexpr int G = U::G;
    const int lane = threadIdx.x & 31;
    decode_unit_tiles<G>(coord, u * G, ntiles, W, ll);
    const uint32_t base = u * kUnit;
    const uint32_t cnt = min((uint32_t)kUnit, total - base);
#pragma unroll 4
    for (uint32_t c = lane; c < cnt; c += 32) sv[c] = in[base + c];
    __syncwarp();                              // coord written by lane 0
    for (int h = lane; h < G * H; h += 32) {
        const int g = h / H, k = h - g * H;
        bool p;
        sv[U::HALO + h] = halo_value<T, S>(in, coord[g], hl[k][0], hl[k][1], hrank[k], rb, order,
                                           &p);
        if (pres) pres[h] = p ? 1 : 0;
    }
    if (lane == 0) sv[U::ZERO] = T(0);
    __syncwarp();
    return cnt;
}

// Six CTAs an SM, 40 registers: left alone the compiler takes 40 or 32 (and the
// serial loads that go with 32) as the rest of the file changes.  us at 40 and
// 32: rho 32, row-major, level 15, 37.5 and 39.1; rho 4, level 10, 23.0 and 23.9;
// rho 16, row-major, level 15, 48.1 and 50.9 (level 16, 139.7 and 136.9).
template <int S>
__global__ void __launch_bounds__(kUnitThreads, 6)
compact_ca_kernel(const uint8_t *__restrict__ in, uint8_t *__restrict__ out, int r, int order,
                  uint32_t total)
{
    using M = StencilSmem<uint8_t, S, kCaHalo, kUnit * 16>;
    extern __shared__ __align__(16) unsigned char smem[];
    const CompactPattern<S> &pat = compact_pattern<S>();
    // per position: the staged-value index of each of its 8 neighbours
    uint4 *nbt = reinterpret_cast<uint4 *>(smem);
    for (int c = threadIdx.x; c < kUnit; c += kUnitThreads) {
        const int g = c / CompactPattern<S>::C, e = c - g * CompactPattern<S>::C;
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            w[k] = stage_slot<S, kCaHalo>(pat.ca_nb[e][2 * k], g) |
                   (stage_slot<S, kCaHalo>(pat.ca_nb[e][2 * k + 1], g) << 16);
        nbt[c] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *region = smem + M::TABLE + warp * M::WARP;
    uint2 *coord = reinterpret_cast<uint2 *>(region + M::COORD);
    uint8_t *sv = region + M::VALS;
    const int rb = r - S;
    const uint32_t ntiles = total / CompactPattern<S>::C, units = (total + kUnit - 1) / kUnit;
    LambdaLane ll;
    ll.init(lane, rb, order);
    const uint32_t W = pi_word(order, rb);
    const uint32_t nwarps = gridDim.x * kUnitWarps;
    for (uint32_t u = blockIdx.x * kUnitWarps + warp; u < units; u += nwarps) {
        __syncwarp();                          // the previous unit is finished
        const uint32_t cnt = stage_unit<uint8_t, S, kCaHalo>(
            sv, coord, nullptr, in, u, total, ntiles, W, ll, pat.ca_halo, pat.ca_halo_rank, rb,
            order);
        uint8_t *o = out + u * kUnit;
#pragma unroll 4
        for (uint32_t c = lane; c < cnt; c += 32) {
            const uint4 t = nbt[c];
            const uint32_t count = (uint32_t)sv[t.x & 0xFFFFu] + sv[t.x >> 16] +
                                   sv[t.y & 0xFFFFu] + sv[t.y >> 16] + sv[t.z & 0xFFFFu] +
                                   sv[t.z >> 16] + sv[t.w & 0xFFFFu] + sv[t.w >> 16];
            o[c] = (uint8_t)(((count | (uint32_t)sv[c]) == 3u) ? 1 : 0);
        }
    }
}

// ---------------------------------------------------------------------------
// CA, rho = 64: bit-sliced rows (the row codec of sg_compact.cuh moves a
// tile row between its compact run and a 64-bit word).  A warp takes one
// tile (729 elements) at a time:
//   1. ballots turn the 729 states (0 / 1) into 23 words of compact bits;
//   2. each lane deposits rows 2*lane and 2*lane + 1 into 64-bit row words,
//      a block at a time through dep[y & 7][block];
//   3. the B3/S23 rule runs on whole rows: horizontal 3-sums and 2-sums by
//      bitwise full adders, the rows above and below through shuffles, the
//      halo cells of the neighbouring tiles as edge bits;
//   4. the next rows are gathered back (cmp[y & 7][byte]) into compact bits
//      and stored as bytes.
// Non-member columns hold 0 in every row word and are dropped by the gather,
// so the rule can run on them freely.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t maj3(uint64_t a, uint64_t b, uint64_t c)
{
    return (a & b) | (c & (a ^ b));
}

// Horizontal sums of a row (bit x: cells x-1, x, x+1), with the cells left
// of column 0 and right of column 63 given as edge bits.
struct RowSums {
    uint64_t t0, t1;    // 3-sum L + v + R, bit planes
    uint64_t d0, d1;    // 2-sum L + R
};

__device__ __forceinline__ RowSums row_sums(uint64_t v, uint32_t left, uint32_t right)
{
    const uint64_t L = (v << 1) | (uint64_t)left, R = (v >> 1) | ((uint64_t)right << 63);
    RowSums s;
    s.t0 = L ^ v ^ R;
    s.t1 = maj3(L, v, R);
    s.d0 = L ^ R;
    s.d1 = L & R;
    return s;
}

// B3/S23 on a row from the 3-sums above and below and its own 2-sum.
__device__ __forceinline__ uint64_t life_row(uint64_t u0, uint64_t u1, uint64_t m0, uint64_t m1,
                                             uint64_t b0, uint64_t b1, uint64_t self)
{
    const uint64_t s0 = u0 ^ m0 ^ b0, k0 = maj3(u0, m0, b0);
    const uint64_t t = u1 ^ m1 ^ b1, k1 = maj3(u1, m1, b1);
    const uint64_t s1 = t ^ k0, k2 = t & k0;
    // count = s0 + 2*s1 + 4*(k1 + k2): 2 or 3 iff s1 and no carry out of bit 1
    return s1 & ~(k1 | k2) & (s0 | self);
}

__device__ __forceinline__ uint64_t shfl_up64(uint64_t v)
{
    const uint32_t lo = __shfl_up_sync(0xffffffffu, (uint32_t)v, 1);
    const uint32_t hi = __shfl_up_sync(0xffffffffu, (uint32_t)(v >> 32), 1);
    return (uint64_t)lo | ((uint64_t)hi << 32);
}

__device__ __forceinline__ uint64_t shfl_down64(uint64_t v)
{
    const uint32_t lo = __shfl_down_sync(0xffffffffu, (uint32_t)v, 1);
    const uint32_t hi = __shfl_down_sync(0xffffffffu, (uint32_t)(v >> 32), 1);
    return (uint64_t)lo | ((uint64_t)hi << 32);
}

__global__ void __launch_bounds__(kUnitThreads, 5)
compact_ca_bits_kernel(const uint8_t *__restrict__ in, uint8_t *__restrict__ out, int r, int order,
                       uint32_t total)
{
    constexpr int S = 6, WORDS = (kUnit + 31) / 32;           // 23 words of compact bits
    __shared__ RowCodec tc;
    __shared__ uint32_t cbits[kUnitWarps][WORDS + 3], obits[kUnitWarps][WORDS + 3];
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(&kRowCodec);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&tc);
        for (int i = threadIdx.x; i < (int)(sizeof(RowCodec) / 4); i += kUnitThreads)
            dst[i] = src[i];
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t *cb = cbits[warp], *ob = obits[warp];
    if (lane >= WORDS && lane < WORDS + 3) cb[lane] = 0u;     // guard words
    __syncthreads();
    static_assert(sizeof(RowCodec) % 4 == 0, "copied as words");

    const CompactPattern<S> &pat = compact_pattern<S>();
    const int rb = r - S;
    const uint32_t units = total / kUnit;                     // whole tiles: r >= 6
    LambdaLane ll;
    ll.init(lane, rb, order);
    const uint32_t W = pi_word(order, rb);
    const uint32_t y0 = 2u * lane, y1 = y0 + 1u;
    const uint32_t o0 = tc.row_start[y0], o1 = tc.row_start[y1];
    // halo cell k of lane k: its place around the tile, (ex, ey) in [-1, 64]
    int ex = 0, ey = 0;
    if (lane < kCaHalo) {
        ex = pat.ca_halo[lane][0] * 64 + pat.ca_halo[lane][2];
        ey = pat.ca_halo[lane][1] * 64 + pat.ca_halo[lane][3];
    }
    const uint32_t nwarps = gridDim.x * kUnitWarps;
    for (uint32_t u = blockIdx.x * kUnitWarps + warp; u < units; u += nwarps) {
        const uint32_t bq = u / W, aq = u - bq * W;
        const uint2 b = ll.decode(aq, bq);
        const uint32_t base = u * kUnit;
        // halo cells (lanes 0..7): their loads are issued first
        uint32_t hv = 0;
        if (lane < kCaHalo) {
            bool p;
            hv = halo_value<uint8_t, S>(in, b, pat.ca_halo[lane][0], pat.ca_halo[lane][1],
                                        pat.ca_halo_rank[lane], rb, order, &p);
        }
        // 1. compact bits: lane `it` keeps word `it`
        uint32_t mine = 0;
#pragma unroll
        for (int it = 0; it < WORDS; ++it) {
            const int c = 32 * it + lane;
            const uint8_t v = c < kUnit ? in[base + c] : 0;
            const uint32_t w = __ballot_sync(0xffffffffu, v != 0);
            if (lane == it) mine = w;
        }
        const bool alive = hv != 0;
        __syncwarp();                  // the previous tile's reads of cb are done
        if (lane < WORDS) cb[lane] = mine;
        if (lane < WORDS + 3) ob[lane] = 0u;
        // edge bits and the rows above row 0 and below row 63
        const uint32_t up_body = __ballot_sync(0xffffffffu, alive && ey == -1 && ex == 0);
        const uint32_t up_right = __ballot_sync(0xffffffffu, alive && ey == -1 && ex == 64);
        const uint32_t dn_body0 = __ballot_sync(0xffffffffu, alive && ey == 64 && ex == 0);
        const uint32_t dn_body1 = __ballot_sync(0xffffffffu, alive && ey == 64 && ex == 1);
        const uint32_t dn_left = __ballot_sync(0xffffffffu, alive && ey == 64 && ex == -1);
        const uint32_t l0 = __ballot_sync(0xffffffffu, alive && ey == 0 && ex == -1);
        const uint32_t r0 = __ballot_sync(0xffffffffu, alive && ey == 0 && ex == 64);
        const uint32_t r1 = __ballot_sync(0xffffffffu, alive && ey == 1 && ex == 64);
        __syncwarp();
        // 2. rows
        const uint64_t v0 = deposit_row(tc, bits_at(cb, o0), y0);
        const uint64_t v1 = deposit_row(tc, bits_at(cb, o1), y1);
        // 3. the rule; only lane 0 has cells beside the left and right edges
        const bool first = lane == 0, last = lane == 31;
        const RowSums a = row_sums(v0, first && l0, first && r0);
        const RowSums c = row_sums(v1, 0u, first && r1);
        uint64_t u0 = shfl_up64(c.t0), u1 = shfl_up64(c.t1);       // row y0 - 1
        uint64_t b0 = shfl_down64(a.t0), b1 = shfl_down64(a.t1);   // row y1 + 1
        if (first) {
            const RowSums h = row_sums(up_body ? 1ull : 0ull, 0u, up_right != 0u);
            u0 = h.t0;
            u1 = h.t1;
        }
        if (last) {
            const RowSums h = row_sums((dn_body0 ? 1ull : 0ull) | (dn_body1 ? 2ull : 0ull),
                                       dn_left != 0u, 0u);
            b0 = h.t0;
            b1 = h.t1;
        }
        const uint64_t n0 = life_row(u0, u1, a.d0, a.d1, c.t0, c.t1, v0);
        const uint64_t n1 = life_row(a.t0, a.t1, c.d0, c.d1, b0, b1, v1);
        // 4. back to compact bits, then bytes
        or_bits_at(ob, o0, gather_row(tc, n0, y0));
        or_bits_at(ob, o1, gather_row(tc, n1, y1));
        __syncwarp();
#pragma unroll
        for (int it = 0; it < WORDS; ++it) {
            const int cc = 32 * it + lane;
            if (cc < kUnit) out[base + cc] = (uint8_t)((ob[it] >> lane) & 1u);
        }
    }
}

template <int S>
__global__ void __launch_bounds__(kUnitThreads)
compact_diffuse_kernel(const float *__restrict__ in, float *__restrict__ out, int r, int order,
                       uint32_t total, float alpha)
{
    using M = StencilSmem<float, S, kDiffHalo, kUnit * 16>;
    extern __shared__ __align__(16) unsigned char smem[];
    const CompactPattern<S> &pat = compact_pattern<S>();
    // per position: staged-value indices of (left, right), (above, below);
    // the tile within the unit and the gasket neighbours inside the tile; and
    // which halo presence bytes count towards the degree
    uint4 *nbt = reinterpret_cast<uint4 *>(smem);
    for (int c = threadIdx.x; c < kUnit; c += kUnitThreads) {
        const int g = c / CompactPattern<S>::C, e = c - g * CompactPattern<S>::C;
        uint32_t hsel = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint16_t v = pat.df_nb[e][k];
            if (v != kNoCell && (v & kHaloBit)) hsel |= 1u << (8 * (v & 3u));
        }
        nbt[c] = make_uint4(stage_slot<S, kDiffHalo>(pat.df_nb[e][0], g) |
                                (stage_slot<S, kDiffHalo>(pat.df_nb[e][1], g) << 16),
                            stage_slot<S, kDiffHalo>(pat.df_nb[e][2], g) |
                                (stage_slot<S, kDiffHalo>(pat.df_nb[e][3], g) << 16),
                            (uint32_t)pat.df_deg_in[e] | ((uint32_t)g << 8), hsel);
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *region = smem + M::TABLE + warp * M::WARP;
    uint2 *coord = reinterpret_cast<uint2 *>(region + M::COORD);
    uint8_t *pres = region + M::PRES;
    const uint32_t *presw = reinterpret_cast<const uint32_t *>(region + M::PRES);
    float *sv = reinterpret_cast<float *>(region + M::VALS);
    const int rb = r - S;
    const uint32_t ntiles = total / CompactPattern<S>::C, units = (total + kUnit - 1) / kUnit;
    LambdaLane ll;
    ll.init(lane, rb, order);
    const uint32_t W = pi_word(order, rb);
    const uint32_t nwarps = gridDim.x * kUnitWarps;
    for (uint32_t u = blockIdx.x * kUnitWarps + warp; u < units; u += nwarps) {
        __syncwarp();
        const uint32_t cnt = stage_unit<float, S, kDiffHalo>(
            sv, coord, pres, in, u, total, ntiles, W, ll, pat.df_halo, pat.df_halo_rank, rb,
            order);
        float *o = out + u * kUnit;
#pragma unroll 4
        for (uint32_t c = lane; c < cnt; c += 32) {
            const uint4 t = nbt[c];
            uint32_t deg = t.z & 0xFFu;
            if (t.w) deg += __popc(presw[t.z >> 8] & t.w);
            const float l = sv[t.x & 0xFFFFu], rr = sv[t.x >> 16];
            const float up = sv[t.y & 0xFFFFu], dn = sv[t.y >> 16];
            o[c] = diffuse_update(sv[c], l, rr, up, dn, (float)deg, alpha);
        }
    }
}

// ---------------------------------------------------------------------------
// Diffusion, rho >= 16: triples.  The gasket cells come in threes A = (X, Y),
// B = (X+1, Y), C = (X, Y+1) with X, Y even and (X & Y) == 0.  Of a triple's
// 4-neighbours, A has B, C and one cell outside at most (the B to its left or
// the C above it, never both), B has A and the A to its right, C has A and the
// A below it.  A unit's 729 elements are 243 triples, one per thread in
// row-major order, so that A and B are consecutive elements, C follows in the
// next row, and consecutive threads read and write consecutive elements
// straight from and to HBM; the three outside values go through shared memory
// (three stores and three loads per triple).  At a tile's corners they come
// from the neighbouring tile, whose launch index follows from the digits of
// this one (corner_tile); a warp of its own looks them up ahead.
//
// Bound: HBM (reads and writes 8 bytes a cell, contiguous: 17 us at level 15).
// Each thread keeps two units' loads in flight while it updates two; one
// barrier per pair (two publishing buffers).  Five gathers and a table entry per
// cell, and here, over several inputs in turn: level 15, rho 64, 37.3 and 21.6 us;
// rho 16, 45.3 and 24.4; level 14, rho 64, 17.6 and 9.1; level 10 (in the L2), 6.9
// and 2.2.  One input again and again, level 15, rho 64: 20.6 (one unit at a time
// 23.6; 7 CTAs an SM with 32 registers and spills 30.6, 5 with 40 registers here).
// ---------------------------------------------------------------------------

// The tile that touches corner `kind` (0: A, 1: B, 2: C) of tile q in the
// 4-neighbour graph, as a launch index of the interleaved order (~0u: none).
// The digits of q are the levels' choices, finest first: 0 the lower, 1 the
// upper left, 2 the right third.  The finest digits that agree with the corner
// are skipped; the first that does not says which sibling lies across, and
// that tile's finer digits are those of the corner it touches with.  *above:
// at corner A, the tile lies above (else to the left).
__device__ __forceinline__ uint32_t corner_tile(uint32_t q, uint32_t kind, int rb, bool *above)
{
    const uint32_t at = kind == 0u ? 1u : kind == 1u ? 2u : 0u;         // digit at the corner
    uint32_t pw = 1u, rest = q, d = at;
    int j = 0;
    for (; j < rb; ++j, pw *= 3u) {
        const uint32_t n = rest / 3u;
        d = rest - 3u * n;
        rest = n;
        if (d != at) break;
    }
    *above = d == 0u;
    if (j == rb || (kind != 0u && d != 1u)) return ~0u;    // the gasket's own corner; a diagonal
    const uint32_t ones = (pw - 1u) / 2u;                  // finer digits all 1
    return kind == 0u ? q - ones - d * pw + pw + (d == 2u ? 2u * ones : 0u)
                      : q - at * ones - pw + at * pw + ones;
}

// The same for a launch index of the row-major order, whose digits are dealt in
// turn to omega_y (the finest first) and omega_x: q = omega_y * W + omega_x.  A
// digit of omega_y thus weighs W times a power of 3, one of omega_x the power;
// else as above (the finer digits become d, the first that differs `at`).  Few
// digits are looked at: moving the index to the other order and back, ten digits
// each way, made the corner warp the slowest of its CTA (level 16, rho 32, 120.0
// us against 99.7 for the gathers it replaced).
__device__ __forceinline__ uint32_t corner_tile_rowmajor(uint32_t q, uint32_t kind, int rb,
                                                         uint32_t W, bool *above)
{
    const uint32_t at = kind == 0u ? 1u : kind == 1u ? 2u : 0u;
    uint32_t w = q / W, v = q - w * W;       // the word the next digit comes from, the other
    uint32_t pw = W, pv = 1u, ones = 0u, d = at;
    int j = 0;
    for (; j < rb; ++j) {
        const uint32_t n = w / 3u;
        d = w - 3u * n;
        if (d != at) break;
        ones += pw;
        const uint32_t p = 3u * pw;
        w = v;
        v = n;
        pw = pv;
        pv = p;
    }
    *above = d == 0u;
    if (j == rb || (kind != 0u && d != 1u)) return ~0u;
    return q + (d - at) * ones + (at - d) * pw;
}

// Per triple of a level-S tile, in row-major order: the element of A (B is the
// next) and of C, and the words the outside values come from (plane * 243 +
// triple; kNoTriple: none in the tile).  corner: 1, 2, 3 for the tile's corner
// A, B, C.  (kNoTriple is also the word that holds 0.)
constexpr uint16_t kNoTriple = 3 * 243;
template <int S> struct TriplePattern {
    static constexpr int T = pow3i(S - 1);
    uint16_t a[T], c[T], rp[T], rq[T], rr[T];
    uint8_t corner[T];
};
template <int S> constexpr TriplePattern<S> make_triple_pattern()
{
    constexpr int H = 1 << (S - 1);
    TriplePattern<S> p{};
    uint16_t id[H][H] = {};
    int t = 0;
    for (int y = 0; y < H; ++y)
        for (int x = 0; x < H; ++x)
            if ((x & y) == 0) id[y][x] = (uint16_t)t++;
    t = 0;
    for (int y = 0; y < H; ++y) {
        int m = 0;
        for (int x = 0; x < H; ++x) m += (x & y) == 0;
        const int first = t;
        for (int x = 0; x < H; ++x) {
            if ((x & y) != 0) continue;
            p.a[t] = (uint16_t)(3 * first + 2 * (t - first));
            p.c[t] = (uint16_t)(3 * first + 2 * m + (t - first));
            p.rp[t] = p.rq[t] = p.rr[t] = kNoTriple;
            if (x > 0 && ((x - 1) & y) == 0) p.rp[t] = (uint16_t)(243 + id[y][x - 1]);
            else if (y > 0 && (x & (y - 1)) == 0) p.rp[t] = (uint16_t)(486 + id[y - 1][x]);
            if (x + 1 < H && ((x + 1) & y) == 0) p.rq[t] = id[y][x + 1];
            if (y + 1 < H && (x & (y + 1)) == 0) p.rr[t] = id[y + 1][x];
            if (x == 0 && y == 0) p.corner[t] = 1;
            if (x == H - 1 && y == 0) p.corner[t] = 2;
            if (x == 0 && y == H - 1) p.corner[t] = 3;
            ++t;
        }
    }
    return p;
}
__device__ const TriplePattern<4> kTriples4 = make_triple_pattern<4>();
__device__ const TriplePattern<5> kTriples5 = make_triple_pattern<5>();
__device__ const TriplePattern<6> kTriples6 = make_triple_pattern<6>();
template <int S> __device__ __forceinline__ const TriplePattern<S> &triple_pattern()
{
    if constexpr (S == 4) return kTriples4;
    else if constexpr (S == 5) return kTriples5;
    else return kTriples6;
}

constexpr int kTripleThreads = 288;      // eight warps of triples, one for the tiles' corners
constexpr int kTripleUnits = 2;          // units a CTA has in hand at a time

template <int S>
__global__ void __launch_bounds__(kTripleThreads, 5)
compact_diffuse_triples_kernel(const float *__restrict__ in, float *__restrict__ out, int r,
                               int order, uint32_t total, float alpha)
{
    constexpr int T = pow3i(S - 1), C = pow3i(S), G = kUnit / C, RHO = 1 << S, N = kTripleUnits;
    constexpr int EXT = kNoTriple + 1, FLAG = EXT + 3 * G;       // corner values, and what they are
    __shared__ float pub[2][N][FLAG + 3 * G];
    const int tid = threadIdx.x;
    const int rb = r - S;
    const uint32_t ntiles = total / C, units = (ntiles + G - 1) / G;
    if (tid < 2 * N) pub[tid & 1][tid >> 1][kNoTriple] = 0.f;

    if (tid >= 256) {
        // The corner warp: lane i fetches the value outside corner i % 3 of
        // tile i / 3 of the unit (flag: 0 none, 1 there, 2 there and above).
        const int lane = tid - 256;
        const uint32_t g = (uint32_t)lane / 3u, kind = (uint32_t)lane - 3u * g;
        const uint32_t W = pi_word(order, rb);
        float e[N], f[N];
        auto fetch = [&](uint32_t u, int i) {
            const uint32_t q = u * G + g;
            e[i] = f[i] = 0.f;
            if (lane >= 3 * G || q >= ntiles) return;
            bool above = false;
            const uint32_t nq = order == kOrderInterleaved
                                    ? corner_tile(q, kind, rb, &above)
                                    : corner_tile_rowmajor(q, kind, rb, W, &above);
            if (nq == ~0u) return;
            // outside corner A lies the tile's corner B or C, else its corner A
            const uint32_t at = kind != 0u ? 0u : above ? (uint32_t)C - 1u : (uint32_t)RHO - 1u;
            e[i] = __ldg(in + (uint64_t)nq * C + at);
            f[i] = kind == 0u && above ? 2.f : 1.f;
        };
        uint32_t u = blockIdx.x;
#pragma unroll
        for (int i = 0; i < N; ++i) fetch(min(u + i * gridDim.x, units), i);
        for (int buf = 0; u < units; buf ^= 1) {
            if (lane < 3 * G) {
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    pub[buf][i][EXT + lane] = e[i];
                    pub[buf][i][FLAG + lane] = f[i];
                }
            }
            u += N * gridDim.x;
#pragma unroll
            for (int i = 0; i < N; ++i) fetch(min(u + i * gridDim.x, units), i);
            __syncthreads();
        }
        return;
    }

    const int g = tid / T, t = tid - g * T;
    const bool mine = tid < 243;
    uint32_t ea = 0, ec = 0, rp = kNoTriple, rq = kNoTriple, rr = kNoTriple, corner = 0;
    float da = 2.f, db = 1.f, dc = 1.f;
    bool left = false;
    if (mine) {
        const TriplePattern<S> &pat = triple_pattern<S>();
        ea = g * C + pat.a[t];
        ec = g * C + pat.c[t];
        corner = pat.corner[t];
        rp = pat.rp[t];
        rq = pat.rq[t];
        rr = pat.rr[t];
        left = rp < 486u;
        if (rp != kNoTriple) { rp += g * T; da = 3.f; }
        if (rq != kNoTriple) { rq += g * T; db = 2.f; }
        if (rr != kNoTriple) { rr += g * T; dc = 2.f; }
        if (corner == 1u) rp = EXT + 3 * g;
        if (corner == 2u) rq = EXT + 3 * g + 1;
        if (corner == 3u) rr = EXT + 3 * g + 2;
    }
    float a[N], b[N], c[N];
    uint32_t u = blockIdx.x;
    const uint32_t step = gridDim.x * kUnit, to_c = ec - ea;
    const float *src = in + u * kUnit + ea;
    float *dst = out + u * kUnit + ea;
    // the units this thread has a triple in: u < lim (whole ones, or the only one)
    const uint32_t lim = !mine ? 0u : (uint32_t)g < ntiles ? (ntiles - (uint32_t)g + G - 1) / G : 0u;
    auto load = [&] {
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (u + i * gridDim.x < lim) {
                a[i] = __ldg(src + i * step);
                b[i] = __ldg(src + i * step + 1);
                c[i] = __ldg(src + i * step + to_c);
            }
    };
    load();
    for (int buf = 0; u < units; buf ^= 1) {
        float ca[N], cb[N], cc[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            float *w = pub[buf][i];
            ca[i] = a[i];
            cb[i] = b[i];
            cc[i] = c[i];
            if (mine) {
                w[tid] = a[i];
                w[243 + tid] = b[i];
                w[486 + tid] = c[i];
            }
        }
        const uint32_t cur = u;
        u += N * gridDim.x;
        src += N * step;
        load();                             // in flight across the barrier and the update
        __syncthreads();
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if (cur + i * gridDim.x >= lim) break;
            const float *w = pub[buf][i];
            const float p = w[rp], q = w[rq], s = w[rr];
            if (corner != 0u) {
                const float f = w[FLAG + 3 * g + (int)corner - 1];
                const float n = f != 0.f ? 1.f : 0.f;
                if (corner == 1u) { da = 2.f + n; left = f < 2.f; }
                if (corner == 2u) db = 1.f + n;
                if (corner == 3u) dc = 1.f + n;
            }
            dst[i * step] = diffuse_update(ca[i], left ? p : 0.f, cb[i], left ? 0.f : p, cc[i], da, alpha);
            dst[i * step + 1] = diffuse_update(cb[i], ca[i], q, 0.f, 0.f, db, alpha);
            dst[i * step + to_c] = diffuse_update(cc[i], 0.f, 0.f, ca[i], s, dc, alpha);
        }
        dst += N * step;
    }
}

template <int S>
cudaError_t launch_ca_t(int r, int order, const uint8_t *in, uint8_t *out, cudaStream_t st,
                        const LaunchCfg &cfg)
{
    static std::atomic<int> occ{0};
    const uint32_t total = (uint32_t)pow3i(r);
    const uint64_t units = (total + kUnit - 1) / kUnit;
    unsigned grid = 1;
    if constexpr (S == 6) {
        // on words of 32 tiles from level 14 on (over several inputs in turn, level
        // 14, 9.6 us against 11.3; level 15, 16.0 against 27.5; level 16, 38.6
        // against 75.1; one input again and again, level 13, 7.7 against 6.1)
        if (r >= 14) return launch_compact_ca_words(r, 6, order, in, out, 1, st, cfg);
        auto k = compact_ca_bits_kernel;
        cudaError_t e = persistent_grid(k, kUnitThreads, 0, (units + kUnitWarps - 1) / kUnitWarps,
                                        cfg, &grid, &occ);
        if (e != cudaSuccess) return e;
        k<<<grid, kUnitThreads, 0, st>>>(in, out, r, order, total);
    } else {
        static std::atomic<uint64_t> attr{0};
        auto k = compact_ca_kernel<S>;
        constexpr int smem = StencilSmem<uint8_t, S, kCaHalo, kUnit * 16>::BYTES;
        cudaError_t e = dyn_smem_grid(k, smem, (units + kUnitWarps - 1) / kUnitWarps, cfg, &grid,
                                      &occ, &attr);
        if (e != cudaSuccess) return e;
        k<<<grid, kUnitThreads, smem, st>>>(in, out, r, order, total);
    }
    return cudaGetLastError();
}

template <int S>
cudaError_t launch_diffuse_t(int r, int order, const float *in, float *out, float alpha,
                             cudaStream_t st, const LaunchCfg &cfg)
{
    static std::atomic<int> occ{0};
    const uint32_t total = (uint32_t)pow3i(r);
    const uint64_t units = (total + kUnit - 1) / kUnit;
    unsigned grid = 1;
    if constexpr (S >= 4) {
        auto k = compact_diffuse_triples_kernel<S>;
        cudaError_t e = persistent_grid(k, kTripleThreads, 0, units, cfg, &grid, &occ);
        if (e != cudaSuccess) return e;
        k<<<grid, kTripleThreads, 0, st>>>(in, out, r, order, total, alpha);
    } else {
        static std::atomic<uint64_t> attr{0};
        auto k = compact_diffuse_kernel<S>;
        constexpr int smem = StencilSmem<float, S, kDiffHalo, kUnit * 16>::BYTES;
        cudaError_t e = dyn_smem_grid(k, smem, (units + kUnitWarps - 1) / kUnitWarps, cfg, &grid,
                                      &occ, &attr);
        if (e != cudaSuccess) return e;
        k<<<grid, kUnitThreads, smem, st>>>(in, out, r, order, total, alpha);
    }
    return cudaGetLastError();
}

#define SG_COMPACT_S_SWITCH(s, CALL)         \
    switch (s) {                             \
    case 0: return CALL(0);                  \
    case 1: return CALL(1);                  \
    case 2: return CALL(2);                  \
    case 3: return CALL(3);                  \
    case 4: return CALL(4);                  \
    case 5: return CALL(5);                  \
    case 6: return CALL(6);                  \
    default: return cudaErrorInvalidValue;   \
    }

}  // namespace

cudaError_t launch_compact_ca(int r, int s, int order, const uint8_t *in, uint8_t *out,
                              cudaStream_t st, const LaunchCfg &cfg)
{
    // 16- and 32-tiles in the interleaved order on words (us, gathered against
    // words: rho 16, level 8, 7.9 and 6.5; rho 32, 6.9 and 6.3; over several inputs
    // in turn, level 15, 46.6 and 16.1; 37.4 and 16.1)
    if ((s == 4 || s == 5) && order == kOrderInterleaved && r >= 6)
        return launch_compact_ca_words(r, s, order, in, out, 1, st, cfg);
#define CALL(S) launch_ca_t<S>(r, order, in, out, st, cfg)
    SG_COMPACT_S_SWITCH(s, CALL)
#undef CALL
}

cudaError_t launch_compact_diffuse(int r, int s, int order, const float *in, float *out,
                                   float alpha, cudaStream_t st, const LaunchCfg &cfg)
{
#define CALL(S) launch_diffuse_t<S>(r, order, in, out, alpha, st, cfg)
    SG_COMPACT_S_SWITCH(s, CALL)
#undef CALL
}

}  // namespace sg
