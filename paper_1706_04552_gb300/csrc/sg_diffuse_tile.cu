// sg_diffuse_tile.cu -- k <= 8 diffusion steps under lambda, one warp per
// 64-tile, every cell in a register.
//
// A lane holds one 8 x 8 piece of the tile: 27 gasket cells in three 4 x 4 blocks
// of nine, (0,0), (1,0) and (0,1) of the piece, each the level-2 gasket
//
//     j = 0:  (0,0) (1,0) (2,0) (3,0)
//     j = 1:  (0,1)       (2,1)
//     j = 2:  (0,2) (1,2)
//     j = 3:  (0,3)
//
// The tile is the 27 pieces of lanes 0..26 (lane = base-3 digits of the piece's
// place: 0 upper left, 1 right, 2 lower third, finest first).  A triangle of
// the gasket touches another only at its corners, and in the 4-neighbour graph
// by one link: corner A = (0,0) to the B corner of the triangle on its left or
// the C corner of the one above (never both), corner B = (7,0) to the A corner
// on its right, corner C = (0,7) to the A corner below.  So a step needs four
// shuffles per 27 cells and no shared memory, and the halo of a tile is not a
// frame around it but the three 8 x 8 pieces across its corners, on lanes 27,
// 28 and 29: everything within 8 steps of the tile's cells.  A halo piece's own
// far corners take no neighbour; that error starts 9 steps away from the tile.
// Lanes 30 and 31 hold zeros, which a missing neighbour reads.
//
// Every cell goes through diffuse_update with the operands of the single-step
// tile kernels (a neighbour off the gasket is the 0 the state holds there), so
// the results are theirs bit for bit, and k steps equal k single steps.
//
// Bound: DRAM's rate for the touched sectors (at level 15, 272 MB read and written
// at 3.3 TB/s).  Over several inputs in turn, 8 steps take 83.1 us and one 81.8,
// where 32 x 32 units with a frame of halo took 106.1 and chunks staged through
// shared memory 85.7 to 145; level 14: 27.9 and 27.4 against 38.6 and 31.1 to 50.
// (About 1150 warp instructions per tile and 8 steps, 5000 before.)
#include "sg_stencil.cuh"
#include "sg_words.cuh"

namespace sg {

namespace {

constexpr int kDiffWarps = 4;                 // independent warps per CTA
constexpr int kIdleLane = 31;

struct Block9 {
    float u00, u10, u20, u30, u01, u21, u02, u12, u03;
};

// One step of a block from its four outside neighbours and the degrees that
// depend on them.
__device__ __forceinline__ Block9 block_step(const Block9 &b, float l, float up, float rt, float dn,
                                             float d00, float d30, float d03, float alpha)
{
    // diffuse_update(u, left, right, up, down, degree, alpha)
    Block9 o;
    o.u00 = diffuse_update(b.u00, l, b.u10, up, b.u01, d00, alpha);
    o.u10 = diffuse_update(b.u10, b.u00, b.u20, 0.f, 0.f, 2.f, alpha);
    o.u20 = diffuse_update(b.u20, b.u10, b.u30, 0.f, b.u21, 3.f, alpha);
    o.u30 = diffuse_update(b.u30, b.u20, rt, 0.f, 0.f, d30, alpha);
    o.u01 = diffuse_update(b.u01, 0.f, 0.f, b.u00, b.u02, 2.f, alpha);
    o.u21 = diffuse_update(b.u21, 0.f, 0.f, b.u20, 0.f, 1.f, alpha);
    o.u02 = diffuse_update(b.u02, 0.f, b.u12, b.u01, b.u03, 3.f, alpha);
    o.u12 = diffuse_update(b.u12, b.u02, 0.f, 0.f, 0.f, 1.f, alpha);
    o.u03 = diffuse_update(b.u03, 0.f, 0.f, b.u02, dn, d03, alpha);
    return o;
}

// Eight floats of a row: one access if both grids are 32-byte aligned (`wide`).
__device__ __forceinline__ void load8(float (&v)[8], const float *p, bool wide)
{
    if (wide) {
        uint32_t w[8];
        ld_global_v8(p, w);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(w[i]);
    } else {
        const float4 a = *reinterpret_cast<const float4 *>(p);
        const float4 b = *reinterpret_cast<const float4 *>(p + 4);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
}
__device__ __forceinline__ void store8(float *p, float4 a, float4 b, bool wide)
{
    if (wide) {
        const uint32_t w[8] = {__float_as_uint(a.x), __float_as_uint(a.y), __float_as_uint(a.z),
                               __float_as_uint(a.w), __float_as_uint(b.x), __float_as_uint(b.y),
                               __float_as_uint(b.z), __float_as_uint(b.w)};
        st_global_v8(p, w);
    } else {
        *reinterpret_cast<float4 *>(p) = a;
        *reinterpret_cast<float4 *>(p + 4) = b;
    }
}

__global__ void __launch_bounds__(32 * kDiffWarps, 6)
diffuse_tile_kernel(const float *__restrict__ in, float *__restrict__ out, int r, int order,
                    uint32_t ntiles, int k, float alpha)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t n = 1ull << r;
    const int rb = r - 6;
    const uint32_t nb = 1u << rb;
    const bool wide = (((uintptr_t)in | (uintptr_t)out) & 31u) == 0u;
    LambdaLane ll;
    ll.init(lane, rb, order);
    const uint32_t W = pi_word(order, rb);

    // the lane's piece and, inside the tile, the lanes across its corners
    const bool own = lane < 27;
    const uint2 pc = gasket_coords(own ? (uint32_t)lane : 0u, 3);
    uint32_t nx, ny;
    uint32_t kind = corner_neighbour<0>(pc.x, pc.y, 8u, nx, ny);
    const int in_l = own && kind == 1u ? (int)gasket_digits(nx, ny, 3) : kIdleLane;
    const int in_u = own && kind == 2u ? (int)gasket_digits(nx, ny, 3) : kIdleLane;
    kind = corner_neighbour<1>(pc.x, pc.y, 8u, nx, ny);
    const int in_r = own && kind == 1u ? (int)gasket_digits(nx, ny, 3) : kIdleLane;
    kind = corner_neighbour<2>(pc.x, pc.y, 8u, nx, ny);
    const int in_d = own && kind == 1u ? (int)gasket_digits(nx, ny, 3) : kIdleLane;

    for (uint32_t q = blockIdx.x * kDiffWarps + warp; q < ntiles; q += gridDim.x * kDiffWarps) {
        const uint2 c = decode_tile<kMapLambda>(q, ntiles, rb, W, ll);     // warp-collective
        // the tiles across the tile's corners (uniform in the warp)
        uint32_t ax, ay, bx, by, cx, cy;
        const uint32_t ka = corner_neighbour<0>(c.x, c.y, nb, ax, ay);
        const uint32_t kb = corner_neighbour<1>(c.x, c.y, nb, bx, by);
        const uint32_t kc = corner_neighbour<2>(c.x, c.y, nb, cx, cy);
        int src_l = in_l, src_u = in_u, src_r = in_r, src_d = in_d;
        uint32_t x = 64u * c.x + 8u * pc.x, y = 64u * c.y + 8u * pc.y;
        bool on = own;
        if (lane == 0) {
            if (ka == 1u) src_l = 27;
            if (ka == 2u) src_u = 27;
        }
        if (lane == 13 && kb == 1u) src_r = 28;          // corner B of the tile
        if (lane == 26 && kc == 1u) src_d = 29;          // corner C
        if (lane == 27) {                                // the left tile's corner B, or the
            on = ka != 0u;                               // upper tile's corner C
            x = 64u * ax + (ka == 1u ? 56u : 0u);
            y = 64u * ay + (ka == 2u ? 56u : 0u);
            if (ka == 1u) src_r = 0;
            if (ka == 2u) src_d = 0;
        }
        if (lane == 28) {                                // the right tile's corner A
            on = kb == 1u;
            x = 64u * bx;
            y = 64u * by;
            if (on) src_l = 13;
        }
        if (lane == 29) {                                // the lower tile's corner A
            on = kc == 1u;
            x = 64u * cx;
            y = 64u * cy;
            if (on) src_u = 26;
        }

        const uint64_t at = (uint64_t)y * n + x;
        Block9 b0 = {}, b1 = {}, b2 = {};
        if (on) {
            const float *p = in + at;
            float v[4][8];
#pragma unroll
            for (int i = 0; i < 4; ++i) load8(v[i], p + i * n, wide);
            const float *s = p + 4 * n;
            const float4 s0 = *reinterpret_cast<const float4 *>(s);
            const float4 s1 = *reinterpret_cast<const float4 *>(s + n);
            const float2 s2 = *reinterpret_cast<const float2 *>(s + 2 * n);
            const float s3 = s[3 * n];
            b0 = Block9{v[0][0], v[0][1], v[0][2], v[0][3], v[1][0], v[1][2], v[2][0], v[2][1], v[3][0]};
            b1 = Block9{v[0][4], v[0][5], v[0][6], v[0][7], v[1][4], v[1][6], v[2][4], v[2][5], v[3][4]};
            b2 = Block9{s0.x, s0.y, s0.z, s0.w, s1.x, s1.z, s2.x, s2.y, s3};
        }
        const float da = 2.f + (float)(src_l != kIdleLane || src_u != kIdleLane);
        const float db = 1.f + (float)(src_r != kIdleLane), dc = 1.f + (float)(src_d != kIdleLane);
#pragma unroll 1
        for (int s = 0; s < k; ++s) {
            const float l = __shfl_sync(~0u, b1.u30, src_l), up = __shfl_sync(~0u, b2.u03, src_u);
            const float rt = __shfl_sync(~0u, b0.u00, src_r), dn = __shfl_sync(~0u, b0.u00, src_d);
            const Block9 o0 = block_step(b0, l, up, b1.u00, b2.u00, da, 2.f, 2.f, alpha);
            const Block9 o1 = block_step(b1, b0.u30, 0.f, rt, 0.f, 3.f, db, 1.f, alpha);
            const Block9 o2 = block_step(b2, 0.f, b0.u03, 0.f, dn, 3.f, 1.f, dc, alpha);
            b0 = o0;
            b1 = o1;
            b2 = o2;
        }
        if (own) {
            // whole sectors: the other half of the lower rows' holds no gasket cell
            float *p = out + at;
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            store8(p, make_float4(b0.u00, b0.u10, b0.u20, b0.u30),
                   make_float4(b1.u00, b1.u10, b1.u20, b1.u30), wide);
            store8(p + n, make_float4(b0.u01, 0.f, b0.u21, 0.f),
                   make_float4(b1.u01, 0.f, b1.u21, 0.f), wide);
            store8(p + 2 * n, make_float4(b0.u02, b0.u12, 0.f, 0.f),
                   make_float4(b1.u02, b1.u12, 0.f, 0.f), wide);
            store8(p + 3 * n, make_float4(b0.u03, 0.f, 0.f, 0.f),
                   make_float4(b1.u03, 0.f, 0.f, 0.f), wide);
            p += 4 * n;
            store8(p, make_float4(b2.u00, b2.u10, b2.u20, b2.u30), z, wide);
            store8(p + n, make_float4(b2.u01, 0.f, b2.u21, 0.f), z, wide);
            store8(p + 2 * n, make_float4(b2.u02, b2.u12, 0.f, 0.f), z, wide);
            store8(p + 3 * n, make_float4(b2.u03, 0.f, 0.f, 0.f), z, wide);
        }
    }
}

}  // namespace

cudaError_t launch_diffuse_tile(int r, const float *in, float *out, float alpha, int k,
                                cudaStream_t st, const LaunchCfg &cfg)
{
    static std::atomic<int> occ{0};
    const uint32_t ntiles = (uint32_t)pow3i(r - 6);
    unsigned grid = 1;
    cudaError_t e = persistent_grid(diffuse_tile_kernel, 32 * kDiffWarps, 0,
                                    (ntiles + kDiffWarps - 1) / kDiffWarps, cfg, &grid, &occ);
    if (e != cudaSuccess) return e;
    diffuse_tile_kernel<<<grid, 32 * kDiffWarps, 0, st>>>(in, out, r, cfg.order, ntiles, k, alpha);
    return cudaGetLastError();
}

}  // namespace sg
