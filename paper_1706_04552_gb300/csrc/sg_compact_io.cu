// sg_compact_io.cu -- moving between the embedded and the compact layout
// (pack, unpack) and the map-and-write pass on a compact array.
//
// Each warp of a persistent grid takes units of 729 elements (G whole tiles,
// layout in sg_compact.cuh) on its own: it decodes the unit's tiles with the
// lambda reduction of Theorem 1 into its own shared memory, then its lanes
// walk the unit's elements, 32 consecutive ones per step.  The compact side
// is therefore read or written in whole sectors; the embedded side is
// touched only at gasket cells, as the embedded write pass touches it.  The
// per-position table (tile within the unit, tile-relative coordinates) is
// expanded into shared memory once per CTA; after that barrier the warps
// never wait for one another.
#include "sg_compact.cuh"
#include "sg_stencil.cuh"

namespace sg {

namespace {

// Shared memory of a CTA: the unit table, then one region per warp.
template <int S> struct IoSmem {
    static constexpr int G = CompactPattern<S>::G;
    // every region starts on a 16-byte boundary (the per-warp arrays hold
    // 8-byte elements)
    static constexpr int TABLE = (kUnit * 4 + 15) / 16 * 16;     // unit_cell per position
    static constexpr int WARP = ((G * 8) + 15) / 16 * 16;        // per-tile words
    static constexpr int BYTES = TABLE + kUnitWarps * WARP;
    static_assert(TABLE % 16 == 0 && WARP % 16 == 0, "16-byte aligned regions");
};

template <int S>
__device__ __forceinline__ uint32_t *build_cell_table(unsigned char *smem)
{
    uint32_t *cells = reinterpret_cast<uint32_t *>(smem);
    for (int c = threadIdx.x; c < kUnit; c += kUnitThreads) cells[c] = unit_cell<S>(c);
    __syncthreads();
    return cells;
}

// MODE 0: pack (grid -> compact), 1: unpack (compact -> grid).
template <typename T, int S, int MODE>
__global__ void __launch_bounds__(kUnitThreads)
compact_move_kernel(const T *__restrict__ src, T *__restrict__ dst, int r, int order,
                    uint32_t total)
{
    using M = IoSmem<S>;
    constexpr int G = M::G;
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t *cells = build_cell_table<S>(smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint2 *coord = reinterpret_cast<uint2 *>(smem + M::TABLE + warp * M::WARP);
    const int rb = r - S;
    const uint32_t ntiles = total / CompactPattern<S>::C, units = (total + kUnit - 1) / kUnit;
    LambdaLane ll;
    ll.init(lane, rb, order);
    const uint32_t W = pi_word(order, rb);
    const uint32_t nwarps = gridDim.x * kUnitWarps;
    for (uint32_t u = blockIdx.x * kUnitWarps + warp; u < units; u += nwarps) {
        __syncwarp();                 // the previous unit's reads of coord are done
        decode_unit_tiles<G>(coord, u * G, ntiles, W, ll);
        __syncwarp();
        const uint32_t base = u * kUnit;
        const uint32_t cnt = min((uint32_t)kUnit, total - base);
#pragma unroll 4
        for (uint32_t c = lane; c < cnt; c += 32) {
            const uint32_t cell = cells[c];
            const uint2 b = coord[cell & 0x3FFu];
            const uint32_t x = (b.x << S) | ((cell >> 10) & 0x3Fu);
            const uint32_t y = (b.y << S) | (cell >> 16);
            const uint64_t at = ((uint64_t)y << r) | x;
            if constexpr (MODE == 0) dst[base + c] = src[at];
            else dst[at] = src[base + c];
        }
    }
}

// Byte offset of the per-warp staging buffers of the write kernel, and their
// size: a unit's values plus room to align them like their destination.
template <int S> __host__ __device__ constexpr int write_stage_offset()
{
    return IoSmem<S>::BYTES + ((kUnit * 2 + 15) / 16) * 16;
}
template <typename T> __host__ __device__ constexpr int write_stage_bytes()
{
    return (kUnit * (int)sizeof(T) + 16 + 15) / 16 * 16;
}

// WIDE: stage each unit in shared memory and store it in whole aligned
// 16-byte chunks (for a destination in host memory, across the host link);
// otherwise every lane stores its values directly (device memory, rho <= 8).
template <typename T, int VK, int S, bool WIDE>
__global__ void __launch_bounds__(kUnitThreads)
compact_write_kernel(T *__restrict__ compact, int r, int order, uint32_t total, uint64_t vs)
{
    using M = IoSmem<S>;
    constexpr int G = M::G;
    constexpr int STAGE = write_stage_bytes<T>();
    extern __shared__ __align__(16) unsigned char smem[];
    // per position: the value-key offset of the cell within its tile (the
    // same in every tile), and the tile within the unit
    uint32_t *koff = reinterpret_cast<uint32_t *>(smem);
    for (int c = threadIdx.x; c < kUnit; c += kUnitThreads) {
        const uint32_t cell = unit_cell<S>(c);
        koff[c] = CellValue<T, VK>::offset_of((cell >> 10) & 0x3Fu, cell >> 16, r);
    }
    uint16_t *tile_of = reinterpret_cast<uint16_t *>(smem + M::BYTES);
    for (int c = threadIdx.x; c < kUnit; c += kUnitThreads)
        tile_of[c] = (uint16_t)(c / CompactPattern<S>::C);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t *vbase = reinterpret_cast<uint32_t *>(smem + M::TABLE + warp * M::WARP);
    unsigned char *stage = smem + write_stage_offset<S>() + warp * STAGE;
    const int rb = r - S;
    const uint32_t ntiles = total / CompactPattern<S>::C, units = (total + kUnit - 1) / kUnit;
    const CellValue<T, VK> cv{vs * kGoldenGamma, (uint32_t)vs};
    LambdaLane ll;
    ll.init(lane, rb, order);
    const uint32_t W = pi_word(order, rb);
    const uint32_t nwarps = gridDim.x * kUnitWarps;
    for (uint32_t u = blockIdx.x * kUnitWarps + warp; u < units; u += nwarps) {
        __syncwarp();
        for (int g = 0; g < G; ++g) {
            const uint32_t q = u * G + (uint32_t)g;
            if (q < ntiles) {
                const uint32_t bq = q / W, aq = q - bq * W;
                const uint2 b = ll.decode(aq, bq);
                if (lane == 0) vbase[g] = CellValue<T, VK>::base_of(b.x << S, b.y << S, r);
            }
        }
        __syncwarp();
        const uint32_t base = u * kUnit;
        const uint32_t cnt = min((uint32_t)kUnit, total - base);
        if constexpr (!WIDE) {
            T *dst = compact + base;
#pragma unroll 4
            for (uint32_t c = lane; c < cnt; c += 32) {
                const uint32_t vb = G == 1 ? vbase[0] : vbase[tile_of[c]];
                dst[c] = cv(vb, koff[c]);
            }
            continue;
        }
        // the values go to shared memory at the destination's offset within
        // 16 bytes, then out as whole aligned 16-byte chunks (byte stores
        // only for the unit's ragged ends)
        unsigned char *out = reinterpret_cast<unsigned char *>(compact + base);
        const uint32_t lead = (uint32_t)(reinterpret_cast<uintptr_t>(out) & 15u);
        T *sv = reinterpret_cast<T *>(stage + lead);
#pragma unroll 4
        for (uint32_t c = lane; c < cnt; c += 32) {
            const uint32_t vb = G == 1 ? vbase[0] : vbase[tile_of[c]];
            sv[c] = cv(vb, koff[c]);
        }
        __syncwarp();
        const uint32_t nb = cnt * (uint32_t)sizeof(T);
        const uint32_t head = min((16u - lead) & 15u, nb);
        const uint32_t chunks = (nb - head) / 16u, body_end = head + 16u * chunks;
        for (uint32_t i = lane; i < head; i += 32) out[i] = stage[lead + i];
        for (uint32_t k = lane; k < chunks; k += 32)
            *reinterpret_cast<uint4 *>(out + head + 16u * k) =
                *reinterpret_cast<const uint4 *>(stage + lead + head + 16u * k);
        for (uint32_t i = body_end + lane; i < nb; i += 32) out[i] = stage[lead + i];
    }
}

// rho >= 16, device memory: a lane computes four consecutive elements at an
// aligned address and stores them at once.  729 u mod 4 = u mod 4, and a warp's
// units are a multiple of 8 apart, so all of them start at the same place
// within four elements: the value-key offsets of a lane's 24 elements never
// change and stay in registers, and the loop over units touches no shared
// memory.  Only a unit's first and last words, shared with its neighbours,
// store element by element.
//
// Bound: integer issue (the hash: ALU 68 %, and moving its adds and shifts to
// the multipliers was slower, 41.3 and 43.7 us).  uint8, level 16, with a table
// load and a byte store per element and here: rho 64, 43.5 and 39.0 us; rho 16,
// 75.2 and 51.5 (a shuffle per element finds its tile's base); float32, level
// 15, rho 16: 29.2 and 20.1.  (Launches back to back; through the call, with three
// arrays in turn, 45.1 and 41.0 at rho 64.)
template <typename T, int VK, int S>
__global__ void __launch_bounds__(kUnitThreads)
compact_write4_kernel(T *__restrict__ compact, int r, int order, uint32_t total, uint64_t vs)
{
    constexpr int C = CompactPattern<S>::C, G = CompactPattern<S>::G, WORDS = 6;
    static_assert(G <= 32, "a lane per tile of the unit");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rb = r - S;
    const uint32_t ntiles = total / C, units = (total + kUnit - 1) / kUnit;
    const CellValue<T, VK> cv{vs * kGoldenGamma, (uint32_t)vs};
    const uint32_t W = pi_word(order, rb);
    LambdaLane ll;
    ll.init(lane, rb, order);
    const uint32_t u0 = blockIdx.x * kUnitWarps + warp, nwarps = gridDim.x * kUnitWarps;
    // elements before the unit's first aligned word of four
    const int lead = (int)(((uint32_t)(reinterpret_cast<uintptr_t>(compact) / sizeof(T)) + u0) & 3u);
    // word i of the lane: elements 4 (lane + 32 i) - lead + 0..3 of the unit
    uint32_t koff[WORDS][4], tile[WORDS];
#pragma unroll
    for (int i = 0; i < WORDS; ++i) {
        tile[i] = 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = min(max(4 * (lane + 32 * i) - lead + k, 0), kUnit - 1);
            const uint32_t cell = unit_cell<S>(c);
            koff[i][k] = CellValue<T, VK>::offset_of((cell >> 10) & 0x3Fu, cell >> 16, r);
            tile[i] |= (cell & 0x3FFu) << (8 * k);
        }
    }
    for (uint32_t u = u0; u < units; u += nwarps) {
        uint32_t vbase = 0u;                           // of tile `lane` of the unit
        if constexpr (G == 1) {
            const uint32_t bq = u / W, aq = u - bq * W;
            const uint2 b = ll.decode(aq, bq);
            vbase = CellValue<T, VK>::base_of(b.x << S, b.y << S, r);
        } else {
            const uint32_t q = u * G + (uint32_t)min(lane, G - 1);
            if (q < ntiles) {
                const uint2 b = lambda_block(q, rb, order, W);
                vbase = CellValue<T, VK>::base_of(b.x << S, b.y << S, r);
            }
        }
        const int cnt = (int)min((uint32_t)kUnit, total - u * kUnit);
        T *dst = compact + (uint64_t)u * kUnit - lead + 4 * lane;
#pragma unroll
        for (int i = 0; i < WORDS; ++i, dst += 128) {
            uint32_t base[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                base[k] = G == 1 ? vbase
                                 : __shfl_sync(~0u, vbase, (int)((tile[i] >> (8 * k)) & 31u));
            const int e = 4 * (lane + 32 * i) - lead;
            if constexpr (sizeof(T) == 1) {
                // the four values as one word: the top bytes of the hash words
                uint32_t v[4], sel = VK == kValHash ? 0x0073u : 0x0040u;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if constexpr (VK == kValHash) v[k] = cv.hash_word(base[k], koff[i][k]);
                    else v[k] = cv(base[k], koff[i][k]);
                }
                const uint32_t w = __byte_perm(__byte_perm(v[0], v[1], sel),
                                               __byte_perm(v[2], v[3], sel), 0x5410);
                if (e >= 0 && e + 3 < cnt) {
                    *reinterpret_cast<uint32_t *>(dst) = w;
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (e + k >= 0 && e + k < cnt) dst[k] = (uint8_t)(w >> (8 * k));
                }
            } else {
                float v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) v[k] = cv.float_value(base[k], koff[i][k]);
                if (e >= 0 && e + 3 < cnt) {
                    *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (e + k >= 0 && e + k < cnt) dst[k] = v[k];
                }
            }
        }
    }
}

template <typename T, int S, bool WIDE> constexpr int write_smem_bytes()
{
    return write_stage_offset<S>() + (WIDE ? kUnitWarps * write_stage_bytes<T>() : 0);
}

template <typename T, int S, int MODE>
cudaError_t launch_move_t(int r, int order, const T *src, T *dst, cudaStream_t st,
                          const LaunchCfg &cfg)
{
    static std::atomic<int> occ{0};
    static std::atomic<uint64_t> attr{0};
    const uint32_t total = (uint32_t)pow3i(r);
    const uint64_t units = (total + kUnit - 1) / kUnit;
    unsigned grid = 1;
    auto k = compact_move_kernel<T, S, MODE>;
    constexpr int smem = IoSmem<S>::BYTES;
    cudaError_t e = dyn_smem_grid(k, smem, (units + kUnitWarps - 1) / kUnitWarps, cfg, &grid,
                                  &occ, &attr);
    if (e != cudaSuccess) return e;
    k<<<grid, kUnitThreads, smem, st>>>(src, dst, r, order, total);
    return cudaGetLastError();
}

template <typename T, int VK, int S, bool WIDE>
cudaError_t launch_write_t(int r, int order, T *compact, uint64_t vs, cudaStream_t st,
                           const LaunchCfg &cfg)
{
    static std::atomic<int> occ{0};
    const uint32_t total = (uint32_t)pow3i(r);
    const uint64_t units = (total + kUnit - 1) / kUnit;
    unsigned grid = 1;
    if constexpr (!WIDE && S >= 4) {
        auto k4 = compact_write4_kernel<T, VK, S>;
        cudaError_t e = persistent_grid(k4, kUnitThreads, 0, (units + kUnitWarps - 1) / kUnitWarps,
                                        cfg, &grid, &occ);
        if (e != cudaSuccess) return e;
        k4<<<grid, kUnitThreads, 0, st>>>(compact, r, order, total, vs);
        return cudaGetLastError();
    } else {
        static std::atomic<uint64_t> attr{0};
        auto k = compact_write_kernel<T, VK, S, WIDE>;
        constexpr int smem = write_smem_bytes<T, S, WIDE>();
        cudaError_t e = dyn_smem_grid(k, smem, (units + kUnitWarps - 1) / kUnitWarps, cfg, &grid,
                                      &occ, &attr);
        if (e != cudaSuccess) return e;
        k<<<grid, kUnitThreads, smem, st>>>(compact, r, order, total, vs);
        return cudaGetLastError();
    }
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

template <typename T, int MODE>
cudaError_t launch_move(int r, int s, int order, const T *src, T *dst, cudaStream_t st,
                        const LaunchCfg &cfg)
{
#define CALL(S) launch_move_t<T, S, MODE>(r, order, src, dst, st, cfg)
    SG_COMPACT_S_SWITCH(s, CALL)
#undef CALL
}

template <typename T, int VK, bool WIDE>
cudaError_t launch_write_vk(int r, int s, int order, T *compact, uint64_t vs, cudaStream_t st,
                            const LaunchCfg &cfg)
{
#define CALL(S) launch_write_t<T, VK, S, WIDE>(r, order, compact, vs, st, cfg)
    SG_COMPACT_S_SWITCH(s, CALL)
#undef CALL
}

template <typename T, bool WIDE>
cudaError_t launch_write_dt(int r, int s, int order, int vk, T *compact, uint64_t vs,
                            cudaStream_t st, const LaunchCfg &cfg)
{
    switch (vk) {
    case kValConst: return launch_write_vk<T, kValConst, WIDE>(r, s, order, compact, vs, st, cfg);
    case kValLinear31:
        return launch_write_vk<T, kValLinear31, WIDE>(r, s, order, compact, vs, st, cfg);
    case kValHash: return launch_write_vk<T, kValHash, WIDE>(r, s, order, compact, vs, st, cfg);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_compact_pack(int r, int s, int order, int elem, const void *grid,
                                void *compact, cudaStream_t st, const LaunchCfg &cfg)
{
    if (elem == 1)
        return launch_move<uint8_t, 0>(r, s, order, (const uint8_t *)grid, (uint8_t *)compact,
                                       st, cfg);
    return launch_move<float, 0>(r, s, order, (const float *)grid, (float *)compact, st, cfg);
}

cudaError_t launch_compact_unpack(int r, int s, int order, int elem, const void *compact,
                                  void *grid, cudaStream_t st, const LaunchCfg &cfg)
{
    if (elem == 1)
        return launch_move<uint8_t, 1>(r, s, order, (const uint8_t *)compact, (uint8_t *)grid,
                                       st, cfg);
    return launch_move<float, 1>(r, s, order, (const float *)compact, (float *)grid, st, cfg);
}

cudaError_t launch_compact_write(int r, int s, int order, int elem, int vk, void *compact,
                                 uint64_t vs, cudaStream_t st, const LaunchCfg &cfg, bool wide)
{
    if (elem == 1)
        return wide ? launch_write_dt<uint8_t, true>(r, s, order, vk, (uint8_t *)compact, vs, st, cfg)
                    : launch_write_dt<uint8_t, false>(r, s, order, vk, (uint8_t *)compact, vs, st,
                                                      cfg);
    return wide ? launch_write_dt<float, true>(r, s, order, vk, (float *)compact, vs, st, cfg)
                : launch_write_dt<float, false>(r, s, order, vk, (float *)compact, vs, st, cfg);
}

}  // namespace sg
