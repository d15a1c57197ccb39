// Per-lane shared-memory views used by the codec kernels (codec.cu, batch.cu).
// Every warp owns its tiles; lane l works in its own column, so no view
// needs a barrier other than the warp's own __syncwarp around the copies in
// and out of a tile.
#pragma once
#include <cstdint>

namespace zfpx {

// Bit planes of one block in this lane's column of a [plane][lane] tile
// (a warp touches 32 consecutive words: conflict-free).
struct SmemPlanes {
    uint64_t *sm;
    int lane;
    __device__ __forceinline__ void store(int k, uint64_t X) { sm[k * 32 + lane] = X; }
    // the low (half 0) or high (half 1) 32 bits of plane k
    __device__ __forceinline__ uint32_t load_half(int k, int half) const
    {
        return reinterpret_cast<const uint32_t *>(sm)[2 * (k * 32 + lane) + half];
    }
};

// The 32 16-bit planes of a 2-D block in this lane's column of a [word][lane]
// tile of 16 words: word k holds planes k and k + 16 as halves.
struct SmemPlanes16 {
    uint32_t *sm;
    int lane;
    __device__ __forceinline__ void store_half(int k, int, uint32_t v)
    {
        reinterpret_cast<uint16_t *>(sm)[2 * ((k & 15) * 32 + lane) + (k >> 4)] = (uint16_t)v;
    }
};
__device__ __forceinline__ uint32_t plane_pair(const SmemPlanes16 &pl, int k) { return pl.sm[k * 32 + pl.lane]; }

// Stream tile of one warp: 32-bit words in a [word][lane] layout (word i of
// lane l at i * 32 + l), so every lane reads its own column without bank
// conflicts; two zero rows follow the stream, so the 64-bit window read at
// any position before the stream's end stays inside the tile.
struct StreamTile {
    const uint32_t *sm;
    int lane;
    __device__ __forceinline__ uint32_t get(int i) const { return sm[i * 32 + lane]; }
};

// drop_group_bits of eight bits: ones at offsets p go to p - t, t ones before.  Two
// lookups give 16 bits, two more 32 (rarely needed), each byte's ones moved down
// by the ones before it; the loop over the ones runs as often as the lane with
// the most of them needs.  Decompressing a 1280 x 640 x 137 field over 8 x 8 ranks:
// 289 -> 278 us at rate 8, 361 -> 350 at rate 16; 2-D blocks (decode_block2_tile)
// 5 % (with all four lookups at once 2 % and none).
struct __align__(16) DropTable {
    uint32_t w[64];
};
constexpr DropTable make_drop_table()
{
    DropTable t{};
    for (int c = 0; c < 256; c++) {
        uint32_t out = 0;
        int ones = 0;
        for (int p = 0; p < 8; p++)
            if ((c >> p) & 1) out |= 1u << (p - ones++);
        t.w[c / 4] |= out << (8 * (c % 4));
    }
    return t;
}
static __device__ const DropTable g_drop = make_drop_table();
// A copy for the CTA; __syncthreads() before use.
template <int THREADS>
__device__ __forceinline__ void load_drop(DropTable &tab)
{
    if (THREADS >= 64) {
        if (threadIdx.x < 64) tab.w[threadIdx.x] = __ldg(g_drop.w + threadIdx.x);
    } else {
#pragma unroll
        for (int i = 0; i < 64; i += THREADS) tab.w[i + threadIdx.x] = __ldg(g_drop.w + i + threadIdx.x);
    }
}

// The same copied asynchronously by the first warp; ready after cp.async.wait_all
// by its threads and a __syncthreads().
__device__ __forceinline__ void load_drop_async(DropTable &tab)
{
    if (threadIdx.x < 16)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(tab.w + 4 * threadIdx.x)),
                     "l"(g_drop.w + 4 * threadIdx.x) : "memory");
}

// A stream tile with the table.
template <class Tile>
struct WithDrop : Tile {
    const uint8_t *drop;
    __device__ __forceinline__ WithDrop(const Tile &t, const DropTable &tab)
        : Tile(t), drop(reinterpret_cast<const uint8_t *>(tab.w)) {}
};
template <class Tile>
__device__ __forceinline__ uint32_t drop_bits(const WithDrop<Tile> &t, uint32_t V)
{
    uint32_t nw = t.drop[V & 255u] | ((uint32_t)t.drop[(V >> 8) & 255u] << (8 - __popc(V & 255u)));
    if (V >> 16)
        nw |= ((uint32_t)t.drop[(V >> 16) & 255u] << (16 - __popc(V & 0xffffu))) |
              ((uint32_t)t.drop[V >> 24] << (24 - __popc(V & 0xffffffu)));
    return nw;
}

}  // namespace zfpx
