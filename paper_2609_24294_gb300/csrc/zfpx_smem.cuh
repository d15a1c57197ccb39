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
    __device__ __forceinline__ uint64_t load(int k) const { return sm[k * 32 + lane]; }
    // the low (half 0) or high (half 1) 32 bits of plane k
    __device__ __forceinline__ void store_half(int k, int half, uint32_t v)
    {
        reinterpret_cast<uint32_t *>(sm)[2 * (k * 32 + lane) + half] = v;
    }
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

}  // namespace zfpx
