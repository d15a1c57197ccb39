// 3-D codec with a warp per block, for launches too small to fill the chip
// with a lane per block.  There a kernel's time is one warp's serial walk over a
// whole block per lane (some 3000 instructions); here the 32 lanes share it:
// two coefficients a lane through the transform, one bit plane a lane through
// the coder.  In the encoder nothing about a plane but its place in the stream
// depends on the planes before it: the coefficients already significant are the
// running maximum of the planes' highest ones, a plane's length follows from its
// word, and the places are the running sum of the lengths.  The decoder's walk
// from plane to plane stays serial and every lane repeats it; the rest is shared.
// Per block the chip issues several times the instructions of a lane per block, so
// codec.cu takes this path only while a launch leaves most of its warps idle
// (the rule and both sides' times stand there).  What bounds it: latency, the
// loads of message table and values in the encoder, the walk in the decoder.
#pragma once
#include "zfpx_block.cuh"

namespace zfpx {
namespace warp3 {

using namespace blk;

__device__ const uint8_t kSeqDev[64] = ZFPX_SEQ3;

// One warp's shared memory: the block's values, its planes, its stream and
// zero words after it (the decoder's 64-bit reads, the encoder's last carries).
template <int RATE>
struct Shared {
    int32_t q[64];
    uint64_t planes[32];
    uint32_t stream[2 * RATE + 4];
};

struct Words {
    const uint32_t *sm;
    __device__ __forceinline__ uint32_t get(int i) const { return sm[i]; }
};
struct Planes {
    uint64_t *sm;
    __device__ __forceinline__ void store(int k, uint64_t X) { sm[k] = X; }
};

// Bit t of lane L's result is bit L of lane t's word.
__device__ __forceinline__ uint32_t transpose(uint32_t x, int lane)
{
#pragma unroll
    for (int s = 16; s; s >>= 1) {
        const uint32_t m = s == 16 ? 0x0000ffffu : s == 8 ? 0x00ff00ffu : s == 4 ? 0x0f0f0f0fu : s == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, s);
        x = lane & s ? (x & ~m) | ((y >> s) & m) : (x & m) | ((y & m) << s);
    }
    return x;
}

// The lifting along one axis of q (steps of `stride`), a row of four per lane.
template <bool FWD>
__device__ __forceinline__ void lift_axis(int32_t *q, int lane, int stride)
{
    __syncwarp();
    if (lane < 16) {
        int32_t *r = q + (stride == 1 ? 4 * lane : stride == 4 ? 16 * (lane >> 2) + (lane & 3) : lane);
        int32_t a = r[0], b = r[stride], c = r[2 * stride], d = r[3 * stride];
        if (FWD) lift_fwd(a, b, c, d);
        else lift_inv(a, b, c, d);
        r[0] = a; r[stride] = b; r[2 * stride] = c; r[3 * stride] = d;
    }
    __syncwarp();
}

// Codes the block of values x0 (index lane) and x1 (index lane + 32) into
// sh.stream's 2 RATE words.
template <int RATE>
__device__ __forceinline__ void encode(float x0, float x1, Shared<RATE> &sh, int lane)
{
    constexpr int END = 64 * RATE;
    for (int w = lane; w < 2 * RATE + 4; w += 32) sh.stream[w] = 0u;
    const int t0 = kSeqDev[lane], t1 = kSeqDev[32 + lane];
    const uint32_t amax = __reduce_max_sync(0xffffffffu, max(f2u(x0) & 0x7fffffffu, f2u(x1) & 0x7fffffffu));
    const int E = (int)(amax >> 23);
    if (amax >= 0x00400000u && E != 255) {              // otherwise a single 0 bit
        const QuantScale qs(E);
        sh.q[lane] = qs(x0);
        sh.q[32 + lane] = qs(x1);
        lift_axis<true>(sh.q, lane, 1);
        lift_axis<true>(sh.q, lane, 4);
        lift_axis<true>(sh.q, lane, 16);
        // lane L: plane 31 - L
        const uint32_t lo = transpose(__brev(to_negabinary(sh.q[t0])), lane);
        const uint32_t hi = transpose(__brev(to_negabinary(sh.q[t1])), lane);
        const uint64_t X = ((uint64_t)hi << 32) | lo;
        int n = 64 - __clzll((long long)X);             // running maximum of the highest ones, then that before this plane
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, n, s);
            if (lane >= s) n = max(n, y);
        }
        n = __shfl_up_sync(0xffffffffu, n, 1);
        if (lane == 0) n = 0;
        // n verbatim bits, then a group bit ahead of every run of zeros and its
        // one, and a last group bit 0; the one of coefficient 63 is implied and ends the plane
        uint64_t x = shr_any(X, n);
        const int span = 64 - __clzll((long long)x), ones = __popcll(x);
        const int len = n == 64 ? 64 : n + ones + span + (n + span == 64 ? -1 : 1);
        int pos = len;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, pos, s);
            if (lane >= s) pos += y;
        }
        pos += 9 - len;
        if (lane == 0) atomicOr(sh.stream, 1u | ((uint32_t)(E + 1) << 1));
        if (pos < END) {
            const uint64_t v = X & low_mask(n);
            if (v) {
                const int w = pos >> 5, s = pos & 31;
                const uint32_t v0 = (uint32_t)v, v1 = (uint32_t)(v >> 32);
                atomicOr(sh.stream + w, v0 << s);
                atomicOr(sh.stream + w + 1, __funnelshift_l(v0, v1, s));
                atomicOr(sh.stream + w + 2, __funnelshift_l(v1, 0u, s));
            }
            int g = pos + n;                            // the next group bit
            for (int c = n; x && g < END;) {
                const int run = __ffsll((long long)x);  // zeros and the one
                atomicOr(sh.stream + (g >> 5), 1u << (g & 31));
                c += run;
                g += run;
                if (c < 64 && g < END) atomicOr(sh.stream + (g >> 5), 1u << (g & 31));
                g++;
                x = shr_any(x, run);
            }
        }
    }
    __syncwarp();
}

// The block's values (indexes lane and lane + 32) from sh.stream, its 2 RATE
// words followed by zeros.
template <int RATE>
__device__ __forceinline__ void decode(float &x0, float &x1, Shared<RATE> &sh, int lane)
{
    const int t0 = kSeqDev[lane], t1 = kSeqDev[32 + lane];
    const Words words{sh.stream};
    const uint32_t head = sh.stream[0];
    x0 = x1 = 0.0f;
    if (!(head & 1u)) return;
    const int e = (int)((head >> 1) & 0xffu);
    Planes pl{sh.planes};
    const int kmin = parse_planes64<true>(words, 9, 64 * RATE, 31, pl);   // every lane writes the same words
    __syncwarp();
    const uint64_t X = 31 - lane >= kmin ? sh.planes[31 - lane] : 0ull;
    sh.q[t0] = from_negabinary(__brev(transpose((uint32_t)X, lane)));
    sh.q[t1] = from_negabinary(__brev(transpose((uint32_t)(X >> 32), lane)));
    lift_axis<false>(sh.q, lane, 16);
    lift_axis<false>(sh.q, lane, 4);
    lift_axis<false>(sh.q, lane, 1);
    const float sc = dequant_scale(e >= 31 ? e : 31);
    x0 = e >= 31 ? dequantize_fast(sh.q[lane], sc) : dequantize_small(sh.q[lane], e);
    x1 = e >= 31 ? dequantize_fast(sh.q[32 + lane], sc) : dequantize_small(sh.q[32 + lane], e);
}

}  // namespace warp3
}  // namespace zfpx
