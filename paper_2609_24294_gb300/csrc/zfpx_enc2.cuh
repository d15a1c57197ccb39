// The 2-D block encoder of the codec kernels (paper Sec. II-C; Sec. IV-B), one
// lane per 4 x 4 block; produces the stream of encode_block2 in zfpx_block.cuh
// bit for bit.
//
// Layout per warp (shared memory, each lane in its own column):
//   tile   [RATE / 2 + 1][32] 32-bit words: the lane's stream and a slack word
//          for a last plane that runs past the budget.  Zero on entry;
//          store_stream() copies the stream out and zeroes the tile again.
//   planes [16][32] 32-bit: word k holds bit planes k and k + 16 as halves.
//
// With 16 coefficients a plane takes at most 31 bits -- n verbatim bits, the
// group bit and the group-tested part of the other 16 - n -- so a plane is put
// together in one register, the part from two table lookups of eight
// coefficients each (enc3::Expand), and ORed into at most two stream words.  Once
// every coefficient is significant the remaining planes go out verbatim, two
// per word.
//
// What bounds it: instruction issue (issue slots 73 % busy, ALU pipe 72 %).  1800
// warp instructions per 32 blocks at rate 16, where one step per newly
// significant coefficient in a second pass, a 64-bit bit writer and a 32 x 32
// transpose took 2875; compressing a 1280 x 640 x 37 field level by level over 4
// x 4 ranks went from 173 to 115 us at rate 8 and from 193 to 131 us at rate 16.
#pragma once
#include <cstdint>

#include "zfpx_enc3.cuh"

namespace zfpx {
namespace enc2 {

using namespace blk;

template <int RATE>
constexpr int kWords = RATE / 2 + 1;

struct View {
    uint32_t *tile;
    uint32_t *planes;
    const uint16_t *expand;
};

template <int RATE>
struct Shared {
    uint32_t tile[kWords<RATE> * 32];
    uint32_t planes[16 * 32];
    __device__ __forceinline__ View view(const enc3::Expand &tab) { return View{tile, planes, tab.e}; }
};

template <int RATE>
__device__ __forceinline__ void encode(const float (&x)[16], bool valid, const View &sh, int lane)
{
    using enc3::red_or;
    constexpr int kSeq[16] = ZFPX_SEQ2;
    constexpr int END = 16 * RATE;
    uint32_t *tile = sh.tile + lane, *planes = sh.planes + lane;
    float am = 0.0f;
#pragma unroll
    for (int i = 0; i < 16; i += 2) am = enc3::max3_abs(am, x[i], x[i + 1]);
    const uint32_t amax = f2u(am) & 0x7fffffffu;
    const int E = (int)(amax >> 23);
    const bool act = valid && amax >= 0x00400000u && E != 255;   // else a single 0 bit
    // nothing to code in the whole warp (dry or masked areas): the streams are zero,
    // as the tile is (120 zero levels of 1280 x 640 at rate 8: 119 -> 82 us)
    if (!__any_sync(0xffffffffu, act)) return;
    const QuantScale qs(act ? E : 127);
    int32_t q[16];
#pragma unroll
    for (int i = 0; i < 16; i++) q[i] = qs(x[i]);
    xform2_fwd(q);
    // Constant blocks in the whole warp (masked areas): z empty planes, the first
    // coefficient's plane, then for every later plane its bit and an empty group --
    // the planes one by one took 511 us for 120 constant levels of 1280 x 640 at rate
    // 8, this takes 91, and the test 0.3 % of the encoder elsewhere (temperature: 354.9
    // -> 355.7 us at rate 8, 406.6 -> 407.6 at rate 16).
    uint32_t ac = 0;
#pragma unroll
    for (int i = 1; i < 16; i++) ac |= (uint32_t)q[i];
    if (__all_sync(0xffffffffu, !act || ac == 0)) {
        if (act) {
            const uint32_t dc = to_negabinary(q[0]);
            const int z = leading_zeros32(dc), at = 12 + z;
            const uint32_t rest = shr_any(reverse32(dc), z + 1);   // plane 30 - z first
            const uint64_t run = ((uint64_t)spread2(rest >> 16) << 32) | spread2(rest);
            const uint64_t lo = (1u | ((uint32_t)(E + 1) << 1)) | (z < 32 ? 3ull << (9 + z) : 0ull) | run << at;
            const uint64_t hi = run >> (64 - at);
            tile[0] = (uint32_t)lo;
            tile[32] = (uint32_t)(lo >> 32);
            tile[64] = (uint32_t)hi;
            tile[96] = (uint32_t)(hi >> 32);
        }
        return;
    }
    // negabinary: the add here, the xor as the complement of the odd planes
    uint32_t u[32];
#pragma unroll
    for (int t = 0; t < 16; t++) u[t] = (uint32_t)q[kSeq[t]] + 0xAAAAAAAAu;
    transpose16_pairs(u);
#pragma unroll
    for (int k = 0; k < 16; k++) planes[32 * k] = k & 1 ? ~u[k] : u[k];
    if (act) tile[0] = 1u | ((uint32_t)(E + 1) << 1);
    auto plane = [&](int k) { return (planes[32 * (k & 15)] >> (k & 16)) & 0xffffu; };

    const uint32_t tb = enc3::smem(tile), xb = enc3::smem(sh.expand);
    int n1 = 1, pos = 9, k = act ? 31 : -1;                      // n + 1
    uint32_t lm = 0;                                             // low n bits
#pragma unroll 1
    for (; k >= 0; k--) {
        const uint32_t X = plane(k), Y = X & ~lm, Z = Y >> (n1 - 1);
        const uint32_t c0 = Z & 255u, c1 = Z >> 8;
        uint32_t P = (X & lm) | (Y ? lm + 1u : 0u);              // verbatim bits, group bit
        const int at = n1;
        if (Y) {
            const int h = highest_set32(Y);
            n1 = h + 2;
            lm = (2u << h) - 1u;
        }
        const uint32_t last = n1 == 17 ? 1024u : 512u;           // table offset of the eight that end the part
        uint16_t e0, e1;
        asm("ld.shared.u16 %0, [%1];" : "=h"(e0) : "r"(xb + (c1 ? 0u : last) + 2u * c0));
        asm("ld.shared.u16 %0, [%1];" : "=h"(e1) : "r"(xb + (c1 ? last : 0u) + 2u * c1));
        P |= ((uint32_t)e0 | ((uint32_t)e1 << (8 + popc32(c0)))) << at;
        const uint32_t s = (uint32_t)pos & 31u, w = tb + 4u * (uint32_t)(pos & ~31);
        red_or<0>(w, P << s);
        red_or<128>(w, enc3::shr(P, 32u - s));
        pos += popc32(Y) + n1;
        if (n1 == 17 || pos >= END) break;
    }
    __syncwarp();
    if (n1 == 17) {                                              // coefficient 15's one is implied: no value or group bit
        pos -= 2;
        const uint32_t s = (uint32_t)pos & 31u;
        uint32_t prev = 0;
#pragma unroll 1
        for (int w = pos >> 5, first = 1; w < RATE / 2; w++, first = 0) {
            const uint32_t hi = k >= 1 ? plane(k - 1) : 0u, lo = k >= 2 ? plane(k - 2) : 0u;
            const uint32_t pair = hi | (lo << 16);
            k -= 2;
            if (first) red_or<0>(tb + 128u * (uint32_t)w, pair << s);
            else tile[32 * w] = enc3::funnel(prev, pair, s);
            prev = pair;
        }
    }
}

// Copies this lane's RATE / 2 stream words to dst (16-byte aligned) when
// `valid`, and zeroes the lane's tile column for the next block.
template <int RATE>
__device__ __forceinline__ void store_stream(const View &sh, int lane, bool valid, uint8_t *dst)
{
    uint32_t *tile = sh.tile + lane;
#pragma unroll
    for (int i = 0; i < RATE / 8; i++) {
        const uint4 v = make_uint4(tile[32 * (4 * i)], tile[32 * (4 * i + 1)], tile[32 * (4 * i + 2)],
                                   tile[32 * (4 * i + 3)]);
        if (valid) reinterpret_cast<uint4 *>(dst)[i] = v;
    }
#pragma unroll
    for (int w = 0; w < kWords<RATE>; w++) tile[32 * w] = 0u;
}

}  // namespace enc2
}  // namespace zfpx
