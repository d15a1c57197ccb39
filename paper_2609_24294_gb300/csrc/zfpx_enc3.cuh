// The 3-D block encoder of the codec kernels (paper Sec. II-C; Sec. IV-B),
// one lane per block, written so that the lanes of a warp never take
// different paths: every loop runs while any lane still has work, and a lane
// without work runs the same instructions on values that change nothing.
// The readings are those of encode_block3 in zfpx_block.cuh, which this
// produces bit for bit; all stream arithmetic is on 32-bit words.
//
// Layout per warp (shared memory, each lane in its own column, so the lanes'
// accesses never share a bank):
//   tile   [RATE * 2 + 4][32] 32-bit words, word w of lane l at w * 32 + l:
//          the lane's stream (2 RATE words, then four slack words that catch
//          the bits of a plane running past the budget).  Zero on entry;
//          store_stream() copies the stream out and zeroes the tile again.
//   planes [32][32] 64-bit: bit plane k of lane l at k * 32 + l; phase A
//          reuses the slots of planes already read for its list of unfinished
//          group-tested parts (entry f at slot 31 - f).
//
// The stream of a block is its header (a 1 bit and e_max + 127 in 8 bits),
// then the bit planes from the top.  Plane k, with n coefficients already
// significant, holds n verbatim bits, then (n < 64) a group bit, which is 1
// if bits n .. 63 of the plane hold ones, c of them with the highest at h;
// then, coefficient by coefficient from n, a value bit for each coefficient
// up to h, each one followed by a group bit (1 while more ones follow), the
// one at coefficient 63 implied (neither bit).  So the plane takes n + 1 bits
// without new ones and n + 1 + (h - n + 1) + c bits with them (two fewer when
// h = 63); the stream is cut at exactly 64 RATE bits.
//
// Phase A walks the planes while n < 64: it writes the verbatim bits and, for
// a plane with new ones, the group bit and the code of the first eight
// coefficients from n on, which a table gives as up to 16 bits (Expand).  Half
// the group-tested parts end there; the others wait in the list, the lane's
// remaining coefficients and their position in one 64-bit word.  Phase B: once
// n = 64 every later plane is its 64 bits verbatim, so the rest of the stream
// is the remaining planes back to back, one funnel shift per 32-bit word.  The
// list is walked last, eight coefficients per step: each lane steps through its
// own entries, so the warp takes the most steps of one lane (about 6) where
// finishing each plane on the spot would take the sum over the planes of the
// most steps of any lane (about 22).
//
// What bounds it: instruction issue, half of it on the ALU pipe (ncu: issue
// slots 63-68 % busy, ALU pipe 67-73 %, 15 to 17 warps per SM), and the latency of
// the gather.  Per 32 blocks at rate 8 about 3500 warp instructions: gather and
// store 270, block maximum and quantisation 210, lifting 610, planes 440, the
// coder the rest.  With one new coefficient per step instead of eight
// through the table, each plane's part finished in a second pass, and the block
// maximum by integer compares it was 4200; compressing a 1280 x 640 x 137
// field over 8 x 8 ranks took 336 us at rate 8 and 420 us at rate 16 then, 274
// and 348 us now.
//
// How the lanes are kept together: phase A is one straight run of instructions
// per plane (a lane without new ones codes zeros), each lane leaving it when
// its own planes are done; the list is walked while any lane has entries.
#pragma once
#include <cstdint>

#include "zfpx_block.cuh"

namespace zfpx {
namespace enc3 {

using namespace blk;

// 32-bit tile words per lane at `rate`
template <int RATE>
constexpr int kWords = 2 * RATE + 4;

// The group-tested code of eight coefficients (bit i: coefficient i is newly
// significant), LSB first: a value bit each, a group bit 1 after each one.
// Entries 256 + c: the last one's group bit 0 (the plane's part ends there);
// 512 + c: the last one is coefficient 63, whose value and group bit are not
// sent.  A CTA keeps a copy in shared memory.
struct __align__(16) Expand {
    uint16_t e[3 * 256];
};
constexpr Expand make_expand()
{
    Expand t{};
    for (int c = 0; c < 256; c++) {
        uint32_t out = 0, top = 0;
        int len = 0;
        for (int i = 0; i < 8; i++) {
            if ((c >> i) & 1) {
                top = 1u << len;
                out |= 3u << len;
                len++;
            }
            len++;
        }
        t.e[c] = (uint16_t)out;
        t.e[256 + c] = (uint16_t)(out & ~(2u * top));
        t.e[512 + c] = (uint16_t)(out & ~(3u * top));
    }
    return t;
}
static __device__ const Expand g_expand = make_expand();

// Copies the table asynchronously (every thread of the CTA takes part); ready
// after wait_expand() by every thread and a __syncthreads().
__device__ __forceinline__ void load_expand(Expand &tab)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(tab.e);
    for (int i = threadIdx.x; i < (int)sizeof(Expand) / 16; i += blockDim.x)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d + 16u * (uint32_t)i), "l"(g_expand.e + 8 * i)
                     : "memory");
}
__device__ __forceinline__ void wait_expand() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Lowest bit plane a block of exponent e_max keeps in the variable-rate modes:
// the accuracy rule, or 32 - prec in precision mode (prec > 0).
struct PlaneCut {
    int minexp, prec;
    __device__ __forceinline__ int kmin(int emax) const
    {
        if (prec > 0) return 32 - prec;
        const int k = minexp - emax + 22;
        return k < 0 ? 0 : (k > 32 ? 32 : k);
    }
};

// One warp's shared memory: tile (kWords<RATE> * 32 words, or more) and planes
// (32 * 32); the CTA's table.
struct View {
    uint32_t *tile;
    uint64_t *planes;
    const uint16_t *expand;
};

// Storage of one warp at `rate`.
template <int RATE>
struct Shared {
    uint32_t tile[kWords<RATE> * 32];
    uint64_t planes[32 * 32];
    __device__ __forceinline__ View view(const Expand &tab) { return View{tile, planes, tab.e}; }
};

__device__ __forceinline__ uint32_t shr(uint32_t a, uint32_t s)
{
    uint32_t r;
    asm("shr.b32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(s));   // s >= 32 gives 0
    return r;
}
// high word of (hi:lo) << s, 0 <= s < 32
__device__ __forceinline__ uint32_t funnel(uint32_t lo, uint32_t hi, uint32_t s) { return __funnelshift_l(lo, hi, s); }
// max(|a|, |b|, |c|), NaN if one of them is
__device__ __forceinline__ float max3_abs(float a, float b, float c)
{
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ uint32_t smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// ORs v into the shared word at address a + OFF (32-bit shared addresses: no
// 64-bit pointer arithmetic in the coder's loops)
template <int OFF>
__device__ __forceinline__ void red_or(uint32_t a, uint32_t v)
{
    asm volatile("red.shared.or.b32 [%0+%2], %1;" ::"r"(a), "r"(v), "n"(OFF) : "memory");
}

__device__ __forceinline__ void store_word(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// One step of a group-tested part: the code of the next eight coefficients
// (the low bits of zh:zl, shifted out) ORed into the lane's stream after bit A,
// with e0 at bit A itself (the plane's group bit ahead of its first eight);
// A moves on by the code's length.  `last`: table offset in bytes for the
// eight that end the part.
__device__ __forceinline__ void chunk(uint32_t &zl, uint32_t &zh, int &A, uint32_t e0, uint32_t tb, uint32_t xb,
                                      uint32_t last)
{
    const uint32_t c = zl & 255u;
    zl = __funnelshift_r(zl, zh, 8);
    zh >>= 8;
    uint16_t code;
    asm("ld.shared.u16 %0, [%1];" : "=h"(code) : "r"(xb + ((zl | zh) ? 0u : last) + 2u * c));
    const uint32_t e = 2u * code + e0, s = (uint32_t)A & 31u, w = tb + 4u * (uint32_t)(A & ~31);
    red_or<0>(w, e << s);
    red_or<128>(w, shr(e, 32u - s));
    A += 8 + popc32(c);
}

// The coder: bit planes ktop, ktop - 1, ... (plane k at planes[32 k]) into the
// lane's stream at shared address tb from bit pos on, cut at bit END; lanes that
// are not `act` code nothing.  finish_low() is called before the first plane
// below kLow is read.  LEN: returns how many bits of the stream planes ktop ..
// kmin take (END at most; 1 for an inactive lane, the zero block's bit);
// planes below kmin may then be left out of it.  Every lane of the warp calls it.
template <bool LEN, class FinishLow>
__device__ __forceinline__ int code(uint32_t tb, uint32_t xb, uint64_t *planes, int ktop, int pos, const int END,
                                    int kmin, bool act, const int kLow, FinishLow &&finish_low)
{
    // ---- phase A: planes while n < 64
    int n1 = 1, kB = -1;                               // n + 1
    uint64_t lm = 0;                                   // low n bits
    bool low_done = false;
    const uint32_t list0 = smem(planes + 32 * ktop);
    uint32_t list = list0;                             // where the next entry goes
#pragma unroll 1
    for (int k = act ? ktop : -1; k >= kmin; k--) {
        if (k == kLow - 1) {
            finish_low();
            low_done = true;
        }
        const uint64_t X = planes[32 * k];
        const uint64_t Y = X & ~lm, V = X & lm;
        const uint32_t vl = (uint32_t)V, vh = (uint32_t)(V >> 32), s = (uint32_t)pos & 31u;
        const uint32_t w = tb + 4u * (uint32_t)(pos & ~31);
        red_or<0>(w, vl << s);
        red_or<128>(w, funnel(vl, vh, s));
        red_or<256>(w, funnel(vh, 0u, s));
        // the group bit and the first eight coefficients of the group-tested
        // part now (the next eight too where more than 52 remain), the rest
        // listed; without new ones all of it is zeros
        const bool any = Y != 0;
        const uint64_t Z = Y >> (n1 - 1);
        uint32_t zl = (uint32_t)Z, zh = (uint32_t)(Z >> 32);
        int A = pos + n1 - 1;                          // the group bit
        if (any) {
            const int lead = 63 - highest_set64(Y);
            lm = ~0ull >> lead;
            n1 = 65 - lead;
        }
        pos += popc64(Y) + n1;
        const uint32_t last = n1 == 65 ? 1024u : 512u;
        chunk(zl, zh, A, any ? 1u : 0u, tb, xb, last);
        if (zh >> 20) chunk(zl, zh, A, 0u, tb, xb, last);
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(list), "r"(zl),
                     "r"(zh | (n1 == 65 ? 1u << 20 : 0u) | ((uint32_t)A << 21)) : "memory");
        if ((zl | zh) && A < END) list -= 256;
        kB = k - 1;
        if (n1 == 65 || pos >= END) break;
    }
    __syncwarp();                                      // the lanes go on together
    if (n1 == 65) pos -= 2;                            // coefficient 63's one is implied: no value or group bit

    int len = 0;
    if (LEN) len = act ? min(END, pos + (n1 == 65 ? 64 * max(0, kB - kmin + 1) : 0)) : 1;

    // ---- phase B: planes kB, kB - 1, ... verbatim from bit pos
    if (n1 == 65 && pos < END) {
        const uint32_t s = (uint32_t)pos & 31u;
        const int w0 = pos >> 5, nw = END >> 5;
        // the lowest plane read here: kB - m for the m with w0 + 2 m < nw
        if (!low_done && kB - ((nw - w0 + 1) / 2 - 1) < kLow) finish_low();
        uint32_t prev = 0;
#pragma unroll 1
        for (int wa = w0; wa < nw; wa += 2) {
            const uint64_t X = kB >= 0 ? planes[32 * kB] : 0ull;
            const uint32_t xl = (uint32_t)X, xh = (uint32_t)(X >> 32);
            if (wa == w0) red_or<0>(tb + 128u * wa, xl << s);
            else store_word(tb + 128u * wa, funnel(prev, xl, s));
            store_word(tb + 128u * (wa + 1), funnel(xl, xh, s));
            prev = xh;
            kB--;
        }
    }
    __syncwarp();

    // ---- the list: eight coefficients per step, each lane through its own
    // entries; a lane without any ORs zeros
    {
        uint32_t next = list0, zl = 0, zh = 0, last = 512u;
        int A = 0;
#pragma unroll 1
        while (__any_sync(0xffffffffu, (zl | zh) != 0 || next != list)) {
            if ((zl | zh) == 0 && next != list) {
                asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(zl), "=r"(zh) : "r"(next));
                next -= 256;
                A = (int)(zh >> 21);
                last = zh & (1u << 20) ? 1024u : 512u;
                zh &= (1u << 20) - 1u;
            }
            if (A >= END) {                            // positions only grow: nothing later is sent
                zl = zh = 0;
                next = list;
                A = 0;
            }
            chunk(zl, zh, A, 0u, tb, xb, last);
        }
    }
    return len;
}

// LEN: also returns how many bits the block's planes 31 .. kmin take (at most
// 64 RATE; 1 for a zero block), kmin by `cut` from the block's exponent; planes
// below kmin may be left out of the stream.
template <int RATE, bool LEN = false>
__device__ __forceinline__ int encode(const float (&x)[64], bool valid, const View &sh, int lane, PlaneCut cut = {})
{
    constexpr int kSeq[64] = ZFPX_SEQ3;
    constexpr int END = 64 * RATE;
    uint32_t *tile = sh.tile + lane;                   // word w at tile[32 w]
    uint64_t *planes = sh.planes + lane;               // plane k at planes[32 k]
    // largest magnitude: the bits of max |x|, NaN where a NaN takes part
    // (max.NaN propagates it), so its exponent field is 255 as for infinities
    float am = 0.0f;
#pragma unroll
    for (int i = 0; i < 64; i += 2) am = max3_abs(am, x[i], x[i + 1]);
    const uint32_t amax = f2u(am) & 0x7fffffffu;
    // E = e_max + 126; a block whose maximum is zero, below 2^-127 or not
    // finite is a single 0 bit (the tile is already zero)
    const int E = (int)(amax >> 23);
    const bool act = valid && amax >= 0x00400000u && E != 255;
    const QuantScale qs(act ? E : 127);
    int32_t q[64];
    if (act && E < 29) {                               // tiny blocks (rare): the scale in two factors
#pragma unroll
        for (int i = 0; i < 64; i++) q[i] = qs(x[i]);
    } else {
#pragma unroll
        for (int i = 0; i < 64; i++) q[i] = f2i_rz(x[i] * qs.s2);
    }
    xform3_fwd(q);
    // negabinary is (q + M) ^ M with M = 0xAA..A: the add here, the xor as the
    // complement of the odd planes once they are transposed (it folds into the
    // last stage's logic operations)
    uint32_t lo[32], hi[32];
#pragma unroll
    for (int t = 0; t < 32; t++) {
        lo[t] = (uint32_t)q[kSeq[t]] + 0xAAAAAAAAu;
        hi[t] = (uint32_t)q[kSeq[32 + t]] + 0xAAAAAAAAu;
    }
    // planes kLow .. 31 finished now, 0 .. kLow - 1 half-transposed until a
    // lane needs them (the budget rarely reaches below plane 16 at rate 8,
    // plane 8 at rate 16)
    constexpr int kLow = RATE == 8 ? 16 : 8;
    uint32_t *p32 = reinterpret_cast<uint32_t *>(planes);   // half h of plane k at p32[64 k + h]
#pragma unroll 1
    for (int half = 0; half < 2; half++) {
        if (half) {
#pragma unroll
            for (int t = 0; t < 32; t++) lo[t] = hi[t];
        }
        transpose32_part1<kLow>(lo);
#pragma unroll
        for (int k = 0; k < 32; k++) p32[64 * k + half] = k >= kLow && (k & 1) ? ~lo[k] : lo[k];
    }
    auto finish_low = [&]() {
        uint32_t a[32], b[32];
#pragma unroll
        for (int i = 0; i < kLow; i++) {
            a[i] = p32[64 * i];
            b[i] = p32[64 * i + 1];
        }
        transpose32_part2<kLow>(a);
        transpose32_part2<kLow>(b);
#pragma unroll
        for (int i = 0; i < kLow; i++) {
            const uint32_t c = i & 1 ? 0xffffffffu : 0u;
            planes[32 * i] = ((uint64_t)(b[i] ^ c) << 32) | (a[i] ^ c);
        }
    };
    if (act) tile[0] = 1u | ((uint32_t)(E + 1) << 1);
    return code<LEN>(smem(tile), smem(sh.expand), planes, 31, 9, END, LEN ? cut.kmin(E - 126) : 0, act, kLow, finish_low);
}

// Copies this lane's 2 RATE stream words to dst (16-byte aligned, the
// block's slot) with 16-byte stores when `valid`, and zeroes the lane's tile
// column for the next block.  Every lane of the warp calls it.
template <int RATE>
__device__ __forceinline__ void store_stream(const View &sh, int lane, bool valid, uint8_t *dst)
{
    uint32_t *tile = sh.tile + lane;
#pragma unroll
    for (int i = 0; i < RATE / 2; i++) {
        const uint4 v = make_uint4(tile[32 * (4 * i)], tile[32 * (4 * i + 1)], tile[32 * (4 * i + 2)],
                                   tile[32 * (4 * i + 3)]);
        if (valid) reinterpret_cast<uint4 *>(dst)[i] = v;
    }
#pragma unroll
    for (int w = 0; w < kWords<RATE>; w++) tile[32 * w] = 0u;
}

// Zeroes this lane's column of the first `words` tile words.
__device__ __forceinline__ void clear(const View &sh, int lane, int words)
{
    for (int w = 0; w < words; w++) sh.tile[32 * w + lane] = 0u;
}

}  // namespace enc3
}  // namespace zfpx
