// One ZFP fixed-rate block: encode and decode (paper Sec. II-C; Sec. IV-B).
//
// Readings (identical to the CPU oracle, stated in include/zfpx.h):
//   e_max = frexp exponent of max|x|; a block whose e_max + 127 <= 0 (max|x|
//   below 2^-127, zero included) or whose max is non-finite is a single 0 bit
//   and zero fill, decoding to +0.0;
//   header = 1 bit, then e_max + 127 in 8 bits, LSB first;
//   q = trunc(x 2^(30 - e_max)); five-step integer lifting with floor halving
//   along x, then y, then z; 3-D coefficients in total-sequency order;
//   negabinary; bit planes 31..0 with group testing, cut at exactly 4^d r
//   bits; truncated bits decode as 0; x = (float)(q 2^(e_max - 30)) with one
//   rounding to nearest even.
//
// The functions are __host__ __device__ so the same block code serves the
// kernels and can be compiled for a CPU.  On the GPU the 64 coefficients of a
// 3-D block sit in registers, their 32 bit planes are built with two 32x32
// bit-matrix transposes.  The kernels decode with decode_block*_tile and the 1-D
// functions of this file and encode 2-D and 3-D blocks with zfpx_enc2.cuh and
// zfpx_enc3.cuh.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define ZFPX_HD __host__ __device__ __forceinline__
#else
#define ZFPX_HD inline
#endif

namespace zfpx {
namespace blk {

// ----------------------------------------------------------------- primitives
ZFPX_HD uint32_t f2u(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t u; std::memcpy(&u, &x, 4); return u;
#endif
}
ZFPX_HD float u2f(uint32_t u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float x; std::memcpy(&x, &u, 4); return x;
#endif
}
ZFPX_HD uint32_t byte_perm(uint32_t a, uint32_t b, uint32_t sel)
{
#ifdef __CUDA_ARCH__
    return __byte_perm(a, b, sel);
#else
    const uint64_t v = ((uint64_t)b << 32) | a;
    uint32_t r = 0;
    for (int i = 0; i < 4; i++) r |= (uint32_t)((v >> (8 * ((sel >> (4 * i)) & 7))) & 0xff) << (8 * i);
    return r;
#endif
}
// index of the lowest set bit (x != 0)
ZFPX_HD int lowest_set(uint64_t x)
{
#ifdef __CUDA_ARCH__
    return __ffsll((long long)x) - 1;
#else
    return __builtin_ctzll(x);
#endif
}
ZFPX_HD int lowest_set32(uint32_t x)
{
#ifdef __CUDA_ARCH__
    return __ffs((int)x) - 1;
#else
    return __builtin_ctz(x);
#endif
}
ZFPX_HD int popc32(uint32_t x)
{
#ifdef __CUDA_ARCH__
    return __popc(x);
#else
    return __builtin_popcount(x);
#endif
}
ZFPX_HD int popc64(uint64_t x)
{
#ifdef __CUDA_ARCH__
    return __popcll(x);
#else
    return __builtin_popcountll(x);
#endif
}
// index of the highest set bit (x != 0)
ZFPX_HD int highest_set64(uint64_t x)
{
#ifdef __CUDA_ARCH__
    return 63 - __clzll((long long)x);
#else
    return 63 - __builtin_clzll(x);
#endif
}
ZFPX_HD int highest_set32(uint32_t x)
{
#ifdef __CUDA_ARCH__
    return 31 - __clz((int)x);
#else
    return 31 - __builtin_clz(x);
#endif
}
ZFPX_HD uint64_t low_mask(int n) { return n >= 64 ? ~0ull : ((1ull << n) - 1); }
ZFPX_HD int imin(int a, int b) { return a < b ? a : b; }

ZFPX_HD uint32_t reverse32(uint32_t x)
{
#ifdef __CUDA_ARCH__
    return __brev(x);
#else
    x = (x >> 16) | (x << 16);
    x = ((x >> 8) & 0x00ff00ffu) | ((x & 0x00ff00ffu) << 8);
    x = ((x >> 4) & 0x0f0f0f0fu) | ((x & 0x0f0f0f0fu) << 4);
    x = ((x >> 2) & 0x33333333u) | ((x & 0x33333333u) << 2);
    return ((x >> 1) & 0x55555555u) | ((x & 0x55555555u) << 1);
#endif
}
ZFPX_HD int leading_zeros32(uint32_t x)                          // 32 for 0
{
#ifdef __CUDA_ARCH__
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}
// Shifts by any s >= 0, giving 0 from the width on.
ZFPX_HD uint32_t shl_any(uint32_t x, int s)
{
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
    return r;
#else
    return s < 32 ? x << s : 0u;
#endif
}
ZFPX_HD uint32_t shr_any(uint32_t x, int s)
{
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("shr.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
    return r;
#else
    return s < 32 ? x >> s : 0u;
#endif
}
ZFPX_HD uint64_t shl_any(uint64_t x, int s)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
#else
    return s < 64 ? x << s : 0ull;
#endif
}
ZFPX_HD uint64_t shr_any(uint64_t x, int s)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
#else
    return s < 64 ? x >> s : 0ull;
#endif
}

// int32 ring arithmetic: wraps like the hardware, without signed overflow.
ZFPX_HD int32_t wadd(int32_t a, int32_t b) { return (int32_t)((uint32_t)a + (uint32_t)b); }
ZFPX_HD int32_t wsub(int32_t a, int32_t b) { return (int32_t)((uint32_t)a - (uint32_t)b); }

// ----------------------------------------------------------------- block float
ZFPX_HD int32_t f2i_rz(float y)
{
#ifdef __CUDA_ARCH__
    return __float2int_rz(y);
#else
    return (int32_t)y;
#endif
}
ZFPX_HD float i2f_rn(int32_t q)
{
#ifdef __CUDA_ARCH__
    return __int2float_rn(q);
#else
    return (float)q;
#endif
}

// q = trunc(x 2^(30 - e_max)), e_max = E - 126 (E: biased exponent of the
// block maximum, 0..254).  The scale 2^(156 - E) is applied as two exact
// power-of-two products, (x * s1) * s2 with s1 = 1 for E >= 29 and 2^64
// below, so every factor is a normal float and no product rounds wherever
// the integer part is non-zero.  No branch, no double precision.
struct QuantScale {
    float s1, s2;
    ZFPX_HD explicit QuantScale(int E)
    {
        const bool small = E < 29;
        s1 = small ? 18446744073709551616.0f : 1.0f;                 // 2^64
        s2 = u2f((uint32_t)((small ? 92 - E : 156 - E) + 127) << 23);
    }
    ZFPX_HD int32_t operator()(float x) const { return f2i_rz((x * s1) * s2); }
};

ZFPX_HD float u2f_rn(uint32_t a)
{
#ifdef __CUDA_ARCH__
    return __uint2float_rn(a);
#else
    return (float)a;
#endif
}

// x = (float)(q 2^(e - 157)) rounded once to nearest even (e = e_max + 127).
// For e >= 31 the scale is a normal float and converting q then scaling is
// exact after the conversion's single rounding.
ZFPX_HD float dequantize_fast(int32_t q, float scale) { return i2f_rn(q) * scale; }
ZFPX_HD float dequant_scale(int e) { return u2f((uint32_t)(e - 30) << 23); }

// The rare headers e < 31, where the result may be subnormal: integer
// rounding at the subnormal quantum 2^-149, no double precision.
ZFPX_HD float dequantize_small(int32_t q, int e)
{
    if (q == 0) return 0.0f;
    const uint32_t sign = q < 0 ? 0x80000000u : 0u;
    const uint32_t a = q < 0 ? 0u - (uint32_t)q : (uint32_t)q;        // |q| <= 2^31
    uint32_t bits;
    if ((uint64_t)a >= (1ull << (31 - e))) {
        // normal result (>= 2^-126): the conversion rounds once, the two
        // power-of-two scalings (2^-64, then 2^(e-93)) are exact
        bits = f2u((u2f_rn(a) * 5.42101086242752217e-20f) * u2f((uint32_t)(e + 34) << 23));
    } else if (e >= 8) {
        bits = a << (e - 8);                                             // exact subnormal
    } else {
        const int d = 8 - e;                                             // a / 2^d to nearest even
        const uint32_t m = a >> d, rem = a & ((1u << d) - 1u), half = 1u << (d - 1);
        bits = m + ((rem > half || (rem == half && (m & 1u))) ? 1u : 0u);
    }
    return u2f(bits | sign);
}

// ----------------------------------------------------------------- transform
// Five lifting steps of the 4-point decorrelating transform (floor halving).
ZFPX_HD void lift_fwd(int32_t &a, int32_t &b, int32_t &c, int32_t &d)
{
    a = wadd(a, d) >> 1; d = wsub(d, a);
    c = wadd(c, b) >> 1; b = wsub(b, c);
    a = wadd(a, c) >> 1; c = wsub(c, a);
    d = wadd(d, b) >> 1; b = wsub(b, d);
    d = wadd(d, b >> 1); b = wsub(b, d >> 1);
}
// The same steps undone in reverse order.
ZFPX_HD void lift_inv(int32_t &a, int32_t &b, int32_t &c, int32_t &d)
{
    b = wadd(b, d >> 1); d = wsub(d, b >> 1);
    b = wadd(b, d); d = wsub(wadd(d, d), b);
    c = wadd(c, a); a = wsub(wadd(a, a), c);
    b = wadd(b, c); c = wsub(wadd(c, c), b);
    d = wadd(d, a); a = wsub(wadd(a, a), d);
}

ZFPX_HD void xform3_fwd(int32_t (&q)[64])
{
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int j = 0; j < 4; j++)
            lift_fwd(q[16 * k + 4 * j], q[16 * k + 4 * j + 1], q[16 * k + 4 * j + 2], q[16 * k + 4 * j + 3]);
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int i = 0; i < 4; i++)
            lift_fwd(q[16 * k + i], q[16 * k + i + 4], q[16 * k + i + 8], q[16 * k + i + 12]);
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
        for (int i = 0; i < 4; i++)
            lift_fwd(q[4 * j + i], q[4 * j + i + 16], q[4 * j + i + 32], q[4 * j + i + 48]);
}

ZFPX_HD void xform3_inv(int32_t (&q)[64])
{
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
        for (int i = 0; i < 4; i++)
            lift_inv(q[4 * j + i], q[4 * j + i + 16], q[4 * j + i + 32], q[4 * j + i + 48]);
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int i = 0; i < 4; i++)
            lift_inv(q[16 * k + i], q[16 * k + i + 4], q[16 * k + i + 8], q[16 * k + i + 12]);
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int j = 0; j < 4; j++)
            lift_inv(q[16 * k + 4 * j], q[16 * k + 4 * j + 1], q[16 * k + 4 * j + 2], q[16 * k + 4 * j + 3]);
}

ZFPX_HD uint32_t to_negabinary(int32_t q) { return ((uint32_t)q + 0xAAAAAAAAu) ^ 0xAAAAAAAAu; }
ZFPX_HD int32_t from_negabinary(uint32_t u) { return (int32_t)((u ^ 0xAAAAAAAAu) - 0xAAAAAAAAu); }

// Coefficient (i + 4j + 16k) coded at position t: total sequency i+j+k
// ascending, ties by i^2+j^2+k^2, then by the index.
#define ZFPX_SEQ3 {0, 1, 4, 16, 5, 17, 20, 2, 8, 32, 21, 6, 9, 18, 24, 33, 36, 3, 12, 48, 22, 25,   \
                   37, 10, 34, 40, 7, 13, 19, 28, 49, 52, 26, 38, 41, 23, 29, 53, 11, 14, 35, 44, \
                   50, 56, 42, 27, 30, 39, 45, 54, 57, 15, 51, 60, 43, 46, 58, 31, 55, 61, 47,    \
                   59, 62, 63}

// In-place transpose of a 32x32 bit matrix: afterwards bit i of w[k] is
// what bit k of w[i] was.  Off-diagonal blocks are swapped at sizes 16, 8,
// 4, 2, 1; the 16- and 8-bit swaps are single byte permutes.
//
// The five stages swap one bit of the row index with the same bit of the
// column index each, so they commute and may run in any order; a stage of
// size S < L keeps each L-aligned group of words to itself.
// tstage<S, B, E>: the stage of size S on the pairs (i, i + S), B <= i < E.
template <int S, int B, int E>
ZFPX_HD void tstage(uint32_t (&w)[32])
{
#pragma unroll
    for (int i = B; i < E; i++) {
        if (i & S) continue;
        const uint32_t a = w[i], b = w[i + S];
        if (S == 16) {
            w[i] = byte_perm(a, b, 0x5410);
            w[i + S] = byte_perm(a, b, 0x7632);
        } else if (S == 8) {
            w[i] = byte_perm(a, b, 0x6240);
            w[i + S] = byte_perm(a, b, 0x7351);
        } else {
            constexpr uint32_t m = S == 4 ? 0x0F0F0F0Fu : S == 2 ? 0x33333333u : 0x55555555u;
            const uint32_t t = ((a >> S) ^ b) & m;
            w[i + S] = b ^ t;
            w[i] = a ^ (t << S);
        }
    }
}

ZFPX_HD void transpose32(uint32_t (&w)[32])
{
    tstage<16, 0, 32>(w);
    tstage<8, 0, 32>(w);
    tstage<4, 0, 32>(w);
    tstage<2, 0, 32>(w);
    tstage<1, 0, 32>(w);
}

// The transpose in two parts, for coding planes from the top: part 1
// finishes output words L..31 (L = 8 or 16) and leaves words 0..L-1 halfway;
// part 2 finishes those.
template <int L>
ZFPX_HD void transpose32_part1(uint32_t (&w)[32])
{
    tstage<16, 0, 32>(w);
    if (L == 8) tstage<8, 0, 32>(w);
    else tstage<8, 16, 32>(w);
    tstage<4, L, 32>(w);
    tstage<2, L, 32>(w);
    tstage<1, L, 32>(w);
}
template <int L>
ZFPX_HD void transpose32_part2(uint32_t (&w)[32])
{
    if (L == 16) tstage<8, 0, 16>(w);
    tstage<4, 0, L>(w);
    tstage<2, 0, L>(w);
    tstage<1, 0, L>(w);
}

// The transpose of a matrix whose words 0..L-1 are zero (L = 8 or 16): the
// stages smaller than L only touch words L..31.
template <int L>
ZFPX_HD void transpose32_zero_low(uint32_t (&w)[32])
{
#pragma unroll
    for (int i = 0; i < L; i++) w[i] = 0u;
    if (L == 16) tstage<8, 16, 32>(w);
    tstage<4, L, 32>(w);
    tstage<2, L, 32>(w);
    tstage<1, L, 32>(w);
    if (L == 8) tstage<8, 0, 32>(w);
    tstage<16, 0, 32>(w);
}

// ----------------------------------------------------------------- coder
// Group-tested coding of one bit plane X of S coefficients, n of which are
// already significant, spending at most R bits.  Writer: put(bits, len),
// 1 <= len <= 64, bits < 2^len.
template <int S, class Writer>
ZFPX_HD void code_plane(Writer &wr, uint64_t X, int &n, int &R)
{
    const int m = imin(n, R);
    if (m > 0) { wr.put(X & low_mask(m), m); R -= m; }
    while (R > 0 && n < S) {
        const uint64_t rest = X >> n;
        if (rest == 0) { wr.put(0ull, 1); R -= 1; break; }
        const int p = lowest_set(rest);              // zeros before the next one
        int len;
        uint64_t pat;
        if (n + p == S - 1) { len = p + 1; pat = 1ull; }                  // last one implied
        else { len = p + 2; pat = 1ull | (1ull << (p + 1)); }
        if (len > R) { wr.put(pat & low_mask(R), R); R = 0; break; }
        wr.put(pat, len);
        R -= len;
        n += p + 1;
    }
}

// Mirror of code_plane.  Reader: peek() = next 64 stream bits, skip(k).
// Bits past the budget are never consumed, so whatever follows the stream
// in the window cannot change the result.
template <int S, class Reader>
ZFPX_HD uint64_t decode_plane(Reader &rd, int &n, int &R)
{
    uint64_t X = 0;
    const int m = imin(n, R);
    if (m > 0) { X = rd.peek() & low_mask(m); rd.skip(m); R -= m; }
    while (R > 0 && n < S) {
        const uint64_t w = rd.peek();
        if (!(w & 1ull)) { rd.skip(1); R -= 1; break; }          // group empty
        const uint64_t after = w >> 1;                           // 63 bits after the group bit
        const int tz = after ? lowest_set(after) : 63;
        const int lim = S - 1 - n;                               // readable before the implied one
        if (tz < lim) {
            if (R < tz + 2) { R = 0; break; }                    // budget ends inside the zeros
            rd.skip(tz + 2); R -= tz + 2;
            X |= 1ull << (n + tz);
            n += tz + 1;
        } else {
            if (R < lim + 1) { R = 0; break; }
            rd.skip(lim + 1); R -= lim + 1;
            X |= 1ull << (S - 1);                                // implied
            n = S;
        }
    }
    return X;
}

// ----------------------------------------------------------------- 3-D block
// Encodes 64 values (x[i + 4j + 16k]) into exactly 64 RATE bits.  (The plain
// statement of the stream, which the CPU tests compile; the kernels' encoder is
// enc3::encode.)
//
// Two passes over the bit planes, so that lanes coding different blocks do
// not diverge per plane.  Pass 1 walks the planes with closed forms: plane k
// with n significant coefficients costs n verbatim bits, a group bit and, if
// its bits n..63 hold c ones with the highest at h, (h - n + 1) value bits
// and c group bits after them (one value bit and one group bit less when
// h = 63, whose one is implied).  It writes the verbatim bits and the first
// group bit and leaves zeros for the rest.  Pass 2 visits each newly
// significant coefficient once: the t-th one (t = 0, 1, ...) of a plane, at
// coefficient p, sits at (plane start + n + 1) + (p - n) + t, that is plane
// start + 1 + p + t, with its group bit right after; pass 2 ORs those bits
// into the stream.
//
// Writer: RATE + 2 64-bit words, the last two slack that the caller drops;
// put(bits, len) for 1 <= len <= 64, zeros(len), finish() (flush and
// zero-fill to RATE words), orw(i, v) (OR v into word i after finish).
// Planes: store(k, X) / load(k), store_half(k, h, w), 32 slots.
template <int RATE, class Writer, class Planes>
ZFPX_HD void encode_block3(const float (&x)[64], Writer &wr, Planes &pl)
{
    constexpr int kSeq[64] = ZFPX_SEQ3;
    constexpr int END = 64 * RATE;
    uint32_t amax = 0;
#pragma unroll
    for (int i = 0; i < 64; i++) {
        const uint32_t a = f2u(x[i]) & 0x7fffffffu;
        amax = a > amax ? a : amax;
    }
    // E = e_max + 126; a subnormal max in [2^-127, 2^-126) has e_max = -126 too
    const int E = (int)(amax >> 23);
    if (amax < 0x00400000u || E == 255) { wr.finish(); return; }
    const QuantScale qs(E);
    int32_t q[64];
#pragma unroll
    for (int i = 0; i < 64; i++) q[i] = qs(x[i]);
    xform3_fwd(q);
    uint32_t lo[32], hi[32];
#pragma unroll
    for (int t = 0; t < 32; t++) {
        lo[t] = to_negabinary(q[kSeq[t]]);
        hi[t] = to_negabinary(q[kSeq[32 + t]]);
    }
    // One transpose body for both halves keeps the kernel's code compact.
    // The budget rarely reaches below plane 16 at rate 8 (plane 8 at rate
    // 16): the planes above are finished here, and the words below wait
    // half-transposed in their slots until the coder first needs them.
    constexpr int kLow = RATE == 8 ? 16 : 8;
#pragma unroll 1
    for (int half = 0; half < 2; half++) {
        if (half) {
#pragma unroll
            for (int t = 0; t < 32; t++) lo[t] = hi[t];
        }
        transpose32_part1<kLow>(lo);
#pragma unroll
        for (int k = 0; k < 32; k++) pl.store_half(k, half, lo[k]);
    }
    wr.put(1ull | ((uint64_t)(E + 1) << 1), 9);
    // pass 1: plane costs, verbatim bits, first group bits.  The last plane
    // may run past the budget: its excess lands in the writer's two slack
    // words, so no bit count is clipped here.  A plane with new ones keeps
    // them in its own slot (already read) and is flagged in evm.
    int n = 0, pos = 9;
    uint32_t evm = 0;
    uint64_t lm = 0;                                             // low_mask(n)
#pragma unroll 1
    for (int k = 31; k >= 0 && pos < END; k--) {
        if (k == kLow - 1) {                                     // finish planes 0..kLow-1
            uint32_t a[32], b[32];
#pragma unroll
            for (int i = 0; i < kLow; i++) {
                a[i] = pl.load_half(i, 0);
                b[i] = pl.load_half(i, 1);
            }
            transpose32_part2<kLow>(a);
            transpose32_part2<kLow>(b);
#pragma unroll
            for (int i = 0; i < kLow; i++) pl.store(i, ((uint64_t)b[i] << 32) | a[i]);
        }
        const uint64_t X = pl.load(k);
        if (n >= 64) {                                           // every coefficient significant
            wr.put(X, 64);
            pos += 64;
            continue;
        }
        const uint64_t Y = X & ~lm;                              // candidates for significance
        wr.put((X & lm) | (Y ? lm + 1ull : 0ull), n + 1);        // verbatim bits, group bit
        int L = n + 1;
        if (Y) {
            const int h = highest_set64(Y);
            L = h < 63 ? h + 2 + popc64(Y) : h + popc64(Y);
            wr.zeros(L - n - 1);
            pl.store(k, Y);
            evm |= 1u << k;
            n = h + 1;
            lm = low_mask(n);
        }
        pos += L;
    }
    wr.finish();
    // pass 2: the bits of each newly significant coefficient, in stream
    // order.  A flagged plane's start follows from the previous one's: that
    // plane's cost, then one bit more than the significant count for each
    // plane without new ones in between.
    uint64_t rest = 0, cacc = 0;
    int ap = 0, t = 0, cw = 0, kp = 32, endp = 9, np = 0;
#pragma unroll 1
    for (;;) {
        if (!rest) {
            if (!evm) break;
            const int k = highest_set32(evm);
            evm &= ~(1u << k);
            rest = pl.load(k);
            const int start = endp + (kp - 1 - k) * (np + 1);
            ap = start + 1;
            const int h = highest_set64(rest), c = popc64(rest);
            endp = start + (h < 63 ? h + 2 + c : h + c);
            np = h + 1;
            kp = k;
            t = 0;
        }
        const int p = lowest_set(rest);
        rest &= rest - 1;
        const int A = ap + p + t;
        t++;
        if (A >= END) break;                                     // positions only grow
        // coefficient 63's one is implied; the group bit (more ones follow)
        // may fall at END, in a slack word
        const uint64_t b = (p != 63 ? 1ull : 0ull) | (rest ? 2ull : 0ull);
        const int w = A >> 6, s = A & 63;
        if (w != cw) {
            if (cacc) wr.orw(cw, cacc);
            cw = w;
            cacc = 0;
        }
        cacc |= b << s;
        if (s == 63 && (b & 2ull)) {
            wr.orw(cw, cacc);
            cw = w + 1;
            cacc = 1ull;
        }
    }
    if (cacc) wr.orw(cw, cacc);
}

// ----------------------------------------------------------------- 3-D decoder over a stream tile
// Reads are 64-bit windows funnel-shifted out of three tile words.  The tile
// holds the 2 RATE stream words and kTileZeroRows<RATE> zero words after
// them: three let the decoder read a window at the stream's end without a
// test; at rate 16 the decoder tests instead and two suffice, which is what
// lets six 3-warp CTAs share an SM.
template <int RATE>
constexpr int kTileZeroRows = RATE == 16 ? 2 : 3;
template <class Tile>
ZFPX_HD uint64_t tile_peek(const Tile &t, int pos)
{
    const int i = pos >> 5, sh = pos & 31;
    const uint32_t a = t.get(i), b = t.get(i + 1), c = t.get(i + 2);
#ifdef __CUDA_ARCH__
    const uint32_t lo = __funnelshift_r(a, b, sh), hi = __funnelshift_r(b, c, sh);
#else
    const uint32_t lo = (uint32_t)((((uint64_t)b << 32) | a) >> sh);
    const uint32_t hi = (uint32_t)((((uint64_t)c << 32) | b) >> sh);
#endif
    return ((uint64_t)hi << 32) | lo;
}

// 32 stream bits from bit pos on (tile words pos / 32 and the next).
template <class Tile>
ZFPX_HD uint32_t tile_peek32(const Tile &t, int pos)
{
    const int i = pos >> 5, sh = pos & 31;
    const uint32_t a = t.get(i), b = t.get(i + 1);
#ifdef __CUDA_ARCH__
    return __funnelshift_r(a, b, sh);
#else
    return (uint32_t)((((uint64_t)b << 32) | a) >> sh);
#endif
}

// The group-tested part of a plane, read from a window W that starts on a
// value bit.  The part is a run of tokens: "0" (a coefficient that stays
// insignificant) or "1g" (a newly significant one and the group bit after it);
// it ends at the first g = 0, or without a closing bit where the last
// coefficient is reached, whose one is implied.  Inside the part every run of
// ones starts on a value bit and alternates value, group, value, ...; a run of
// odd length ends on a value bit, and the 0 after it closes the part.  Returns
// the value ones of W read that way (exact below the part's end) and in `term`
// the closing-0 candidates.
template <class T>
ZFPX_HD T group_values(T W, T &term)
{
    constexpr T kEven = (T)0x5555555555555555ull;
    const T starts = W & ~(W << 1);
    const T even_runs = W & ~(W + (starts & kEven));            // the carry clears runs that start even
    const T val = (even_runs & kEven) | (W & ~even_runs & ~kEven);
    const T ends = W & ~(W >> 1) & ((T)~(T)0 >> 1);              // a run at the window's top may go on
    term = (ends & val) << 1;
    return val;
}

// The value ones V of a window to the coefficients they stand for: the t-th
// one, at offset p, is coefficient p - t (t ones before it took a group bit
// each), so the ones are taken lowest first and the rest moves down one place
// after each.
template <class T>
ZFPX_HD T drop_group_bits(T V)
{
    T nw = 0;
    while (V) {
        const T rest = V & (V - 1);
        nw |= V ^ rest;
        V = rest >> 1;
    }
    return nw;
}

// The same for 32 bits as the tile does it: a tile may hold a table of it.
template <class Tile>
ZFPX_HD uint32_t drop_bits(const Tile &, uint32_t V) { return drop_group_bits<uint32_t>(V); }

// The bit planes of a 64-coefficient block, planes ktop, ktop - 1, ... from
// stream bit pos on, with the budget ending at bit END: a plane's n verbatim
// bits and its group bit from one 64-bit window, its group-tested part 32 bits
// at a time (most parts close inside the first).  SAFE: the tile holds at least
// three zero words after the budget, so a window may be read at any position a
// part can reach without a test.  Stores every plane it reaches (pl.store) and
// returns the lowest; the planes below stay for the caller to clear.
// Issue-bound like the encoder; with the part taken in a 64-bit window, twice
// the instructions of a 32-bit one, decompressing a 1280 x 640 x 137 field over
// 8 x 8 ranks took 308 us at rate 8 and 386 at rate 16, now 278 and 350.
template <bool SAFE, class Tile, class Planes>
ZFPX_HD int parse_planes64(const Tile &tile, int pos, const int END, const int ktop, Planes &pl)
{
    int n = 0, k = ktop;
    uint64_t lm = 0;                                             // low_mask(n)
#pragma unroll 1
    for (; k >= 0 && n < 64; k--) {
        const int rem = END - pos;
        if (rem <= 0) return k + 1;
        const uint64_t w = tile_peek(tile, pos);
        uint64_t X = w & lm;
        if (rem <= n) { pl.store(k, w & low_mask(rem)); return k; }  // budget ends in the verbatim bits
        pos += n + 1;
        if (w & (lm + 1ull)) {                                   // the group bit (lm + 1 = bit n)
            // The tile is zero past the budget, so no one and no closing 0 can
            // be read there: a part cut by the budget shows as one that runs
            // on, and only the implied one needs the check that its zeros fit.
#pragma unroll 1
            for (;;) {
                uint32_t term;
                const uint32_t W = SAFE || pos < END ? tile_peek32(tile, pos) : 0u;
                const uint32_t val = group_values<uint32_t>(W, term);
                const uint32_t below = (term - 1u) & ~term;      // the bits before the closing 0 (all: none)
                // a value one in the window's last bit waits for its group bit
                const uint32_t V = val & (term ? below : 0x7fffffffu);
                const int B = term ? popc32(below) + 1 : 32 - (int)(val >> 31);   // bits taken
                uint32_t nw = drop_bits(tile, V);
                const int c = n + B - popc32(V);                 // the next coefficient
                if (c < 63 || (term && c == 63)) {
                    X |= (uint64_t)nw << n;
                    pos += B;
                    n = c;
                    if (term) break;
                    continue;
                }
                // the part reaches coefficient 63: the ones up to coefficient
                // 62 stand, the one at 63 is implied if the bits ahead of it fit
                nw &= shl_any(1u, 63 - n) - 1u;
                X |= (uint64_t)nw << n;
                pos += 63 - n + popc32(nw);
                if (pos > END) { pl.store(k, X); return k; }
                X |= 1ull << 63;
                n = 64;
                break;
            }
            lm = low_mask(n);
        }
        pl.store(k, X);
    }
    // every coefficient significant: the planes that the budget still holds, verbatim
#pragma unroll 1
    for (; k >= 0 && pos < END; k--, pos += 64) {
        const uint64_t w = tile_peek(tile, pos);
        pl.store(k, END - pos < 64 ? w & low_mask(END - pos) : w);
    }
    return k + 1;
}

// Decodes one block from this lane's stream tile: its planes by
// parse_planes64, then the transposes, the inverse transform and the
// dequantisation.
template <int RATE, class Tile, class Planes>
ZFPX_HD void decode_block3_tile(const Tile &tile, float (&x)[64], Planes &pl)
{
    constexpr int kSeq[64] = ZFPX_SEQ3;
    constexpr int END = 64 * RATE;
    const uint64_t head = tile_peek(tile, 0);
    if (!(head & 1ull)) {
#pragma unroll
        for (int i = 0; i < 64; i++) x[i] = 0.0f;
        return;
    }
    const int e = (int)((head >> 1) & 0xffu);
    // planes below kmin stay zero
    const int kmin = parse_planes64<kTileZeroRows<RATE> >= 3>(tile, 9, END, 31, pl);
    uint32_t lo[32], hi[32];
    // Planes below kmin are zero; when that holds for planes 0..kLow-1 in
    // every lane of the warp, the stages smaller than kLow skip them.
    constexpr int kLow = RATE == 8 ? 16 : 8;
#ifdef __CUDA_ARCH__
    const bool low_zero = __all_sync(__activemask(), kmin >= kLow);
#else
    const bool low_zero = kmin >= kLow;
#endif
    if (low_zero) {
#pragma unroll
        for (int kk = kLow; kk < 32; kk++) {
            lo[kk] = kk >= kmin ? pl.load_half(kk, 0) : 0u;
            hi[kk] = kk >= kmin ? pl.load_half(kk, 1) : 0u;
        }
        transpose32_zero_low<kLow>(lo);
        transpose32_zero_low<kLow>(hi);
    } else {
#pragma unroll
        for (int kk = 0; kk < 32; kk++) {
            lo[kk] = kk >= kmin ? pl.load_half(kk, 0) : 0u;
            hi[kk] = kk >= kmin ? pl.load_half(kk, 1) : 0u;
        }
        transpose32(lo);
        transpose32(hi);
    }
    int32_t q[64];
#pragma unroll
    for (int t = 0; t < 32; t++) {
        q[kSeq[t]] = from_negabinary(lo[t]);
        q[kSeq[32 + t]] = from_negabinary(hi[t]);
    }
    xform3_inv(q);
    if (e >= 31) {
        const float sc = dequant_scale(e);
#pragma unroll
        for (int i = 0; i < 64; i++) x[i] = dequantize_fast(q[i], sc);
    } else {
        // tiny exponents (rare): a rolled loop over a local copy
        int32_t t[64];
#pragma unroll
        for (int i = 0; i < 64; i++) t[i] = q[i];
#pragma unroll 1
        for (int i = 0; i < 64; i++) t[i] = (int32_t)f2u(dequantize_small(t[i], e));
#pragma unroll
        for (int i = 0; i < 64; i++) x[i] = u2f((uint32_t)t[i]);
    }
}

// ----------------------------------------------------------------- 2-D block
// A 2-D block is 4 x 4 values x[i + 4j] (i along axis 0, j along axis 1) of
// one level, coded into exactly 16 RATE bits (128 at rate 8, 256 at rate 16).
// Transform: the lifting along i for every j, then along j for every i.
// Coefficient (i + 4j) coded at position t: total sequency i + j ascending,
// ties by i^2 + j^2, then by the index (the 3-D rule with k = 0).
#define ZFPX_SEQ2 {0, 1, 4, 5, 2, 8, 6, 9, 3, 12, 10, 7, 13, 11, 14, 15}

ZFPX_HD void xform2_fwd(int32_t (&q)[16])
{
#pragma unroll
    for (int j = 0; j < 4; j++) lift_fwd(q[4 * j], q[4 * j + 1], q[4 * j + 2], q[4 * j + 3]);
#pragma unroll
    for (int i = 0; i < 4; i++) lift_fwd(q[i], q[i + 4], q[i + 8], q[i + 12]);
}

ZFPX_HD void xform2_inv(int32_t (&q)[16])
{
#pragma unroll
    for (int i = 0; i < 4; i++) lift_inv(q[i], q[i + 4], q[i + 8], q[i + 12]);
#pragma unroll
    for (int j = 0; j < 4; j++) lift_inv(q[4 * j], q[4 * j + 1], q[4 * j + 2], q[4 * j + 3]);
}

// Encodes x[i + 4j] into 16 RATE bits.  (The plain statement of the stream, as
// encode_block3, which the CPU tests compile; the kernels' encoder is enc2::encode,
// which the GPU tests compare with the oracle.)  The 16 coefficients' bit planes come
// from one 32x32 transpose whose lower 16 rows are zero (the coefficients sit
// in rows 16..31, so plane k is the high 16 bits of word k and the stages
// below 16 only touch the upper rows), parked in the lane's plane slots;
// the planes are coded in the two passes of encode_block3.  Writer: as for
// encode_block3 (put, zeros, finish, orw; two slack words past 16 RATE
// bits).  Planes: store_half(k, 0, w) / load_half(k, 0), 32 slots of 32 bits.
template <int RATE, class Writer, class Planes>
ZFPX_HD void encode_block2(const float (&x)[16], Writer &wr, Planes &pl)
{
    constexpr int kSeq[16] = ZFPX_SEQ2;
    uint32_t amax = 0;
#pragma unroll
    for (int i = 0; i < 16; i++) {
        const uint32_t a = f2u(x[i]) & 0x7fffffffu;
        amax = a > amax ? a : amax;
    }
    const int E = (int)(amax >> 23);
    if (amax < 0x00400000u || E == 255) { wr.finish(); return; }
    const QuantScale qs(E);
    int32_t q[16];
#pragma unroll
    for (int i = 0; i < 16; i++) q[i] = qs(x[i]);
    xform2_fwd(q);
    uint32_t w[32];
#pragma unroll
    for (int t = 0; t < 16; t++) w[16 + t] = to_negabinary(q[kSeq[t]]);
    transpose32_zero_low<16>(w);
#pragma unroll
    for (int k = 0; k < 32; k++) pl.store_half(k, 0, w[k] >> 16);
    wr.put(1ull | ((uint64_t)(E + 1) << 1), 9);
    // The two passes of encode_block3 with 16 coefficients: pass 1 writes each
    // plane's verbatim bits and first group bit and leaves zeros for its
    // group-tested part (the last plane may run into the writer's slack
    // words); planes with new ones keep them in their slot, flagged in evm.
    constexpr int END = 16 * RATE;
    int n = 0, pos = 9;
    uint32_t evm = 0, lm = 0;                                    // lm = low_mask(n)
#pragma unroll 1
    for (int k = 31; k >= 0 && pos < END; k--) {
        const uint32_t X = pl.load_half(k, 0);
        if (n >= 16) {                                           // every coefficient significant
            wr.put(X, 16);
            pos += 16;
            continue;
        }
        const uint32_t Y = X & ~lm;
        wr.put((X & lm) | (Y ? lm + 1u : 0u), n + 1);
        int L = n + 1;
        if (Y) {
            const int h = highest_set32(Y), c = popc32(Y);
            L = h < 15 ? h + 2 + c : h + c;
            wr.zeros(L - n - 1);
            pl.store_half(k, 0, Y);
            evm |= 1u << k;
            n = h + 1;
            lm = (2u << h) - 1u;
        }
        pos += L;
    }
    wr.finish();
    // pass 2: the bits of each newly significant coefficient (the t-th one of
    // a plane, at coefficient p, sits at plane start + 1 + p + t, its group
    // bit right after; coefficient 15's one is implied)
    uint32_t rest = 0;
    uint64_t cacc = 0;
    int ap = 0, t = 0, cw = 0, kp = 32, endp = 9, np = 0;
#pragma unroll 1
    for (;;) {
        if (!rest) {
            if (!evm) break;
            const int k = highest_set32(evm);
            evm &= ~(1u << k);
            rest = pl.load_half(k, 0);
            const int start = endp + (kp - 1 - k) * (np + 1);
            ap = start + 1;
            const int h = highest_set32(rest), c = popc32(rest);
            endp = start + (h < 15 ? h + 2 + c : h + c);
            np = h + 1;
            kp = k;
            t = 0;
        }
        const int p = lowest_set32(rest);
        rest &= rest - 1u;
        const int A = ap + p + t;
        t++;
        if (A >= END) break;                                     // positions only grow
        const uint64_t b = (p != 15 ? 1ull : 0ull) | (rest ? 2ull : 0ull);
        const int w = A >> 6, sh = A & 63;
        if (w != cw) {
            if (cacc) wr.orw(cw, cacc);
            cw = w;
            cacc = 0;
        }
        cacc |= b << sh;
        if (sh == 63 && (b & 2ull)) {
            wr.orw(cw, cacc);
            cw = w + 1;
            cacc = 1ull;
        }
    }
    if (cacc) wr.orw(cw, cacc);
}

// Planes k and k + 16 of a 2-D block as the halves of one word.
template <class Planes>
ZFPX_HD uint32_t plane_pair(const Planes &pl, int k)
{
    return pl.load_half(k, 0) | (pl.load_half(k + 16, 0) << 16);
}

// The bit planes of 16 words as 16 pairs and back: afterwards bit i of the low
// (high) half of w[k] is what bit k (k + 16) of w[i] was.
ZFPX_HD void transpose16_pairs(uint32_t (&w)[32])
{
    tstage<8, 0, 16>(w);
    tstage<4, 0, 16>(w);
    tstage<2, 0, 16>(w);
    tstage<1, 0, 16>(w);
}

// Decodes one 2-D block from this lane's stream tile (2 RATE / 4 words of 32
// bits, then at least one zero word).  With 16 coefficients a plane takes at most
// 31 bits (n verbatim bits, the group bit, and a value and a group bit for
// each of the rest but the implied last one), so one 32-bit window holds it.
// Issue-bound; with 64-bit windows and 32-word transposes decompressing a 1280
// x 640 x 37 field level by level over 4 x 4 ranks took 172 us at rate 8 and 201
// at rate 16, now 117 and 132.
template <int RATE, class Tile, class Planes>
ZFPX_HD void decode_block2_tile(const Tile &tile, float (&x)[16], Planes &pl)
{
    constexpr int kSeq[16] = ZFPX_SEQ2;
    constexpr int END = 16 * RATE;
    const uint32_t head = tile_peek32(tile, 0);
    if (!(head & 1u)) {
#pragma unroll
        for (int i = 0; i < 16; i++) x[i] = 0.0f;
        return;
    }
    const int e = (int)((head >> 1) & 0xffu);
    // The tile is zero past the budget, so a part the budget cuts reads on as
    // zeros: no one and no closing 0 appear there, and only the implied one of
    // coefficient 15 needs the check that its bits fit (the 3-D decoder's
    // reading, with 16 coefficients).
    int pos = 9, n = 0, k = 31;
    uint32_t lm = 0;                                             // low n bits
    bool cut = false;
#pragma unroll 1
    for (; k >= 0 && n < 16 && pos < END && !cut; k--) {
        const int rem = END - pos;
        const uint32_t W = tile_peek32(tile, pos);
        uint32_t X = W & lm;
        pos += n + 1;
        if (rem > n && (W & (lm + 1u))) {                        // the group bit
            uint32_t term;
            const uint32_t val = group_values<uint32_t>(W >> (n + 1), term);
            const uint32_t below = (term - 1u) & ~term;          // the bits before the closing 0 (all: none)
            const uint32_t V = val & below;
            uint32_t nw = drop_bits(tile, V);
            // ones past coefficient 14 lie beyond a part that ends at the implied one
            const uint32_t keep = (1u << (15 - n)) - 1u;
            const bool over = (nw & ~keep) != 0u;
            nw &= keep;
            X |= nw << n;
            if (!over && term) {                                 // closed by a 0 below coefficient 15
                const int T = popc32(below);
                n += T - popc32(V) + 1;
                lm = (1u << n) - 1u;
                pos += T + 1;
            } else {
                const int E = 15 - n + popc32(nw);               // the part ends at the implied one
                if (E > END - pos) {
                    cut = true;
                } else {
                    X |= 0x8000u;
                    n = 16;
                }
                pos += E;
            }
        }
        pl.store_half(k, 0, X);                                  // past the budget W and so X is 0
    }
    // every coefficient significant: the planes that the budget still holds, verbatim
#pragma unroll 1
    for (; k >= 0 && pos < END && !cut; k--, pos += 16) pl.store_half(k, 0, tile_peek32(tile, pos) & 0xffffu);
#pragma unroll 1
    for (; k >= 0; k--) pl.store_half(k, 0, 0u);
    // u ^ 0xAA..A of the negabinary map as the complement of the odd planes
    uint32_t w[32];
#pragma unroll
    for (int i = 0; i < 16; i++) w[i] = i & 1 ? ~plane_pair(pl, i) : plane_pair(pl, i);
    transpose16_pairs(w);
    int32_t q[16];
#pragma unroll
    for (int t = 0; t < 16; t++) q[kSeq[t]] = (int32_t)(w[t] - 0xAAAAAAAAu);
    xform2_inv(q);
    if (e >= 31) {
        const float sc = dequant_scale(e);
#pragma unroll
        for (int i = 0; i < 16; i++) x[i] = dequantize_fast(q[i], sc);
    } else {
        // tiny exponents (rare): a rolled loop over a local copy
        int32_t t[16];
#pragma unroll
        for (int i = 0; i < 16; i++) t[i] = q[i];
#pragma unroll 1
        for (int i = 0; i < 16; i++) t[i] = (int32_t)f2u(dequantize_small(t[i], e));
#pragma unroll
        for (int i = 0; i < 16; i++) x[i] = u2f((uint32_t)t[i]);
    }
}

// ----------------------------------------------------------------- 1-D block
// A 1-D block is 4 RATE <= 64 bits, returned in one word (LSB = first bit).
struct RegWriter {
    uint64_t acc;
    int nb;
    ZFPX_HD void put(uint64_t bits, int len) { acc |= bits << nb; nb += len; }
};
struct WordReader {
    uint64_t w;
    int off;
    ZFPX_HD uint64_t peek() const { return off < 64 ? (w >> off) : 0ull; }
    ZFPX_HD void skip(int k) { off += k; }
};

// With four coefficients the code has little structure left, and both coders
// take it by runs instead of plane by plane.  While n coefficients are
// significant and no new one appears, a plane is n verbatim bits and a 0, so a
// run of such planes is a bit interleave: of nothing (n = 0), of one
// coefficient with zeros (n = 1) or of two with zeros (n = 2).  From n = 3 on a
// plane is just its four bits: with n = 3 the group bit says whether
// coefficient 3, whose one is then implied, is new.  So a block is at most
// three runs, each ended by one plane with new ones, and a tail of 4-bit
// planes; the length of a run is a count of leading zeros.  A plane with new
// ones is coded from a table built from code_plane / decode_plane: encoder
// entry (n, X) = code bits 0..6, length bits 7..9, new n bits 10..12; decoder
// entry (n, the next seven bits) = X bits 0..3, length bits 4..6, new n bits
// 7..9.
// The encoder's output is the first 4 RATE bits of the unbounded code, which
// is the width of the word it builds: what runs past the budget shifts out.
// The decoder reads zeros past the budget, which add no one except, in a plane
// with new ones that the budget cuts, the implied one of coefficient 3, which
// needs the whole plane and so is dropped.
// The planes are taken bit-reversed (plane 31 in bit 0), in stream order.
// This bounds the 1-D kernels by instruction issue still, at about half the
// instructions of one table lookup per plane.
struct Plane4Enc {
    uint16_t e[5 * 16];
};
struct Plane4Dec {
    uint16_t d[5 * 128];
};

ZFPX_HD uint16_t plane4_enc_entry(int n, uint32_t X)
{
    RegWriter wr{0ull, 0};
    int nn = n, R = 64;
    code_plane<4>(wr, X, nn, R);
    return (uint16_t)((uint32_t)wr.acc | ((uint32_t)wr.nb << 7) | ((uint32_t)nn << 10));
}

ZFPX_HD uint16_t plane4_dec_entry(int n, uint32_t w7)
{
    WordReader rd{w7, 0};
    int nn = n, R = 64;
    const uint32_t X = (uint32_t)decode_plane<4>(rd, nn, R);
    return (uint16_t)(X | ((uint32_t)rd.off << 4) | ((uint32_t)nn << 7));
}

// Fills a table with `nthreads` threads, thread `t` taking every nthreads-th
// entry (the caller synchronises).
ZFPX_HD void plane4_fill(Plane4Enc &tab, int t, int nthreads)
{
    for (int i = t; i < 5 * 16; i += nthreads) tab.e[i] = plane4_enc_entry(i >> 4, (uint32_t)i & 15u);
}
ZFPX_HD void plane4_fill(Plane4Dec &tab, int t, int nthreads)
{
    for (int i = t; i < 5 * 128; i += nthreads) tab.d[i] = plane4_dec_entry(i >> 7, (uint32_t)i & 127u);
}

// Bit i of x to bit 2 i, 3 i or 4 i (16, 10 and 8 bits fit a 32-bit word), and
// back from the bits there.
ZFPX_HD uint32_t spread2(uint32_t x)
{
    x &= 0xffffu;
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    return (x | (x << 1)) & 0x55555555u;
}
ZFPX_HD uint32_t spread3(uint32_t x)
{
    x &= 0x3ffu;
    x = (x | (x << 16)) & 0x030000ffu;
    x = (x | (x << 8)) & 0x0300f00fu;
    x = (x | (x << 4)) & 0x030c30c3u;
    return (x | (x << 2)) & 0x09249249u;
}
ZFPX_HD uint32_t spread4(uint32_t x)
{
    x &= 0xffu;
    x = (x | (x << 12)) & 0x000f000fu;
    x = (x | (x << 6)) & 0x03030303u;
    return (x | (x << 3)) & 0x11111111u;
}
ZFPX_HD uint32_t gather2(uint32_t x)
{
    x &= 0x55555555u;
    x = (x | (x >> 1)) & 0x33333333u;
    x = (x | (x >> 2)) & 0x0f0f0f0fu;
    x = (x | (x >> 4)) & 0x00ff00ffu;
    return (x | (x >> 8)) & 0xffffu;
}
ZFPX_HD uint32_t gather3(uint32_t x)
{
    x &= 0x09249249u;
    x = (x | (x >> 2)) & 0x030c30c3u;
    x = (x | (x >> 4)) & 0x0300f00fu;
    x = (x | (x >> 8)) & 0x030000ffu;
    return (x | (x >> 16)) & 0x3ffu;
}
ZFPX_HD uint32_t gather4(uint32_t x)
{
    x &= 0x11111111u;
    x = (x | (x >> 3)) & 0x03030303u;
    x = (x | (x >> 6)) & 0x000f000fu;
    return (x | (x >> 12)) & 0xffu;
}

struct SpreadBits {                                                // spread4 by shifts
    ZFPX_HD uint32_t operator()(uint32_t x) const { return spread4(x); }
};

// The word a 1-D block's 4 RATE bits fill, and the interleaves in it: as many
// planes as can matter from bit 9 on.
template <int RATE>
struct Word1 {
    typedef uint64_t T;
    ZFPX_HD static T runs1(uint32_t a) { return ((T)spread2(a >> 16) << 32) | spread2(a); }
    ZFPX_HD static T runs2(uint32_t a, uint32_t b)
    {
        return ((T)(spread3(a >> 10) | (spread3(b >> 10) << 1)) << 30) | spread3(a) | (spread3(b) << 1);
    }
    template <class Spread>
    ZFPX_HD static T tail(const uint32_t (&v)[4], int p, const Spread &spread)
    {
        T r = 0;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const uint32_t a = shr_any(v[i], p);
            r |= (((T)spread(a >> 8) << 32) | spread(a)) << i;
        }
        return r;
    }
    ZFPX_HD static uint32_t of_runs1(T w) { return gather2((uint32_t)w) | (gather2((uint32_t)(w >> 32)) << 16); }
    ZFPX_HD static uint32_t of_runs2(T w) { return gather3((uint32_t)w) | (gather3((uint32_t)(w >> 30)) << 10); }
    ZFPX_HD static uint32_t of_tail(T w, int i)
    {
        return gather4((uint32_t)(w >> i)) | (gather4((uint32_t)(w >> 32) >> i) << 8);
    }
    static constexpr T kGroup1 = 0xaaaaaaaaaaaaaaaaull, kGroup2 = 0x4924924924924924ull;
    ZFPX_HD static int low(T w) { return lowest_set(w); }
};
template <>
struct Word1<8> {
    typedef uint32_t T;
    ZFPX_HD static T runs1(uint32_t a) { return spread2(a); }
    ZFPX_HD static T runs2(uint32_t a, uint32_t b) { return spread3(a) | (spread3(b) << 1); }
    template <class Spread>
    ZFPX_HD static T tail(const uint32_t (&v)[4], int p, const Spread &spread)
    {
        T r = 0;
#pragma unroll
        for (int i = 0; i < 4; i++) r |= spread(shr_any(v[i], p)) << i;
        return r;
    }
    ZFPX_HD static uint32_t of_runs1(T w) { return gather2(w); }
    ZFPX_HD static uint32_t of_runs2(T w) { return gather3(w); }
    ZFPX_HD static uint32_t of_tail(T w, int i) { return gather4(w >> i); }
    static constexpr T kGroup1 = 0xaaaaaaaau, kGroup2 = 0x24924924u;
    ZFPX_HD static int low(T w) { return lowest_set32(w); }
};

// Encodes K blocks x[b][0..3]; w[b] = the block's 4 RATE bits.
template <int RATE, int K, class Spread = SpreadBits>
ZFPX_HD void encode_blocks1(const float (&x)[K][4], const Plane4Enc &tab, uint64_t (&w)[K], const Spread &spread = Spread())
{
    typedef typename Word1<RATE>::T T;
#pragma unroll
    for (int b = 0; b < K; b++) {
        uint32_t amax = 0;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const uint32_t a = f2u(x[b][i]) & 0x7fffffffu;
            amax = a > amax ? a : amax;
        }
        const int E = (int)(amax >> 23);
        const bool zero = amax < 0x00400000u || E == 255;          // a single 0 bit
        const QuantScale qs(zero ? 127 : E);
        int32_t q0 = qs(x[b][0]), q1 = qs(x[b][1]), q2 = qs(x[b][2]), q3 = qs(x[b][3]);
        lift_fwd(q0, q1, q2, q3);
        const uint32_t u[4] = {to_negabinary(q0), to_negabinary(q1), to_negabinary(q2), to_negabinary(q3)};
        const uint32_t v[4] = {reverse32(u[0]), reverse32(u[1]), reverse32(u[2]), reverse32(u[3])};
        const uint32_t o2 = u[2] | u[3], o1 = u[1] | o2, o0 = u[0] | o1;
        T r = (T)(1u | ((uint32_t)(E + 1) << 1));                  // header, 9 bits
        int n = 0, pos = 9, p = 0;                                 // p: the next plane (31 - p)
        // a plane with new ones: its table entry, for plane 31 - e
        auto event = [&](int e) {
            const uint32_t X = (shr_any(v[0], e) & 1u) | ((shr_any(v[1], e) & 1u) << 1) |
                               ((shr_any(v[2], e) & 1u) << 2) | ((shr_any(v[3], e) & 1u) << 3);
            const uint32_t c = tab.e[n * 16 + (int)X];
            r |= shl_any((T)(c & 127u), pos);
            pos += (int)((c >> 7) & 7u);
            n = (int)(c >> 10);
            p = e + 1;
        };
        const int e0 = leading_zeros32(o0);                        // zeros up to the first one
        pos += e0;
        if (e0 < 32) event(e0);
        if (n == 1) {
            const int e1 = leading_zeros32(o1), run = e1 - p;
            r |= shl_any(Word1<RATE>::runs1(shr_any(v[0], p) & (shl_any(1u, run) - 1u)), pos);
            pos += 2 * run;
            if (e1 < 32) event(e1);
        }
        if (n == 2) {
            const int e2 = leading_zeros32(o2), run = e2 - p;
            const uint32_t m = shl_any(1u, run) - 1u;
            r |= shl_any(Word1<RATE>::runs2(shr_any(v[0], p) & m, shr_any(v[1], p) & m), pos);
            pos += 3 * run;
            if (e2 < 32) event(e2);
        }
        if (n >= 3) r |= shl_any(Word1<RATE>::tail(v, p, spread), pos);
        w[b] = zero ? 0ull : (uint64_t)r;
    }
}

// The planes from p on of w, every coefficient significant, into v by shifts.
struct TailBits {
    template <class Word>
    ZFPX_HD void add(typename Word::T w, int p, uint32_t (&v)[4]) const
    {
#pragma unroll
        for (int i = 0; i < 4; i++) v[i] |= shl_any(Word::of_tail(w, i), p);
    }
};

// Decodes K blocks from their 4 RATE-bit words.
template <int RATE, int K, class Tail = TailBits>
ZFPX_HD void decode_blocks1(const uint64_t (&win)[K], const Plane4Dec &tab, float (&x)[K][4], const Tail &tail = Tail())
{
    typedef typename Word1<RATE>::T T;
    constexpr int END = 4 * RATE;
#pragma unroll
    for (int b = 0; b < K; b++) {
        T w = (T)win[b] >> 9;
        uint32_t v[4] = {0u, 0u, 0u, 0u};                          // planes from 31 down, bit-reversed
        int n = 0, pos = 9, p = 0;
        // a plane with new ones at the start of w, for plane 31 - e (e < 32)
        auto event = [&](int e) {
            const uint32_t d = tab.d[n * 128 + (int)((uint32_t)w & 127u)];
            const int len = (int)((d >> 4) & 7u);
            const bool cut = len > END - pos;                      // the budget ends inside it
            const uint32_t X = cut ? d & 7u : d & 15u;
#pragma unroll
            for (int i = 0; i < 4; i++) v[i] |= ((X >> i) & 1u) << e;
            w = cut ? (T)0 : w >> len;
            pos += len;
            n = cut ? -1 : (int)(d >> 7);
            p = e + 1;
        };
        if (w) {
            const int e0 = Word1<RATE>::low(w);
            w >>= e0;
            pos += e0;
            if (e0 < 32) event(e0);
        }
        if (n == 1) {
            const T t = w & Word1<RATE>::kGroup1;
            const int run = t ? Word1<RATE>::low(t) >> 1 : 32;
            const T m = shl_any((T)1, 2 * run) - (T)1;
            v[0] |= shl_any(Word1<RATE>::of_runs1(w & m), p);
            w = shr_any(w, 2 * run);
            pos += 2 * run;
            if (p + run < 32 && t) event(p + run);
            else n = -1;
        }
        if (n == 2) {
            const T t = w & Word1<RATE>::kGroup2;
            const int run = t ? (Word1<RATE>::low(t) * 43) >> 7 : 32;    // the group bits are at 3 i + 2
            const T m = shl_any((T)1, 3 * run) - (T)1;
            v[0] |= shl_any(Word1<RATE>::of_runs2(w & m), p);
            v[1] |= shl_any(Word1<RATE>::of_runs2((w & m) >> 1), p);
            w = shr_any(w, 3 * run);
            pos += 3 * run;
            if (p + run < 32 && t) event(p + run);
            else n = -1;
        }
        if (n >= 3) tail.template add<Word1<RATE>>(w, p, v);
        if (!(win[b] & 1ull)) {
            x[b][0] = x[b][1] = x[b][2] = x[b][3] = 0.0f;
            continue;
        }
        const int e = (int)((win[b] >> 1) & 0xffu);
        int32_t q0 = from_negabinary(reverse32(v[0])), q1 = from_negabinary(reverse32(v[1]));
        int32_t q2 = from_negabinary(reverse32(v[2])), q3 = from_negabinary(reverse32(v[3]));
        lift_inv(q0, q1, q2, q3);
        if (e >= 31) {
            const float sc = dequant_scale(e);
            x[b][0] = dequantize_fast(q0, sc); x[b][1] = dequantize_fast(q1, sc);
            x[b][2] = dequantize_fast(q2, sc); x[b][3] = dequantize_fast(q3, sc);
        } else {
            x[b][0] = dequantize_small(q0, e); x[b][1] = dequantize_small(q1, e);
            x[b][2] = dequantize_small(q2, e); x[b][3] = dequantize_small(q3, e);
        }
    }
}

}  // namespace blk
}  // namespace zfpx
