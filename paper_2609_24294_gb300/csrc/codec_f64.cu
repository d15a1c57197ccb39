// float64 fields, 3-D blocks, fixed rate (raw arrays).  The float32 method
// with the double format's sizes (readings identical in the CPU oracle):
// e_max = frexp exponent of max|x|; zero block (one 0 bit) if max|x| is 0,
// below 2^-1023 or non-finite; header = a 1 bit and e_max + 1023 in 11 bits;
// q = trunc(x 2^(62 - e_max)) in int64; the five-step lifting in int64 along
// x, y, z; the 3-D coefficient order; 64-bit negabinary; group-tested bit
// planes 63 .. 0 cut at exactly 64 r bits; decode x = q 2^(e_max - 62)
// rounded once to nearest even.
//
// One lane per block, 32 consecutive blocks per warp.  A block's 64 int64
// values live in the lane's registers (128 of them) through the gather,
// quantisation, transform and negabinary map; the bit planes come from 32x32
// register transposes (low / high 32 coefficients x low / high 32 bits) and wait
// in shared memory ([plane][lane]) for the coder, the float32 encoder's
// (enc3::code), which writes the lane's column of a [word][lane] stream tile.  The
// low 32 planes are transposed only where a budget reaches them (from about 24
// bits per value on); until then the encoder parks the coefficients' low words
// in their slots, and the decoder knows them to be zero.  Rates 1 .. 32 bits
// per value.
// What bounds it: latency at ten to twelve warps per SM (registers and shared
// memory), and the int64 arithmetic.  With all four transposes, a per-lane coder
// that wrote bit by bit through 64-bit words and 64-bit index divisions, a 640 x
// 320 x 91 field took 175 / 153 us to encode / decode at rate 8, 207 / 182 at 16
// and 235 / 219 at 32, now 127 / 127, 139 / 156 and 164 / 211.
#include <algorithm>
#include <climits>
#include <cuda_runtime.h>

#include "zfpx_internal.h"
#include "zfpx_block.cuh"
#include "zfpx_smem.cuh"
#include "zfpx_enc3.cuh"

namespace zfpx {
namespace {

using namespace blk;

constexpr int kMaxRate = 32;
constexpr int kEncWarps = 2;            // the encoder's warps share its table
constexpr int kF64MinWarps = 10;        // warps per SM the registers are budgeted for
constexpr uint64_t kNega64 = 0xAAAAAAAAAAAAAAAAull;

__device__ __forceinline__ int64_t add64(int64_t a, int64_t b) { return (int64_t)((uint64_t)a + (uint64_t)b); }
__device__ __forceinline__ int64_t sub64(int64_t a, int64_t b) { return (int64_t)((uint64_t)a - (uint64_t)b); }

// One lane's stream in a [64-bit word][lane] tile; peek(pos) = the 64 stream
// bits from bit pos on (reads words pos / 64 and pos / 64 + 1).
struct Tile64 {
    const uint64_t *sm;
    int lane;
    __device__ __forceinline__ uint64_t peek(int pos) const
    {
        const int w = pos >> 6, sh = pos & 63;
        const uint64_t a = sm[w * 32 + lane];
        return sh ? (a >> sh) | (sm[(w + 1) * 32 + lane] << (64 - sh)) : a;
    }
};

// The same stream as 32-bit words (word i is the low half of 64-bit word
// i / 2 for even i, the high half for odd i), for the float32 path's plane
// parser.
struct Tile64As32 {
    const uint32_t *sm;
    int lane;
    __device__ __forceinline__ uint32_t get(int i) const { return sm[2 * ((i >> 1) * 32 + lane) + (i & 1)]; }
};

struct Geom64 {
    int64_t n[3], s[3];
    int64_t bx, by, nblocks, nunits;
    uint32_t bxm, bym;      // 32-bit divisors of bx and by (used while the block count fits)
    int32_t bxl, byl;
    int rate;
    int vec;        // unit x stride, even y and z strides, 16-byte aligned base: rows of a block are
                    // two 16-byte moves each
};

__device__ __forceinline__ void block_origin(const Geom64 &g, int64_t b, int64_t &x0, int64_t &y0, int64_t &z0)
{
    if (g.nblocks <= INT_MAX) {
        const uint32_t t = divu((uint32_t)b, g.bxm, g.bxl), z = divu(t, g.bym, g.byl);
        x0 = 4 * (int64_t)((uint32_t)b - t * (uint32_t)g.bx);
        y0 = 4 * (int64_t)(t - z * (uint32_t)g.by);
        z0 = 4 * (int64_t)z;
        return;
    }
    const int64_t t = b / g.bx;
    x0 = 4 * (b - t * g.bx);
    y0 = 4 * (t % g.by);
    z0 = 4 * (t / g.by);
}

// exponent: 0 for a zero block, else e_max + 1023 (1 .. 2046)
// from the high word of the largest magnitude
__device__ __forceinline__ int block_exponent(uint32_t amax_hi)
{
    const int E = (int)(amax_hi >> 20);
    if (E == 2047 || amax_hi < 0x00080000u) return 0;            // non-finite, or below 2^-1023
    return E == 0 ? 1 : E + 1;                                   // frexp exponent + 1023
}

// The quantisation and the dequantisation of the common case in integer
// operations on the bits: on this GPU the float64 pipe runs at a small
// fraction of the integer one, and these are the path's only float64
// arithmetic.  Both give the bits of the float64 formulas exactly (the
// products by powers of two there are exact, so only the truncation and the
// one rounding of q to 53 bits remain).
//
// q = trunc(x 2^(62 - e_max)), e = e_max + 1023 the block's exponent: x =
// +-M 2^(E - 1075) with E the biased exponent (taken as 1 for subnormals) and
// M the significand (with the implicit bit for normals), so |q| is M shifted
// left by E + 10 - e (at most 10, in the value whose exponent set e): M 2^10
// shifted right by e - E.
__device__ __forceinline__ int64_t quantize64(uint64_t bits, int e)
{
    const uint32_t hi = (uint32_t)(bits >> 32), lo = (uint32_t)bits;
    const int E = (int)((hi >> 20) & 0x7ffu);
    const uint32_t m = (hi & 0x000fffffu) | (E ? 0x00100000u : 0u);
    const uint64_t M = ((uint64_t)__funnelshift_l(lo, m, 10) << 32) | (lo << 10);
    const uint64_t a = shr_any(M, e - (E ? E : 1));
    const uint64_t s = (uint64_t)(int64_t)((int32_t)hi >> 31);   // all ones for a negative value
    return (int64_t)((a ^ s) - s);
}

// x = q 2^(e - 1085) rounded once to nearest even, for e >= 63, where every
// non-zero result is normal (or, past the largest double, infinite): the one
// rounding is the conversion of q, and the power-of-two scaling an integer
// add to the exponent field (infinity where it passes the largest exponent).
__device__ __forceinline__ double dequantize64_normal(int64_t q, int e)
{
    const uint64_t b = (uint64_t)__double_as_longlong(__ll2double_rn(q));
    const int E = (int)((b >> 52) & 0x7ffu);                     // 0 only for q = 0
    const int ne = E + e - 1085;                                 // >= 1 for q != 0
    const uint64_t r = ne >= 2047 ? (b & 0x8000000000000000ull) | 0x7ff0000000000000ull
                                  : b + ((uint64_t)(int64_t)(e - 1085) << 52);
    return __longlong_as_double((long long)(E ? r : b));
}

// The 3-D transform on a block held in registers (int64 v[i + 4j + 16k]).
__device__ __forceinline__ void lift_fwd64r(int64_t &a, int64_t &b, int64_t &c, int64_t &d)
{
    a = add64(a, d) >> 1; d = sub64(d, a);
    c = add64(c, b) >> 1; b = sub64(b, c);
    a = add64(a, c) >> 1; c = sub64(c, a);
    d = add64(d, b) >> 1; b = sub64(b, d);
    d = add64(d, b >> 1); b = sub64(b, d >> 1);
}
__device__ __forceinline__ void lift_inv64r(int64_t &a, int64_t &b, int64_t &c, int64_t &d)
{
    b = add64(b, d >> 1); d = sub64(d, b >> 1);
    b = add64(b, d); d = sub64(add64(d, d), b);
    c = add64(c, a); a = sub64(add64(a, a), c);
    b = add64(b, c); c = sub64(add64(c, c), b);
    d = add64(d, a); a = sub64(add64(a, a), d);
}
__device__ __forceinline__ void xform3_fwd64(int64_t (&v)[64])
{
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int j = 0; j < 4; j++)
            lift_fwd64r(v[16 * k + 4 * j], v[16 * k + 4 * j + 1], v[16 * k + 4 * j + 2], v[16 * k + 4 * j + 3]);
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int i = 0; i < 4; i++)
            lift_fwd64r(v[16 * k + i], v[16 * k + i + 4], v[16 * k + i + 8], v[16 * k + i + 12]);
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
        for (int i = 0; i < 4; i++)
            lift_fwd64r(v[4 * j + i], v[4 * j + i + 16], v[4 * j + i + 32], v[4 * j + i + 48]);
}
__device__ __forceinline__ void xform3_inv64(int64_t (&v)[64])
{
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
        for (int i = 0; i < 4; i++)
            lift_inv64r(v[4 * j + i], v[4 * j + i + 16], v[4 * j + i + 32], v[4 * j + i + 48]);
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int i = 0; i < 4; i++)
            lift_inv64r(v[16 * k + i], v[16 * k + i + 4], v[16 * k + i + 8], v[16 * k + i + 12]);
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int j = 0; j < 4; j++)
            lift_inv64r(v[16 * k + 4 * j], v[16 * k + 4 * j + 1], v[16 * k + 4 * j + 2], v[16 * k + 4 * j + 3]);
}

// Shared memory of one decoder warp: the 64 bit planes ([plane][lane]) and the
// stream tile ([64-bit word][lane], rate words and two zero words); of an
// encoder CTA: per warp the planes and the stream tile ([32-bit word][lane], 2
// rate words and four slack words), and the table.
__host__ __device__ constexpr size_t f64_dec_smem_bytes(int rate) { return (size_t)(64 + rate + 2) * 32 * 8; }
__host__ __device__ constexpr size_t f64_enc_smem_bytes(int rate)
{
    return sizeof(enc3::Expand) + (size_t)kEncWarps * (64 * 32 * 8 + (size_t)(2 * rate + 4) * 32 * 4);
}

__global__ void __launch_bounds__(32 * kEncWarps, kF64MinWarps / kEncWarps)
encode_f64_kernel(const double *__restrict__ src, uint8_t *__restrict__ out, Geom64 g)
{
    extern __shared__ __align__(16) uint64_t sm64[];
    enc3::Expand &expand = *reinterpret_cast<enc3::Expand *>(sm64);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = 2 * g.rate;
    uint64_t *wplanes = sm64 + sizeof(enc3::Expand) / 8 + (size_t)wid * (64 * 32 + (size_t)(nw + 4) * 16);
    uint32_t *tile = reinterpret_cast<uint32_t *>(wplanes + 64 * 32) + lane;
    uint64_t *planes = wplanes + lane;                          // plane k at planes[32 k]
    uint32_t *p32 = reinterpret_cast<uint32_t *>(planes);        // half h of plane k at p32[64 k + h]
    constexpr int kSeq[64] = ZFPX_SEQ3;
    enc3::load_expand(expand);
    for (int w = 0; w < nw + 4; w++) tile[32 * w] = 0u;
    enc3::wait_expand();
    __syncthreads();
    const bool out16 = (g.rate & 1) == 0 && !((uintptr_t)out & 15u);
    for (int64_t u = (int64_t)blockIdx.x * kEncWarps + wid; u < g.nunits; u += (int64_t)gridDim.x * kEncWarps) {
        const int64_t b0 = u * 32;
        const int nact = (int)min((int64_t)32, g.nblocks - b0);
        const bool valid = lane < nact;
        int64_t x0, y0, z0;
        // lanes past the unit's last block load that block and code nothing
        block_origin(g, b0 + (valid ? lane : nact - 1), x0, y0, z0);
        int64_t v[64];
        if (g.vec && x0 + 4 <= g.n[0] && y0 + 4 <= g.n[1] && z0 + 4 <= g.n[2]) {
            // an interior block: two 16-byte loads per row
            const double *p = src + z0 * g.s[2] + y0 * g.s[1] + x0;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const double *row = p;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const double2 a = __ldg(reinterpret_cast<const double2 *>(row));
                    const double2 b = __ldg(reinterpret_cast<const double2 *>(row) + 1);
                    v[16 * k + 4 * j] = __double_as_longlong(a.x);
                    v[16 * k + 4 * j + 1] = __double_as_longlong(a.y);
                    v[16 * k + 4 * j + 2] = __double_as_longlong(b.x);
                    v[16 * k + 4 * j + 3] = __double_as_longlong(b.y);
                    row += g.s[1];
                }
                p += g.s[2];
            }
        } else {
            // edge blocks and other layouts: element loads, the last row, level
            // and point repeated past the array's end, through a local array
            // kept rolled so the hot path's code stays compact
            int64_t t[64];
#pragma unroll 1
            for (int r = 0; r < 64; r++) {
                const int i = r & 3, j = (r >> 2) & 3, k = r >> 4;
                t[r] = __double_as_longlong(__ldg(src + min(z0 + k, g.n[2] - 1) * g.s[2] +
                                                  min(y0 + j, g.n[1] - 1) * g.s[1] +
                                                  min(x0 + i, g.n[0] - 1) * g.s[0]));
            }
#pragma unroll
            for (int r = 0; r < 64; r++) v[r] = t[r];
        }
        uint32_t amax = 0;                                       // high word of the largest magnitude
#pragma unroll
        for (int r = 0; r < 64; r++) amax = max(amax, (uint32_t)((uint64_t)v[r] >> 32) & 0x7fffffffu);
        const int e = block_exponent(amax);
        const bool act = valid && e;
        // nothing to code in the whole warp: the streams are zero (640 x 320 x 91 zeros:
        // 98 -> 50 us at rate 8, 110 -> 66 at 32; nothing more for other fields)
        if (!__any_sync(0xffffffffu, act)) {
            uint8_t *dst = out + (b0 + lane) * (int64_t)g.rate * 8;
            if (valid && out16)
                for (int i = 0; i < g.rate; i += 2) *reinterpret_cast<uint4 *>(dst + 8 * i) = make_uint4(0u, 0u, 0u, 0u);
            else if (valid)
                for (int i = 0; i < g.rate; i++) *reinterpret_cast<uint2 *>(dst + 8 * i) = make_uint2(0u, 0u);
            continue;
        }
#pragma unroll
        for (int r = 0; r < 64; r++) v[r] = quantize64((uint64_t)v[r], e);
        xform3_fwd64(v);
        // negabinary: the add here, the xor as the complement of the odd planes
#pragma unroll
        for (int r = 0; r < 64; r++) v[r] = (int64_t)((uint64_t)v[r] + kNega64);
        // planes 32 .. 63 from the high words of the coefficients in coding
        // order; the low words wait in the slots of planes 0 .. 31.  The loop over
        // the coefficients' halves stays rolled (a select picks the coefficient):
        // half the code, which the instruction cache holds better beside the
        // unrolled lifting
#pragma unroll 1
        for (int ch = 0; ch < 2; ch++) {
            uint32_t w[32];
#pragma unroll
            for (int t = 0; t < 32; t++) {
                const uint64_t c = (uint64_t)(ch ? v[kSeq[32 + t]] : v[kSeq[t]]);
                w[t] = (uint32_t)(c >> 32);
                p32[64 * t + ch] = (uint32_t)c;
            }
            transpose32(w);
#pragma unroll
            for (int k = 0; k < 32; k++) p32[64 * (32 + k) + ch] = k & 1 ? ~w[k] : w[k];
        }
        auto finish_low = [&]() {
#pragma unroll 1
            for (int ch = 0; ch < 2; ch++) {
                uint32_t w[32];
#pragma unroll
                for (int t = 0; t < 32; t++) w[t] = p32[64 * t + ch];
                transpose32(w);
#pragma unroll
                for (int k = 0; k < 32; k++) p32[64 * k + ch] = k & 1 ? ~w[k] : w[k];
            }
        };
        if (act) tile[0] = 1u | ((uint32_t)e << 1);
        enc3::code<false>(enc3::smem(tile), enc3::smem(expand.e), planes, 63, 12, 64 * g.rate, 0, act, 32, finish_low);
        __syncwarp();
        uint8_t *dst = out + (b0 + lane) * (int64_t)g.rate * 8;
        if (out16) {
            for (int i = 0; i < nw; i += 4) {
                const uint4 c = make_uint4(tile[32 * i], tile[32 * (i + 1)], tile[32 * (i + 2)], tile[32 * (i + 3)]);
                if (valid) *reinterpret_cast<uint4 *>(dst + 4 * i) = c;
            }
        } else {
            for (int i = 0; i < nw; i += 2) {
                const uint2 c = make_uint2(tile[32 * i], tile[32 * (i + 1)]);
                if (valid) *reinterpret_cast<uint2 *>(dst + 4 * i) = c;
            }
        }
        for (int w = 0; w < nw + 4; w++) tile[32 * w] = 0u;
        __syncwarp();
    }
}

// x = q 2^(e_max - 62) rounded once to nearest even, e_max = e - 1023 (every
// exponent; the kernels take dequantize64_normal where it applies).
__device__ __forceinline__ double dequantize64(int64_t q, int e)
{
    const int s = e - 1023 - 62;                                 // x = q 2^s
    if (s >= -1022 || q == 0) {
        // (double)q rounds once; the scaling by 2^s is exact while the result
        // is normal, which holds for every q != 0 once s >= -1022
        const int s1 = s < -600 ? -600 : s;
        return (__ll2double_rn(q) * __longlong_as_double((long long)(s1 + 1023) << 52)) *
               __longlong_as_double((long long)(s - s1 + 1023) << 52);
    }
    const uint64_t a = q < 0 ? 0ull - (uint64_t)q : (uint64_t)q;
    const uint64_t sign = q < 0 ? 0x8000000000000000ull : 0ull;
    // normal result: a 2^s >= 2^-1022, i.e. a >= 2^(-1022 - s)
    const int t = -1022 - s;                                     // >= 1 here
    if (t < 64 && a >= (1ull << t)) {
        const int s1 = s < -600 ? -600 : s;
        const double r = (__ull2double_rn(a) * __longlong_as_double((long long)(s1 + 1023) << 52)) *
                         __longlong_as_double((long long)(s - s1 + 1023) << 52);
        return sign ? -r : r;
    }
    // subnormal: a 2^(s + 1074) units of 2^-1074, rounded to nearest even
    const int u = s + 1074;
    uint64_t m;
    if (u >= 0) {
        m = a << u;                                              // a < 2^(t) so this stays below 2^52
    } else {
        const int d = -u;
        if (d >= 64) {
            m = 0;                                               // below half the smallest subnormal
        } else {
            const uint64_t lo = a & ((1ull << d) - 1ull), half = 1ull << (d - 1);
            m = a >> d;
            m += (lo > half || (lo == half && (m & 1ull))) ? 1ull : 0ull;
        }
    }
    return __longlong_as_double((long long)(m | sign));
}

__global__ void __launch_bounds__(32, kF64MinWarps) decode_f64_kernel(const uint8_t *__restrict__ in,
                                                                      double *__restrict__ dst, Geom64 g)
{
    extern __shared__ uint64_t sm64[];
    __shared__ DropTable drop;
    load_drop<32>(drop);
    __syncthreads();
    uint64_t *tile = sm64 + 64 * 32;
    const int lane = threadIdx.x;
    const Tile64 st{tile, lane};
    SmemPlanes pl{sm64, lane};
    constexpr int kSeq[64] = ZFPX_SEQ3;
    for (int64_t u = blockIdx.x; u < g.nunits; u += gridDim.x) {
        const int64_t b0 = u * 32;
        const int nact = (int)min((int64_t)32, g.nblocks - b0);
        if (lane >= nact) continue;
        const int64_t b = b0 + lane;
        const uint64_t *s64 = reinterpret_cast<const uint64_t *>(in) + b * g.rate;
#pragma unroll 4
        for (int i = 0; i < g.rate; i++) tile[i * 32 + lane] = __ldg(s64 + i);
        tile[g.rate * 32 + lane] = 0ull;
        tile[(g.rate + 1) * 32 + lane] = 0ull;
        int64_t x0, y0, z0;
        block_origin(g, b, x0, y0, z0);
        const uint64_t head = st.peek(0);
        double x[64];
        if (!(head & 1ull)) {
#pragma unroll
            for (int r = 0; r < 64; r++) x[r] = 0.0;
        } else {
            const int e = (int)((head >> 1) & 0x7ffu);
            // the planes from bit 12 on; the tile's two zero 64-bit words let the
            // parser read past the budget without a test
            const WithDrop<Tile64As32> t32(Tile64As32{reinterpret_cast<const uint32_t *>(tile), lane}, drop);
            const int kmin = parse_planes64<true>(t32, 12, 64 * g.rate, 63, pl);
            // planes below kmin are zero; the negabinary xor is the complement of
            // the odd planes
            int64_t v[64];
#pragma unroll
            for (int ch = 0; ch < 2; ch++) {
                uint32_t w[32];
#pragma unroll
                for (int k = 0; k < 32; k++) {
                    const uint32_t c = 32 + k >= kmin ? pl.load_half(32 + k, ch) : 0u;
                    w[k] = k & 1 ? ~c : c;
                }
                transpose32(w);
#pragma unroll
                for (int t = 0; t < 32; t++) v[kSeq[32 * ch + t]] = (int64_t)((uint64_t)w[t] << 32);
            }
            if (__all_sync(__activemask(), kmin >= 32)) {
                // no low plane in any lane: every low word is M - M = 0
#pragma unroll
                for (int r = 0; r < 64; r++) v[r] = sub64(v[r], (int64_t)(kNega64 & 0xffffffff00000000ull));
            } else {
#pragma unroll
                for (int ch = 0; ch < 2; ch++) {
                    uint32_t w[32];
#pragma unroll
                    for (int k = 0; k < 32; k++) {
                        const uint32_t c = k >= kmin ? pl.load_half(k, ch) : 0u;
                        w[k] = k & 1 ? ~c : c;
                    }
                    transpose32(w);
#pragma unroll
                    for (int t = 0; t < 32; t++) {
                        int64_t &c = v[kSeq[32 * ch + t]];
                        c = sub64((int64_t)((uint64_t)c | w[t]), (int64_t)kNega64);
                    }
                }
            }
            xform3_inv64(v);
            if (e >= 63) {
#pragma unroll
                for (int r = 0; r < 64; r++) x[r] = dequantize64_normal(v[r], e);
            } else {
                // tiny exponents (rare): a rolled loop over a local copy
                int64_t t[64];
#pragma unroll
                for (int r = 0; r < 64; r++) t[r] = v[r];
#pragma unroll 1
                for (int r = 0; r < 64; r++) t[r] = __double_as_longlong(dequantize64(t[r], e));
#pragma unroll
                for (int r = 0; r < 64; r++) x[r] = __longlong_as_double(t[r]);
            }
        }
        if (g.vec && x0 + 4 <= g.n[0] && y0 + 4 <= g.n[1] && z0 + 4 <= g.n[2]) {
            // an interior block: two 16-byte stores per row
#pragma unroll
            for (int k = 0; k < 4; k++)
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    double2 *row = reinterpret_cast<double2 *>(dst + (z0 + k) * g.s[2] + (y0 + j) * g.s[1] + x0);
                    row[0] = make_double2(x[16 * k + 4 * j], x[16 * k + 4 * j + 1]);
                    row[1] = make_double2(x[16 * k + 4 * j + 2], x[16 * k + 4 * j + 3]);
                }
        } else {
            // edge blocks and other layouts: element stores inside the array,
            // through a local array kept rolled
            double t[64];
#pragma unroll
            for (int r = 0; r < 64; r++) t[r] = x[r];
#pragma unroll 1
            for (int r = 0; r < 64; r++) {
                const int i = r & 3, j = (r >> 2) & 3, k = r >> 4;
                if (x0 + i < g.n[0] && y0 + j < g.n[1] && z0 + k < g.n[2])
                    dst[(z0 + k) * g.s[2] + (y0 + j) * g.s[1] + (x0 + i) * g.s[0]] = t[r];
            }
        }
    }
}

Geom64 make_geom(const int64_t n[3], const int64_t s[3], int rate, const void *base)
{
    Geom64 g;
    g.vec = s[0] == 1 && s[1] % 2 == 0 && s[2] % 2 == 0 && !((uintptr_t)base & 15u);
    for (int a = 0; a < 3; a++) { g.n[a] = n[a]; g.s[a] = s[a]; }
    g.bx = (n[0] + 3) / 4; g.by = (n[1] + 3) / 4;
    g.nblocks = g.bx * g.by * ((n[2] + 3) / 4);
    block_divisor((uint32_t)std::min<int64_t>(g.bx, INT_MAX), g.bxm, g.bxl);
    block_divisor((uint32_t)std::min<int64_t>(g.by, INT_MAX), g.bym, g.byl);
    g.nunits = (g.nblocks + 31) / 32;
    g.rate = rate;
    return g;
}

unsigned grid_f64(const void *fn, int warps, int64_t nunits, size_t smem)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * warps, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    const int64_t cap = (int64_t)num_sms() * per_sm;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((nunits + warps - 1) / warps, cap));
}

bool valid_f64_args(int rate, const int64_t n[3], const int64_t stride[3])
{
    if (rate < 1 || rate > kMaxRate || !n || !stride) return false;
    for (int a = 0; a < 3; a++) if (n[a] < 1 || stride[a] < 0) return false;
    return true;
}

}  // namespace
}  // namespace zfpx

using namespace zfpx;

extern "C" {

size_t zfpx_stream_bytes_f64(int rate, const int64_t n[3])
{
    if (!n || rate < 1 || rate > kMaxRate) return 0;
    for (int a = 0; a < 3; a++) if (n[a] < 1) return 0;
    return (size_t)(((n[0] + 3) / 4) * ((n[1] + 3) / 4) * ((n[2] + 3) / 4) * 8 * rate);
}

int zfpx_encode_f64(int rate, const double *d_in, const int64_t n[3], const int64_t stride[3], uint8_t *d_out,
                    size_t cap, void *stream)
{
    if (!d_in || !d_out || !valid_f64_args(rate, n, stride)) return ZFPX_EINVAL;
    if (((uintptr_t)d_out & 7u) || ((uintptr_t)d_in & 7u)) return ZFPX_EINVAL;
    if (cap < zfpx_stream_bytes_f64(rate, n)) return ZFPX_ESIZE;
    const Geom64 g = make_geom(n, stride, rate, d_in);
    const size_t smem = f64_enc_smem_bytes(rate);
    const int rc = allow_smem((const void *)encode_f64_kernel, smem);
    if (rc) return rc;
    encode_f64_kernel<<<grid_f64((const void *)encode_f64_kernel, kEncWarps, g.nunits, smem), 32 * kEncWarps, smem,
                        (cudaStream_t)stream>>>(d_in, d_out, g);
    count_launch();
    return check_launch();
}

int zfpx_decode_f64(int rate, const uint8_t *d_in, size_t len, const int64_t n[3], const int64_t stride[3],
                    double *d_out, void *stream)
{
    if (!d_in || !d_out || !valid_f64_args(rate, n, stride)) return ZFPX_EINVAL;
    if (((uintptr_t)d_out & 7u) || ((uintptr_t)d_in & 7u)) return ZFPX_EINVAL;
    if (len < zfpx_stream_bytes_f64(rate, n)) return ZFPX_ESIZE;
    const Geom64 g = make_geom(n, stride, rate, d_out);
    const size_t smem = f64_dec_smem_bytes(rate);
    const int rc = allow_smem((const void *)decode_f64_kernel, smem);
    if (rc) return rc;
    decode_f64_kernel<<<grid_f64((const void *)decode_f64_kernel, 1, g.nunits, smem), 32, smem, (cudaStream_t)stream>>>(
        d_in, d_out, g);
    count_launch();
    return check_launch();
}

}  // extern "C"
