// Fused pack + ZFP fixed-rate encode, and fused decode + unpack, for sm_103a.
//
// The codec is ZFP's fixed-rate mode as the paper uses it (Sec. II-C: 4^d
// blocks coded independently by a lifting transform and precision
// reduction; Sec. IV-B: rate 8 and 16, fixed message size), in the readings
// stated in include/zfpx.h:
//   e_max = frexp exponent of max|x|; zero block if max|x| is 0, subnormal or
//   non-finite; q = trunc(x 2^(30-e_max)); five-step integer lifting along
//   x, y, z; coefficients in total-sequency order; negabinary; group-tested
//   bit planes from 31 down, cut at exactly 4^d r bits.
//
// Mapping to the GPU: one lane owns one block (a warp owns one in the smallest
// 3-D launches).  A warp takes 32 consecutive blocks of one message, so its
// compressed output (or input) is one contiguous run of 32 * 8r bytes; each
// lane moves its own stream with 16-byte accesses and keeps it in its own
// column of a [word][lane] tile of shared memory.  The 64 coefficients of a
// block live in registers; their 32 bit planes are formed with two in-register
// 32x32 bit-matrix transposes (byte permutes for the 16- and 8-bit stages,
// masked shifts below), after which each plane is one 64-bit word; the
// encoder writes its group-tested part eight coefficients at a time through a
// table (zfpx_enc3.cuh), the decoder reads it in 32-bit windows
// (parse_planes64).  Each warp processes a contiguous range of 32-block
// chunks, so the message lookup is a forward scan.
#include <atomic>
#include <climits>
#include <cuda_runtime.h>

#include "zfpx_internal.h"
#include "zfpx_block.cuh"
#include "zfpx_smem.cuh"
#include "zfpx_enc3.cuh"
#include "zfpx_enc2.cuh"
#include "zfpx_warp3.cuh"

namespace zfpx {
namespace {

using namespace blk;

constexpr int kWarps = 4;
constexpr int kThreads = 32 * kWarps;
// Launch shapes of the 3-D kernels, chosen by measurement on GB300: encoder
// CTAs of 2 warps, eight to an SM (the shared memory of a ninth is there at rate
// 8, but five warps on a scheduler leave 96 registers and a few spills: 287 us
// against 274 for a 1280 x 640 x 137 field over 8 x 8 ranks); decoder CTAs of 4
// warps, except the rate-16 decoder, whose 3-warp CTAs fit six to an SM (two zero
// rows after its stream tile make the shared memory fit); the rate-8 decoder is
// compiled for five resident CTAs, which its shared memory allows and capping its
// registers to match pays for (four: 10 % slower).
template <int RATE>
constexpr int kEnc3Warps = 2;
constexpr int kEnc3MinBlocks = 8;
template <int RATE>
constexpr int kDec3Warps = RATE == 16 ? 3 : 4;
template <int RATE>
constexpr int kDec3MinBlocks = RATE == 8 ? 5 : 6;

// ----------------------------------------------------------------- message walk
struct MsgWalk {
    const MsgDev *msgs;
    int nmsg, mi;
    int64_t next0;
    __device__ __forceinline__ void start(const MsgDev *m, int n, int64_t u)
    {
        msgs = m; nmsg = n;
        mi = find_msg(m, n, u);
        next0 = mi + 1 < n ? m[mi + 1].unit0 : LLONG_MAX;
    }
    __device__ __forceinline__ void advance(int64_t u)
    {
        while (u >= next0) {
            mi++;
            next0 = mi + 1 < nmsg ? msgs[mi + 1].unit0 : LLONG_MAX;
        }
    }
};

// Work split of the 3-D kernels: warp w of the grid codes the upw consecutive
// 32-block units starting at w * upw (the grid has ceil(units / (upw * warps))
// CTAs), and the hardware's CTA scheduler balances the CTAs over the SMs.  No
// counters in device memory: launches on any streams may overlap, and a CUDA
// graph replays a launch as it was recorded.
struct UnitRange {
    int64_t c, c1;
    __device__ __forceinline__ UnitRange(const LaunchGeom &g, int warps, int wid)
    {
        c = ((int64_t)blockIdx.x * warps + wid) * g.upw;
        c1 = min(c + (int64_t)g.upw, g.nunits);
    }
};

// ----------------------------------------------------------------- rows of a 3-D block
// Rows that don't start on 16 bytes (a longitude split 3, 6, 7 ... ways, a padded
// row pitch): with unit x stride and even y and z strides every row of a
// message starts alike, on 8 bytes or 4 past them, and moves as two 8-byte
// accesses or as 4 + 8 + 4 bytes.  Any other layout moves value by value.
enum RowKind { ROWS_8 = 0, ROWS_4_8_4 = 1, ROWS_ANY = 2 };
__device__ __forceinline__ int row_kind(const void *first, const int64_t *s)
{
    if (s[0] != 1 || ((s[1] | s[2]) & 1)) return ROWS_ANY;
    return ((uintptr_t)first >> 2) & 1 ? ROWS_4_8_4 : ROWS_8;
}

// The 64 values of the block at p (rows past the end of the box repeat its
// last row); every row complete in x.
template <int KIND>
__device__ __forceinline__ void load_rows(const float *p, const int64_t *s, int ny, int nz, float (&x)[64])
{
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const float *row = p;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            float *v = x + 16 * k + 4 * j;
            if (KIND == ROWS_8) {
                const float2 a = __ldg(reinterpret_cast<const float2 *>(row));
                const float2 b = __ldg(reinterpret_cast<const float2 *>(row) + 1);
                v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
            } else if (KIND == ROWS_4_8_4) {
                const float2 b = __ldg(reinterpret_cast<const float2 *>(row + 1));
                v[0] = __ldg(row); v[1] = b.x; v[2] = b.y; v[3] = __ldg(row + 3);
            } else {
#pragma unroll
                for (int i = 0; i < 4; i++) v[i] = __ldg(row + (int64_t)i * s[0]);
            }
            if (j + 1 < ny) row += s[1];
        }
        if (k + 1 < nz) p += s[2];
    }
}

// The same with partial rows (nx < 4 values, the last one repeated): four
// values at a time through `own`, the lane's own words of the plane tile ([32][32]
// 64-bit, this lane's column, two values a word), kept rolled so that the
// complete blocks' code stays compact.  No other lane's words are touched, so
// the other lanes may be storing planes, or still reading them, meanwhile.
__device__ __forceinline__ void load_edge(const float *p, const int64_t *s, int nx, int ny, int nz, uint64_t *own,
                                          float (&x)[64])
{
#pragma unroll 1
    for (int r = 0; r < 16; r++) {
        const float *row = p + (int64_t)min(r >> 2, nz - 1) * s[2] + (int64_t)min(r & 3, ny - 1) * s[1];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const float a = __ldg(row + (int64_t)min(2 * h, nx - 1) * s[0]);
            const float b = __ldg(row + (int64_t)min(2 * h + 1, nx - 1) * s[0]);
            own[32 * (2 * r + h)] = (uint64_t)f2u(b) << 32 | f2u(a);
        }
    }
#pragma unroll
    for (int r = 0; r < 32; r++) {
        const uint64_t v = own[32 * r];
        x[2 * r] = u2f((uint32_t)v);
        x[2 * r + 1] = u2f((uint32_t)(v >> 32));
    }
}

// The inverses: only rows inside the box are written.
template <int KIND>
__device__ __forceinline__ void store_rows(float *p, const int64_t *s, int ny, int nz, const float (&x)[64])
{
#pragma unroll
    for (int k = 0; k < 4; k++) {
#pragma unroll
        for (int j = 0; j < 4; j++) {
            float *row = p + (int64_t)k * s[2] + (int64_t)j * s[1];
            const float *v = x + 16 * k + 4 * j;
            if (k < nz && j < ny) {
                if (KIND == ROWS_8) {
                    reinterpret_cast<float2 *>(row)[0] = make_float2(v[0], v[1]);
                    reinterpret_cast<float2 *>(row)[1] = make_float2(v[2], v[3]);
                } else if (KIND == ROWS_4_8_4) {
                    row[0] = v[0];
                    *reinterpret_cast<float2 *>(row + 1) = make_float2(v[1], v[2]);
                    row[3] = v[3];
                } else {
#pragma unroll
                    for (int i = 0; i < 4; i++) row[(int64_t)i * s[0]] = v[i];
                }
            }
        }
    }
}
__device__ __forceinline__ void store_edge(float *p, const int64_t *s, int nx, int ny, int nz, uint64_t *own,
                                           const float (&x)[64])
{
#pragma unroll
    for (int r = 0; r < 32; r++) own[32 * r] = (uint64_t)f2u(x[2 * r + 1]) << 32 | f2u(x[2 * r]);
#pragma unroll 1
    for (int r = 0; r < 16; r++) {
        if ((r >> 2) >= nz || (r & 3) >= ny) continue;
        float *row = p + (int64_t)(r >> 2) * s[2] + (int64_t)(r & 3) * s[1];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const uint64_t v = own[32 * (2 * r + h)];
            if (2 * h < nx) row[(int64_t)(2 * h) * s[0]] = u2f((uint32_t)v);
            if (2 * h + 1 < nx) row[(int64_t)(2 * h + 1) * s[0]] = u2f((uint32_t)(v >> 32));
        }
    }
}

// ================================================================= 3-D kernels
// VEC: every block's rows start on 16 bytes (the view's row and level strides
// and every message's x origin are multiples of 4 values, the base aligned),
// so full rows move as 16-byte loads and stores.  Otherwise a separate
// instantiation moves the rows by their kind (load_rows), keeping the vector
// kernel's code as it is.  Blocks partial in x go through load_edge in both.
// Four scalar accesses per row and partial blocks value by value through a local
// array took 5760 (compress) and 5130 (decompress) warp instructions per 32
// blocks of a 1000 x 501 x 91 field on 3 x 3 ranks, against 3540 and 4040 for
// aligned rows: 192 / 174 us at rate 8, now 168 / 125; a 233 x 117 x 137 array of
// aligned rows, one partial block in 59, went from 26.6 / 26.6 to 20.5 / 18.5 us.
// LEN: the variable-rate modes, which also want every block's bit count (acc).
template <int RATE, bool VEC, bool LEN>
__global__ void __launch_bounds__(32 * kEnc3Warps<RATE>, kEnc3MinBlocks)
encode3_kernel(const float *__restrict__ src, uint8_t *__restrict__ out, LaunchGeom g, int layout, AccEncode acc)
{
    __shared__ enc3::Shared<RATE> sh[kEnc3Warps<RATE>];
    __shared__ enc3::Expand expand;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const enc3::View v = sh[wid].view(expand);
    enc3::load_expand(expand);
    const UnitRange ur(g, kEnc3Warps<RATE>, wid);
    enc3::clear(v, lane, enc3::kWords<RATE>);
    MsgWalk walk;
    if (ur.c < ur.c1) walk.start(g.msgs, g.nmsg, ur.c);
    enc3::wait_expand();
    __syncthreads();
    for (int64_t c = ur.c; c < ur.c1; c++) {
        walk.advance(c);
        const MsgDev &m = g.msgs[walk.mi];
        const int64_t unit0 = m.unit0, nblocks = m.nblocks, src_off = m.src_off;
        const int64_t boff = layout ? m.off[1] : m.off[0];
        const int nx = m.nx, ny = m.ny, nz = m.nz, bxn = m.bx, byn = m.by;
        const int64_t b0 = (c - unit0) * 32;
        const int nact = (int)min((int64_t)32, nblocks - b0);
        const bool valid = lane < nact;
        float x[64];
        {
            // lanes past the unit's last block load that block and code nothing
            const int b = (int)b0 + (valid ? lane : nact - 1);
            const int t = (int)divu((uint32_t)b, m.bxm, m.bxl), bxi = b - t * bxn;
            const int bzi = (int)divu((uint32_t)t, m.bym, m.byl), byi = t - bzi * byn;
            const int x0 = 4 * bxi, y0 = 4 * byi, z0 = 4 * bzi;
            const float *base = src + src_off;
            if (VEC && x0 + 4 <= nx) {
                // the common case: sixteen 16-byte row loads (rows past the
                // end of the box repeat its last row)
                const float *p = base + (int64_t)z0 * g.ss[2] + (int64_t)y0 * g.ss[1] + x0;
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const float *row = p;
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const float4 f = __ldg(reinterpret_cast<const float4 *>(row));
                        x[16 * k + 4 * j] = f.x; x[16 * k + 4 * j + 1] = f.y;
                        x[16 * k + 4 * j + 2] = f.z; x[16 * k + 4 * j + 3] = f.w;
                        if (y0 + j + 1 < ny) row += g.ss[1];
                    }
                    if (z0 + k + 1 < nz) p += g.ss[2];
                }
            } else {
                const float *p = base + (int64_t)z0 * g.ss[2] + (int64_t)y0 * g.ss[1] + (int64_t)x0 * g.ss[0];
                const int kind = VEC ? ROWS_ANY : row_kind(base, g.ss);
                if (x0 + 4 > nx)
                    load_edge(p, g.ss, nx - x0, ny - y0, nz - z0, v.planes + lane, x);
                else if (!VEC && kind == ROWS_8)
                    load_rows<ROWS_8>(p, g.ss, ny - y0, nz - z0, x);
                else if (!VEC && kind == ROWS_4_8_4)
                    load_rows<ROWS_4_8_4>(p, g.ss, ny - y0, nz - z0, x);
                else if (!VEC)
                    load_rows<ROWS_ANY>(p, g.ss, ny - y0, nz - z0, x);
            }
        }
        const int len = enc3::encode<RATE, LEN>(x, valid, v, lane, enc3::PlaneCut{acc.minexp, acc.prec});
        if (LEN && valid) acc.lengths[(acc.msgs ? acc.msgs[walk.mi].gb0 : 0) + b0 + lane] = (uint16_t)len;
        __syncwarp();
        enc3::store_stream<RATE>(v, lane, valid, out + boff + (b0 + lane) * RATE * 8);
        __syncwarp();
    }
}

// Cuts a unit's nact blocks, from block b0 of message mi on, out of the payload
// into the lanes' tile columns: 1024 bits each, those past a block's length 0.
__device__ __forceinline__ void load_payload(const AccDecode &acc, int mi, int64_t b0, int nact, int lane,
                                             uint32_t *t32, uint64_t *stage)
{
    const int64_t gr0 = acc.msgs ? acc.msgs[mi].gr0 : 0;
    const int64_t gl = gr0 + b0 + (lane < nact ? lane : nact - 1);
    auto bit = [&](int64_t q) { return acc.tile_off[q / kAccTile] + acc.local[q]; };
    const uint64_t off = (acc.pay ? (uint64_t)acc.pay[mi] * 64 : 0ull) + (bit(gl) - bit(gr0));
    const int L = min((int)acc.lengths[gl], 1024);
    const int64_t j0 = (int64_t)(__shfl_sync(0xffffffffu, off, 0) >> 6);
    const int64_t j1 = (int64_t)(__shfl_sync(0xffffffffu, off + (uint64_t)L + 63, nact - 1) >> 6);
    if (j1 - j0 > 32 * 16 + 1) {                                 // lengths above 1024 bits: not the encoder's
        if (lane < nact) {
            auto word = [&](int64_t j) { return j < acc.pwords ? __ldg(acc.payload + j) : 0ull; };
#pragma unroll 1
            for (int i = 0; i < 16; i++) {
                const int64_t j = (int64_t)(off >> 6) + i;
                const int sh = (int)(off & 63), rem = L - 64 * i;
                uint64_t v = rem > 0 ? (sh ? (word(j) >> sh) | (word(j + 1) << (64 - sh)) : word(j)) : 0ull;
                if (rem > 0 && rem < 64) v &= (1ull << rem) - 1ull;
                t32[(2 * i) * 32 + lane] = (uint32_t)v;
                t32[(2 * i + 1) * 32 + lane] = (uint32_t)(v >> 32);
            }
        }
        return;
    }
    const int nw = (int)(j1 - j0);
    for (int i = lane; i <= nw; i += 32) {                       // one word more, for the last funnel
        const int64_t j = j0 + i;
        stage[i] = i < nw && j < acc.pwords ? __ldg(acc.payload + j) : 0ull;
    }
    __syncwarp();
    const uint32_t *s32 = reinterpret_cast<const uint32_t *>(stage);
    const int p = (int)(off - (uint64_t)j0 * 64);
    const int w = p >> 5, sh = p & 31;
    uint32_t a = s32[w];
#pragma unroll
    for (int i = 0; i < 32; i++) {
        const int rem = L - 32 * i;
        uint32_t v = 0;
        if (rem > 0) {
            const uint32_t b = s32[w + i + 1];
            v = __funnelshift_r(a, b, sh);
            if (rem < 32) v &= (1u << rem) - 1u;
            a = b;
        }
        t32[i * 32 + lane] = v;
    }
    __syncwarp();                                                // the planes go over the staged words next
}

// PAY: the variable-rate modes, whose blocks lie back to back in a payload at
// the bit offsets that the scan of their lengths gives (acc); a unit's bits are
// one run of words, copied to shared memory (the planes' space, not yet in
// use) in whole and cut into the lanes' columns from there.
template <int RATE, bool VEC, bool PAY>
__global__ void __launch_bounds__(32 * kDec3Warps<RATE>, kDec3MinBlocks<RATE>)
decode3_kernel(const uint8_t *__restrict__ in, float *__restrict__ dstf, LaunchGeom g, int layout, AccDecode acc)
{
    __shared__ uint32_t stile[kDec3Warps<RATE>][(2 * RATE + kTileZeroRows<RATE>) * 32];
    __shared__ uint64_t splanes[kDec3Warps<RATE>][32 * 32];
    __shared__ DropTable drop;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t *t32 = stile[wid];
    SmemPlanes pl{splanes[wid], lane};
    const WithDrop<StreamTile> tile(StreamTile{t32, lane}, drop);
    load_drop<32 * kDec3Warps<RATE>>(drop);
#pragma unroll
    for (int r = 0; r < kTileZeroRows<RATE>; r++) t32[(2 * RATE + r) * 32 + lane] = 0u;
    const UnitRange ur(g, kDec3Warps<RATE>, wid);
    __syncthreads();
    if (ur.c >= ur.c1) return;
    MsgWalk walk;
    walk.start(g.msgs, g.nmsg, ur.c);
    for (int64_t c = ur.c; c < ur.c1; c++) {
        walk.advance(c);
        const MsgDev &m = g.msgs[walk.mi];
        const int64_t unit0 = m.unit0, nblocks = m.nblocks, dst_off = m.dst_off;
        const int64_t boff = layout ? m.off[1] : m.off[0];
        const int nx = m.nx, ny = m.ny, nz = m.nz, bxn = m.bx, byn = m.by;
        const int64_t b0 = (c - unit0) * 32;
        const int nact = (int)min((int64_t)32, nblocks - b0);
        if (PAY) load_payload(acc, walk.mi, b0, nact, lane, t32, splanes[wid]);
        if (lane < nact) {
            const int b = (int)b0 + lane;
            if (!PAY) {
                // this lane's block: RATE / 2 16-byte loads into its own tile column
                const uint4 *src4 = reinterpret_cast<const uint4 *>(in + boff) + (int64_t)b * (RATE / 2);
#pragma unroll
                for (int i = 0; i < RATE / 2; i++) {
                    const uint4 v = __ldg(src4 + i);
                    t32[(4 * i) * 32 + lane] = v.x;
                    t32[(4 * i + 1) * 32 + lane] = v.y;
                    t32[(4 * i + 2) * 32 + lane] = v.z;
                    t32[(4 * i + 3) * 32 + lane] = v.w;
                }
            }
            const int t = (int)divu((uint32_t)b, m.bxm, m.bxl), bxi = b - t * bxn;
            const int bzi = (int)divu((uint32_t)t, m.bym, m.byl), byi = t - bzi * byn;
            const int x0 = 4 * bxi, y0 = 4 * byi, z0 = 4 * bzi;
            float v[64];
            decode_block3_tile<RATE>(tile, v, pl);
            float *base = dstf + dst_off;
            if (VEC && x0 + 4 <= nx) {
#pragma unroll
                for (int k = 0; k < 4; k++) {
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        float *row = base + (int64_t)(z0 + k) * g.ds[2] + (int64_t)(y0 + j) * g.ds[1] + x0;
                        if (z0 + k < nz && y0 + j < ny)
                            *reinterpret_cast<float4 *>(row) = make_float4(v[16 * k + 4 * j], v[16 * k + 4 * j + 1],
                                                                           v[16 * k + 4 * j + 2], v[16 * k + 4 * j + 3]);
                    }
                }
            } else {
                float *p = base + (int64_t)z0 * g.ds[2] + (int64_t)y0 * g.ds[1] + (int64_t)x0 * g.ds[0];
                const int kind = VEC ? ROWS_ANY : row_kind(base, g.ds);
                if (x0 + 4 > nx)
                    store_edge(p, g.ds, nx - x0, ny - y0, nz - z0, splanes[wid] + lane, v);
                else if (!VEC && kind == ROWS_8)
                    store_rows<ROWS_8>(p, g.ds, ny - y0, nz - z0, v);
                else if (!VEC && kind == ROWS_4_8_4)
                    store_rows<ROWS_4_8_4>(p, g.ds, ny - y0, nz - z0, v);
                else if (!VEC)
                    store_rows<ROWS_ANY>(p, g.ds, ny - y0, nz - z0, v);
            }
        }
        __syncwarp();
    }
}

// A warp per block (zfpx_warp3.cuh): warp w of a unit's 32 codes its block w.
// Values move one by one, two a lane, in the block's order.
struct WarpBlock {
    int64_t boff;             // the block's message in the stream buffer
    int b, nx, ny, nz;        // block, and the values it holds along each axis
    int64_t view;             // its first value in the view
    __device__ __forceinline__ bool find(const LaunchGeom &g, const int64_t *s, int64_t view_off(const MsgDev &), int layout, int wid)
    {
        const int64_t c = blockIdx.x / (32 / kWarps);
        MsgWalk walk;
        walk.start(g.msgs, g.nmsg, c);
        const MsgDev &m = g.msgs[walk.mi];
        const int64_t q = (c - m.unit0) * 32 + blockIdx.x % (32 / kWarps) * kWarps + wid;
        if (q >= m.nblocks) return false;
        b = (int)q;
        boff = layout ? m.off[1] : m.off[0];
        const int t = (int)divu((uint32_t)b, m.bxm, m.bxl), z = (int)divu((uint32_t)t, m.bym, m.byl);
        const int x0 = 4 * (b - t * m.bx), y0 = 4 * (t - z * m.by), z0 = 4 * z;
        nx = m.nx - x0; ny = m.ny - y0; nz = m.nz - z0;
        view = view_off(m) + (int64_t)z0 * s[2] + (int64_t)y0 * s[1] + (int64_t)x0 * s[0];
        return true;
    }
};

template <int RATE>
__global__ void __launch_bounds__(kThreads)
encode3_warp_kernel(const float *__restrict__ src, uint8_t *__restrict__ out, LaunchGeom g, int layout)
{
    __shared__ warp3::Shared<RATE> sh[kWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    WarpBlock k;
    if (!k.find(g, g.ss, [](const MsgDev &m) { return m.src_off; }, layout, wid)) return;
    // rows past the end of the box repeat its last row, values its last value
    const float *p = src + k.view + (int64_t)min(lane & 3, k.nx - 1) * g.ss[0] +
                     (int64_t)min((lane >> 2) & 3, k.ny - 1) * g.ss[1];
    const float x0 = __ldg(p + (int64_t)min(lane >> 4, k.nz - 1) * g.ss[2]);
    const float x1 = __ldg(p + (int64_t)min((lane >> 4) + 2, k.nz - 1) * g.ss[2]);
    warp3::encode<RATE>(x0, x1, sh[wid], lane);
    if (lane < 2 * RATE)
        reinterpret_cast<uint32_t *>(out + k.boff)[(int64_t)k.b * 2 * RATE + lane] = sh[wid].stream[lane];
}

template <int RATE>
__global__ void __launch_bounds__(kThreads)
decode3_warp_kernel(const uint8_t *__restrict__ in, float *__restrict__ dstf, LaunchGeom g, int layout)
{
    __shared__ warp3::Shared<RATE> sh[kWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    WarpBlock k;
    if (!k.find(g, g.ds, [](const MsgDev &m) { return m.dst_off; }, layout, wid)) return;
    uint32_t *w = sh[wid].stream;
    if (lane < 2 * RATE) w[lane] = __ldg(reinterpret_cast<const uint32_t *>(in + k.boff) + (int64_t)k.b * 2 * RATE + lane);
    if (lane < 4) w[2 * RATE + lane] = 0u;
    __syncwarp();
    float x0, x1;
    warp3::decode<RATE>(x0, x1, sh[wid], lane);
    if ((lane & 3) >= k.nx || ((lane >> 2) & 3) >= k.ny) return;
    float *p = dstf + k.view + (int64_t)(lane & 3) * g.ds[0] + (int64_t)((lane >> 2) & 3) * g.ds[1];
    if ((lane >> 4) < k.nz) p[(int64_t)(lane >> 4) * g.ds[2]] = x0;
    if ((lane >> 4) + 2 < k.nz) p[(int64_t)((lane >> 4) + 2) * g.ds[2]] = x1;
}

// ================================================================= 1-D kernels
// Blocks of 4 values along x; a block is 4r bits (32 or 64), kept in one
// register and moved with one coalesced 4- or 8-byte access per lane.  A lane
// takes a block of each of kUnits1 consecutive units of its warp's range at a
// time, all loads ahead of the coding.
constexpr int kUnits1 = 2;

// x origin and row offset (elements, view strides s) of block b of message m
__device__ __forceinline__ int64_t block1_row(const MsgDev &m, const int64_t *s, uint32_t b, int &x0)
{
    const uint32_t t = divu(b, m.bxm, m.bxl), z = divu(t, m.bym, m.byl);
    x0 = 4 * (int)(b - t * (uint32_t)m.bx);
    return (int64_t)z * s[2] + (int64_t)(t - z * (uint32_t)m.by) * s[1];
}

// Once every coefficient is significant a block's bits are its planes as
// nibbles: spread4 of a byte, and a byte of nibbles back to two bits of each
// coefficient (bits 8 i, 8 i + 1), by tables, since the ALU pipe bounds these
// kernels and the load pipe idles.  1280 x 640 x 37 values, compress / decompress:
// 98 / 119 us at rate 8 and 123 / 152 at rate 16 by shifts, now 94 / 115 and 115 / 139.
struct SpreadTable {
    const uint32_t *e;
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const { return e[x & 255u]; }
};

struct TailTable {
    const uint32_t *e;
    __device__ __forceinline__ uint32_t planes8(uint32_t w) const   // bits 8 i .. 8 i + 7: coefficient i of eight planes
    {
        return e[w & 255u] + 4u * e[(w >> 8) & 255u] + 16u * e[(w >> 16) & 255u] + 64u * e[w >> 24];
    }
    template <class Word>
    __device__ __forceinline__ void add(typename Word::T w, int p, uint32_t (&v)[4]) const
    {
        const uint32_t a = planes8((uint32_t)w);
        if (sizeof(w) == 8) {
            const uint32_t b = planes8((uint32_t)((uint64_t)w >> 32));
#pragma unroll
            for (int i = 0; i < 4; i++) v[i] |= shl_any(__byte_perm(a, b, i | (4 + i) << 4) & 0xffffu, p);
        } else {
#pragma unroll
            for (int i = 0; i < 4; i++) v[i] |= shl_any((a >> (8 * i)) & 255u, p);
        }
    }
};

template <int RATE>
__global__ void __launch_bounds__(kThreads)
encode1_kernel(const float *__restrict__ src, uint8_t *__restrict__ out, LaunchGeom g, int layout, int vec)
{
    __shared__ Plane4Enc tab;
    __shared__ uint32_t spread[256];
    plane4_fill(tab, threadIdx.x, blockDim.x);
    for (int i = threadIdx.x; i < 256; i += kThreads) spread[i] = spread4(i);
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t W = (int64_t)gridDim.x * kWarps;
    const int64_t gw = (int64_t)blockIdx.x * kWarps + wid;
    int64_t c = gw * g.nunits / W;
    const int64_t c1 = (gw + 1) * g.nunits / W;
    if (c >= c1) return;
    MsgWalk walk;
    walk.start(g.msgs, g.nmsg, c);
    while (c < c1) {
        walk.advance(c);
        const MsgDev &m = g.msgs[walk.mi];
        const int take = (int)min((int64_t)kUnits1, min(c1, walk.next0) - c);
        const uint32_t b0 = (uint32_t)(c - m.unit0) * 32u + lane;
        const uint32_t end = (uint32_t)min(m.nblocks, (c - m.unit0 + take) * 32);
        const int nx = m.nx;
        const float *base = src + m.src_off;
        float r[kUnits1][4];
#pragma unroll
        for (int k = 0; k < kUnits1; k++) {
            const uint32_t b = b0 + 32u * k;
            int x0;
            const float *row = base + block1_row(m, g.ss, b < end ? b : 0u, x0);   // past the end: some block's values
            if (vec && x0 + 4 <= nx) {
                const float4 f = __ldg(reinterpret_cast<const float4 *>(row + x0));
                r[k][0] = f.x; r[k][1] = f.y; r[k][2] = f.z; r[k][3] = f.w;
            } else {
#pragma unroll
                for (int i = 0; i < 4; i++) r[k][i] = __ldg(row + (int64_t)min(x0 + i, nx - 1) * g.ss[0]);
            }
        }
        uint64_t w[kUnits1];
        encode_blocks1<RATE, kUnits1>(r, tab, w, SpreadTable{spread});
        uint8_t *dst = out + (layout ? m.off[1] : m.off[0]);
#pragma unroll
        for (int k = 0; k < kUnits1; k++) {
            const uint32_t b = b0 + 32u * k;
            if (b >= end) continue;
            if (RATE == 16) reinterpret_cast<uint64_t *>(dst)[b] = w[k];
            else reinterpret_cast<uint32_t *>(dst)[b] = (uint32_t)w[k];
        }
        c += take;
    }
}

template <int RATE>
__global__ void __launch_bounds__(kThreads)
decode1_kernel(const uint8_t *__restrict__ in, float *__restrict__ dstf, LaunchGeom g, int layout, int vec)
{
    __shared__ Plane4Dec tab;
    __shared__ uint32_t nibbles[256];
    plane4_fill(tab, threadIdx.x, blockDim.x);
    for (uint32_t i = threadIdx.x; i < 256; i += kThreads) {
        uint32_t e = 0;
        for (int c = 0; c < 4; c++) e |= (((i >> c) & 1u) | ((i >> (c + 4)) & 1u) << 1) << (8 * c);
        nibbles[i] = e;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t W = (int64_t)gridDim.x * kWarps;
    const int64_t gw = (int64_t)blockIdx.x * kWarps + wid;
    int64_t c = gw * g.nunits / W;
    const int64_t c1 = (gw + 1) * g.nunits / W;
    if (c >= c1) return;
    MsgWalk walk;
    walk.start(g.msgs, g.nmsg, c);
    while (c < c1) {
        walk.advance(c);
        const MsgDev &m = g.msgs[walk.mi];
        const int take = (int)min((int64_t)kUnits1, min(c1, walk.next0) - c);
        const uint32_t b0 = (uint32_t)(c - m.unit0) * 32u + lane;
        const uint32_t end = (uint32_t)min(m.nblocks, (c - m.unit0 + take) * 32);
        const int nx = m.nx;
        const uint8_t *src = in + (layout ? m.off[1] : m.off[0]);
        float *base = dstf + m.dst_off;
        uint64_t w[kUnits1];
#pragma unroll
        for (int k = 0; k < kUnits1; k++) {
            const uint32_t b = b0 + 32u * k;
            w[k] = 0;
            if (b >= end) continue;
            if (RATE == 16) w[k] = __ldg(reinterpret_cast<const uint64_t *>(src) + b);
            else w[k] = __ldg(reinterpret_cast<const uint32_t *>(src) + b);
        }
        float v[kUnits1][4];
        decode_blocks1<RATE, kUnits1>(w, tab, v, TailTable{nibbles});
#pragma unroll
        for (int k = 0; k < kUnits1; k++) {
            const uint32_t b = b0 + 32u * k;
            if (b >= end) continue;
            int x0;
            float *row = base + block1_row(m, g.ds, b, x0);
            if (vec && x0 + 4 <= nx) {
                *reinterpret_cast<float4 *>(row + x0) = make_float4(v[k][0], v[k][1], v[k][2], v[k][3]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; i++)
                    if (x0 + i < nx) row[(int64_t)(x0 + i) * g.ds[0]] = v[k][i];
            }
        }
        c += take;
    }
}

// ================================================================= 2-D kernels
// Blocks of 4 x 4 values over axes 0 and 1 of one level; one lane per block,
// a warp takes 32 consecutive blocks of one message (units split statically
// over the warps).  Each lane moves its own stream with 16-byte accesses.
template <int RATE>
__global__ void __launch_bounds__(kThreads)
encode2_kernel(const float *__restrict__ src, uint8_t *__restrict__ out, LaunchGeom g, int layout, int vec)
{
    __shared__ enc2::Shared<RATE> sh[kWarps];
    __shared__ enc3::Expand expand;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const enc2::View v = sh[wid].view(expand);
    enc3::load_expand(expand);
    const int64_t W = (int64_t)gridDim.x * kWarps;
    const int64_t gw = (int64_t)blockIdx.x * kWarps + wid;
    int64_t c = gw * g.nunits / W;
    const int64_t c1 = (gw + 1) * g.nunits / W;
#pragma unroll
    for (int w = 0; w < enc2::kWords<RATE>; w++) v.tile[32 * w + lane] = 0u;
    MsgWalk walk;
    if (c < c1) walk.start(g.msgs, g.nmsg, c);
    enc3::wait_expand();
    __syncthreads();
    for (; c < c1; c++) {
        walk.advance(c);
        const MsgDev &m = g.msgs[walk.mi];
        const int64_t b0 = (c - m.unit0) * 32;
        const int nact = (int)min((int64_t)32, m.nblocks - b0);
        const bool valid = lane < nact;
        const int64_t boff = layout ? m.off[1] : m.off[0];
        float x[16];
        {
            // lanes past the unit's last block load that block and code nothing
            const int nx = m.nx, ny = m.ny;
            const uint32_t b = (uint32_t)b0 + (uint32_t)(valid ? lane : nact - 1);
            const uint32_t t = divu(b, m.bxm, m.bxl), z = divu(t, m.bym, m.byl);
            const int x0 = 4 * (int)(b - t * (uint32_t)m.bx), y0 = 4 * (int)(t - z * (uint32_t)m.by);
            const float *base = src + m.src_off + (int64_t)z * g.ss[2] + (int64_t)y0 * g.ss[1];
            if (vec && x0 + 4 <= nx) {
                // four 16-byte row loads (rows past the box repeat its last row)
                const float *row = base + x0;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const float4 f = __ldg(reinterpret_cast<const float4 *>(row));
                    x[4 * j] = f.x; x[4 * j + 1] = f.y; x[4 * j + 2] = f.z; x[4 * j + 3] = f.w;
                    if (y0 + j + 1 < ny) row += g.ss[1];
                }
            } else {
#pragma unroll
                for (int r = 0; r < 16; r++) {
                    const int i = r & 3, j = r >> 2;
                    x[r] = __ldg(base + (int64_t)min(j, ny - 1 - y0) * g.ss[1] + (int64_t)min(x0 + i, nx - 1) * g.ss[0]);
                }
            }
        }
        enc2::encode<RATE>(x, valid, v, lane);
        __syncwarp();
        enc2::store_stream<RATE>(v, lane, valid, out + boff + (b0 + lane) * (2 * RATE));
        __syncwarp();
    }
}

template <int RATE>
__global__ void __launch_bounds__(kThreads)
decode2_kernel(const uint8_t *__restrict__ in, float *__restrict__ dstf, LaunchGeom g, int layout, int vec)
{
    constexpr int NW = RATE / 2;              // 32-bit words per block
    __shared__ uint32_t stile[kWarps][(NW + 1) * 32];
    __shared__ uint32_t splanes[kWarps][16 * 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t *t32 = stile[wid];
    SmemPlanes16 pl{splanes[wid], lane};
    __shared__ DropTable drop;
    const WithDrop<StreamTile> tile(StreamTile{t32, lane}, drop);
    load_drop<kThreads>(drop);
    __syncthreads();
    t32[NW * 32 + lane] = 0u;                 // a zero word after the stream
    const int64_t W = (int64_t)gridDim.x * kWarps;
    const int64_t gw = (int64_t)blockIdx.x * kWarps + wid;
    int64_t c = gw * g.nunits / W;
    const int64_t c1 = (gw + 1) * g.nunits / W;
    if (c >= c1) return;
    MsgWalk walk;
    walk.start(g.msgs, g.nmsg, c);
    for (; c < c1; c++) {
        walk.advance(c);
        const MsgDev &m = g.msgs[walk.mi];
        const int64_t b0 = (c - m.unit0) * 32;
        const int nact = (int)min((int64_t)32, m.nblocks - b0);
        if (lane >= nact) continue;
        const int nx = m.nx, ny = m.ny;
        const int64_t boff = layout ? m.off[1] : m.off[0];
        const uint32_t b = (uint32_t)b0 + lane;
        // this lane's block: 16-byte loads into its own tile column
        const uint4 *src4 = reinterpret_cast<const uint4 *>(in + boff) + (int64_t)b * (NW / 4);
#pragma unroll
        for (int i = 0; i < NW / 4; i++) {
            const uint4 v = __ldg(src4 + i);
            t32[(4 * i) * 32 + lane] = v.x;
            t32[(4 * i + 1) * 32 + lane] = v.y;
            t32[(4 * i + 2) * 32 + lane] = v.z;
            t32[(4 * i + 3) * 32 + lane] = v.w;
        }
        float v[16];
        decode_block2_tile<RATE>(tile, v, pl);
        const uint32_t t = divu(b, m.bxm, m.bxl), z = divu(t, m.bym, m.byl);
        const int x0 = 4 * (int)(b - t * (uint32_t)m.bx), y0 = 4 * (int)(t - z * (uint32_t)m.by);
        float *base = dstf + m.dst_off + (int64_t)z * g.ds[2] + (int64_t)y0 * g.ds[1];
        if (vec && x0 + 4 <= nx) {
            float *row = base + x0;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                if (y0 + j < ny)
                    *reinterpret_cast<float4 *>(row) = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                row += g.ds[1];
            }
        } else {
#pragma unroll
            for (int r = 0; r < 16; r++) {
                const int i = r & 3, j = r >> 2;
                if (x0 + i < nx && y0 + j < ny) base[(int64_t)j * g.ds[1] + (int64_t)(x0 + i) * g.ds[0]] = v[r];
            }
        }
    }
}

// ================================================================= launch
template <class K>
int grid_for(K kernel, int64_t nunits, int warps = kWarps)
{
    const int occ = occupancy((const void *)kernel, 32 * warps);
    const int64_t want = (nunits + warps - 1) / warps;
    const int64_t cap = (int64_t)num_sms() * occ;
    return (int)std::max<int64_t>(1, std::min(want, cap));
}

bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// Consecutive 32-block units per warp of the 3-D kernels, [encode][rate 16?];
// 0 = default: two, and one in launches of at most kFewUnits units per
// resident warp.  A warp's units run one after the other, so where a launch is
// little more than one wave of warps a second unit doubles its time (a 64 x 32
// x 8 field: 18.4 us a kernel with two, 10.2 with one; 233 x 117 x 137: 36.9 /
// 36.9 us against 26.6 / 26.6 compress / decompress), and one also ends a launch of a
// few waves more evenly (640 x 320 x 137 over 4 x 4 ranks, five waves: 73.7 /
// 75.8 against 71.7 / 73.7); in longer launches two halve the start-up of the
// warps (message search, tables; eight waves: 158 / 166 us against 174 / 188).
// The autotuner can override it; results never depend on it.
std::atomic<int> g_upw[2][2] = {{{0}, {0}}, {{0}, {0}}};
constexpr int kDefaultUpw = 2;
constexpr int kFewUnits = 6;

// One launch of a 3-D codec kernel (either alignment instantiation): one
// warp per upw consecutive units.
template <class In, class Out, class Acc>
void launch3(void (*kernel)(In, Out, LaunchGeom, int, Acc), int warps, int encode, int rate, LaunchGeom g,
             cudaStream_t st, In in, Out out, int layout, const Acc &acc = Acc{})
{
    g.upw = units_per_warp(encode, rate);
    if (g.upw <= 0) {
        const int64_t resident = (int64_t)num_sms() * occupancy((const void *)kernel, 32 * warps) * warps;
        g.upw = g.nunits <= kFewUnits * resident ? 1 : kDefaultUpw;
    }
    const int64_t per_cta = (int64_t)g.upw * warps;
    const int64_t grid = (g.nunits + per_cta - 1) / per_cta;
    kernel<<<(unsigned)grid, 32 * warps, 0, st>>>(in, out, g, layout, acc);
}

// A warp per block (zfpx_warp3.cuh) where that leaves an SM no more than 14 warps,
// unless the units per warp were set.  Up to there a launch's time is one
// warp's: 256 blocks at rate 8 / 16 compress in 6.2 / 6.2 us where a lane per block takes
// 8.2 / 9.2, decompress in 8.2 / 8.2 against 10.3 / 12.3; 2048 blocks 6.2 / 6.2 against
// 8.2 / 10.3 and 8.2 / 10.3 against 10.3 / 12.3.  Beyond, the eight times as many
// instructions show: 4000 blocks 8.2 / 8.2 and 12.1 / 12.3 us (the same as a lane per
// block, or more), 8192 blocks 11.1 / 11.3 and 16.4 / 18.5 against 8.2 / 10.3 and 10.3 / 12.3.
constexpr int kWarpPerBlockPerSm = 14;
bool warp_per_block(int encode, int rate, int64_t nunits)
{
    return units_per_warp(encode, rate) <= 0 && nunits * 32 <= (int64_t)kWarpPerBlockPerSm * num_sms();
}

// vec: rows start on 16 bytes wherever a block starts (x0 multiple of 4).
bool vec_ok(const void *ptr, const int64_t s[3], const zfpx_plan_s *p, int which /*0 src,1 dst*/)
{
    if (!aligned16(ptr) || s[0] != 1 || (s[1] & 3) || (s[2] & 3)) return false;
    (void)which;
    for (const HostMsg &m : p->msgs)
        if (m.x0 & 3) return false;
    return true;
}

}  // namespace

bool codec_vec_ok(const void *ptr, const int64_t s[3], const zfpx_plan_s *p) { return vec_ok(ptr, s, p, 0); }

int launch_encode(int dims, int rate, const float *src, uint8_t *out, const LaunchGeom &g, int layout, int vec,
                  cudaStream_t st)
{
    if (g.nunits == 0) return ZFPX_OK;
    if (dims == 3 && warp_per_block(1, rate, g.nunits)) {
        const unsigned grid = (unsigned)g.nunits * (32 / kWarps);
        if (rate == 8) encode3_warp_kernel<8><<<grid, kThreads, 0, st>>>(src, out, g, layout);
        else encode3_warp_kernel<16><<<grid, kThreads, 0, st>>>(src, out, g, layout);
    } else if (dims == 3) {
        if (rate == 8)
            launch3(vec ? encode3_kernel<8, true, false> : encode3_kernel<8, false, false>, kEnc3Warps<8>, 1, 8, g, st, src, out,
                    layout);
        else
            launch3(vec ? encode3_kernel<16, true, false> : encode3_kernel<16, false, false>, kEnc3Warps<16>, 1, 16, g, st, src, out,
                    layout);
    } else if (dims == 2) {
        if (rate == 8) encode2_kernel<8><<<grid_for(encode2_kernel<8>, g.nunits), kThreads, 0, st>>>(src, out, g, layout, vec);
        else encode2_kernel<16><<<grid_for(encode2_kernel<16>, g.nunits), kThreads, 0, st>>>(src, out, g, layout, vec);
    } else {
        if (rate == 8) encode1_kernel<8><<<grid_for(encode1_kernel<8>, g.nunits), kThreads, 0, st>>>(src, out, g, layout, vec);
        else encode1_kernel<16><<<grid_for(encode1_kernel<16>, g.nunits), kThreads, 0, st>>>(src, out, g, layout, vec);
    }
    count_launch();
    return check_launch();
}

int launch_decode(int dims, int rate, const uint8_t *in, float *dst, const LaunchGeom &g, int layout, int vec,
                  cudaStream_t st)
{
    if (g.nunits == 0) return ZFPX_OK;
    if (dims == 3 && warp_per_block(0, rate, g.nunits)) {
        const unsigned grid = (unsigned)g.nunits * (32 / kWarps);
        if (rate == 8) decode3_warp_kernel<8><<<grid, kThreads, 0, st>>>(in, dst, g, layout);
        else decode3_warp_kernel<16><<<grid, kThreads, 0, st>>>(in, dst, g, layout);
    } else if (dims == 3) {
        if (rate == 8)
            launch3(vec ? decode3_kernel<8, true, false> : decode3_kernel<8, false, false>, kDec3Warps<8>, 0, 8, g, st, in, dst,
                    layout);
        else
            launch3(vec ? decode3_kernel<16, true, false> : decode3_kernel<16, false, false>, kDec3Warps<16>, 0, 16, g, st, in, dst,
                    layout);
    } else if (dims == 2) {
        if (rate == 8) decode2_kernel<8><<<grid_for(decode2_kernel<8>, g.nunits), kThreads, 0, st>>>(in, dst, g, layout, vec);
        else decode2_kernel<16><<<grid_for(decode2_kernel<16>, g.nunits), kThreads, 0, st>>>(in, dst, g, layout, vec);
    } else {
        if (rate == 8) decode1_kernel<8><<<grid_for(decode1_kernel<8>, g.nunits), kThreads, 0, st>>>(in, dst, g, layout, vec);
        else decode1_kernel<16><<<grid_for(decode1_kernel<16>, g.nunits), kThreads, 0, st>>>(in, dst, g, layout, vec);
    }
    count_launch();
    return check_launch();
}

int launch_encode_lengths(const float *src, uint8_t *slots, const LaunchGeom &g, int vec, const AccEncode &a,
                          cudaStream_t st)
{
    if (g.nunits == 0) return ZFPX_OK;
    launch3(vec ? encode3_kernel<16, true, true> : encode3_kernel<16, false, true>, kEnc3Warps<16>, 1, 16, g, st, src,
            slots, (int)ZFPX_LAYOUT_SEND, a);
    count_launch();
    return check_launch();
}

int launch_decode_payload(float *dst, const LaunchGeom &g, int vec, const AccDecode &a, cudaStream_t st)
{
    if (g.nunits == 0) return ZFPX_OK;
    launch3(vec ? decode3_kernel<16, true, true> : decode3_kernel<16, false, true>, kDec3Warps<16>, 0, 16, g, st,
            (const uint8_t *)nullptr, dst, (int)ZFPX_LAYOUT_RECV, a);
    count_launch();
    return check_launch();
}

int units_per_warp(int encode, int rate)
{
    return g_upw[encode ? 1 : 0][rate == 16 ? 1 : 0].load(std::memory_order_relaxed);
}
}  // namespace zfpx

using namespace zfpx;

extern "C" {

int zfpx_set_units_per_warp(int encode, int rate, int upw)
{
    if (!valid_codec_rate(rate) || upw < 0 || upw > 4096) return ZFPX_EINVAL;
    g_upw[encode ? 1 : 0][rate == 16 ? 1 : 0].store(upw, std::memory_order_relaxed);
    return ZFPX_OK;
}

int zfpx_get_units_per_warp(int encode, int rate)
{
    if (!valid_codec_rate(rate)) return ZFPX_EINVAL;
    return units_per_warp(encode, rate);
}

int zfpx_pack_compress(zfpx_plan p, int rate, const float *d_src, uint8_t *d_out, size_t cap, int layout,
                       void *stream)
{
    if (!p || !d_src || !d_out || !valid_codec_rate(rate)) return ZFPX_EINVAL;
    if (layout != ZFPX_LAYOUT_SEND && layout != ZFPX_LAYOUT_RECV) return ZFPX_EINVAL;
    if ((uintptr_t)d_out & 15u) return ZFPX_EINVAL;
    if ((int64_t)cap < buffer_bytes(p, rate)) return ZFPX_ESIZE;
    DevTable *t = nullptr;
    int rc = get_table(p, rate, UNIT_BLOCKS32, &t);
    if (rc) return rc;
    LaunchGeom g{};
    g.msgs = t->d_msgs; g.nmsg = (int)p->msgs.size(); g.nunits = t->nunits;
    for (int a = 0; a < 3; a++) { g.ss[a] = p->ss[a]; g.ds[a] = p->ds[a]; }
    const int vec = vec_ok(d_src, p->ss, p, 0) ? 1 : 0;
    return launch_encode(p->dims, rate, d_src, d_out, g, layout, vec, (cudaStream_t)stream);
}

int zfpx_decompress_unpack(zfpx_plan p, int rate, const uint8_t *d_in, size_t len, float *d_dst, int layout,
                           void *stream)
{
    if (!p || !d_in || !d_dst || !valid_codec_rate(rate)) return ZFPX_EINVAL;
    if (layout != ZFPX_LAYOUT_SEND && layout != ZFPX_LAYOUT_RECV) return ZFPX_EINVAL;
    if ((uintptr_t)d_in & 15u) return ZFPX_EINVAL;
    if ((int64_t)len < buffer_bytes(p, rate)) return ZFPX_ESIZE;
    DevTable *t = nullptr;
    int rc = get_table(p, rate, UNIT_BLOCKS32, &t);
    if (rc) return rc;
    LaunchGeom g{};
    g.msgs = t->d_msgs; g.nmsg = (int)p->msgs.size(); g.nunits = t->nunits;
    for (int a = 0; a < 3; a++) { g.ss[a] = p->ss[a]; g.ds[a] = p->ds[a]; }
    const int vec = vec_ok(d_dst, p->ds, p, 1) ? 1 : 0;
    return launch_decode(p->dims, rate, d_in, d_dst, g, layout, vec, (cudaStream_t)stream);
}

size_t zfpx_stream_bytes(int dims, int rate, const int64_t n[3])
{
    if (!n || dims < 1 || dims > 3 || !valid_codec_rate(rate)) return 0;
    for (int a = 0; a < 3; a++) if (n[a] < 1) return 0;
    const int64_t bx = (n[0] + 3) / 4;
    if (dims == 3) return (size_t)(bx * ((n[1] + 3) / 4) * ((n[2] + 3) / 4) * 8 * rate);
    if (dims == 2) return (size_t)(bx * ((n[1] + 3) / 4) * n[2] * 2 * rate);
    return (size_t)(bx * n[1] * n[2] * rate / 2);
}

}  // extern "C"

// The raw-array entry points run the same kernels on a one-message table
// that lives in a small per-device cache of plans keyed by shape.
#include <map>
#include <tuple>
namespace zfpx {
namespace {
std::mutex g_raw_mu;
std::map<std::tuple<int, int, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t>, zfpx_plan> g_raw_plans;
}  // namespace

int raw_plan(int dims, const int64_t n[3], const int64_t s[3], zfpx_plan *out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ZFPX_ECUDA;
    auto key = std::make_tuple(dev, dims, n[0], n[1], n[2], s[0], s[1], s[2]);
    std::lock_guard<std::mutex> g(g_raw_mu);
    auto it = g_raw_plans.find(key);
    if (it != g_raw_plans.end()) { *out = it->second; return ZFPX_OK; }
    if (g_raw_plans.size() > 256) {   // bounded cache
        for (auto &kv : g_raw_plans) zfpx_plan_destroy(kv.second);
        g_raw_plans.clear();
    }
    zfpx_view3 v;
    for (int a = 0; a < 3; a++) { v.n[a] = n[a]; v.stride[a] = s[a]; }
    int rc = zfpx_plan_create(out, &v, &v, 1, 1, 0, dims, ZFPX_SPLIT_BALANCED);
    if (rc) return rc;
    g_raw_plans[key] = *out;
    return ZFPX_OK;
}
}  // namespace zfpx

extern "C" {

int zfpx_encode(int dims, int rate, const float *d_in, const int64_t n[3], const int64_t stride[3],
                uint8_t *d_out, size_t cap, void *stream)
{
    if (!d_in || !d_out || !n || !stride || dims < 1 || dims > 3 || !valid_codec_rate(rate)) return ZFPX_EINVAL;
    for (int a = 0; a < 3; a++) if (n[a] < 1 || stride[a] < 0) return ZFPX_EINVAL;
    if (cap < zfpx_stream_bytes(dims, rate, n)) return ZFPX_ESIZE;
    zfpx_plan p = nullptr;
    int rc = raw_plan(dims, n, stride, &p);
    if (rc) return rc;
    return zfpx_pack_compress(p, rate, d_in, d_out, cap + 256, ZFPX_LAYOUT_SEND, stream);
}

int zfpx_decode(int dims, int rate, const uint8_t *d_in, size_t len, const int64_t n[3], const int64_t stride[3],
                float *d_out, void *stream)
{
    if (!d_in || !d_out || !n || !stride || dims < 1 || dims > 3 || !valid_codec_rate(rate)) return ZFPX_EINVAL;
    for (int a = 0; a < 3; a++) if (n[a] < 1 || stride[a] < 0) return ZFPX_EINVAL;
    if (len < zfpx_stream_bytes(dims, rate, n)) return ZFPX_ESIZE;
    zfpx_plan p = nullptr;
    int rc = raw_plan(dims, n, stride, &p);
    if (rc) return rc;
    return zfpx_decompress_unpack(p, rate, d_in, len + 256, d_out, ZFPX_LAYOUT_SEND, stream);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// A transposition that allocates nothing.
//
// For callers that cannot allocate device memory at the point of the call --
// code running inside another framework's memory pool or allocator, real-time
// loops that must not pay for an allocation, programs with a fixed device
// memory map -- zfpx_transpose_noalloc keeps everything it needs beyond the
// caller's source and destination fields in one file-scope device array: the
// message table of the plan and the compressed messages (written straight
// into the receive layout, then decoded).  The array is ZFPX_NOALLOC_SCRATCH_BYTES
// long and stays reserved on every GPU that loads the library until the
// process exits.  Every call shares it and leaves its contents behind; nothing
// here depends on what an earlier call left (each call rewrites the table and
// every stream byte it later reads), but calls that overlap on the GPU -- on
// different streams, or from different host threads -- race on it.
#include <algorithm>
#include <mutex>
#include <vector>

static __device__ __align__(256) unsigned char g_noalloc_scratch[ZFPX_NOALLOC_SCRATCH_BYTES];

namespace zfpx {
namespace {
// device address of the scratch array, looked up once per device with that
// device current (a host-side name of the array is not a device address)
std::mutex g_noalloc_mu;
void *g_noalloc_ptr[64] = {nullptr};

int noalloc_scratch(void **out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return ZFPX_ECUDA;
    std::lock_guard<std::mutex> g(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return ZFPX_ECUDA;
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return ZFPX_OK;
}
}  // namespace
}  // namespace zfpx

extern "C" int zfpx_transpose_noalloc(zfpx_plan p, int rate, const float *d_src, float *d_dst, void *stream)
{
    if (!p || !d_src || !d_dst || !valid_codec_rate(rate)) return ZFPX_EINVAL;
    // message table (32-block work units, receive-layout offsets), built on the host
    const size_t M = p->msgs.size();
    std::vector<MsgDev> h(M);
    int64_t units = 0, so = 0, ro = 0;
    std::vector<int64_t> recv_off(M, 0);
    {
        std::vector<size_t> order(M);
        for (size_t i = 0; i < M; i++) order[i] = i;
        std::stable_sort(order.begin(), order.end(), [&](size_t a, size_t b) {
            const HostMsg &x = p->msgs[a], &y = p->msgs[b];
            return x.dst != y.dst ? x.dst < y.dst : x.src_peer < y.src_peer;
        });
        for (size_t i : order) {
            recv_off[i] = ro;
            ro = (ro + message_bytes(p, p->msgs[i], rate) + 255) / 256 * 256;
        }
    }
    for (size_t i = 0; i < M; i++) {
        const HostMsg &m = p->msgs[i];
        MsgDev &d = h[i];
        const int64_t bx = (m.nx + 3) / 4;
        const int64_t by = p->dims >= 2 ? (m.ny + 3) / 4 : m.ny;
        const int64_t bz = p->dims == 3 ? (m.nz + 3) / 4 : m.nz;
        d.src_off = m.x0 * p->ss[0] + m.y0 * p->ss[1] + m.z0 * p->ss[2];
        d.dst_off = m.x0 * p->ds[0] + m.y0 * p->ds[1] + m.z0 * p->ds[2];
        d.off[0] = so;
        d.off[1] = recv_off[i];
        so = (so + message_bytes(p, m, rate) + 255) / 256 * 256;
        d.nx = (int32_t)m.nx; d.ny = (int32_t)m.ny; d.nz = (int32_t)m.nz;
        d.bx = (int32_t)bx; d.by = (int32_t)by; d.bz = (int32_t)bz;
        d.nblocks = bx * by * bz;
        set_block_divisors(d);
        d.unit0 = units;
        units += (d.nblocks + 31) / 32;
    }
    const size_t table_bytes = (M * sizeof(MsgDev) + 255) / 256 * 256;
    const size_t stream_bytes = (size_t)ro;
    // layout of the array: the message table, then the compressed messages
    if (table_bytes + stream_bytes > ZFPX_NOALLOC_SCRATCH_BYTES) return ZFPX_ESIZE;
    cudaStream_t st = (cudaStream_t)stream;
    // the table is copied from pageable host memory, which a stream capture
    // cannot record: refuse while the stream is capturing
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return ZFPX_ECUDA;
    if (cs != cudaStreamCaptureStatusNone) return ZFPX_EINVAL;
    void *scratch = nullptr;
    int rc = noalloc_scratch(&scratch);
    if (rc) return rc;
    if (units == 0) return ZFPX_OK;
    // pageable source: the copy has read h before this call returns
    uint8_t *base = static_cast<uint8_t *>(scratch);
    if (cudaMemcpyAsync(base, h.data(), M * sizeof(MsgDev), cudaMemcpyHostToDevice, st) != cudaSuccess)
        return ZFPX_ECUDA;
    uint8_t *buf = base + table_bytes;
    LaunchGeom g{};
    g.msgs = reinterpret_cast<const MsgDev *>(base);
    g.nmsg = (int)M;
    g.nunits = units;
    for (int a = 0; a < 3; a++) { g.ss[a] = p->ss[a]; g.ds[a] = p->ds[a]; }
    rc = launch_encode(p->dims, rate, d_src, buf, g, ZFPX_LAYOUT_RECV, vec_ok(d_src, p->ss, p, 0) ? 1 : 0, st);
    if (rc) return rc;
    return launch_decode(p->dims, rate, buf, d_dst, g, ZFPX_LAYOUT_RECV, vec_ok(d_dst, p->ds, p, 1) ? 1 : 0, st);
}
