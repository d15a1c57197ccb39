// Accuracy and precision modes: variable-rate coding of 3-D blocks to an
// absolute error tolerance, or to a fixed number of bit planes per block (the
// ZFP modes the paper names and leaves for future work, Sec. II-C), built on
// the fixed-rate kernels.  Precision p keeps planes 31 .. 32 - p; the rest of
// what follows holds for both.
//
// Readings (identical in the CPU oracle): minexp = floor(log2 tol); a block
// with exponent e_max keeps its bit planes 31 .. kmin, kmin = clamp(minexp -
// e_max + 22, 0, 32), cut at the rate-16 budget of 1024 bits; a zero block is
// its one 0 bit, a block with kmin = 32 its 9 header bits.  Because the plane
// coder is embedded, a block's accuracy-mode bits are the first L bits of its
// rate-16 stream, and the rate-16 decoder reads the same block from those L
// bits followed by zeros (zeros after the last coded plane are empty planes).
//
// Encode: the rate-16 encoder writes every block to a 128-byte slot and, as it
// walks the planes, its bit count L; an exclusive scan of the L (per 1024-block
// tile, then over the tiles) gives every block's bit offset; one warp per 32
// blocks shifts their bits together in shared memory and writes the payload
// words that start in them, each once (the last with the leading bits of the
// blocks that follow), so the payload needs no zeroing but its tail and no
// atomics in global memory.  Decode: the same scan, then the rate-16
// decoder, which cuts each block's bits out of the payload as it loads them.
// What bounds it: the codec; the rest moves a slot once out and once in.  With a
// parse of every slot for L, a zeroed payload filled by atomics, and slots
// copied out for the decoder, compress, exchange and decompress of a 640 x 320 x
// 137 field over 4 x 4 ranks at tolerance 1e-3 took 351, 93 and 212 us; now 138,
// 23 and 126.
#include <algorithm>
#include <cmath>
#include <vector>
#include <cuda_runtime.h>

#include "zfpx_internal.h"

namespace zfpx {
namespace {

constexpr int kTile = kAccTile;              // blocks per scan tile (one CTA)

// Exclusive scan of the lengths inside each tile of kTile blocks; the tile's
// total goes to totals[tile].
__global__ void __launch_bounds__(kTile) acc_scan_tiles_kernel(const uint16_t *__restrict__ lengths,
                                                               int64_t nblocks, uint32_t *__restrict__ local,
                                                               uint64_t *__restrict__ totals)
{
    __shared__ uint32_t warp_sum[kTile / 32];
    start_next();
    wait_previous(lengths);
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int64_t b = (int64_t)blockIdx.x * kTile + t;
    const uint32_t v = b < nblocks ? lengths[b] : 0u;
    uint32_t x = v;                                        // inclusive scan in the warp
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) warp_sum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t s = warp_sum[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, s, d);
            if (lane >= d) s += y;
        }
        warp_sum[lane] = s;                                // inclusive over warps
    }
    __syncthreads();
    const uint32_t before = (wid ? warp_sum[wid - 1] : 0u) + x - v;
    if (b < nblocks) local[b] = before;
    if (t == kTile - 1) totals[blockIdx.x] = warp_sum[kTile / 32 - 1];
}

// Exclusive sum over a CTA of kTile threads (`sums`: kTile / 32 shared values);
// *total gets the sum of all.  Every thread calls it; sums may be reused after
// the next barrier.
__device__ __forceinline__ uint64_t cta_scan(uint64_t v, uint64_t *sums, uint64_t *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint64_t s = sums[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, s, d);
            if (lane >= d) s += y;
        }
        sums[lane] = s;
    }
    __syncthreads();
    *total = sums[kTile / 32 - 1];
    return (wid ? sums[wid - 1] : 0ull) + x - v;
}

// Exclusive scan of the tile totals (one CTA, sequential over chunks of
// kTile tiles); the grand total goes to *total_bits.
__global__ void __launch_bounds__(kTile) acc_scan_totals_kernel(const uint64_t *__restrict__ totals, int64_t ntiles,
                                                                uint64_t *__restrict__ tile_off,
                                                                uint64_t *__restrict__ total_bits)
{
    __shared__ uint64_t sums[kTile / 32];
    start_next();
    wait_previous(totals);
    uint64_t carry = 0, all;
    for (int64_t base = 0; base < ntiles; base += kTile) {
        const int64_t i = base + threadIdx.x;
        const uint64_t before = cta_scan(i < ntiles ? totals[i] : 0ull, sums, &all);
        if (i < ntiles) tile_off[i] = carry + before;
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total_bits = carry;
}

// The block list a pack kernel walks: M messages in send order (msgs NULL: one
// message, its slots from 0 on, its payload from word 0 on).
struct AccList {
    const AccMsg *msgs;
    const int64_t *pay;        // first payload word of each message
    const uint16_t *lengths;
    const uint32_t *local;
    const uint64_t *tile_off;
    int M;
    int64_t G;
    __device__ __forceinline__ uint64_t bit(int64_t g) const { return tile_off[g / kTile] + local[g]; }
    // the last message whose blocks start at or before g
    __device__ __forceinline__ int message(int64_t g) const
    {
        int lo = 0, hi = M - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (msgs[mid].gb0 <= g) lo = mid; else hi = mid - 1;
        }
        return lo;
    }
    // block g's first bit in the payload and its slot's first byte
    __device__ __forceinline__ void place(int64_t g, uint64_t &off, int64_t &slot) const
    {
        if (!msgs) {
            off = bit(g);
            slot = g * 128;
            return;
        }
        const int m = message(g);
        const AccMsg a = msgs[m];
        off = (uint64_t)pay[m] * 64 + (bit(g) - bit(a.gb0));
        slot = a.slot_send + (g - a.gb0) * 128;
    }
};

// One warp per 32 consecutive blocks writes the payload words whose first bit
// lies in them.  Block by block the lanes read the slot's 32 words, shift them
// to the block's place in the warp's shared words and OR them in; the word the
// last block ends in also takes the first bits of the blocks that follow, up to
// 63 of them.  (Messages start on words, so every word's first bit is in some
// block.)
constexpr int kPackWarps = 4;
constexpr int kPackWords = 32 * 32 + 4;       // 32-bit words: 32 blocks of at most 16 64-bit words, and the last word
__global__ void __launch_bounds__(32 * kPackWarps) acc_pack_kernel(AccList P, const uint8_t *__restrict__ slots,
                                                                   uint64_t *__restrict__ payload)
{
    __shared__ __align__(8) uint32_t buf[kPackWarps][kPackWords];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t g0 = ((int64_t)blockIdx.x * kPackWarps + wid) * 32;
    start_next();
    uint32_t *w = buf[wid];
    for (int i = lane; i < kPackWords; i += 32) w[i] = 0u;
    wait_previous(slots);
    if (g0 >= P.G) return;
    const int n = (int)min((int64_t)32, P.G - g0);
    const int64_t g = g0 + min(lane, n - 1);
    uint64_t off;
    int64_t slot;
    P.place(g, off, slot);
    const int L = P.lengths[g];
    const uint64_t first = __shfl_sync(0xffffffffu, off, 0), end = __shfl_sync(0xffffffffu, off + L, n - 1);
    const uint64_t base = first & ~63ull;      // w[0] holds the payload's bits from here on
    const uint32_t rel = (uint32_t)(off - base);
    __syncwarp();
    // eight blocks at a time, all their loads ahead of the shifting (past the
    // warp's last block lengths are 0)
    const int Lw = lane < n ? L : 0;
#pragma unroll 1
    for (int b0 = 0; b0 < n; b0 += 8) {
        uint32_t v[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int len = __shfl_sync(0xffffffffu, Lw, b0 + k) - 32 * lane;
            const int64_t s = __shfl_sync(0xffffffffu, slot, b0 + k);
            v[k] = len > 0 ? __ldg(reinterpret_cast<const uint32_t *>(slots + s) + lane) : 0u;
            if (len > 0 && len < 32) v[k] &= (1u << len) - 1u;
        }
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const uint32_t r = __shfl_sync(0xffffffffu, rel, b0 + k);
            const uint64_t x = (uint64_t)v[k] << (r & 31u);
            if ((uint32_t)x) atomicOr(w + (r >> 5) + lane, (uint32_t)x);
            if ((uint32_t)(x >> 32)) atomicOr(w + (r >> 5) + lane + 1, (uint32_t)(x >> 32));
        }
    }
    // the words owned: those starting at or after `first`, up to the one `end` lies in
    const uint64_t j0 = (first + 63) >> 6, j1 = (end + 63) >> 6;
    if (j1 > j0 && (end & 63u)) {
        const uint64_t wend = j1 * 64;
        for (int64_t t = g0 + n + lane; ; t += 32) {
            uint64_t o = wend;
            int64_t sl = 0;
            if (t < P.G) P.place(t, o, sl);
            if (o < wend) {
                uint64_t v = __ldg(reinterpret_cast<const uint64_t *>(slots + sl));
                const int len = P.lengths[t];
                if (len < 64) v &= (1ull << len) - 1ull;
                v <<= o & 63u;
                uint32_t *d = w + (uint32_t)((wend - 64 - base) >> 5);
                if ((uint32_t)v) atomicOr(d, (uint32_t)v);
                if ((uint32_t)(v >> 32)) atomicOr(d + 1, (uint32_t)(v >> 32));
            }
            if (!__all_sync(0xffffffffu, o < wend)) break;
        }
    }
    __syncwarp();
    const uint64_t *w64 = reinterpret_cast<const uint64_t *>(w);
    for (uint64_t j = j0 + lane; j < j1; j += 32) payload[j] = w64[j - (base >> 6)];
}

// Zeroes the payload's words from its end on: *count words (bits rounded up
// to words where `bits` is set) up to `words`.
__global__ void __launch_bounds__(256) acc_zero_tail_kernel(uint64_t *__restrict__ payload,
                                                            const uint64_t *__restrict__ count, int bits, int64_t words)
{
    start_next();
    wait_previous(count);
    const int64_t used = (int64_t)(bits ? (*count + 63) / 64 : *count);
    for (int64_t i = used + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words;
         i += (int64_t)gridDim.x * blockDim.x)
        payload[i] = 0ull;
}

struct AccWork {
    uint64_t *slots;
    uint32_t *local;
    uint64_t *totals, *tile_off, *total;
    int64_t nblocks, ntiles;
};

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

int64_t acc_blocks(const int64_t n[3]) { return ((n[0] + 3) / 4) * ((n[1] + 3) / 4) * ((n[2] + 3) / 4); }

size_t acc_work_bytes(int64_t nb)
{
    const int64_t nt = (nb + kTile - 1) / kTile;
    return align256((size_t)nb * 128) + align256((size_t)nb * 4) + 2 * align256((size_t)nt * 8) + 256;
}

AccWork acc_carve(void *work, int64_t nb)
{
    AccWork a;
    a.nblocks = nb;
    a.ntiles = (nb + kTile - 1) / kTile;
    char *p = static_cast<char *>(work);
    a.slots = reinterpret_cast<uint64_t *>(p); p += align256((size_t)nb * 128);
    a.local = reinterpret_cast<uint32_t *>(p); p += align256((size_t)nb * 4);
    a.totals = reinterpret_cast<uint64_t *>(p); p += align256((size_t)a.ntiles * 8);
    a.tile_off = reinterpret_cast<uint64_t *>(p); p += align256((size_t)a.ntiles * 8);
    a.total = reinterpret_cast<uint64_t *>(p);
    return a;
}

int plan_geom(zfpx_plan p, LaunchGeom &g)
{
    DevTable *t = nullptr;
    const int rc = get_table(p, 16, UNIT_BLOCKS32, &t);
    if (rc) return rc;
    g.msgs = t->d_msgs; g.nmsg = (int)p->msgs.size(); g.nunits = t->nunits;
    for (int a = 0; a < 3; a++) { g.ss[a] = p->ss[a]; g.ds[a] = p->ds[a]; }
    return ZFPX_OK;
}

int acc_scan(const AccWork &a, const uint16_t *lengths, uint64_t *total_bits, cudaStream_t st)
{
    launch_after(acc_scan_tiles_kernel, (unsigned)a.ntiles, kTile, 0, st, lengths, a.nblocks, a.local, a.totals);
    count_launch();
    launch_after(acc_scan_totals_kernel, 1, kTile, 0, st, a.totals, a.ntiles, a.tile_off, total_bits);
    count_launch();
    return check_launch();
}

// Packs the slots of the listed blocks; *count (words, or bits) ends the payload.
int acc_pack(const AccList &P, const uint8_t *slots, uint8_t *payload, const uint64_t *count, int bits, cudaStream_t st)
{
    const int64_t per_cta = 32 * kPackWarps;
    launch_after(acc_pack_kernel, (unsigned)((P.G + per_cta - 1) / per_cta), 32 * kPackWarps, 0, st, P, slots, reinterpret_cast<uint64_t *>(payload));
    count_launch();
    const int64_t words = P.G * 16, want = (words + 255) / 256;
    launch_after(acc_zero_tail_kernel, (unsigned)std::min<int64_t>(want, (int64_t)num_sms() * 8), 256, 0, st, reinterpret_cast<uint64_t *>(payload), count, bits, words);
    count_launch();
    return check_launch();
}

// Launch geometry of a raw array (its one-message table) for the rate-16 codec.
int raw_geom(const int64_t n[3], const int64_t stride[3], const void *base, LaunchGeom &g, int &vec)
{
    zfpx_plan p = nullptr;
    int rc = raw_plan(3, n, stride, &p);
    if (!rc) rc = plan_geom(p, g);
    if (!rc) vec = codec_vec_ok(base, stride, p) ? 1 : 0;
    return rc;
}

bool aligned(const void *p, size_t a) { return ((uintptr_t)p % a) == 0; }

}  // namespace
}  // namespace zfpx

using namespace zfpx;

extern "C" {

size_t zfpx_accuracy_workspace_bytes(const int64_t n[3])
{
    if (!n || n[0] < 1 || n[1] < 1 || n[2] < 1) return 0;
    return acc_work_bytes(acc_blocks(n));
}

size_t zfpx_accuracy_max_payload_bytes(const int64_t n[3])
{
    if (!n || n[0] < 1 || n[1] < 1 || n[2] < 1) return 0;
    return (size_t)acc_blocks(n) * 128;
}

static int encode_variable(const float *d_in, const int64_t n[3], const int64_t stride[3], int minexp, int prec,
                           uint16_t *d_lengths, uint8_t *d_payload, size_t cap, uint64_t *d_total_bits,
                           void *d_work, size_t work_bytes, void *stream)
{
    if (!d_in || !n || !stride || !d_lengths || !d_payload || !d_total_bits || !d_work) return ZFPX_EINVAL;
    for (int a = 0; a < 3; a++) if (n[a] < 1 || stride[a] < 0) return ZFPX_EINVAL;
    if (!aligned(d_payload, 8) || !aligned(d_work, 256) || !aligned(d_lengths, 2) || !aligned(d_total_bits, 8))
        return ZFPX_EINVAL;
    const int64_t nb = acc_blocks(n);
    if (cap < (size_t)nb * 128 || work_bytes < acc_work_bytes(nb)) return ZFPX_ESIZE;
    cudaStream_t st = (cudaStream_t)stream;
    const AccWork a = acc_carve(d_work, nb);
    LaunchGeom g{};
    int vec = 0, rc = raw_geom(n, stride, d_in, g, vec);
    if (rc) return rc;
    if ((rc = launch_encode_lengths(d_in, reinterpret_cast<uint8_t *>(a.slots), g, vec,
                                    AccEncode{d_lengths, nullptr, minexp, prec}, st)))
        return rc;
    if ((rc = acc_scan(a, d_lengths, d_total_bits, st))) return rc;
    return acc_pack(AccList{nullptr, nullptr, d_lengths, a.local, a.tile_off, 1, nb},
                    reinterpret_cast<const uint8_t *>(a.slots), d_payload, d_total_bits, 1, st);
}

int zfpx_encode_accuracy(const float *d_in, const int64_t n[3], const int64_t stride[3], double tolerance,
                         uint16_t *d_lengths, uint8_t *d_payload, size_t cap, uint64_t *d_total_bits,
                         void *d_work, size_t work_bytes, void *stream)
{
    if (!(tolerance > 0.0) || !(tolerance < HUGE_VAL)) return ZFPX_EINVAL;
    int e = 0;
    (void)frexp(tolerance, &e);                         // floor(log2 tolerance) = e - 1
    return encode_variable(d_in, n, stride, e - 1, 0, d_lengths, d_payload, cap, d_total_bits, d_work,
                           work_bytes, stream);
}

int zfpx_encode_precision(const float *d_in, const int64_t n[3], const int64_t stride[3], int precision,
                          uint16_t *d_lengths, uint8_t *d_payload, size_t cap, uint64_t *d_total_bits,
                          void *d_work, size_t work_bytes, void *stream)
{
    if (precision < 1 || precision > 32) return ZFPX_EINVAL;
    return encode_variable(d_in, n, stride, 0, precision, d_lengths, d_payload, cap, d_total_bits, d_work,
                           work_bytes, stream);
}

int zfpx_decode_accuracy(const uint16_t *d_lengths, const uint8_t *d_payload, size_t len, const int64_t n[3],
                         const int64_t stride[3], float *d_out, void *d_work, size_t work_bytes, void *stream)
{
    if (!d_lengths || !d_payload || !n || !stride || !d_out || !d_work) return ZFPX_EINVAL;
    for (int a = 0; a < 3; a++) if (n[a] < 1 || stride[a] < 0) return ZFPX_EINVAL;
    if (!aligned(d_payload, 8) || !aligned(d_work, 256) || !aligned(d_lengths, 2)) return ZFPX_EINVAL;
    const int64_t nb = acc_blocks(n);
    if (work_bytes < acc_work_bytes(nb)) return ZFPX_ESIZE;
    cudaStream_t st = (cudaStream_t)stream;
    const AccWork a = acc_carve(d_work, nb);
    LaunchGeom g{};
    int vec = 0, rc = raw_geom(n, stride, d_out, g, vec);
    if (rc || (rc = acc_scan(a, d_lengths, a.total, st))) return rc;
    return launch_decode_payload(d_out, g, vec,
                                 AccDecode{reinterpret_cast<const uint64_t *>(d_payload), (int64_t)(len / 8), d_lengths,
                                           a.local, a.tile_off, nullptr, nullptr},
                                 st);
}

}  // extern "C"

// ============================================================================
// The accuracy mode on a transposition plan: every message is coded as in the
// raw accuracy mode (its box's 3-D blocks, edge-replicated inside the box);
// messages become variable in size, so the exchange is an all-to-all-v: the
// per-message word counts go first, then the payloads.  On one GPU both are
// device-local copies.  A message's payload starts on a 64-bit word.
namespace zfpx {
std::vector<int64_t> layout_offsets(const zfpx_plan_s *p, int rate, int layout, int64_t *total);
namespace {

struct PlanAcc {
    const AccMsg *msgs;       // M, send order
    const int32_t *rorder;    // M: send index of the message at receive position r
    int64_t *pay_send;        // M: payload word offset in the send buffer
    int64_t *pay_recv;        // M: payload word offset in the receive buffer
    int M;
    int64_t G;                // blocks in all messages
};

// Word counts and payload offsets of the messages: one CTA, kTile messages at a
// time.  With `send` the counts come from the block scan of the send-order
// lengths and are written to words[]; otherwise words[] is input.  *used (if
// not NULL) gets the sum of the counts.
__global__ void __launch_bounds__(kTile) pacc_messages_kernel(PlanAcc P, const uint32_t *__restrict__ local,
                                                              const uint64_t *__restrict__ tile_off,
                                                              const uint64_t *__restrict__ total,
                                                              uint64_t *words, int send, uint64_t *used)
{
    __shared__ uint64_t sums[kTile / 32];
    start_next();
    wait_previous(local, tile_off, total);
    auto bit = [&](int64_t g) { return g < P.G ? tile_off[g / kTile] + local[g] : *total; };
    uint64_t carry = 0, all;
    for (int base = 0; base < P.M; base += kTile) {
        const int m = base + threadIdx.x;
        uint64_t v = 0;
        if (m < P.M) {
            if (send) {
                const AccMsg a = P.msgs[m];
                v = (bit(a.gb0 + a.nb) - bit(a.gb0) + 63) / 64;
                words[m] = v;
            } else {
                v = words[m];
            }
        }
        const uint64_t before = cta_scan(v, sums, &all);
        if (m < P.M) P.pay_send[m] = (int64_t)(carry + before);
        carry += all;
        __syncthreads();                          // sums, and words[] for the next loop
    }
    if (used && threadIdx.x == 0) *used = carry;
    carry = 0;
    for (int base = 0; base < P.M; base += kTile) {
        const int r = base + threadIdx.x;
        const int m = r < P.M ? P.rorder[r] : 0;
        const uint64_t before = cta_scan(r < P.M ? words[m] : 0ull, sums, &all);
        if (r < P.M) P.pay_recv[m] = (int64_t)(carry + before);
        carry += all;
        __syncthreads();
    }
}

// The all-to-all-v on one GPU: CTAs (m, *) move message m's payload words and
// its block bit counts from the send to the receive buffers, in equal parts.
__global__ void __launch_bounds__(256) pacc_exchange_kernel(PlanAcc P, const uint64_t *__restrict__ words,
                                                            const uint64_t *__restrict__ pay_in,
                                                            uint64_t *__restrict__ pay_out,
                                                            const uint16_t *__restrict__ len_in,
                                                            uint16_t *__restrict__ len_out, int64_t cap_words)
{
    start_next();
    wait_previous(words, pay_in, len_in);
    const int m = blockIdx.x;
    const AccMsg a = P.msgs[m];
    // counts that would run past either buffer are cut there
    const int64_t nw = min((int64_t)min(words[m], (uint64_t)cap_words),
                           cap_words - max(P.pay_send[m], P.pay_recv[m]));
    const uint64_t *s = pay_in + P.pay_send[m];
    uint64_t *d = pay_out + P.pay_recv[m];
    const int64_t t = (int64_t)blockIdx.y * blockDim.x + threadIdx.x, step = (int64_t)gridDim.y * blockDim.x;
#pragma unroll 4
    for (int64_t i = t; i < nw; i += step) d[i] = __ldg(s + i);
    for (int64_t i = t; i < a.nb; i += step) len_out[a.gr0 + i] = len_in[a.gb0 + i];
}

struct PlanAccWork {
    PlanAcc P;
    uint8_t *slots;
    AccWork scan;             // local / totals / tile_off / total for G blocks
    size_t bytes;
};

int64_t plan_blocks(const zfpx_plan_s *p, std::vector<AccMsg> *msgs, std::vector<int32_t> *rorder)
{
    const size_t M = p->msgs.size();
    auto c4 = [](int64_t v) { return (v + 3) / 4; };
    std::vector<int64_t> nb(M);
    int64_t G = 0;
    for (size_t i = 0; i < M; i++) {
        const HostMsg &m = p->msgs[i];
        nb[i] = c4(m.nx) * c4(m.ny) * c4(m.nz);
        G += nb[i];
    }
    if (!msgs) return G;
    const std::vector<int64_t> so = layout_offsets(p, 16, ZFPX_LAYOUT_SEND, nullptr);
    std::vector<int32_t> ord(M);
    for (size_t i = 0; i < M; i++) ord[i] = (int32_t)i;
    std::stable_sort(ord.begin(), ord.end(), [&](int32_t a, int32_t b) {
        const HostMsg &x = p->msgs[a], &y = p->msgs[b];
        return x.dst != y.dst ? x.dst < y.dst : x.src_peer < y.src_peer;
    });
    msgs->assign(M, AccMsg{});
    rorder->assign(ord.begin(), ord.end());
    int64_t g = 0;
    for (size_t i = 0; i < M; i++) {
        (*msgs)[i].gb0 = g; (*msgs)[i].nb = nb[i];
        (*msgs)[i].slot_send = so[i];
        g += nb[i];
    }
    g = 0;
    for (size_t r = 0; r < M; r++) {
        (*msgs)[ord[r]].gr0 = g;
        g += nb[ord[r]];
    }
    return G;
}

size_t plan_acc_bytes(const zfpx_plan_s *p, int64_t G)
{
    const size_t M = p->msgs.size();
    // 40 bytes a message and three words where the tables below take 32 and two:
    // the size stays what saved callers hold
    return align256((size_t)buffer_bytes(p, 16)) + acc_work_bytes(G) - align256((size_t)G * 128) +
           align256(M * 40) + align256(M * 4) + 3 * align256(M * 8);
}

static_assert(sizeof(AccMsg) <= 40, "the scratch holds the message table");

// Carves the scratch and uploads the message tables (pageable copies: the
// host vectors have been read when the call returns).
int plan_acc_setup(const zfpx_plan_s *p, void *work, size_t work_bytes, cudaStream_t st, PlanAccWork *w)
{
    std::vector<AccMsg> msgs;
    std::vector<int32_t> rorder;
    const int64_t G = plan_blocks(p, &msgs, &rorder);
    const size_t M = msgs.size();
    if (work_bytes < plan_acc_bytes(p, G)) return ZFPX_ESIZE;
    char *c = static_cast<char *>(work);
    w->slots = reinterpret_cast<uint8_t *>(c); c += align256((size_t)buffer_bytes(p, 16));
    w->scan.nblocks = G;
    w->scan.ntiles = (G + kTile - 1) / kTile;
    w->scan.slots = nullptr;
    w->scan.local = reinterpret_cast<uint32_t *>(c); c += align256((size_t)G * 4);
    w->scan.totals = reinterpret_cast<uint64_t *>(c); c += align256((size_t)w->scan.ntiles * 8);
    w->scan.tile_off = reinterpret_cast<uint64_t *>(c); c += align256((size_t)w->scan.ntiles * 8);
    w->scan.total = reinterpret_cast<uint64_t *>(c); c += 256;
    AccMsg *dm = reinterpret_cast<AccMsg *>(c); c += align256(M * sizeof(AccMsg));
    int32_t *dr = reinterpret_cast<int32_t *>(c); c += align256(M * 4);
    w->P.pay_send = reinterpret_cast<int64_t *>(c); c += align256(M * 8);
    w->P.pay_recv = reinterpret_cast<int64_t *>(c); c += align256(M * 8);
    w->P.msgs = dm; w->P.rorder = dr; w->P.M = (int)M; w->P.G = G;
    if (M && (cudaMemcpyAsync(dm, msgs.data(), M * sizeof(AccMsg), cudaMemcpyHostToDevice, st) != cudaSuccess ||
              cudaMemcpyAsync(dr, rorder.data(), M * 4, cudaMemcpyHostToDevice, st) != cudaSuccess))
        return ZFPX_ECUDA;
    return ZFPX_OK;
}

}  // namespace
}  // namespace zfpx

extern "C" {

size_t zfpx_plan_accuracy_blocks(zfpx_plan p)
{
    return p ? (size_t)plan_blocks(p, nullptr, nullptr) : 0;
}

size_t zfpx_plan_accuracy_workspace_bytes(zfpx_plan p)
{
    if (!p || p->dims != 3) return 0;
    return plan_acc_bytes(p, plan_blocks(p, nullptr, nullptr));
}

static int pack_compress_variable(zfpx_plan p, int minexp, int prec, const float *d_src, uint16_t *d_lengths,
                                  uint8_t *d_payload, size_t cap, uint64_t *d_msg_words, void *d_work,
                                  size_t work_bytes, void *stream)
{
    if (!p || !d_src || !d_lengths || !d_payload || !d_msg_words || !d_work || p->dims != 3) return ZFPX_EINVAL;
    if (!aligned(d_payload, 8) || !aligned(d_work, 256) || !aligned(d_lengths, 2) || !aligned(d_msg_words, 8))
        return ZFPX_EINVAL;
    const int64_t G = plan_blocks(p, nullptr, nullptr);
    if (cap < (size_t)G * 128) return ZFPX_ESIZE;
    cudaStream_t st = (cudaStream_t)stream;
    PlanAccWork w;
    int rc = plan_acc_setup(p, d_work, work_bytes, st, &w);
    if (rc) return rc;
    if (G == 0)                                    // every message empty
        return cudaMemsetAsync(d_msg_words, 0, p->msgs.size() * 8, st) == cudaSuccess ? ZFPX_OK : ZFPX_ECUDA;
    LaunchGeom g{};
    if ((rc = plan_geom(p, g))) return rc;
    if ((rc = launch_encode_lengths(d_src, w.slots, g, codec_vec_ok(d_src, p->ss, p) ? 1 : 0,
                                    AccEncode{d_lengths, w.P.msgs, minexp, prec}, st)))
        return rc;
    if ((rc = acc_scan(w.scan, d_lengths, w.scan.total, st))) return rc;
    // the sum of the word counts, where the payload ends, in the scratch after the total
    uint64_t *used = w.scan.total + 1;
    launch_after(pacc_messages_kernel, 1, kTile, 0, st, w.P, w.scan.local, w.scan.tile_off, w.scan.total, d_msg_words, 1, used);
    count_launch();
    if ((rc = check_launch())) return rc;
    return acc_pack(AccList{w.P.msgs, w.P.pay_send, d_lengths, w.scan.local, w.scan.tile_off, w.P.M, G}, w.slots,
                    d_payload, used, 0, st);
}

int zfpx_pack_compress_accuracy(zfpx_plan p, double tolerance, const float *d_src, uint16_t *d_lengths,
                                uint8_t *d_payload, size_t cap, uint64_t *d_msg_words, void *d_work,
                                size_t work_bytes, void *stream)
{
    if (!(tolerance > 0.0) || !(tolerance < HUGE_VAL)) return ZFPX_EINVAL;
    int e = 0;
    (void)frexp(tolerance, &e);
    return pack_compress_variable(p, e - 1, 0, d_src, d_lengths, d_payload, cap, d_msg_words, d_work, work_bytes,
                                  stream);
}

int zfpx_pack_compress_precision(zfpx_plan p, int precision, const float *d_src, uint16_t *d_lengths,
                                 uint8_t *d_payload, size_t cap, uint64_t *d_msg_words, void *d_work,
                                 size_t work_bytes, void *stream)
{
    if (precision < 1 || precision > 32) return ZFPX_EINVAL;
    return pack_compress_variable(p, 0, precision, d_src, d_lengths, d_payload, cap, d_msg_words, d_work,
                                  work_bytes, stream);
}

int zfpx_exchange_accuracy(zfpx_plan p, const uint64_t *d_msg_words, const uint16_t *d_len_send,
                           const uint8_t *d_pay_send, uint16_t *d_len_recv, uint8_t *d_pay_recv, size_t cap,
                           void *d_work, size_t work_bytes, void *stream)
{
    if (!p || !d_msg_words || !d_len_send || !d_pay_send || !d_len_recv || !d_pay_recv || !d_work || p->dims != 3)
        return ZFPX_EINVAL;
    if (!aligned(d_pay_send, 8) || !aligned(d_pay_recv, 8) || !aligned(d_work, 256)) return ZFPX_EINVAL;
    const int64_t G = plan_blocks(p, nullptr, nullptr);
    if (cap < (size_t)G * 128) return ZFPX_ESIZE;
    cudaStream_t st = (cudaStream_t)stream;
    PlanAccWork w;
    int rc = plan_acc_setup(p, d_work, work_bytes, st, &w);
    if (rc || w.P.M == 0) return rc;
    launch_after(pacc_messages_kernel, 1, kTile, 0, st, w.P, nullptr, nullptr, nullptr, const_cast<uint64_t *>(d_msg_words), 0,
                                              nullptr);
    count_launch();
    // about eight CTAs per SM over all messages
    const unsigned parts = (unsigned)std::max<int64_t>(1, std::min<int64_t>(64, (int64_t)num_sms() * 8 / w.P.M));
    launch_after(pacc_exchange_kernel, dim3((unsigned)w.P.M, parts), 256, 0, st, w.P, d_msg_words,
                                                           reinterpret_cast<const uint64_t *>(d_pay_send),
                                                           reinterpret_cast<uint64_t *>(d_pay_recv), d_len_send,
                                                           d_len_recv, (int64_t)(cap / 8));
    count_launch();
    return check_launch();
}

int zfpx_decompress_unpack_accuracy(zfpx_plan p, const uint64_t *d_msg_words, const uint16_t *d_len_recv,
                                    const uint8_t *d_pay_recv, size_t len, float *d_dst, void *d_work,
                                    size_t work_bytes, void *stream)
{
    if (!p || !d_msg_words || !d_len_recv || !d_pay_recv || !d_dst || !d_work || p->dims != 3) return ZFPX_EINVAL;
    if (!aligned(d_pay_recv, 8) || !aligned(d_work, 256) || !aligned(d_len_recv, 2)) return ZFPX_EINVAL;
    const int64_t G = plan_blocks(p, nullptr, nullptr);
    cudaStream_t st = (cudaStream_t)stream;
    PlanAccWork w;
    int rc = plan_acc_setup(p, d_work, work_bytes, st, &w);
    if (rc || G == 0) return rc;
    launch_after(pacc_messages_kernel, 1, kTile, 0, st, w.P, nullptr, nullptr, nullptr, const_cast<uint64_t *>(d_msg_words), 0,
                                              nullptr);
    count_launch();
    if ((rc = acc_scan(w.scan, d_len_recv, w.scan.total, st))) return rc;
    LaunchGeom g{};
    if ((rc = plan_geom(p, g))) return rc;
    return launch_decode_payload(d_dst, g, codec_vec_ok(d_dst, p->ds, p) ? 1 : 0,
                                 AccDecode{reinterpret_cast<const uint64_t *>(d_pay_recv), (int64_t)(len / 8), d_len_recv,
                                           w.scan.local, w.scan.tile_off, w.P.msgs, w.P.pay_recv},
                                 st);
}

}  // extern "C"
