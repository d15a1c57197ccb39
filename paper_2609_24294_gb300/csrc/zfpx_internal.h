// Internal declarations shared by the library's translation units.
#pragma once

#include <cstdint>
#include <cstddef>
#include <vector>
#include <mutex>
#include <map>

#include <cuda_runtime.h>

#include "../../include/zfpx.h"

namespace zfpx {

// One message as the kernels see it.  Element offsets are into the plan's
// src / dst views; byte offsets into the send / receive layouts.
struct MsgDev {
    int64_t src_off;    // element offset of the box origin in the source view
    int64_t dst_off;    // element offset of the box origin in the destination view
    int64_t off[2];     // byte offset in the send [0] and receive [1] layout
    int64_t unit0;      // first work unit (warp chunk or row quad) of this message
    int32_t nx, ny, nz; // box extents
    int32_t bx, by, bz; // block counts (dims 3: ceil(n/4) each; dims 1: ceil(nx/4), ny, nz)
    int64_t nblocks;    // bx * by * bz
    uint32_t bxm, bym;  // divisors of bx and by for divu (set_block_divisors)
    int32_t bxl, byl;
};

// Exact unsigned 32-bit division by an invariant d >= 1 as a high multiply,
// an add and shifts (Granlund and Montgomery, "Division by invariant integers
// using multiplication", 1994): l = ceil(log2 d), m = floor(2^32 (2^l - d) / d)
// + 1, then n / d = (t + ((n - t) >> 1)) >> (l - 1) with t = mulhi(n, m), and
// n itself when d = 1.
inline void block_divisor(uint32_t d, uint32_t &m, int32_t &l)
{
    l = 0;
    while (l < 32 && ((uint64_t)1 << l) < d) l++;
    m = (uint32_t)(((((uint64_t)1 << l) - d) << 32) / d + 1);
}
inline void set_block_divisors(MsgDev &d)
{
    block_divisor((uint32_t)d.bx, d.bxm, d.bxl);
    block_divisor((uint32_t)d.by, d.bym, d.byl);
}
#ifdef __CUDACC__
// Launches that overlap the end of the kernel before them on the stream
// (programmatic dependent launch).  start_next() lets the next kernel's CTAs
// come in as soon as every CTA of this one has started; every thread of a kernel
// launched by launch_after() passes wait_previous() before it touches global
// memory or exits.  wait_previous() returns once the kernel before has completed
// with all its writes visible, so completion stays in stream order through any
// chain of such launches; kernels, copies and events of other origin wait for
// full completion as always.  Used for the chain of short kernels of the
// variable-rate modes, where the gap between two shrinks by 2 to 3 us (fixed
// accuracy 1e-3, 640 x 320 x 137: encode, exchange and decode 308 -> 289 us).  Not
// for the codec and pack kernels: their CTAs that come in early settle unevenly
// over the SMs and take room from work on other streams (one rank's pencil
// 42.6 -> 45.4 us, a captured pair of transpositions 1594 -> 1637 us).
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// The read-only pointers of a kernel pass through the wait: their loads may be
// of the kind that a compiler moves across a memory barrier, not across this.
template <class... T>
__device__ __forceinline__ void wait_previous(const T *__restrict__ &...p)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    ((void)([&] { asm volatile("" : "+l"(p) :: "memory"); }()), ...);
}
template <class... P, class... A>
void launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);   // errors: check_launch()
}

__device__ __forceinline__ uint32_t divu(uint32_t n, uint32_t m, int32_t l)
{
    const uint32_t t = __umulhi(n, m);
    return l ? (t + ((n - t) >> 1)) >> (l - 1) : n;
}
// The last message whose units start at or before u, by the whole warp: every
// round the lanes look at 32 messages spread over the range that is left, so 512
// messages take two rounds of loads where halving takes nine, each waiting for
// the one before at the start of every warp.
__device__ __forceinline__ int find_msg(const MsgDev *msgs, int nmsg, int64_t u)
{
    const int lane = threadIdx.x & 31;
    int lo = 0, n = nmsg;
    while (n > 1) {
        const int step = (n + 31) >> 5;
        const bool before = lane * step < n && msgs[lo + lane * step].unit0 <= u;
        const int k = __popc(__ballot_sync(0xffffffffu, before)) - 1;    // msgs[lo] starts at or before u
        lo += k * step;
        n = min(step, n - k * step);
    }
    return lo;
}
#endif

// Arguments common to every plan-driven launch.
struct LaunchGeom {
    const MsgDev *msgs; // device table (nmsg entries)
    int nmsg;
    int64_t nunits;     // total work units
    int64_t ss[3];      // source strides (elements)
    int64_t ds[3];      // destination strides (elements)
    int32_t upw;        // 3-D codec kernels: consecutive work units per warp (grid = units / (upw * warps))
};

struct HostMsg {
    int32_t src, dst, src_peer, dst_peer;
    int64_t x0, nx, y0, ny, z0, nz;
};

// Device tables of one (rate, unit kind, device) for a plan.
struct DevTable {
    MsgDev *d_msgs = nullptr;   // the message table
    int64_t nunits = 0;
};

}  // namespace zfpx

struct zfpx_plan_s {
    int64_t n[3];
    int64_t ss[3], ds[3];
    int pr, pc, P, transposition, dims, split_mode;
    std::vector<zfpx::HostMsg> msgs;              // send order
    std::mutex mu;
    std::map<long long, zfpx::DevTable> tables;   // key: (device, rate, unit kind)
};

namespace zfpx {

// Work-unit kinds: codec kernels take 32 blocks (one warp) per unit; packs
// take 4-value quads of one row per unit; the permutation 16 stream bytes.
enum UnitKind { UNIT_BLOCKS32 = 0, UNIT_QUADS = 1, UNIT_CHUNK16 = 2 };

int64_t message_bytes(const zfpx_plan_s *p, const HostMsg &m, int rate);
// Offsets of every message (send-order index) in the given layout; the total in *total.
std::vector<int64_t> layout_offsets(const zfpx_plan_s *p, int rate, int layout, int64_t *total);
int64_t buffer_bytes(const zfpx_plan_s *p, int rate);
// Fetches (building on first use) the device table; returns ZFPX_OK or an error.
int get_table(zfpx_plan_s *p, int rate, UnitKind kind, DevTable **out);
// Host copy of the table of the messages `subset` (send-order indices; empty
// = every message), work units numbered from 0 within it; returns the units.
// Offsets stay those of the whole plan's layouts.
int64_t host_table(const zfpx_plan_s *p, int rate, UnitKind kind, const std::vector<int> &subset,
                   std::vector<MsgDev> &h);
// Uploads a host table into a new device allocation (t->d_msgs, freed by the owner).
int upload_table(const std::vector<MsgDev> &h, int64_t units, DevTable *t);

// One message of a plan in the variable-rate modes (send-order index).
struct AccMsg {
    int64_t gb0;        // first block in the send-order block list (and lengths array)
    int64_t gr0;        // first block in the receive-order block list
    int64_t nb;         // blocks
    int64_t slot_send;  // byte offset of its rate-16 slots in the send layout
};
// Where the variable-rate kernels find a table's messages; a NULL array stands
// for one message that starts at 0.
struct AccEncode {
    uint16_t *lengths;        // bits per block, send order
    const AccMsg *msgs;
    int minexp, prec;         // the plane cut (prec > 0: precision mode)
};
struct AccDecode {
    const uint64_t *payload;  // 64-bit words
    int64_t pwords;
    const uint16_t *lengths;  // receive order
    const uint32_t *local;    // exclusive scan of the lengths: tile_off[g / kAccTile] + local[g]
    const uint64_t *tile_off;
    const AccMsg *msgs;
    const int64_t *pay;       // first payload word of each message (send-order index)
};
constexpr int kAccTile = 1024;               // blocks per scan tile

// The rate-16 3-D codec of the variable-rate modes over a table: encode into
// 128-byte slots with every block's bit count, decode straight from the payload.
int launch_encode_lengths(const float *src, uint8_t *slots, const LaunchGeom &g, int vec, const AccEncode &a,
                          cudaStream_t st);
int launch_decode_payload(float *dst, const LaunchGeom &g, int vec, const AccDecode &a, cudaStream_t st);
// The one-message plan of a raw array (cached by shape).
int raw_plan(int dims, const int64_t n[3], const int64_t s[3], zfpx_plan *out);

// Kernel launchers over a table (geometry g: table, units, view strides).
// vec: every row the kernel touches starts on 16 bytes.
int launch_encode(int dims, int rate, const float *src, uint8_t *out, const LaunchGeom &g, int layout, int vec,
                  cudaStream_t st);
int launch_decode(int dims, int rate, const uint8_t *in, float *dst, const LaunchGeom &g, int layout, int vec,
                  cudaStream_t st);
int launch_permute(const uint8_t *send, uint8_t *recv, const LaunchGeom &g, int rate, int dims, cudaStream_t st);
// vec test of the codec kernels for a pointer and view strides over the plan's messages.
bool codec_vec_ok(const void *ptr, const int64_t s[3], const zfpx_plan_s *p);

int num_sms();
// Resident CTAs per SM of `fn` at `threads` threads (cached per kernel).
int occupancy(const void *fn, int threads);
// For a launch of `fn` with `smem` bytes of dynamic shared memory: lifts the
// kernel's limit on them to what the device offers beside its static ones, once per
// device.  The limit is the kernel's, not the call's, so one set to each call's own
// size could be lowered by another thread between a call's set and its launch.
// ZFPX_ECUDA if smem is more than the device offers.
int allow_smem(const void *fn, size_t smem);
void count_launch();
void uncount_launches(uint64_t n);   // launches recorded into a graph, not run
bool valid_codec_rate(int rate);
int check_launch();   // cudaGetLastError -> ZFPX_OK / ZFPX_ECUDA
// Work units per warp of the 3-D codec kernels set for (direction, rate); 0 = the
// library's choice by the launch's size.  Set through zfpx_set_units_per_warp.
int units_per_warp(int encode, int rate);

}  // namespace zfpx
