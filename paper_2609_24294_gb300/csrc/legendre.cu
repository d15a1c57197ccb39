// The Legendre transform: the latitude half of the spectral transform, run on
// theta-pencils after the second transposition (Sec. II-A: associated
// Legendre functions on Gauss-Legendre latitudes; Sec. II-B: the lambda ->
// theta all-to-all makes every latitude column local).  For the wavenumber
// fields F_m(mu_j) (real and imaginary parts, [lev][lat][m]) it returns
//     a_l^m = sum_j w_j Pbar_l^m(mu_j) F_m(mu_j),   0 <= m <= l <= T,
// with Pbar normalised to int Pbar^2 dmu = 1 (Condon-Shortley phase), mu_j the
// Gauss-Legendre nodes north to south and w_j their weights.
//
// Pbar_l^m(-mu) = (-1)^(l+m) Pbar_l^m(mu) and the nodes and weights are
// symmetric, so with S_j = F(mu_j) + F(-mu_j) and A_j = F(mu_j) - F(-mu_j)
// over the northern half (j < nlat/2)
//     a_l^m = sum_{j < nlat/2} w_j Pbar_l^m(mu_j) (l + m even ? S_j : A_j),
// half the work of the full sum.  For each order m and parity p of l + m this
// is a product (rows l of that parity) x (nlat/2) times (nlat/2) x (2 nlev)
// (columns: the real parts of all levels, then the imaginary parts).
//
// The plan holds the table w_j Pbar_l^m(mu_j), j < nlat/2, built on the host
// in double precision (Newton iteration for the nodes, the three-term
// recurrences for Pbar) and rounded once to float; values below the double
// range near the poles for large m are 0.  Both operands are stored K-major
// (the latitude index j contiguous): the table as rows l of each (m, p)
// block, and the folded operand, which a fold kernel writes per call into the
// caller's workspace, as rows (m, p, column).
//
// The products run on the tensor cores (tcgen05.mma, kind::tf32) with float32
// accuracy from a three-term split: a = a_hi + a_lo with a_hi = a truncated
// to TF32 (what the MMA reads of a float32 operand) and a_lo = a - a_hi rounded
// to TF32, and a b = a_hi b_hi + a_hi b_lo + a_lo b_hi, accumulated in float32
// in tensor memory; the dropped a_lo b_lo and the TF32 rounding of the lo
// parts leave about 2^-21 of sum |a b| per product, far below the float32
// dot-product bound the transform is held to.  One CTA per SM walks 128-row x
// Nt-column tiles of the (m, p) blocks (legendre_mma_kernel below); each warp
// role waits only on mbarriers, every wait is bounded, and a wait that runs
// out sets the plan's status word and the CTA stops.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <new>
#include <vector>
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include "zfpx_internal.h"

struct LegItem {
    int32_t m, p, r0, nr;   // order, parity of l + m, first row (of that parity), rows in this tile
    int64_t arow;           // first table row of this (m, p) block (rows of the K-major table tensor)
};

struct zfpx_legendre_s {
    int nlat = 0, T = 0, nh = 0, nhs = 0, device = 0;
    int64_t table_rows = 0;
    float *d_table = nullptr;   // K-major: [table_rows][nhs] floats, columns >= nh zero
    LegItem *d_items = nullptr;
    int *d_status = nullptr;    // 0, or the code of a wait that ran out
    int nitems = 0;
    CUtensorMap tmap_table;     // TMA view of the table: {nh, table_rows}, boxes {32, 128}
};

namespace zfpx {
namespace {

constexpr int kBM = 128;        // rows per CTA tile (the MMA's M)
constexpr int kBK = 32;         // K per stage: one 128-byte swizzle row of float32
constexpr long long kSpinLimit = 1ll << 26;   // about a second of polling

struct LegGeom {
    int nlat, nh, nhs, T, nlev;
    int N;                   // columns: 2 nlev
    int nt, ntiles;          // columns per tile (a multiple of 16, <= 256), tiles
    int ncp;                 // column rows per (m, p) in the workspace: ntiles * nt
    int64_t is1, is2;        // input strides: latitude, level (floats; wavenumber stride 1)
    int64_t os;              // output level stride (floats)
};

__host__ __device__ __forceinline__ int64_t tri_offset(int m, int T)
{
    return (int64_t)m * (T + 1) - (int64_t)m * (m - 1) / 2;
}

// G[((m * 2 + p) * ncp + c) * nhs + j], c = part * nlev + lev: S (p = 0) and A
// (p = 1) of part `part` of F at level lev, latitude pair (j, nlat - 1 - j),
// order m; columns j in [nh, nhs) are written as zeros.  Block (32, 8) over 32
// orders x 32 latitudes of one (level, part).
__global__ void __launch_bounds__(256) legendre_fold_kernel(const float *__restrict__ re, const float *__restrict__ im,
                                                            float *__restrict__ G, LegGeom g)
{
    __shared__ float sS[32][33], sA[32][33];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int m0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
    const int lev = blockIdx.z >> 1, part = blockIdx.z & 1;
    const float *F = (part ? im : re) + lev * g.is2;
    for (int i = ty; i < 32; i += 8) {
        const int j = j0 + i, m = m0 + tx;
        float a = 0.f, b = 0.f;
        if (j < g.nh && m <= g.T) {
            a = __ldg(F + (int64_t)j * g.is1 + m);
            b = __ldg(F + (int64_t)(g.nlat - 1 - j) * g.is1 + m);
        }
        sS[i][tx] = a + b;                            // [j][m]
        sA[i][tx] = a - b;
    }
    __syncthreads();
    const int c = part * g.nlev + lev;
    for (int i = ty; i < 32; i += 8) {
        const int m = m0 + i, j = j0 + tx;
        if (m <= g.T && j < g.nhs) {
            const int64_t row = ((int64_t)m * 2 * g.ncp + c) * g.nhs + j;
            G[row] = sS[tx][i];
            G[row + (int64_t)g.ncp * g.nhs] = sA[tx][i];
        }
    }
}

// The same fold for fields whose rows start on 16 bytes (latitude and level
// strides multiples of 4, 16-byte aligned bases): tiles of 128 orders x 32
// latitudes, every load and store a 16-byte vector (four orders in, four
// latitudes out).  Block (32, 8).
__global__ void __launch_bounds__(256) legendre_fold4_kernel(const float *__restrict__ re,
                                                             const float *__restrict__ im, float *__restrict__ G,
                                                             LegGeom g)
{
    __shared__ float sS[32][129], sA[32][129];          // [latitude][order]
    const int tx = threadIdx.x, ty = threadIdx.y, t = ty * 32 + tx;
    const int m0 = blockIdx.x * 128, j0 = blockIdx.y * 32;
    const int lev = blockIdx.z >> 1, part = blockIdx.z & 1;
    const float *F = (part ? im : re) + lev * g.is2;
    const int m = m0 + 4 * tx;
    for (int i = ty; i < 32; i += 8) {
        const int j = j0 + i;
        float a[4] = {0.f, 0.f, 0.f, 0.f}, b[4] = {0.f, 0.f, 0.f, 0.f};
        if (j < g.nh) {
            const float *rn = F + (int64_t)j * g.is1, *rs = F + (int64_t)(g.nlat - 1 - j) * g.is1;
            if (m + 3 <= g.T) {
                const float4 u = __ldg(reinterpret_cast<const float4 *>(rn + m));
                const float4 v = __ldg(reinterpret_cast<const float4 *>(rs + m));
                a[0] = u.x; a[1] = u.y; a[2] = u.z; a[3] = u.w;
                b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
            } else {
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (m + q <= g.T) {
                        a[q] = __ldg(rn + m + q);
                        b[q] = __ldg(rs + m + q);
                    }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; q++) {
            sS[i][4 * tx + q] = a[q] + b[q];
            sA[i][4 * tx + q] = a[q] - b[q];
        }
    }
    __syncthreads();
    const int c = part * g.nlev + lev;
    const int jj = 4 * (t & 7), j = j0 + jj;              // latitudes j .. j + 3 (nhs is a multiple of 4)
    if (j >= g.nhs) return;
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const int k = (t >> 3) + 32 * r, mm = m0 + k;
        if (mm > g.T) break;
        const int64_t row = ((int64_t)mm * 2 * g.ncp + c) * g.nhs + j;
        *reinterpret_cast<float4 *>(G + row) = make_float4(sS[jj][k], sS[jj + 1][k], sS[jj + 2][k], sS[jj + 3][k]);
        *reinterpret_cast<float4 *>(G + row + (int64_t)g.ncp * g.nhs) =
            make_float4(sA[jj][k], sA[jj + 1][k], sA[jj + 2][k], sA[jj + 3][k]);
    }
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// tcgen05 shared-memory descriptor of a K-major, 128-byte-swizzled operand
// tile starting at `saddr` (8-row groups 1024 bytes apart)
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);           // start address / 16
    d |= (uint64_t)1u << 16;                             // leading byte offset (not used by swizzled K-major)
    d |= (uint64_t)(1024u >> 4) << 32;                   // stride byte offset / 16
    d |= (uint64_t)1u << 46;                             // descriptor version
    d |= (uint64_t)2u << 61;                             // 128-byte swizzle
    return d;
}

__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity)
{
    for (long long i = 0; i < kSpinLimit; i++) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t mbar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(dst), "l"(map), "r"(x), "r"(y), "r"(mbar) : "memory");
}

__device__ __forceinline__ void mbar_expect(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(mbar), "r"(bytes) : "memory");
}

// The 3 x TF32 split of a float32 a: hi = a with its 13 low mantissa bits
// cleared (what the tensor core reads of a), lo = a - hi (exact) rounded to
// TF32, to nearest with ties away from zero, by adding half of the last kept
// bit to the magnitude bits and clearing the rest (the rounding of PTX's
// cvt.rna.tf32.f32, as integer operations).
__device__ __forceinline__ float tf32_lo(float a)
{
    const float l = a - __uint_as_float(__float_as_uint(a) & 0xffffe000u);
    return __uint_as_float((__float_as_uint(l) + 0x1000u) & 0xffffe000u);
}

// lo = tf32_lo(a) over n <= 8 nthr 16-byte chunks, by the nthr threads numbered
// t: every load ahead of the first store
__device__ __forceinline__ void split_lo(const uint8_t *raw, uint8_t *lo, int n, int t, int nthr)
{
    float4 a[8];
#pragma unroll
    for (int r = 0; r < 8; r++)
        if (t + r * nthr < n) a[r] = reinterpret_cast<const float4 *>(raw)[t + r * nthr];
#pragma unroll
    for (int r = 0; r < 8; r++)
        if (t + r * nthr < n)
            reinterpret_cast<float4 *>(lo)[t + r * nthr] =
                make_float4(tf32_lo(a[r].x), tf32_lo(a[r].y), tf32_lo(a[r].z), tf32_lo(a[r].w));
}

// Persistent and warp-specialised: one CTA per SM walks the tiles t =
// blockIdx.x, blockIdx.x + gridDim.x, ... (a tile: 128 rows x nt columns of one
// (m, p) block).  Roles:
//   warp 0 (one lane)  TMA producer: the K slices (32 deep) of every tile in
//                      turn, up to `stages` ahead, a stage refilled once the
//                      MMAs that read it have completed (mma_bar); of the table
//                      only the 32-row boxes that hold rows of the tile;
//   warp 1 (one lane)  waits for a slice's operands (lo_bar), issues its twelve
//                      MMAs into the tile's accumulator and commits them to
//                      the stage, and after a tile's last slice to acc_full;
//   warps 4-7          bring the table slice from shared to tensor memory, a
//                      thread per row: its 32 values and their low parts;
//   warps 2, 3, 8-11   derive the data slice's low parts in shared memory;
//   warps 12-15        epilogue: once a tile's accumulator is complete, each
//                      reads the 32 rows of its TMEM lane quadrant, scatters
//                      them into the triangular output and frees the
//                      accumulator (acc_empty).
// Tensor memory: two accumulators that alternate between tiles, so that a
// tile's epilogue overlaps the next tile's MMAs, and two or three table slots.
// Dynamic shared memory: `stages` x {table, data, data lo}, 1024-aligned.
// What bounds it: reads from L2 (the loads alone take 173 us of the 273 at T639 on
// 137 levels), then shared-memory traffic.  Measured there and at T319 on 91 levels,
// us without the fold:
//   low parts of both operands in shared memory, the table's read from a table
//   of their own, one barrier over eleven warps per slice       350, 83
//   a role per step, joined by mbarriers alone                  302, 84
//   table through tensor memory, its low parts derived          328, 80
//   the output's addresses kept instead of computed per store   280, 48
//   only the table boxes with rows                              273, 48
// Neither more split or epilogue warps (292) nor five stages with two low-part
// buffers (283) is faster, nor tiles of both parities with 8-byte stores (96
// columns so that four accumulators fit: 408).
constexpr int kMaxStages = 4;
constexpr int kTableWarps = 4, kDataWarps = 6;  // warps 4-7; warps 2, 3, 8-11
constexpr int kMmaThreads = 512;                // 16 warps
constexpr int kBoxRows = 32;                    // rows per TMA copy of the table
constexpr int kTmemCols = 512;                  // all of the SM's tensor memory
constexpr int kMaxTile = 192;                   // columns per tile: two accumulators and two table slots fit

// A bounded wait that also gives up once another role has failed.
__device__ __forceinline__ bool role_wait(uint32_t mbar, uint32_t parity, volatile int *fail)
{
    for (long long i = 0; i < kSpinLimit; i++) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
        if (ok) return true;
        if ((i & 1023) == 1023 && *fail) return false;
    }
    return false;
}

// How often stage s of `stages` has been used once `n` slices have gone through
// them in turn: its barrier's last phase is the one before that.
__host__ __device__ constexpr int stage_uses(int n, int s, int stages) { return (n - s + stages - 1) / stages; }
static_assert(stage_uses(0, 0, 4) == 0 && stage_uses(0, 3, 4) == 0 && stage_uses(1, 0, 4) == 1 && stage_uses(1, 1, 4) == 0 &&
              stage_uses(4, 3, 4) == 1 && stage_uses(5, 0, 4) == 2 && stage_uses(5, 1, 4) == 1 && stage_uses(7, 2, 2 + 1) == 2,
              "uses of a stage");

// 32 columns of this warp's 32 tensor-memory lanes
__device__ __forceinline__ void tmem_store32(uint32_t addr, const uint32_t (&v)[32])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
                 :: "r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
                 : "memory");
}

__device__ __forceinline__ void tmem_load16(uint32_t addr, uint32_t (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(addr));
}

__global__ void __launch_bounds__(kMmaThreads, 1)
legendre_mma_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                    const LegItem *__restrict__ items, LegGeom g, int stages, int ntiles_total,
                    float *__restrict__ are, float *__restrict__ aim, int *__restrict__ status)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kMaxStages], lo_bar[kMaxStages], mma_bar[kMaxStages], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base;
    __shared__ int fail;
    __shared__ int issued[2];                            // slices loaded, slices whose MMAs were committed
    volatile int *vfail = &fail;
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int nt = g.nt;
    const uint32_t a_bytes = kBM * 128, b_bytes = (uint32_t)nt * 128;
    const uint32_t stage_bytes = a_bytes + 2 * b_bytes;
    auto a_raw = [&](int s) { return smem + s * stage_bytes; };
    auto b_raw = [&](int s) { return smem + s * stage_bytes + a_bytes; };
    auto b_lo = [&](int s) { return smem + s * stage_bytes + a_bytes + b_bytes; };
    // tensor memory: two accumulators, then the table slots (32 columns of high,
    // 32 of low parts: one slice each)
    const int acc_cols = (nt + 31) / 32 * 32;
    const int slots = min(stages, (kTmemCols - 2 * acc_cols) / (2 * kBK));

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&tmem_base)), "n"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        fail = 0;
        for (int s = 0; s < stages; s++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&full_bar[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&mma_bar[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(&lo_bar[s])), "n"(kTableWarps + kDataWarps));
        }
        for (int a = 0; a < 2; a++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&acc_full[a])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" :: "r"(smem_u32(&acc_empty[a])));
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" :: "l"(&tmap_a) : "memory");
        asm volatile("prefetch.tensormap [%0];" :: "l"(&tmap_b) : "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    const int nk = (g.nh + kBK - 1) / kBK;

    if (warp == 0) {
        // ---- producer
        if (tid == 0) {
            int i = 0;                                   // slice count over all tiles of this CTA
            for (int t = blockIdx.x; t < ntiles_total && !*vfail; t += gridDim.x) {
                const LegItem it = items[t / g.ntiles];
                const int ct = t % g.ntiles;
                const int arow = (int)(it.arow + it.r0), abox = (it.nr + kBoxRows - 1) / kBoxRows;
                const int brow = (int)(((int64_t)it.m * 2 + it.p) * g.ncp + (int64_t)ct * nt);
                for (int k = 0; k < nk; k++, i++) {
                    const int s = i % stages;
                    if (i >= stages && !role_wait(smem_u32(&mma_bar[s]), (uint32_t)(i / stages - 1) & 1u, vfail)) {
                        *vfail = 1;
                        break;
                    }
                    const uint32_t fb = smem_u32(&full_bar[s]);
                    mbar_expect(fb, abox * kBoxRows * 128 + b_bytes);
                    for (int b = 0; b < abox; b++)
                        tma_load_2d(smem_u32(a_raw(s) + b * kBoxRows * 128), &tmap_a, k * kBK, arow + b * kBoxRows, fb);
                    tma_load_2d(smem_u32(b_raw(s)), &tmap_b, k * kBK, brow, fb);
                }
            }
            issued[0] = i;
        }
    } else if (warp == 1) {
        // ---- MMAs
        if (tid == 32) {
            const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(nt >> 3) << 17) |
                                   ((uint32_t)(kBM >> 4) << 24);
            int i = 0, j = 0;                            // slices, tiles of this CTA
            for (int t = blockIdx.x; t < ntiles_total && !*vfail; t += gridDim.x, j++) {
                const int acc = j & 1;
                const uint32_t d = tmem + (uint32_t)(acc * acc_cols);
                // the accumulator's previous tile must have been read out
                if (j >= 2 && !role_wait(smem_u32(&acc_empty[acc]), (uint32_t)(j / 2 - 1) & 1u, vfail)) {
                    *vfail = 1;
                    break;
                }
                for (int k = 0; k < nk; k++, i++) {
                    const int s = i % stages;
                    if (!role_wait(smem_u32(&lo_bar[s]), (uint32_t)(i / stages) & 1u, vfail)) {
                        *vfail = 1;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t ah = tmem + (uint32_t)(2 * acc_cols + i % slots * (2 * kBK)), al = ah + kBK;
                    const uint32_t bh = smem_u32(b_raw(s)), bl = smem_u32(b_lo(s));
#pragma unroll
                    for (int q = 0; q < kBK / 8; q++) {     // 8-deep K steps, 32 bytes apart in the swizzle row
                        const uint64_t dbh = sw128_desc(bh + 32 * q), dbl = sw128_desc(bl + 32 * q);
#pragma unroll
                        for (int e = 0; e < 3; e++) {
                            const uint32_t a = (e == 2 ? al : ah) + 8 * q;
                            const uint64_t db = e == 1 ? dbl : dbh;
                            const uint32_t accum = (k > 0 || q > 0 || e > 0) ? 1u : 0u;
                            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                         "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}"
                                         :: "r"(d), "r"(a), "l"(db), "r"(idesc), "r"(accum));
                        }
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                                 :: "r"(smem_u32(&mma_bar[s])) : "memory");
                    if (k == nk - 1)
                        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                                     :: "r"(smem_u32(&acc_full[acc])) : "memory");
                }
            }
            issued[1] = i;
        }
    } else if (warp >= 4 && warp <= 7) {
        // ---- table slices to tensor memory: a thread per row, its 32 values and
        // their low parts; warp 4 + q reaches the lanes (rows) 32 q .. 32 q + 31
        const int row = 32 * (warp - 4) + (tid & 31);
        const uint32_t lanes = (uint32_t)(32 * (warp - 4)) << 16;
        int i = 0;
        bool stop = false;
        for (int t = blockIdx.x; t < ntiles_total && !stop; t += gridDim.x)
            for (int k = 0, live = 32 * (warp - 4) < items[t / g.ntiles].nr; k < nk; k++, i++) {
                const int s = i % stages, f = i - slots;     // f: the slice whose slot this one takes
                bool got = role_wait(smem_u32(&full_bar[s]), (uint32_t)(i / stages) & 1u, vfail);
                if (got && f >= 0)
                    got = role_wait(smem_u32(&mma_bar[f % stages]), (uint32_t)(f / stages) & 1u, vfail);
                if (!__all_sync(0xffffffffu, got)) { *vfail = 1; stop = true; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (live) {
                    const uint8_t *a = a_raw(s) + row * 128;
                    uint32_t v[kBK];
#pragma unroll
                    for (int ch = 0; ch < 8; ch++) {             // 16-byte chunk ch of a swizzled row
                        const uint4 x = *reinterpret_cast<const uint4 *>(a + 16 * (ch ^ (row & 7)));
                        v[4 * ch] = x.x; v[4 * ch + 1] = x.y; v[4 * ch + 2] = x.z; v[4 * ch + 3] = x.w;
                    }
                    const uint32_t slot = tmem + lanes + (uint32_t)(2 * acc_cols + i % slots * (2 * kBK));
                    tmem_store32(slot, v);
#pragma unroll
                    for (int e = 0; e < kBK; e++) v[e] = __float_as_uint(tf32_lo(__uint_as_float(v[e])));
                    tmem_store32(slot + kBK, v);
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if ((tid & 31) == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&lo_bar[s])) : "memory");
            }
    } else if (warp <= 11) {
        // ---- low parts of the data
        const int c = tid - (warp < 4 ? 64 : 192);
        int i = 0;
        bool stop = false;
        for (int t = blockIdx.x; t < ntiles_total && !stop; t += gridDim.x)
            for (int k = 0; k < nk; k++, i++) {
                const int s = i % stages;
                const bool got = role_wait(smem_u32(&full_bar[s]), (uint32_t)(i / stages) & 1u, vfail);
                if (!__all_sync(0xffffffffu, got)) { *vfail = 1; stop = true; break; }
                split_lo(b_raw(s), b_lo(s), (int)(b_bytes / 16), c, 32 * kDataWarps);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if ((tid & 31) == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&lo_bar[s])) : "memory");
            }
    } else {
        // ---- epilogue: warp 12 + q reads TMEM lanes 32 q .. 32 q + 31 (its warp
        // index mod 4 is q, the lane quadrant tcgen05.ld lets it reach)
        const int q = warp - 12, lane = tid & 31;
        int j = 0;
        for (int t = blockIdx.x; t < ntiles_total; t += gridDim.x, j++) {
            const int acc = j & 1;
            const bool got = role_wait(smem_u32(&acc_full[acc]), (uint32_t)(j / 2) & 1u, vfail);
            if (!__all_sync(0xffffffffu, got)) { *vfail = 1; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const LegItem it = items[t / g.ntiles];
            const int ct = t % g.ntiles;
            const int row = 32 * q + lane;
            const bool live = row < it.nr;
            // the row's output column c is at base[part] + c os, part 1 from column nlev on
            const int64_t o = tri_offset(it.m, g.T) + it.p + 2 * (int64_t)(it.r0 + row);
            float *const base0 = are + o, *const base1 = aim + o - g.nlev * g.os;
            const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * acc_cols);
            for (int c0 = 0; c0 < nt; c0 += 16) {
                uint32_t v[16];
                tmem_load16(taddr + c0, v);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                const int c = ct * nt + c0;
                int64_t off = (int64_t)c * g.os;
                if (live) {
#pragma unroll
                    for (int e = 0; e < 16; e++, off += g.os)
                        if (c + e < g.N) (c + e < g.nlev ? base0 : base1)[off] = __uint_as_float(v[e]);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&acc_empty[acc])) : "memory");
        }
    }
    __syncthreads();
    if (*vfail && tid == 0) {
        atomicExch(status, 1);
        // let copies and MMAs still in flight land before the CTA leaves: the last
        // phase that each stage's barriers have been given
        for (int s = 0; s < stages; s++) {
            const int loads = stage_uses(issued[0], s, stages), mmas = stage_uses(issued[1], s, stages);
            if (loads) mbar_wait(smem_u32(&full_bar[s]), (uint32_t)(loads - 1) & 1u);
            if (mmas) mbar_wait(smem_u32(&mma_bar[s]), (uint32_t)(mmas - 1) & 1u);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "n"(kTmemCols));
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, []() {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// TMA view of a K-major float32 matrix: `rows` rows of `k` values (`ld`
// floats apart, ld * 4 a multiple of 16), read as {32 x box_rows} boxes with
// 128-byte swizzle; values past k or rows read as zero.
int make_tmap(CUtensorMap *map, const float *base, int64_t k, int64_t rows, int64_t ld, int box_rows)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn) return ZFPX_ECUDA;
    const cuuint64_t dims[2] = {(cuuint64_t)k, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? ZFPX_OK : ZFPX_ECUDA;
}

// the workspace's columns per (m, p) for N = 2 nlev columns, as nt * ntiles
void column_tiles(int N, int &nt, int &ntiles)
{
    ntiles = (N + 255) / 256;
    nt = ((N + ntiles - 1) / ntiles + 15) / 16 * 16;
}

size_t stage_bytes(int nt) { return kBM * 128 + 2 * (size_t)nt * 128; }

// as many stages (2 .. 4) as fit beside one CTA's static shared memory
int mma_stages(int nt)
{
    const size_t budget = 220 * 1024 - 1024;
    return (int)std::max<size_t>(2, std::min<size_t>(kMaxStages, budget / stage_bytes(nt)));
}

size_t mma_smem_bytes(int nt) { return 1024 + (size_t)mma_stages(nt) * stage_bytes(nt); }

// Gauss-Legendre nodes (north to south) and weights: Newton's iteration on
// P_n from the initial guesses cos(pi (i + 3/4) / (n + 1/2)), the upper half
// mirrored.
void gauss_legendre(int n, std::vector<double> &mu, std::vector<double> &w)
{
    const double pi = 3.14159265358979323846264338327950288;
    mu.assign(n, 0.0);
    w.assign(n, 0.0);
    for (int i = 0; i < (n + 1) / 2; i++) {
        double x = std::cos(pi * (i + 0.75) / (n + 0.5)), dp = 1.0;
        for (int it = 0; it < 100; it++) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= n; k++) {
                const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            if (n == 1) { p1 = x; p0 = 1.0; }
            dp = n * (x * p1 - p0) / -((1.0 - x) * (1.0 + x));
            const double dx = p1 / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-16) break;
        }
        // recompute the derivative at the converged node for the weight
        double p0 = 1.0, p1 = x;
        for (int k = 2; k <= n; k++) {
            const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        if (n == 1) { p1 = x; p0 = 1.0; }
        dp = n * (x * p1 - p0) / -((1.0 - x) * (1.0 + x));
        mu[i] = x;
        mu[n - 1 - i] = -x;
        w[i] = w[n - 1 - i] = 2.0 / ((1.0 - x) * (1.0 + x) * dp * dp);   // 1 - x^2 without cancellation
    }
}

}  // namespace
}  // namespace zfpx

using namespace zfpx;

namespace {

int legendre_create(zfpx_legendre *out, int nlat, int T)
{
    std::unique_ptr<zfpx_legendre_s> hold(new zfpx_legendre_s());
    zfpx_legendre_s *p = hold.get();
    p->nlat = nlat; p->T = T; p->nh = nlat / 2;
    p->nhs = (p->nh + 3) / 4 * 4;                        // row pitch: a multiple of 16 bytes
    if (cudaGetDevice(&p->device) != cudaSuccess) return ZFPX_ECUDA;
    const int nh = p->nh, nhs = p->nhs;
    // rows: for m = 0..T, parity 0 then 1, one row per l = m + p + 2 i, K-major
    int64_t rows = 0;
    for (int m = 0; m <= T; m++)
        for (int par = 0; par < 2; par++) rows += (T - m - par) >= 0 ? (T - m - par) / 2 + 1 : 0;
    p->table_rows = rows;
    // a table of more than half the device's memory is refused
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return ZFPX_ECUDA;
    if ((double)std::max<int64_t>(rows, 1) * nhs * 2 * sizeof(float) > (double)total_b) return ZFPX_ENOMEM;
    std::vector<double> mu, w;
    gauss_legendre(nlat, mu, w);
    std::vector<double> s(nh);
    for (int j = 0; j < nh; j++) s[j] = std::sqrt(std::max(0.0, 1.0 - mu[j] * mu[j]));
    std::vector<float> tab((size_t)std::max<int64_t>(rows, 1) * nhs, 0.0f);
    std::vector<LegItem> items;
    std::vector<double> pmm(nh, std::sqrt(0.5));
    std::vector<std::vector<double>> prow;
    int64_t r = 0;
    for (int m = 0; m <= T; m++) {
        if (m > 0) {
            const double f = -std::sqrt((2.0 * m + 1.0) / (2.0 * m));
            for (int j = 0; j < nh; j++) pmm[j] *= f * s[j];
        }
        const int L = T - m + 1;
        prow.assign(L, std::vector<double>(nh));
        prow[0] = pmm;
        if (L > 1)
            for (int j = 0; j < nh; j++) prow[1][j] = std::sqrt(2.0 * m + 3.0) * mu[j] * pmm[j];
        for (int i = 2; i < L; i++) {
            const double l = m + i;
            const double a = std::sqrt((4.0 * l * l - 1.0) / (l * l - (double)m * m));
            const double b = std::sqrt(((l - 1.0) * (l - 1.0) - (double)m * m) / (4.0 * (l - 1.0) * (l - 1.0) - 1.0));
            for (int j = 0; j < nh; j++) prow[i][j] = a * (mu[j] * prow[i - 1][j] - b * prow[i - 2][j]);
        }
        for (int par = 0; par < 2; par++) {
            const int cnt = par < L ? (L - 1 - par) / 2 + 1 : 0;
            for (int c = 0; c < cnt; c++)
                for (int j = 0; j < nh; j++) tab[(size_t)(r + c) * nhs + j] = (float)(w[j] * prow[par + 2 * c][j]);
            for (int r0 = 0; r0 < cnt; r0 += kBM)
                items.push_back(LegItem{m, par, r0, std::min(kBM, cnt - r0), r});
            r += cnt;
        }
    }
    p->nitems = (int)items.size();
    if (cudaMalloc(&p->d_table, tab.size() * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&p->d_items, std::max<size_t>(items.size(), 1) * sizeof(LegItem)) != cudaSuccess ||
        cudaMalloc(&p->d_status, sizeof(int)) != cudaSuccess ||
        cudaMemcpy(p->d_table, tab.data(), tab.size() * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(p->d_items, items.data(), items.size() * sizeof(LegItem), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess ||
        make_tmap(&p->tmap_table, p->d_table, nh, std::max<int64_t>(rows, 1), nhs, kBoxRows) != ZFPX_OK) {
        cudaFree(p->d_table);
        cudaFree(p->d_items);
        cudaFree(p->d_status);
        return ZFPX_ECUDA;
    }
    *out = hold.release();
    return ZFPX_OK;
}

}  // namespace

extern "C" {

int zfpx_legendre_create(zfpx_legendre *out, int nlat, int T)
{
    if (!out) return ZFPX_EINVAL;
    *out = nullptr;
    if (nlat < 2 || nlat % 2 || nlat > 1 << 15 || T < 0 || T + 1 > nlat) return ZFPX_EINVAL;   // grid z = nlat
    // the host tables are built before any device memory is taken: a failed
    // host allocation leaves nothing behind
    try {
        return legendre_create(out, nlat, T);
    } catch (const std::bad_alloc &) {
        return ZFPX_ENOMEM;
    }
}

int zfpx_gauss_legendre(int n, double *mu, double *w)
{
    if (n < 1 || n > (1 << 15) || !mu || !w) return ZFPX_EINVAL;
    std::vector<double> m, ww;
    gauss_legendre(n, m, ww);
    for (int i = 0; i < n; i++) { mu[i] = m[i]; w[i] = ww[i]; }
    return ZFPX_OK;
}

void zfpx_legendre_destroy(zfpx_legendre p)
{
    if (!p) return;
    cudaFree(p->d_table);
    cudaFree(p->d_items);
    cudaFree(p->d_status);
    delete p;
}

size_t zfpx_legendre_workspace_bytes(zfpx_legendre p, int64_t nlev)
{
    if (!p || nlev < 1 || nlev > (1 << 20)) return 0;
    int nt, ntiles;
    column_tiles((int)(2 * nlev), nt, ntiles);
    return (size_t)((int64_t)(p->T + 1) * 2 * ntiles * nt * p->nhs * (int64_t)sizeof(float));
}

int zfpx_legendre_status(zfpx_legendre p)
{
    if (!p) return ZFPX_EINVAL;
    int v = 0;
    if (cudaMemcpy(&v, p->d_status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return ZFPX_ECUDA;
    return v ? ZFPX_ETIMEOUT : ZFPX_OK;
}

int zfpx_legendre_forward(zfpx_legendre p, const float *d_re, const float *d_im, const int64_t n[3],
                          const int64_t stride[3], float *d_are, float *d_aim, int64_t out_stride, void *d_work,
                          size_t work_bytes, void *stream)
{
    if (!p || !d_re || !d_im || !n || !stride || !d_are || !d_aim || !d_work) return ZFPX_EINVAL;
    if (n[0] < p->T + 1 || n[1] != p->nlat || n[2] < 1 || n[2] > (1 << 20)) return ZFPX_EINVAL;
    if (stride[0] != 1 || stride[1] < 0 || stride[2] < 0) return ZFPX_EINVAL;
    if (out_stride < (int64_t)(p->T + 1) * (p->T + 2) / 2) return ZFPX_EINVAL;
    if (((uintptr_t)d_re & 3u) || ((uintptr_t)d_im & 3u) || ((uintptr_t)d_are & 3u) || ((uintptr_t)d_aim & 3u) ||
        ((uintptr_t)d_work & 15u))
        return ZFPX_EINVAL;
    if (work_bytes < zfpx_legendre_workspace_bytes(p, n[2])) return ZFPX_ESIZE;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ZFPX_ECUDA;
    if (dev != p->device) return ZFPX_EINVAL;
    // the tensor map is encoded through the driver, which wants a current context:
    // a host thread that has made no runtime call yet has none
    if (cudaSetDevice(dev) != cudaSuccess) return ZFPX_ECUDA;
    LegGeom g{};
    g.nlat = p->nlat; g.nh = p->nh; g.nhs = p->nhs; g.T = p->T; g.nlev = (int)n[2];
    g.N = 2 * g.nlev;
    column_tiles(g.N, g.nt, g.ntiles);
    g.ncp = g.nt * g.ntiles;
    g.ntiles = (g.N + kMaxTile - 1) / kMaxTile;
    g.nt = ((g.N + g.ntiles - 1) / g.ntiles + 15) / 16 * 16;
    g.is1 = stride[1]; g.is2 = stride[2]; g.os = out_stride;
    const int64_t grows = (int64_t)(p->T + 1) * 2 * g.ncp;
    if (grows > 0x7fffffff || p->table_rows > 0x7fffffff) return ZFPX_EINVAL;
    float *G = static_cast<float *>(d_work);
    CUtensorMap tmap_g;
    int rc = make_tmap(&tmap_g, G, p->nh, grows, p->nhs, g.nt);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    if (2 * g.nlev > 65535) return ZFPX_EINVAL;
    const bool vec4 = stride[1] % 4 == 0 && stride[2] % 4 == 0 && !((uintptr_t)d_re & 15u) && !((uintptr_t)d_im & 15u);
    if (vec4) {
        const dim3 fgrid((p->T + 1 + 127) / 128, (p->nhs + 31) / 32, 2 * g.nlev);
        legendre_fold4_kernel<<<fgrid, dim3(32, 8), 0, st>>>(d_re, d_im, G, g);
    } else {
        const dim3 fgrid((p->T + 1 + 31) / 32, (p->nhs + 31) / 32, 2 * g.nlev);
        legendre_fold_kernel<<<fgrid, dim3(32, 8), 0, st>>>(d_re, d_im, G, g);
    }
    count_launch();
    rc = check_launch();
    if (rc) return rc;
    const int64_t nblk = (int64_t)p->nitems * g.ntiles;
    if (nblk > 0x7fffffff) return ZFPX_EINVAL;
    if (nblk == 0) return ZFPX_OK;
    const size_t smem = mma_smem_bytes(g.nt);
    if ((rc = allow_smem((const void *)legendre_mma_kernel, smem))) return rc;
    const int grid = (int)std::min<int64_t>(nblk, num_sms());      // persistent: one CTA per SM
    legendre_mma_kernel<<<grid, kMmaThreads, smem, st>>>(p->tmap_table, tmap_g, p->d_items, g,
                                                          mma_stages(g.nt), (int)nblk,
                                                          d_are, d_aim, p->d_status);
    count_launch();
    return check_launch();
}

}  // extern "C"
