// Device pieces of the longitude FFT (fourier.cu), shared with the fused
// decode + FFT kernel (rfft_fused.cu): the radix stages of the self-sorting
// H-point complex FFT and the split of its result into the N = 2H-point real
// transform's wavenumbers (see fourier.cu for the method).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace zfpx {
namespace fft {

constexpr int kMaxStages = 16;
constexpr int kMaxHalf = 4096;                  // N <= 8192

// n / d for n d < 2^32 as one multiply-high by m = ceil(2^32 / d) (exact in
// that range: m d - 2^32 < d); d = 1 has m = 0 and returns n.
struct FastDiv {
    uint32_t d, m;
    __device__ __forceinline__ uint32_t div(uint32_t n) const { return m ? __umulhi(n, m) : n; }
};
__host__ __device__ constexpr FastDiv make_fastdiv(uint32_t d)
{
    return FastDiv{d, d == 1 ? 0u : (uint32_t)((((uint64_t)1 << 32) + d - 1) / d)};
}

struct FftGeom {
    int N, H, K, nst;
    int r1;                   // > 0: N = 64 r1, taken in two register passes (rfft_row64); 0: the stages below
    int radix[kMaxStages];
    FastDiv rp[kMaxStages];   // r / p of each stage
    int64_t nrows, ny;
    int64_t is1, is2;         // input row strides (floats)
    int64_t os1, os2;         // output row strides (floats)
};

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -(a.y * b.y)), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// multiply by -i
__device__ __forceinline__ float2 cmul_mi(float2 a) { return make_float2(a.y, -a.x); }

__device__ __forceinline__ void dft4(float2 a0, float2 a1, float2 a2, float2 a3, float2 &v0, float2 &v1, float2 &v2,
                                     float2 &v3)
{
    // w_4 = -i: v_s = sum_q a_q (-i)^{s q}
    const float2 a = cadd(a0, a2), b = csub(a0, a2);
    const float2 c = cadd(a1, a3), d = cmul_mi(csub(a1, a3));
    v0 = cadd(a, c);
    v1 = cadd(b, d);
    v2 = csub(a, c);
    v3 = csub(b, d);
}

// 3 and 5 points by the symmetric and antisymmetric sums of the inputs j and
// P - j: half the products of the plain sums
__device__ __forceinline__ void dft3(float2 a0, float2 a1, float2 a2, float2 &v0, float2 &v1, float2 &v2)
{
    constexpr float s = 0.86602540378443864676f;               // sin(2 pi / 3)
    const float2 t = cadd(a1, a2), d = csub(a1, a2);
    v0 = cadd(a0, t);
    const float2 p = make_float2(fmaf(-0.5f, t.x, a0.x), fmaf(-0.5f, t.y, a0.y));
    v1 = make_float2(fmaf(s, d.y, p.x), fmaf(-s, d.x, p.y));
    v2 = make_float2(fmaf(-s, d.y, p.x), fmaf(s, d.x, p.y));
}
__device__ __forceinline__ void dft5(float2 a0, float2 a1, float2 a2, float2 a3, float2 a4, float2 &v0, float2 &v1,
                                     float2 &v2, float2 &v3, float2 &v4)
{
    constexpr float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;   // cos(2 pi / 5), cos(4 pi / 5)
    constexpr float s1 = 0.95105651629515357212f, s2 = 0.58778525229247312917f;    // sin(2 pi / 5), sin(4 pi / 5)
    const float2 t1 = cadd(a1, a4), t2 = cadd(a2, a3), d1 = csub(a1, a4), d2 = csub(a2, a3);
    v0 = cadd(a0, cadd(t1, t2));
    const float2 p1 = make_float2(fmaf(c2, t2.x, fmaf(c1, t1.x, a0.x)), fmaf(c2, t2.y, fmaf(c1, t1.y, a0.y)));
    const float2 p2 = make_float2(fmaf(c1, t2.x, fmaf(c2, t1.x, a0.x)), fmaf(c1, t2.y, fmaf(c2, t1.y, a0.y)));
    const float2 q1 = make_float2(fmaf(s2, d2.x, s1 * d1.x), fmaf(s2, d2.y, s1 * d1.y));
    const float2 q2 = make_float2(fmaf(-s1, d2.x, s2 * d1.x), fmaf(-s1, d2.y, s2 * d1.y));
    v1 = make_float2(p1.x + q1.y, p1.y - q1.x);                 // p1 - i q1
    v4 = make_float2(p1.x - q1.y, p1.y + q1.x);
    v2 = make_float2(p2.x + q2.y, p2.y - q2.x);
    v3 = make_float2(p2.x - q2.y, p2.y + q2.x);
}

// v_s = sum_q u_q w_P^{s q}, with w[j] = w_P^j.  P = 8 and 16 as two levels:
// q = B a + b, s = c + 4 d (B = P / 4): a 4-point DFT over a for every b, the
// twiddle w_P^{b c}, then a B-point DFT over b for every c.
template <int P>
__device__ __forceinline__ void small_dft(const float2 (&u)[P], float2 (&v)[P], const float2 (&w)[P])
{
    if constexpr (P == 2) {
        v[0] = cadd(u[0], u[1]);
        v[1] = csub(u[0], u[1]);
    } else if constexpr (P == 4) {
        dft4(u[0], u[1], u[2], u[3], v[0], v[1], v[2], v[3]);
    } else if constexpr (P == 8 || P == 16) {
        constexpr int B = P / 4;
        float2 t[B][4];
#pragma unroll
        for (int b = 0; b < B; b++) {
            dft4(u[b], u[B + b], u[2 * B + b], u[3 * B + b], t[b][0], t[b][1], t[b][2], t[b][3]);
#pragma unroll
            for (int c = 1; c < 4; c++)
                if (b) t[b][c] = cmul(t[b][c], w[(b * c) % P]);
        }
#pragma unroll
        for (int c = 0; c < 4; c++) {
            if constexpr (B == 2) {
                v[c] = cadd(t[0][c], t[1][c]);
                v[c + 4] = csub(t[0][c], t[1][c]);
            } else {
                dft4(t[0][c], t[1][c], t[2][c], t[3][c], v[c], v[c + 4], v[c + 8], v[c + 12]);
            }
        }
    } else if constexpr (P == 3) {
        dft3(u[0], u[1], u[2], v[0], v[1], v[2]);
    } else {
        dft5(u[0], u[1], u[2], u[3], u[4], v[0], v[1], v[2], v[3], v[4]);
    }
}

// FIRST: the first stage (L = 1, so f = 0 and every twiddle is 1).
template <int P, bool FIRST>
__device__ __forceinline__ void fft_stage(const float2 *x, float2 *y, const float2 *__restrict__ tw, int N, int H,
                                          int L, int lane, FastDiv drp)
{
    const int Lp = L * P, r = H / L, rp = (int)drp.d, nb = H / P;
    float2 w[P];
#pragma unroll
    for (int j = 0; j < P; j++) w[j] = __ldg(tw + (int64_t)j * (N / P));
    const int tstep = N / Lp;                   // w_{pL}^{t} = e^{-2 pi i t / (pL)} = tw[t N / (pL)]
    for (int b = lane; b < nb; b += 32) {
        const int f = (int)drp.div(b), k = b - f * rp;
        float2 u[P], v[P];
#pragma unroll
        for (int q = 0; q < P; q++) {
            const float2 a = x[k + rp * q + r * f];
            u[q] = (FIRST || !q) ? a : cmul(a, __ldg(tw + f * q * tstep));
        }
        small_dft<P>(u, v, w);
#pragma unroll
        for (int s = 0; s < P; s++) y[k + rp * (f + L * s)] = v[s];
    }
}


// A row of H complex values (8-byte aligned) into shared memory by
// asynchronous copies, every copy of the lane in flight at once (16 bytes each
// when both addresses are on 16 bytes and H is even, else 8), as one commit
// group; wait_rows() waits for the lane's groups.
__device__ __forceinline__ void load_row_async(float2 *dst, const float2 *src, int H, int lane)
{
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(dst);
    if (((((uint32_t)(uintptr_t)src) | s) & 15u) == 0 && (H & 1) == 0) {
        for (int k = lane; k < H / 2; k += 32)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s + 16u * (uint32_t)k), "l"(src + 2 * k)
                         : "memory");
    } else {
        for (int k = lane; k < H; k += 32)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s + 8u * (uint32_t)k), "l"(src + k)
                         : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void wait_rows() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// X holds Z_f at f < H; writes X_m / N, m < K, to ore / oim.  X_m = E_m + P_m
// with E_m = (Z_m + conj Z_{H-m}) / 2, P_m = e^{-2 pi i m / N} (Z_m - conj
// Z_{H-m}) / (2i), and from the same two X_{H-m} = conj(E_m - P_m).  One warp.
// STREAM: the output is marked as not to be kept in the caches (1280 x 640 rows of
// 1280: 165.9 -> 161.8 us; not where the input comes from L2, as in the fused
// kernel, 624.6 -> 630.3).
template <bool STREAM>
__device__ __forceinline__ void split_real(const float2 *X, const float2 *__restrict__ tw, int H, int K, float scale,
                                           int lane, float *ore, float *oim)
{
    auto put = [](float *p, float v) { if (STREAM) __stcs(p, v); else *p = v; };
#pragma unroll 2
    for (int m = lane; 2 * m <= H; m += 32) {
        const float2 zm = X[m], zc = X[m ? H - m : 0];
        const float2 E = make_float2(0.5f * (zm.x + zc.x), 0.5f * (zm.y - zc.y));
        const float2 O = make_float2(0.5f * (zm.y + zc.y), -0.5f * (zm.x - zc.x));
        const float2 P = cmul(O, __ldg(tw + m));
        if (m < K) {
            put(ore + m, (E.x + P.x) * scale);
            put(oim + m, (E.y + P.y) * scale);
        }
        if (H - m < K && 2 * m != H) {
            put(ore + H - m, (E.x - P.x) * scale);
            put(oim + H - m, (P.y - E.y) * scale);
        }
    }
    __syncwarp();
}

// One row: X holds the H complex values z_k = x_2k + i x_2k+1 on entry; Y is
// scratch of H values; writes X_m / N, m < K, to ore / oim.  One warp.
template <bool STREAM>
__device__ __forceinline__ void rfft_row(float2 *X, float2 *Y, const float2 *__restrict__ tw, const FftGeom &g,
                                         int lane, float *ore, float *oim)
{
    const int H = g.H;
    const float scale = 1.0f / (float)g.N;
    int L = 1;
    for (int s = 0; s < g.nst; s++) {
        const int p = g.radix[s];
        if (s == 0) {
            if (p == 16) fft_stage<16, true>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
            else if (p == 8) fft_stage<8, true>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
            else if (p == 4) fft_stage<4, true>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
            else if (p == 2) fft_stage<2, true>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
            else if (p == 3) fft_stage<3, true>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
            else fft_stage<5, true>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
        } else {
            if (p == 16) fft_stage<16, false>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
            else if (p == 8) fft_stage<8, false>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
            else if (p == 4) fft_stage<4, false>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
            else if (p == 2) fft_stage<2, false>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
            else if (p == 3) fft_stage<3, false>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
            else fft_stage<5, false>(X, Y, tw, g.N, H, L, lane, g.rp[s]);
        }
        __syncwarp();
        float2 *t = X; X = Y; Y = t;
        L *= p;
    }
    split_real<STREAM>(X, tw, H, g.K, scale, lane, ore, oim);
}

// rfft_row for a length whose stages P ... are fixed when it is compiled: the same
// values in half the instructions (no dispatch over the radices, and every index
// and twiddle distance a constant).
template <int N, int L, int P, int... REST>
__device__ __forceinline__ float2 *fixed_stages(float2 *X, float2 *Y, const float2 *__restrict__ tw, int lane)
{
    fft_stage<P, L == 1>(X, Y, tw, N, N / 2, L, lane, make_fastdiv(N / 2 / L / P));
    __syncwarp();
    if constexpr (sizeof...(REST) > 0) return fixed_stages<N, L * P, REST...>(Y, X, tw, lane);
    return Y;
}
template <bool STREAM, int N, int... P>
__device__ __forceinline__ void rfft_row_fixed(float2 *X, float2 *Y, const float2 *__restrict__ tw, int K, int lane,
                                               float *ore, float *oim)
{
    split_real<STREAM>(fixed_stages<N, 1, P...>(X, Y, tw, lane), tw, N / 2, K, 1.0f / (float)N, lane, ore, oim);
}
// Built for the multiples of 32 below the two register passes, in
// factor_half_impl's order: their stages leave lanes idle, so the dispatch weighs
// most there, and pairs of outputs (split_real) take longer than an output a lane.
// us for 262144 rows, K = N / 2, general stages with an output a lane, with pairs,
// and these: N = 32: 164, 178, 94; 64: 216, 229, 105; 96: 244, 232, 121; 128: 228,
// 244, 134; 160: 277, 263, 161; 192: 305, 308, 164.
// Fn: a macro taking N and the radices.
#define ZFPX_FFT_FIXED_LENGTHS(F) F(32, 16) F(64, 16, 2) F(96, 16, 3) F(128, 16, 4) F(160, 16, 5) F(192, 16, 2, 3)

// ------------------------------------------------------------------ N = 64 r1
// The H = 32 r1 points in two passes of registers.  Pass 1: lane k takes the r1
// points z_{k + 32 q} straight from global memory (every load of the warp one
// run of 256 bytes), transforms them and applies the twiddle w_H^{k s} to
// output s; pass 2: lane s < r1 transforms the 32 values of output s, which gives
// Z at s + r1 t.  One trip through shared memory between the passes and one to
// the split, in one buffer (every lane has read before any writes), where the
// stages above take a trip per radix and two buffers.
// Bounds it: the instructions of the two transforms and the split.  For N = 1280
// the stages of 16, 4 and 5 (the first with 40 butterflies on 32 lanes) took
// 2860 warp instructions a row and 302 us for 1280 x 640 x 137, these passes
// 1410 and 164 us, 0.8 of the copy rate.

// e^{-2 pi i j / R}, computed in double and rounded once
template <int R>
struct Roots {
    float c[R], s[R];
};
__host__ __device__ constexpr double roots_sin(double x)                             // 0 <= x <= pi / 4
{
    double t = x, r = x;
    for (int k = 1; k < 12; k++) { t *= -x * x / ((2 * k) * (2 * k + 1)); r += t; }
    return r;
}
__host__ __device__ constexpr double roots_cos(double x)
{
    double t = 1.0, r = 1.0;
    for (int k = 1; k < 12; k++) { t *= -x * x / ((2 * k - 1) * (2 * k)); r += t; }
    return r;
}
// cos(2 pi j / p), 0 <= j < p, by reduction to an eighth of the circle
__host__ __device__ constexpr double roots_cos_turn(int j, int p)
{
    constexpr double two_pi = 6.283185307179586476925286766559;
    if (2 * j > p) j = p - j;
    const bool neg = 4 * j > p;
    // quarter turn: j / p, or 1 / 2 - j / p, as a fraction of 2 p
    const int num = neg ? p - 2 * j : 2 * j;                     // angle / (2 pi) = num / (2 p)
    const double r = 8 * num > 2 * p ? roots_sin(two_pi * ((double)(p - 2 * num) / (4.0 * p)))
                                     : roots_cos(two_pi * ((double)num / (2.0 * p)));
    return neg ? -r : r;
}
template <int R>
__host__ __device__ constexpr Roots<R> make_roots()
{
    Roots<R> w{};
    for (int j = 0; j < R; j++) {
        w.c[j] = (float)roots_cos_turn(j, R);
        // sin(2 pi j / R) = cos(2 pi (4 j - R) / (4 R))
        const int q = (4 * j - R + 4 * R) % (4 * R);
        w.s[j] = (float)roots_cos_turn(q, 4 * R);
    }
    return w;
}

// a e^{-2 pi i j / R}; j is a constant once the caller's loops are unrolled
template <int R>
__device__ __forceinline__ float2 rotate(float2 a, int j)
{
    constexpr Roots<R> W = make_roots<R>();
    j %= R;
    if (j == 0) return a;
    if (4 * j == R) return make_float2(a.y, -a.x);
    if (2 * j == R) return make_float2(-a.x, -a.y);
    if (4 * j == 3 * R) return make_float2(-a.y, a.x);
    return cmul(a, make_float2(W.c[j], -W.s[j]));
}

// v_s = sum_q u_q w_R^{s q} in registers; R = A B as B transforms of A points,
// twiddles, A transforms of B points (q = B a + b, s = c + A d)
template <int R>
__device__ __forceinline__ void reg_dft(const float2 (&u)[R], float2 (&v)[R])
{
    if constexpr (R == 1) {
        v[0] = u[0];
    } else if constexpr (R == 2) {
        v[0] = cadd(u[0], u[1]);
        v[1] = csub(u[0], u[1]);
    } else if constexpr (R == 3) {
        dft3(u[0], u[1], u[2], v[0], v[1], v[2]);
    } else if constexpr (R == 4) {
        dft4(u[0], u[1], u[2], u[3], v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 5) {
        dft5(u[0], u[1], u[2], u[3], u[4], v[0], v[1], v[2], v[3], v[4]);
    } else {
        constexpr int A = R % 4 == 0 ? 4 : R % 2 == 0 ? 2 : R % 3 == 0 ? 3 : 5, B = R / A;
        float2 t[A][B];
#pragma unroll
        for (int b = 0; b < B; b++) {
            float2 x[A], y[A];
#pragma unroll
            for (int a = 0; a < A; a++) x[a] = u[B * a + b];
            reg_dft<A>(x, y);
#pragma unroll
            for (int c = 0; c < A; c++) t[c][b] = rotate<R>(y[c], b * c);
        }
#pragma unroll
        for (int c = 0; c < A; c++) {
            float2 y[B];
            reg_dft<B>(t[c], y);
#pragma unroll
            for (int d = 0; d < B; d++) v[c + A * d] = y[d];
        }
    }
}

// Complex values of shared memory per warp: pass 1's output in rows of 33
__host__ __device__ constexpr int row64_values(int r1) { return 33 * r1; }

// One row (src: its H complex values in global memory) through `buf`
// (row64_values(R1) values); tw2[32 s + k] = w_H^{k s}.  One warp.
template <int R1, bool STREAM>
__device__ __forceinline__ void rfft_row64(const float2 *src, float2 *buf, const float2 *__restrict__ tw,
                                           const float2 *__restrict__ tw2, int K, int lane, float *ore, float *oim)
{
    constexpr int H = 32 * R1;
    {
        float2 u[R1], v[R1];
#pragma unroll
        for (int q = 0; q < R1; q++) u[q] = src[lane + 32 * q];
        reg_dft<R1>(u, v);
        buf[lane] = v[0];
#pragma unroll
        for (int s = 1; s < R1; s++) buf[33 * s + lane] = cmul(v[s], __ldg(tw2 + 32 * s + lane));
    }
    __syncwarp();
    {
        float2 u[32], v[32];
        const int s = lane < R1 ? lane : 0;
#pragma unroll
        for (int k = 0; k < 32; k++) u[k] = buf[33 * s + k];
        __syncwarp();
        if (lane < R1) {
            reg_dft<32>(u, v);
#pragma unroll
            for (int t = 0; t < 32; t++) buf[lane + R1 * t] = v[t];
        }
    }
    __syncwarp();
    split_real<STREAM>(buf, tw, H, K, 1.0f / (float)(2 * H), lane, ore, oim);
}

// The first radices rfft_row64 is built for: the 2-3-5 numbers from 4 to 20.  us
// for 65536 rows, K = N / 2, the stages above against the two passes: N = 256: 76,
// 58; 320: 88, 62; 384: 93, 68; 512: 124, 70; 576: 126, 75; 640: 115, 82; 768: 133,
// 86; 960: 179, 101; 1024: 187, 99; 1152: 214, 119; 1280: 201, 122.  Longer rows take
// the stages: the passes are neither built nor measured for them.
// Fn: a macro taking the radix.
#define ZFPX_FFT_ROW64_RADICES(F) F(4) F(5) F(6) F(8) F(9) F(10) F(12) F(15) F(16) F(18) F(20)
inline bool row64_radix(int r1)
{
#define ZFPX_FFT_IS(R) || r1 == R
    return false ZFPX_FFT_ROW64_RADICES(ZFPX_FFT_IS);
#undef ZFPX_FFT_IS
}

}  // namespace fft

// Host side (fourier.cu): e^{-2 pi i t / N}, t < N, per (device, N), built once
// and never freed, followed for N = 64 r1 by w_H^{k s} at 32 s + k (s < r1, k <
// 32); and the radix plan of H (false if H has a prime factor other than 2, 3,
// 5).
int fft_twiddles(int N, const float2 **out);
bool fft_plan_half(int H, fft::FftGeom &g);

}  // namespace zfpx
