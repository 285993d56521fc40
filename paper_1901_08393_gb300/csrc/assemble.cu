// Assembly of the Galerkin matrix V[i][j] = (1/4pi) int_Ti int_Tj 1/|x-y| on
// piecewise constants (Eq. 2.4-2.5; primal P0 form of App. A, Eq. A.1).
//
//  * Far field (no common vertex): 7 x 7 product of Radon's degree-5 rule,
//      V_ij = |Ti||Tj|/(4pi) sum_a w_a sum_b w_b / |x_a - y_b|.
//    One thread per column j holds its 7 points (FP64, FP32: in registers; DF64: its
//    triangle's table in shared memory); the CTA stages R row triangles in
//    shared memory and walks them (broadcast reads; R x C tile variants, chosen per
//    size class by timing them).  Only
//    entries with i <= j are computed; the strict lower triangle is mirrored, so
//    V is exactly symmetric and an incremental re-assembly reproduces the full
//    one bit for bit.  Three arithmetic variants:
//      DF64 -- FP64-accurate double-float on the FP32 pipe.  The centroid difference
//              d = c_i - c_j is taken exactly from three-float centroids.  Pairs at
//              least 1.5 (R_i + R_j) apart (R: the largest distance of a triangle's
//              points from its centroid; almost all far pairs) expand |x_a - y_b|^2
//              into dot products of d and the points' offsets, split on one
//              power-of-two grid chosen for the pair so that hi parts add exactly;
//              closer pairs form x_a - y_b by two-sums, gathered so that whole warps
//              take them.  1/|r| by the MUFU reciprocal square root and one step in
//              double-float.  Entries within 3e-13 of FP64 (r.m.s. 3e-14).  V stored
//              as hi/lo pairs.
//      F64  -- native FP64 (GB300 issues FP64 at 1/64 of the FP32 rate): 7 FP64
//              operations per point pair, the reciprocal root's estimate and its
//              quadratic correction on the FP32 pipe.
//      F32  -- centroid difference from hi + lo float centroids, offsets in FP32, MUFU rsqrt;
//              no FP64 operation per pair (GB300 issues FP64 at 1/64 of the FP32 rate).
//  * Near field (common vertex, common edge, identical): Sauter-Schwab
//    regularising transformations.  The 4-d integrand of each region is a power
//    of the radial variables times a function of the others (the kernel is
//    homogeneous of degree -1 on flat panels), so the radial integrals are taken
//    exactly (1/3 for xi^2, 1/2 for rho) -- the same value that a Gauss-Legendre
//    rule with >= 2 points gives in those variables -- and the remaining
//    variables use n Gauss-Legendre points each: identical 6 hexagon sectors x n,
//    common edge 4 sub-regions x n^2, common vertex 2 regions x n^3.  FP64.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "bem_internal.cuh"
#include "dfloat.cuh"

namespace bem {

__constant__ double c_w7[kQ];
__constant__ float2 c_w7df[kQ];
__constant__ float2 c_inv4pi_df;
__constant__ double c_inv4pi_f32;  // 1 / (4 pi (sum of the FP32 Radon weights)^2)
__constant__ double c_glx[kMaxSS + 1][kMaxSS];
__constant__ double c_glw[kMaxSS + 1][kMaxSS];

static bool g_asm_ready[64] = {false};

// Gauss-Legendre rule with n points on [0, 1]: roots of P_n by Newton's method on
// the three-term recurrence, weights 2 / ((1 - x^2) P_n'(x)^2) halved.
static void gauss_legendre(int n, double *x, double *w)
{
    const double pi = 3.14159265358979323846;
    for (int i = 0; i < n; ++i) {
        double r = std::cos(pi * (i + 0.75) / (n + 0.5));
        double d = 0.0;
        for (int it = 0; it < 60; ++it) {
            double pm1 = 1.0, p = r;  // P_0, P_1
            for (int k = 1; k < n; ++k) {
                const double pn = ((2.0 * k + 1.0) * r * p - k * pm1) / (k + 1.0);
                pm1 = p;
                p = pn;
            }
            if (n == 1) { p = r; pm1 = 1.0; }
            d = n * (pm1 - r * p) / (1.0 - r * r);  // P_n'(r)
            const double step = p / d;
            r -= step;
            if (std::fabs(step) <= 1e-17) break;
        }
        double pm1 = 1.0, p = r;
        for (int k = 1; k < n; ++k) {
            const double pn = ((2.0 * k + 1.0) * r * p - k * pm1) / (k + 1.0);
            pm1 = p;
            p = pn;
        }
        if (n == 1) { p = r; pm1 = 1.0; }
        d = n * (pm1 - r * p) / (1.0 - r * r);
        x[n - 1 - i] = 0.5 * (1.0 + r);
        w[n - 1 - i] = 1.0 / ((1.0 - r * r) * d * d);
    }
}

static bem_status assembly_constants(bem_ctx *ctx)
{
    if (ctx->device < 64 && g_asm_ready[ctx->device]) return BEM_OK;
    const double r15 = std::sqrt(15.0);
    const double wa = (155.0 - r15) / 1200.0, wb = (155.0 + r15) / 1200.0;
    const double w7[kQ] = {9.0 / 40.0, wa, wa, wa, wb, wb, wb};
    double X[kMaxSS + 1][kMaxSS] = {}, W[kMaxSS + 1][kMaxSS] = {};
    for (int n = 1; n <= kMaxSS; ++n) gauss_legendre(n, X[n], W[n]);
    float2 w7df[kQ];
    for (int a = 0; a < kQ; ++a) {
        const float h = (float)w7[a];
        w7df[a] = make_float2(h, (float)(w7[a] - (double)h));
    }
    BEM_CK(ctx, cudaMemcpyToSymbol(c_w7, w7, sizeof(w7)));
    BEM_CK(ctx, cudaMemcpyToSymbol(c_w7df, w7df, sizeof(w7df)));
    const float ih = (float)kInv4Pi;
    const float2 inv4pi = make_float2(ih, (float)(kInv4Pi - (double)ih));
    BEM_CK(ctx, cudaMemcpyToSymbol(c_inv4pi_df, &inv4pi, sizeof(inv4pi)));
    double wsum = 0.0;  // exact: seven floats of similar size
    for (int a = 0; a < kQ; ++a) wsum += (double)w7df[a].x;
    const double inv4pi_f32 = kInv4Pi / (wsum * wsum);
    BEM_CK(ctx, cudaMemcpyToSymbol(c_inv4pi_f32, &inv4pi_f32, sizeof(inv4pi_f32)));
    BEM_CK(ctx, cudaMemcpyToSymbol(c_glx, X, sizeof(X)));
    BEM_CK(ctx, cudaMemcpyToSymbol(c_glw, W, sizeof(W)));
    if (ctx->device < 64) g_asm_ready[ctx->device] = true;
    return BEM_OK;
}

static inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// Element storage: FP64, double-float hi/lo pair, or FP32.
template <typename T> struct Elem;
template <> struct Elem<double> {
    __device__ static double from_double(double v) { return v; }
    __host__ __device__ static double to_double(double v) { return v; }
};
template <> struct Elem<float> {
    __device__ static float from_double(double v) { return (float)v; }
    __host__ __device__ static double to_double(float v) { return (double)v; }
};
template <> struct Elem<float2> {
    __device__ static float2 from_double(double v) { return df_from_double(v); }
    __host__ __device__ static double to_double(float2 v) { return df_to_double(v); }
};

// ------------------------------------------------------------------ far field
// Pair tiles: a CTA of C threads (one column each) walks R row triangles staged in
// shared memory.  Every variant computes each entry with the same operations, so V
// is bit-identical whichever is used; the fastest depends on N (small meshes want
// more, smaller CTAs) and on the arithmetic, and is chosen by timing (autotune).
struct FarTileS {
    int rows, cols;
    int min_ctas;  // DF64: > 0 -- registers capped so that this many CTAs fit an SM
};
constexpr FarTileS kFarTiles[kFarTileVariants] = {
    {32, 256, 0}, {16, 256, 0}, {64, 256, 0}, {8, 128, 0}, {16, 128, 0}, {32, 128, 0}, {8, 128, 5},
    {16, 128, 5}, {32, 128, 5}, {4, 128, 5},  {8, 64, 10}, {4, 64, 10},  {2, 64, 10}, {1, 64, 10}};
constexpr bool far_rows_divide_cols()
{
    for (const FarTileS &t : kFarTiles)
        if (t.cols % t.rows) return false;
    return true;
}
static_assert(far_rows_divide_cols(), "a column tile holds whole row tiles (far_items)");

// The far-field bodies take the tile origin (first row i0, first column cbase) as
// arguments: the per-operator kernels derive it from the block index, the batched
// kernel (several operators in one launch) from its work list.
// v rounded to the nearest multiple of q = 2^(e-23), for |v| < 2^(e-1) and big =
// 1.5 * 2^e: v + big lies in [2^e, 2^(e+1)], whose spacing is q, and the subtraction
// of big is exact (Sterbenz).
__device__ __forceinline__ float grid_snap(float v, float big) { return __fsub_rn(__fadd_rn(v, big), big); }

// 1.5 * 2^(k + up) for a normal v in [2^k, 2^(k+1))
__device__ __forceinline__ float grid_big(float v, unsigned up)
{
    return __uint_as_float(((__float_as_uint(v) & 0x7f800000u) + (up << 23)) | 0x400000u);
}

constexpr double kSqrt15 = 3.87298334620741688518;
constexpr double kW0 = 9.0 / 40.0, kW1 = (155.0 - kSqrt15) / 1200.0, kW2 = (155.0 + kSqrt15) / 1200.0;
constexpr float kFarSpread2 = 2.2505f;  // 1.5^2, rounded up past the FP32 errors of the test

// FP64 <-> FP32 by integer operations, for magnitudes in the normal FP32 range (a
// conversion costs as much as an FP64 operation): a positive v truncated.
__device__ __forceinline__ float f64_to_f32_trunc(double v)
{
    return __uint_as_float(__funnelshift_l((unsigned)__double2loint(v), (unsigned)__double2hiint(v) - (896u << 20), 3));
}
// |v| truncated, at least 2^-127; |v| < 2^128
__device__ __forceinline__ float f64_to_f32_abs(double v)
{
    const unsigned h = max((unsigned)__double2hiint(v) & 0x7fffffffu, 896u << 20) - (896u << 20);
    return __uint_as_float(__funnelshift_l((unsigned)__double2loint(v), h, 3));
}
// The same for any v: infinity or NaN from 2^128 on (infinity and NaN among them), so that no
// comparison takes it for an ordinary length.
__device__ __forceinline__ float f64_to_f32_len(double v)
{
    const unsigned h = min(max((unsigned)__double2hiint(v) & 0x7fffffffu, 896u << 20), 1151u << 20) - (896u << 20);
    return __uint_as_float(__funnelshift_l((unsigned)__double2loint(v), h, 3));
}
// -2 v for a normal v (a zero becomes -+2^-1022)
__device__ __forceinline__ double f64_m2(double v)
{
    return __hiloint2double((int)(((unsigned)__double2hiint(v) ^ 0x80000000u) + (1u << 20)), __double2loint(v));
}
// a positive v exactly (zero: 2^-127)
__device__ __forceinline__ double f32_to_f64_pos(float v)
{
    const unsigned b = __float_as_uint(v);
    return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}

// Entry (i, j) of a close pair (see far_f64_body): every difference in FP64.
__device__ __noinline__ double far_f64_close(const double *__restrict__ qi, const double *__restrict__ qj)
{
    double acc = 0.0;
#pragma unroll 1
    for (int a = 0; a < kQ; ++a) {
        const double xa = qi[3 * a], ya = qi[3 * a + 1], za = qi[3 * a + 2];
        double s = 0.0;
#pragma unroll 1
        for (int b = 0; b < kQ; ++b) {
            const double dx = xa - qj[3 * b], dy = ya - qj[3 * b + 1], dz = za - qj[3 * b + 2];
            s += c_w7[b] * rsqrt(dx * dx + dy * dy + dz * dz);
        }
        acc += c_w7[a] * s;
    }
    return qi[21] * (qj[21] * kInv4Pi) * acc;
}

// Pairs at least 1.5 (R_i + R_j) apart (R: the largest distance of a triangle's points from
// its centroid) take |x_a - y_b|^2 = E_a + n_b - 2 e_a.o_b, e_a = x_a - c_j, o_b = y_b -
// c_j, n_b = |o_b|^2: 4 FP64 operations per point pair instead of 6.  The reciprocal root is
// the FP32 MUFU estimate on a grid (estimates of equal weight add exactly in FP32) and the
// correction y t / 2 + 3/8 y t^2, t = 1 - S y^2: 3 FP64 operations (y^2, t, the sum of y t)
// and the t^2 term, below 2^-34, in FP32, where rsqrt took about 8.  Conversions are integer
// operations.  7 FP64 operations per point pair instead of 15; bound by the FP64 pipe (2
// lanes per SM and cycle: 91% of it, 402 operations per entry).  Rotated polycubes, best tile:
// N = 604 434 -> 238 us, N = 2,416 3.40 -> 2.43 ms, N = 9,664 51.2 -> 34.7 ms.  Error of an
// entry against extended precision on the same points, emulated on cubes, graded cubes and
// polycubes: r.m.s. 8.1 - 8.3e-17, at most 4e-16; 8.9 - 9.2e-17 and 4e-16 for FP64 sums of
// rsqrt.  Close pairs are put aside per warp as in far_df_body.
template <int R, int C>
__device__ __forceinline__ void far_f64_body(const double *__restrict__ q64, const double *__restrict__ cent,
                                             double *__restrict__ V, int64_t ld, int64_t r1, int64_t c1, int64_t i0,
                                             int64_t cbase)
{
    __shared__ double sx[R][kQ64Stride];
    __shared__ double sc[R][3];
    __shared__ unsigned short close_s[C / 32][64];
    if (i0 > cbase + C - 1 || i0 >= r1) return;  // tile strictly below the diagonal
    for (int k = threadIdx.x; k < R * kQ64Stride; k += C) {
        const int r = k / kQ64Stride, c = k % kQ64Stride;
        const int64_t i = i0 + r < r1 ? i0 + r : r1 - 1;
        sx[r][c] = q64[i * kQ64Stride + c];
        if (c < 3) sc[r][c] = cent[4 * i + c];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t jw = cbase + 32 * warp, j = jw + lane, jc = j < c1 ? j : c1 - 1;
    if (jw >= c1) return;
    const double cj[3] = {cent[4 * jc], cent[4 * jc + 1], cent[4 * jc + 2]};
    double o[3 * kQ], n[kQ];
#pragma unroll
    for (int b = 0; b < kQ; ++b) {
#pragma unroll
        for (int c = 0; c < 3; ++c) o[3 * b + c] = q64[jc * kQ64Stride + 3 * b + c] - cj[c];
        n[b] = fma(o[3 * b + 2], o[3 * b + 2], fma(o[3 * b + 1], o[3 * b + 1], o[3 * b] * o[3 * b]));
    }
    const double Aj = q64[jc * kQ64Stride + 21] * kInv4Pi;
    const float Rj = (float)q64[jc * kQ64Stride + 23];
    unsigned short *list = close_s[warp];
    int n_close = 0;
    auto flush = [&](int m) {  // the first m pairs put aside (m <= 32)
        __syncwarp();
        if (lane < m) {
            const int e = list[lane];
            const int64_t i = i0 + (e >> 5), jj = jw + (e & 31);
            V[i * ld + jj] = far_f64_close(q64 + i * kQ64Stride, q64 + jj * kQ64Stride);
        }
        __syncwarp();
    };
    int rows = (int)((r1 - i0) < R ? (r1 - i0) : R);
    if (jw + 32 - i0 < rows) rows = (int)(jw + 32 - i0);  // rows past the warp's last column: below the diagonal
    for (int r = 0; r < rows; ++r) {
        const int64_t i = i0 + r;
        const bool valid = j < c1 && i <= j;
        const float fx = f64_to_f32_len(sc[r][0] - cj[0]), fy = f64_to_f32_len(sc[r][1] - cj[1]),
                    fz = f64_to_f32_len(sc[r][2] - cj[2]);
        const float D2 = fx * fx + fy * fy + fz * fz, Rs = f64_to_f32_len(sx[r][23]) + Rj;
        // where the bounds hold and |x - y|^2 is a normal FP32 number; not for NaN
        const bool wide = D2 >= kFarSpread2 * (Rs * Rs) && D2 >= 0x1p-68f && D2 <= 0x1p100f;
        if (valid && wide) {
            float y0;
            asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(D2));
            const float by = grid_big(y0, 6);
            // class sums by weight: w0^2, w0 w1, w0 w2, w1^2, w1 w2, w2^2
            float s[6], q[6];
            double l[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                s[k] = q[k] = 0.0f;
                l[k] = 0.0;
            }
#pragma unroll
            for (int a = 0; a < kQ; ++a) {
                const double ex = sx[r][3 * a] - cj[0], ey = sx[r][3 * a + 1] - cj[1], ez = sx[r][3 * a + 2] - cj[2];
                const double E = fma(ez, ez, fma(ey, ey, ex * ex));
                const double mx = f64_m2(ex), my = f64_m2(ey), mz = f64_m2(ez);
#pragma unroll
                for (int b = 0; b < kQ; ++b) {
                    constexpr int kClass[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
                    const int k = kClass[(a + 2) / 3][(b + 2) / 3];
                    const double S = fma(mz, o[3 * b + 2], fma(my, o[3 * b + 1], fma(mx, o[3 * b], E + n[b])));
                    float y;
                    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f64_to_f32_trunc(S)));
                    y = grid_snap(y, by);
                    const double yd = f32_to_f64_pos(y);
                    const double t = fma(-S, yd * yd, 1.0);
                    const float tf = f64_to_f32_abs(t);
                    s[k] = __fadd_rn(s[k], y);
                    l[k] = fma(yd, t, l[k]);
                    q[k] = __fmaf_rn(y * tf, tf, q[k]);
                }
            }
            constexpr double w[6] = {kW0 * kW0, kW0 * kW1, kW0 * kW2, kW1 * kW1, kW1 * kW2, kW2 * kW2};
            double acc = 0.0;
#pragma unroll
            for (int k = 0; k < 6; ++k)
                acc = fma(w[k], fma(0.5, l[k], f32_to_f64_pos(s[k])) + f32_to_f64_pos(0.375f * q[k]), acc);
            V[i * ld + j] = sx[r][21] * Aj * acc;
        }
        const bool put = valid && !wide && i != j;  // (i, i) is the near field's
        const unsigned mask = __ballot_sync(0xffffffffu, put);
        if (mask) {
            if (put) list[n_close + __popc(mask & ((1u << lane) - 1u))] = (unsigned short)(r * 32 + lane);
            n_close += __popc(mask);
            if (n_close >= 32) {
                flush(32);
                n_close -= 32;
                unsigned short rest = 0;
                if (lane < n_close) rest = list[32 + lane];
                __syncwarp();
                if (lane < n_close) list[lane] = rest;
                __syncwarp();
            }
        }
    }
    if (n_close) flush(n_close);
}

template <int R, int C>
__global__ void __launch_bounds__(C) k_far_f64(const double *__restrict__ q64, const double *__restrict__ cent,
                                               double *__restrict__ V, int64_t ld, int64_t r0, int64_t r1, int64_t c0,
                                               int64_t c1)
{
    far_f64_body<R, C>(q64, cent, V, ld, r1, c1, r0 + (int64_t)blockIdx.y * R, c0 + (int64_t)blockIdx.x * C);
}

template <int R, int C>
__device__ __forceinline__ void far_f32_body(const float *__restrict__ q32, const double *__restrict__ cent,
                                             float *__restrict__ V, int64_t ld, int64_t r1, int64_t c1,
                                             int64_t i0, int64_t cbase)
{
    // FP32 only in the pair loop: centroids as hi + lo floats, so that the centroid
    // difference (hi_i - hi_j) + (lo_i - lo_j) keeps FP32 relative accuracy for
    // distant pairs; weights and areas rounded to FP32 once
    __shared__ float4 so[R][kQ32Stride / 4];  // offsets (21 of 24 floats)
    __shared__ float4 sc[R][2];               // centroid hi (3) and area, lo (3)
    static_assert(kQ32Stride % 4 == 0 && kQ32Stride >= 3 * kQ, "rows of whole float4");
    if (i0 > cbase + C - 1 || i0 >= r1) return;
    for (int k = threadIdx.x; k < R * (kQ32Stride / 4); k += C) {
        const int r = k / (kQ32Stride / 4), c = k % (kQ32Stride / 4);
        const int64_t i = i0 + r < r1 ? i0 + r : r1 - 1;
        so[r][c] = reinterpret_cast<const float4 *>(q32 + i * kQ32Stride)[c];
    }
    for (int r = threadIdx.x; r < R; r += C) {
        const int64_t i = i0 + r < r1 ? i0 + r : r1 - 1;
        float h[4], l[3];
        for (int c = 0; c < 4; ++c) {
            const double v = cent[i * 4 + c];
            h[c] = (float)v;
            if (c < 3) l[c] = (float)(v - (double)h[c]);
        }
        sc[r][0] = make_float4(h[0], h[1], h[2], h[3]);
        sc[r][1] = make_float4(l[0], l[1], l[2], 0.0f);
    }
    __syncthreads();
    const int64_t j = cbase + threadIdx.x;
    if (j >= c1) return;
    float y[3 * kQ];
#pragma unroll
    for (int c = 0; c < 3 * kQ; ++c) y[c] = q32[j * kQ32Stride + c];
    float ch[3], cl[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double v = cent[4 * j + c];
        ch[c] = (float)v;
        cl[c] = (float)(v - (double)ch[c]);
    }
    // 1/(4pi) with the weights' rounding undone: the FP32 Radon weights all round down
    // (their sum is 1 - 2.98e-8), which would scale every far entry by (sum w)^2; the
    // factor 1 / (sum of the FP32 weights)^2 is folded into the column's area term
    const float Aj = (float)(cent[4 * j + 3] * c_inv4pi_f32);
    float wf[kQ];  // the weights rounded to FP32 once (c_w7df[.].x = nearest float)
#pragma unroll
    for (int a = 0; a < kQ; ++a) wf[a] = c_w7df[a].x;
    const int rows = (int)((r1 - i0) < R ? (r1 - i0) : R);
    for (int r = 0; r < rows; ++r) {
        const int64_t i = i0 + r;
        if (i > j) break;
        const float4 h4 = sc[r][0], l4 = sc[r][1];
        const float Dx = (h4.x - ch[0]) + (l4.x - cl[0]);
        const float Dy = (h4.y - ch[1]) + (l4.y - cl[1]);
        const float Dz = (h4.z - ch[2]) + (l4.z - cl[2]);
        float o[kQ32Stride];
#pragma unroll
        for (int k = 0; k < kQ32Stride / 4; ++k) {
            const float4 v = so[r][k];
            o[4 * k] = v.x;
            o[4 * k + 1] = v.y;
            o[4 * k + 2] = v.z;
            o[4 * k + 3] = v.w;
        }
        // The bare MUFU estimate gives rsqrtf's bits for normal arguments without the
        // scaling of subnormal ones (about 4 of 11 instructions per point pair); a
        // subnormal |d|^2 is infinity there, and the sum is then taken again with rsqrtf.
        // Bound by issue, then by MUFU (49 per entry, 16 lanes per SM and cycle: 103
        // Gpairs/s): N = 2,416 69.9 -> 55.2 us, N = 21,744 4.08 -> 3.31 ms (58.0 -> 71.4
        // Gpairs/s), the same bits.
        auto sum = [&](auto bare) {
            float acc = 0.0f;
#pragma unroll
            for (int a = 0; a < kQ; ++a) {
                const float xa = Dx + o[3 * a], ya = Dy + o[3 * a + 1], za = Dz + o[3 * a + 2];
                float s = 0.0f;
#pragma unroll
                for (int b = 0; b < kQ; ++b) {
                    const float dx = xa - y[3 * b], dy = ya - y[3 * b + 1], dz = za - y[3 * b + 2];
                    const float d2 = dx * dx + dy * dy + dz * dz;
                    float q;
                    if (decltype(bare)::value)
                        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(d2));
                    else
                        q = rsqrtf(d2);
                    s += wf[b] * q;
                }
                acc += wf[a] * s;
            }
            return acc;
        };
        float acc = sum(std::true_type());
        if (!(acc < INFINITY) && i != j) acc = sum(std::false_type());  // (i, i) is the near field's
        V[i * ld + j] = h4.w * Aj * acc;
    }
}

template <int R, int C>
__global__ void __launch_bounds__(C) k_far_f32(const float *__restrict__ q32,
                                                      const double *__restrict__ cent, float *__restrict__ V,
                                                      int64_t ld, int64_t r0, int64_t r1, int64_t c0,
                                                      int64_t c1)
{
    far_f32_body<R, C>(q32, cent, V, ld, r1, c1, r0 + (int64_t)blockIdx.y * R, c0 + (int64_t)blockIdx.x * C);
}

// Double-float far field: see the file comment.
//
// s + e = a + b exactly for a, b >= 0 (Dekker's fast two-sum with the larger first).
__device__ __forceinline__ void pos_two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    e = __fsub_rn(fminf(a, b), __fsub_rn(s, fmaxf(a, b)));
}

// sh + sl += w (y + yl) with the two-sum of the running sum
__device__ __forceinline__ void df_acc_w(float2 w, float y, float yl, float &sh, float &sl)
{
    float ph, pe, u, ue;
    two_prod(w.x, y, ph, pe);
    pe = __fmaf_rn(w.x, yl, pe);
    pe = __fmaf_rn(w.y, y, pe);
    two_sum(sh, ph, u, ue);
    sh = u;
    sl = __fadd_rn(sl, __fadd_rn(pe, ue));
}

// Centroid difference c_i - c_j from the three-float centroids, one coordinate.
__device__ __forceinline__ void centroid_diff(float a0, float a1, float a2, float b0, float b1, float b2, float &dh,
                                              float &dl)
{
    float s1, e1, s2, e2, h, l;
    two_sum(a0, -b0, s1, e1);
    two_sum(a1, -b1, s2, e2);
    two_sum(s1, s2, h, l);
    l = __fadd_rn(l, __fadd_rn(__fadd_rn(e1, e2), __fsub_rn(a2, b2)));
    fast_two_sum(h, l, dh, dl);
}

// Entry (i, j) of a pair whose triangles are close (|c_i - c_j| < 1.5 (R_i + R_j)):
// sum_a w_a sum_b w_b / |x_a - y_b| with x_a - y_b = (D + o_a) - o_b in double-float by
// two-sums, D = c_i - c_j, o the offsets from the centroids, and 1/|d| = y + y t / 2 from
// the MUFU estimate y by one Newton step, t = 1 - S y^2 with y^2 by a two-product (the
// estimate's relative error is below 2^-22, so 1 - Sh y2 is below 2^-20 in size and its
// single rounding in the FMA is below 2^-44).  74 FP32 operations per point pair; called
// for the few close pairs of a tile together (far_df_body), so kept out of line.
__device__ __noinline__ float2 far_df_close(const float *__restrict__ qi, const float *__restrict__ qj)
{
    float Dh[3], Dl[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
        centroid_diff(qi[42 + 3 * c], qi[43 + 3 * c], qi[44 + 3 * c], qj[42 + 3 * c], qj[43 + 3 * c], qj[44 + 3 * c],
                      Dh[c], Dl[c]);
    const float2 *oi = reinterpret_cast<const float2 *>(qi), *oj = reinterpret_cast<const float2 *>(qj);
    float acc_h = 0.0f, acc_l = 0.0f;
#pragma unroll 1
    for (int a = 0; a < kQ; ++a) {
        float eh[3], el[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float2 o = oi[3 * a + c];
            float s, e;
            two_sum(Dh[c], o.x, s, e);
            e = __fadd_rn(e, __fadd_rn(Dl[c], o.y));
            fast_two_sum(s, e, eh[c], el[c]);
        }
        float sh = 0.0f, sl = 0.0f;
#pragma unroll 1
        for (int b = 0; b < kQ; ++b) {
            // d = e_a - o_b; |d|^2 = sum h^2 + 2 h l (two-product, two-sum)
            float Sh = 0.0f, Sl = 0.0f;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float h, e;
                const float2 o = oj[3 * b + c];
                two_sum(eh[c], -o.x, h, e);
                const float l = __fadd_rn(e, __fsub_rn(el[c], o.y));
                float p, pe;
                two_prod(h, h, p, pe);
                pe = __fmaf_rn(__fmul_rn(2.0f, h), l, pe);
                if (c == 0) {
                    Sh = p;
                    Sl = pe;
                } else {
                    float t, te;
                    two_sum(Sh, p, t, te);
                    Sh = t;
                    Sl = __fadd_rn(Sl, __fadd_rn(pe, te));
                }
            }
            const float y = rsqrtf(Sh);
            float y2, y2e;
            two_prod(y, y, y2, y2e);
            float t = __fmaf_rn(-Sh, y2, 1.0f);
            t = __fmaf_rn(-Sh, y2e, t);
            t = __fmaf_rn(-Sl, y2, t);
            df_acc_w(c_w7df[b], y, __fmul_rn(__fmul_rn(0.5f, y), t), sh, sl);
        }
        df_acc_w(c_w7df[a], sh, sl, acc_h, acc_l);
    }
    float h, l;
    fast_two_sum(acc_h, acc_l, h, l);
    return df_mul(df_mul(make_float2(qi[51], qi[52]), df_mul(make_float2(qj[51], qj[52]), c_inv4pi_df)),
                  make_float2(h, l));
}

// The expanded form, for every other pair.  Radon's points of a triangle are its
// centroid and two orbits o_1k = t v_k, o_2k = s o_1k (v_k: vertex k from the centroid,
// t = (1 + sqrt 15) / 7, s = (1 - sqrt 15) / (1 + sqrt 15)), and o_12 = -(o_10 + o_11), so
//   |x_a - y_b|^2 = |d|^2 + A_a + B_b - C_ab,  d = c_i - c_j,
//   A_1k = 2 d.o_1k + |o_1k|^2,   A_2k = s 2 d.o_1k + |o_2k|^2   (B alike, with -2 d.o),
//   C = G, s G or s^2 G with G_kl = 2 o_1k.o_1l:
// 9 dot products of three terms for all 49 squared distances, instead of three
// differences and three squares for each.  Every product is split on one power-of-two
// grid of the pair, q = 2^(e-23) with 2^(e-1) > 1.34 |d|^2: its hi part is the multiple of
// q next to it (an FMA onto 1.5 * 2^e and a subtraction), its lo part the rest (an FMA),
// so that hi parts add exactly in plain additions: no term exceeds 4/3 |d|^2 and no sum
// 3 |d|^2 < 2^24 q while |d| >= 1.5 (R_i + R_j).  The lo parts add up with an error of a
// few units of 2^-24 q; every |x_a - y_b|^2 is at least |d|^2 / 9.  The MUFU estimate of
// 1/|x_a - y_b| is itself put on a grid (a multiple of 2^-17 .. 2^-18 of 1/|d|), so that
// estimates of equal weight add exactly; the step from there, y t (1/2 + 3/8 t) with t =
// 1 - S y^2 below 2^-16, goes to the lo sum.  Error of an entry (CPU emulation on cubes,
// graded cubes with needles, Fichera, polycubes): 2.2e-13 at most, 3e-14 r.m.s., no bias.
//
// 16 FP32 operations per point pair and about 520 per entry, against 50 and 336 of the
// form that took each of the 49 differences on a grid (three subtractions and squares
// each).  Bound by FP32 issue (72% of the 128 lanes per SM and cycle, 81% of the issue
// slots).  Measured on rotated
// polycubes, best tile of each: N = 604 116 -> 35 us, N = 2,416 418 -> 166 us, N = 9,664
// 4.60 -> 2.03 ms, N = 21,744 22.3 -> 9.88 ms (10.6 -> 23.9 Gpairs/s).
constexpr double kOrbS = (1.0 - kSqrt15) / (1.0 + kSqrt15);
constexpr float kOrbSh = (float)kOrbS, kOrbSl = (float)(kOrbS - (double)kOrbSh);
constexpr float kOrbS2h = (float)(kOrbS * kOrbS), kOrbS2l = (float)(kOrbS * kOrbS - (double)kOrbS2h);

// h + l = (ah + al) (bh + bl), h on the grid
__device__ __forceinline__ void grid_prod(float ah, float al, float bh, float bl, float big, float &h, float &l)
{
    h = __fsub_rn(__fmaf_rn(ah, bh, big), big);
    l = __fmaf_rn(ah, bl, __fmaf_rn(al, bh, __fmaf_rn(ah, bh, -h)));
}

// h + l = a.b for double-float vectors (h, l) x 3
__device__ __forceinline__ void grid_dot(const float *ah, const float *al, const float *bh, const float *bl, float big,
                                         float &h, float &l)
{
    float p[3], r[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) grid_prod(ah[c], al[c], bh[c], bl[c], big, p[c], r[c]);
    h = __fadd_rn(__fadd_rn(p[0], p[1]), p[2]);
    l = __fadd_rn(__fadd_rn(r[0], r[1]), r[2]);
}

// The offset terms of one triangle's orbits: h1 + l1 = p + |o_1|^2, h2 + l2 = s p +
// |o_2|^2 for the projection p of vertex k; n: (|o_1|^2 hi, lo, |o_2|^2 hi, lo).
__device__ __forceinline__ void orbit_terms(float ph, float pl, float4 n, float big, float &h1, float &l1, float &h2,
                                            float &l2)
{
    const float g1 = grid_snap(n.x, big), g2 = grid_snap(n.z, big);
    h1 = __fadd_rn(ph, g1);
    l1 = __fadd_rn(pl, __fadd_rn(__fsub_rn(n.x, g1), n.y));
    grid_prod(kOrbSh, kOrbSl, ph, pl, big, h2, l2);
    h2 = __fadd_rn(h2, g2);
    l2 = __fadd_rn(l2, __fadd_rn(__fsub_rn(n.z, g2), n.w));
}

// s + l += 1 / sqrt(H + L)
__device__ __forceinline__ void inv_root_acc(float H, float L, float by, float &s, float &l)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(H));  // H: a normal number
    y = grid_snap(y, by);
    float y2, y2e;
    two_prod(y, y, y2, y2e);
    float t = __fmaf_rn(-H, y2, 1.0f);
    t = __fmaf_rn(-H, y2e, t);
    t = __fmaf_rn(-L, y2, t);
    s = __fadd_rn(s, y);
    l = __fmaf_rn(y, __fmul_rn(t, __fmaf_rn(t, 0.375f, 0.5f)), l);
}

// acc += w (s + l), all positive
__device__ __forceinline__ void class_acc(double w, float s, float l, float &h, float &lo)
{
    const float wh = (float)w, wl = (float)(w - (double)wh);
    float p, e, u, ue;
    two_prod(wh, s, p, e);
    e = __fmaf_rn(wl, s, __fmaf_rn(wh, l, e));
    pos_two_sum(h, p, u, ue);
    h = u;
    lo = __fadd_rn(lo, __fadd_rn(e, ue));
}

// ri: the row triangle's nine float4 of the table (kQdfExp), cj: the column triangle's,
// stride C; dh, dl: c_i - c_j.
template <int C>
__device__ __forceinline__ void far_df_expanded(const float4 *ri, const float4 *cj, const float *dh, const float *dl,
                                                float big, float &h_out, float &l_out)
{
    float d2h[3], d2l[3];  // 2 d
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        d2h[c] = __fadd_rn(dh[c], dh[c]);
        d2l[c] = __fadd_rn(dl[c], dl[c]);
    }
    float Dh, Dl;
    {
        float p[3], r[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            p[c] = __fsub_rn(__fmaf_rn(dh[c], dh[c], big), big);
            r[c] = __fmaf_rn(d2h[c], dl[c], __fmaf_rn(dh[c], dh[c], -p[c]));
        }
        Dh = __fadd_rn(__fadd_rn(p[0], p[1]), p[2]);
        Dl = __fadd_rn(__fadd_rn(r[0], r[1]), r[2]);
    }
    float y0;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(Dh));
    const float by = grid_big(y0, 6);
    // class sums by weight: w0^2, w0 w1, w0 w2, w1^2, w1 w2, w2^2
    float s[6], l[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) s[k] = l[k] = 0.0f;
    inv_root_acc(Dh, Dl, by, s[0], l[0]);
    // column side: B_1l, B_2l, and the orbit offsets of vertices 0 and 1
    float wh[2][3], wl[2][3], B1h[3], B1l[3], B2h[3], B2l[3];
    {
        const float4 a = cj[0], b = cj[C], c = cj[2 * C];
        wh[0][0] = a.x; wl[0][0] = a.y; wh[0][1] = a.z; wl[0][1] = a.w; wh[0][2] = b.x; wl[0][2] = b.y;
        wh[1][0] = b.z; wl[1][0] = b.w; wh[1][1] = c.x; wl[1][1] = c.y; wh[1][2] = c.z; wl[1][2] = c.w;
        float qh[3], ql[3];
        grid_dot(d2h, d2l, wh[0], wl[0], big, qh[0], ql[0]);
        grid_dot(d2h, d2l, wh[1], wl[1], big, qh[1], ql[1]);
        qh[2] = -__fadd_rn(qh[0], qh[1]);
        ql[2] = -__fadd_rn(ql[0], ql[1]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            orbit_terms(-qh[k], -ql[k], cj[(3 + k) * C], big, B1h[k], B1l[k], B2h[k], B2l[k]);
            inv_root_acc(__fadd_rn(Dh, B1h[k]), __fadd_rn(Dl, B1l[k]), by, s[1], l[1]);
            inv_root_acc(__fadd_rn(Dh, B2h[k]), __fadd_rn(Dl, B2l[k]), by, s[2], l[2]);
        }
    }
    float psh = 0.0f, psl = 0.0f, Gsh[3] = {0.0f, 0.0f, 0.0f}, Gsl[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float ph, pl, Gh[3], Gl[3];
        if (k < 2) {
            float vh[3], vl[3];
            if (k == 0) {
                const float4 a = ri[0], b = ri[1];
                vh[0] = a.x; vl[0] = a.y; vh[1] = a.z; vl[1] = a.w; vh[2] = b.x; vl[2] = b.y;
            } else {
                const float4 b = ri[1], c = ri[2];
                vh[0] = b.z; vl[0] = b.w; vh[1] = c.x; vl[1] = c.y; vh[2] = c.z; vl[2] = c.w;
            }
            grid_dot(d2h, d2l, vh, vl, big, ph, pl);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                vh[c] = __fadd_rn(vh[c], vh[c]);
                vl[c] = __fadd_rn(vl[c], vl[c]);
            }
            grid_dot(vh, vl, wh[0], wl[0], big, Gh[0], Gl[0]);
            grid_dot(vh, vl, wh[1], wl[1], big, Gh[1], Gl[1]);
            Gh[2] = -__fadd_rn(Gh[0], Gh[1]);
            Gl[2] = -__fadd_rn(Gl[0], Gl[1]);
            psh = __fadd_rn(psh, ph);
            psl = __fadd_rn(psl, pl);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                Gsh[j] = __fadd_rn(Gsh[j], Gh[j]);
                Gsl[j] = __fadd_rn(Gsl[j], Gl[j]);
            }
        } else {  // vertex 2's offsets are minus the sum of the others'
            ph = -psh;
            pl = -psl;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                Gh[j] = -Gsh[j];
                Gl[j] = -Gsl[j];
            }
        }
        float A1h, A1l, A2h, A2l;
        orbit_terms(ph, pl, ri[3 + k], big, A1h, A1l, A2h, A2l);
        A1h = __fadd_rn(A1h, Dh);
        A1l = __fadd_rn(A1l, Dl);
        A2h = __fadd_rn(A2h, Dh);
        A2l = __fadd_rn(A2l, Dl);
        inv_root_acc(A1h, A1l, by, s[1], l[1]);
        inv_root_acc(A2h, A2l, by, s[2], l[2]);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float C1h, C1l, C2h, C2l;  // s G, s^2 G
            grid_prod(kOrbSh, kOrbSl, Gh[j], Gl[j], big, C1h, C1l);
            grid_prod(kOrbS2h, kOrbS2l, Gh[j], Gl[j], big, C2h, C2l);
            inv_root_acc(__fsub_rn(__fadd_rn(A1h, B1h[j]), Gh[j]), __fsub_rn(__fadd_rn(A1l, B1l[j]), Gl[j]), by, s[3],
                         l[3]);
            inv_root_acc(__fsub_rn(__fadd_rn(A1h, B2h[j]), C1h), __fsub_rn(__fadd_rn(A1l, B2l[j]), C1l), by, s[4],
                         l[4]);
            inv_root_acc(__fsub_rn(__fadd_rn(A2h, B1h[j]), C1h), __fsub_rn(__fadd_rn(A2l, B1l[j]), C1l), by, s[4],
                         l[4]);
            inv_root_acc(__fsub_rn(__fadd_rn(A2h, B2h[j]), C2h), __fsub_rn(__fadd_rn(A2l, B2l[j]), C2l), by, s[5],
                         l[5]);
        }
    }
    float acc_h = 0.0f, acc_l = 0.0f;
    class_acc(kW0 * kW0, s[0], l[0], acc_h, acc_l);
    class_acc(kW0 * kW1, s[1], l[1], acc_h, acc_l);
    class_acc(kW0 * kW2, s[2], l[2], acc_h, acc_l);
    class_acc(kW1 * kW1, s[3], l[3], acc_h, acc_l);
    class_acc(kW1 * kW2, s[4], l[4], acc_h, acc_l);
    class_acc(kW2 * kW2, s[5], l[5], acc_h, acc_l);
    fast_two_sum(acc_h, acc_l, h_out, l_out);
}

// The column triangles' table rows are kept in dynamic shared memory (9 x C float4,
// one column of the array per thread: conflict-free), the row triangles' beside them
// (broadcast reads).
template <int C>
constexpr size_t far_df_smem() { return sizeof(float4) * 9 * C; }
static_assert(far_df_smem<256>() + 64 * 9 * sizeof(float4) + 8 * 64 * sizeof(unsigned short) <= 48 * 1024,
              "the largest tile (64 x 256) fits the default shared memory per CTA");

// Close pairs (below 1.5 (R_i + R_j): 0.1-0.7% of the pairs from N = 5,000 on, most of them
// on meshes of a few hundred triangles) cost three times the others: each warp puts its
// own aside (row, lane) and computes them 32 at a time, so that a warp with one such pair
// does not run both forms for a whole row.  The last ones run with the lanes there are.
template <int R, int C>
__device__ __forceinline__ void far_df_body(const float *__restrict__ qdf, float2 *__restrict__ V, int64_t ld,
                                            int64_t r1, int64_t c1, int64_t i0, int64_t cbase)
{
    __shared__ float4 sq[R][9];
    __shared__ unsigned short close_s[C / 32][64];
    extern __shared__ float4 far_dsm[];
    if (i0 > cbase + C - 1 || i0 >= r1) return;
    const float4 *q4 = reinterpret_cast<const float4 *>(qdf + kQdfExp);
    constexpr int kS4 = kQdfStride / 4;
    for (int k = threadIdx.x; k < R * 9; k += C) {
        const int r = k / 9, c = k % 9;
        const int64_t i = i0 + r < r1 ? i0 + r : r1 - 1;
        sq[r][c] = q4[i * kS4 + c];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t jw = cbase + 32 * warp, j = jw + lane;
    float4 *cj = far_dsm + threadIdx.x;
    {
        const float4 *src = q4 + (j < c1 ? j : c1 - 1) * kS4;
#pragma unroll
        for (int k = 0; k < 9; ++k) cj[k * C] = src[k];
    }
    __syncthreads();
    if (jw >= c1) return;
    unsigned short *list = close_s[warp];
    int n_close = 0;
    auto flush = [&](int n) {  // the first n pairs put aside (n <= 32)
        __syncwarp();
        if (lane < n) {
            const int e = list[lane];
            const int64_t i = i0 + (e >> 5), jc = jw + (e & 31);
            V[i * ld + jc] = far_df_close(qdf + i * kQdfStride, qdf + jc * kQdfStride);
        }
        __syncwarp();
    };
    const float2 Aj = df_mul(make_float2(cj[7 * C].w, cj[8 * C].w), c_inv4pi_df);
    int rows = (int)((r1 - i0) < R ? (r1 - i0) : R);
    if (jw + 32 - i0 < rows) rows = (int)(jw + 32 - i0);  // rows past the warp's last column: below the diagonal
    for (int r = 0; r < rows; ++r) {
        const int64_t i = i0 + r;
        const bool valid = j < c1 && i <= j;
        float dh[3], dl[3], Rs, Ah, Al;
        {
            const float4 *ri = sq[r];
            const float4 a0 = ri[6], a1 = ri[7], a2 = ri[8], b0 = cj[6 * C], b1 = cj[7 * C], b2 = cj[8 * C];
            centroid_diff(a0.x, a1.x, a2.x, b0.x, b1.x, b2.x, dh[0], dl[0]);
            centroid_diff(a0.y, a1.y, a2.y, b0.y, b1.y, b2.y, dh[1], dl[1]);
            centroid_diff(a0.z, a1.z, a2.z, b0.z, b1.z, b2.z, dh[2], dl[2]);
            Rs = a0.w + b0.w;
            Ah = a1.w;
            Al = a2.w;
        }
        const float D2 = dh[0] * dh[0] + dh[1] * dh[1] + dh[2] * dh[2];
        const float m = 1.34f * D2;
        // the expanded form where its bounds hold (and no product of it can leave the
        // normal FP32 range); not for NaN
        const bool wide = D2 >= kFarSpread2 * (Rs * Rs) && m >= 0x1p-68f && m <= 0x1p100f;
        if (valid && wide) {
            float h, l;
            far_df_expanded<C>(sq[r], cj, dh, dl, grid_big(m, 2), h, l);
            V[i * ld + j] = df_mul(df_mul(make_float2(Ah, Al), Aj), make_float2(h, l));
        }
        const bool put = valid && !wide && i != j;  // (i, i) is the near field's
        const unsigned mask = __ballot_sync(0xffffffffu, put);
        if (mask) {
            if (put) list[n_close + __popc(mask & ((1u << lane) - 1u))] = (unsigned short)(r * 32 + lane);
            n_close += __popc(mask);
            if (n_close >= 32) {
                flush(32);
                n_close -= 32;
                unsigned short rest = 0;
                if (lane < n_close) rest = list[32 + lane];
                __syncwarp();
                if (lane < n_close) list[lane] = rest;
                __syncwarp();
            }
        }
    }
    if (n_close) flush(n_close);
}

// MB > 0: MB CTAs per SM requested (registers capped to fit)
template <int R, int C>
__global__ void __launch_bounds__(C) k_far_df(const float *__restrict__ qdf, float2 *__restrict__ V, int64_t ld,
                                              int64_t r0, int64_t r1, int64_t c0, int64_t c1)
{
    far_df_body<R, C>(qdf, V, ld, r1, c1, r0 + (int64_t)blockIdx.y * R, c0 + (int64_t)blockIdx.x * C);
}

template <int R, int C, int MB>
__global__ void __launch_bounds__(C, MB) k_far_df_s(const float *__restrict__ qdf, float2 *__restrict__ V, int64_t ld,
                                                    int64_t r0, int64_t r1, int64_t c0, int64_t c1)
{
    far_df_body<R, C>(qdf, V, ld, r1, c1, r0 + (int64_t)blockIdx.y * R, c0 + (int64_t)blockIdx.x * C);
}

// Mirror the strict lower triangle of rows [r0, r1): V[i][j] = V[j][i], j < i,
// through 32 x 32 shared-memory tiles (coalesced on both sides).
template <typename T>
__device__ __forceinline__ void mirror_tile(T *V, int64_t ld, int64_t r0, int64_t r1, int64_t bi, int64_t bj)
{
    __shared__ T tile[32][33];
    if (bj > bi) return;
    const int tx = threadIdx.x, ty = threadIdx.y;
    // load source block rows bj.., cols bi.. (upper part)
    for (int k = ty; k < 32; k += 8) {
        const int64_t sr = bj + k, sc = bi + tx;
        tile[k][tx] = (sr < r1 && sc < r1) ? V[sr * ld + sc] : T();
    }
    __syncthreads();
    for (int k = ty; k < 32; k += 8) {
        const int64_t i = bi + k, j = bj + tx;
        if (i >= r0 && i < r1 && j < i) V[i * ld + j] = tile[tx][k];
    }
}

template <typename T>
__global__ void k_mirror(T *V, int64_t ld, int64_t r0, int64_t r1)
{
    // destination row tile, destination column tile
    mirror_tile<T>(V, ld, r0, r1, (int64_t)blockIdx.y * 32 + (r0 / 32) * 32, (int64_t)blockIdx.x * 32);
}

// ------------------------------------------------------------------ near field
struct Tri {
    double p[3][3];
};

__device__ __forceinline__ double inv_norm3(double x, double y, double z)
{
    return rsqrt(x * x + y * y + z * z);
}

// The near-field quadratures below return one thread's share of the sum: thread sub of
// a group of kNearGroup takes every kNearGroup-th index of the outermost loop, and the
// group's shares are added in a fixed order before the constant factor is applied.
constexpr int kNearGroup = 4;

// Identical panels: (1/6) sum over the 6 hexagon sectors of int_0^1 1/|J w(eta)|.
__device__ double ss_identical(const Tri &P, int n, int sub)
{
    const double *gx = c_glx[n], *gw = c_glw[n];
    const double J1[3] = {P.p[1][0] - P.p[0][0], P.p[1][1] - P.p[0][1], P.p[1][2] - P.p[0][2]};
    const double J2[3] = {P.p[2][0] - P.p[1][0], P.p[2][1] - P.p[1][1], P.p[2][2] - P.p[1][2]};
    const double H[7][2] = {{1, 0}, {1, 1}, {0, 1}, {-1, 0}, {-1, -1}, {0, -1}, {1, 0}};
    double s = 0.0;
    for (int k = sub; k < 6; k += kNearGroup) {
        const double px = H[k][0], py = H[k][1], qx = H[k + 1][0], qy = H[k + 1][1];
        for (int g = 0; g < n; ++g) {
            const double z1 = px + gx[g] * (qx - px), z2 = py + gx[g] * (qy - py);
            s += gw[g] * inv_norm3(z1 * J1[0] + z2 * J2[0], z1 * J1[1] + z2 * J2[1], z1 * J1[2] + z2 * J2[2]);
        }
    }
    return s;  // times 1/6
}

// Common edge: P = (A,B,C), Q = (A,B,D).  x - y = xi rho (+-a e + t1 fP - t2 fQ).
__device__ double ss_edge(const Tri &P, const Tri &Q, int n, int sub)
{
    const double *gx = c_glx[n], *gw = c_glw[n];
    double e[3], fP[3], fQ[3];
    for (int c = 0; c < 3; ++c) {
        e[c] = P.p[1][c] - P.p[0][c];
        fP[c] = P.p[2][c] - P.p[1][c];
        fQ[c] = Q.p[2][c] - Q.p[1][c];
    }
    double s = 0.0;
    for (int iu = sub; iu < n; iu += kNearGroup)
        for (int iv = 0; iv < n; ++iv) {
            const double u = gx[iu], v = gx[iv], w = gw[iu] * gw[iv];
            // sub-region a: (own, a, other) = (1, u(1-v), uv), weight u
            // sub-region b: (own, a, other) = (u, 1-v, v),    weight 1
            const double oa = 1.0, aa = u * (1.0 - v), ha = u * v;
            const double ob = u, ab = 1.0 - v, hb = v;
            double t = 0.0;
            // region 1 (s1 = xi): vec = a e + own fP - other fQ
            t += u * inv_norm3(aa * e[0] + oa * fP[0] - ha * fQ[0], aa * e[1] + oa * fP[1] - ha * fQ[1],
                               aa * e[2] + oa * fP[2] - ha * fQ[2]);
            t += inv_norm3(ab * e[0] + ob * fP[0] - hb * fQ[0], ab * e[1] + ob * fP[1] - hb * fQ[1],
                           ab * e[2] + ob * fP[2] - hb * fQ[2]);
            // region 2 (s2 = xi): vec = -a e + other fP - own fQ
            t += u * inv_norm3(-aa * e[0] + ha * fP[0] - oa * fQ[0], -aa * e[1] + ha * fP[1] - oa * fQ[1],
                               -aa * e[2] + ha * fP[2] - oa * fQ[2]);
            t += inv_norm3(-ab * e[0] + hb * fP[0] - ob * fQ[0], -ab * e[1] + hb * fP[1] - ob * fQ[1],
                           -ab * e[2] + hb * fP[2] - ob * fQ[2]);
            s += w * t;
        }
    return s;  // times 1/6
}

// Common vertex: P = (A,B,C), Q = (A,D,E).  Regions x = (1,e1), y = e2 (1,e3) and
// x = e2 (1,e1), y = (1,e3), weight e2.
__device__ double ss_vertex(const Tri &P, const Tri &Q, int n, int sub)
{
    const double *gx = c_glx[n], *gw = c_glw[n];
    double a1[3], a2[3], b1[3], b2[3];
    for (int c = 0; c < 3; ++c) {
        a1[c] = P.p[1][c] - P.p[0][c];
        a2[c] = P.p[2][c] - P.p[1][c];
        b1[c] = Q.p[1][c] - Q.p[0][c];
        b2[c] = Q.p[2][c] - Q.p[1][c];
    }
    double s = 0.0;
    for (int i1 = sub; i1 < n; i1 += kNearGroup) {
        double xa[3];
        for (int c = 0; c < 3; ++c) xa[c] = a1[c] + gx[i1] * a2[c];
        for (int i3 = 0; i3 < n; ++i3) {
            double yb[3];
            for (int c = 0; c < 3; ++c) yb[c] = b1[c] + gx[i3] * b2[c];
            double t = 0.0;
            for (int i2 = 0; i2 < n; ++i2) {
                const double e2 = gx[i2];
                const double r1 = inv_norm3(xa[0] - e2 * yb[0], xa[1] - e2 * yb[1], xa[2] - e2 * yb[2]);
                const double r2 = inv_norm3(e2 * xa[0] - yb[0], e2 * xa[1] - yb[1], e2 * xa[2] - yb[2]);
                t += gw[i2] * e2 * (r1 + r2);
            }
            s += gw[i1] * gw[i3] * t;
        }
    }
    return s;  // times 1/3
}

__device__ __forceinline__ void load_tri(const double *verts, const int32_t *v, Tri &T)
{
    for (int k = 0; k < 3; ++k)
        for (int c = 0; c < 3; ++c) T.p[k][c] = verts[3 * (int64_t)v[k] + c];
}

// kind 0: identical pairs i = j = K + idx; 1: common-vertex list; 2: common-edge list.
// Pairs (i < j) with j < K are skipped (their entries are reused).  Called by every
// thread of a warp (valid false for the padding): the kNearGroup threads of a pair each
// integrate their share, the shares are summed in a fixed order ((s0 + s1) + (s2 + s3))
// by shuffles, and the group's first thread writes the entry.
template <typename T>
__device__ __forceinline__ void near_entry(const double *__restrict__ verts, const int32_t *__restrict__ tris,
                                           const double *__restrict__ area, const int32_t *__restrict__ pairs,
                                           int64_t idx, int kind, int64_t K, int n, T *V, int64_t ld, bool valid)
{
    static_assert(kNearGroup == 4, "the group sum below adds four shares");
    const int sub = (int)(threadIdx.x % kNearGroup);
    int64_t i = 0, j = 0;
    bool write = false;
    double I = 0.0;
    if (valid) {
        if (kind == 0) {
            i = j = K + idx;
        } else {
            i = pairs[2 * idx];
            j = pairs[2 * idx + 1];
        }
        write = kind == 0 || j >= K;
    }
    if (write) {
        const int32_t *ti = tris + 3 * i, *tj = tris + 3 * j;
        if (kind == 0) {
            Tri P;
            load_tri(verts, ti, P);
            I = ss_identical(P, n, sub);
        } else if (kind == 2) {
            // (u, v) = the shared vertices in the order they appear in triangle i
            int32_t u = -1, v = -1, ci = -1, cj = -1;
            for (int k = 0; k < 3; ++k) {
                const bool in = (ti[k] == tj[0] || ti[k] == tj[1] || ti[k] == tj[2]);
                if (in) {
                    if (u < 0) u = ti[k];
                    else v = ti[k];
                } else {
                    ci = ti[k];
                }
            }
            for (int k = 0; k < 3; ++k)
                if (tj[k] != u && tj[k] != v) cj = tj[k];
            const int32_t pi[3] = {u, v, ci}, pj[3] = {u, v, cj};
            Tri P, Q;
            load_tri(verts, pi, P);
            load_tri(verts, pj, Q);
            I = ss_edge(P, Q, n, sub);
        } else {
            int ki = 0, kj = 0;
            for (int a = 0; a < 3; ++a)
                for (int b = 0; b < 3; ++b)
                    if (ti[a] == tj[b]) {
                        ki = a;
                        kj = b;
                    }
            const int32_t pi[3] = {ti[ki], ti[(ki + 1) % 3], ti[(ki + 2) % 3]};
            const int32_t pj[3] = {tj[kj], tj[(kj + 1) % 3], tj[(kj + 2) % 3]};
            Tri P, Q;
            load_tri(verts, pi, P);
            load_tri(verts, pj, Q);
            I = ss_vertex(P, Q, n, sub);
        }
    }
    I += __shfl_xor_sync(0xffffffffu, I, 1);
    I += __shfl_xor_sync(0xffffffffu, I, 2);
    if (write && sub == 0) {
        I = kind == 1 ? I / 3.0 : I / 6.0;
        const double v = 4.0 * area[i] * area[j] * I * kInv4Pi;
        const T e = Elem<T>::from_double(v);
        V[i * ld + j] = e;
        if (i != j) V[j * ld + i] = e;
    }
}

// All touching pairs of an assembly in one launch, kNearGroup threads per pair: the
// common-vertex pairs (the longest quadrature) first, then the common-edge pairs, then
// the identical pairs of the new triangles, so that the three lists overlap instead of
// running one after another.  Each list starts on a warp boundary (its pair count
// rounded up to kNearPairsPerWarp), so that no warp runs two of the quadratures.
constexpr int kNearPairsPerWarp = 32 / kNearGroup;
inline int64_t near_pad(int64_t n) { return (n + kNearPairsPerWarp - 1) / kNearPairsPerWarp * kNearPairsPerWarp; }

template <typename T>
__global__ void k_near(const double *__restrict__ verts, const int32_t *__restrict__ tris,
                       const double *__restrict__ area, const int32_t *__restrict__ vert_pairs, int64_t n_vert,
                       const int32_t *__restrict__ edge_pairs, int64_t n_edge, int64_t n_ident, int64_t K, int n,
                       T *V, int64_t ld)
{
    const int64_t nvp = (n_vert + kNearPairsPerWarp - 1) / kNearPairsPerWarp * kNearPairsPerWarp;
    const int64_t nep = (n_edge + kNearPairsPerWarp - 1) / kNearPairsPerWarp * kNearPairsPerWarp;
    int64_t idx = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kNearGroup;
    if (idx < nvp) {
        near_entry<T>(verts, tris, area, vert_pairs, idx, 1, K, n, V, ld, idx < n_vert);
    } else if ((idx -= nvp) < nep) {
        near_entry<T>(verts, tris, area, edge_pairs, idx, 2, K, n, V, ld, idx < n_edge);
    } else {
        idx -= nep;
        near_entry<T>(verts, tris, area, nullptr, idx, 0, K, n, V, ld, idx < n_ident);
    }
}

// ------------------------------------------------------------------ reuse and diagonal
// V'[i][j] = Vc[parent[i]][parent[j]] for i, j < K (unrefined triangles), by 64 x 64
// tiles: CTA (bx, by) copies rows 64 by.. and columns 64 bx.., thread t column t % 64 and
// the 16 rows 16 (t / 64).. of the tile (16 independent loads in flight; a warp reads
// 32 nearly consecutive entries of a coarse row, the kept triangles keeping their
// order).  upper: entries i <= j only (tiles below the diagonal return at once; the
// kept triangles keep their order, so these come from the coarse operator's upper
// triangle).
template <typename T>
__global__ void __launch_bounds__(256) k_gather_kept(const T *__restrict__ Vc, int64_t ldc,
                                                     const int32_t *__restrict__ parent, int64_t K,
                                                     T *__restrict__ V, int64_t ld, int upper)
{
    if (upper && blockIdx.y > blockIdx.x) return;
    const int64_t j = (int64_t)blockIdx.x * 64 + (threadIdx.x & 63);
    const int64_t i0 = (int64_t)blockIdx.y * 64 + 16 * (threadIdx.x >> 6);
    if (j >= K) return;
    const int64_t pj = parent[j];
    const int64_t iend = upper ? (j + 1 < K ? j + 1 : K) : K;
    T v[16];
#pragma unroll
    for (int r = 0; r < 16; ++r)
        if (i0 + r < iend) v[r] = Vc[(int64_t)parent[i0 + r] * ldc + pj];
#pragma unroll
    for (int r = 0; r < 16; ++r)
        if (i0 + r < iend) V[(i0 + r) * ld + j] = v[r];
}

// Mirror of the diagonal 64 x 64 blocks only: 32 x 32 tiles (2D, 2D), (2D+1, 2D),
// (2D+1, 2D+1) of block D, item t = 3 D + (0, 1, 2).
template <typename T>
__global__ void k_mirror_diag(T *V, int64_t ld, int64_t N)
{
    const int64_t t = blockIdx.x, D = t / 3, r = t % 3;
    const int64_t bi = 2 * D + (r > 0 ? 1 : 0), bj = 2 * D + (r == 2 ? 1 : 0);
    mirror_tile<T>(V, ld, 0, N, 32 * bi, 32 * bj);
}

template <typename T>
__global__ void k_diag(const T *V, int64_t ld, int64_t N, double *d)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) d[i] = Elem<T>::to_double(V[i * ld + i]);
}

// ------------------------------------------------------------------ drivers
template <typename T, int R, int C, int MB = 0>
static void far_kernel(bem_operator *op, dim3 grid, int64_t r0, int64_t r1, int64_t c0, int64_t c1)
{
    bem_mesh *m = op->mesh;
    cudaStream_t s = m->ctx->stream;
    if (op->precision == BEM_PREC_F64)
        k_far_f64<R, C><<<grid, C, 0, s>>>(m->q64, m->cent, (double *)op->V, op->ld, r0, r1, c0, c1);
    else if (op->precision == BEM_PREC_DF64)
    {
        if constexpr (MB > 0)
            k_far_df_s<R, C, MB><<<grid, C, far_df_smem<C>(), s>>>(m->qdf, (float2 *)op->V, op->ld, r0, r1,
                                                                   c0, c1);
        else
            k_far_df<R, C><<<grid, C, far_df_smem<C>(), s>>>(m->qdf, (float2 *)op->V, op->ld, r0, r1, c0, c1);
    }
    else
        k_far_f32<R, C><<<grid, C, 0, s>>>(m->q32, m->cent, (float *)op->V, op->ld, r0, r1, c0, c1);
}

// Far-field entries i <= j of the block [r0, r1) x [c0, c1) with tile variant v.
template <typename T>
static bem_status launch_far(bem_operator *op, int v, int64_t r0, int64_t r1, int64_t c0, int64_t c1,
                             bool profile = true)
{
    if (r1 <= r0 || c1 <= c0) return BEM_OK;
    bem_mesh *m = op->mesh;
    bem_ctx *ctx = m->ctx;
    const int R = kFarTiles[v].rows, C = kFarTiles[v].cols;
    const int64_t gx = (c1 - c0 + C - 1) / C;
    const int64_t gy = (r1 - r0 + R - 1) / R;
    if (gy > 65535) {
        // split rows into chunks that fit the grid's y limit
        for (int64_t rs = r0; rs < r1; rs += 65535LL * R) {
            const int64_t re = rs + 65535LL * R < r1 ? rs + 65535LL * R : r1;
            bem_status st = launch_far<T>(op, v, rs, re, c0, c1, profile);
            if (st) return st;
        }
        return BEM_OK;
    }
    dim3 grid((unsigned)gx, (unsigned)gy);
    // entries with i <= j in the block: whole rows above the columns' first, then a triangle
    const int64_t full = (r1 < c0 ? r1 : c0) - r0, t0 = r0 > c0 ? r0 : c0, t1 = r1 < c1 ? r1 : c1;
    const double units = (full > 0 ? (double)full * (double)(c1 - c0) : 0.0) +
                         (t1 > t0 ? 0.5 * (double)(t1 - t0) * (double)((c1 - t0) + (c1 - t1 + 1)) : 0.0);
    const int prof = profile ? prof_start(ctx, BEM_KERNEL_FAR, units) : -1;
    switch (v) {
    case 0: far_kernel<T, 32, 256>(op, grid, r0, r1, c0, c1); break;
    case 1: far_kernel<T, 16, 256>(op, grid, r0, r1, c0, c1); break;
    case 2: far_kernel<T, 64, 256>(op, grid, r0, r1, c0, c1); break;
    case 3: far_kernel<T, 8, 128>(op, grid, r0, r1, c0, c1); break;
    case 4: far_kernel<T, 16, 128>(op, grid, r0, r1, c0, c1); break;
    case 5: far_kernel<T, 32, 128>(op, grid, r0, r1, c0, c1); break;
    case 6: far_kernel<T, 8, 128, 5>(op, grid, r0, r1, c0, c1); break;
    case 7: far_kernel<T, 16, 128, 5>(op, grid, r0, r1, c0, c1); break;
    case 8: far_kernel<T, 32, 128, 5>(op, grid, r0, r1, c0, c1); break;
    case 9: far_kernel<T, 4, 128, 5>(op, grid, r0, r1, c0, c1); break;
    case 10: far_kernel<T, 8, 64, 10>(op, grid, r0, r1, c0, c1); break;
    case 11: far_kernel<T, 4, 64, 10>(op, grid, r0, r1, c0, c1); break;
    case 12: far_kernel<T, 2, 64, 10>(op, grid, r0, r1, c0, c1); break;
    default: far_kernel<T, 1, 64, 10>(op, grid, r0, r1, c0, c1); break;
    }
    BEM_COUNT(ctx);
    if (profile) prof_stop(ctx, prof);
    BEM_CK_LAUNCH(ctx);
    return BEM_OK;
}

// Size classes of the tile cache: N < 1,024, < 4,096, < 16,384, larger.
static int far_bucket(int64_t N) { return N < 1024 ? 0 : N < 4096 ? 1 : N < 16384 ? 2 : 3; }

// The tile variant of this assembly: the requested one, else the context's choice
// for (precision, size class), timed now on this assembly's own far-field block if
// the class has none yet -- every variant once to load its module, then once timed,
// the fastest kept.  No timing while the stream is being captured into a graph (the
// variant is then the cached one, or variant 0).
template <typename T>
static bem_status far_variant(bem_operator *op, int64_t K, int64_t N, int *v_out)
{
    bem_ctx *ctx = op->mesh->ctx;
    if (op->tile > 0) {
        *v_out = op->tile - 1;
        return BEM_OK;
    }
    int8_t &slot = ctx->far_tile[op->precision][far_bucket(N)];
    *v_out = slot >= 0 ? slot : 0;
    if (slot >= 0 || N - K <= 0) return BEM_OK;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    BEM_CK(ctx, cudaStreamIsCapturing(ctx->stream, &cs));
    if (cs != cudaStreamCaptureStatusNone) return BEM_OK;
    float best = 0.0f;
    int bv = 0;
    for (int pass = 0; pass < 2; ++pass)
        for (int v = 0; v < kFarTileVariants; ++v) {
            BEM_CK(ctx, cudaEventRecord(ctx->ev[4], ctx->stream));
            bem_status st = launch_far<T>(op, v, K, N, K, N, false);
            if (st) return st;
            BEM_CK(ctx, cudaEventRecord(ctx->ev[5], ctx->stream));
            BEM_CK(ctx, cudaEventSynchronize(ctx->ev[5]));
            float ms = 0.0f;
            BEM_CK(ctx, cudaEventElapsedTime(&ms, ctx->ev[4], ctx->ev[5]));
            if (pass == 1 && (v == 0 || ms < best)) {
                best = ms;
                bv = v;
            }
        }
    slot = (int8_t)bv;
    *v_out = bv;
    return BEM_OK;
}

// A batch lists its tiles: below kFarBatchArea entries each the list would outgrow what is
// set aside for it, so only meshes of the smallest class (N < 1,024) take such tiles there.
constexpr int kFarBatchArea = 512;
int far_batch_variant(const bem_ctx *ctx, int precision, int64_t N)
{
    const int v = std::max<int>(0, ctx->far_tile[precision][far_bucket(N)]);
    return far_bucket(N) > 0 && kFarTiles[v].rows * kFarTiles[v].cols < kFarBatchArea ? 6 : v;
}

// Tiles of variant v that reach the diagonal of N rows or above: K column tiles; the rows of
// column tile m take K - m of them.
static int64_t far_items(int v, int64_t N)
{
    const int64_t R = kFarTiles[v].rows, C = kFarTiles[v].cols, K = (N + C - 1) / C;
    return C / R * (K * (K + 1) / 2 - 1) + (N - (K - 1) * C + R - 1) / R;
}

double far_batch_items_bound(int tile, int64_t N)
{
    if (tile > 0) return (double)far_items(tile - 1, N);
    int64_t most = 0;
    for (int v = 0; v < kFarTileVariants; ++v)
        if (far_bucket(N) == 0 || kFarTiles[v].rows * kFarTiles[v].cols >= kFarBatchArea)
            most = std::max(most, far_items(v, N));
    return (double)most;
}

bem_status far_tune(bem_operator *op)
{
    int v = 0;
    const int64_t N = op->mesh->N;
    if (op->precision == BEM_PREC_F64) return far_variant<double>(op, 0, N, &v);
    if (op->precision == BEM_PREC_DF64) return far_variant<float2>(op, 0, N, &v);
    return far_variant<float>(op, 0, N, &v);
}

template <typename T>
static bem_status launch_mirror(bem_operator *op, int64_t r0, int64_t r1)
{
    if (r1 <= r0) return BEM_OK;
    bem_ctx *ctx = op->mesh->ctx;
    const int64_t t0 = r0 / 32, t1 = (r1 + 31) / 32;
    for (int64_t ts = t0; ts < t1; ts += 65535) {
        const int64_t te = ts + 65535 < t1 ? ts + 65535 : t1;
        dim3 grid((unsigned)te, (unsigned)(te - ts));
        k_mirror<T><<<grid, dim3(32, 8), 0, ctx->stream>>>((T *)op->V, op->ld, ts * 32 > r0 ? ts * 32 : r0,
                                                           te * 32 < r1 ? te * 32 : r1); BEM_COUNT(ctx);
        BEM_CK_LAUNCH(ctx);
    }
    return BEM_OK;
}

template <typename T>
static bem_status launch_near(bem_operator *op, int64_t K)
{
    bem_mesh *m = op->mesh;
    bem_ctx *ctx = m->ctx;
    const int n = op->ss_order;
    const int prof = prof_start(ctx, BEM_KERNEL_NEAR, (double)(m->N - K + m->n_vert_pairs + m->n_edge_pairs));
    const int64_t n_ident = m->N > K ? m->N - K : 0;
    const int64_t total = near_pad(m->n_vert_pairs) + near_pad(m->n_edge_pairs) + n_ident;
    if (total > 0) {
        k_near<T><<<nblk(total * kNearGroup, 128), 128, 0, ctx->stream>>>(m->verts, m->tris, m->area, m->vert_pairs,
                                                             m->n_vert_pairs, m->edge_pairs, m->n_edge_pairs, n_ident,
                                                             K, n, (T *)op->V, op->ld);
        BEM_COUNT(ctx);
    }
    prof_stop(ctx, prof);
    BEM_CK_LAUNCH(ctx);
    return BEM_OK;
}

// Zero the padding columns [N, ld) of every row (the far field, the mirror, the near
// field and the reused block write every entry of [0, N) x [0, N)).
template <typename T>
__global__ void k_zero_padding(T *V, int64_t ld, int64_t N)
{
    const int64_t i = blockIdx.x, j = N + threadIdx.x;
    if (i < N && j < ld) V[i * ld + j] = T();
}

template <typename T>
static bem_status launch_mirror_diag(bem_operator *op)
{
    bem_ctx *ctx = op->mesh->ctx;
    const int64_t T32 = (op->N + 31) / 32, items = 3 * (T32 / 2) + (T32 % 2);
    if (items > 0) {
        k_mirror_diag<T><<<(unsigned)items, dim3(32, 8), 0, ctx->stream>>>((T *)op->V, op->ld, op->N); BEM_COUNT(ctx);
        BEM_CK_LAUNCH(ctx);
    }
    return BEM_OK;
}

// upper: fill only the upper triangle and the diagonal blocks (op->upper_only)
template <typename T>
static bem_status assemble_t(bem_operator *op, const bem_operator *coarse, bool upper)
{
    bem_mesh *m = op->mesh;
    bem_ctx *ctx = m->ctx;
    const int64_t N = m->N;
    if (op->ld > N) {
        k_zero_padding<T><<<(unsigned)N, 64, 0, ctx->stream>>>((T *)op->V, op->ld, N); BEM_COUNT(ctx);
    }
    bem_status st;
    int64_t K = 0;
    if (coarse) {
        K = m->n_kept;
        if (K > 0) {
            dim3 grid(nblk(K, 64), nblk(K, 64));
            k_gather_kept<T><<<grid, 256, 0, ctx->stream>>>((const T *)coarse->V, coarse->ld, m->parent, K,
                                                            (T *)op->V, op->ld,
                                                            (upper || coarse->upper_only) ? 1 : 0); BEM_COUNT(ctx);
            BEM_CK_LAUNCH(ctx);
        }
    }
    int v = 0;
    if ((st = far_variant<T>(op, K, N, &v))) return st;
    if (K > 0 && (st = launch_far<T>(op, v, 0, K, K, N))) return st;
    if ((st = launch_far<T>(op, v, K, N, K, N))) return st;
    if (upper) {
        if ((st = launch_mirror_diag<T>(op))) return st;
    } else {
        // a coarse operator with its upper triangle alone gave the kept block's upper half
        const int64_t m0 = (coarse && coarse->upper_only) ? 0 : (K > 0 ? K : 0);
        if ((st = launch_mirror<T>(op, m0, N))) return st;
    }
    op->upper_only = upper ? 1 : 0;
    if ((st = launch_near<T>(op, K))) return st;
    k_diag<T><<<nblk(N, 256), 256, 0, ctx->stream>>>((const T *)op->V, op->ld, N, op->diag); BEM_COUNT(ctx);
    BEM_CK_LAUNCH(ctx);
    return BEM_OK;
}

// ------------------------------------------------------------------ batched assembly
// The assembly of every operator of a batch wave in one launch per phase: the far
// field over a work list of (problem, row tile, column tile) items, the mirror over
// the 32 x 32 tile pairs of all problems, the near field over the concatenated
// identical / common-vertex / common-edge lists.  Every entry is computed by the same
// device code as the per-operator kernels, so the operators are bit-identical to
// bem_assemble_V's.

// Problem p with prefix[p] <= k < prefix[p + 1] (prefix: P + 1 ascending entries).
__device__ __forceinline__ int batch_find(const int64_t *__restrict__ prefix, int P, int64_t k)
{
    int lo = 0, hi = P - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= k)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

template <typename T, int R, int C, int MB>
__global__ void __launch_bounds__(C, (MB > 0 ? MB : 1))
    k_far_batch(const BatchAsmProb *__restrict__ prob, const int4 *__restrict__ items)
{
    const int4 it = items[blockIdx.x];
    const BatchAsmProb *pb = prob + it.x;
    const int64_t N = pb->N, ld = pb->ld;
    if constexpr (std::is_same<T, double>::value)
        far_f64_body<R, C>(pb->q64, pb->cent, (double *)pb->V, ld, N, N, it.y, it.z);
    else if constexpr (std::is_same<T, float2>::value)
        far_df_body<R, C>(pb->qdf, (float2 *)pb->V, ld, N, N, it.y, it.z);
    else
        far_f32_body<R, C>(pb->q32, pb->cent, (float *)pb->V, ld, N, N, it.y, it.z);
}

// Tile pair t of a problem: row tile bi >= column tile bj, t = bi (bi + 1) / 2 + bj.
// A batch's operators are read only through their upper triangle (the packed tiles, the
// DF64 tile products, the symmetric reads of the block preconditioner), so only the
// 64 x 64 diagonal blocks, whose lower halves those tiles include, are mirrored: 32 x 32
// tiles (2D, 2D), (2D+1, 2D), (2D+1, 2D+1) of block D, item t = 3 D + (0, 1, 2).
template <typename T>
__global__ void k_mirror_batch(const BatchAsmProb *__restrict__ prob, const int64_t *__restrict__ pref, int P)
{
    const int64_t k = blockIdx.x;
    const int p = batch_find(pref, P, k);
    const int64_t t = k - pref[p];
    const int64_t D = t / 3, r = t % 3;
    const int64_t bi = 2 * D + (r > 0 ? 1 : 0), bj = 2 * D + (r == 2 ? 1 : 0);
    const BatchAsmProb *pb = prob + p;
    mirror_tile<T>((T *)pb->V, pb->ld, 0, pb->N, 32 * bi, 32 * bj);
}

// Item k of a problem: identical pairs [0, N), common-vertex pairs, common-edge pairs.
// kNearGroup threads per item (every thread of a warp reaches near_entry's group sum).
template <typename T>
__global__ void k_near_batch(const BatchAsmProb *__restrict__ prob, const int64_t *__restrict__ pref, int P,
                             int64_t total, int n)
{
    const int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kNearGroup;
    const bool valid = k < total;
    const int p = batch_find(pref, P, valid ? k : total - 1);
    const BatchAsmProb *pb = prob + p;
    int64_t idx = (valid ? k : total - 1) - pref[p];
    const int64_t N = pb->N;
    if (idx < N) {
        near_entry<T>(pb->verts, pb->tris, pb->area, nullptr, idx, 0, 0, n, (T *)pb->V, pb->ld, valid);
    } else if ((idx -= N) < pb->n_vert) {
        near_entry<T>(pb->verts, pb->tris, pb->area, pb->vert_pairs, idx, 1, 0, n, (T *)pb->V, pb->ld, valid);
    } else {
        idx -= pb->n_vert;
        near_entry<T>(pb->verts, pb->tris, pb->area, pb->edge_pairs, idx, 2, 0, n, (T *)pb->V, pb->ld, valid);
    }
}

int far_variant_rows(int v) { return kFarTiles[v].rows; }
int far_variant_cols(int v) { return kFarTiles[v].cols; }

void batch_far_items(int v, int p, int64_t N, std::vector<int4> &items)
{
    const int64_t R = kFarTiles[v].rows, C = kFarTiles[v].cols;
    for (int64_t i0 = 0; i0 < N; i0 += R)
        for (int64_t c = (i0 / C) * C; c < N; c += C)  // tiles reaching the diagonal or above
            if (i0 <= c + C - 1) items.push_back(make_int4(p, (int)i0, (int)c, 0));
}

template <typename T, int R, int C, int MB = 0>
static void far_batch_launch(const BatchAsm &b, cudaStream_t s)
{
    const size_t smem = std::is_same<T, float2>::value ? far_df_smem<C>() : 0;
    k_far_batch<T, R, C, MB><<<(unsigned)b.n_far, C, smem, s>>>(b.prob, b.far_items);
}

// Event record that also fires when a captured graph replays (an external event node
// while the stream is being captured; a plain record otherwise).
bem_status record_timing_event(bem_ctx *ctx, cudaEvent_t e)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    BEM_CK(ctx, cudaStreamIsCapturing(ctx->stream, &cs));
    BEM_CK(ctx, cudaEventRecordWithFlags(e, ctx->stream,
                                         cs == cudaStreamCaptureStatusActive ? cudaEventRecordExternal
                                                                             : cudaEventRecordDefault));
    return BEM_OK;
}

template <typename T>
static bem_status batch_assemble_t(bem_ctx *ctx, const BatchAsm &b, cudaEvent_t *ev)
{
    cudaStream_t s = ctx->stream;
    bem_status st;
    if (ev && (st = record_timing_event(ctx, ev[0]))) return st;
    if (b.n_far > 0) {
        switch (b.variant) {
        case 0: far_batch_launch<T, 32, 256>(b, s); break;
        case 1: far_batch_launch<T, 16, 256>(b, s); break;
        case 2: far_batch_launch<T, 64, 256>(b, s); break;
        case 3: far_batch_launch<T, 8, 128>(b, s); break;
        case 4: far_batch_launch<T, 16, 128>(b, s); break;
        case 5: far_batch_launch<T, 32, 128>(b, s); break;
        case 6: far_batch_launch<T, 8, 128, 5>(b, s); break;
        case 7: far_batch_launch<T, 16, 128, 5>(b, s); break;
        case 8: far_batch_launch<T, 32, 128, 5>(b, s); break;
        case 9: far_batch_launch<T, 4, 128, 5>(b, s); break;
        case 10: far_batch_launch<T, 8, 64, 10>(b, s); break;
        case 11: far_batch_launch<T, 4, 64, 10>(b, s); break;
        case 12: far_batch_launch<T, 2, 64, 10>(b, s); break;
        default: far_batch_launch<T, 1, 64, 10>(b, s); break;
        }
        BEM_COUNT(ctx);
        BEM_CK_LAUNCH(ctx);
    }
    if (ev && (st = record_timing_event(ctx, ev[1]))) return st;
    if (b.n_mirror > 0) {
        k_mirror_batch<T><<<(unsigned)b.n_mirror, dim3(32, 8), 0, s>>>(b.prob, b.mirror_pref, b.P); BEM_COUNT(ctx);
        BEM_CK_LAUNCH(ctx);
    }
    if (ev && (st = record_timing_event(ctx, ev[2]))) return st;
    if (b.n_near > 0) {
        k_near_batch<T><<<nblk(b.n_near * kNearGroup, 128), 128, 0, s>>>(b.prob, b.near_pref, b.P, b.n_near,
                                                                          b.ss_order);
        BEM_COUNT(ctx);
        BEM_CK_LAUNCH(ctx);
    }
    if (ev && (st = record_timing_event(ctx, ev[3]))) return st;
    return BEM_OK;
}

bem_status batch_assemble(bem_ctx *ctx, const BatchAsm &b, cudaEvent_t *ev)
{
    if (b.precision == BEM_PREC_F64) return batch_assemble_t<double>(ctx, b, ev);
    if (b.precision == BEM_PREC_DF64) return batch_assemble_t<float2>(ctx, b, ev);
    return batch_assemble_t<float>(ctx, b, ev);
}

bem_status assembly_prepare(bem_ctx *ctx) { return assembly_constants(ctx); }

bem_status gauss_legendre_upload(int n)
{
    (void)n;
    return BEM_OK;
}

bem_status assemble_full(bem_operator *op, bool upper_only)
{
    bem_status st = assembly_constants(op->mesh->ctx);
    if (st) return st;
    if (op->precision == BEM_PREC_F64) return assemble_t<double>(op, nullptr, upper_only);
    if (op->precision == BEM_PREC_DF64) return assemble_t<float2>(op, nullptr, upper_only);
    return assemble_t<float>(op, nullptr, upper_only);
}

bem_status assemble_update(bem_operator *op, const bem_operator *coarse, bool upper_only)
{
    bem_status st = assembly_constants(op->mesh->ctx);
    if (st) return st;
    if (op->precision == BEM_PREC_F64) return assemble_t<double>(op, coarse, upper_only);
    if (op->precision == BEM_PREC_DF64) return assemble_t<float2>(op, coarse, upper_only);
    return assemble_t<float>(op, coarse, upper_only);
}

// The lower triangle of an upper-only operator, mirrored from the upper one (bit-
// identical copies) before a reader of whole rows.
bem_status ensure_full(bem_operator *op)
{
    if (!op || !op->upper_only) return BEM_OK;
    bem_status st;
    if (op->precision == BEM_PREC_F64) st = launch_mirror<double>(op, 0, op->N);
    else if (op->precision == BEM_PREC_DF64) st = launch_mirror<float2>(op, 0, op->N);
    else st = launch_mirror<float>(op, 0, op->N);
    if (!st) op->upper_only = 0;
    return st;
}

bem_status operator_diag(bem_operator *op)
{
    bem_ctx *ctx = op->mesh->ctx;
    if (op->precision == BEM_PREC_F64)
        { k_diag<double><<<nblk(op->N, 256), 256, 0, ctx->stream>>>((const double *)op->V, op->ld, op->N, op->diag); BEM_COUNT(ctx); }
    else if (op->precision == BEM_PREC_DF64)
        { k_diag<float2><<<nblk(op->N, 256), 256, 0, ctx->stream>>>((const float2 *)op->V, op->ld, op->N, op->diag); BEM_COUNT(ctx); }
    else
        { k_diag<float><<<nblk(op->N, 256), 256, 0, ctx->stream>>>((const float *)op->V, op->ld, op->N, op->diag); BEM_COUNT(ctx); }
    BEM_CK_LAUNCH(ctx);
    return BEM_OK;
}

}  // namespace bem
