// near64.cuh -- device code shared by the FP64 form's kernels (lmfmm_apply.cu) and
// their double-float near field (lmfmm_near_df.cu): box geometries, the density
// exponent and the free-space kernel.
#pragma once
#include "df.cuh"
#include "internal.h"

// Box geometry of a launch: block i works on box id(i), whose centre and width
// come from centre().
struct GridLeaves { // uniform tree: leaf i of the leaf lattice
    LeafGeom g;
    __device__ int64_t id(int64_t i) const { return i; }
    __device__ void centre(int64_t b, double *cx, double *cy, double *w) const
    {
        leaf_centre(g, b, cx, cy);
        *w = g.w;
    }
};
struct EdgeRowLeaves { // uniform tree: the leaves of the top row, then (nrow > 1) of the bottom row
    LeafGeom g;
    int64_t nrow;
    __device__ int64_t id(int64_t i) const { return ((nrow == 1 || i < g.ncol) ? 0 : nrow - 1) * g.ncol + i % g.ncol; }
    __device__ void centre(int64_t b, double *cx, double *cy, double *w) const
    {
        leaf_centre(g, b, cx, cy);
        *w = g.w;
    }
};
struct ListBoxes { // adaptive tree: box ids[i], centres and widths from arrays
    const int32_t *ids;
    const double *bx, *by, *bw;
    __device__ int64_t id(int64_t i) const { return ids[i]; }
    __device__ void centre(int64_t b, double *cx, double *cy, double *w) const
    {
        *cx = bx[b];
        *cy = by[b];
        *w = bw[b];
    }
};

struct GridParents { // uniform tree: parent i of a level with ncol columns; children one level down
    int64_t ncol;
    __device__ int64_t parent(int64_t i) const { return i; }
    __device__ int64_t child(int64_t b, int pos) const
    {
        const int64_t r = b / ncol, c = b % ncol;
        return (2 * r + (pos >> 1)) * (2 * ncol) + 2 * c + (pos & 1);
    }
};
struct ListParents { // adaptive tree: parent ids[i], children from the box links
    const int32_t *ids, *kids;
    __device__ int64_t parent(int64_t i) const { return ids[i]; }
    __device__ int64_t child(int64_t b, int pos) const { return kids[4 * b + pos]; }
};


// binary exponent of a vector's densities: each vector is scaled by its own, so that its result does not
// depend on the others of the call (one exponent for all flushed a vector 2^-126 of the largest to zero)
__device__ __forceinline__ int qexp_of(const int *qexp, int v)
{
    const int e = qexp[v];
    return e < -2000 ? 0 : e; // all densities zero: no scaling
}

// ---------------------------------------------------------------------------
// Free-space kernel (i/4) H0^(1)(x) = (i/4)(J0(x) + i Y0(x)) of a near pair in
// FP64.  For x <= 2 the ascending series (Abramowitz & Stegun 9.1.12, 9.1.13),
// with z = x^2/4:
//   J0 = sum_m (-z)^m / (m!)^2,
//   Y0 = (2/pi) [(ln(x/2) + gamma) J0 - sum_{m>=1} H_m (-z)^m / (m!)^2],
// H_m the harmonic numbers, gamma Euler's constant; 14 terms leave the first
// omitted one below 2e-21 for z <= 1 (within 5e-16 of scipy's J0, Y0 on
// (0, 2]).  Horner form: 28 FMAs and one log in place of the library's j0 and
// y0 (1M FP64 strip: leaf kernel 72.0 -> 65.7 ms).  Larger x: j0, y0.
// ---------------------------------------------------------------------------
#define H0S_TERMS 14
struct H0Series {
    double cj[H0S_TERMS], cy[H0S_TERMS]; // (-1)^m / (m!)^2, -(-1)^m H_m / (m!)^2
    constexpr H0Series() : cj(), cy()
    {
        double f = 1.0, h = 0.0; // 1/(m!)^2, H_m
        for (int m = 0; m < H0S_TERMS; ++m) {
            if (m > 0) {
                f /= (double)m * (double)m;
                h += 1.0 / m;
            }
            cj[m] = (m & 1) ? -f : f;
            cy[m] = (m & 1) ? h * f : -h * f;
        }
    }
};
static __constant__ H0Series c_h0s = H0Series();
// J1 and Y1 for the target gradient (A&S 9.1.10, 9.1.11 with n = 1):
//   J1 = (x/2) sum_m (-z)^m / (m! (m+1)!),
//   Y1 = -2/(pi x) + (2/pi) ln(x/2) J1 - (x/(2 pi)) sum_m (-z)^m (psi(m+1) + psi(m+2)) / (m! (m+1)!),
// psi(m+1) = H_m - gamma; within 5e-16 of scipy's J1, Y1 on (0, 2]
struct H1Series {
    double c[H0S_TERMS], e[H0S_TERMS]; // (-1)^m / (m! (m+1)!), (-1)^m (psi(m+1) + psi(m+2)) / (m! (m+1)!)
    constexpr H1Series() : c(), e()
    {
        double f = 1.0, h = 0.0; // 1/(m! (m+1)!), H_m
        for (int m = 0; m < H0S_TERMS; ++m) {
            if (m > 0) {
                f /= (double)m * (double)(m + 1);
                h += 1.0 / m;
            }
            const double psi = (h - 0.57721566490153286061) + (h + 1.0 / (m + 1) - 0.57721566490153286061);
            c[m] = (m & 1) ? -f : f;
            e[m] = (m & 1) ? -psi * f : psi * f;
        }
    }
};
static __constant__ H1Series c_h1s = H1Series();
// (i/4) H0^(1)(x) and (i/4) H1^(1)(x) together (series for x <= 2, else the library's)
__device__ __forceinline__ void h01_free64(double x, zd *h0, zd *h1)
{
    if (x > 2.0) {
        *h0 = zd{-0.25 * y0(x), 0.25 * j0(x)};
        *h1 = zd{-0.25 * y1(x), 0.25 * j1(x)};
        return;
    }
    const double z = 0.25 * x * x;
    double j = c_h0s.cj[H0S_TERMS - 1], sy = c_h0s.cy[H0S_TERMS - 1];
    double a = c_h1s.c[H0S_TERMS - 1], b = c_h1s.e[H0S_TERMS - 1];
#pragma unroll
    for (int m = H0S_TERMS - 2; m >= 0; --m) {
        j = fma(j, z, c_h0s.cj[m]);
        sy = fma(sy, z, c_h0s.cy[m]);
        a = fma(a, z, c_h1s.c[m]);
        b = fma(b, z, c_h1s.e[m]);
    }
    const double tpi = 0.63661977236758134308, lg = log(0.5 * x);
    const double yv0 = tpi * ((lg + 0.57721566490153286061) * j + sy);
    const double jv1 = 0.5 * x * a;
    const double yv1 = -tpi / x + tpi * lg * jv1 - 0.5 * tpi * 0.5 * x * b;
    *h0 = zd{-0.25 * yv0, 0.25 * j};
    *h1 = zd{-0.25 * yv1, 0.25 * jv1};
}
__device__ __forceinline__ zd h0_free64(double x)
{
    if (x > 2.0) return zd{-0.25 * y0(x), 0.25 * j0(x)};
    const double z = 0.25 * x * x;
    double j = c_h0s.cj[H0S_TERMS - 1], sy = c_h0s.cy[H0S_TERMS - 1];
#pragma unroll
    for (int m = H0S_TERMS - 2; m >= 0; --m) {
        j = fma(j, z, c_h0s.cj[m]);
        sy = fma(sy, z, c_h0s.cy[m]);
    }
    const double y = 0.63661977236758134308 * ((log(0.5 * x) + 0.57721566490153286061) * j + sy);
    return zd{-0.25 * y, 0.25 * j};
}

// ---------------------------------------------------------------------------
// The same in double-float.  A kernel value g = g_re + i g_im is kept as (A, J), g_re =
// -A/(4 pi), g_im = J/4: A = (ln z + 2 gamma) J + 2 V, J = J0, z = (k r / 2)^2, so the constants
// are applied once per target.
// ---------------------------------------------------------------------------
#define ND_TINY 8.0779357e-28f // 2^-90: closer pairs, and z > 1, take the FP64 functions
// Series coefficients as double-floats (A&S 9.1.12, 9.1.13; H0Series of near64.cuh)
struct H0DF {
    float jh[H0S_TERMS], jl[H0S_TERMS], vh[H0S_TERMS], vl[H0S_TERMS];
    constexpr H0DF() : jh(), jl(), vh(), vl()
    {
        const H0Series s = H0Series();
        for (int m = 0; m < H0S_TERMS; ++m) {
            jh[m] = df_hi(s.cj[m]);
            jl[m] = df_lo(s.cj[m]);
            vh[m] = df_hi(s.cy[m]);
            vl[m] = df_lo(s.cy[m]);
        }
    }
};
static __constant__ H0DF c_h0df = H0DF();

// (A, J) of a free pair at z = (k r / 2)^2.  The first D terms of both series in
// double-float, the rest up to T in FP32: z^D / (D!)^2 < 2^-24 and z^T / (T!)^2 <
// 2^-50 for z up to the instantiation's limit (1: D = 7, T = 12; 1/16: D = 4, T = 7).
template <int D, int T>
__device__ __forceinline__ void h0_df(const DfSmem &tab, df z, df *A, df *J)
{
    float fj = c_h0df.jh[T - 1], fv = c_h0df.vh[T - 1];
#pragma unroll
    for (int m = T - 2; m >= D; --m) {
        fj = fmaf(fj, z.h, c_h0df.jh[m]);
        fv = fmaf(fv, z.h, c_h0df.vh[m]);
    }
    df j = {fj, 0.f}, v = {fv, 0.f};
#pragma unroll
    for (int m = D - 1; m >= 0; --m) {
        j = df_horner(df{c_h0df.jh[m], c_h0df.jl[m]}, z, j);
        if (m >= 1) v = df_horner(df{c_h0df.vh[m], c_h0df.vl[m]}, z, v);
    }
    const df lz = df_add(df_log(tab, z), df{1.1544313f, -1.3275548e-08f}); // ln z + 2 gamma
    const df a = df_mul(lz, j);
    df b = df_mul_raw(z, v);
    b = df{2.f * b.h, 2.f * b.l};
    *A = df_add(a, b);
    *J = j;
}
// the same from the FP64 functions, x = k r of the FP64 coordinates
static __device__ __noinline__ void h0_slow(double x, df *A, df *J)
{
    const zd g = h0_free64(x);
    *A = df_of(-4.0 * M_PI * g.re);
    *J = df_of(4.0 * g.im);
}
