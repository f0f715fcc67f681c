// df.cuh -- double-float arithmetic on the FP32 pipes (Dekker 1971, Knuth's
// TwoSum): a value is hi + lo, two FP32 numbers, 48 significand bits.  GB300
// issues 128 FP32 FMAs per clock and SM against 2 FP64 ones, so a double-float
// product (7 instructions) or sum (11) costs a fraction of its FP64 counterpart
// (64 issue slots).  Every rounding below is written with the _rn intrinsics, so
// the compiler neither contracts nor reorders the error terms.
#pragma once
#include "common.cuh"

struct df {
    float h, l;
};

__device__ __forceinline__ df df_of(double a)
{
    const float h = __double2float_rn(a);
    return df{h, __double2float_rn(a - (double)h)};
}
__device__ __forceinline__ double df_double(df a) { return (double)a.h + (double)a.l; }
// a + b exactly as s + e; the quick form needs |a| >= |b| (or a = 0)
__device__ __forceinline__ df two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return df{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ df quick_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return df{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return df{p, fmaf(a, b, -p)};
}
__device__ __forceinline__ df df_add(df a, df b)
{
    df s = two_sum(a.h, b.h);
    s.l = __fadd_rn(s.l, __fadd_rn(a.l, b.l));
    return quick_two_sum(s.h, s.l);
}
__device__ __forceinline__ df df_neg(df a) { return df{-a.h, -a.l}; }
__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, df_neg(b)); }
// product, not renormalised: |lo| stays below a few ulp of hi
__device__ __forceinline__ df df_mul_raw(df a, df b)
{
    df p = two_prod(a.h, b.h);
    p.l = fmaf(a.h, b.l, p.l);
    p.l = fmaf(a.l, b.h, p.l);
    return p;
}
__device__ __forceinline__ df df_mul(df a, df b)
{
    const df p = df_mul_raw(a, b);
    return quick_two_sum(p.h, p.l);
}
__device__ __forceinline__ df df_mulf(df a, float b)
{
    df p = two_prod(a.h, b);
    p.l = fmaf(a.l, b, p.l);
    return quick_two_sum(p.h, p.l);
}
__device__ __forceinline__ df df_sq(df a)
{
    df p = two_prod(a.h, a.h);
    p.l = fmaf(__fadd_rn(a.h, a.h), a.l, p.l);
    return p;
}
// c + z a for |c| >= |z a| (a Horner step)
__device__ __forceinline__ df df_horner(df c, df z, df a)
{
    const df p = df_mul_raw(z, a);
    df s = quick_two_sum(c.h, p.h);
    s.l = __fadd_rn(s.l, __fadd_rn(c.l, p.l));
    return s;
}
// running sum (sh, sl) += a b; sl collects the rounding errors
__device__ __forceinline__ void df_mac(float &sh, float &sl, float ah, float al, float bh, float bl)
{
    const float p = __fmul_rn(ah, bh);
    float e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, e);
    e = fmaf(al, bh, e);
    const float s = __fadd_rn(sh, p);
    const float bb = __fsub_rn(s, sh);
    const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    sh = s;
    sl = __fadd_rn(sl, __fadd_rn(err, e));
}
__device__ __forceinline__ void df_mac(df &s, df a, df b) { df_mac(s.h, s.l, a.h, a.l, b.h, b.l); }

// a complex number as (re hi, re lo, im hi, im lo)
__device__ __forceinline__ df df_re(float4 a) { return df{a.x, a.y}; }
__device__ __forceinline__ df df_im(float4 a) { return df{a.z, a.w}; }
__device__ __forceinline__ float4 df_pack(df re, df im) { return make_float4(re.h, re.l, im.h, im.l); }
__device__ __forceinline__ float4 df_split(zd a) { return df_pack(df_of(a.re), df_of(a.im)); }
// acc += t m
__device__ __forceinline__ void dfc_mac(float4 &acc, const float4 t, const float4 m)
{
    df_mac(acc.x, acc.y, t.x, t.y, m.x, m.y);
    df_mac(acc.x, acc.y, -t.z, -t.w, m.z, m.w);
    df_mac(acc.z, acc.w, t.x, t.y, m.z, m.w);
    df_mac(acc.z, acc.w, t.z, t.w, m.x, m.y);
}
__device__ __forceinline__ float4 dfc_mul(float4 a, float4 b)
{
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    dfc_mac(r, a, b);
    const df re = quick_two_sum(r.x, r.y), im = quick_two_sum(r.z, r.w);
    return df_pack(re, im);
}
__device__ __forceinline__ float4 dfc_add(float4 a, float4 b)
{
    return df_pack(df_add(df_re(a), df_re(b)), df_add(df_im(a), df_im(b)));
}
__device__ __forceinline__ float4 df_norm(float4 a)
{
    return df_pack(quick_two_sum(a.x, a.y), quick_two_sum(a.z, a.w));
}
__device__ __forceinline__ float4 shfl4(float4 a, int o)
{
    return make_float4(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o),
                       __shfl_xor_sync(0xffffffffu, a.z, o), __shfl_xor_sync(0xffffffffu, a.w, o));
}
// sum over the lanes lane ^ o, o = first, 2 first, .. < 32 (fixed order)
__device__ __forceinline__ df df_warp_sum(df a, int first = 1)
{
    for (int o = 16; o >= first; o >>= 1)
        a = df_add(a, df{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)});
    return a;
}

// ---------------------------------------------------------------------------
// Tables of the exponential and the logarithm (both table-driven in the manner
// of Tang, ACM TOMS 15 (1989) and 16 (1990)), copied to shared memory by the
// kernels that use them:
//   cs[i]  = (cos, sin)(2 pi i / 256) as double-floats,
//   ex[i]  = 2^(i/64),
//   lg[i]  = (r, -, -ln r) with r about 1/m, m the middle of [1 + i/128, 1 + (i+1)/128).
// ---------------------------------------------------------------------------
struct f4 { // float4 with a constant-expression constructor
    float x, y, z, w;
};
constexpr float df_hi(double a) { return (float)a; }
constexpr float df_lo(double a) { return (float)(a - (double)(float)a); }
struct DfTables {
    f4 cs[256], lg[128];
    float ex[64][2];
    constexpr DfTables() : cs(), lg(), ex()
    {
        for (int i = 0; i < 256; ++i) { // octant-reduced series
            const int o = (i + 16) / 32; // nearest multiple of pi/4
            const double a = 6.283185307179586476925 * (i - 32 * o) / 256.0;
            double c = 0.0, s = 0.0, f = 1.0;
            for (int m = 0; m < 24; ++m) {
                if (m & 1) s += (m & 2) ? -f : f;
                else c += (m & 2) ? -f : f;
                f *= a / (m + 1);
            }
            const double q = 0.70710678118654752440;
            const double C8[8] = {1, q, 0, -q, -1, -q, 0, q}, S8[8] = {0, q, 1, q, 0, -q, -1, -q};
            const double co = C8[o & 7], so = S8[o & 7];
            const double cc = co * c - so * s, ss = so * c + co * s;
            cs[i] = f4{df_hi(cc), df_lo(cc), df_hi(ss), df_lo(ss)};
        }
        for (int i = 0; i < 64; ++i) {
            const double a = 0.693147180559945309417 * i / 64.0;
            double e = 0.0, f = 1.0;
            for (int m = 0; m < 26; ++m) {
                e += f;
                f *= a / (m + 1);
            }
            ex[i][0] = df_hi(e);
            ex[i][1] = df_lo(e);
        }
        for (int i = 0; i < 128; ++i) {
            const float r = (float)(1.0 / (1.0 + (i + 0.5) / 128.0));
            // -ln r = 2 atanh((1 - r)/(1 + r)), r in (1/2, 1)
            const double t = (1.0 - (double)r) / (1.0 + (double)r);
            double s = 0.0, f = t;
            for (int m = 0; m < 40; ++m) {
                s += f / (2 * m + 1);
                f *= t * t;
            }
            lg[i] = f4{r, 0.f, df_hi(2.0 * s), df_lo(2.0 * s)};
        }
    }
};
static __device__ const DfTables d_dft = DfTables();

struct DfSmem {
    float4 cs[256], lg[128];
    float2 ex[64];
    __device__ __forceinline__ void load() // by the whole block; the caller synchronises
    {
        for (int i = threadIdx.x; i < 256; i += blockDim.x) cs[i] = *(const float4 *)&d_dft.cs[i];
        for (int i = threadIdx.x; i < 128; i += blockDim.x) lg[i] = *(const float4 *)&d_dft.lg[i];
        for (int i = threadIdx.x; i < 64; i += blockDim.x) ex[i] = make_float2(d_dft.ex[i][0], d_dft.ex[i][1]);
    }
};

// e^{x + i y} with x in units of ln 2 / 64 and y in units of 2 pi / 256 (the
// callers' tables carry the factors): x and y split into the table index and a
// remainder of at most half a unit, exact by construction.  Relative error below
// 1e-13 (the exponential's series ends at t^4: 5e-14 at most).
__device__ __forceinline__ float4 df_cexp(const DfSmem &T, df x, df y)
{
    // 2^(n/64) (1 + t + t^2/2 + t^3/6 + t^4/24), t = r ln 2 / 64, |t| < 0.0055
    const float xn = rintf(x.h);
    const df xr = quick_two_sum(__fsub_rn(x.h, xn), x.l); // |x.h - xn| <= 1/2 exactly; x.l is below it or xr is tiny
    const int n = (int)fmaxf(xn, -9600.f); // 2^(-150): below FP32's range the value is zero
    const float uh = 0.010830425f, ul = -2.9760222e-11f; // ln 2 / 64
    df t = two_prod(xr.h, uh);
    t.l = fmaf(xr.h, ul, fmaf(xr.l, uh, t.l));
    const float q = __fmul_rn(t.h, t.h);
    const float ql = fmaf(t.h, t.h, -q);
    df e1 = quick_two_sum(t.h, 0.5f * q);
    e1.l = __fadd_rn(e1.l, fmaf(0.5f, ql, fmaf(t.h, t.l, fmaf(q * t.h, fmaf(t.h, 0.041666667f, 0.16666667f), t.l))));
    const float2 b = T.ex[n & 63];
    df E = df_mul_raw(df{b.x, b.y}, e1);
    {
        const df s = quick_two_sum(b.x, E.h);
        E = df{s.h, __fadd_rn(s.l, __fadd_rn(b.y, E.l))};
    }
    // 2^(n >> 6) in two factors, so that gradual underflow and n down to -150 stay finite
    const int k = n >> 6, k1 = max(k, -120), k2 = max(k - k1, -120);
    const float f1 = __int_as_float((min(k1, 127) + 127) << 23), f2 = __int_as_float((k2 + 127) << 23);
    // (cos, sin) of the table angle plus r 2 pi / 256, |.| < 0.0123
    const float yn = rintf(y.h);
    const df yr = quick_two_sum(__fsub_rn(y.h, yn), y.l);
    const float4 cs = T.cs[((int)yn) & 255];
    const float vh = 0.024543693f, vl = -6.8299044e-10f; // 2 pi / 256
    df s = two_prod(yr.h, vh);
    s.l = fmaf(yr.h, vl, fmaf(yr.l, vh, s.l));
    const float w = __fmul_rn(s.h, s.h), wl = fmaf(s.h, s.h, -w);
    // sin = s - s^3/6 + s^5/120, cos - 1 = -s^2/2 + s^4/24
    const float c1 = -0.5f * w, c1l = fmaf(w * w, 0.041666667f, fmaf(-0.5f, wl, -(s.h * s.l)));
    s.l = fmaf(s.h * w, fmaf(w, 0.0083333333f, -0.16666667f), s.l);
    const df C = {cs.x, cs.y}, S = {cs.z, cs.w};
    // C + C c1 - S s and S + S c1 + C s
    df a = two_prod(C.h, c1), p = df_mul_raw(S, s);
    df r = two_sum(a.h, -p.h);
    r.l += fmaf(C.l, c1, fmaf(C.h, c1l, a.l - p.l));
    df co = two_sum(C.h, r.h);
    co.l += C.l + r.l;
    a = two_prod(S.h, c1);
    p = df_mul_raw(C, s);
    r = two_sum(a.h, p.h);
    r.l += fmaf(S.l, c1, fmaf(S.h, c1l, a.l + p.l));
    df si = two_sum(S.h, r.h);
    si.l += S.l + r.l;
    E.h *= f1;
    E.l *= f1;
    df re = df_mul(co, E), im = df_mul(si, E);
    return make_float4(re.h * f2, re.l * f2, im.h * f2, im.l * f2);
}

// ln z for a normal z.h > 0: exponent, table value and ln(1 + r), |r| < 2^-7.9
__device__ __forceinline__ df df_log(const DfSmem &T, df z)
{
    const int zi = __float_as_int(z.h), e = (zi >> 23) - 127;
    const float mh = __int_as_float((zi & 0x7fffff) | 0x3f800000), ml = z.l * __int_as_float((127 - e) << 23);
    const float4 t = T.lg[(zi >> 16) & 127];
    const df p = two_prod(mh, t.x);
    df r = quick_two_sum(__fsub_rn(p.h, 1.0f), 0.0f);
    r.l = fmaf(ml, t.x, p.l);
    r = two_sum(r.h, r.l);
    const float q = __fmul_rn(r.h, r.h), ql = fmaf(r.h, r.h, -q);
    df s = two_sum(r.h, -0.5f * q);
    // - r^2/2 (low part) + r^3/3 - r^4/4 + r^5/5 - r^6/6
    const float tail = q * r.h * fmaf(r.h, fmaf(r.h, fmaf(r.h, -0.16666667f, 0.2f), -0.25f), 0.33333333f);
    s.l += r.l + (tail - fmaf(0.5f, ql, r.h * r.l));
    // e ln 2: the leading part of ln 2 has 15 bits, so its product with e is exact
    const float fe = (float)e;
    const float L1 = 0.693145751953125f, L2 = 1.4286068e-06f, L3 = 5.497923e-14f;
    df b = two_prod(fe, L2);
    b.l = fmaf(fe, L3, b.l);
    df u = two_sum(fe * L1, t.z);
    u.l += t.w;
    df v = two_sum(u.h, s.h);
    df w = two_sum(v.h, b.h);
    w.l += (v.l + b.l) + (u.l + s.l);
    return quick_two_sum(w.h, w.l);
}
