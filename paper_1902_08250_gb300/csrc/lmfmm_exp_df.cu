// lmfmm_exp_df.cu -- expansions of the FP64 form in double-float on the FP32
// pipes: S2M, M2M, M2L, L2L and L2T.  Multipoles and local expansions are kept as
// float4 (re hi, re lo, im hi, im lo), scaled by 2^-qexp[vector], [box][2p+1][nvec]: an FP64
// value takes the same 16 bytes, but converting it costs FP64 instructions (64 issue
// slots each), and with nvec instead of 16 slots per order the one-vector apply
// reads whole lines.
//
// The Bessel basis of S2M and L2T comes from its power series.  With (rx, ry) the
// point's offset from the box centre, Z = (rx + i ry)/w and t = (k r / 2)^2,
//     Jhat_n(k r) e^{i n theta} = Z^n g_n(t),   g_n = 0F1(; n + 1; -t) (DLMF 10.16.9),
// Jhat_n = J_n / S(n).  g is evaluated from its series at orders N and N + 1, N >= p,
// and carried down by 0F1's contiguous relation (DLMF 16.3.6 for 0F1)
//     g_{n-1} = g_n - t / (n (n + 1)) g_{n+1}.
// No division, no angle and no normalisation is left per point; the former backward
// recurrence divided in FP64 twice per order and took one thread through 70 orders.
#include <math.h>
#include <algorithm>

#include "df.cuh"
#include "internal.h"
#include "near64.cuh"

static int gridn(int64_t n, int b) { return (int)((n + b - 1) / b); }

// Z^n g_n, n = 0..P, of one point into row[0..P]; rel: offset from the box centre times k/2;
// iw = 2/(k w)
__device__ __forceinline__ void basis_row(const BesselDF &B, int P, float4 rel, df iw, float4 *row)
{
    const df x = df_re(rel), y = df_im(rel);
    const df t = df_add(df_sq(x), df_sq(y)), mt = df_neg(t);
    df g0 = {1.f, 0.f}, g1 = {1.f, 0.f}; // g_N, g_{N+1}
    for (int m = B.nt; m >= 1; --m) {
        const float2 a = B.c[B.N + m], b = B.c[B.N + B.nt + m];
        g0 = df_horner(df{1.f, 0.f}, df_mul(mt, df{a.x, a.y}), g0);
        g1 = df_horner(df{1.f, 0.f}, df_mul(mt, df{b.x, b.y}), g1);
    }
    for (int n = B.N; n >= 1; --n) {
        if (n <= P) *(float2 *)&row[n] = make_float2(g0.h, g0.l);
        const float2 c = B.c[n];
        const df p = df_mul_raw(df_mul(mt, df{c.x, c.y}), g1);
        g1 = g0;
        g0 = df_add(g0, p);
    }
    row[0] = df_pack(g0, df{0.f, 0.f});
    const float4 Z = df_pack(df_mul(x, iw), df_mul(y, iw));
    float4 zp = Z;
    for (int n = 1; n <= P; ++n) {
        const float2 g = *(const float2 *)&row[n];
        row[n] = df_pack(df_mul(df_re(zp), df{g.x, g.y}), df_mul(df_im(zp), df{g.x, g.y}));
        if (n < P) zp = dfc_mul(zp, Z);
    }
}

// ---------------------------------------------------------------------------
// S2M (Eq. (multipole_coef)), scaled: Mhat_q = sum_j q_j Jhat_q(k r_j) e^{-i q theta_j}.
// One block per leaf, 32 points a round: a thread forms a point's basis row, then
// a thread per (order n >= 0, vector) sums the four products b.re, b.im x q.re, q.im,
// from which the orders n and -n both follow.  Bound by FP32 issue.  250k strip, 16 vectors:
// 0.36 ms (4.4 ms in FP64).
// ---------------------------------------------------------------------------
#define XD_PTS 32
template <int NV, class Geo>
__global__ void __launch_bounds__(128) k_s2m_df(Geo geo, int P, double k, BesselDF B, const float4 *rel,
                                                const int64_t *ls, const float4 *qd, int nv, float4 *M)
{
    extern __shared__ float4 xs_sm[];
    const int np = 2 * P + 1, rs = (P + 1) | 1; // odd row stride: no bank conflicts among the rows
    float4 *b = xs_sm, *q = xs_sm + XD_PTS * rs;
    constexpr int THR = NV >= 4 ? 128 : 64, MAXI = ((LM_MAXP + 1) * NV + THR - 1) / THR; // launched with THR threads
    const int64_t box = geo.id(blockIdx.x), lo = ls[box], hi = ls[box + 1];
    __shared__ float2 siw;
    if (threadIdx.x == 0) {
        double cx, cy, w;
        geo.centre(box, &cx, &cy, &w);
        const df a = df_of(2.0 / (k * w));
        siw = make_float2(a.h, a.l);
    }
    float4 s0[MAXI], s1[MAXI]; // (sum q.re b.re, sum q.im b.im), (sum q.im b.re, sum q.re b.im)
#pragma unroll
    for (int i = 0; i < MAXI; ++i) s0[i] = s1[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int nitem = (P + 1) * nv;
    for (int64_t p0 = lo; p0 < hi; p0 += XD_PTS) {
        const int cnt = (int)min((int64_t)XD_PTS, hi - p0);
        __syncthreads();
        if (threadIdx.x < cnt) basis_row(B, P, rel[p0 + threadIdx.x], df{siw.x, siw.y}, b + threadIdx.x * rs);
        for (int i = threadIdx.x; i < cnt * nv; i += blockDim.x) q[i] = qd[p0 * nv + i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < MAXI; ++i) {
            const int it = threadIdx.x + i * blockDim.x;
            if (it < nitem) {
                const int n = it / nv, v = it - n * nv;
                for (int j = 0; j < cnt; ++j) {
                    const float4 bb = b[j * rs + n], qq = q[j * nv + v];
                    df_mac(s0[i].x, s0[i].y, bb.x, bb.y, qq.x, qq.y);
                    df_mac(s0[i].z, s0[i].w, bb.z, bb.w, qq.z, qq.w);
                    df_mac(s1[i].x, s1[i].y, bb.x, bb.y, qq.z, qq.w);
                    df_mac(s1[i].z, s1[i].w, bb.z, bb.w, qq.x, qq.y);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < MAXI; ++i) {
        const int it = threadIdx.x + i * blockDim.x;
        if (it < nitem) {
            const int n = it / nv, v = it - n * nv;
            const df rr = df_re(s0[i]), ii = df_im(s0[i]), ir = df_re(s1[i]), ri = df_im(s1[i]);
            // order n: q conj(b); order -n: (-1)^n q b
            M[(box * np + P + n) * nv + v] = df_pack(df_add(rr, ii), df_sub(ir, ri));
            const float sg = (n & 1) ? -1.f : 1.f;
            df re = df_sub(rr, ii), im = df_add(ir, ri);
            if (n > 0)
                M[(box * np + P - n) * nv + v] = make_float4(sg * re.h, sg * re.l, sg * im.h, sg * im.l);
        }
    }
}

// ---------------------------------------------------------------------------
// L2T (Eq. (local)): u = sum_n Lhat_n Z^n g_n over |n| <= P; with b_n = Z^n g_n and
// b_{-n} = (-1)^n conj(b_n),
//     u = L_0 b_0 + sum_{n >= 1} [(L_n + s L_{-n}) b_n.re + i (L_n - s L_{-n}) b_n.im], s = (-1)^n.
// GRAD: also du/dx and du/dy, local expansions of order P + 1 themselves,
//     (d/dx + i d/dy) J_n e^{i n t} = -k J_{n+1} e^{i(n+1)t}, (d/dx - i d/dy) J_n e^{i n t} = k J_{n-1} e^{i(n-1)t};
// in scaled coefficients the shifts carry S(n)/S(n -+ 1).  Values are set in FP64: u in tree
// order, or (GRAD) u, ux, uy in input order through perm.  A thread per point forms its basis row, then
// one per (point, vector) sums it.  Bound by FP32 issue: 250k strip, 16 vectors 0.27 ms.
// ---------------------------------------------------------------------------
struct L2TOut {
    zd *u, *ux, *uy;
    const int64_t *perm;
};
template <bool GRAD, class Geo>
__global__ void __launch_bounds__(128) k_l2t_df(Geo geo, int P, double k, BesselDF B, const float4 *rel,
                                                const int64_t *ls, const float4 *L, int nvl, int v0, int nv,
                                                const int *qexp, int64_t n, L2TOut out)
{
    extern __shared__ float4 xs_sm[];
    constexpr int SETS = GRAD ? 3 : 1;
    const int PB = P + (GRAD ? 1 : 0), np = 2 * P + 1, rs = (PB + 1) | 1;
    float4 *b = xs_sm, *C = xs_sm + XD_PTS * rs; // C: [SETS][PB + 1][nv][2]
    const int64_t box = geo.id(blockIdx.x), lo = ls[box], hi = ls[box + 1];
    if (lo == hi) return;
    __shared__ float2 siw;
    double cx, cy, w;
    geo.centre(box, &cx, &cy, &w);
    if (threadIdx.x == 0) {
        const df a = df_of(2.0 / (k * w));
        siw = make_float2(a.h, a.l);
    }
    const float4 *Lb = L + box * np * nvl + v0;
    auto get = [&](int m, int v) { return abs(m) <= P ? Lb[(P + m) * nvl + v] : make_float4(0.f, 0.f, 0.f, 0.f); };
    auto scl = [](float4 a, double f) { // a f
        const df ff = df_of(f);
        return df_pack(df_mul(df_re(a), ff), df_mul(df_im(a), ff));
    };
    auto put = [&](int set, int m, int v, float4 lp, float4 lm) { // orders m and -m
        const float sg = (m & 1) ? -1.f : 1.f;
        const float4 sl = make_float4(sg * lm.x, sg * lm.y, sg * lm.z, sg * lm.w);
        const float4 a = m ? dfc_add(lp, sl) : lp;
        const float4 d = m ? dfc_add(lp, make_float4(-sl.x, -sl.y, -sl.z, -sl.w)) : make_float4(0.f, 0.f, 0.f, 0.f);
        float4 *c = C + 2 * ((set * (PB + 1) + m) * nv + v);
        c[0] = a;
        c[1] = make_float4(-d.z, -d.w, d.x, d.y); // i d
    };
    for (int i = threadIdx.x; i < (PB + 1) * nv; i += blockDim.x) {
        const int m = i / nv, v = i - m * nv;
        put(0, m, v, get(m, v), get(-m, v));
        if (GRAD) {
            // dm_n = -k L_{n-1} S(|n|)/S(|n-1|), dp_n = k L_{n+1} S(|n|)/S(|n+1|); S(m)/S(m-1) = hs/m
            const double hs = 0.5 * k * w;
            auto up = [&](int a) { return (double)(a + 1) / hs; };   // S(a)/S(a+1)
            auto dn = [&](int a) { return hs / (double)a; };          // S(a)/S(a-1)
            float4 d[2][2]; // [+m, -m][dp, dm]
            d[0][0] = scl(get(m + 1, v), k * up(m));
            d[0][1] = m ? scl(get(m - 1, v), -k * dn(m)) : scl(get(-1, v), -k * up(0));
            d[1][0] = m ? scl(get(1 - m, v), k * dn(m)) : d[0][0];
            d[1][1] = m ? scl(get(-m - 1, v), -k * up(m)) : d[0][1];
            float4 x[2], y[2];
            for (int s = 0; s < 2; ++s) {
                const float4 p = d[s][0], q = d[s][1];
                const float4 a = dfc_add(p, q), e = dfc_add(p, make_float4(-q.x, -q.y, -q.z, -q.w));
                x[s] = make_float4(0.5f * a.x, 0.5f * a.y, 0.5f * a.z, 0.5f * a.w);
                y[s] = make_float4(-0.5f * e.z, -0.5f * e.w, 0.5f * e.x, 0.5f * e.y); // i (dp - dm)/2
            }
            put(1, m, v, x[0], x[1]);
            put(2, m, v, y[0], y[1]);
        }
    }
    for (int64_t p0 = lo; p0 < hi; p0 += XD_PTS) {
        const int cnt = (int)min((int64_t)XD_PTS, hi - p0);
        __syncthreads();
        if (threadIdx.x < cnt) basis_row(B, PB, rel[p0 + threadIdx.x], df{siw.x, siw.y}, b + threadIdx.x * rs);
        __syncthreads();
        for (int it = threadIdx.x; it < cnt * nv * SETS; it += blockDim.x) {
            const int j = it % cnt, sv = it / cnt, v = sv % nv, set = sv / nv;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int m = 0; m <= PB; ++m) {
                const float4 bb = b[j * rs + m];
                const float4 *c = C + 2 * ((set * (PB + 1) + m) * nv + v);
                df_mac(a.x, a.y, c[0].x, c[0].y, bb.x, bb.y);
                df_mac(a.z, a.w, c[0].z, c[0].w, bb.x, bb.y);
                df_mac(a.x, a.y, c[1].x, c[1].y, bb.z, bb.w);
                df_mac(a.z, a.w, c[1].z, c[1].w, bb.z, bb.w);
            }
            const int ex = qexp_of(qexp, v0 + v);
            const zd r = {ldexp(df_double(df_re(a)), ex), ldexp(df_double(df_im(a)), ex)};
            if (GRAD) {
                zd *o = set == 0 ? out.u : set == 1 ? out.ux : out.uy;
                if (o) o[(int64_t)v * n + out.perm[p0 + j]] = r;
            } else
                out.u[(int64_t)v * n + p0 + j] = r;
        }
    }
}

// ---------------------------------------------------------------------------
// Translations.  Tables transposed, [q][p]: the lanes of a warp take consecutive
// orders p, so a table row is one contiguous read and the multipole a broadcast.
// A thread holds VPT = min(NV, 4) vectors of one order: a table entry (16 bytes)
// is read once for VPT multiply-adds of 48 FP32 instructions.
// ---------------------------------------------------------------------------
// (vectors beyond nv are summed with their neighbours' data, inside the 16-slot buffers, and not stored)
template <int VPT>
__device__ __forceinline__ void dot_q(float4 *acc, const float4 *T, const float4 *m, int nq, int np, int nv)
{
    int q = 0;
    for (; q + 4 <= nq; q += 4) { // four table entries in flight
        float4 t[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = T[(q + j) * np];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < VPT; ++i)
                dfc_mac(acc[i], t[j], m[(q + j) * nv + i]);
    }
    for (; q < nq; ++q)
#pragma unroll
        for (int i = 0; i < VPT; ++i)
            dfc_mac(acc[i], T[q * np], m[q * nv + i]);
}

// M2M: one block per (parent, group of VPT vectors); a thread per (part of the sum over q, child
// position, order).  Each position's parts are added in order, then the positions.  QS parts of the
// sum (2 while 512 threads hold them) depend on the order alone: a vector's result does not depend on
// the others.  Bound by FP32 issue on large levels, by the chain of multiply-adds on small ones: 250k
// strip, 16 vectors, the four levels above 5120 boxes 456 us with a thread for the four positions of
// (order, 4 vectors), 167 us; adjoint of 20k points, 2 vectors, 69 us with QS = 1, 52 us with 2.
template <int VPT, class Geo>
__global__ void __launch_bounds__(512) k_m2m_dx(Geo geo, int P, int nv, int QS, const float4 *tabs, const float4 *Mc, float4 *Mp)
{
    extern __shared__ float4 red[]; // [4 QS - 1][np][VPT]
    const int np = 2 * P + 1, v0 = blockIdx.y * VPT, nvv = min(VPT, nv - v0);
    const int64_t b = geo.parent(blockIdx.x);
    const int p = threadIdx.x % np, r = threadIdx.x / np, pos = r & 3, qs = r >> 2;
    const int q0 = qs * np / QS, q1 = (qs + 1) * np / QS;
    float4 acc[VPT];
#pragma unroll
    for (int i = 0; i < VPT; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (qs < QS) {
        dot_q<VPT>(acc, tabs + ((int64_t)pos * np + q0) * np + p, Mc + (geo.child(b, pos) * np + q0) * nv + v0, q1 - q0, np, nv);
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            acc[i] = df_norm(acc[i]);
            if (r > 0) red[((r - 1) * np + p) * VPT + i] = acc[i];
        }
    }
    __syncthreads();
    if (r > 0) return;
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        float4 tot = acc[i];
        for (int c = 0; c < 4; ++c) {
            float4 part = c == 0 ? acc[i] : red[((c - 1) * np + p) * VPT + i];
            for (int h = 1; h < QS; ++h) part = dfc_add(part, red[((c + 4 * h - 1) * np + p) * VPT + i]);
            tot = c == 0 ? part : dfc_add(tot, part);
        }
        if (i < nvv) Mp[(b * np + p) * nv + v0 + i] = tot;
    }
}

// L2L: one block per (parent, group of vectors), threads as in M2M; adds to the child's L
template <int VPT, class Geo>
__global__ void __launch_bounds__(512) k_l2l_dx(Geo geo, int P, int nv, int QS, const float4 *tabs, const float4 *Lp, float4 *Lc)
{
    extern __shared__ float4 red[]; // [4 QS - 4][np][VPT]
    const int np = 2 * P + 1, v0 = blockIdx.y * VPT, nvv = min(VPT, nv - v0);
    const int64_t b = geo.parent(blockIdx.x);
    const int p = threadIdx.x % np, r = threadIdx.x / np, pos = r & 3, qs = r >> 2;
    const int q0 = qs * np / QS, q1 = (qs + 1) * np / QS;
    float4 acc[VPT];
#pragma unroll
    for (int i = 0; i < VPT; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (qs < QS) {
        dot_q<VPT>(acc, tabs + ((int64_t)pos * np + q0) * np + p, Lp + (b * np + q0) * nv + v0, q1 - q0, np, nv);
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            acc[i] = df_norm(acc[i]);
            if (qs > 0) red[((r - 4) * np + p) * VPT + i] = acc[i];
        }
    }
    if (QS > 1) __syncthreads();
    if (qs > 0) return;
    float4 *o = Lc + (geo.child(b, pos) * np + p) * nv + v0;
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        for (int h = 1; h < QS; ++h) acc[i] = dfc_add(acc[i], red[((r + 4 * h - 4) * np + p) * VPT + i]);
        if (i < nvv) o[i] = dfc_add(o[i], acc[i]);
    }
}

// M2L over the V lists of every level in one launch: one block per target box; sets L.
// The entries form GS interleaved subsets (3, or 12 for small trees), each summed on its own; the
// sums of equal index mod 3 are added in order, then the three: a vector's result does not depend on
// how many vectors are applied or on how many threads share a box.  G groups of threads (GS, 3 or 1)
// take the subsets.  Bound by FP32 issue on large trees (24 multiply-adds a complex product) and by the
// reads of table and multipoles in the two or three blocks an SM gets on small ones.
template <int NV, int MINB>
__global__ void __launch_bounds__(512, MINB) k_m2l_dx(const M2LLevelDF *lev, int nlev, int P, int nv, int GS, int G)
{
    constexpr int VPT = NV < 4 ? NV : 4;
    extern __shared__ float4 red[]; // [G - 1][items][VPT]
    const int np = 2 * P + 1, vg = (nv + VPT - 1) / VPT, item = np * vg;
    int l = nlev - 1;
    while ((int64_t)blockIdx.x < lev[l].box0) --l;
    const M2LLevelDF &v = lev[l];
    const int64_t b = blockIdx.x - v.box0, e0 = v.vstart[b], e1 = v.vstart[b + 1];
    const int it = threadIdx.x % item, g = threadIdx.x / item, p = it % np, v0 = it / np * VPT, nvv = min(VPT, nv - v0);
    const int k3 = min(3, GS); // the last level of the sum
    float4 tot[VPT];
#pragma unroll
    for (int i = 0; i < VPT; ++i) tot[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (g < G) {
        // G = GS: subset g; G = 3: subsets g, g + 3, ..; G = 1: all of them, class by class
        for (int c = G == 1 ? 0 : g; c < (G == 1 ? k3 : g + 1); ++c) {
            float4 part[VPT];
            for (int s = c; s < (G == GS && G > 1 ? c + 1 : GS); s += 3) {
                float4 acc[VPT];
#pragma unroll
                for (int i = 0; i < VPT; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int64_t e = e0 + s; e < e1; e += GS)
                    dot_q<VPT>(acc, v.tab + (int64_t)v.vslot[e] * np * np + p, v.M + (int64_t)v.vsrc[e] * np * nv + v0, np, np, nv);
#pragma unroll
                for (int i = 0; i < VPT; ++i) part[i] = s == c ? df_norm(acc[i]) : dfc_add(part[i], df_norm(acc[i]));
            }
#pragma unroll
            for (int i = 0; i < VPT; ++i) tot[i] = G > 1 || c == 0 ? part[i] : dfc_add(tot[i], part[i]);
        }
    }
    if (G > 1) {
        if (g > 0 && g < G)
#pragma unroll
            for (int i = 0; i < VPT; ++i) red[((g - 1) * item + it) * VPT + i] = tot[i];
        __syncthreads();
        if (g == 0)
#pragma unroll
            for (int i = 0; i < VPT; ++i) {
                auto at = [&](int s) { return red[((s - 1) * item + it) * VPT + i]; };
                for (int s = 3; s < G; s += 3) tot[i] = dfc_add(tot[i], at(s));
                for (int c = 1; c < k3; ++c) {
                    float4 part = at(c);
                    for (int s = c + 3; s < G; s += 3) part = dfc_add(part, at(s));
                    tot[i] = dfc_add(tot[i], part);
                }
            }
    }
    if (g == 0)
#pragma unroll
        for (int i = 0; i < VPT; ++i)
            if (i < nvv) v.L[(b * np + p) * nv + v0 + i] = tot[i];
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
__global__ void k_tab_df_t(const zd *tab, int64_t count, int np, float4 *out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= count) return;
    const int64_t slot = i / ((int64_t)np * np);
    const int r = (int)(i % ((int64_t)np * np)), p = r / np, q = r % np;
    out[slot * np * np + (int64_t)q * np + p] = df_split(tab[i]);
}

static int nv_slots(int nv) { return nv <= 1 ? 1 : nv <= 2 ? 2 : nv <= 4 ? 4 : nv <= 8 ? 8 : 16; }
#define NV_DISPATCH(nv, ...)                                  \
    switch (nv_slots(nv)) {                                   \
    case 1: { constexpr int NV = 1; __VA_ARGS__; } break;     \
    case 2: { constexpr int NV = 2; __VA_ARGS__; } break;     \
    case 4: { constexpr int NV = 4; __VA_ARGS__; } break;     \
    case 8: { constexpr int NV = 8; __VA_ARGS__; } break;     \
    default: { constexpr int NV = 16; __VA_ARGS__; } break;   \
    }
static int round32(int n) { return (n + 31) / 32 * 32; }
#define TRY_X(x)                     \
    do {                             \
        lm_status s_ = (x);          \
        if (s_ != LM_OK) return s_;  \
    } while (0)

// Largest (k r / 2)^2 of a point in its leaf that the basis takes: beyond it g_n, about
// e^{-k r / 2} at n = k r / 4, would leave FP32's range (k w > 140; no order up to 48 resolves such a box)
#define XD_TMAX 2500.0
bool lm_exp_df_fits(double k2, double wmax) { return 0.125 * k2 * k2 * wmax * wmax <= XD_TMAX; }

void lm_bessel_df(int P, double k, double wmax, std::vector<float> &h, int *N, int *nt)
{
    const double tmax = 0.125 * k * k * wmax * wmax;
    *N = std::max(P + 1, (int)ceil(tmax));
    *nt = 1;
    for (double v = tmax / (*N + 1); v > 1e-16; ++*nt) v *= tmax / ((*nt + 1.0) * (*N + *nt + 1.0));
    h.assign(2 * (*N + 2 * *nt + 1), 0.f);
    auto put = [&](int i, double v) {
        h[2 * i] = (float)v;
        h[2 * i + 1] = (float)(v - (double)(float)v);
    };
    for (int n = 1; n <= *N; ++n) put(n, 1.0 / ((double)n * (n + 1.0)));
    for (int m = 1; m <= *nt; ++m) {
        put(*N + m, 1.0 / ((double)m * (*N + m)));
        put(*N + *nt + m, 1.0 / ((double)m * (*N + 1.0 + m)));
    }
}

void lm_tab_df_t(const zd *tab, int64_t ncls, int np, float4 *out, cudaStream_t st)
{
    const int64_t cnt = ncls * np * np;
    k_tab_df_t<<<gridn(cnt, 256), 256, 0, st>>>(tab, cnt, np, out);
}

// Bessel coefficients, transposed double-float tables, level descriptors; t->ndf.wmax is set
lm_status lm_setup_exp_df(lm_tree_s *t, cudaStream_t st)
{
    ExpDF &E = t->xdf;
    const int P = t->p, np = 2 * P + 1;
    std::vector<float> h;
    lm_bessel_df(P, t->med.k2, t->ndf.wmax, h, &E.N, &E.nt);
    TRY_X(lm_dalloc(t, &E.bes, h.size() / 2));
    LM_CUDA(cudaMemcpyAsync(E.bes, h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice, st));
    auto conv = [&](const zd *tab, int64_t ncls, float4 **out) -> lm_status {
        const int64_t cnt = std::max<int64_t>(1, ncls) * np * np;
        TRY_X(lm_dalloc(t, out, cnt));
        k_tab_df_t<<<gridn(cnt, 256), 256, 0, st>>>(tab, cnt, np, *out);
        return LM_OK;
    };
    for (Level &lv : t->lev) {
        if (lv.m2m) TRY_X(conv(lv.m2m, 4, &lv.m2mdf)); // 4 child positions
        if (lv.l2l) TRY_X(conv(lv.l2l, 4, &lv.l2ldf));
    }
    std::vector<M2LLevelDF> lev;
    E.nblk = 0;
    if (t->adaptive) {
        AdaptTree &A = t->at;
        TRY_X(conv(A.tab, (int64_t)A.cls_term.size(), &A.tabdft));
        lev.push_back({0, A.vstart, A.vsrc, A.vslot, A.tabdft, (const float4 *)A.M, (float4 *)A.Lc});
        E.nblk = A.nbox;
    } else
        for (Level &lv : t->lev) {
            if (lm_oz_level(t, lv.l)) continue; // on the tensor cores
            TRY_X(conv(lv.tab, (int64_t)lv.cls_term.size(), &lv.tabdft));
            lev.push_back({E.nblk, lv.vstart, lv.vsrc, lv.vslot, lv.tabdft, (const float4 *)lv.M, (float4 *)lv.Lc});
            E.nblk += lv.nbox;
        }
    M2LLevelDF *d;
    TRY_X(lm_dalloc(t, &d, lev.size()));
    E.lev = d;
    E.nlev = (int)lev.size();
    LM_CUDA(cudaMemcpyAsync(d, lev.data(), lev.size() * sizeof(M2LLevelDF), cudaMemcpyHostToDevice, st));
    LM_CUDA(cudaStreamSynchronize(st)); // host temporaries
    LM_CUDA(cudaGetLastError());
    E.ready = true;
    return LM_OK;
}

template <class Geo>
static void launch_s2m(const BesselDF &B, Geo geo, int64_t nleaf, int P, double k, const float4 *rel, const int64_t *ls,
                       const float4 *q, int nv, float4 *M, cudaStream_t st)
{
    const size_t shm = (size_t)XD_PTS * (((P + 1) | 1) + nv) * sizeof(float4);
    NV_DISPATCH(nv, k_s2m_df<NV><<<(unsigned)nleaf, NV >= 4 ? 128 : 64, shm, st>>>(geo, P, k, B, rel, ls, q, nv, M))
}
// L2T of vectors v0 .. v0 + nw - 1 of the nvl in L
template <bool GRAD, class Geo>
static void launch_l2t(const BesselDF &B, Geo geo, int64_t nleaf, int P, double k, const float4 *rel, const int64_t *ls,
                       const float4 *L, int nvl, int v0, int nw, const int *qexp, int64_t n, const L2TOut &out, cudaStream_t st)
{
    const int PB = P + (GRAD ? 1 : 0);
    const size_t shm = ((size_t)XD_PTS * ((PB + 1) | 1) + (GRAD ? 3 : 1) * (PB + 1) * nw * 2) * sizeof(float4);
    k_l2t_df<GRAD><<<(unsigned)nleaf, nw > 2 || GRAD ? 128 : 64, shm, st>>>(geo, P, k, B, rel, ls, L, nvl, v0, nw, qexp, n, out);
}
// as many vectors at a time as the coefficients fit in 48 KB beside the basis; us: [nv][n], tree order
template <class Geo>
static int launch_l2t_all(const BesselDF &B, Geo geo, int64_t nleaf, int P, double k, const float4 *rel, const int64_t *ls,
                          const float4 *L, int nv, const int *qexp, int64_t n, zd *us, cudaStream_t st)
{
    const int room = 48 * 1024 / 16 - XD_PTS * ((P + 1) | 1), step = std::max(1, std::min(nv, room / (2 * (P + 1))));
    int k_ = 0;
    for (int w0 = 0; w0 < nv; w0 += step, ++k_)
        launch_l2t<false>(B, geo, nleaf, P, k, rel, ls, L, nv, w0, std::min(step, nv - w0), qexp, n,
                          L2TOut{us + (int64_t)w0 * n, nullptr, nullptr, nullptr}, st);
    return k_;
}
// parts of the sum over q of M2M and L2L
static int shift_parts(int np) { return 8 * np <= 512 ? 2 : 1; }
#define VPT_DISPATCH(nv, ...)                            \
    switch (nv) {                                         \
    case 1: { constexpr int VPT = 1; __VA_ARGS__; } break; \
    case 2: { constexpr int VPT = 2; __VA_ARGS__; } break; \
    default: { constexpr int VPT = 4; __VA_ARGS__; } break;\
    }
template <class Geo>
static void launch_m2m(Geo geo, int64_t npar, int P, int nv, const float4 *tab, const float4 *Mc, float4 *Mp, cudaStream_t st)
{
    const int np = 2 * P + 1, QS = shift_parts(np);
    VPT_DISPATCH(nv, {
        k_m2m_dx<VPT><<<dim3((unsigned)npar, (nv + VPT - 1) / VPT), round32(4 * QS * np), (size_t)(4 * QS - 1) * np * VPT * sizeof(float4),
                        st>>>(geo, P, nv, QS, tab, Mc, Mp);
    });
}
template <class Geo>
static void launch_l2l(Geo geo, int64_t npar, int P, int nv, const float4 *tab, const float4 *Lp, float4 *Lc, cudaStream_t st)
{
    const int np = 2 * P + 1, QS = shift_parts(np);
    VPT_DISPATCH(nv, {
        k_l2l_dx<VPT><<<dim3((unsigned)npar, (nv + VPT - 1) / VPT), round32(4 * QS * np), (size_t)(4 * QS - 4) * np * VPT * sizeof(float4),
                        st>>>(geo, P, nv, QS, tab, Lp, Lc);
    });
}
static void launch_m2l(const M2LLevelDF *lev, int nlev, int64_t nblk, int P, int nv, cudaStream_t st)
{
    const int np = 2 * P + 1;
    // subsets of a box's entries: 12 for small trees, whose boxes leave SMs idle, if 512 threads hold them
    const int GS = nblk < 1216 && 12 * np <= 512 ? 12 : 3;
    NV_DISPATCH(nv, {
        constexpr int VPT = NV < 4 ? NV : 4;
        const int item = np * ((nv + VPT - 1) / VPT);
        const int G = item * GS <= 512 && (GS - 1) * item * VPT <= 3072 ? GS : (item * 3 <= 512 ? 3 : 1); // 48 KB of sums
        const size_t shm = (size_t)(G - 1) * item * VPT * sizeof(float4);
        // one vector on many boxes (four waves of 8 blocks per SM): 64 registers, more warps; clustered 100k
        // 2.07 ms against 2.27 ms with 102.  Fewer boxes or more vectors: the registers (two vectors on
        // 1000 boxes: the whole apply 0.69 ms against 0.77 ms with 64).
        if (NV == 1 && nblk >= 4864)
            k_m2l_dx<NV, NV == 1 ? 2 : 1><<<(unsigned)nblk, round32(item * G), shm, st>>>(lev, nlev, P, nv, GS, G);
        else
            k_m2l_dx<NV, 1><<<(unsigned)nblk, round32(item * G), shm, st>>>(lev, nlev, P, nv, GS, G);
    });
}

// The same for the cross-layer operator's two trees (lmfmm_cross.cu), whose levels share one lattice
void lm_df_s2m(const BesselDF &B, const LeafGeom &g, int64_t nleaf, int P, double k, const float4 *rel, const int64_t *ls,
               const float4 *q, int nv, float4 *M, cudaStream_t st)
{
    launch_s2m(B, GridLeaves{g}, nleaf, P, k, rel, ls, q, nv, M, st);
}
void lm_df_l2t(const BesselDF &B, const LeafGeom &g, int64_t nleaf, int P, double k, const float4 *rel, const int64_t *ls,
               const float4 *L, int nv, const int *qexp, int64_t n, zd *us, cudaStream_t st)
{
    launch_l2t_all(B, GridLeaves{g}, nleaf, P, k, rel, ls, L, nv, qexp, n, us, st);
}
void lm_df_m2m(int64_t ncol, int64_t npar, int P, int nv, const float4 *tab, const float4 *Mc, float4 *Mp, cudaStream_t st)
{
    launch_m2m(GridParents{ncol}, npar, P, nv, tab, Mc, Mp, st);
}
void lm_df_l2l(int64_t ncol, int64_t npar, int P, int nv, const float4 *tab, const float4 *Lp, float4 *Lc, cudaStream_t st)
{
    launch_l2l(GridParents{ncol}, npar, P, nv, tab, Lp, Lc, st);
}
void lm_df_m2l(const M2LLevelDF *lev, int nlev, int64_t nblk, int P, int nv, cudaStream_t st)
{
    launch_m2l(lev, nlev, nblk, P, nv, st);
}

__global__ void k_permute_in(const zd *q, const int64_t *perm, int64_t n, int nvec, int conjugate, zd *qs);
__global__ void k_permute_out(const zd *us, const int64_t *perm, int64_t n, int nvec, int conjugate, zd *u);

// FP64 form in double-float, both tree kinds; with ux set, step 4 also evaluates the target gradient
// and writes u (or null), ux, uy
lm_status lm_run_df(lm_tree_s *t, const zd *q, int nvec, zd *u, bool adjoint, zd *ux, zd *uy, cudaStream_t st)
{
    const int L = t->L;
    const int64_t n = t->n;
    AdaptTree &A = t->at;
    const bool ad = t->adaptive;
    const ListBoxes leaves{A.leaves, A.cx, A.cy, A.w};
    const GridLeaves gleaves{LeafGeom{t->lev[L].ncol, t->x0, t->lev[L].w}};
    const int64_t nleaf = ad ? A.nleaf : t->lev[L].nbox;
    const BesselDF B{t->xdf.bes, t->xdf.N, t->xdf.nt};
    const int P = t->p;
    const double k2 = t->med.k2;
    zd *qs = t->qs ? t->qs : t->us; // (lm_setup_df)
    auto Mof = [&](int l) { return (float4 *)(ad ? A.M : t->lev[l].M); };
    auto Lof = [&](int l) { return (float4 *)(ad ? A.Lc : t->lev[l].Lc); };
    for (int v0 = 0; v0 < nvec; v0 += LM_MAXV) {
        const int nv = std::min(LM_MAXV, nvec - v0);
        lm_phase_begin(t, PH_PERMUTE, st);
        k_permute_in<<<gridn(n, 256), 256, 0, st>>>(q + (int64_t)v0 * n, t->perm, n, nv, adjoint, qs);
        TRY_X(lm_launch_q_df(qs, n, nv, t->qexp, t->ndf.q, st));
        lm_phase_end(t, PH_PERMUTE, st, 3);
        // step 2: S2M at every leaf, M2M up the levels
        lm_phase_begin(t, PH_S2M, st);
        if (ad) launch_s2m(B, leaves, nleaf, P, k2, t->ndf.rel, t->leaf_start, t->ndf.q, nv, Mof(L), st);
        else launch_s2m(B, gleaves, nleaf, P, k2, t->ndf.rel, t->leaf_start, t->ndf.q, nv, Mof(L), st);
        lm_phase_end(t, PH_S2M, st, 1);
        if (L > 0) lm_phase_begin(t, PH_M2M, st);
        int nl = 0, lm2m = L;
        if (!ad) TRY_X(lm_launch_m2m_oz(t, nv, st, &lm2m, &nl));
        for (int l = lm2m - 1; l >= 0; --l) {
            const int64_t npar = ad ? A.nl_start[l + 1] - A.nl_start[l] : t->lev[l].nbox;
            if (npar == 0) continue;
            if (ad) launch_m2m(ListParents{A.nonleaf + A.nl_start[l], A.child}, npar, P, nv, t->lev[l].m2mdf, Mof(0), Mof(0), st);
            else launch_m2m(GridParents{t->lev[l].ncol}, npar, P, nv, t->lev[l].m2mdf, Mof(l + 1), Mof(l), st);
            ++nl;
        }
        if (L > 0) lm_phase_end(t, PH_M2M, st, nl);
        // step 3: M2L of every level, then L2L down the levels
        lm_phase_begin(t, PH_M2L, st);
        int km = 0;
        TRY_X(lm_launch_m2l_oz(t, nv, st, &km));
        if (t->xdf.nblk > 0) launch_m2l((const M2LLevelDF *)t->xdf.lev, t->xdf.nlev, t->xdf.nblk, P, nv, st);
        lm_phase_end(t, PH_M2L, st, km + (t->xdf.nblk > 0));
        if (L > 0) lm_phase_begin(t, PH_L2L, st);
        nl = 0;
        for (int l = 1; l <= L; ++l) {
            const int64_t npar = ad ? A.nl_start[l] - A.nl_start[l - 1] : t->lev[l - 1].nbox;
            if (npar == 0) continue;
            if (lm_oz_shift(t, l)) {
                int k = 0;
                TRY_X(lm_launch_l2l_oz(t, l, nv, st, &k));
                nl += k;
                continue;
            }
            if (ad) launch_l2l(ListParents{A.nonleaf + A.nl_start[l - 1], A.child}, npar, P, nv, t->lev[l].l2ldf, Lof(0), Lof(0), st);
            else launch_l2l(GridParents{t->lev[l - 1].ncol}, npar, P, nv, t->lev[l].l2ldf, Lof(l - 1), Lof(l), st);
            ++nl;
        }
        if (L > 0) lm_phase_end(t, PH_L2L, st, nl);
        // step 4: L2T and the direct list at every leaf
        lm_phase_begin(t, PH_LEAF, st);
        int nnear = 0;
        if (ux) {
            for (int w0 = 0; w0 < nv; w0 += 4) {
                const int nw = std::min(4, nv - w0);
                const int64_t off = (int64_t)(v0 + w0) * n;
                const L2TOut out{u ? u + off : nullptr, ux + off, uy + off, t->perm};
                if (ad) launch_l2t<true>(B, leaves, nleaf, P, k2, t->ndf.rel, t->leaf_start, Lof(L), nv, w0, nw, t->qexp, n, out, st);
                else launch_l2t<true>(B, gleaves, nleaf, P, k2, t->ndf.rel, t->leaf_start, Lof(L), nv, w0, nw, t->qexp, n, out, st);
                if (t->ndf.ready) TRY_X(lm_launch_near_grad_df(t, nv, w0, nw, out.u, out.ux, out.uy, st));
                else TRY_X(lm_launch_near64(t, w0, nw, out.u, out.ux, out.uy, st));
                nnear += 2;
            }
            lm_phase_end(t, PH_LEAF, st, nnear);
            LM_CUDA(cudaGetLastError());
            continue;
        }
        nnear = ad ? launch_l2t_all(B, leaves, nleaf, P, k2, t->ndf.rel, t->leaf_start, Lof(L), nv, t->qexp, n, t->us, st)
                   : launch_l2t_all(B, gleaves, nleaf, P, k2, t->ndf.rel, t->leaf_start, Lof(L), nv, t->qexp, n, t->us, st);
        int k = 1;
        if (t->ndf.ready) TRY_X(lm_launch_near_df(t, nv, st, &k));
        else TRY_X(lm_launch_near64(t, 0, nv, nullptr, nullptr, nullptr, st));
        lm_phase_end(t, PH_LEAF, st, nnear + k);
        lm_phase_begin(t, PH_PERMUTE, st);
        k_permute_out<<<gridn(n, 256), 256, 0, st>>>(t->us, t->perm, n, nv, adjoint, u + (int64_t)v0 * n);
        lm_phase_end(t, PH_PERMUTE, st, 1);
        LM_CUDA(cudaGetLastError());
    }
    return LM_OK;
}
