// lmfmm_near_df.cu -- direct interactions of the FP64 form in double-float on the
// FP32 pipes: kernel values (free-space H0, the reflected terms' contour tails,
// the factorised segment) and the multiply-adds over the vectors.
//
// GB300 issues an FP64 instruction per warp in 64 slots of a sub-core, against one
// for FP32, so the FP64 leaf kernel spent its time in H0 (28 DFMAs, a log, a
// hypot) and in the tails (48 complex exponentials a pair, about 75 DFMAs each).
// In double-float a free pair takes about 250 FP32 instructions and a tail node
// about 170.  The kernel values carry about 47 bits: one leaf of 60 points is 8e-15 from the IEEE
// form, its gradient 1.3e-14, beside the FMM's own truncation (1e-13 to 1e-10 for p = 24 to 18).
//
// Units: coordinates are scaled by k2/2, so that z = dx^2 + dy^2 = (k2 r / 2)^2 is
// the argument of the ascending series; densities by 2^-qexp, an exponent per vector
// (as the multipoles).
// A kernel value g = g_re + i g_im is kept as (A, J), g_re = -A/(4 pi), g_im = J/4:
// for the free pair A = (ln z + 2 gamma) J + 2 V, J = J0, so the constants are
// applied once per target.  A pair closer than 2^-6 leaf widths takes its offset from the
// FP64 coordinates: the leaf-relative ones are good to 2^-49 of the leaf, an offset of s leaf widths to
// 2^-48 / s, which the gradient shows (with 2^-10 the y-derivative of 3000 points within 0.02 of an interface was 4.5e-13 from
// the IEEE form's, 4.8e-14 now, that of 100k clustered points 8.2e-14, 2.6e-14 now; times the same;
// 2^-4 costs the gradient step 2 %).  Pairs outside the
// series' range (z > 1, or closer than 2^-45 in these units) take the FP64 functions.
#include <algorithm>
#include <type_traits>

#include "df.cuh"
#include "internal.h"
#include "near64.cuh"

static int gridn(int64_t n, int b) { return (int)((n + b - 1) / b); }
__host__ __device__ constexpr int min_i(int a, int b) { return a < b ? a : b; }

// 16 vectors: 256 threads a block, the sums of a row spread over 4 warps (WIDE); else 128
__host__ __device__ constexpr bool nd_wide(int nv, bool grad) { return !grad && nv == 16; }
__host__ __device__ constexpr int nd_threads(int nv, bool grad) { return nd_wide(nv, grad) ? 256 : 128; }
#define ND_ENT 64 // U entries a round
#define ND_SRC 64 // near sources a round
// targets of a block's pass: 16, 8 for the gradient, whose sums take three times the registers; up to 2
// vectors twice as many on large uniform trees whose leaves hold more than that (launch_near)
__host__ __device__ constexpr int nd_tgt(int nv, bool grad) { return grad ? 8 : 16; }

// (A, J) and their z-derivatives (target gradient): A' = J/z + (ln z + 2 gamma) J' + 2 V'
struct HVal {
    df A, J, dA, dJ;
};
template <int D, int T>
__device__ __forceinline__ void h0_df_grad(const DfSmem &tab, df z, HVal *o)
{
    float fj = c_h0df.jh[T - 1], fv = c_h0df.vh[T - 1], gj = (T - 1) * c_h0df.jh[T - 1], gv = (T - 1) * c_h0df.vh[T - 1];
#pragma unroll
    for (int m = T - 2; m >= D; --m) {
        fj = fmaf(fj, z.h, c_h0df.jh[m]);
        fv = fmaf(fv, z.h, c_h0df.vh[m]);
        gj = fmaf(gj, z.h, m * c_h0df.jh[m]);
        gv = fmaf(gv, z.h, m * c_h0df.vh[m]);
    }
    df j = {fj, 0.f}, v = {fv, 0.f}, dj = {gj, 0.f}, dv = {gv, 0.f};
#pragma unroll
    for (int m = D - 1; m >= 0; --m) {
        const df cj = {c_h0df.jh[m], c_h0df.jl[m]}, cv = {c_h0df.vh[m], c_h0df.vl[m]};
        j = df_horner(cj, z, j);
        if (m >= 1) {
            v = df_horner(cv, z, v);
            dj = df_horner(df_mulf(cj, (float)m), z, dj);
            dv = df_horner(df_mulf(cv, (float)m), z, dv);
        }
    }
    const df lz = df_add(df_log(tab, z), df{1.1544313f, -1.3275548e-08f});
    const df b = df_mul(z, v);
    o->A = df_add(df_mul(lz, j), df{2.f * b.h, 2.f * b.l});
    o->J = j;
    // J / z by one correction step
    const float q0 = j.h / z.h;
    const df r = df_sub(j, df_mulf(z, q0));
    const df jz = quick_two_sum(q0, (r.h + r.l) / z.h);
    o->dA = df_add(df_add(jz, df{2.f * dv.h, 2.f * dv.l}), df_mul(lz, dj));
    o->dJ = dj;
}
__device__ __noinline__ void h0_slow_grad(double x, HVal *o)
{
    zd g, g1;
    h01_free64(x, &g, &g1);
    const double c = -2.0 / x; // d/dz = (dx/dz) d/dx, z = x^2/4; d/dx H0 = -H1
    o->A = df_of(-4.0 * M_PI * g.re);
    o->J = df_of(4.0 * g.im);
    o->dA = df_of(-4.0 * M_PI * c * g1.re);
    o->dJ = df_of(4.0 * c * g1.im);
}
// ---------------------------------------------------------------------------
// Tables
// ---------------------------------------------------------------------------
// a node as (X and h or Y coefficients of the exponent, then of the phase), in df_cexp's units
__device__ __forceinline__ void put_node(float4 *o, double ex, double ey, double px, double py)
{
    const double u = 64.0 / 0.693147180559945309417, v = 256.0 / 6.283185307179586476925;
    const df a = df_of(ex * u), b = df_of(ey * u), c = df_of(px * v), d = df_of(py * v);
    o[0] = make_float4(a.h, a.l, b.h, b.l);
    o[1] = make_float4(c.h, c.l, d.h, d.l);
}
// tail nodes: e^{i lambda X - s2 h} in X, h scaled by kap; weights P Re(E) + i M Im(E) as (A, J)
__global__ void k_tail_tab(int tot, double kap, const zd *lam, const zd *s2, const zd *w, float4 *node, float4 *wt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= tot) return;
    const zd l = lam[i], s = s2[i];
    if (node) put_node(node + 2 * i, -l.im / kap, -s.re / kap, l.re / kap, -s.im / kap);
    for (int m = 0; w && m < 2; ++m) {
        const zd P = w[(int64_t)(2 * m) * tot + i], M = w[(int64_t)(2 * m + 1) * tot + i];
        const df a = df_of(-4.0 * M_PI * P.re), b = df_of(4.0 * M_PI * M.im), c = df_of(4.0 * P.im), d = df_of(4.0 * M.re);
        wt[2 * ((int64_t)m * tot + i)] = make_float4(a.h, a.l, b.h, b.l);
        wt[2 * ((int64_t)m * tot + i) + 1] = make_float4(c.h, c.l, d.h, d.l);
    }
}
// segment nodes: e^{i lambda X + s2 Y}, and their weights
__global__ void k_seg_tab(int nseg, double kap, const zd *lam, const zd *s2, const zd *w, float4 *node, float4 *wt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nseg) return;
    const zd l = lam[i], s = s2[i];
    put_node(node + 2 * i, -l.im / kap, s.re / kap, l.re / kap, s.im / kap);
    for (int m = 0; m < 2; ++m) wt[m * nseg + i] = df_split(w[m * nseg + i]);
}
// The target gradient's tail weights: with E = e^{i lambda X - s2 h} the value, d/dX and d/dh
// are P Re(f E) + i M Im(f E), f = 1, i lambda, -s2, written as weights of Re E and Im E; c
// (or null): the part of P, M that the h-derivative leaves out (see near_refl64_grad).
// wt: [term][node][6]: A of the three, then J of the three
__global__ void k_tail_tab_grad(int tot, const zd *lam, const zd *s2, const zd *w, const zd *c, float4 *wt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= tot) return;
    for (int m = 0; m < 2; ++m)
        for (int k = 0; k < 3; ++k) {
            const zd f = k == 0 ? zd{1.0, 0.0} : k == 1 ? zd{-lam[i].im, lam[i].re} : -s2[i];
            zd P = w[(int64_t)(2 * m) * tot + i], M = w[(int64_t)(2 * m + 1) * tot + i];
            if (k == 2 && c) {
                P = P - c[(int64_t)(2 * m) * tot + i];
                M = M - c[(int64_t)(2 * m + 1) * tot + i];
            }
            const zd iM = {-M.im, M.re};
            // Re(f E) = f.re E.re - f.im E.im, Im(f E) = f.im E.re + f.re E.im
            const zd wr = f.re * P + f.im * iM, wi = f.re * iM - f.im * P;
            float4 *o = wt + 6 * ((int64_t)m * tot + i);
            o[k] = df_pack(df_of(-4.0 * M_PI * wr.re), df_of(-4.0 * M_PI * wi.re));
            o[3 + k] = df_pack(df_of(4.0 * wr.im), df_of(4.0 * wi.im));
        }
}
// segment weights of the gradient: W, i lambda W, -s2 (W - c); [term][node][3]
__global__ void k_seg_tab_grad(int nseg, const zd *lam, const zd *s2, const zd *w, const zd *c, float4 *wt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nseg) return;
    for (int m = 0; m < 2; ++m) {
        const zd W = w[m * nseg + i], l = lam[i];
        float4 *o = wt + 3 * (m * nseg + i);
        o[0] = df_split(W);
        o[1] = df_split(zd{-l.im, l.re} * W);
        o[2] = df_split(-(s2[i] * (c ? W - c[m * nseg + i] : W)));
    }
}
// points of the leaf boxes: offset from the box centre, and heights y and y + d, scaled by kap
template <class Geo>
__global__ void k_near_pts(Geo geo, double kap, double d, const double *xs, const double *ys, const int64_t *ls,
                           float4 *rel, float4 *hgt)
{
    const int64_t b = geo.id(blockIdx.x);
    double cx, cy, w;
    geo.centre(b, &cx, &cy, &w);
    for (int64_t i = ls[b] + threadIdx.x; i < ls[b + 1]; i += blockDim.x) {
        const df a = df_of((xs[i] - cx) * kap), c = df_of((ys[i] - cy) * kap);
        rel[i] = df_pack(a, c);
        hgt[i] = df_pack(df_of(ys[i] * kap), df_of((ys[i] + d) * kap));
    }
}

// densities in tree order [nvec][n] -> double-float [n][nvec], scaled by 2^-qexp[vector]
__global__ void k_q_df(const zd *qs, int64_t n, int nvec, const int *qexp, float4 *q)
{
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= n * nvec) return;
    const int64_t i = idx / nvec;
    const int v = (int)(idx % nvec), e = -qexp_of(qexp, v);
    const zd a = qs[(int64_t)v * n + i];
    q[idx] = df_split(zd{ldexp(a.re, e), ldexp(a.im, e)});
}

// ---------------------------------------------------------------------------
// Pairs
// ---------------------------------------------------------------------------
struct NearDF {
    int nray, ntail, cplx, a_zero;
    const float4 *node, *w, *w2; // tail nodes and weights (w2: multiple reflections between two walls, or null)
    df d2;                       // 2d scaled: the multiple reflections' extra height
    float hray;                  // added to h when the ray is chosen (see NearQuad)
    double rinf[2];
    // target gradient: segment nodes and weights (a pair's own; the apply factorises it), beta per wall
    int nseg;
    const float4 *seg, *segw_g;
    double beta[2];
};
struct GradOut { // GRAD: outputs in input order through perm
    zd *u, *ux, *uy;
    const int64_t *perm;
    int v0; // first vector of the launch
};
__device__ __forceinline__ int ray_of(const NearDF &q, float X, float h)
{
    return q.nray > 1 ? (int)rintf(atan2f(X, h) * (float)(q.nray - 1) * 0.63661977f) : 0;
}
// x X + y Y of a node's two coefficients
__device__ __forceinline__ df dot2(float4 c, df X, df Y)
{
    df s = df_mul_raw(df{c.x, c.y}, X);
    df_mac(s.h, s.l, c.z, c.w, Y.h, Y.l);
    return quick_two_sum(s.h, s.l);
}
__device__ __noinline__ void tail_df(const DfSmem &tab, const NearDF &q, const float4 *w, int ray, df X, df h, df *A, df *J)
{
    const float4 *nd = q.node + 2 * (int64_t)ray * q.ntail, *wt = w + 2 * (int64_t)ray * q.ntail;
    df a = *A, j = *J;
    for (int i = 0; i < q.ntail; ++i) {
        const float4 e = df_cexp(tab, dot2(nd[2 * i], X, h), dot2(nd[2 * i + 1], X, h));
        const float4 p = wt[2 * i];
        df_mac(a, df_re(e), df_re(p));
        df_mac(a, df_im(e), df_im(p));
        if (q.cplx) {
            const float4 r = wt[2 * i + 1];
            df_mac(j, df_re(e), df_re(r));
            df_mac(j, df_im(e), df_im(r));
        }
    }
    *A = quick_two_sum(a.h, a.l);
    *J = quick_two_sum(j.h, j.l);
}

// value, d/dX and d/dh of a reflected pair: A and J of each
struct GradVal {
    df A[3], J[3];
};
__device__ __noinline__ void tail_df_grad(const DfSmem &tab, const NearDF &q, const float4 *w, int ray, df X, df h, GradVal *o)
{
    const float4 *nd = q.node + 2 * (int64_t)ray * q.ntail, *wt = w + 6 * (int64_t)ray * q.ntail;
    GradVal s = *o;
    for (int i = 0; i < q.ntail; ++i) {
        const float4 e = df_cexp(tab, dot2(nd[2 * i], X, h), dot2(nd[2 * i + 1], X, h));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float4 p = wt[6 * i + k];
            df_mac(s.A[k], df_re(e), df_re(p));
            df_mac(s.A[k], df_im(e), df_im(p));
            if (q.cplx) {
                const float4 r = wt[6 * i + 3 + k];
                df_mac(s.J[k], df_re(e), df_re(r));
                df_mac(s.J[k], df_im(e), df_im(r));
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        o->A[k] = quick_two_sum(s.A[k].h, s.A[k].l);
        o->J[k] = quick_two_sum(s.J[k].h, s.J[k].l);
    }
}
__device__ __noinline__ void seg_df_grad(const DfSmem &tab, const NearDF &q, int m, df X, df h, GradVal *o)
{
    float4 s[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) s[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    const df Y = df_neg(h), Xn = df_neg(X);
    for (int i = 0; i < q.nseg; ++i) {
        const float4 *nd = q.seg + 2 * i, *w = q.segw_g + 3 * (m * q.nseg + i);
        const float4 e1 = df_cexp(tab, dot2(nd[0], X, Y), dot2(nd[1], X, Y));
        const float4 e2 = df_cexp(tab, dot2(nd[0], Xn, Y), dot2(nd[1], Xn, Y));
        const float4 ep = dfc_add(e1, e2), em = dfc_add(e1, make_float4(-e2.x, -e2.y, -e2.z, -e2.w));
        dfc_mac(s[0], w[0], ep);
        dfc_mac(s[1], w[1], em);
        dfc_mac(s[2], w[2], ep);
    }
    const df cA = {-12.566371f, 3.496911e-07f}; // -4 pi
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        o->A[k] = df_mul(quick_two_sum(s[k].x, s[k].y), cA);
        const df im = quick_two_sum(s[k].z, s[k].w);
        o->J[k] = df{4.f * im.h, 4.f * im.l};
    }
}

// A pair of points at the same place: the kernel is infinite, which no double-float sum holds (inf - inf in its error
// terms).  What FP64 gives, an infinity with the density's sign (not a number for the derivatives), goes to the output
// at once; the block adds its finite sums to it later.
__device__ __noinline__ void add_coincident(const float4 *q, int nv, int64_t n, int64_t i, zd *u, zd *ux, zd *uy)
{
    for (int v = 0; v < nv; ++v) {
        const int64_t k = (int64_t)v * n + i;
        if (u) {
            atomicAdd(&u[k].re, INFINITY * df_double(df_re(q[v])));
            atomicAdd(&u[k].im, INFINITY * df_double(df_im(q[v])));
        }
        if (ux) ux[k] = uy[k] = zd{NAN, NAN};
    }
}

// One block: up to tb targets of a leaf at a time against the leaf's flattened near
// sources.  Round: 64 sources staged (coordinates in the target leaf's frame,
// densities), the kernel values of all (target, source) pairs evaluated a lane per
// source into shared memory, then summed with a lane per (source subset, vector).
// Bound by FP32 issue (free pairs about 250 instructions, tails 170 per node, 48
// per complex multiply-add), half of whose slots go to the barriers between the rounds
// and instruction fetch.  200k uniform points, 1 vector: 0.46 ms (6.1 ms in FP64);
// 250k strip, 16 vectors: 2.19 ms (16.6 ms).
template <int NV, int D, int T, bool GRAD, int TG, class Geo>
__global__ void __launch_bounds__(nd_threads(NV, GRAD), GRAD ? 3 : 512 / nd_threads(NV, GRAD))
    k_near_df(Geo geo, double k, double kap, const double *xs, const double *ys, const int64_t *ls, const float4 *rel,
              const float4 *hgt, const int64_t *ustart, const int32_t *usrc, const int32_t *uterm, NearDF nq,
              const float4 *qd, int nvq, const int *qexp, int64_t n, int nv, int tb, int free_on, zd *us, GradOut go)
{
    constexpr int SETS = GRAD ? 3 : 1, SRC = GRAD ? 32 : ND_SRC, THR = nd_threads(NV, GRAD);
    __shared__ DfSmem tab;
    __shared__ int64_t fj0[ND_ENT];
    __shared__ int fpre[ND_ENT + 1], fterm[ND_ENT];
    __shared__ float4 foff[ND_ENT];
    __shared__ float4 sp[SRC], tr[TG], th[TG];
    __shared__ int64_t sj[SRC];
    __shared__ int st[SRC];
    __shared__ float4 g[SETS][TG][SRC];
    float4 *ur = &g[0][0][0];      // [TG][SETS][2 NV]: the sums, once the values are done with
    extern __shared__ float4 sq[]; // [SRC][NV]
    const int64_t b = geo.id(blockIdx.x);
    const int64_t lo = ls[b], hi = ls[b + 1];
    if (lo + (int64_t)blockIdx.y * tb >= hi) return;
    tab.load();
    double cx, cy, bw;
    geo.centre(b, &cx, &cy, &bw);
    const float zclose = (float)(kap * kap * bw * bw) * 0x1p-12f; // pairs closer than 2^-6 leaf widths
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t u0 = ustart[b], u1 = ustart[b + 1];
    constexpr int ROWS = TG / (THR / 32), HALF = SRC / 32;
    // Sums over the sources: 8 interleaved subsets whatever the number of vectors, added in the same
    // order, so that a vector's result does not depend on how many others are applied with it.  A lane
    // holds ACC subsets of vector v for LR of its warp's ROWS rows; WIDE (16 vectors): one subset of every
    // second row, so that a leaf's rows are spread evenly over the warps whatever their number and a
    // density is read once for up to 8 rows.
    constexpr bool WIDE = nd_wide(NV, GRAD);
    constexpr int SUB = 8, ACC = WIDE ? 1 : NV * SUB > 32 ? NV * SUB / 32 : 1, LS = WIDE ? 2 : SUB / ACC,
                  RSTEP = WIDE ? 1 : min_i(ROWS, 32 / (NV * LS));
    constexpr int LR = WIDE ? TG / 2 : ROWS / RSTEP;
    const int v = lane % NV, sub = (lane / NV) % LS, rh = lane / (NV * LS);
    const int wg = warp & 3, wr = warp >> 2; // WIDE: subsets 2 wg + sub, rows wr + 2 r
    const bool on = rh < RSTEP; // one vector, 8 targets a pass: half the lanes have no row
    for (int64_t t0 = lo + (int64_t)blockIdx.y * tb; t0 < hi; t0 += (int64_t)gridDim.y * tb) {
        const int nt = (int)min((int64_t)tb, hi - t0);
        float4 acA[SETS][LR][ACC], acJ[SETS][LR][ACC]; // sums of A q and J q (complex)
#pragma unroll
        for (int c = 0; c < SETS; ++c)
#pragma unroll
            for (int r = 0; r < LR; ++r)
#pragma unroll
                for (int a = 0; a < ACC; ++a) acA[c][r][a] = acJ[c][r][a] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        if (tid < nt) {
            tr[tid] = rel[t0 + tid];
            th[tid] = hgt[t0 + tid];
        }
        for (int64_t c0 = u0; c0 < u1; c0 += ND_ENT) {
            const int nc = (int)min((int64_t)ND_ENT, u1 - c0);
            __syncthreads(); // the previous entries' sources are done
            int cnt = 0;
            if (tid < nc) {
                const int32_t s = usrc[c0 + tid], term = uterm[c0 + tid];
                const int64_t j0 = ls[s];
                fj0[tid] = j0;
                fterm[tid] = term;
                cnt = (term == 0 && !free_on) ? 0 : (int)(ls[s + 1] - j0);
                double sx, sy, sw;
                geo.centre(s, &sx, &sy, &sw);
                foff[tid] = df_pack(df_of((sx - cx) * kap), df_of((sy - cy) * kap));
            }
            if (tid < ND_ENT) { // inclusive scan of the counts (two warps)
                for (int o = 1; o < 32; o <<= 1) {
                    const int x = __shfl_up_sync(0xffffffffu, cnt, o);
                    if (lane >= o) cnt += x;
                }
                fpre[tid + 1] = cnt;
            }
            if (tid == 0) fpre[0] = 0;
            __syncthreads();
            if (tid >= 32 && tid < ND_ENT) fpre[tid + 1] += fpre[32];
            __syncthreads();
            const int tot = fpre[nc];
            for (int f0 = 0; f0 < tot; f0 += SRC) {
                const int ns = min(SRC, tot - f0);
                if (tid < ns) {
                    const int f = f0 + tid;
                    int e = 0; // the entry holding source f
#pragma unroll
                    for (int o = ND_ENT / 2; o > 0; o >>= 1)
                        if (e + o < nc && fpre[e + o] <= f) e += o;
                    const int64_t j = fj0[e] + (f - fpre[e]);
                    const int term = fterm[e];
                    const float4 p = rel[j], of = foff[e];
                    const df x = df_add(df_re(p), df_re(of));
                    const float4 hh = hgt[j];
                    // free: y in the target leaf's frame; tt: y; bb: y + d
                    const df y = term == 0 ? df_add(df_im(p), df_im(of)) : (term == 1 ? df_re(hh) : df_im(hh));
                    sp[tid] = df_pack(x, y);
                    sj[tid] = j;
                    st[tid] = term;
                }
                if (nv < NV)
                    for (int i = tid; i < SRC * NV; i += THR) sq[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                __syncthreads();
                for (int i = tid; i < ns * nv; i += THR) {
                    const int s = i / nv, vv = i - s * nv;
                    sq[s * NV + vv] = qd[sj[s] * nvq + go.v0 + vv];
                }
                for (int it = warp; it < HALF * nt; it += THR / 32) {
                    const int row = it / HALF, s = (it % HALF) * 32 + lane;
                    if (s >= ns) continue;
                    const float4 tp = tr[row], p = sp[s];
                    const int term = st[s];
                    df dx = df_sub(df_re(tp), df_re(p));
                    GradVal G; // [1..]: d/dx, d/dy (GRAD)
#pragma unroll
                    for (int c = 0; c < 3; ++c) G.A[c] = G.J[c] = df{0.f, 0.f};
                    if (term == 0) {
                        if (sj[s] != t0 + row) {
                            df dy = df_sub(df_im(tp), df_im(p));
                            df z = df_add(df_sq(dx), df_sq(dy));
                            if (z.h < zclose) {
                                dx = df_of((xs[t0 + row] - xs[sj[s]]) * kap);
                                dy = df_of((ys[t0 + row] - ys[sj[s]]) * kap);
                                z = df_add(df_sq(dx), df_sq(dy));
                            }
                            const bool slow = z.h > 1.0f || z.h < ND_TINY;
                            if (slow && xs[t0 + row] == xs[sj[s]] && ys[t0 + row] == ys[sj[s]])
                                add_coincident(qd + sj[s] * nvq + go.v0, nv, n, GRAD ? go.perm[t0 + row] : t0 + row,
                                               GRAD ? go.u : us, GRAD ? go.ux : nullptr, GRAD ? go.uy : nullptr);
                            else if (GRAD) {
                                HVal H;
                                if (slow) h0_slow_grad(k * hypot(xs[t0 + row] - xs[sj[s]], ys[t0 + row] - ys[sj[s]]), &H);
                                else h0_df_grad<D, T>(tab, z, &H);
                                const float f = (float)(2.0 * kap), fl = (float)(2.0 * kap - (double)f);
                                const df ex = df_mul(dx, df{f, fl}), ey = df_mul(dy, df{f, fl}); // dz/dx, dz/dy
                                G.A[0] = H.A, G.J[0] = H.J;
                                G.A[1] = df_mul(H.dA, ex), G.J[1] = df_mul(H.dJ, ex);
                                G.A[2] = df_mul(H.dA, ey), G.J[2] = df_mul(H.dJ, ey);
                            } else if (slow)
                                h0_slow(k * hypot(xs[t0 + row] - xs[sj[s]], ys[t0 + row] - ys[sj[s]]), &G.A[0], &G.J[0]);
                            else
                                h0_df<D, T>(tab, z, &G.A[0], &G.J[0]);
                        }
                    } else {
                        const int m = term - 1;
                        const float4 hh = th[row];
                        df h = df_add(m == 0 ? df_re(hh) : df_im(hh), df_im(p));
                        if (m == 0) h = df_neg(h); // tt: -(y + y0); bb: (y + d) + (y0 + d)
                        if (dx.h * dx.h + h.h * h.h < zclose) dx = df_of((xs[t0 + row] - xs[sj[s]]) * kap);
                        const df X = dx.h < 0.f ? df_neg(dx) : dx;
                        const int64_t wo = (int64_t)m * (GRAD ? 6 : 2) * nq.nray * nq.ntail;
                        if (GRAD) seg_df_grad(tab, nq, m, X, h, &G);
                        auto tail = [&](const float4 *w, float hr) {
                            if (GRAD) tail_df_grad(tab, nq, w + wo, ray_of(nq, X.h, hr), X, h, &G);
                            else tail_df(tab, nq, w + wo, ray_of(nq, X.h, hr), X, h, &G.A[0], &G.J[0]);
                        };
                        if (nq.w2) {
                            if (!nq.a_zero) tail(nq.w, h.h);
                            tail(nq.w2, h.h + nq.d2.h);
                        } else
                            tail(nq.w, h.h + nq.hray);
                        const float ri = (float)nq.rinf[m]; // 0, 1 or -1
                        if (ri != 0.f) { // the wall's image in closed form
                            const df z = df_add(df_sq(X), df_sq(h));
                            const bool slow = z.h > 1.0f || z.h < ND_TINY;
                            HVal H;
                            const double x = slow ? 2.0 * hypot(df_double(X), df_double(h)) : 0.0;
                            if (GRAD) {
                                if (slow) h0_slow_grad(x, &H);
                                else h0_df_grad<D, T>(tab, z, &H);
                                const df f2 = df_of(2.0 * kap * nq.rinf[m]);
                                const df ex = df_mul(X, f2), eh = df_mul(h, f2);
                                G.A[1] = df_add(G.A[1], df_mul(H.dA, ex)), G.J[1] = df_add(G.J[1], df_mul(H.dJ, ex));
                                G.A[2] = df_add(G.A[2], df_mul(H.dA, eh)), G.J[2] = df_add(G.J[2], df_mul(H.dJ, eh));
                                if (nq.beta[m] != 0.0) { // -2 i beta (i/4) H0 of the h-derivative's closed form
                                    G.A[2] = df_add(G.A[2], df_mul(H.J, df_of(-2.0 * M_PI * nq.beta[m])));
                                    G.J[2] = df_add(G.J[2], df_mul(H.A, df_of(2.0 / M_PI * nq.beta[m])));
                                }
                            } else if (slow)
                                h0_slow(x, &H.A, &H.J);
                            else
                                h0_df<D, T>(tab, z, &H.A, &H.J);
                            G.A[0] = df_add(G.A[0], df{ri * H.A.h, ri * H.A.l});
                            G.J[0] = df_add(G.J[0], df{ri * H.J.h, ri * H.J.l});
                        }
                        if (GRAD) { // d/dx = sign(x - x0) d/dX, d/dy = -d/dh (tt), d/dh (bb)
                            const float sx = dx.h > 0.f ? 1.f : (dx.h < 0.f ? -1.f : 0.f), sy = m == 0 ? -1.f : 1.f;
                            G.A[1] = df{sx * G.A[1].h, sx * G.A[1].l}, G.J[1] = df{sx * G.J[1].h, sx * G.J[1].l};
                            G.A[2] = df{sy * G.A[2].h, sy * G.A[2].l}, G.J[2] = df{sy * G.J[2].h, sy * G.J[2].l};
                        }
                    }
#pragma unroll
                    for (int c = 0; c < SETS; ++c) g[c][row][s] = df_pack(G.A[c], G.J[c]);
                }
                __syncthreads();
                if (WIDE) {
                    for (int s0 = 2 * wg; s0 < ns; s0 += SUB) {
                        const bool in = s0 + sub < ns;
                        const int s = in ? s0 + sub : s0;
                        const float4 q = in ? sq[s * NV + v] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int r = 0; r < LR; ++r)
                            if (wr + 2 * r < nt) {
                                const float4 gg = g[0][wr + 2 * r][s];
                                float4 &x = acA[0][r][0], &y = acJ[0][r][0];
                                df_mac(x.x, x.y, gg.x, gg.y, q.x, q.y);
                                df_mac(x.z, x.w, gg.x, gg.y, q.z, q.w);
                                df_mac(y.x, y.y, gg.z, gg.w, q.x, q.y);
                                df_mac(y.z, y.w, gg.z, gg.w, q.z, q.w);
                            }
                    }
                } else
#pragma unroll
                for (int r = 0; r < LR; ++r) {
                    const int row = warp + (r * RSTEP + rh) * (THR / 32);
                    if (on && row < nt)
                        for (int s0 = 0; s0 < ns; s0 += SUB)
#pragma unroll
                            for (int a = 0; a < ACC; ++a) {
                                const int s = s0 + sub + a * LS;
                                if (s >= ns) continue;
                                const float4 q = sq[s * NV + v];
#pragma unroll
                                for (int c = 0; c < SETS; ++c) {
                                    const float4 gg = g[c][row][s];
                                    float4 &x = acA[c][r][a], &y = acJ[c][r][a];
                                    df_mac(x.x, x.y, gg.x, gg.y, q.x, q.y);
                                    df_mac(x.z, x.w, gg.x, gg.y, q.z, q.w);
                                    df_mac(y.x, y.y, gg.z, gg.w, q.x, q.y);
                                    df_mac(y.z, y.w, gg.z, gg.w, q.z, q.w);
                                }
                            }
                }
                __syncthreads(); // sources and values are overwritten by the next round
            }
        }
        // the subsets' sums: neighbours first
        if (WIDE) {
#pragma unroll
            for (int r = 0; r < LR; ++r) {
                const int row = wr + 2 * r;
                if (row >= nt) break;
                float4 a = df_norm(acA[0][r][0]), j = df_norm(acJ[0][r][0]);
                a = dfc_add(a, shfl4(a, NV));
                j = dfc_add(j, shfl4(j, NV));
                if (sub == 0) {
                    ur[(row * 4 + wg) * NV + v] = a;
                    sq[(row * 4 + wg) * NV + v] = j;
                }
            }
        } else
#pragma unroll
        for (int r = 0; r < LR; ++r) {
            const int row = warp + (r * RSTEP + rh) * (THR / 32);
#pragma unroll
            for (int c = 0; c < SETS; ++c) {
                float4 x[ACC], y[ACC];
#pragma unroll
                for (int i = 0; i < ACC; ++i) {
                    x[i] = df_norm(acA[c][r][i]), y[i] = df_norm(acJ[c][r][i]);
#pragma unroll
                    for (int o = NV; o < NV * LS; o <<= 1) {
                        x[i] = dfc_add(x[i], shfl4(x[i], o));
                        y[i] = dfc_add(y[i], shfl4(y[i], o));
                    }
                }
#pragma unroll
                for (int h = 1; h < ACC; h <<= 1)
#pragma unroll
                    for (int i = 0; i < ACC; i += 2 * h) x[i] = dfc_add(x[i], x[i + h]), y[i] = dfc_add(y[i], y[i + h]);
                if (on && row < nt && sub == 0) {
                    ur[((row * SETS + c) * NV + v) * 2] = x[0];
                    ur[((row * SETS + c) * NV + v) * 2 + 1] = y[0];
                }
            }
        }
        __syncthreads();
        for (int i = tid; i < nt * nv * SETS; i += THR) {
            const int row = i % nt, vc = i / nt, vv = vc % nv, c = vc / nv;
            float4 a, j;
            if (WIDE) {
                const float4 *pa = ur + row * 4 * NV + vv, *pj = sq + row * 4 * NV + vv;
                a = dfc_add(dfc_add(pa[0], pa[NV]), dfc_add(pa[2 * NV], pa[3 * NV]));
                j = dfc_add(dfc_add(pj[0], pj[NV]), dfc_add(pj[2 * NV], pj[3 * NV]));
            } else {
                a = ur[((row * SETS + c) * NV + vv) * 2];
                j = ur[((row * SETS + c) * NV + vv) * 2 + 1];
            }
            const double f = -1.0 / (4.0 * M_PI);
            zd r = {f * df_double(df_re(a)) - 0.25 * df_double(df_im(j)), f * df_double(df_im(a)) + 0.25 * df_double(df_re(j))};
            const int ex = qexp_of(qexp, go.v0 + vv);
            r = zd{ldexp(r.re, ex), ldexp(r.im, ex)};
            if (GRAD) {
                zd *o = c == 0 ? go.u : c == 1 ? go.ux : go.uy;
                if (o) {
                    zd &w = o[(int64_t)vv * n + go.perm[t0 + row]];
                    w = zd{__ldcg(&w.re), __ldcg(&w.im)} + r;
                }
            } else { // (past L1, for add_coincident's atomics)
                zd &o = us[(int64_t)vv * n + t0 + row];
                o = zd{__ldcg(&o.re), __ldcg(&o.im)} + r;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// The factorised segment of the reflected terms (see k_pw_src64 and k_near_pw64 for
// the factorisation): a source leaf's coefficients C, then per target leaf the sum
// B over its U entries and its evaluation.
// ---------------------------------------------------------------------------
// e^{s i lambda x + s2 Y}, Y = y (tt) or -(y + d) (bb)
__device__ __forceinline__ float4 seg_exp(const DfSmem &tab, const float4 *nd, float sg, df x, df Y)
{
    const df sx = {sg * x.h, sg * x.l};
    return df_cexp(tab, dot2(nd[0], sx, Y), dot2(nd[1], sx, Y));
}
__device__ __forceinline__ df seg_height(int m, float4 h) { return m == 0 ? df_re(h) : df_neg(df_im(h)); }

template <int NV, class Geo>
__global__ void __launch_bounds__(256) k_pw_src_df(Geo geo, int nseg, const float4 *node, const float4 *rel,
                                                   const float4 *hgt, const int64_t *ls, const int64_t *ustart,
                                                   const int32_t *uterm, const float4 *qd, int nv, float4 *C)
{
    __shared__ DfSmem tab;
    __shared__ int any[2];
    const int nk = 2 * nseg;
    const int64_t slot = blockIdx.x, b = geo.id(slot);
    if (ls[b + 1] == ls[b]) return; // an empty leaf: its coefficients are never read
    tab.load();
    if (threadIdx.x < 2) any[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t e = ustart[b] + threadIdx.x; e < ustart[b + 1]; e += blockDim.x)
        if (uterm[e] > 0) any[uterm[e] - 1] = 1;
    __syncthreads();
    for (int m = 0; m < 2; ++m) {
        if (!any[m]) continue;
        float4 *Cm = C + (slot * 2 + m) * nk * nv;
        for (int k = threadIdx.x; k < nk; k += blockDim.x) {
            const float sg = (k & 1) ? 1.f : -1.f; // -s
            float4 acc[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int64_t j = ls[b]; j < ls[b + 1]; ++j) {
                const float4 f = seg_exp(tab, node + (k & ~1), sg, df_re(rel[j]), seg_height(m, hgt[j]));
#pragma unroll
                for (int v = 0; v < NV; ++v)
                    if (v < nv) dfc_mac(acc[v], f, qd[j * nv + v]);
            }
#pragma unroll
            for (int v = 0; v < NV; ++v)
                if (v < nv) Cm[k * nv + v] = df_pack(quick_two_sum(acc[v].x, acc[v].y), quick_two_sum(acc[v].z, acc[v].w));
        }
    }
}

#define PW_WARPS 8 // of a block of k_near_pw_df
template <int NV, class Geo>
__global__ void __launch_bounds__(32 * PW_WARPS) k_near_pw_df(Geo geo, double kap, int nseg, const float4 *node, const float4 *wt,
                                                    const float4 *rel, const float4 *hgt, const int64_t *ls,
                                                    const int64_t *ustart, const int32_t *usrc, const int32_t *uterm,
                                                    const float4 *C, const int32_t *pwidx, const int *qexp, int64_t n,
                                                    int nv, zd *us)
{
    __shared__ DfSmem tab;
    __shared__ float4 ur[PW_WARPS][NV];
    extern __shared__ float4 B[]; // [nk][nv]
    const int nk = 2 * nseg;
    const int64_t b = geo.id(blockIdx.x), lo = ls[b], hi = ls[b + 1];
    if (hi == lo) return; // no targets
    tab.load();
    double xT, yT, wT;
    geo.centre(b, &xT, &yT, &wT);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    for (int m = 0; m < 2; ++m) {
        __syncthreads(); // tables loaded, the previous term's B done
        bool any = false;
        for (int k = threadIdx.x; k < nk; k += blockDim.x) // a thread owns its B[k]
            for (int v = 0; v < nv; ++v) B[k * nv + v] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int64_t e = ustart[b]; e < ustart[b + 1]; ++e) {
            if (uterm[e] != m + 1) continue;
            const int64_t s = usrc[e];
            if (ls[s + 1] == ls[s]) continue; // no sources (uniform over the block)
            any = true;
            double cs, ysc, wsc;
            geo.centre(s, &cs, &ysc, &wsc);
            const df dx = df_of((cs - xT) * kap);
            const float4 *Cs = C + ((int64_t)pwidx[s] * 2 + m) * nk * nv;
            for (int k = threadIdx.x; k < nk; k += blockDim.x) {
                const float sg = (k & 1) ? 1.f : -1.f; // -s
                const float4 f = seg_exp(tab, node + (k & ~1), sg, dx, df{0.f, 0.f});
                for (int v = 0; v < nv; ++v) dfc_mac(B[k * nv + v], f, Cs[k * nv + v]);
            }
        }
        if (!any) continue; // block-uniform
        for (int k = threadIdx.x; k < nk; k += blockDim.x)
            for (int v = 0; v < nv; ++v) B[k * nv + v] = dfc_mul(wt[m * nseg + (k >> 1)], B[k * nv + v]);
        __syncthreads();
        for (int64_t i0 = lo; i0 < hi; i0 += nwarp) { // a warp per target, lanes over the nodes
            const int64_t i = i0 + warp;
            if (i < hi) {
                float4 acc[NV];
#pragma unroll
                for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
                const df x = df_re(rel[i]), Y = seg_height(m, hgt[i]);
                for (int k = lane; k < nk; k += 32) {
                    const float4 f = seg_exp(tab, node + (k & ~1), (k & 1) ? -1.f : 1.f, x, Y);
#pragma unroll
                    for (int v = 0; v < NV; ++v)
                        if (v < nv) dfc_mac(acc[v], f, B[k * nv + v]);
                }
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const df re = df_warp_sum(df_re(acc[v])), im = df_warp_sum(df_im(acc[v]));
                    if (lane == v) ur[warp][v] = df_pack(re, im);
                }
            }
            __syncthreads();
            const int cnt = (int)min((int64_t)nwarp, hi - i0);
            for (int t = threadIdx.x; t < cnt * nv; t += blockDim.x) {
                const float4 a = ur[t % cnt][t / cnt];
                const int ex = qexp_of(qexp, t / cnt);
                zd &o = us[(int64_t)(t / cnt) * n + i0 + t % cnt];
                o = o + zd{ldexp(df_double(df_re(a)), ex), ldexp(df_double(df_im(a)), ex)};
            }
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
static int nv_slots(int nv) { return nv <= 1 ? 1 : nv <= 2 ? 2 : nv <= 4 ? 4 : nv <= 8 ? 8 : 16; }
#define NV_DISPATCH(nv, ...)                                  \
    switch (nv_slots(nv)) {                                   \
    case 1: { constexpr int NV = 1; __VA_ARGS__; } break;     \
    case 2: { constexpr int NV = 2; __VA_ARGS__; } break;     \
    case 4: { constexpr int NV = 4; __VA_ARGS__; } break;     \
    case 8: { constexpr int NV = 8; __VA_ARGS__; } break;     \
    default: { constexpr int NV = 16; __VA_ARGS__; } break;   \
    }

lm_status lm_setup_near_df(lm_tree_s *t, cudaStream_t st)
{
    NearTabDF &N = t->ndf;
    N.ready = false;
    const NearQuad &q = t->nq;
    const double kap = 0.5 * t->med.k2, d = t->med.d;
    const int tot = q.nray * q.ntail;
    lm_status s;
    if ((s = lm_dalloc(t, &N.rel, (size_t)t->n)) != LM_OK) return s;
    if ((s = lm_dalloc(t, &N.hgt, (size_t)t->n)) != LM_OK) return s;
    if ((s = lm_dalloc(t, &N.q, (size_t)t->n * LM_MAXV)) != LM_OK) return s;
    const double wmax = N.wmax; // near pairs of adjacent leaves are at most 2 sqrt(2) widths apart
    if (t->adaptive) {
        const AdaptTree &A = t->at;
        k_near_pts<<<(unsigned)A.nleaf, 32, 0, st>>>(ListBoxes{A.leaves, A.cx, A.cy, A.w}, kap, d, t->xs, t->ys,
                                                     t->leaf_start, N.rel, N.hgt);
    } else {
        const Level &lv = t->lev[t->L];
        k_near_pts<<<(unsigned)lv.nbox, 64, 0, st>>>(GridLeaves{LeafGeom{lv.ncol, t->x0, lv.w}}, kap, d, t->xs, t->ys,
                                                     t->leaf_start, N.rel, N.hgt);
    }
    LM_CUDA(cudaGetLastError());
    N.zmax = 8.0 * wmax * wmax * kap * kap;
    if (!t->near_pw64) return LM_OK; // segment coefficients too many for shared memory: FP64 pairs (k_leaf64)
    if ((s = lm_dalloc(t, &N.node, 2 * (size_t)tot)) != LM_OK) return s;
    if ((s = lm_dalloc(t, &N.w, 4 * (size_t)tot)) != LM_OK) return s;
    if (q.split && (s = lm_dalloc(t, &N.w2, 4 * (size_t)tot)) != LM_OK) return s;
    if ((s = lm_dalloc(t, &N.seg, 2 * (size_t)q.nseg)) != LM_OK) return s;
    if ((s = lm_dalloc(t, &N.segw, 2 * (size_t)q.nseg)) != LM_OK) return s;
    k_tail_tab<<<gridn(tot, 64), 64, 0, st>>>(tot, kap, q.tail_lam, q.tail_s2, q.tail_w, N.node, N.w);
    if (q.split) k_tail_tab<<<gridn(tot, 64), 64, 0, st>>>(tot, kap, q.tail_lam, q.tail_s2, q.tail_w2, nullptr, N.w2);
    k_seg_tab<<<gridn(q.nseg, 64), 64, 0, st>>>(q.nseg, kap, q.seg_lam, q.seg_s2, q.seg_w, N.seg, N.segw);
    // target gradient: its own, longer tails, and per-pair segment weights
    const int tg = q.nray * q.ntail_g;
    if ((s = lm_dalloc(t, &N.node_g, 2 * (size_t)tg)) != LM_OK) return s;
    if ((s = lm_dalloc(t, &N.w_g, 12 * (size_t)tg)) != LM_OK) return s;
    if (q.split && (s = lm_dalloc(t, &N.w2_g, 12 * (size_t)tg)) != LM_OK) return s;
    if ((s = lm_dalloc(t, &N.segw_g, 6 * (size_t)q.nseg)) != LM_OK) return s;
    k_tail_tab<<<gridn(tg, 64), 64, 0, st>>>(tg, kap, q.tail_lam_g, q.tail_s2_g, nullptr, N.node_g, nullptr);
    k_tail_tab_grad<<<gridn(tg, 64), 64, 0, st>>>(tg, q.tail_lam_g, q.tail_s2_g, q.tail_w_g, q.tail_c_g, N.w_g);
    if (q.split)
        k_tail_tab_grad<<<gridn(tg, 64), 64, 0, st>>>(tg, q.tail_lam_g, q.tail_s2_g, q.tail_w2_g, nullptr, N.w2_g);
    k_seg_tab_grad<<<gridn(q.nseg, 64), 64, 0, st>>>(q.nseg, q.seg_lam, q.seg_s2, q.seg_w, q.seg_c, N.segw_g);
    LM_CUDA(cudaGetLastError());
    // one limit for every tree: raised, never lowered under another tree's launch.  A launch asks for the
    // dynamic part (largest at 16 vectors) and k_near_pw_df's own arrays; 48 KB need no attribute
    const int lim = 200 * 1024;
    if (lm_near_pw64_smem(q.nseg) + sizeof(DfSmem) + PW_WARPS * LM_MAXV * sizeof(float4) > 48 * 1024) {
        const void *f[] = {(const void *)k_near_pw_df<1, EdgeRowLeaves>, (const void *)k_near_pw_df<2, EdgeRowLeaves>,
                           (const void *)k_near_pw_df<4, EdgeRowLeaves>, (const void *)k_near_pw_df<8, EdgeRowLeaves>,
                           (const void *)k_near_pw_df<16, EdgeRowLeaves>, (const void *)k_near_pw_df<1, ListBoxes>,
                           (const void *)k_near_pw_df<2, ListBoxes>, (const void *)k_near_pw_df<4, ListBoxes>,
                           (const void *)k_near_pw_df<8, ListBoxes>, (const void *)k_near_pw_df<16, ListBoxes>};
        for (const void *p : f) LM_CUDA(cudaFuncSetAttribute(p, cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
    }
    N.ready = true;
    return LM_OK;
}

template <int NV, bool GRAD, class Geo>
static void launch_near(lm_tree_s *t, Geo geo, int64_t nleaf, int nvq, int nv, const GradOut &go, cudaStream_t st)
{
    const NearTabDF &N = t->ndf;
    const NearQuad &q = t->nq;
    const double kap = 0.5 * t->med.k2;
    const bool imp = t->med.opt.top_bc == LM_BC_IMPEDANCE || t->med.opt.bottom_bc == LM_BC_IMPEDANCE;
    const NearDF nq{q.nray, GRAD ? q.ntail_g : q.ntail, imp ? 1 : 0, q.a_zero ? 1 : 0, GRAD ? N.node_g : N.node,
                    GRAD ? N.w_g : N.w, GRAD ? N.w2_g : N.w2, df{(float)(2.0 * t->med.d * kap), 0.f},
                    (float)(q.hray * kap), {q.rinf[0], q.rinf[1]}, q.nseg, N.seg, N.segw_g, {q.beta[0], q.beta[1]}};
    // targets a pass: TG or, where a leaf holds more and they leave 8 waves of 4 blocks per SM, 2 TG (a pass
    // stages every near source: 200k uniform points with 19 a leaf, 1 vector 531 us with 16, 458 us with 32;
    // gradient of 2 1.93 and 1.83 ms with 8 and 16; 30k points, 2.5 waves, 138 and 151 us; adaptive 100k, whose
    // leaves hold fewer, 797 and 849 us); fewer while that leaves fewer than 4 blocks per SM (small trees), down
    // to an item of kernel values a warp (2 rows x 2 halves of the sources, 4 rows for the gradient; 1000
    // points 116 us with 4, 75 us with 2)
    const int64_t per = std::max<int64_t>(1, (t->n + nleaf - 1) / nleaf);
    constexpr int TG = nd_tgt(NV, GRAD), TW = NV <= 2 && std::is_same<Geo, GridLeaves>::value ? 2 * TG : TG;
    const bool wide = TW > TG && per > TG && nleaf * ((per + TW - 1) / TW) >= 4864;
    int tb = wide ? TW : TG;
    while (tb > (GRAD ? 4 : 2) && nleaf * ((per + tb - 1) / tb) < 608) tb >>= 1;
    const unsigned gy = (unsigned)std::min<int64_t>(64, (per + tb - 1) / tb);
    const size_t shm = (size_t)(GRAD ? 32 : ND_SRC) * NV * sizeof(float4);
    const int free_on = t->med.opt.kernel == LM_KERNEL_G;
    auto run = [&](auto kern) {
        kern<<<dim3((unsigned)nleaf, gy), nd_threads(NV, GRAD), shm, st>>>(geo, t->med.k2, kap, t->xs, t->ys, t->leaf_start, N.rel,
                                                                 N.hgt, t->ustart, t->usrc, t->uterm, nq, N.q, nvq, t->qexp,
                                                                 t->n, nv, tb, free_on, t->us, go);
    };
    if (N.zmax <= 1.0 / 16.0) wide ? run(k_near_df<NV, 4, 7, GRAD, TW, Geo>) : run(k_near_df<NV, 4, 7, GRAD, TG, Geo>);
    else wide ? run(k_near_df<NV, 7, 12, GRAD, TW, Geo>) : run(k_near_df<NV, 7, 12, GRAD, TG, Geo>);
}
template <int NV, class Geo>
static void launch_pw(lm_tree_s *t, Geo geo, int64_t npw, int nv, cudaStream_t st)
{
    const NearTabDF &N = t->ndf;
    const int nseg = t->nq.nseg;
    const double kap = 0.5 * t->med.k2;
    k_pw_src_df<NV><<<(unsigned)npw, 256, 0, st>>>(geo, nseg, N.seg, N.rel, N.hgt, t->leaf_start, t->ustart, t->uterm, N.q,
                                                   nv, (float4 *)t->pwC);
    const size_t shm = (size_t)2 * nseg * nv * sizeof(float4);
    k_near_pw_df<NV><<<(unsigned)npw, 32 * PW_WARPS, shm, st>>>(geo, kap, nseg, N.seg, N.segw, N.rel, N.hgt, t->leaf_start, t->ustart,
                                                      t->usrc, t->uterm, (const float4 *)t->pwC, t->pwidx, t->qexp, t->n,
                                                      nv, t->us);
}

// the direct interactions of nv vectors (t->ndf.q), added to t->us
lm_status lm_launch_near_df(lm_tree_s *t, int nv, cudaStream_t st, int *launches)
{
    *launches = 1;
    const GradOut go{nullptr, nullptr, nullptr, nullptr, 0};
    if (t->adaptive) {
        const AdaptTree &A = t->at;
        const ListBoxes leaves{A.leaves, A.cx, A.cy, A.w}, pwl{A.pwleaves, A.cx, A.cy, A.w};
        NV_DISPATCH(nv, launch_near<NV, false>(t, leaves, A.nleaf, nv, nv, go, st));
        if (A.npw > 0) {
            NV_DISPATCH(nv, launch_pw<NV>(t, pwl, A.npw, nv, st));
            *launches += 2;
        }
    } else {
        const Level &lv = t->lev[t->L];
        const LeafGeom g{lv.ncol, t->x0, lv.w};
        NV_DISPATCH(nv, launch_near<NV, false>(t, GridLeaves{g}, lv.nbox, nv, nv, go, st));
        const int64_t npw = lv.nrow == 1 ? lv.ncol : 2 * lv.ncol;
        NV_DISPATCH(nv, launch_pw<NV>(t, EdgeRowLeaves{g, lv.nrow}, npw, nv, st));
        *launches += 2;
    }
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}

// value and target gradient of vectors v0 .. v0 + nv - 1 (nv <= 4) of the apply's nvq, added to u
// (or null), ux, uy in input order
lm_status lm_launch_near_grad_df(lm_tree_s *t, int nvq, int v0, int nv, zd *u, zd *ux, zd *uy, cudaStream_t st)
{
    const GradOut go{u, ux, uy, t->perm, v0};
    auto run = [&](auto geo, int64_t nleaf) {
        if (nv == 1) launch_near<1, true>(t, geo, nleaf, nvq, nv, go, st);
        else if (nv == 2) launch_near<2, true>(t, geo, nleaf, nvq, nv, go, st);
        else launch_near<4, true>(t, geo, nleaf, nvq, nv, go, st);
    };
    if (t->adaptive) run(ListBoxes{t->at.leaves, t->at.cx, t->at.cy, t->at.w}, t->at.nleaf);
    else run(GridLeaves{LeafGeom{t->lev[t->L].ncol, t->x0, t->lev[t->L].w}}, t->lev[t->L].nbox);
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}
