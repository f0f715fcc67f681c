// lmfmm_few32.cu -- FP32 kernels of the mixed form for applies of up to 4 vectors:
// S2M, L2T with the direct interactions, the factorised segment of the reflected
// terms, and the adaptive tree's M2L.  With few vectors the work per pair is its
// kernel value, so the lanes of a warp take the sources of a target (a leaf of 20
// points leaves two thirds of a 64-thread block idle when a thread takes a target),
// and a leaf's targets may be dealt out to several blocks.
#include <algorithm>

#include "internal.h"
#include "mixed_near.cuh"

static int gridf(int64_t n, int b) { return (int)((n + b - 1) / b); }

// Z^n g_n, n = 0..P, of one point (see basis_row in lmfmm_exp_df.cu): x, y the offset from
// the box centre, iw = 1/w, k2 = k/2
__device__ __forceinline__ void basis_row32(const BesselDF &B, int P, float x, float y, float iw, float k2, zf *row)
{
    const float xx = k2 * x, yy = k2 * y, t = fmaf(xx, xx, yy * yy);
    float g0 = 1.f, g1 = 1.f;
    for (int m = B.nt; m >= 1; --m) {
        g0 = fmaf(-t * B.c[B.N + m].x, g0, 1.f);
        g1 = fmaf(-t * B.c[B.N + B.nt + m].x, g1, 1.f);
    }
    for (int n = B.N; n >= 1; --n) {
        if (n <= P) row[n].re = g0;
        const float g = fmaf(-t * B.c[n].x, g1, g0);
        g1 = g0;
        g0 = g;
    }
    row[0] = zf{g0, 0.f};
    const zf Z = {x * iw, y * iw};
    zf zp = Z;
    for (int n = 1; n <= P; ++n) {
        const float g = row[n].re;
        row[n] = zf{g * zp.re, g * zp.im};
        zp = zp * Z;
    }
}

// ---------------------------------------------------------------------------
// S2M: one block per leaf, 32 points a round (each round summed on its own): a thread forms a
// point's basis row, then a thread per (order n >= 0, vector) sums the four products from which the
// orders n and -n follow.  Writes 4 vector slots, zeros beyond nv.
// ---------------------------------------------------------------------------
#define F32_PTS 32
template <class G>
__global__ void __launch_bounds__(64) k_s2m_f32(G geo, int P, float k, BesselDF B, const float *xl, const float *yl,
                                                const int64_t *ls, const zf *qs, int nv, zf *M)
{
    __shared__ zf b[F32_PTS][25 | 1];
    __shared__ zf q[F32_PTS][4];
    const int np = 2 * P + 1, nitem = (P + 1) * 4;
    const int64_t box = geo.id(blockIdx.x), lo = ls[box], hi = ls[box + 1];
    const float iw = 1.f / geo.width(box);
    float4 s[2]; // up to 100 items on 64 threads: sums re re, im im, re im, im re of basis and density
    s[0] = s[1] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t p0 = lo; p0 < hi; p0 += F32_PTS) {
        const int cnt = (int)min((int64_t)F32_PTS, hi - p0);
        __syncthreads();
        if (threadIdx.x < cnt) basis_row32(B, P, xl[p0 + threadIdx.x], yl[p0 + threadIdx.x], iw, 0.5f * k, b[threadIdx.x]);
        for (int i = threadIdx.x; i < cnt * 4; i += blockDim.x) {
            const int j = i >> 2, v = i & 3;
            q[j][v] = v < nv ? qs[(p0 + j) * LM_MAXV + v] : zf{0.f, 0.f};
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int it = threadIdx.x + 64 * h;
            if (it < nitem) {
                const int n = it >> 2, v = it & 3;
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int j = 0; j < cnt; ++j) {
                    const zf bb = b[j][n], qq = q[j][v];
                    a.x = fmaf(bb.re, qq.re, a.x);
                    a.y = fmaf(bb.im, qq.im, a.y);
                    a.z = fmaf(bb.re, qq.im, a.z);
                    a.w = fmaf(bb.im, qq.re, a.w);
                }
                s[h] = make_float4(s[h].x + a.x, s[h].y + a.y, s[h].z + a.z, s[h].w + a.w);
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int it = threadIdx.x + 64 * h;
        if (it < nitem) {
            const int n = it >> 2, v = it & 3;
            M[(box * np + P + n) * LM_MAXV + v] = zf{s[h].x + s[h].y, s[h].z - s[h].w}; // q conj(b)
            const float sg = (n & 1) ? -1.f : 1.f;
            if (n > 0) M[(box * np + P - n) * LM_MAXV + v] = zf{sg * (s[h].x - s[h].y), sg * (s[h].z + s[h].w)};
        }
    }
}

// ---------------------------------------------------------------------------
// L2T and the direct interactions.  One block: up to tb targets of a leaf at a time, ROWS rows per
// warp.  The leaf's near sources are flattened and staged 64 at a time in the target leaf's frame; each
// lane takes two of them against the warp's rows, kernel value and multiply-adds in registers, and the
// lanes' sums are folded once per target by exchanging halves.  Reflected pairs add their tails (the
// segment part comes from k_near_pw_f32).  DEG as in k_leaf32.
// Bound by FP32 issue and, between the rounds, by the staging and the barriers: more rows a warp
// spread those over more pairs.  Uniform 100k points, 1 vector: 193 us with 4 rows, 153 us with 8;
// 12 trees of 4 vectors: 3.46 ms with 4 rows, 3.29 ms with 6 (8 spill).  Clustered adaptive 100k, whose
// leaves hold fewer points than 32: 186 us with 4 rows, 256 us with 8.
// ---------------------------------------------------------------------------
// rows of a warp on large uniform trees (4 vectors' sums take more registers), F32_ROWS elsewhere
__host__ __device__ constexpr int f32_rows(int nv) { return nv == 4 ? 6 : 8; }
#define F32_ROWS 4
#define F32_SRC 64
#define F32_ENT 64
template <int NV, int DEG, int ROWS, class G>
__global__ void __launch_bounds__(128) k_leaf_f32(G geo, int P, float k, float d, BesselDF B, const float *xl, const float *yl,
                                                  const float *y32, const int64_t *ls, const int64_t *ustart,
                                                  const int32_t *usrc, const int32_t *uterm, NearQuadF nq, const zf *Lc,
                                                  const zf *qs, zf *us, int nv, int tb, int free_on)
{
    constexpr int TGT = 4 * ROWS;
    __shared__ int fj0[F32_ENT], fpre[F32_ENT + 1], fterm[F32_ENT];
    __shared__ float2 foff[F32_ENT];
    __shared__ float2 sp[F32_SRC];
    __shared__ int sj[F32_SRC], st[F32_SRC];
    __shared__ zf sq[F32_SRC][NV];
    __shared__ float4 tr[TGT]; // x, y relative to the leaf centre, absolute y
    __shared__ zf bz[TGT][25], PQ[25][NV][2], uL[TGT][NV];
    const int np = 2 * P + 1;
    const int64_t b = geo.id(blockIdx.x);
    const int lo = (int)ls[b], hi = (int)ls[b + 1];
    if (lo + (int)blockIdx.y * tb >= hi) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float iw = 1.f / geo.width(b), k24 = 0.25f * k * k;
    const int e0 = (int)ustart[b], e1 = (int)ustart[b + 1];
    for (int i = tid; i < (P + 1) * NV; i += 128) { // L_n + s L_{-n} and i (L_n - s L_{-n}), s = (-1)^n
        const int n = i / NV, v = i - n * NV;
        const zf a = Lc[(b * np + P + n) * LM_MAXV + v], c = Lc[(b * np + P - n) * LM_MAXV + v];
        const float s = (n & 1) ? -1.f : 1.f;
        PQ[n][v][0] = n ? zf{a.re + s * c.re, a.im + s * c.im} : a;
        PQ[n][v][1] = n ? zf{-(a.im - s * c.im), a.re - s * c.re} : zf{0.f, 0.f};
    }
    for (int t0 = lo + (int)blockIdx.y * tb; t0 < hi; t0 += (int)gridDim.y * tb) {
        const int nt = min(tb, hi - t0);
        __syncthreads();
        if (tid < nt) {
            const float x = xl[t0 + tid], y = yl[t0 + tid];
            tr[tid] = make_float4(x, y, y32[t0 + tid], 0.f);
            basis_row32(B, P, x, y, iw, 0.5f * k, bz[tid]);
        }
        __syncthreads();
        for (int i = tid; i < nt * NV; i += 128) {
            const int j = i / NV, v = i - j * NV;
            zf a = {0.f, 0.f};
            for (int n = 0; n <= P; ++n) {
                const zf bb = bz[j][n], p = PQ[n][v][0], q = PQ[n][v][1];
                a.re = fmaf(p.re, bb.re, fmaf(q.re, bb.im, a.re));
                a.im = fmaf(p.im, bb.re, fmaf(q.im, bb.im, a.im));
            }
            uL[j][v] = a;
        }
        float tx[ROWS], ty[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const float4 t = tr[min(warp + 4 * r, nt - 1)];
            tx[r] = t.x;
            ty[r] = t.y;
        }
        zf acc[ROWS][NV];
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[r][v] = zf{0.f, 0.f};
        for (int c0 = e0; c0 < e1; c0 += F32_ENT) {
            const int nc = min(F32_ENT, e1 - c0);
            __syncthreads(); // the previous entries' sources are done
            int cnt = 0;
            if (tid < nc) {
                const int s = usrc[c0 + tid], term = uterm[c0 + tid];
                fj0[tid] = (int)ls[s];
                fterm[tid] = term;
                cnt = (term == 0 && !free_on) ? 0 : (int)(ls[s + 1] - ls[s]);
                float ox, oy;
                geo.offset(b, s, ox, oy);
                foff[tid] = make_float2(ox, oy);
            }
            if (tid < F32_ENT) { // inclusive scan of the counts (two warps)
                for (int o = 1; o < 32; o <<= 1) {
                    const int x = __shfl_up_sync(0xffffffffu, cnt, o);
                    if (lane >= o) cnt += x;
                }
                fpre[tid + 1] = cnt;
            }
            if (tid == 0) fpre[0] = 0;
            __syncthreads();
            if (tid >= 32 && tid < F32_ENT) fpre[tid + 1] += fpre[32];
            __syncthreads();
            const int tot = fpre[nc];
            for (int f0 = 0; f0 < tot; f0 += F32_SRC) {
                const int ns = min(F32_SRC, tot - f0);
                if (tid < ns) {
                    const int f = f0 + tid;
                    int e = 0; // the entry holding source f
#pragma unroll
                    for (int o = F32_ENT / 2; o > 0; o >>= 1)
                        if (e + o < nc && fpre[e + o] <= f) e += o;
                    const int j = fj0[e] + (f - fpre[e]), term = fterm[e];
                    const float2 of = foff[e];
                    // free: in the target leaf's frame; reflected: absolute y
                    sp[tid] = make_float2(xl[j] - of.x, term ? y32[j] : yl[j] - of.y);
                    sj[tid] = j;
                    st[tid] = term;
#pragma unroll
                    for (int v = 0; v < NV; ++v) sq[tid][v] = v < nv ? qs[(int64_t)j * LM_MAXV + v] : zf{0.f, 0.f};
                }
                __syncthreads();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int s = 32 * h + lane;
                    if (s >= ns) continue;
                    const float2 p = sp[s];
                    const int term = st[s], j = sj[s];
                    zf q[NV];
#pragma unroll
                    for (int v = 0; v < NV; ++v) q[v] = sq[s][v];
                    if (term == 0) {
#pragma unroll
                        for (int r = 0; r < ROWS; ++r) {
                            if (warp + 4 * r >= nt) break;
                            const float dx = tx[r] - p.x, dy = ty[r] - p.y;
                            const bool self = j == t0 + warp + 4 * r;
                            const float t = self ? 1.0f : k24 * fmaf(dx, dx, dy * dy);
                            zf g;
                            if (DEG) g = green_free32_series_d<DEG ? DEG : 8>(t);
                            else {
                                g = green_free32_series(t);
                                if (t > 1.0f) g = green_free32_far(t);
                            }
                            if (self) g = zf{0.f, 0.f};
#pragma unroll
                            for (int v = 0; v < NV; ++v) cfmaf(acc[r][v], g, q[v]);
                        }
                    } else {
#pragma unroll
                        for (int r = 0; r < ROWS; ++r) {
                            if (warp + 4 * r >= nt) break;
                            const float ya = tr[warp + 4 * r].z;
                            const float hh = term == 1 ? -(ya + p.y) : ya + p.y + 2.0f * d;
                            const zf g = near_tail32(nq, term - 1, fabsf(tx[r] - p.x), hh);
#pragma unroll
                            for (int v = 0; v < NV; ++v) cfmaf(acc[r][v], g, q[v]);
                        }
                    }
                }
                __syncthreads(); // the sources are overwritten by the next round
            }
        }
        // 2 NV sums of each row over the lanes, RP rows at a time: at each step a lane keeps one half of
        // them
        constexpr int RP = NV * ROWS <= 16 ? ROWS : 2, CNT = 2 * NV * RP; // 8, 16 or 32 sums
#pragma unroll
        for (int r0 = 0; r0 < ROWS; r0 += RP) {
            if (r0 > 0 && warp + 4 * r0 >= nt) break;
            float val[CNT];
#pragma unroll
            for (int r = 0; r < RP; ++r)
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    val[2 * (r * NV + v)] = acc[r0 + r][v].re;
                    val[2 * (r * NV + v) + 1] = acc[r0 + r][v].im;
                }
            int cnt = CNT;
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                if (cnt > 1) {
                    cnt >>= 1;
#pragma unroll
                    for (int i = 0; i < CNT / 2; ++i)
                        if (i < cnt) {
                            const float x = val[i], y = val[i + cnt];
                            const bool up = (lane & o) != 0;
                            val[i] = (up ? y : x) + __shfl_xor_sync(0xffffffffu, up ? x : y, o);
                        }
                } else
                    val[0] += __shfl_xor_sync(0xffffffffu, val[0], o);
            }
            constexpr int REP = 32 / CNT; // lanes holding the same sum
            const int id = lane / REP, row = warp + 4 * (r0 + id / (2 * NV)), vv = (id / 2) % NV;
            if (lane % REP == 0 && row < nt && vv < nv) {
                const zf l = uL[row][vv];
                ((float *)&us[(int64_t)(t0 + row) * LM_MAXV + vv])[id & 1] = val[0] + ((id & 1) ? l.im : l.re);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// The factorised segment of the reflected terms, as k_pw_src64 and k_near_pw64 split it: a source
// leaf's coefficients once, then per target leaf the sum over its U entries and its evaluation
// (a warp per target, lanes over the nodes).
// ---------------------------------------------------------------------------
__device__ __forceinline__ zf seg_exp32(zf lam, zf s2, float sg, float x, float Y)
{
    const float a = expf(fmaf(-sg * lam.im, x, s2.re * Y));
    float sn, cs;
    sincosf(fmaf(sg * lam.re, x, s2.im * Y), &sn, &cs);
    return zf{a * cs, a * sn};
}
template <int NV, class G>
__global__ void __launch_bounds__(128) k_pw_src_f32(G geo, float d, const float *xl, const float *y32, const int64_t *ls,
                                                    const int64_t *ustart, const int32_t *uterm, NearQuadF nq, const zf *qs,
                                                    zf *C)
{
    __shared__ int any[2];
    const int nk = 2 * nq.nseg;
    const int64_t slot = blockIdx.x, b = geo.id(slot);
    if (ls[b + 1] == ls[b]) return; // an empty leaf: its coefficients are never read
    if (threadIdx.x < 2) any[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t e = ustart[b] + threadIdx.x; e < ustart[b + 1]; e += blockDim.x)
        if (uterm[e] > 0) any[uterm[e] - 1] = 1;
    __syncthreads();
    for (int m = 0; m < 2; ++m) {
        if (!any[m]) continue;
        for (int k = threadIdx.x; k < nk; k += blockDim.x) {
            const zf lam = nq.seg_lam[k >> 1], s2 = nq.seg_s2[k >> 1];
            zf acc[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[v] = zf{0.f, 0.f};
            for (int64_t j = ls[b]; j < ls[b + 1]; ++j) {
                const zf f = seg_exp32(lam, s2, (k & 1) ? 1.f : -1.f, xl[j], m == 0 ? y32[j] : -(y32[j] + d));
#pragma unroll
                for (int v = 0; v < NV; ++v) cfmaf(acc[v], f, qs[j * LM_MAXV + v]);
            }
#pragma unroll
            for (int v = 0; v < NV; ++v) C[((slot * 2 + m) * nk + k) * 4 + v] = acc[v];
        }
    }
}
template <int NV, class G>
__global__ void __launch_bounds__(256) k_near_pw_f32(G geo, float d, const float *xl, const float *y32, const int64_t *ls,
                                                     const int64_t *ustart, const int32_t *usrc, const int32_t *uterm,
                                                     NearQuadF nq, const zf *C, const int32_t *pwidx, zf *us)
{
    extern __shared__ zf Bf[]; // [nk][NV]
    const int nk = 2 * nq.nseg;
    const int64_t b = geo.id(blockIdx.x), lo = ls[b], hi = ls[b + 1];
    if (hi == lo) return; // no targets
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    for (int m = 0; m < 2; ++m) {
        __syncthreads(); // the previous term's B is done with
        bool any = false;
        for (int k = threadIdx.x; k < nk; k += blockDim.x) // a thread owns its B[k]
#pragma unroll
            for (int v = 0; v < NV; ++v) Bf[k * NV + v] = zf{0.f, 0.f};
        for (int64_t e = ustart[b]; e < ustart[b + 1]; ++e) {
            if (uterm[e] != m + 1) continue;
            const int64_t s = usrc[e];
            if (ls[s + 1] == ls[s]) continue; // no sources (uniform over the block)
            any = true;
            float ox, oy;
            geo.offset(s, b, ox, oy); // centre_s - centre_T
            const zf *Cs = C + ((int64_t)pwidx[s] * 2 + m) * nk * 4;
            for (int k = threadIdx.x; k < nk; k += blockDim.x) {
                const zf f = seg_exp32(nq.seg_lam[k >> 1], zf{0.f, 0.f}, (k & 1) ? 1.f : -1.f, ox, 0.f);
#pragma unroll
                for (int v = 0; v < NV; ++v) cfmaf(Bf[k * NV + v], f, Cs[k * 4 + v]);
            }
        }
        if (!any) continue; // block-uniform
        for (int k = threadIdx.x; k < nk; k += blockDim.x) {
            const zf w = nq.seg_w[m * nq.nseg + (k >> 1)];
#pragma unroll
            for (int v = 0; v < NV; ++v) Bf[k * NV + v] = w * Bf[k * NV + v];
        }
        __syncthreads();
        for (int64_t i = lo + warp; i < hi; i += nwarp) { // a warp per target, lanes over the nodes
            zf acc[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[v] = zf{0.f, 0.f};
            const float x = xl[i], Y = m == 0 ? y32[i] : -(y32[i] + d);
            for (int k = lane; k < nk; k += 32) {
                const zf f = seg_exp32(nq.seg_lam[k >> 1], nq.seg_s2[k >> 1], (k & 1) ? -1.f : 1.f, x, Y);
#pragma unroll
                for (int v = 0; v < NV; ++v) cfmaf(acc[v], f, Bf[k * NV + v]);
            }
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                float re = acc[v].re, im = acc[v].im;
                for (int o = 16; o > 0; o >>= 1) {
                    re += __shfl_xor_sync(0xffffffffu, re, o);
                    im += __shfl_xor_sync(0xffffffffu, im, o);
                }
                if (lane == v) us[i * LM_MAXV + v] = us[i * LM_MAXV + v] + zf{re, im};
            }
        }
    }
}

// ---------------------------------------------------------------------------
// M2L over the adaptive V list: one block per target box, a thread per (order, one of 4 subsets of
// the entries); tables transposed ([q][p]) so that a warp reads contiguous rows.  Each entry is
// summed on its own; sets L (L2L adds to it).  Bound by the L2 reads of the tables (a table per
// entry).
// ---------------------------------------------------------------------------
__global__ void k_tab32_t(const zf *tab, int64_t count, int np, zf *out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= count) return;
    const int64_t slot = i / ((int64_t)np * np);
    const int r = (int)(i % ((int64_t)np * np)), p = r / np, q = r % np;
    out[slot * np * np + (int64_t)q * np + p] = tab[i];
}
template <int NV>
__global__ void __launch_bounds__(224) k_m2l_f32(int P, const int64_t *vstart, const int32_t *vsrc, const int32_t *vslot,
                                                 const zf *tab, const zf *M, zf *L)
{
    __shared__ zf red[3][49][NV];
    const int np = 2 * P + 1, p = threadIdx.x % np, g = threadIdx.x / np;
    const int64_t b = blockIdx.x, e0 = vstart[b], e1 = vstart[b + 1];
    zf tot[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) tot[v] = zf{0.f, 0.f};
    if (g < 4)
        for (int64_t e = e0 + g; e < e1; e += 4) {
            const zf *T = tab + (int64_t)vslot[e] * np * np + p, *m = M + (int64_t)vsrc[e] * np * LM_MAXV;
            zf acc[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[v] = zf{0.f, 0.f};
            int q = 0;
            for (; q + 4 <= np; q += 4) { // four table entries in flight
                zf t[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) t[j] = T[(q + j) * np];
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int v = 0; v < NV; ++v) cfmaf(acc[v], t[j], m[(q + j) * LM_MAXV + v]);
            }
            for (; q < np; ++q)
#pragma unroll
                for (int v = 0; v < NV; ++v) cfmaf(acc[v], T[q * np], m[q * LM_MAXV + v]);
#pragma unroll
            for (int v = 0; v < NV; ++v) tot[v] = tot[v] + acc[v];
        }
    if (g > 0 && g < 4)
#pragma unroll
        for (int v = 0; v < NV; ++v) red[g - 1][p][v] = tot[v];
    __syncthreads();
    if (g == 0)
#pragma unroll
        for (int v = 0; v < NV; ++v) L[(b * np + p) * LM_MAXV + v] = ((tot[v] + red[0][p][v]) + red[1][p][v]) + red[2][p][v];
}

// The same for one vector, class by class: a table serves one product an entry, so k_m2l_f32 reads all of
// them from L2.  Blocks take 64 entries of one class, sorted at build: table and source multipoles are staged
// once, a thread holds 8 orders of an entry; the products go to memory by entry, then a target's are summed
// in k_m2l_f32's order (the same bits).  Clustered 100k, p = 14: 409 us there, 229 us here.
#define CLS_TILE 64
struct ClsTile {
    int32_t slot, first, cnt, pad;
};
// slices of whole target boxes of at most about 2^20 entries share the products' buffer
struct ClsSlice {
    int64_t tile0, ntile, box0, nbox, e0;
};
// M: the vector's multipoles alone, [box][2p+1] (from the 16-slot layout a gather takes a sector an order: 247
// instead of 192 us)
__global__ void k_m2l_pack_f32(const zf *M, int64_t n, zf *out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = M[i * LM_MAXV];
}
__global__ void __launch_bounds__(448) k_m2l_cls_f32(int P, const ClsTile *tiles, const int32_t *psrc, const int32_t *ppos,
                                                     const zf *tab, const zf *M, zf *C)
{
    extern __shared__ float4 cls_sm[];
    const int np = 2 * P + 1, NG = (np + 7) / 8, PW = 8 * NG, MS = CLS_TILE + 1;
    zf *Ts = (zf *)cls_sm, *Ms = Ts + np * PW; // [np][PW] (q, p), [np][MS]
    const ClsTile t = tiles[blockIdx.x];
    const zf *T = tab + (int64_t)t.slot * np * np;
    for (int i = threadIdx.x; i < np * np; i += blockDim.x) Ts[i / np * PW + i % np] = T[i];
    for (int i = threadIdx.x; i < t.cnt * np; i += blockDim.x) {
        const int j = i / np, q = i % np;
        Ms[q * MS + j] = M[(int64_t)psrc[t.first + j] * np + q];
    }
    __syncthreads();
    const int j = threadIdx.x % CLS_TILE, p0 = threadIdx.x / CLS_TILE * 8;
    if (j >= t.cnt) return;
    zf acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = zf{0.f, 0.f};
    for (int q = 0; q < np; ++q) {
        const zf m = Ms[q * MS + j];
        const float4 *r = (const float4 *)(Ts + q * PW + p0);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 x = r[i];
            cfmaf(acc[2 * i], zf{x.x, x.y}, m);
            cfmaf(acc[2 * i + 1], zf{x.z, x.w}, m);
        }
    }
    zf *o = C + (int64_t)ppos[t.first + j] * np + p0;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (p0 + i < np) o[i] = acc[i];
}
__global__ void __launch_bounds__(224) k_m2l_sum_f32(int P, int64_t box0, int64_t base, const int64_t *vstart, const zf *C, zf *L)
{
    __shared__ zf red[3][49];
    const int np = 2 * P + 1, p = threadIdx.x % np, g = threadIdx.x / np;
    const int64_t b = box0 + blockIdx.x, e0 = vstart[b], e1 = vstart[b + 1];
    zf tot = {0.f, 0.f};
    if (g < 4)
        for (int64_t e = e0 + g; e < e1; e += 4) tot = tot + C[(e - base) * np + p];
    if (g > 0 && g < 4) red[g - 1][p] = tot;
    __syncthreads();
    if (g == 0) L[(b * np + p) * LM_MAXV] = ((tot + red[0][p]) + red[1][p]) + red[2][p];
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
#define NV_FEW(nv, ...)                                   \
    switch (nv) {                                         \
    case 1: { constexpr int NV = 1; __VA_ARGS__; } break; \
    case 2: { constexpr int NV = 2; __VA_ARGS__; } break; \
    default: { constexpr int NV = 4; __VA_ARGS__; } break;\
    }
#define TRY_F(x)                     \
    do {                             \
        lm_status s_ = (x);          \
        if (s_ != LM_OK) return s_;  \
    } while (0)

// V entries by class for k_m2l_cls_f32, where a tile holds enough of them to pay for its table
static lm_status setup_classes(lm_tree_s *t, cudaStream_t st)
{
    AdaptTree &A = t->at;
    const int np = 2 * t->p + 1;
    const int64_t ne = A.nv, ncls = (int64_t)A.cls_term.size();
    A.cls_slices.clear();
    if (ne == 0 || ne > INT32_MAX) return LM_OK;
    std::vector<int64_t> vs(A.nbox + 1);
    std::vector<int32_t> src(ne), slot(ne), psrc(ne), ppos(ne);
    LM_CUDA(cudaMemcpyAsync(vs.data(), A.vstart, vs.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    LM_CUDA(cudaMemcpyAsync(src.data(), A.vsrc, ne * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    LM_CUDA(cudaMemcpyAsync(slot.data(), A.vslot, ne * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    LM_CUDA(cudaStreamSynchronize(st));
    std::vector<ClsTile> tiles;
    std::vector<ClsSlice> slices;
    int64_t most = 0;
    for (int64_t b0 = 0, b1; b0 < A.nbox; b0 = b1) {
        for (b1 = b0 + 1; b1 < A.nbox && vs[b1 + 1] - vs[b0] <= (int64_t)1 << 20;) ++b1;
        const int64_t e0 = vs[b0], e1 = vs[b1];
        std::vector<int32_t> at(ncls + 1, 0);
        for (int64_t e = e0; e < e1; ++e) ++at[slot[e] + 1];
        for (int64_t c = 0; c < ncls; ++c) at[c + 1] += at[c];
        const int64_t tile0 = (int64_t)tiles.size();
        for (int64_t c = 0; c < ncls; ++c)
            for (int32_t f = at[c]; f < at[c + 1]; f += CLS_TILE)
                tiles.push_back({(int32_t)c, (int32_t)(e0 + f), std::min(CLS_TILE, at[c + 1] - f), 0});
        for (int64_t e = e0; e < e1; ++e) {
            const int64_t k = e0 + at[slot[e]]++;
            psrc[k] = src[e];
            ppos[k] = (int32_t)(e - e0);
        }
        slices.push_back({tile0, (int64_t)tiles.size() - tile0, b0, b1 - b0, e0});
        most = std::max(most, e1 - e0);
    }
    if (ne < 24 * (int64_t)tiles.size()) return LM_OK;
    ClsTile *dt;
    TRY_F(lm_dalloc(t, &dt, tiles.size()));
    TRY_F(lm_dalloc(t, &A.cls_src, (size_t)ne));
    TRY_F(lm_dalloc(t, &A.cls_pos, (size_t)ne));
    TRY_F(lm_dalloc(t, &A.cls_C, (size_t)most * np));
    TRY_F(lm_dalloc(t, &A.cls_M, (size_t)A.nbox * np));
    A.cls_tiles = dt;
    LM_CUDA(cudaMemcpyAsync(dt, tiles.data(), tiles.size() * sizeof(ClsTile), cudaMemcpyHostToDevice, st));
    LM_CUDA(cudaMemcpyAsync(A.cls_src, psrc.data(), ne * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    LM_CUDA(cudaMemcpyAsync(A.cls_pos, ppos.data(), ne * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    for (const ClsSlice &x : slices) A.cls_slices.insert(A.cls_slices.end(), {x.tile0, x.ntile, x.box0, x.nbox, x.e0});
    return LM_OK;
}

// basis coefficients, interface-leaf slots and coefficient buffer, transposed tables (adaptive)
lm_status lm_setup_few32(lm_tree_s *t, cudaStream_t st)
{
    double wmax = t->adaptive ? 0.0 : t->lev[t->L].w; // the widest leaf
    if (t->adaptive)
        for (int64_t b = 0; b < t->at.nbox; ++b)
            if (t->at.hbox[4 * b + 3]) wmax = std::max(wmax, ldexp(t->med.d, -(int)t->at.hbox[4 * b]));
    t->few32 = false;
    if (!lm_exp_df_fits(t->med.k2, wmax)) return LM_OK;
    std::vector<float> h;
    lm_bessel_df(t->p, t->med.k2, wmax, h, &t->xdf.N, &t->xdf.nt);
    TRY_F(lm_dalloc(t, &t->xdf.bes, h.size() / 2));
    LM_CUDA(cudaMemcpyAsync(t->xdf.bes, h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice, st));
    int64_t npw = 0;
    TRY_F(lm_setup_pwidx(t, &npw, st));
    zf *C;
    TRY_F(lm_dalloc(t, &C, (size_t)std::max<int64_t>(1, npw) * 2 * 2 * t->nq.nseg * 4));
    t->pwC = (zd *)C;
    if (t->adaptive) {
        const int np = 2 * t->p + 1;
        const int64_t cnt = std::max<int64_t>(1, (int64_t)t->at.cls_term.size()) * np * np;
        TRY_F(lm_dalloc(t, &t->at.tab32t, (size_t)cnt));
        k_tab32_t<<<gridf(cnt, 256), 256, 0, st>>>(t->at.tab32, cnt, np, t->at.tab32t);
    }
    if (t->adaptive) TRY_F(setup_classes(t, st));
    LM_CUDA(cudaGetLastError());
    t->few32 = true;
    return LM_OK;
}

void lm_few32_s2m(lm_tree_s *t, int nv, cudaStream_t st)
{
    const BesselDF B{t->xdf.bes, t->xdf.N, t->xdf.nt};
    const float k = (float)t->med.k2;
    if (t->adaptive) {
        const AdaptTree &A = t->at;
        k_s2m_f32<<<(unsigned)A.nleaf, 64, 0, st>>>(List32{A.leaves, A.cx, A.cy, A.w}, t->p, k, B, t->xl32, t->yl32,
                                                   t->leaf_start, t->qs32, nv, A.M32);
    } else {
        const Level &lv = t->lev[t->L];
        k_s2m_f32<<<(unsigned)lv.nbox, 64, 0, st>>>(Grid32{lv.ncol, (float)lv.w}, t->p, k, B, t->xl32, t->yl32, t->leaf_start,
                                                   t->qs32, nv, lv.M32);
    }
}

// M2L of the adaptive tree (sets L); returns the kernels launched
int lm_few32_m2l(lm_tree_s *t, int nv, cudaStream_t st)
{
    const AdaptTree &A = t->at;
    const int np = 2 * t->p + 1, thr = (4 * np + 31) / 32 * 32;
    if (nv == 1 && !A.cls_slices.empty()) { // (more vectors share a table's reading in k_m2l_f32)
        const int NG = (np + 7) / 8;
        const size_t shm = (size_t)np * (8 * NG + CLS_TILE + 1) * sizeof(zf);
        int k = 1;
        k_m2l_pack_f32<<<gridf(A.nbox * np, 256), 256, 0, st>>>(A.M32, A.nbox * np, A.cls_M);
        for (size_t i = 0; i < A.cls_slices.size(); i += 5) {
            const int64_t *x = &A.cls_slices[i]; // tile0, ntile, box0, nbox, e0
            if (x[1] > 0) {
                k_m2l_cls_f32<<<(unsigned)x[1], CLS_TILE * NG, shm, st>>>(t->p, (const ClsTile *)A.cls_tiles + x[0], A.cls_src,
                                                                          A.cls_pos, A.tab32t, A.cls_M, A.cls_C);
                ++k;
            }
            k_m2l_sum_f32<<<(unsigned)x[3], thr, 0, st>>>(t->p, x[2], x[4], A.vstart, A.cls_C, A.L32);
            ++k;
        }
        return k;
    }
    NV_FEW(nv, (k_m2l_f32<NV><<<(unsigned)A.nbox, thr, 0, st>>>(t->p, A.vstart, A.vsrc, A.vslot, A.tab32t, A.M32, A.L32)));
    return 1;
}

// L2T, direct interactions and the reflected segment; returns the kernels launched
int lm_few32_leaf(lm_tree_s *t, const NearQuadF &nq, int nv, cudaStream_t st)
{
    const BesselDF B{t->xdf.bes, t->xdf.N, t->xdf.nt};
    const float k = (float)t->med.k2, d = (float)t->med.d;
    const int free_on = t->med.opt.kernel == LM_KERNEL_G;
    const int64_t nleaf = t->adaptive ? t->at.nleaf : t->lev[t->L].nbox;
    // targets a pass: 32 (24 for 4 vectors) on a uniform tree that fills 4 blocks per SM with them,
    // else 16, fewer while that leaves fewer than 4 blocks per SM (small trees)
    const int64_t per = std::max<int64_t>(1, (t->n + nleaf - 1) / nleaf);
    const int big = 4 * f32_rows(nv <= 2 ? nv : 4);
    const bool wide = !t->adaptive && nleaf * ((per + big - 1) / big) >= 608;
    int tb = wide ? big : 4 * F32_ROWS;
    while (tb > 4 && nleaf * ((per + tb - 1) / tb) < 608) tb >>= 1;
    const unsigned gy = (unsigned)std::min<int64_t>(64, (per + tb - 1) / tb);
    const size_t shm = (size_t)2 * t->nq.nseg * (nv <= 2 ? nv : 4) * sizeof(zf);
    auto leaf = [&](auto kern, auto geo, const zf *L) {
        kern<<<dim3((unsigned)nleaf, gy), 128, 0, st>>>(geo, t->p, k, d, B, t->xl32, t->yl32, t->y32, t->leaf_start, t->ustart,
                                                        t->usrc, t->uterm, nq, L, t->qs32, t->us32, nv, tb, free_on);
    };
    auto pw = [&](auto src, auto tgt, auto geo, int64_t npw) {
        src<<<(unsigned)npw, 128, 0, st>>>(geo, d, t->xl32, t->y32, t->leaf_start, t->ustart, t->uterm, nq, t->qs32, (zf *)t->pwC);
        tgt<<<(unsigned)npw, 256, shm, st>>>(geo, d, t->xl32, t->y32, t->leaf_start, t->ustart, t->usrc, t->uterm, nq,
                                             (const zf *)t->pwC, t->pwidx, t->us32);
    };
    if (t->adaptive) {
        const AdaptTree &A = t->at;
        const List32 g{A.leaves, A.cx, A.cy, A.w}, e{A.pwleaves, A.cx, A.cy, A.w};
        NV_FEW(nv, (leaf(k_leaf_f32<NV, 0, F32_ROWS, List32>, g, A.L32)));
        if (A.npw == 0) return 1;
        NV_FEW(nv, (pw(k_pw_src_f32<NV, List32>, k_near_pw_f32<NV, List32>, e, A.npw)));
        return 3;
    }
    const Level &lv = t->lev[t->L];
    const Grid32 g{lv.ncol, (float)lv.w};
    EdgeGrid32 e;
    e.ncol = lv.ncol;
    e.w = (float)lv.w;
    e.nrow = lv.nrow;
    // largest k r of a direct pair: two leaves apart diagonally
    const double xmax = t->med.k2 * lv.w * 2.0 * 1.4142135623730951 * 1.0001;
    const bool deg6 = xmax <= 2.0 && lm_h0_terms(xmax) <= 6;
    NV_FEW(nv, (deg6 ? (wide ? leaf(k_leaf_f32<NV, 6, f32_rows(NV), Grid32>, g, lv.L32) : leaf(k_leaf_f32<NV, 6, F32_ROWS, Grid32>, g, lv.L32))
                     : (wide ? leaf(k_leaf_f32<NV, 0, f32_rows(NV), Grid32>, g, lv.L32) : leaf(k_leaf_f32<NV, 0, F32_ROWS, Grid32>, g, lv.L32))));
    NV_FEW(nv, (pw(k_pw_src_f32<NV, EdgeGrid32>, k_near_pw_f32<NV, EdgeGrid32>, e, lv.nrow == 1 ? lv.ncol : 2 * lv.ncol)));
    return 3;
}
