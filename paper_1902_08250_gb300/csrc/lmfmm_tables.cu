// lmfmm_tables.cu -- the FP64 translation tables of a tree: M2L of the free
// space and the four image terms for every class of the lists (both tree
// kinds), and the M2M / L2L shift tables of every level.
//
// Image terms (Lemma M2L, reading G2 for the phase i^{p-q}):
//   A_pq = (i^{p-q}/4pi) Int Z_t^p Z_s^q e^{i lambda dx - s2 h} sigma_m / s2 d lambda,
//   Z_t = (lambda + tau s2)/k2, Z_s = (lambda + vs s2)/k2,
// scaled by S_t(p) S_s(q), S(n) = (k2 w/2)^|n| / |n|!.  Since (lambda + s2)
// (lambda - s2) = k2^2, Z_s = Z_t for tt and bb (vs = tau) and Z_s = 1/Z_t for
// tb and bt (vs = -tau): A_pq depends on p and q through n = p + q or p - q
// alone, and a table needs the 4P + 1 integrals
//   I_n = (1/4pi) Int Z^n e^{i lambda dx - s2 h} sigma_m / s2 d lambda, |n| <= 2P,
// instead of (2P + 1)^2.  They are kept scaled, Ihat_n = I_n (sc/2)^|n| / |n|!
// with sc the larger of the two boxes' k2 w, so that
//   A_pq S_t(p) S_s(q) = i^{p-q} Ihat_n (|n|! / (|p|! |q|!)) (sc/2)^{|p|+|q|-|n|}
//                        (sc_t/sc)^|p| (sc_s/sc)^|q|.
// With lambda -> -lambda (Z -> -1/Z, the rest even): I_n(-dx) = (-1)^n I_{-n}(dx),
// so classes that differ in the sign of dx share their integrals.
#include <math.h>
#include <algorithm>
#include <map>
#include <tuple>

#include "internal.h"
#include "tables.cuh"

namespace {

#define TI_CHUNK 64   // nodes a round
#define TI_THREADS 128
#define TI_ROUNDS 8   // rounds of one block

struct ImgInt { // one set of integrals: (term, dx >= 0, h) at scale sc
    TabContour C;
    double dx, h, sc;
    int term, item0, item1; // its partial sums
};
struct ImgItem { // a block's share of the rounds of integrals `u`
    int u, round0, round1;
};
struct ImgCls { // one table
    zd *out;
    double rt, rs; // sc_t / sc, sc_s / sc
    int u, flip;   // integrals, and whether the class has dx < 0
};
struct FreeCls {
    zd *out;
    const double *st, *ss;
    double cx, cy;
};

__device__ inline int ti_seg_rounds(const TabContour &C) { return (C.nseg() + TI_CHUNK - 1) / TI_CHUNK; }

// Partial sums of the 4P + 1 integrals over some rounds of 64 node pairs (a node
// of the right half contour and its mirror image on the left).  Thread j < 64
// evaluates the right node's weight and the powers Z^n, thread 64 + j the left
// node's weight and the powers Z^-n; the mirror's powers are (-1)^n Z^-n
// (segment, lambda -> -lambda) or (-1)^n conj(Z^-n) (ray, lambda -> -conj lambda).
// Bound by the FP64 pipe (2 DFMA per clock and SM): about 1600 DFMAs to evaluate
// a pair of nodes, 12P + 8 (4P + 1) per pair for powers and sums.  100k mixed tree
// of five levels (p = 14): 0.66 ms, k_image_expand 0.02 ms; 78.0 ms with a block per
// class for its (2P + 1)^2 integrals.
__global__ void __launch_bounds__(TI_THREADS) k_image_int(MediumD m, int P, const ImgInt *ints, const ImgItem *items,
                                                          zd *part)
{
    extern __shared__ zd ti_smem[];
    const int nn = 4 * P + 1;
    zd *ZP = ti_smem;             // [TI_CHUNK][nn]: powers -2P..2P
    zd *BW = ZP + TI_CHUNK * nn;  // [2][TI_CHUNK]: weights right, left
    __shared__ double fs[4 * LM_MAXP / 2 + 1]; // sc / (2 n)
    const ImgItem it = items[blockIdx.x];
    const ImgInt &I = ints[it.u];
    const int tau = (I.term == 2 || I.term == 4) ? 1 : -1, is = I.term == 1 ? 0 : (I.term == 2 ? 1 : 2);
    const int j = threadIdx.x & (TI_CHUNK - 1), left = threadIdx.x / TI_CHUNK;
    for (int n = 1 + threadIdx.x; n <= 2 * P; n += TI_THREADS) fs[n] = 0.5 * I.sc / n;
    const int segr = ti_seg_rounds(I.C), nseg = I.C.nseg(), ntail = I.C.ntail();
    zd aR[2], aL[2]; // 4P + 1 <= 193 integrals on 128 threads
    for (int e = 0; e < 2; ++e) aR[e] = aL[e] = zd{0.0, 0.0};
    for (int r = it.round0; r < it.round1; ++r) {
        const bool tail = r >= segr; // a round holds nodes of one kind
        const int o = (tail ? r - segr : r) * TI_CHUNK + j, lim = tail ? ntail : nseg;
        __syncthreads();
        zd *row = ZP + j * nn + 2 * P;
        if (o < lim) {
            zd lam, dl, s2, sig[3];
            tab_node(I.C, tail ? nseg + o : o, left ? -1 : 1, &lam, &dl);
            densities(m, lam, &s2, sig);
            const zd ex = cexpd(zd{-lam.im * I.dx, lam.re * I.dx} - I.h * s2);
            BW[left * TI_CHUNK + j] = cdiv(dl * ex * sig[is], s2) * (1.0 / (4.0 * M_PI));
            if (left) { // back to the right node, for its powers
                lam = tail ? -conj(lam) : -lam;
                if (tail) s2 = conj(s2);
            }
            // Z = (lam + tau s2)/k2 and 1/Z = (lam - tau s2)/k2, in the form without cancellation
            const zd ap = lam + (double)tau * s2, am = lam - (double)tau * s2;
            const bool up = abs2(ap) >= abs2(am);
            const zd zp = up ? (1.0 / m.k2) * ap : cdiv(zd{m.k2, 0.0}, am);
            const zd zm = up ? cdiv(zd{m.k2, 0.0}, ap) : (1.0 / m.k2) * am;
            const zd z = left ? zm : zp;
            const int st = left ? -1 : 1;
            zd v = {1.0, 0.0};
            if (!left) row[0] = v;
            for (int n = 1; n <= 2 * P; ++n) {
                v = v * (fs[n] * z);
                row[st * n] = v;
            }
        } else {
            BW[left * TI_CHUNK + j] = zd{0.0, 0.0};
            for (int n = left ? -2 * P : 0; n <= (left ? -1 : 2 * P); ++n) row[n] = zd{0.0, 0.0};
        }
        __syncthreads();
        const double cj = tail ? -1.0 : 1.0;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int n = threadIdx.x + e * TI_THREADS;
            if (n >= nn) break;
            const zd *zr = ZP + n, *zl = ZP + nn - 1 - n;
            for (int i = 0; i < TI_CHUNK; ++i) {
                cfma(aR[e], BW[i], zr[i * nn]);
                const zd a = zl[i * nn];
                cfma(aL[e], BW[TI_CHUNK + i], zd{a.re, cj * a.im});
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int n = threadIdx.x + e * TI_THREADS;
        if (n < nn) part[(int64_t)blockIdx.x * nn + n] = (n & 1) ? aR[e] - aL[e] : aR[e] + aL[e]; // 2P is even
    }
}

// The tables of the image classes from their integrals: one block per class.
__global__ void __launch_bounds__(256) k_image_expand(int P, const ImgInt *ints, const ImgCls *cls, const zd *part,
                                                      int *flag)
{
    const int np = 2 * P + 1, nn = 4 * P + 1;
    __shared__ zd In[4 * LM_MAXP + 1];
    __shared__ double fact[2 * LM_MAXP + 1], pw[LM_MAXP + 1], rt[LM_MAXP + 1], rs[LM_MAXP + 1];
    const ImgCls c = cls[blockIdx.x];
    const ImgInt &I = ints[c.u];
    for (int n = threadIdx.x; n < nn; n += blockDim.x) {
        zd s = {0.0, 0.0};
        for (int k = I.item0; k < I.item1; ++k) s = s + part[(int64_t)k * nn + n];
        // dx < 0: I_n(-dx) = (-1)^n I_{-n}(dx)
        In[c.flip ? nn - 1 - n : n] = (c.flip && (n & 1)) ? -s : s;
    }
    if (threadIdx.x < 4) {
        double v = 1.0;
        const int lim = threadIdx.x == 0 ? 2 * P : P;
        double *a = threadIdx.x == 0 ? fact : threadIdx.x == 1 ? pw : threadIdx.x == 2 ? rt : rs;
        for (int n = 0; n <= lim; ++n) {
            a[n] = v;
            v *= threadIdx.x == 0 ? (double)(n + 1) : threadIdx.x == 1 ? 0.5 * I.sc : threadIdx.x == 2 ? c.rt : c.rs;
        }
    }
    __syncthreads();
    const bool sum = I.term <= 2; // tt, bb: n = p + q; tb, bt: n = p - q
    for (int idx = threadIdx.x; idx < np * np; idx += blockDim.x) {
        const int p = idx / np - P, q = idx % np - P, n = sum ? p + q : p - q;
        const int ap = abs(p), aq = abs(q), an = abs(n);
        // (sc/2)^{|p|+|q|-|n|} as two equal powers beside their factorials: the whole power alone passes FP64's
        // range for sc above 3235 at P = 48, where the entries do not
        const double h = pw[(ap + aq - an) >> 1], f = fact[an] * (h / fact[ap] * rt[ap]) * (h / fact[aq] * rs[aq]);
        const zd v = f * In[n + 2 * P];
        const int ph = ((p - q) % 4 + 4) % 4; // i^{p-q}
        const zd r = ph == 0 ? v : ph == 1 ? zd{-v.im, v.re} : ph == 2 ? -v : zd{v.im, -v.re};
        if (!isfinite(r.re) || !isfinite(r.im)) atomicOr(flag, 16);
        c.out[idx] = r;
    }
}

// Free-space M2L (Rokhlin's translation): A_pq = (i/4) H_{q-p}(k rho) e^{i (q-p) theta},
// c = target centre - source centre; scaled by S_t(p) S_s(q).  One block per class:
// the 2P + 1 Hankel values and 4P + 1 phases are formed once (a thread each: jn and
// yn are serial recurrences), then every entry is a product.
__global__ void __launch_bounds__(256) k_free_tab(double k, int P, const FreeCls *cls)
{
    const int np = 2 * P + 1;
    __shared__ double jv[2 * LM_MAXP + 1], yv[2 * LM_MAXP + 1];
    __shared__ zd ph[2 * LM_MAXP + 1];
    const FreeCls c = cls[blockIdx.x];
    const double rho = hypot(c.cx, c.cy), th = atan2(c.cy, c.cx);
    for (int i = threadIdx.x; i < 3 * np; i += blockDim.x) {
        const int n = i % np, what = i / np;
        if (what == 0) jv[n] = jn(n, k * rho);
        else if (what == 1) yv[n] = yn(n, k * rho);
        else ph[n] = zd{cos(n * th), sin(n * th)};
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < np * np; idx += blockDim.x) {
        const int p = idx / np - P, q = idx % np - P, n = q - p, a = abs(n);
        const double sg = (n < 0 && (a & 1)) ? -1.0 : 1.0, s = sg * c.st[abs(p)] * c.ss[abs(q)];
        const zd h = {-0.25 * yv[a] * s, 0.25 * jv[a] * s}; // (i/4)(J + iY) S_t S_s
        c.out[idx] = h * (n < 0 ? conj(ph[a]) : ph[a]);
    }
}

// M2M and L2L tables, one block per (job, child position):
//  M2M (Lemma M2M, reading G3): M_p += sum_q M_q J_{p-q}(k r) e^{-i (p-q) theta},
//     (r, theta) = child centre - parent centre; scaled by S_child(q)/S_parent(p).
//  L2L (Lemma L2L, reading G3): the same kernel with (r, theta) = parent centre -
//     child centre; scaled by S_child(p)/S_parent(q).
__global__ void __launch_bounds__(256) k_shift_tab(int P, const ShiftJob *jobs)
{
    const int np = 2 * P + 1;
    __shared__ double jv[2 * LM_MAXP + 1];
    __shared__ zd ph[2 * LM_MAXP + 1];
    const ShiftJob J = jobs[blockIdx.x >> 2];
    const int pos = blockIdx.x & 3, dy = pos >> 1, dx = pos & 1;
    const double sx = (dx - 0.5) * J.wc, sy = -(dy - 0.5) * J.wc; // child centre - parent centre
    const double r = hypot(sx, sy), th = atan2(sy, sx);
    for (int i = threadIdx.x; i < 2 * np; i += blockDim.x) {
        const int n = i % np;
        if (i < np) jv[n] = jn(n, J.k * r);
        else ph[n] = zd{cos(n * th), -sin(n * th)}; // e^{-i n theta}
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < np * np; idx += blockDim.x) {
        const int p = idx / np - P, q = idx % np - P, n = p - q, a = abs(n);
        const double jn_ = (n < 0 && (a & 1)) ? -jv[a] : jv[a];
        const zd e = n < 0 ? conj(ph[a]) : ph[a];
        const int64_t o = (int64_t)pos * np * np + idx;
        if (J.m2m) J.m2m[o] = (jn_ * (J.sc_child[abs(q)] / J.sc_par[abs(p)])) * e;
        // theta + pi: e^{-i n (theta + pi)} = (-1)^n e^{-i n theta}
        if (J.l2l) J.l2l[o] = (((a & 1) ? -jn_ : jn_) * (J.sc_child[abs(p)] / J.sc_par[abs(q)])) * e;
    }
}

template <typename T> size_t put(std::vector<unsigned char> &buf, const std::vector<T> &v)
{
    const size_t at = (buf.size() + 15) / 16 * 16;
    buf.resize(at + v.size() * sizeof(T));
    if (!v.empty()) std::copy((const unsigned char *)v.data(), (const unsigned char *)(v.data() + v.size()), buf.begin() + at);
    return at;
}

} // namespace

lm_status lm_build_shift_tables(int P, const std::vector<ShiftJob> &jobs, LmArena &tmp, cudaStream_t st)
{
    if (jobs.empty()) return LM_OK;
    ShiftJob *d;
    const lm_status r = lm_dalloc(tmp, &d, jobs.size());
    if (r != LM_OK) return r;
    LM_CUDA(cudaMemcpyAsync(d, jobs.data(), jobs.size() * sizeof(ShiftJob), cudaMemcpyHostToDevice, st));
    k_shift_tab<<<(unsigned)(4 * jobs.size()), 256, 0, st>>>(P, d);
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}

lm_status lm_build_m2l_tables(const MediumD &md, int P, const std::vector<M2LClass> &cls, int *dflag, LmArena &tmp, cudaStream_t st)
{
    const int nn = 4 * P + 1;
    const double km = fmax(md.k1, fmax(md.k2, md.k3)), kmin = fmin(md.k1, fmin(md.k2, md.k3));
    std::vector<FreeCls> fc;
    std::vector<ImgCls> ic;
    std::vector<ImgInt> ints;
    std::vector<ImgItem> items;
    std::map<std::tuple<int, double, double, double>, int> seen; // term, |dx|, h, scale
    for (const M2LClass &c : cls) {
        if (c.term == 0) {
            if (!md.deriv) fc.push_back(FreeCls{c.out, c.scale_t, c.scale_s, c.dx, c.dy});
            continue;
        }
        const double sc = std::max(c.sc_t, c.sc_s);
        auto ins = seen.insert({{c.term, fabs(c.dx), c.dy, sc}, (int)ints.size()});
        if (ins.second) {
            ImgInt I;
            I.C = tab_contour(km, kmin, P, fabs(c.dx), c.dy);
            I.dx = fabs(c.dx);
            I.h = c.dy;
            I.sc = sc;
            I.term = c.term;
            I.item0 = (int)items.size();
            const int nr = (I.C.nseg() + TI_CHUNK - 1) / TI_CHUNK + (I.C.ntail() + TI_CHUNK - 1) / TI_CHUNK;
            for (int r = 0; r < nr; r += TI_ROUNDS) items.push_back({(int)ints.size(), r, std::min(nr, r + TI_ROUNDS)});
            I.item1 = (int)items.size();
            ints.push_back(I);
        }
        ic.push_back(ImgCls{c.out, c.sc_t / sc, c.sc_s / sc, ins.first->second, c.dx < 0.0});
    }
    std::vector<unsigned char> buf;
    const size_t of = put(buf, fc), oc = put(buf, ic), oi = put(buf, ints), ot = put(buf, items);
    if (buf.empty()) return LM_OK;
    const size_t op = (buf.size() + 15) / 16 * 16;
    unsigned char *d;
    const lm_status r = lm_dalloc(tmp, &d, op + items.size() * nn * sizeof(zd));
    if (r != LM_OK) return r;
    LM_CUDA(cudaMemcpyAsync(d, buf.data(), buf.size(), cudaMemcpyHostToDevice, st));
    if (!fc.empty()) k_free_tab<<<(unsigned)fc.size(), 256, 0, st>>>(md.k2, P, (const FreeCls *)(d + of));
    if (!ic.empty()) {
        const size_t shm = ((size_t)TI_CHUNK * nn + 2 * TI_CHUNK) * sizeof(zd);
        LM_CUDA(lm_raise_smem((const void *)k_image_int, LM_SMEM_IMAGE_M2L, (int)shm));
        k_image_int<<<(unsigned)items.size(), TI_THREADS, shm, st>>>(md, P, (const ImgInt *)(d + oi),
                                                                   (const ImgItem *)(d + ot), (zd *)(d + op));
        k_image_expand<<<(unsigned)ic.size(), 256, 0, st>>>(P, (const ImgInt *)(d + oi), (const ImgCls *)(d + oc),
                                                            (const zd *)(d + op), dflag);
    }
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}
