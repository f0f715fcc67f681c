// lmfmm_setup.cu -- Algorithm 1, step 1 on the device: the strip-forest
// quadtree, interaction lists, translation tables and near-field quadrature.
#include <math.h>
#include <cmath>
#include <stdio.h>
#include <algorithm>
#include <map>
#include <tuple>

#include "internal.h"
#include "lists.cuh"
#include "tables.cuh"

// ---------------------------------------------------------------------------
// Tree
// ---------------------------------------------------------------------------
__global__ void k_minmax(const double *x, const double *y, int64_t n, double d, double *bmin,
                         double *bmax, int *flag)
{
    __shared__ double smin[256], smax[256];
    double mn = 1e308, mx = -1e308;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        double xi = x[i], yi = y[i];
        if (!isfinite(xi) || !isfinite(yi) || !(yi < 0.0) || !(yi > -d)) atomicOr(flag, 1);
        mn = fmin(mn, xi);
        mx = fmax(mx, xi);
    }
    smin[threadIdx.x] = mn;
    smax[threadIdx.x] = mx;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            smin[threadIdx.x] = fmin(smin[threadIdx.x], smin[threadIdx.x + s]);
            smax[threadIdx.x] = fmax(smax[threadIdx.x], smax[threadIdx.x + s]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        bmin[blockIdx.x] = smin[0];
        bmax[blockIdx.x] = smax[0];
    }
}

// leaf of each point: col = floor((x - x0)/w), row = floor(-y/w), clamped
__global__ void k_keys(const double *x, const double *y, int64_t n, double x0, double w,
                       int64_t ncol, int64_t nrow, int32_t *key, int32_t *cnt)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t c = (int64_t)floor((x[i] - x0) / w), r = (int64_t)floor(-y[i] / w);
    c = c < 0 ? 0 : (c > ncol - 1 ? ncol - 1 : c);
    r = r < 0 ? 0 : (r > nrow - 1 ? nrow - 1 : r);
    int32_t k = (int32_t)(r * ncol + c);
    key[i] = k;
    atomicAdd(&cnt[k], 1);
}

// exclusive scan of cnt[0..m) into start[0..m] by one block
__global__ void k_scan(const int32_t *cnt, int64_t m, int64_t *start)
{
    __shared__ int64_t part[1024];
    int64_t chunk = (m + blockDim.x - 1) / blockDim.x;
    int64_t lo = threadIdx.x * chunk, hi = min(m, lo + chunk);
    int64_t s = 0;
    for (int64_t i = lo; i < hi; ++i) s += cnt[i];
    part[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t acc = 0;
        for (int i = 0; i < (int)blockDim.x; ++i) {
            int64_t v = part[i];
            part[i] = acc;
            acc += v;
        }
        start[m] = acc;
    }
    __syncthreads();
    int64_t acc = part[threadIdx.x];
    for (int64_t i = lo; i < hi; ++i) {
        start[i] = acc;
        acc += cnt[i];
    }
}

__global__ void k_scatter(const int32_t *key, int64_t n, const int64_t *start, int32_t *cursor,
                          int64_t *tmp)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int32_t k = key[i];
    int pos = atomicAdd(&cursor[k], 1);
    tmp[start[k] + pos] = i;
}

// sort each leaf's input indices ascending (bitonic sort in shared memory)
__global__ void k_leafsort(const int64_t *start, int64_t *idx, int *flag)
{
    __shared__ int32_t s[LM_MAXLEAF];
    int64_t b = blockIdx.x;
    int64_t lo = start[b], cnt = start[b + 1] - lo;
    if (cnt <= 1) return;
    if (cnt > LM_MAXLEAF) {
        if (threadIdx.x == 0) atomicOr(flag, 2);
        return;
    }
    int m = 1;
    while (m < cnt) m <<= 1;
    for (int i = threadIdx.x; i < m; i += blockDim.x) s[i] = i < cnt ? (int32_t)idx[lo + i] : INT32_MAX;
    __syncthreads();
    for (int k = 2; k <= m; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < m; i += blockDim.x) {
                int ixj = i ^ j;
                if (ixj > i) {
                    bool up = (i & k) == 0;
                    int32_t a = s[i], c = s[ixj];
                    if ((a > c) == up) {
                        s[i] = c;
                        s[ixj] = a;
                    }
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) idx[lo + i] = s[i];
}

__global__ void k_gather_pts(const double *x, const double *y, const int64_t *perm, int64_t n,
                             double *xs, double *ys)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t j = perm[i];
    xs[i] = x[j];
    ys[i] = y[j];
}

// ---------------------------------------------------------------------------
// Interaction lists.  Image row of source row r for term m at a level with
// nrow rows: free r; tt -1-r (mirror in y = 0); bb 2nrow-1-r (mirror in
// y = -d); tb r-2nrow (shift +2d); bt r+2nrow (shift -2d).
// ---------------------------------------------------------------------------
struct SlotMap {
    int DC;          // dc in [-DC, DC]
    int32_t *map;    // [5][2DC+1][7] slot or -1 (dr in [-3, 3])
};
__host__ __device__ inline int slot_index(int DC, int term, int dc, int dr)
{
    return (term * (2 * DC + 1) + (dc + DC)) * 7 + (dr + 3);
}

// pass 0: count (rstart, optional: the entries that the free-space stencil kernels do not cover);
// pass 1: fill. One thread per target box.
__global__ void k_vlist(int l, int64_t ncol, int64_t nrow, int DC, const int32_t *slotmap,
                        int64_t *vstart, int32_t *vsrc, int32_t *vslot, int32_t *vterm, int pass,
                        int *flag, int64_t *rstart)
{
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= ncol * nrow) return;
    int64_t rt = t / ncol, ct = t % ncol;
    int64_t pos = pass ? vstart[t] : 0, cnt = 0, rest = 0;
    for (int term = 0; term < 5; ++term) {
        // source rows in ascending order
        int64_t rlo = 0, rhi = nrow - 1;
        if (l > 0) {
            int64_t a = src_row(term, rt - 3, nrow), b = src_row(term, rt + 3, nrow);
            rlo = max((int64_t)0, min(a, b));
            rhi = min(nrow - 1, max(a, b));
        }
        int64_t clo = l > 0 ? max((int64_t)0, ct - 3) : 0;
        int64_t chi = l > 0 ? min(ncol - 1, ct + 3) : ncol - 1;
        for (int64_t rs = rlo; rs <= rhi; ++rs) {
            int64_t ri = img_row(term, rs, nrow);
            for (int64_t cs = clo; cs <= chi; ++cs) {
                if (!v_rule(l, ct, rt, cs, ri)) continue;
                if (pass) {
                    int64_t dc = ct - cs, dr = rt - ri;
                    int slot = -1;
                    if (dc >= -DC && dc <= DC && dr >= -3 && dr <= 3)
                        slot = slotmap[slot_index(DC, term, (int)dc, (int)dr)];
                    if (slot < 0) atomicOr(flag, 4);
                    vsrc[pos] = (int32_t)(rs * ncol + cs);
                    vslot[pos] = slot < 0 ? 0 : slot;
                    vterm[pos] = term;
                    ++pos;
                }
                ++cnt;
                rest += l == 0 || term > 0;
            }
        }
    }
    if (!pass) vstart[t] = cnt; // counts, scanned by k_scan_lists
    if (!pass && rstart) rstart[t] = rest;
}

// U list at the leaf level: image adjacent to target (free term includes itself)
// pass 0: count (chunks, optional: of 64 source points, for leaves with points); pass 1: fill
__global__ void k_ulist(int64_t ncol, int64_t nrow, int64_t *ustart, int32_t *usrc, int32_t *uterm,
                        int pass, const int64_t *ls, int64_t *chunks)
{
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= ncol * nrow) return;
    int64_t rt = t / ncol, ct = t % ncol;
    int64_t pos = pass ? ustart[t] : 0, cnt = 0, pts = 0;
    for (int term = 0; term < 5; ++term) {
        int64_t a = src_row(term, rt - 1, nrow), b = src_row(term, rt + 1, nrow);
        int64_t rlo = max((int64_t)0, min(a, b)), rhi = min(nrow - 1, max(a, b));
        for (int64_t rs = rlo; rs <= rhi; ++rs) {
            int64_t ri = img_row(term, rs, nrow);
            for (int64_t cs = max((int64_t)0, ct - 1); cs <= min(ncol - 1, ct + 1); ++cs) {
                if (!adj(ct, rt, cs, ri)) continue;
                if (pass) {
                    usrc[pos] = (int32_t)(rs * ncol + cs);
                    uterm[pos] = term;
                    ++pos;
                }
                ++cnt;
                if (chunks) pts += ls[rs * ncol + cs + 1] - ls[rs * ncol + cs];
            }
        }
    }
    if (!pass) ustart[t] = cnt;
    if (chunks) chunks[t] = ls[t + 1] > ls[t] ? (pts + 63) / 64 : 0;
}

// One block per list: counts c[0..m) -> starts c[0..m], in place; tot: their sum, the largest count and
// the number of nonzero counts, whose boxes go to tgt in ascending order (optional)
struct ScanJob {
    int64_t *c;
    int64_t m;
    int64_t *tot; // [3]
    int32_t *tgt; // [m]
};
__global__ void __launch_bounds__(1024) k_scan_lists(const ScanJob *jobs)
{
    __shared__ int64_t ws[32], wn[32], wm[32];
    const ScanJob J = jobs[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t chunk = (J.m + 1023) / 1024, lo = threadIdx.x * chunk, hi = min(J.m, lo + chunk);
    int64_t s = 0, nz = 0, mx = 0;
    for (int64_t i = lo; i < hi; ++i) {
        const int64_t v = J.c[i];
        s += v;
        nz += v > 0;
        mx = max(mx, v);
    }
    int64_t is = s, in = nz;
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t a = __shfl_up_sync(0xffffffffu, is, o), b = __shfl_up_sync(0xffffffffu, in, o);
        if (lane >= o) {
            is += a;
            in += b;
        }
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 31) {
        ws[warp] = is;
        wn[warp] = in;
        wm[warp] = mx;
    }
    __syncthreads();
    int64_t as = is - s, an = in - nz; // exclusive
    for (int w = 0; w < warp; ++w) {
        as += ws[w];
        an += wn[w];
    }
    if (threadIdx.x == 1023) {
        J.c[J.m] = as + s;
        J.tot[0] = as + s;
        for (int w = 0; w < 32; ++w) mx = max(mx, wm[w]);
        J.tot[1] = mx;
        J.tot[2] = an + nz;
    }
    for (int64_t i = lo; i < hi; ++i) {
        const int64_t v = J.c[i];
        J.c[i] = as;
        as += v;
        if (v > 0 && J.tgt) J.tgt[an++] = (int32_t)i;
    }
}

// ---------------------------------------------------------------------------
// Near-field quadrature tables.
//  Segment (first contour, Sec. 5): a trapezoid from 0 down to delta - i a,
//  along -i a to c - delta - i a, and up to c; the negative half is folded
//  onto it (integrand 2 cos(lambda X) ...).  Gauss-Legendre panels.
//  Tail: rays lambda = c + t e^{i phi_k}, phi_k = k (pi/2) / (nray - 1),
//  t = c v/(1-v), Gauss-Legendre in v.  The half-line integrals of
//  e^{+i lambda X} F and e^{-i lambda X} F go to the ray and its mirror image
//  below the axis, with weights W_u, W_l; with E = e^{i lambda X - s2 h} the
//  mirror's factor is conj(E), so the tail is sum P Re(Z) + i M Im(Z) with
//  P = W_u + W_l, M = W_u - W_l and Z = E (or its X- or h-derivative).  For
//  transmission and Dirichlet/Neumann walls sigma(conj lambda) = conj(sigma)
//  and the tail is real; an impedance wall makes it complex.
// ---------------------------------------------------------------------------
// c_o (optional, [2][nseg]): the weights of 2 i beta / s2 (imp_beta) for the gradient's h-derivative
__global__ void k_near_seg(MediumD m, double c, double a, double delta, int nflat, int order,
                           zd *lam_o, zd *s2_o, zd *w_o, int nseg, zd *c_o = nullptr)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nseg) return;
    int pan = i / order, j = i % order;
    double x, w;
    gl_node(order, j, &x, &w);
    zd z0, z1;
    double flat = (c - 2.0 * delta) / nflat;
    if (pan == 0) {
        z0 = {0.0, 0.0};
        z1 = {delta, -a};
    } else if (pan == nflat + 1) {
        z0 = {c - delta, -a};
        z1 = {c, 0.0};
    } else {
        z0 = {delta + (pan - 1) * flat, -a};
        z1 = {delta + pan * flat, -a};
    }
    zd dz = z1 - z0;
    zd lam = z0 + (0.5 * (x + 1.0)) * dz;
    zd s2, sig[3];
    densities(m, lam, &s2, sig);
    zd base = cdiv((0.5 * w / (4.0 * M_PI)) * dz, s2);
    lam_o[i] = lam;
    s2_o[i] = s2;
    w_o[i] = base * (sig[0] - zd{refl_inf(m, 0), 0.0});
    w_o[nseg + i] = base * (sig[1] - zd{refl_inf(m, 1), 0.0});
    if (c_o)
        for (int mm = 0; mm < 2; ++mm) c_o[mm * nseg + i] = base * cdiv(zd{0.0, 2.0 * imp_beta(m, mm)}, s2);
}

// With w2_o set (walls on both sides, FP64): w_o takes the single reflection R - R_inf
// and w2_o the multiple reflections sigma - R, summed on different rays (see NearQuad).
// c_o (optional, layout of w_o): P, M weights of 2 i beta / s2 for the gradient's h-derivative
__global__ void k_near_tail(MediumD m, double c, int nray, int order, zd *lam_o, zd *s2_o, zd *w_o,
                            zd *w2_o = nullptr, zd *c_o = nullptr)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int tot = nray * order;
    if (i >= tot) return;
    int k = i / order, j = i % order;
    double x, w;
    gl_node(order, j, &x, &w);
    double v = 0.5 * (x + 1.0), wv = 0.5 * w;
    double t = c * v / (1.0 - v), dt = c / ((1.0 - v) * (1.0 - v));
    double phi = (nray > 1) ? k * (0.5 * M_PI) / (nray - 1) : 0.0;
    // upper ray (for e^{+i lam X}) and its mirror below the axis (for e^{-i lam X})
    zd e = {cos(phi), sin(phi)};
    zd lam = zd{c, 0.0} + t * e, laml = conj(lam);
    zd s2, sig[3], s2l, sigl[3];
    densities(m, lam, &s2, sig);
    densities(m, laml, &s2l, sigl);
    zd bu = cdiv((wv * dt / (4.0 * M_PI)) * e, s2), bl = cdiv((wv * dt / (4.0 * M_PI)) * conj(e), s2l);
    lam_o[i] = lam;
    s2_o[i] = s2;
    for (int mm = 0; mm < 2; ++mm) {
        const zd ri = {refl_inf(m, mm), 0.0};
        if (c_o) {
            const zd tb = {0.0, 2.0 * imp_beta(m, mm)};
            const zd cu = bu * cdiv(tb, s2), cl = bl * cdiv(tb, s2l);
            c_o[((size_t)(2 * mm) * tot) + i] = cu + cl;
            c_o[((size_t)(2 * mm + 1) * tot) + i] = cu - cl;
        }
        if (w2_o) {
            const double kj = mm == 0 ? m.k1 : m.k3;
            const zd r = refl_coef(m, mm, s2, sbranch(lam, kj), kj), rl = refl_coef(m, mm, s2l, sbranch(laml, kj), kj);
            const zd au = bu * (r - ri), al = bl * (rl - ri), mu = bu * (sig[mm] - r), ml = bl * (sigl[mm] - rl);
            w_o[((size_t)(2 * mm) * tot) + i] = au + al;
            w_o[((size_t)(2 * mm + 1) * tot) + i] = au - al;
            w2_o[((size_t)(2 * mm) * tot) + i] = mu + ml;
            w2_o[((size_t)(2 * mm + 1) * tot) + i] = mu - ml;
            continue;
        }
        const zd wu = bu * (sig[mm] - ri), wl = bl * (sigl[mm] - ri);
        w_o[((size_t)(2 * mm) * tot) + i] = wu + wl;     // P
        w_o[((size_t)(2 * mm + 1) * tot) + i] = wu - wl; // M
    }
}

// ---------------------------------------------------------------------------
// host orchestration
// ---------------------------------------------------------------------------
cudaError_t LmArena::get(void **p, size_t bytes)
{
    bytes = (bytes + 511) / 512 * 512; // what cudaMalloc aligns to
    if (bytes > left) {
        const size_t unit = std::min<size_t>(64u << 20, std::max<size_t>(4u << 20, total));
        size_t want = bytes > unit / 2 ? bytes : unit;
        slabs.reserve(slabs.size() + 1);
        void *m = nullptr;
        cudaError_t e = cudaMalloc(&m, want);
        if (e == cudaErrorMemoryAllocation && want > bytes) {
            cudaGetLastError();
            e = cudaMalloc(&m, want = bytes);
        }
        if (e != cudaSuccess) return e;
        slabs.push_back(m);
        total += want;
        if (want == bytes) { // the open slab stays open
            *p = m;
            return cudaSuccess;
        }
        cur = (char *)m;
        left = want;
    }
    *p = cur;
    cur += bytes;
    left -= bytes;
    return cudaSuccess;
}
void LmArena::release()
{
    for (void *m : slabs) cudaFree(m);
    slabs.clear();
    cur = nullptr;
    left = total = 0;
}

#define TRY(x)                       \
    do {                             \
        lm_status s_ = (x);          \
        if (s_ != LM_OK) return s_;  \
    } while (0)

static int grid_for(int64_t n, int b) { return (int)((n + b - 1) / b); }

lm_status lm_setup_tree(lm_tree_s *t, const double *x, const double *y, cudaStream_t st)
{
    const int64_t n = t->n;
    const double d = t->med.d;
    TRY(lm_dalloc(t, &t->dflag, 4));
    LM_CUDA(cudaMemsetAsync(t->dflag, 0, 4 * sizeof(int), st));
    int nb = (int)std::min<int64_t>(1024, (n + 255) / 256);
    double *bmin, *bmax;
    TRY(lm_dalloc(t->tmp, &bmin, 2 * nb));
    bmax = bmin + nb;
    k_minmax<<<nb, 256, 0, st>>>(x, y, n, d, bmin, bmax, t->dflag);
    std::vector<double> hmin(2 * nb);
    const double *hmax = hmin.data() + nb;
    int hflag = 0;
    LM_CUDA(cudaMemcpyAsync(hmin.data(), bmin, 2 * nb * sizeof(double), cudaMemcpyDeviceToHost, st));
    LM_CUDA(cudaMemcpyAsync(&hflag, t->dflag, sizeof(int), cudaMemcpyDeviceToHost, st));
    LM_CUDA(cudaStreamSynchronize(st));
    if (hflag & 1) {
        lm_set_error("build_tree: a point is non-finite or not strictly inside -d < y < 0");
        return LM_EINVAL;
    }
    double mn = hmin[0], mx = hmax[0];
    for (int i = 1; i < nb; ++i) {
        mn = fmin(mn, hmin[i]);
        mx = fmax(mx, hmax[i]);
    }
    double f0 = floor(mn / d), f1 = floor(mx / d);
    // the number of d x d roots, checked in double before it becomes an int: an
    // x extent of more than 2^30 thicknesses (or one that overflows) is rejected
    const double roots = f1 - f0 + 1.0;
    if (!std::isfinite(roots) || roots < 1.0 || roots > (double)(1 << 30)) {
        lm_set_error("build_tree: the x extent spans %g layer thicknesses; at most 2^30 roots are supported",
                     roots);
        return LM_EINVAL;
    }
    t->x0 = f0 * d;
    t->R = (int)roots;
    if (t->med.opt.depth >= 0) {
        t->L = t->med.opt.depth;
    } else {
        // least L with n <= leaf_target R 4^L, then deeper while the points share
        // a leaf with more than 1.5 leaf_target points on average over the points
        // (sum n_leaf^2 / n: what the direct interactions cost), as long as the
        // leaves stay fewer than twice the points (clustered inputs)
        int L = 0;
        while ((double)n > (double)t->med.opt.leaf_target * t->R * pow(4.0, L)) ++L;
        int32_t *key = nullptr, *cnt = nullptr;
        TRY(lm_dalloc(t->tmp, &key, n));
        for (;; ++L) {
            const int64_t ncol = (int64_t)t->R << L, nrow = (int64_t)1 << L, nl = ncol * nrow;
            if (L >= 14 || nl > std::max<int64_t>(2 * n, t->R)) {
                --L;
                break;
            }
            TRY(lm_dalloc(t->tmp, &cnt, nl));
            LM_CUDA(cudaMemsetAsync(cnt, 0, nl * sizeof(int32_t), st));
            k_keys<<<grid_for(n, 256), 256, 0, st>>>(x, y, n, t->x0, ldexp(d, -L), ncol, nrow, key, cnt);
            std::vector<int32_t> hc(nl);
            LM_CUDA(cudaMemcpyAsync(hc.data(), cnt, nl * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
            LM_CUDA(cudaStreamSynchronize(st));
            double s2 = 0.0;
            for (int32_t c : hc) s2 += (double)c * c;
            if (s2 / n <= 1.5 * t->med.opt.leaf_target) break;
        }
        t->L = std::max(L, 0);
    }
    const int L = t->L;
    const int64_t ncol = (int64_t)t->R << L, nrow = (int64_t)1 << L;
    t->nleaf = ncol * nrow;
    if (t->nleaf > (int64_t)1 << 30) {
        lm_set_error("build_tree: %lld leaves is beyond this build", (long long)t->nleaf);
        return LM_ENOTSUP;
    }
    int32_t *key, *cnt, *cursor;
    int64_t *tmp;
    TRY(lm_dalloc(t->tmp, &key, n));
    TRY(lm_dalloc(t->tmp, &cnt, 2 * t->nleaf));
    cursor = cnt + t->nleaf;
    TRY(lm_dalloc(t, &t->leaf_start, t->nleaf + 1));
    TRY(lm_dalloc(t, &t->perm, n));
    LM_CUDA(cudaMemsetAsync(cnt, 0, 2 * t->nleaf * sizeof(int32_t), st));
    double w = ldexp(d, -L);
    k_keys<<<grid_for(n, 256), 256, 0, st>>>(x, y, n, t->x0, w, ncol, nrow, key, cnt);
    k_scan<<<1, 1024, 0, st>>>(cnt, t->nleaf, t->leaf_start);
    tmp = t->perm;
    k_scatter<<<grid_for(n, 256), 256, 0, st>>>(key, n, t->leaf_start, cursor, tmp);
    k_leafsort<<<(unsigned)t->nleaf, 256, 0, st>>>(t->leaf_start, t->perm, t->dflag);
    TRY(lm_dalloc(t, &t->xs, n));
    TRY(lm_dalloc(t, &t->ys, n));
    k_gather_pts<<<grid_for(n, 256), 256, 0, st>>>(x, y, t->perm, n, t->xs, t->ys);
    LM_CUDA(cudaGetLastError());
    return LM_OK; // an overfull leaf (k_leafsort's flag) is reported by lm_setup_tables
}

// classes (term, dc, dr) reachable under the list rules at level l
static void enumerate_classes(int l, int R, std::vector<std::tuple<int, int, int>> &out)
{
    const int64_t nrow = (int64_t)1 << l, ncol = (int64_t)R << l;
    std::map<std::tuple<int, int, int>, int> seen;
    for (int term = 0; term < 5; ++term)
        for (int64_t rt = 0; rt < nrow; ++rt) {
            int64_t rlo = 0, rhi = nrow - 1;
            if (l > 0) {
                int64_t a = src_row(term, rt - 3, nrow), b = src_row(term, rt + 3, nrow);
                rlo = std::max((int64_t)0, std::min(a, b));
                rhi = std::min(nrow - 1, std::max(a, b));
            }
            for (int64_t rs = rlo; rs <= rhi; ++rs) {
                int64_t ri = img_row(term, rs, nrow);
                if (l == 0) {
                    for (int64_t cs = 0; cs < ncol; ++cs) {
                        int64_t ct = 0; // all dc are reached by some pair at level 0
                        for (ct = 0; ct < ncol; ++ct)
                            if (v_rule(0, ct, rt, cs, ri)) seen[{term, (int)(ct - cs), (int)(rt - ri)}] = 1;
                    }
                } else {
                    for (int64_t ct = 8; ct <= 9; ++ct)
                        for (int64_t cs = ct - 3; cs <= ct + 3; ++cs)
                            if (v_rule(l, ct, rt, cs, ri)) seen[{term, (int)(ct - cs), (int)(rt - ri)}] = 1;
                }
            }
        }
    for (auto &kv : seen) out.push_back(kv.first);
}

// Levels 0..L of the strip forest: scale vectors, the M2M / L2L tables and,
// with boxes set, the FP64 form's per-level expansion arrays of the uniform tree.
lm_status lm_setup_levels(lm_tree_s *t, int L, bool boxes, cudaStream_t st)
{
    const int P = t->p, np = 2 * P + 1;
    const double k = t->med.k2, d = t->med.d;
    t->lev.resize(L + 1);
    double *scale;
    TRY(lm_dalloc(t, &scale, (size_t)(L + 1) * (P + 1)));
    std::vector<double> sc((size_t)(L + 1) * (P + 1));
    for (int l = 0; l <= L; ++l) {
        Level &lv = t->lev[l];
        lv.l = l;
        lv.ncol = (int64_t)t->R << l;
        lv.nrow = (int64_t)1 << l;
        lv.nbox = lv.ncol * lv.nrow;
        lv.w = ldexp(d, -l);
        double f = 0.5 * k * lv.w, v = 1.0;
        for (int n = 0; n <= P; ++n) {
            sc[(size_t)l * (P + 1) + n] = v;
            v *= f / (n + 1);
        }
        lv.scale = scale + (size_t)l * (P + 1);
        if (boxes && t->precision == LM_FP64) {
            TRY(lm_dalloc(t, &lv.M, lv.nbox * np * LM_MAXV));
            TRY(lm_dalloc(t, &lv.Lc, lv.nbox * np * LM_MAXV));
        }
    }
    LM_CUDA(cudaMemcpyAsync(scale, sc.data(), sc.size() * sizeof(double), cudaMemcpyHostToDevice, st));
    // shift tables
    for (int l = 0; l <= L; ++l) {
        Level &lv = t->lev[l];
        lv.m2m = nullptr;
        lv.l2l = nullptr;
        if (l < L) TRY(lm_dalloc(t, &lv.m2m, 4 * np * np));
        if (l > 0) TRY(lm_dalloc(t, &lv.l2l, 4 * np * np));
    }
    std::vector<ShiftJob> jobs;
    for (int l = 0; l < L; ++l) { // child level l+1 -> parent level l
        const Level &par = t->lev[l], &ch = t->lev[l + 1];
        jobs.push_back({k, ch.w, ch.scale, par.scale, par.m2m, ch.l2l});
    }
    return lm_build_shift_tables(P, jobs, t->tmp, st);
}

// Near-field quadrature tables of the reflected direct terms (shared by both tree kinds)
lm_status lm_setup_near(lm_tree_s *t, cudaStream_t st)
{
    MediumD md{t->med.k1,
               t->med.k2,
               t->med.k3,
               t->med.d,
               t->med.opt.kernel == LM_KERNEL_DG_DD,
               {t->med.opt.top_bc, t->med.opt.bottom_bc},
               {t->med.opt.top_alpha, t->med.opt.bottom_alpha}};
    NearQuad &q = t->nq;
    q.rinf[0] = refl_inf(md, 0);
    q.rinf[1] = refl_inf(md, 1);
    const bool walls = !md.deriv && md.bc[0] != LM_BC_TRANSMISSION && md.bc[1] != LM_BC_TRANSMISSION;
    const bool imp = md.bc[0] == LM_BC_IMPEDANCE || md.bc[1] == LM_BC_IMPEDANCE;
    q.hray = (walls && !imp) ? 2.0 * md.d : 0.0; // single table (mixed form): shift only for constant R
    q.split = walls && t->precision == LM_FP64;   // FP64: single and multiple reflections apart
    q.a_zero = !imp;                              // Dirichlet / Neumann: R - R_inf = 0
    double km = fmax(md.k1, fmax(md.k2, md.k3)), kmin = fmin(md.k1, fmin(md.k2, md.k3));
    q.c = 1.5 * km + 1.0;
    double a = 0.5, delta = fmin(0.25, 0.5 * kmin);
    int nflat = (int)ceil((q.c - 2.0 * delta) / 1.0);
    int order = t->med.opt.seg_order;
    q.nseg = (nflat + 2) * order;
    q.nray = t->med.opt.tail_rays;
    q.ntail = t->med.opt.tail_order;
    TRY(lm_dalloc(t, &q.seg_lam, q.nseg));
    TRY(lm_dalloc(t, &q.seg_s2, q.nseg));
    TRY(lm_dalloc(t, &q.seg_w, 2 * q.nseg));
    int nt = q.nray * q.ntail;
    TRY(lm_dalloc(t, &q.tail_lam, nt));
    TRY(lm_dalloc(t, &q.tail_s2, nt));
    TRY(lm_dalloc(t, &q.tail_w, 4 * nt));
    const bool impc = t->precision == LM_FP64 && (imp_beta(md, 0) != 0.0 || imp_beta(md, 1) != 0.0);
    q.beta[0] = imp_beta(md, 0);
    q.beta[1] = imp_beta(md, 1);
    if (impc) TRY(lm_dalloc(t, &q.seg_c, 2 * q.nseg));
    k_near_seg<<<grid_for(q.nseg, 64), 64, 0, st>>>(md, q.c, a, delta, nflat, order, q.seg_lam, q.seg_s2,
                                                     q.seg_w, q.nseg, impc ? q.seg_c : nullptr);
    if (q.split) TRY(lm_dalloc(t, &q.tail_w2, 4 * nt));
    k_near_tail<<<grid_for(nt, 64), 64, 0, st>>>(md, q.c, q.nray, q.ntail, q.tail_lam, q.tail_s2, q.tail_w,
                                                  q.split ? q.tail_w2 : nullptr);
    if (t->precision == LM_FP64) {
        q.ntail_g = std::max(64, q.ntail);
        const int ng = q.nray * q.ntail_g;
        TRY(lm_dalloc(t, &q.tail_lam_g, ng));
        TRY(lm_dalloc(t, &q.tail_s2_g, ng));
        TRY(lm_dalloc(t, &q.tail_w_g, 4 * ng));
        if (q.split) TRY(lm_dalloc(t, &q.tail_w2_g, 4 * ng));
        if (impc) TRY(lm_dalloc(t, &q.tail_c_g, 4 * ng));
        k_near_tail<<<grid_for(ng, 64), 64, 0, st>>>(md, q.c, q.nray, q.ntail_g, q.tail_lam_g, q.tail_s2_g,
                                                      q.tail_w_g, q.split ? q.tail_w2_g : nullptr,
                                                      impc ? q.tail_c_g : nullptr);
    }
    LM_CUDA(cudaGetLastError());
    // FP64: factorise the segment per leaf when its coefficients fit in shared memory
    const size_t pw = lm_near_pw64_smem(q.nseg);
    t->near_pw64 = false;
    if (t->precision == LM_FP64 && pw <= 200 * 1024) {
        TRY(lm_near_pw64_attr(pw));
        t->near_pw64 = true;
        TRY(lm_setup_pwsrc(t, st));
    }
    return LM_OK;
}

lm_status lm_setup_tables(lm_tree_s *t, cudaStream_t st)
{
    const int L = t->L, P = t->p, np = 2 * P + 1;
    const double k = t->med.k2;
    MediumD md{t->med.k1,
               t->med.k2,
               t->med.k3,
               t->med.d,
               t->med.opt.kernel == LM_KERNEL_DG_DD,
               {t->med.opt.top_bc, t->med.opt.bottom_bc},
               {t->med.opt.top_alpha, t->med.opt.bottom_alpha}};
    TRY(lm_setup_levels(t, L, true, st));
    // M2L classes and lists.  The lists are counted and scanned for all levels before the one
    // synchronisation that their sizes need.
    const bool mixed = t->precision == LM_MIXED;
    std::vector<int32_t> smap;
    std::vector<size_t> smap0;
    std::vector<int> dcs;
    for (int l = 0; l <= L; ++l) {
        Level &lv = t->lev[l];
        std::vector<std::tuple<int, int, int>> cls;
        enumerate_classes(l, t->R, cls);
        int DC = l == 0 ? (int)std::max<int64_t>(3, lv.ncol - 1) : 3;
        smap0.push_back(smap.size());
        dcs.push_back(DC);
        smap.resize(smap.size() + (size_t)5 * (2 * DC + 1) * 7, -1);
        for (size_t i = 0; i < cls.size(); ++i) {
            int term = std::get<0>(cls[i]), dc = std::get<1>(cls[i]), dr = std::get<2>(cls[i]);
            lv.cls_term.push_back(term);
            lv.cls_dc.push_back(dc);
            lv.cls_dr.push_back(dr);
            smap[smap0[l] + slot_index(DC, term, dc, dr)] = (int32_t)i;
        }
    }
    int32_t *dmap;
    ScanJob *djobs;
    int64_t *dtot;
    TRY(lm_dalloc(t->tmp, &dmap, smap.size()));
    LM_CUDA(cudaMemcpyAsync(dmap, smap.data(), smap.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    const int nj = mixed ? 2 * (L + 1) + 2 : L + 2; // V, rest (mixed) of every level; U, chunks (mixed)
    TRY(lm_dalloc(t->tmp, &djobs, nj));
    TRY(lm_dalloc(t->tmp, &dtot, 3 * nj));
    std::vector<ScanJob> sj;
    auto vlist = [&](Level &lv, int pass) {
        k_vlist<<<grid_for(lv.nbox, 128), 128, 0, st>>>(lv.l, lv.ncol, lv.nrow, dcs[lv.l], dmap + smap0[lv.l], lv.vstart,
                                                        lv.vsrc, lv.vslot, lv.vterm, pass, t->dflag, lv.rstart);
    };
    for (Level &lv : t->lev) {
        TRY(lm_dalloc(t, &lv.vstart, lv.nbox + 1));
        sj.push_back({lv.vstart, lv.nbox, dtot + 3 * sj.size(), nullptr});
        if (mixed) {
            TRY(lm_dalloc(t, &lv.rstart, lv.nbox + 1));
            TRY(lm_dalloc(t, &lv.rtgt, lv.nbox));
            sj.push_back({lv.rstart, lv.nbox, dtot + 3 * sj.size(), lv.rtgt});
        }
        vlist(lv, 0);
    }
    const int64_t ncol = (int64_t)t->R << L, nrow = (int64_t)1 << L;
    TRY(lm_dalloc(t, &t->ustart, t->nleaf + 1));
    sj.push_back({t->ustart, t->nleaf, dtot + 3 * sj.size(), nullptr});
    if (mixed) {
        TRY(lm_dalloc(t, &t->lf_cbase, t->nleaf + 1));
        sj.push_back({t->lf_cbase, t->nleaf, dtot + 3 * sj.size(), nullptr});
    }
    k_ulist<<<grid_for(t->nleaf, 128), 128, 0, st>>>(ncol, nrow, t->ustart, nullptr, nullptr, 0, t->leaf_start, t->lf_cbase);
    LM_CUDA(cudaMemcpyAsync(djobs, sj.data(), nj * sizeof(ScanJob), cudaMemcpyHostToDevice, st));
    k_scan_lists<<<nj, 1024, 0, st>>>(djobs);
    LM_CUDA(cudaGetLastError());
    std::vector<int64_t> tot(3 * nj);
    int hflag = 0;
    LM_CUDA(cudaMemcpyAsync(tot.data(), dtot, tot.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    LM_CUDA(cudaMemcpyAsync(&hflag, t->dflag, sizeof(int), cudaMemcpyDeviceToHost, st));
    LM_CUDA(cudaStreamSynchronize(st));
    if (hflag & 2) {
        lm_set_error("build_tree: a leaf holds more than %d points; use a deeper tree", LM_MAXLEAF);
        return LM_ENOTSUP;
    }
    const int64_t *ht = tot.data();
    std::vector<M2LClass> tcls;
    for (Level &lv : t->lev) {
        lv.nv = ht[0];
        ht += 3;
        if (mixed) {
            lv.nrest = ht[0];
            lv.nrtgt = ht[2];
            ht += 3;
        }
        TRY(lm_dalloc(t, &lv.vsrc, lv.nv));
        TRY(lm_dalloc(t, &lv.vslot, lv.nv));
        TRY(lm_dalloc(t, &lv.vterm, lv.nv));
        vlist(lv, 1);
        // tables
        int ncls = (int)lv.cls_term.size();
        TRY(lm_dalloc(t, &lv.tab, (size_t)std::max(1, ncls) * np * np));
        if (md.deriv) // the free part does not depend on d: its tables stay zero
            LM_CUDA(cudaMemsetAsync(lv.tab, 0, (size_t)std::max(1, ncls) * np * np * sizeof(zd), st));
        for (int i = 0; i < ncls; ++i) { // free space: target centre - source centre = (dc w, -dr w)
            const double dy = lv.cls_term[i] == 0 ? -lv.cls_dr[i] * lv.w : fabs((double)lv.cls_dr[i]) * lv.w;
            tcls.push_back({lv.cls_term[i], lv.cls_dc[i] * lv.w, dy, k * lv.w, k * lv.w, lv.scale, lv.scale,
                            lv.tab + (size_t)i * np * np});
        }
    }
    TRY(lm_build_m2l_tables(md, P, tcls, t->dflag, t->tmp, st));
    t->nu = ht[0];
    t->umax = ht[1];
    if (mixed) t->lf_nchunk = ht[3];
    TRY(lm_dalloc(t, &t->usrc, t->nu));
    TRY(lm_dalloc(t, &t->uterm, t->nu));
    k_ulist<<<grid_for(t->nleaf, 128), 128, 0, st>>>(ncol, nrow, t->ustart, t->usrc, t->uterm, 1, nullptr, nullptr);
    TRY(lm_setup_near(t, st));
    LM_CUDA(cudaGetLastError());
    if (mixed) {
        TRY(lm_setup_mixed(t, st));
    } else {
        // tree-order potentials
        TRY(lm_dalloc(t, &t->us, (size_t)LM_MAXV * t->n));
    }
    LM_CUDA(cudaMemcpyAsync(&hflag, t->dflag, sizeof(int), cudaMemcpyDeviceToHost, st));
    LM_CUDA(cudaStreamSynchronize(st));
    if (hflag & 4) {
        lm_set_error("build_tree: internal error, an interaction has no translation class");
        return LM_ECUDA;
    }
    if (hflag & 16) {
        lm_set_error("build_tree: a layered M2L table overflowed; lower p");
        return LM_ENOTSUP;
    }
    return mixed ? LM_OK : lm_setup_df(t, st);
}

lm_status lm_list_to_host(lm_tree_s *t, int which, int level, std::vector<int64_t> &rows,
                          cudaStream_t st)
{
    int64_t nb, ne;
    const int64_t *start;
    const int32_t *src, *term;
    if (which == 0) {
        if (level < 0 || level > t->L) {
            lm_set_error("list_export: level %d out of range", level);
            return LM_EINVAL;
        }
        Level &lv = t->lev[level];
        nb = lv.nbox;
        ne = lv.nv;
        start = lv.vstart;
        src = lv.vsrc;
        term = lv.vterm;
    } else {
        nb = t->nleaf;
        ne = t->nu;
        start = t->ustart;
        src = t->usrc;
        term = t->uterm;
    }
    std::vector<int64_t> hs(nb + 1);
    std::vector<int32_t> hsrc(ne), hterm(ne);
    LM_CUDA(cudaMemcpyAsync(hs.data(), start, (nb + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    if (ne > 0) {
        LM_CUDA(cudaMemcpyAsync(hsrc.data(), src, ne * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        LM_CUDA(cudaMemcpyAsync(hterm.data(), term, ne * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    }
    LM_CUDA(cudaStreamSynchronize(st));
    rows.resize(3 * ne);
    for (int64_t b = 0; b < nb; ++b)
        for (int64_t e = hs[b]; e < hs[b + 1]; ++e) {
            rows[3 * e] = b;
            rows[3 * e + 1] = hterm[e];
            rows[3 * e + 2] = hsrc[e];
        }
    return LM_OK;
}

void lm_free_tree_device(lm_tree_s *t)
{
    t->tmp.release();
    t->mem.release();
    cudaGetLastError(); // teardown leaves no error behind for the caller's next call
}
