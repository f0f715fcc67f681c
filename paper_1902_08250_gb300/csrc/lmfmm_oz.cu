// lmfmm_oz.cu -- the FP64 form's M2L on the tensor cores (tcgen05, kind::f16) by
// error-free slicing (Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012;
// Mukunoki et al., ISC 2020): tables and multipoles are scaled to fixed point and cut
// into 5 signed digits of 10 bits, held exactly in FP16.  The digit pairs i + j <= 4 are
// kept, those of one weight 2^{-10 w}, w = i + j, in one FP32 accumulator, and the 5 sums of
// an output are combined in double-float.
//
// Scales.  Powers of two: one per order of a level's tables (rows), one per vector of a level's multipoles, one per
// box and vector of L2L's sources, whose targets have one entry.  Components are below 1/2 then, row sums at most 4.
// Accuracy is that of fixed point, 2^-50 of the scales: in M2L and M2M a box whose multipole is 10^-k of the level's
// largest keeps k digits fewer than the 15 of the largest, where double-float keeps 48 bits of every box.  The orders'
// and the boxes' scales are for the target gradient, which magnifies order p by |p| / w.  From the IEEE form, 250k
// strip, 16 vectors, p = 20: potentials 4.8e-14, gradient 6.1e-14 (one scale a level: 5.1e-14, 2.7e-13; contractions in
// double-float: 3.2e-13, 2.8e-13); 20k points on leaves of 1/64, sources 1e10 times weaker than those at the
// strip's end, gradient 6 units from there 9.1e-13 (3.1e-12; 1.8e-13).
//
// Exactness.  Digits are at most 2^9, so an entry adds at most 2^9 (A_0 + .. + A_w) to accumulator w, A_j
// the sum of the magnitudes of the j-th digits of its table row.  That is 2^25 and more for 128 orders of
// any size, but a table's rows decay: the set-up adds up A_0 + A_1 over the entries of every reading of the
// level's lists, and so many entries G <= OZ_GRP are summed before a reading that 2^9 times the largest such sum is
// at most 2^24: accumulators 0 and 1 hold their integers exactly whatever the multipoles are.  (M2L with 3
// entries a reading: 0.74 to 0.98 x 2^24 for box widths k w up to 1 and p up to 31; 2 entries 0.98 at k w = 2, one
// 0.55 at 4, 0.87 at 16; M2M 2 or 3.)
// Accumulator 2 stays below 3 x 2^24: it rounds, in units of 2^-40 of the product of the scales, where
// the second digits of several sources are near their largest and match a row's in sign.  For digits that
// do not know of each other its sum is 10 standard deviations below 2^24.  Those of w = 3 and 4 round in
// units of 2^-50 and 2^-60.
//
// Levels of at least OZ_MINBOX boxes of uniform trees, their M2M and L2L
// from OZ_MINSHIFT; the others run on the CUDA cores (lmfmm_exp_df.cu).
//
// A tile is 128 columns: 128 / nvs target boxes of one row and parity class, nvs vectors
// each.  An interior box's V list depends only on its row and its column's parity, so
// the tiles of a (row, parity) share one entry list (table slot, column offset dc, source
// row).  A source outside the strip is a zero box: each row of split multipoles is padded.
// One entry adds D_{i+j}[128 x R] += S_i[128 x K] T_j[R x K]^T over 15 digit pairs, with S
// the sources, T the real-block table ([Re -Im; Im Re], rows and columns 2 n + re / im)
// and K = 2(2p+1) padded to 16.  R <= 96: five accumulators of R columns share the 512 columns
// of tensor memory; orders with more rows take two sweeps.  (Tables as the 128-row operand
// against 64 columns, 38 of whose rows are padding at p = 22, read 6 KB of shared memory an
// MMA for half the columns: 250k strip, 16 vectors, M2L, M2M and L2L 5.85 ms, 3.07 ms
// this way round.)
//
// Operands lie in global memory as [digit][8-wide K chunk][row][8 FP16]: 8 rows of a
// chunk are a core matrix of the canonical K-major no-swizzle layout (stride 128 B between
// 8-row groups), a stage of a table is one bulk copy, and any run of boxes one per digit and
// chunk, whatever its offset.  Stages of up to 48 K (107 KB), two in flight.  Roles as in lmfmm_tc_tiles.cu:
// a producer warp (a lane per copy), an MMA warp, 8 epilogue warps that read the 5
// accumulators once per G entries: there is room for one set of accumulators, so that
// reading them (about 50 FP32 instructions an element) and the MMAs take turns (250k strip, 16
// vectors, the apply with G = 4, 3, 2 and 1 everywhere: 6.95, 7.06, 7.37 and 8.14 ms; 7.19 as chosen).  A lane of an epilogue warp holds a column,
// so that it writes whole components, neighbouring vectors beside each other.
// Bound by the copies from L2 (215 KB an entry and 128 columns at p = 22) and the
// shared-memory reads of the MMAs' operands (7 KB each at 128 B per clock).
#include <algorithm>

#include <cuda_fp16.h>

#include "df.cuh"
#include "internal.h"
#include "lists.cuh"
#include "near64.cuh"
#include "tc_common.cuh"

#define OZ_S 5        // digits
#define OZ_BITS 10
#define OZ_N 128      // columns of a tile
#define OZ_RN 96      // most table rows of a sweep: 5 accumulators of OZ_RN columns in 512 of tensor memory
#define OZ_KC 6       // 8-wide K chunks of a full stage
#define OZ_NST 2
#define OZ_A_BYTES (OZ_S * OZ_KC * OZ_N * 16)  // sources
#define OZ_B_BYTES (OZ_S * OZ_KC * OZ_RN * 16) // tables
#define OZ_STAGE (OZ_A_BYTES + OZ_B_BYTES)
#define OZ_EPI 8
#define OZ_THREADS ((OZ_EPI + 2) * 32)
#define OZ_SMEM (OZ_NST * OZ_STAGE + 128)

// Smaller levels leave most SMs without a tile.  250k strip, 16 vectors: levels of up to 2047 boxes in
// k_m2l_dx 2.67 ms, of up to 255 0.20 ms and 0.15 ms more here.
#define OZ_MINBOX 256
// M2M and L2L read and write a level for one or four entries a tile and split the sources in a launch
// of their own.  250k strip, 16 vectors (levels of 20480 and 5120 boxes): 4.5 ms on the CUDA cores,
// 1.7 ms with these two levels here; walled adjoint of 20k points (no level as large): 658 us, 680 us
// with its levels of 256 boxes here.
#define OZ_MINSHIFT 4096
#define OZ_PADL 2
#define OZ_GRP 4 // most entries summed in the accumulators before they are read

// One level of a contraction: M2L (sources and targets a level's boxes), M2M (sources the children,
// targets a level) or L2L (sources the parents).  Sources lie in planes of consecutive boxes: (row, column
// parity) for M2L and M2M, so that the children (i, j) of consecutive parents are one run; rows for L2L.
struct OzLevel {
    int64_t tile0;          // first tile of the level in the launch
    int32_t ncl, tpr;       // boxes of a target class = of a source plane, tiles of a class
    int32_t tstep, sstep;   // 2: target classes / source planes are (row, parity), 1: rows
    int32_t add, planes;    // L += (L2L); source planes
    int64_t ncol;           // target columns
    const int32_t *e0;      // [classes + 1] entries of each class
    const RowEnt *ents;     // (pad: rs is the source plane itself, its run starts at the tile's first box)
    const unsigned char *A; // split tables
    unsigned char *B;       // split sources
    const int32_t *ea;      // [np] exponent of each order's table rows; [3] largest sum of the first and second digits'
                            // magnitudes over 2, 3, 4 entries of a list
    uint32_t *mmax;         // [LM_MAXV] largest source component per vector; L2L: [sources][LM_MAXV], of each box
    uint32_t *omax;         // the same of the result, or null
    const float4 *M;        // sources
    float4 *L;              // targets
};

__device__ __forceinline__ int oz_exp(uint32_t bits) { return bits ? (int)((bits >> 23) & 0xff) - 127 : -126; }
// entries a reading: 2^9 (their A_0 + A_1) <= 2^24
__device__ __forceinline__ int oz_grp(const int32_t *ea, int np)
{
    for (int g = OZ_GRP; g > 1; --g)
        if (ea[np + g - 2] <= 1 << 15) return g;
    return 1;
}
__device__ __forceinline__ float oz_pow2(int e) { return __int_as_float((max(-126, min(127, e)) + 127) << 23); }
// table rows (2 p + re / im) in sweeps of oz_rows(np), a multiple of 16, at most OZ_RN
__host__ __device__ __forceinline__ int oz_sweeps(int np) { return 2 * np <= OZ_RN ? 1 : 2; }
__host__ __device__ __forceinline__ int oz_rows(int np) { return (2 * np / oz_sweeps(np) + 15) / 16 * 16; }
__host__ __device__ __forceinline__ int oz_chunks(int np) { return (2 * np + 15) / 16 * 2; }
__host__ __device__ __forceinline__ int64_t oz_prow(int ncl, int tb, int nvs) { return (int64_t)(OZ_PADL + ncl + tb + 2) * nvs; }

// ---------------------------------------------------------------------------
// operands
// ---------------------------------------------------------------------------
// largest component and row sum (float bits) of each order over a level's tables
__global__ void __launch_bounds__(128) k_oz_tmax(const zd *tab, int np, uint32_t *tmax)
{
    const zd *T = tab + (int64_t)blockIdx.x * np * np;
    for (int p = threadIdx.x; p < np; p += blockDim.x) {
        float mx = 0.f;
        double s = 0.0;
        for (int q = 0; q < np; ++q) {
            const zd a = T[p * np + q];
            mx = fmaxf(mx, (float)fmax(fabs(a.re), fabs(a.im)));
            s += fabs(a.re) + fabs(a.im);
        }
        if (mx > 0.f) atomicMax(tmax + p, __float_as_uint(mx));
        if (s > 0.0) atomicMax(tmax + np + p, __float_as_uint((float)s));
    }
}
// the orders' exponents: components below 2^(e-1), row sums at most 2^(e+2)
__global__ void k_oz_texp(const uint32_t *tmax, int np, int32_t *ea)
{
    const int p = threadIdx.x;
    if (p < np) ea[p] = max(oz_exp(tmax[p]) + 2, oz_exp(tmax[np + p]) - 1);
}
// W[class][p]: the magnitudes of the first two digits of a row of order p (as k_oz_tsplit cuts them; the rows of the
// real and the imaginary part hold the same components)
__global__ void __launch_bounds__(128) k_oz_tsum(const zd *tab, int np, const int32_t *ea, int32_t *W)
{
    const zd *T = tab + (int64_t)blockIdx.x * np * np;
    for (int p = threadIdx.x; p < np; p += blockDim.x) {
        const double sc = ldexp(1.0, OZ_BITS - ea[p]);
        double s = 0.0;
        for (int k = 0; k < 2 * np; ++k) {
            const zd a = T[p * np + (k >> 1)];
            const double x = sc * ((k & 1) ? a.im : a.re), d = rint(x);
            s += fabs(d) + fabs(rint((x - d) * 1024.0));
        }
        W[(int64_t)blockIdx.x * np + p] = (int32_t)s;
    }
}
// one block per list: its readings' sums of W, for 2, 3 and 4 entries a reading
__global__ void __launch_bounds__(128) k_oz_gsum(const RowEnt *ents, const int32_t *e0, int np, const int32_t *W, int32_t *ea)
{
    const int b = e0[blockIdx.x], e = e0[blockIdx.x + 1];
    for (int g = 2; g <= OZ_GRP; ++g) {
        int mx = 0;
        for (int p = threadIdx.x; p < np; p += blockDim.x)
            for (int i = b; i < e; i += g) {
                int s = 0;
                for (int j = i; j < min(i + g, e); ++j) s += W[(int64_t)ents[j].slot * np + p];
                mx = max(mx, s);
            }
        if (mx) atomicMax(ea + np + g - 2, mx);
    }
}
// one thread per (class, 8-wide K chunk, row): 8 components into 5 digit planes
__global__ void __launch_bounds__(256) k_oz_tsplit(const zd *tab, int64_t ncls, int np, const int32_t *ea,
                                                   unsigned char *A)
{
    const int RN = oz_rows(np), ns = oz_sweeps(np), KC = oz_chunks(np);
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= ncls * ns * KC * RN) return;
    const int lrow = (int)(idx % RN), c = (int)(idx / RN % KC);
    const int64_t cs = idx / ((int64_t)RN * KC), cls = cs / ns;
    const int row = (int)(cs % ns) * RN + lrow, p = row >> 1, im = row & 1;
    const zd *T = tab + cls * np * np;
    const double sc = row < 2 * np ? ldexp(1.0, -ea[p]) : 0.0;
    uint16_t d[OZ_S][8];
    for (int i = 0; i < 8; ++i) {
        const int k = 8 * c + i;
        double x = 0.0;
        if (row < 2 * np && k < 2 * np) {
            const zd a = T[p * np + (k >> 1)];
            x = im == (k & 1) ? a.re : (im ? a.im : -a.im);
        }
        x *= sc;
        for (int s = 0; s < OZ_S; ++s) {
            x *= 1024.0;
            const double r = rint(x);
            d[s][i] = __half_as_ushort(__float2half_rn((float)r));
            x -= r;
        }
    }
    // stage-major: [stage of OZ_KC chunks][digit][chunk][row]
    const int st = c / OZ_KC, c0 = st * OZ_KC, kc = min(OZ_KC, KC - c0);
    unsigned char *o = A + (cs * OZ_S * KC + (int64_t)OZ_S * c0) * RN * 16;
    for (int s = 0; s < OZ_S; ++s)
        *(uint4 *)(o + ((int64_t)(s * kc + c - c0) * RN + lrow) * 16) = *(const uint4 *)d[s];
}

// largest component of each vector over a level's sources
__global__ void __launch_bounds__(256) k_oz_mmax(const OzLevel *lvs, int np, int nv)
{
    const OzLevel &lv = lvs[blockIdx.y];
    const int64_t n = (int64_t)lv.planes * lv.ncl * np;
    const int per = blockDim.x / nv, v = threadIdx.x % nv; // threads per round of orders
    float mx = 0.f;
    if ((int)threadIdx.x < per * nv)
        for (int64_t i = blockIdx.x * (int64_t)per + threadIdx.x / nv; i < n; i += (int64_t)gridDim.x * per) {
            const float4 a = lv.M[i * nv + v];
            mx = fmaxf(mx, fmaxf(fabsf(a.x), fabsf(a.z)));
        }
    __shared__ uint32_t s[LM_MAXV];
    if (threadIdx.x < LM_MAXV) s[threadIdx.x] = 0;
    __syncthreads();
    if (mx > 0.f) atomicMax(&s[v], __float_as_uint(mx));
    __syncthreads();
    if ((int)threadIdx.x < nv && s[threadIdx.x]) atomicMax(&lv.mmax[threadIdx.x], s[threadIdx.x]);
}
// L2L: largest component of each source box and vector, a warp per box
__global__ void __launch_bounds__(256) k_oz_bmax(const OzLevel *lvs, int np, int nv)
{
    const OzLevel &lv = lvs[0];
    __shared__ uint32_t s[8][LM_MAXV];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, step = 32 / nv * nv; // a lane keeps to one vector
    const int64_t n = (int64_t)lv.planes * lv.ncl;
    for (int64_t b = blockIdx.x * (int64_t)8 + w; b < n; b += (int64_t)gridDim.x * 8) {
        if (lane < LM_MAXV) s[w][lane] = 0;
        __syncwarp();
        float mx = 0.f;
        if (lane < step)
            for (int i = lane; i < np * nv; i += step) {
                const float4 a = lv.M[b * np * nv + i];
                mx = fmaxf(mx, fmaxf(fabsf(a.x), fabsf(a.z)));
            }
        if (mx > 0.f) atomicMax(&s[w][lane % nv], __float_as_uint(mx));
        __syncwarp();
        if (lane < nv) lv.mmax[b * LM_MAXV + lane] = s[w][lane];
        __syncwarp();
    }
}
// one thread per (plane, row of it, 8-wide K chunk): 4 orders of a (box, vector) into 5 digit
// planes; the padding boxes and vectors beyond nv are written as zeros.  Bound by memory: 250k strip,
// 16 vectors, all levels 0.18 ms (0.27 ms with the real parts of all orders first, which reads each
// component twice)
__global__ void __launch_bounds__(256) k_oz_split(const OzLevel *lvs, int np, int nv, int nvs)
{
    const OzLevel &lv = lvs[blockIdx.y];
    const int KC = oz_chunks(np);
    const int64_t rows = oz_prow(lv.ncl, OZ_N / nvs, nvs), tot = lv.planes * rows * KC;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < tot; idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = idx % rows, pc = idx / rows;
        const int c = (int)(pc % KC);
        const int64_t plane = pc / KC;
        const int v = (int)(r % nvs);
        const int64_t i = r / nvs - OZ_PADL;
        uint16_t d[OZ_S][8];
        const bool on = i >= 0 && i < lv.ncl && v < nv;
        const int64_t box = lv.sstep == 2 ? (plane >> 1) * 2 * lv.ncl + 2 * i + (plane & 1) : plane * lv.ncl + i;
        const float sc = on ? oz_pow2(-(oz_exp(lv.mmax[(lv.add ? box * LM_MAXV : 0) + v]) + 2)) : 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = 8 * c + j;
            float h = 0.f, l = 0.f;
            if (on && k < 2 * np) {
                const float4 a = lv.M[(box * np + (k >> 1)) * nv + v];
                h = (k & 1 ? a.z : a.x) * sc;
                l = (k & 1 ? a.w : a.y) * sc;
            }
#pragma unroll
            for (int s = 0; s < OZ_S; ++s) { // digits of h + l, exact
                h *= 1024.f;
                l *= 1024.f;
                const float g = rintf(h);
                d[s][j] = __half_as_ushort(__float2half_rn(g));
                const df t = two_sum(__fsub_rn(h, g), l);
                h = t.h;
                l = t.l;
            }
        }
        unsigned char *o = lv.B + (plane * OZ_S * KC + c) * rows * 16 + r * 16;
#pragma unroll
        for (int s = 0; s < OZ_S; ++s) *(uint4 *)(o + (int64_t)s * KC * rows * 16) = *(const uint4 *)d[s];
    }
}

// ---------------------------------------------------------------------------
// M2L
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t oz_desc(uint32_t saddr, uint32_t lbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)(lbo >> 4) << 16;  // K-direction core-matrix stride
    d |= (uint64_t)(128 >> 4) << 32;  // 8-row-group stride
    d |= (uint64_t)1 << 46;
    return d;
}
__device__ __forceinline__ void oz_mma(uint32_t dtmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dtmem),
                 "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}
// 8 columns of each of the 5 accumulators (nc columns apart), one wait
__device__ __forceinline__ void oz_ld8x5(uint32_t t0, uint32_t nc, float d[OZ_S][8])
{
    uint32_t r[OZ_S][8];
#pragma unroll
    for (int k = 0; k < OZ_S; ++k)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[k][0]), "=r"(r[k][1]), "=r"(r[k][2]), "=r"(r[k][3]), "=r"(r[k][4]), "=r"(r[k][5]),
                       "=r"(r[k][6]), "=r"(r[k][7])
                     : "r"(t0 + nc * k));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < OZ_S; ++k)
#pragma unroll
        for (int i = 0; i < 8; ++i) d[k][i] = __uint_as_float(r[k][i]);
}
// tile -> level, class, first box of the class, sweep
__device__ __forceinline__ const OzLevel &oz_tile(const OzLevel *lvs, int nlev, int64_t tile, int ns, int *cls, int *i0, int *sw,
                                                  int tb)
{
    int l = nlev - 1;
    while (tile < lvs[l].tile0) --l;
    const int64_t r = tile - lvs[l].tile0;
    const int x = (int)(r % lvs[l].tpr);
    *cls = (int)(r / lvs[l].tpr);
    *i0 = x / ns * tb;
    *sw = x % ns;
    return lvs[l];
}
__device__ __forceinline__ void oz_fail(volatile int *abort_s, int *err)
{
    *abort_s = 1;
    atomicOr(err, 1);
}

// first_limit >= 0: poll limit of the MMA issuer's first wait for operands (the timeout path's test)
__global__ void __launch_bounds__(OZ_THREADS, 1) k_m2l_oz(const OzLevel *lvs, int nlev, int64_t ntiles, int np, int nv, int nvs,
                                                          int *err, int first_limit)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *bars = (uint64_t *)(smem + OZ_NST * OZ_STAGE);
    uint32_t *tslot = (uint32_t *)(bars + 2 * OZ_NST + 2);
    volatile int *abort_s = (volatile int *)(tslot + 1);
    const uint32_t sbase = smem_u32(smem), bfull = smem_u32(bars), bempty = bfull + 8 * OZ_NST, btfull = bfull + 16 * OZ_NST,
                   btempty = btfull + 8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int KC = oz_chunks(np), RN = oz_rows(np), ns = oz_sweeps(np), nst = (KC + OZ_KC - 1) / OZ_KC, tb = OZ_N / nvs;

    if (threadIdx.x == 0) {
        for (int i = 0; i < OZ_NST; ++i) {
            mbar_init(bfull + 8 * i, 1);
            mbar_init(bempty + 8 * i, 1);
        }
        mbar_init(btfull, 1);
        mbar_init(btempty, OZ_EPI);
        *abort_s = *(volatile int *)err; // an earlier CTA gave up: do no work
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;

    if (warp == OZ_EPI) {
        // ---- producer: lane 0 waits for a free stage; lane 31 then copies the tables, lanes 0..29
        // one multipole piece each (5 digits x up to 6 chunks) ----
        uint32_t it = 0;
        int last[OZ_NST];
#pragma unroll
        for (int s = 0; s < OZ_NST; ++s) last[s] = -1;
        bool stop = false;
        for (int64_t tile = blockIdx.x; tile < ntiles && !stop; tile += gridDim.x) {
            int cls, i0, sw;
            const OzLevel &lv = oz_tile(lvs, nlev, tile, ns, &cls, &i0, &sw, tb);
            const int e0 = lv.e0[cls], e1 = lv.e0[cls + 1], c0 = 2 * i0 + (cls & 1);
            const int64_t rows = oz_prow(lv.ncl, tb, nvs);
            for (int base = e0; base < e1 && !stop; base += 32) {
                const int cnt = min(32, e1 - base);
                const RowEnt mine = lane < cnt ? lv.ents[base + lane] : RowEnt{0, 0, 0, 0};
                for (int i = 0; i < cnt && !stop; ++i) {
                    const int slot = __shfl_sync(0xffffffffu, mine.slot, i), dc = __shfl_sync(0xffffffffu, mine.dc, i),
                              rs = __shfl_sync(0xffffffffu, mine.rs, i), direct = __shfl_sync(0xffffffffu, mine.pad, i);
                    const int cs = c0 - dc, par = cs & 1;
                    const int64_t plane = direct ? rs : (int64_t)rs * 2 + par;
                    const int64_t sbox = (direct ? i0 : (cs - par) >> 1) + OZ_PADL; // first source in its padded plane
                    const unsigned char *a = lv.A + ((int64_t)slot * ns + sw) * OZ_S * KC * RN * 16;
                    const unsigned char *b = lv.B + plane * OZ_S * KC * rows * 16 + sbox * nvs * 16;
                    for (int st = 0; st < nst; ++st, ++it) {
                        const int s = (int)(it % OZ_NST), k0 = st * OZ_KC, kc = min(OZ_KC, KC - k0);
                        int ok = 1;
                        if (lane == 0) {
                            ok = mbar_wait_lim(bempty + 8 * s, ((it / OZ_NST) & 1) ^ 1, TC_WAIT_LIMIT, abort_s, err);
                            if (ok) mbar_expect_tx(bfull + 8 * s, OZ_S * kc * (RN + OZ_N) * 16);
                            else oz_fail(abort_s, err);
                        }
                        ok = __shfl_sync(0xffffffffu, ok, 0);
                        if (!ok) {
                            stop = true;
                            break;
                        }
                        const uint32_t sa = sbase + s * OZ_STAGE, sb = sa + OZ_A_BYTES, fb = bfull + 8 * s;
                        if (lane == 31) // the stage's tables are contiguous
                            bulk_g2s(sb, a + (int64_t)OZ_S * k0 * RN * 16, OZ_S * kc * RN * 16, fb);
                        if (lane < OZ_S * kc) {
                            const int dg = lane / kc, c = lane - dg * kc;
                            bulk_g2s(sa + (dg * OZ_KC + c) * OZ_N * 16, b + ((int64_t)dg * KC + k0 + c) * rows * 16, OZ_N * 16, fb);
                        }
                        last[s] = (int)it;
                        __syncwarp();
                    }
                }
            }
        }
        // copies in flight land before the CTA's shared memory is released
        if (lane == 0)
            for (int s = 0; s < OZ_NST; ++s)
                if (last[s] >= 0) mbar_wait_lim(bfull + 8 * s, (last[s] / OZ_NST) & 1, TC_WAIT_LIMIT, nullptr, nullptr);
        __syncwarp();
    } else if (warp == OZ_EPI + 1) {
        // ---- MMA issuer ----
        if (lane == 0) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(RN >> 3) << 17) | ((uint32_t)(OZ_N >> 4) << 24);
            uint32_t it = 0, item = 0;
            int done = -1;
            bool stop = false;
            for (int64_t tile = blockIdx.x; tile < ntiles && !stop && !*abort_s; tile += gridDim.x) {
                int cls, i0, sw;
                const OzLevel &lv = oz_tile(lvs, nlev, tile, ns, &cls, &i0, &sw, tb);
                const int ne = lv.e0[cls + 1] - lv.e0[cls], grp = oz_grp(lv.ea, np);
                for (int e = 0; e < ne && !stop; e += grp, ++item) {
                    if (!mbar_wait_lim(btempty, (item & 1) ^ 1, TC_WAIT_LIMIT, abort_s, err)) {
                        oz_fail(abort_s, err);
                        stop = true;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    int issued = 0;
                    const int nstg = nst * min(grp, ne - e);
                    for (int q = 0, st = 0; q < nstg; ++q, ++it, st = st + 1 == nst ? 0 : st + 1) {
                        const int s = (int)(it % OZ_NST), kc = min(OZ_KC, KC - st * OZ_KC), ks = kc / 2;
                        const int lim = it == 0 && first_limit >= 0 ? first_limit : TC_WAIT_LIMIT;
                        if (!mbar_wait_lim(bfull + 8 * s, (it / OZ_NST) & 1, lim, abort_s, err)) {
                            oz_fail(abort_s, err);
                            stop = true;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t sa = sbase + s * OZ_STAGE, sb = sa + OZ_A_BYTES;
                        for (int kk = 0; kk < ks; ++kk)
#pragma unroll
                            for (int i = 0; i < OZ_S; ++i)
#pragma unroll
                                for (int j = 0; i + j < OZ_S; ++j)
                                    oz_mma(tmem + RN * (i + j), oz_desc(sa + (i * OZ_KC + 2 * kk) * OZ_N * 16, OZ_N * 16),
                                           oz_desc(sb + (j * kc + 2 * kk) * RN * 16, RN * 16), idesc,
                                           (q > 0 || kk > 0 || i > 0) ? 1u : 0u);
                        tc_commit(bempty + 8 * s);
                        ++issued;
                    }
                    if (issued > 0) { // (after a failed wait too: the drain below then covers every MMA issued)
                        tc_commit(btfull);
                        done = (int)item;
                    }
                }
            }
            // MMAs in flight complete before tensor memory is freed
            if (done >= 0) mbar_wait_lim(btfull, done & 1, TC_WAIT_LIMIT, nullptr, nullptr);
        }
        __syncwarp();
    } else {
        // ---- epilogue: warp (quadrant Q, half H): tile columns 32 Q .. + 31, one a lane, half the sweep's rows ----
        const int Q = warp & 3, H = warp >> 2, col = 32 * Q + lane, nr = RN / 2, j = col / nvs, v = col - j * nvs;
        const uint32_t base = tmem + ((uint32_t)(32 * Q) << 16) + (uint32_t)(nr * H);
        uint32_t item = 0;
        bool bad = false;
        for (int64_t tile = blockIdx.x; tile < ntiles && !bad; tile += gridDim.x) {
            int cls, i0, sw;
            const OzLevel &lv = oz_tile(lvs, nlev, tile, ns, &cls, &i0, &sw, tb);
            const int ne = lv.e0[cls + 1] - lv.e0[cls], grp = oz_grp(lv.ea, np);
            df acc[OZ_RN / 2];
#pragma unroll
            for (int r = 0; r < OZ_RN / 2; ++r) acc[r] = df{0.f, 0.f};
            for (int e = 0; e < ne; e += grp, ++item) {
                if (!mbar_wait_lim(btfull, item & 1, TC_WAIT_LIMIT, abort_s, err)) {
                    oz_fail(abort_s, err);
                    bad = true;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int r8 = 0; r8 < OZ_RN / 2; r8 += 8) {
                    if (r8 >= nr) break;
                    float d[OZ_S][8];
                    oz_ld8x5(base + r8, RN, d);
                    if (r8 + 8 == nr) {
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(btempty);
                    }
#pragma unroll
                    for (int c = 0; c < 8; ++c) { // integers of weight 2^{-10 k}
                        const df s = two_sum(d[0][c], d[1][c] * 0x1p-10f);
                        const df u = two_sum(d[2][c] * 0x1p-20f, fmaf(d[4][c], 0x1p-40f, d[3][c] * 0x1p-30f));
                        acc[r8 + c] = df_add(acc[r8 + c], df_add(s, u));
                    }
                }
            }
            if (bad) break;
            if (i0 + j < lv.ncl && v < nv) {
                const int64_t r0 = lv.tstep == 2 ? (int64_t)(cls >> 1) * lv.ncol + (cls & 1) : cls * lv.ncol;
                const int64_t src = lv.add ? ((int64_t)(cls >> 2) * lv.ncl + i0 + j) * LM_MAXV : 0; // L2L: the parent
                const int x0 = oz_exp(lv.mmax[src + v]) + 2 - 2 * OZ_BITS, p0 = (sw * RN + H * nr) / 2;
                float4 *o = lv.L + ((r0 + lv.tstep * (int64_t)(i0 + j)) * np + p0) * nv + v;
                float omx = 0.f;
#pragma unroll
                for (int r8 = 0; r8 < OZ_RN / 2; r8 += 8) {
                    if (r8 >= nr) break;
                    float4 b[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        b[c] = lv.add && p0 + r8 / 2 + c < np ? o[(int64_t)(r8 / 2 + c) * nv] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (p0 + r8 / 2 + c < np) {
                            const int x = x0 + lv.ea[p0 + r8 / 2 + c];
                            const float f = oz_pow2(x / 2), g = oz_pow2(x - x / 2);
                            const df a = acc[r8 + 2 * c], i = acc[r8 + 2 * c + 1];
                            df yr = {a.h * f * g, a.l * f * g}, yi = {i.h * f * g, i.l * f * g};
                            if (lv.add) {
                                yr = df_add(df{b[c].x, b[c].y}, yr);
                                yi = df_add(df{b[c].z, b[c].w}, yi);
                            }
                            o[(int64_t)(r8 / 2 + c) * nv] = make_float4(yr.h, yr.l, yi.h, yi.l);
                            omx = fmaxf(omx, fmaxf(fabsf(yr.h), fabsf(yi.h)));
                        }
                }
                if (lv.omax) {
                    const uint32_t m = __float_as_uint(omx);
                    if (m > *(volatile uint32_t *)&lv.omax[v]) atomicMax(&lv.omax[v], m);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
#define TRY_O(x)                     \
    do {                             \
        lm_status s_ = (x);          \
        if (s_ != LM_OK) return s_;  \
    } while (0)

// whether level l of a uniform FP64 tree takes the tensor cores: its boxes fill the SMs with tiles, its
// order fits the operand
bool lm_oz_level(const lm_tree_s *t, int l)
{
    return !t->adaptive && t->m2l_df && l >= 1 && 2 * t->np <= 128 && t->lev[l].nbox >= OZ_MINBOX;
}

// M2L descriptors of the tensor-core levels, their M2M to the level above, their L2L from it
enum { OZ_M2L = 0, OZ_M2M = 1, OZ_L2L = 2 };
static std::vector<OzLevel> oz_levels(const lm_tree_s *t, int op, int nvs)
{
    std::vector<OzLevel> v;
    const OzData &Z = t->oz;
    const int tb = OZ_N / nvs;
    const size_t nl = Z.lv.size();
    int64_t tiles = 0;
    for (size_t i = 0; i < nl; ++i) {
        const OzData::Lv &z = Z.lv[i];
        const Level &lv = t->lev[z.l], &up = t->lev[z.l - 1];
        const OzData::Op &x = z.op[op];
        OzLevel o{};
        o.tile0 = op == OZ_M2L ? tiles : 0;
        o.ncl = (int32_t)(lv.ncol / 2);
        o.tpr = (o.ncl + tb - 1) / tb * oz_sweeps(t->np);
        o.tstep = op == OZ_M2M ? 1 : 2;
        o.sstep = op == OZ_L2L ? 1 : 2;
        o.add = op == OZ_L2L;
        o.planes = (int32_t)(op == OZ_L2L ? up.nrow : 2 * lv.nrow);
        o.ncol = op == OZ_M2M ? up.ncol : lv.ncol;
        o.e0 = x.e0;
        o.ents = (const RowEnt *)x.ents;
        o.A = x.A;
        o.ea = x.ea;
        // level i's multipoles and their digits; the parents' local expansions take those of level i + 1
        o.B = op == OZ_L2L ? (i + 1 < nl ? Z.lv[i + 1].B : Z.Btop) : z.B;
        o.mmax = op == OZ_L2L ? Z.bmax : Z.mmax + (size_t)LM_MAXV * i;
        o.omax = op == OZ_M2M && i + 1 < nl ? Z.mmax + (size_t)LM_MAXV * (i + 1) : nullptr;
        o.M = (const float4 *)(op == OZ_L2L ? up.Lc : lv.M);
        o.L = (float4 *)(op == OZ_M2M ? up.M : lv.Lc);
        v.push_back(o);
        tiles += 2 * lv.nrow * o.tpr;
    }
    return v;
}

// split tables [ncls][np][np] of one contraction and its entry lists
static lm_status oz_setup_op(lm_tree_s *t, const zd *tab, size_t ncls, const std::vector<RowEnt> &ents,
                             const std::vector<int32_t> &e0, OzData::Op &x, cudaStream_t st)
{
    const int np = t->np, rows = oz_rows(np) * oz_sweeps(np), KC = oz_chunks(np);
    RowEnt *de;
    TRY_O(lm_dalloc(t, &de, ents.size()));
    x.ents = de;
    TRY_O(lm_dalloc(t, &x.e0, e0.size()));
    TRY_O(lm_dalloc(t, &x.A, ncls * OZ_S * KC * rows * 16));
    TRY_O(lm_dalloc(t, &x.ea, np + 3));
    uint32_t *tmax;
    int32_t *W;
    TRY_O(lm_dalloc(t->tmp, &tmax, 2 * np));
    TRY_O(lm_dalloc(t->tmp, &W, ncls * np));
    LM_CUDA(cudaMemcpyAsync(de, ents.data(), ents.size() * sizeof(RowEnt), cudaMemcpyHostToDevice, st));
    LM_CUDA(cudaMemcpyAsync(x.e0, e0.data(), e0.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    LM_CUDA(cudaMemsetAsync(tmax, 0, 2 * np * sizeof(uint32_t), st));
    LM_CUDA(cudaMemsetAsync(x.ea, 0, (np + 3) * sizeof(int32_t), st));
    k_oz_tmax<<<(unsigned)ncls, 128, 0, st>>>(tab, np, tmax);
    k_oz_texp<<<1, 128, 0, st>>>(tmax, np, x.ea);
    k_oz_tsum<<<(unsigned)ncls, 128, 0, st>>>(tab, np, x.ea, W);
    k_oz_gsum<<<(unsigned)(e0.size() - 1), 128, 0, st>>>(de, x.e0, np, W, x.ea);
    const int64_t nt = (int64_t)ncls * KC * rows;
    k_oz_tsplit<<<(unsigned)((nt + 255) / 256), 256, 0, st>>>(tab, (int64_t)ncls, np, x.ea, x.A);
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}

lm_status lm_setup_oz(lm_tree_s *t, cudaStream_t st)
{
    OzData &Z = t->oz;
    const int KC = oz_chunks(t->np);
    auto buf = [&](int64_t planes, int64_t ncl, unsigned char **B) { // every vector form shares the buffer
        size_t bb = 0;
        for (int s = 1; s <= LM_MAXV; s *= 2)
            bb = std::max(bb, (size_t)(planes * OZ_S * KC) * oz_prow((int)ncl, OZ_N / s, s) * 16);
        return lm_dalloc(t, B, bb);
    };
    for (int l = t->L; l >= 1; --l) { // deepest (most tiles) first
        if (!lm_oz_level(t, l)) continue;
        const Level &lv = t->lev[l], &up = t->lev[l - 1];
        OzData::Lv z{};
        z.l = l;
        std::vector<RowEnt> ents;
        std::vector<int32_t> e0;
        TRY_O(lm_row_entries(lv, ents, e0));
        TRY_O(oz_setup_op(t, lv.tab, std::max<size_t>(1, lv.cls_term.size()), ents, e0, z.op[OZ_M2L], st));
        if (lv.nbox < OZ_MINSHIFT) {
            TRY_O(buf(2 * lv.nrow, lv.ncol / 2, &z.B));
            Z.lv.push_back(z);
            continue;
        }
        // M2M: the children of a parent row, by position; L2L: one parent of a child
        ents.clear();
        e0.assign(1, 0);
        for (int64_t r = 0; r < up.nrow; ++r) {
            for (int pos = 0; pos < 4; ++pos) ents.push_back(RowEnt{pos, 0, (int32_t)(2 * (2 * r + (pos >> 1)) + (pos & 1)), 1});
            e0.push_back((int32_t)ents.size());
        }
        TRY_O(oz_setup_op(t, up.m2m, 4, ents, e0, z.op[OZ_M2M], st));
        ents.clear();
        e0.assign(1, 0);
        for (int64_t c = 0; c < 2 * lv.nrow; ++c) {
            ents.push_back(RowEnt{(int32_t)((c >> 1 & 1) * 2 + (c & 1)), 0, (int32_t)(c >> 2), 1});
            e0.push_back((int32_t)ents.size());
        }
        TRY_O(oz_setup_op(t, lv.l2l, 4, ents, e0, z.op[OZ_L2L], st));
        TRY_O(buf(2 * lv.nrow, lv.ncol / 2, &z.B));
        Z.lv.push_back(z);
        Z.nshift = Z.lv.size();
    }
    if (Z.lv.empty()) return LM_OK;
    const size_t nl = Z.lv.size();
    const Level &top = t->lev[Z.lv.back().l - 1];
    if (Z.nshift == nl) TRY_O(buf(top.nrow, top.ncol, &Z.Btop));
    TRY_O(lm_dalloc(t, &Z.mmax, nl * LM_MAXV)); // multipoles of a level
    if (Z.nshift > 0) TRY_O(lm_dalloc(t, &Z.bmax, (size_t)t->lev[Z.lv[0].l - 1].nbox * LM_MAXV)); // parents of the deepest level
    int f = 0;
    for (int s = 1; s <= 16; s *= 2, ++f) {
        OzLevel *d;
        TRY_O(lm_dalloc(t, &d, 3 * nl));
        Z.desc[f] = d;
        for (int op = 0; op < 3; ++op) {
            const std::vector<OzLevel> lv = oz_levels(t, op, s);
            LM_CUDA(cudaMemcpyAsync(d + op * nl, lv.data(), nl * sizeof(OzLevel), cudaMemcpyHostToDevice, st));
            if (op == OZ_M2L) Z.ntile[f] = lv.back().tile0 + 2 * t->lev[Z.lv.back().l].nrow * lv.back().tpr;
        }
    }
    int dev = 0;
    LM_CUDA(cudaGetDevice(&dev));
    LM_CUDA(cudaDeviceGetAttribute(&Z.nsm, cudaDevAttrMultiProcessorCount, dev));
    LM_CUDA(cudaFuncSetAttribute(k_m2l_oz, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM));
    return LM_OK;
}

static int oz_form(int nv) { return nv <= 1 ? 0 : nv <= 2 ? 1 : nv <= 4 ? 2 : nv <= 8 ? 3 : 4; }
// one contraction of tensor-core level i (M2M, L2L), its sources' digits first
static int oz_step(lm_tree_s *t, int op, size_t i, bool mmax, int nv, cudaStream_t st)
{
    const OzData &Z = t->oz;
    const int f = oz_form(nv), nvs = 1 << f, tb = OZ_N / nvs;
    const OzLevel *d = (const OzLevel *)Z.desc[f] + op * Z.lv.size() + i;
    const Level &lv = t->lev[Z.lv[i].l];
    const int64_t ncl = lv.ncol / 2, planes = op == OZ_L2L ? lv.nrow / 2 : 2 * lv.nrow;
    const int64_t work = planes * oz_prow((int)ncl, tb, nvs) * oz_chunks(t->np);
    if (op == OZ_L2L) k_oz_bmax<<<8 * (unsigned)Z.nsm, 256, 0, st>>>(d, t->np, nv);
    else if (mmax) k_oz_mmax<<<2 * (unsigned)Z.nsm, 256, 0, st>>>(d, t->np, nv);
    k_oz_split<<<(unsigned)std::min<int64_t>(8 * Z.nsm, (work + 255) / 256), 256, 0, st>>>(d, t->np, nv, nvs);
    const int64_t tiles = (op == OZ_M2M ? lv.nrow / 2 : 2 * lv.nrow) * ((ncl + tb - 1) / tb) * oz_sweeps(t->np);
    k_m2l_oz<<<(unsigned)std::min<int64_t>(Z.nsm, tiles), OZ_THREADS, OZ_SMEM, st>>>(d, 1, tiles, t->np, nv, nvs, t->dflag + 1, -1);
    return 2 + (mmax || op == OZ_L2L);
}

// M2M from the levels of at least OZ_MINSHIFT boxes, whose multipoles' digits the M2L takes too; *lmin: the
// level that it has reached
lm_status lm_launch_m2m_oz(lm_tree_s *t, int nv, cudaStream_t st, int *lmin, int *launches)
{
    const OzData &Z = t->oz;
    *launches = 0;
    *lmin = t->L;
    if (Z.lv.empty()) return LM_OK;
    LM_CUDA(cudaMemsetAsync(Z.mmax, 0, Z.lv.size() * LM_MAXV * sizeof(uint32_t), st));
    for (size_t i = 0; i < Z.nshift; ++i) *launches += oz_step(t, OZ_M2M, i, i == 0, nv, st);
    *lmin = t->L - (int)Z.nshift;
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}
bool lm_oz_shift(const lm_tree_s *t, int l) { return t->L - l < (int)t->oz.nshift; }
// L2L to such a level l (adds to its L)
lm_status lm_launch_l2l_oz(lm_tree_s *t, int l, int nv, cudaStream_t st, int *launches)
{
    const size_t i = (size_t)(t->L - l);
    *launches = oz_step(t, OZ_L2L, i, false, nv, st);
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}

// the M2L of the tensor-core levels (sets their L; after their M2M); returns the kernels launched
lm_status lm_launch_m2l_oz(lm_tree_s *t, int nv, cudaStream_t st, int *launches)
{
    const OzData &Z = t->oz;
    *launches = 0;
    if (Z.lv.empty()) return LM_OK;
    const int f = oz_form(nv), nl = (int)Z.lv.size(), n0 = (int)Z.nshift;
    const OzLevel *d = (const OzLevel *)Z.desc[f];
    if (n0 < nl) { // the digits of the levels without M2M here
        k_oz_mmax<<<dim3(2 * (unsigned)Z.nsm, nl - n0), 256, 0, st>>>(d + n0, t->np, nv);
        k_oz_split<<<dim3(8 * (unsigned)Z.nsm, nl - n0), 256, 0, st>>>(d + n0, t->np, nv, 1 << f);
    }
    k_m2l_oz<<<(unsigned)std::min<int64_t>(Z.nsm, Z.ntile[f]), OZ_THREADS, OZ_SMEM, st>>>(
        d, nl, Z.ntile[f], t->np, nv, 1 << f, t->dflag + 1, t->tt_poll_limit);
    t->tt_poll_limit = -1; // a test limit applies to one launch
    *launches = n0 < nl ? 3 : 1;
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}
