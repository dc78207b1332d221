// Density preparation: the input pdfs evaluated on the grid and normalised
// (Algorithm "VUP - Single probability": evaluate the input pdf at the grid
// points and normalise; Sec. 5.3: hard truncation at the domain boundary and
// renormalisation; Eq. gaussh Gaussian measurement uncertainty).
//
// Product densities factor over axes, so W[k, i] = prod_d g_d(k, a_d) / Z_d(k)
// with Z_d = sum_a g_d(k, a).  This kernel writes the per-axis factor tables
// g_d[a][k] (K x sum_d n_d floats -- never the K x N weights) and the FP64
// normalisation statistics.  The contraction and histogram kernels form W on
// the fly as products of these factors.
#include "vup_internal.cuh"

#include <math.h>

#include <algorithm>
#include <vector>

namespace {

struct DensIn {
    const uint8_t *kind;
    const double *mu, *sigma, *lo, *hi;
};

// Neumaier-compensated FP32 accumulator.
struct KSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v) {
        float t = s + v;
        if (fabsf(s) >= fabsf(v)) c += (s - t) + v; else c += (v - t) + s;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// a + b as s + e exactly, for |a| >= |b| (or a + b exact): Dekker's fast two-sum.
__device__ __forceinline__ void fast_two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    e = b - (s - a);
}

// Constants of one (k, d) Gaussian factor in index space, as FP32 pairs.
struct GaussArg {
    double nk;       // integer part of the mean's index coordinate
    float fh, fl;    // fractional part f = fh + fl
    float rh, rl;    // r = h / sigma = rh + rl
    float qh, ql;    // u0^2 = qh + ql (u at the midpoint nearest the mean)
};

// Unnormalised Gaussian factor at index offset A = a - n (an integer held
// exactly in FP32), and u = (A - f) r, the midpoint's distance from the mean
// in units of sigma.  The exponent 0.5 (u^2 - u0^2) is carried as an FP32
// pair (error ~2^-44 relative) and exp is split, exp(-(eh + el)) =
// expf(-eh) (1 - el), so the factor keeps FP32 relative accuracy even far in
// the tails, where the exponent is large and a plain FP32 argument would lose
// ~e * 2^-24.  Dividing by the value at the midpoint nearest the mean (u0) is
// a constant per (k, d) that the normalisation removes; it keeps narrow
// densities from underflowing.
__device__ __forceinline__ float gauss_value(float A, const GaussArg &ga, float &u) {
    // t = A - f exactly as a pair
    float th, tl;
    fast_two_sum(A, -ga.fh, th, tl);  // A is an integer, fh in [0, 1): 0 or larger than fh
    tl -= ga.fl;
    // u = t r
    const float uh = th * ga.rh;
    const float ul = fmaf(th, ga.rh, -uh) + (th * ga.rl + tl * ga.rh);
    u = uh + ul;
    // u^2 - u0^2
    const float sh = uh * uh;
    const float sl = fmaf(uh, uh, -sh) + 2.f * uh * ul;
    // (u0 is the smallest |u|: sh >= qh but where they round to neighbours, whose
    // difference is exact)
    float dh, dl;
    fast_two_sum(sh, -ga.qh, dh, dl);
    dl += sl - ga.ql;
    // e = dh + dl; the halves of e and of its error are exact
    const float e = dh + dl;
    const float l = dl - (e - dh);
    return expf(-0.5f * e) * fmaf(-0.5f, l, 1.f);
}

// Midpoint coordinate of cell a, x_a = lo + (a + 1/2) h, rounded in FP64 in
// this order (the support decisions below compare it with FP64 bounds).
__device__ __forceinline__ double midpoint(double lo, double h, int64_t a) {
    return __dadd_rn(lo, __dmul_rn((double)a + 0.5, h));
}

// First a in [b, e) with pred(a) true, e if none, for a predicate that is
// false then true along a (binary search: a few FP64 evaluations per segment
// instead of one per point).
template <class P>
__device__ __forceinline__ int64_t first_true(int64_t b, int64_t e, P pred) {
    while (b < e) {
        const int64_t m = b + ((e - b) >> 1);
        if (pred(m)) e = m; else b = m + 1;
    }
    return b;
}

// Factor values of one thread's segment [a_begin, a_end) of axis cells,
// written to tab (stride K_pad) and summed (compensated) into S0 = sum g,
// S1 = sum g u, S2 = sum g u^2.  Cells in [in_b, in_e) are inside the
// support (uniform: g = 1 there; truncated normal: the Gaussian there, 0
// outside).  EXACT_F32: every a - n in the segment is below 2^24 in
// magnitude, so A is carried as an FP32 counter; otherwise A is rounded
// from FP64 per cell.
// PLAIN: a warp of Gaussian densities (no supports to look at).
template <bool EXACT_F32, bool STATS, bool PLAIN>
__device__ __forceinline__ void prep_segment(float *__restrict__ tab, int64_t K_pad, int kind, int32_t a_begin,
                                             int32_t a_end, int32_t in_b, int32_t in_e, const GaussArg &ga,
                                             KSum &S0, KSum &S1, KSum &S2) {
    float Af = (float)((double)a_begin - ga.nk);
    tab += a_begin * K_pad;
    for (int32_t a = a_begin; a < a_end; ++a, tab += K_pad) {
        const float A = EXACT_F32 ? Af : (float)((double)a - ga.nk);
        Af += 1.f;
        float u;
        float g = gauss_value(A, ga, u);
        if (!PLAIN) {
            const bool inside = a >= in_b && a < in_e;
            if (kind == VUP_UNIFORM) {
                g = inside ? 1.f : 0.f;
                u = 0.f;
            } else if (kind == VUP_TRUNCNORM && !inside) {
                g = 0.f;
            }
        }
        *tab = g;
        S0.add(g);
        if (STATS) {
            S1.add(g * u);
            S2.add(g * u * u);
        }
    }
}

// Everything one density-prep launch needs for one grid (one instance).
struct DensJob {
    DensIn in;
    int64_t K, K_pad;
    int ndim;
    int64_t n[3];
    double lo[3], h[3];
    int S;  // segments per axis
    DensConst *dconst;
    float *ftab;
    DensStats *dstats;
    int *dstatus;
    // split BF16 A table of the orientation-0 reduction axis (tensor-core path)
    const float *red_tab;
    int64_t nd_red, R_pad;
    __nv_bfloat16 *ahi, *alo;
};

// One CTA: the factors and the normalisation statistics of 32 densities on one
// axis; warp z (threadIdx.y) takes segment z.  Warp 0 first forms the densities'
// constants -- FP64 divisions and, for supports, binary searches -- which every
// segment's thread repeated before (half of the kernel's time, as FP64 issues
// at a 64th of the FP32 rate); the segments' compensated sums are added in order
// (FP64) by the same CTA: Z = sum g, E[u] and E[u^2] under g / Z.  The rest is
// FP32 issue: about 38 instructions per factor.  1024 + 1024 cells x 16384
// densities with the split table, beside a layout build: 165 -> 142 us; 2048 +
// 2048 x 65536 with two split tables: 1133 -> 970.
constexpr int kMaxSeg = 16;
struct DensK {
    GaussArg ga;
    int32_t kind, in_b, in_e;  // cells [in_b, in_e) are inside the support
};
template <bool STATS>
__device__ __forceinline__ void density_prep_body(const DensJob &J, int64_t kb, int d) {
    constexpr int NS = STATS ? 3 : 1;
    __shared__ DensK s_k[32];
    __shared__ float2 s_sum[kMaxSeg][NS][32];
    const int lane = threadIdx.x, z = threadIdx.y;
    const int64_t k = kb * 32 + lane;  // K_pad is a multiple of 128: k < K_pad
    const int64_t K_pad = J.K_pad, p = k * J.ndim + d;
    const DensIn &in = J.in;
    const int32_t nd = (int32_t)J.n[d];
    const bool live = k < J.K;
    int64_t off = 0;
    for (int q = 0; q < d; ++q) off += J.n[q] * K_pad;
    float *tab = J.ftab + off + k;
    if (z == 0 && live) {
        const double lo = J.lo[d], h = J.h[d];
        DensK D;
        D.kind = in.kind[p];
        const double mu = in.mu[p], sigma = in.sigma[p];
        // index coordinate of the mean: (mu - lo) / h - 1/2 = nk + f
        const double c = (mu - lo) / h - 0.5;
        const double nk = floor(c);
        const double fd = c - nk;
        const double rd = h / sigma;
        GaussArg &ga = D.ga;
        ga.nk = nk;
        ga.fh = (float)fd;
        ga.fl = (float)(fd - (double)ga.fh);
        ga.rh = (float)rd;
        ga.rl = (float)(rd - (double)ga.rh);
        // squared index-space distance from the mean to its nearest midpoint
        double anear = floor(c + 0.5);
        anear = fmin(fmax(anear, 0.0), (double)(nd - 1));
        const double u0 = ((anear - nk) - fd) * rd;
        double u0sq = D.kind == VUP_UNIFORM ? 0.0 : u0 * u0;
        if (!(u0sq < 1e30)) u0sq = 0.0;
        ga.qh = (float)u0sq;
        ga.ql = (float)(u0sq - (double)ga.qh);
        // support of a uniform or truncated density: an interval of cells, since
        // x_a is non-decreasing in a
        D.in_b = 0;
        D.in_e = nd;
        if (D.kind == VUP_UNIFORM) {
            const double half = __dmul_rn(0.5, sigma);
            D.in_b = first_true(0, nd, [&](int64_t a) { return __dsub_rn(midpoint(lo, h, a), mu) >= -half; });
            D.in_e = first_true(D.in_b, nd, [&](int64_t a) { return !(__dsub_rn(midpoint(lo, h, a), mu) <= half); });
        } else if (D.kind == VUP_TRUNCNORM) {
            const double tlo = in.lo ? in.lo[p] : 0.0, thi = in.hi ? in.hi[p] : 0.0;
            D.in_b = first_true(0, nd, [&](int64_t a) { return midpoint(lo, h, a) >= tlo; });
            D.in_e = first_true(D.in_b, nd, [&](int64_t a) { return !(midpoint(lo, h, a) <= thi); });
        }
        s_k[lane] = D;
        DensConst dc;
        dc.n = (int32_t)fmax(fmin(nk, 2147483647.0), -2147483647.0);
        dc.f = ga.fh;
        dc.r = ga.rh;
        dc.kind = D.kind;
        J.dconst[p] = dc;
    }
    __syncthreads();
    const int32_t seg = (nd + J.S - 1) / J.S;
    const int32_t a_begin = min(nd, z * seg), a_end = min(nd, a_begin + seg);
    KSum S0, S1, S2;
    if (live) {
        const DensK D = s_k[lane];
        const GaussArg &ga = D.ga;
        const double A0 = (double)a_begin - ga.nk;
        const bool exact = fabs(A0) + (double)(a_end - a_begin) < 16777216.0;
        if (__all_sync(__activemask(), exact && D.kind == VUP_GAUSS))
            prep_segment<true, STATS, true>(tab, K_pad, D.kind, a_begin, a_end, D.in_b, D.in_e, ga, S0, S1, S2);
        else if (exact)
            prep_segment<true, STATS, false>(tab, K_pad, D.kind, a_begin, a_end, D.in_b, D.in_e, ga, S0, S1, S2);
        else
            prep_segment<false, STATS, false>(tab, K_pad, D.kind, a_begin, a_end, D.in_b, D.in_e, ga, S0, S1, S2);
    } else {
        for (int32_t a = a_begin; a < a_end; ++a) tab[a * K_pad] = 0.f;
    }
    s_sum[z][0][lane] = make_float2(S0.s, S0.c);
    if constexpr (STATS) {
        s_sum[z][1][lane] = make_float2(S1.s, S1.c);
        s_sum[z][2][lane] = make_float2(S2.s, S2.c);
    }
    __syncthreads();
    if (z != 0 || !live) return;
    double s[3] = {0.0, 0.0, 0.0};
    for (int q = 0; q < J.S; ++q)
#pragma unroll
        for (int i = 0; i < NS; ++i) s[i] += (double)s_sum[q][i][lane].x + (double)s_sum[q][i][lane].y;
    DensStats ds;
    ds.invZ = s[0] > 0.0 ? 1.0 / s[0] : 0.0;
    ds.Eu = STATS && s[0] > 0.0 ? s[1] / s[0] : 0.0;
    ds.Eu2 = STATS && s[0] > 0.0 ? s[2] / s[0] : 0.0;
    ds.inv_sigma = 1.0 / in.sigma[p];
    J.dstats[p] = ds;
    if (!(s[0] > 0.0)) atomicCAS(J.dstatus, 0, VUP_DSTAT_EMPTY);
}

// A-operand table of the tensor-core contraction: rows k, reduction index a
// contiguous (K-major), each FP32 factor split into BF16 hi + lo (see
// split_transpose_body for the tiling).
// Split of one FP32 value into hi + lo: BF16 pair (tensor kind::f16) or
// TF32 pair stored in floats (kind::tf32).
__device__ __forceinline__ float to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

// Two consecutive reduction indices of one density row split together (one
// 4-byte BF16 pair or 8-byte TF32 pair store per array).
__device__ __forceinline__ void split_store2(__nv_bfloat16 *hi, __nv_bfloat16 *lo, int64_t i, float v0, float v1) {
    const __nv_bfloat16 h0 = __float2bfloat16_rn(v0), h1 = __float2bfloat16_rn(v1);
    *reinterpret_cast<__nv_bfloat162 *>(hi + i) = __halves2bfloat162(h0, h1);
    *reinterpret_cast<__nv_bfloat162 *>(lo + i) = __halves2bfloat162(__float2bfloat16_rn(v0 - __bfloat162float(h0)),
                                                                     __float2bfloat16_rn(v1 - __bfloat162float(h1)));
}
__device__ __forceinline__ void split_store2(float *hi, float *lo, int64_t i, float v0, float v1) {
    const float h0 = to_tf32(v0), h1 = to_tf32(v1);
    *reinterpret_cast<float2 *>(hi + i) = make_float2(h0, h1);
    *reinterpret_cast<float2 *>(lo + i) = make_float2(to_tf32(v0 - h0), to_tf32(v1 - h1));
}

// Block (bx, by) transposes the 64 (a) x 128 (k) tile at a = 64 bx,
// k = 128 by: the 64 rows are read with 16-byte loads (eight per thread, in
// flight together), then each lane writes two consecutive a of one density
// row.  R_pad is a multiple of 64, K_pad of 128.
constexpr int kSplitK = 128;
template <typename T>
__device__ __forceinline__ void split_transpose_body(const float *__restrict__ tab, int64_t nd, int64_t K_pad,
                                                     int64_t R_pad, T *__restrict__ hi, T *__restrict__ lo,
                                                     int64_t bx, int64_t by) {
    __shared__ float t[64][kSplitK + 1];
    const int64_t a0 = bx * 64, k0 = by * kSplitK;
    float4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int64_t a = a0 + threadIdx.y + 8 * i;
        v[i] = a < nd ? *reinterpret_cast<const float4 *>(tab + a * K_pad + k0 + 4 * threadIdx.x)
                      : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float *r = &t[threadIdx.y + 8 * i][4 * threadIdx.x];
        r[0] = v[i].x;
        r[1] = v[i].y;
        r[2] = v[i].z;
        r[3] = v[i].w;
    }
    __syncthreads();
    for (int y = threadIdx.y; y < kSplitK; y += blockDim.y) {
        const int64_t k = k0 + y, a = a0 + 2 * threadIdx.x;
        split_store2(hi, lo, k * R_pad + a, t[2 * threadIdx.x][y], t[2 * threadIdx.x + 1][y]);
    }
    __syncthreads();
}

// STATS: also the sums of g u and g u^2 (E[u], E[u^2] of the IPSA derivatives)
template <bool STATS>
__global__ void __launch_bounds__(32 * kMaxSeg) k_density_prep(DensJob J) {
    pdl_trigger();
    pdl_wait();
    density_prep_body<STATS>(J, blockIdx.x, blockIdx.y);
}
// grid: x = density tiles of 128 (more than the 65535 limit of y for large K), y = axis tiles
template <typename T>
__global__ void k_split_transpose(const float *__restrict__ tab, int64_t nd, int64_t K_pad, int64_t R_pad,
                                  T *__restrict__ hi, T *__restrict__ lo) {
    pdl_trigger();
    pdl_wait();
    split_transpose_body<T>(tab, nd, K_pad, R_pad, hi, lo, blockIdx.y, blockIdx.x);
}

// Batched forms: one launch for the blocks of every instance; items[b] =
// (instance, block coordinates) of block b.
// (blocks of as many warps as the batch's longest axis has segments; the others'
// spare warps have empty segments)
__global__ void __launch_bounds__(32 * kMaxSeg) k_density_prep_batched(const DensJob *__restrict__ jobs,
                                                                       const int4 *__restrict__ items) {
    const int4 it = items[blockIdx.x];
    density_prep_body<false>(jobs[it.x], it.y, it.z);
}
__global__ void k_split_transpose_batched(const DensJob *__restrict__ jobs, const int4 *__restrict__ items) {
    const int4 it = items[blockIdx.x];
    const DensJob &J = jobs[it.x];
    split_transpose_body<__nv_bfloat16>(J.red_tab, J.nd_red, J.K_pad, J.R_pad, J.ahi, J.alo, it.y, it.z);
}

int density_segments(vup_grid g) {
    int64_t nmax = 1;
    for (int q = 0; q < g->ndim; ++q) nmax = std::max(nmax, g->n[q]);
    return (int)std::max<int64_t>(1, std::min<int64_t>(kMaxSeg, nmax / 128));
}

DensJob make_job(vup_grid g, const vup_densities *d) {
    DensJob J{};
    J.in = DensIn{d->kind, d->mu, d->sigma, d->lo, d->hi};
    J.K = d->K;
    J.K_pad = ceil_div64(d->K, 128) * 128;
    J.ndim = g->ndim;
    for (int q = 0; q < 3; ++q) {
        J.n[q] = g->n[q];
        J.lo[q] = g->lo[q];
        J.h[q] = (g->hi[q] - g->lo[q]) / (double)g->n[q];
    }
    J.S = density_segments(g);
    J.dconst = (DensConst *)g->dconst.p;
    J.ftab = (float *)g->ftab.p;
    J.dstats = (DensStats *)g->dstats.p;
    J.dstatus = g->dstatus;
    const Orient &o = g->orient[0];
    int64_t off = 0;
    for (int q = 0; q < o.red_axis0; ++q) off += g->n[q] * J.K_pad;
    J.red_tab = (const float *)g->ftab.p + off;
    J.nd_red = g->n[o.red_axis0];
    J.R_pad = o.R_pad;
    J.ahi = (__nv_bfloat16 *)g->atab_hi.p;
    J.alo = (__nv_bfloat16 *)g->atab_lo.p;
    return J;
}

}  // namespace

size_t vup_ftab_floats(const vup_grid g) {
    size_t s = 0;
    for (int d = 0; d < g->ndim; ++d) s += (size_t)g->n[d];
    return s;
}

// need_bf16_orient_mask: bit o set -> build the split BF16 A table for the
// reduction axis of orientation o.
template <typename T>
static vup_status split_tables(vup_grid g, int mask, int64_t K_pad, T *hi0, T *lo0, cudaStream_t s);

vup_status vup_density_prep(vup_grid g, const vup_densities *d, int need_bf16_orient_mask, cudaStream_t s,
                            bool tf32, bool stats) {
    const DensJob J = make_job(g, d);
    const int64_t K_pad = J.K_pad;
    dim3 grd((unsigned)(K_pad / 32), (unsigned)g->ndim), blk(32, (unsigned)J.S);
    VUP_PROF("density_prep", s, 1 + __builtin_popcount(need_bf16_orient_mask));
    VUP_CHECK_CUDA(stats ? launch_pdl(k_density_prep<true>, grd, blk, 0, s, J)
                         : launch_pdl(k_density_prep<false>, grd, blk, 0, s, J));
    if (tf32) return split_tables<float>(g, need_bf16_orient_mask, K_pad, (float *)g->atf_hi.p,
                                         (float *)g->atf_lo.p, s);
    return split_tables<__nv_bfloat16>(g, need_bf16_orient_mask, K_pad, (__nv_bfloat16 *)g->atab_hi.p,
                                       (__nv_bfloat16 *)g->atab_lo.p, s);
}

// Split tables of the A operand for the orientations in `mask` (T: BF16 or
// TF32-in-float), written to hi / lo.
template <typename T>
static vup_status split_tables(vup_grid g, int mask, int64_t K_pad, T *hi0, T *lo0, cudaStream_t s) {
    for (int o = 0; o < 2; ++o) {
        if (!(mask & (1 << o))) continue;
        const Orient &ori = g->orient[o];
        const int dred = ori.red_axis0;
        int64_t off = 0;
        for (int q = 0; q < dred; ++q) off += g->n[q] * K_pad;
        T *hi = hi0, *lo = lo0;
        if (o == 1) {
            // orientation-1 tables live after the orientation-0 tables
            const size_t o0 = (size_t)K_pad * g->orient[0].R_pad;
            hi += o0;
            lo += o0;
        }
        dim3 tg((unsigned)ceil_div64(K_pad, kSplitK), (unsigned)ceil_div64(ori.R_pad, 64));
        VUP_CHECK_CUDA(launch_pdl(k_split_transpose<T>, tg, dim3(32, 8), 0, s, (const float *)g->ftab.p + off,
                                  (int64_t)g->n[dred], K_pad, ori.R_pad, hi, lo));
    }
    return VUP_OK;
}

// Batched density preparation for n instances (one launch per stage).  The
// job and item tables are built on the host and uploaded into `plan`
// (device memory owned by the caller); returns the device pointers' layout
// via the launch.  Scratch of every grid must already be reserved for its K.
struct DensPlan {
    DevBuf jobs, items;
    int n_prep = 0, n_split = 0, segs = 1;
};

vup_status vup_density_plan(int n, const vup_grid *gs, const vup_densities *ds, bool bf16, void **plan_out) {
    DensPlan *P = new DensPlan();
    std::vector<DensJob> jobs(n);
    std::vector<int4> prep, split;
    for (int i = 0; i < n; ++i) {
        jobs[i] = make_job(gs[i], &ds[i]);
        const DensJob &J = jobs[i];
        P->segs = std::max(P->segs, J.S);
        for (int d = 0; d < J.ndim; ++d)
            for (int64_t kb = 0; kb < J.K_pad / 32; ++kb) prep.push_back(make_int4(i, (int)kb, d, 0));
        if (bf16)
            for (int64_t by = 0; by < ceil_div64(J.K_pad, kSplitK); ++by)
                for (int64_t bx = 0; bx < ceil_div64(J.R_pad, 64); ++bx)
                    split.push_back(make_int4(i, (int)bx, (int)by, 0));
    }
    P->n_prep = (int)prep.size();
    P->n_split = (int)split.size();
    std::vector<int4> all;
    all.insert(all.end(), prep.begin(), prep.end());
    all.insert(all.end(), split.begin(), split.end());
    vup_status st;
    if ((st = devbuf_reserve(P->jobs, sizeof(DensJob) * n)) != VUP_OK ||
        (st = devbuf_reserve(P->items, sizeof(int4) * all.size())) != VUP_OK) {
        devbuf_free(P->jobs);
        devbuf_free(P->items);
        delete P;
        return st;
    }
    VUP_CHECK_CUDA(cudaMemcpy(P->jobs.p, jobs.data(), sizeof(DensJob) * n, cudaMemcpyHostToDevice));
    VUP_CHECK_CUDA(cudaMemcpy(P->items.p, all.data(), sizeof(int4) * all.size(), cudaMemcpyHostToDevice));
    *plan_out = P;
    return VUP_OK;
}

void vup_density_plan_free(void *plan) {
    DensPlan *P = (DensPlan *)plan;
    if (!P) return;
    devbuf_free(P->jobs);
    devbuf_free(P->items);
    delete P;
}

vup_status vup_density_batched(void *plan, cudaStream_t s) {
    const DensPlan *P = (const DensPlan *)plan;
    const DensJob *jobs = (const DensJob *)P->jobs.p;
    const int4 *items = (const int4 *)P->items.p;
    VUP_PROF("density_prep_batched", s, P->n_split ? 2 : 1);
    if (P->n_prep) k_density_prep_batched<<<P->n_prep, dim3(32, P->segs), 0, s>>>(jobs, items);
    VUP_CHECK_LAUNCH();
    if (P->n_split) k_split_transpose_batched<<<P->n_split, dim3(32, 8), 0, s>>>(jobs, items + P->n_prep);
    VUP_CHECK_LAUNCH();
    return VUP_OK;
}
