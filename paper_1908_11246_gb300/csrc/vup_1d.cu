// One-dimensional grids in FP64 (Algorithm "VUP - Single probability" with
// the densities of Eq. VUP, every step in double precision).  One thread-block
// cluster per density: its CTAs share the points, keep every point's density in
// shared memory, and reduce the sums over the cluster; raw moments, central
// moments (second pass about the mean) and the histogram over the bin-sorted
// points (the CSR form of the one-hot model matrix, Eq. MUP) all read the kept
// values.
//
// FP64 arithmetic bounds this path: the GPU issues about two FP64 operations
// per clock and SM, so its time is the number of them.  The density is evaluated once per
// point (it was evaluated for each of the three sums: 338 us for 256 densities
// on 4096 points, now 88), in 4 operations up to the exponent and 12 for a
// table-driven exponential; points whose Gaussian is 0 in FP64, beyond 38.6
// sigma, are skipped (three of five points at sigma = 1/200 of the domain, none
// at 1/40); and sums add across warps and few lanes, as
// a step of a shuffle tree costs an FP64 operation on all 32 lanes (full-warp
// trees, with every warp forming the density's constants, took 116 us).
#include "vup_internal.cuh"

#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

namespace cg = cooperative_groups;

namespace {

constexpr int kThreads = 128, kWarps = kThreads / 32;
constexpr int kMaxCluster = 8;

struct P1 {
    const uint8_t *kind;
    const double *mu, *sigma, *lo, *hi;
};

struct Geo1 {
    int64_t n;
    double lo, h;
};

// 2^(j / 64), j = 0 .. 63, each rounded to FP64
__constant__ double kExpTab[64] = {
    0x1.0000000000000p+0, 0x1.02c9a3e778061p+0, 0x1.059b0d3158574p+0, 0x1.0874518759bc8p+0,
    0x1.0b5586cf9890fp+0, 0x1.0e3ec32d3d1a2p+0, 0x1.11301d0125b51p+0, 0x1.1429aaea92de0p+0,
    0x1.172b83c7d517bp+0, 0x1.1a35beb6fcb75p+0, 0x1.1d4873168b9aap+0, 0x1.2063b88628cd6p+0,
    0x1.2387a6e756238p+0, 0x1.26b4565e27cddp+0, 0x1.29e9df51fdee1p+0, 0x1.2d285a6e4030bp+0,
    0x1.306fe0a31b715p+0, 0x1.33c08b26416ffp+0, 0x1.371a7373aa9cbp+0, 0x1.3a7db34e59ff7p+0,
    0x1.3dea64c123422p+0, 0x1.4160a21f72e2ap+0, 0x1.44e086061892dp+0, 0x1.486a2b5c13cd0p+0,
    0x1.4bfdad5362a27p+0, 0x1.4f9b2769d2ca7p+0, 0x1.5342b569d4f82p+0, 0x1.56f4736b527dap+0,
    0x1.5ab07dd485429p+0, 0x1.5e76f15ad2148p+0, 0x1.6247eb03a5585p+0, 0x1.6623882552225p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6dfb23c651a2fp+0, 0x1.71f75e8ec5f74p+0, 0x1.75feb564267c9p+0,
    0x1.7a11473eb0187p+0, 0x1.7e2f336cf4e62p+0, 0x1.82589994cce13p+0, 0x1.868d99b4492edp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8f1ae99157736p+0, 0x1.93737b0cdc5e5p+0, 0x1.97d829fde4e50p+0,
    0x1.9c49182a3f090p+0, 0x1.a0c667b5de565p+0, 0x1.a5503b23e255dp+0, 0x1.a9e6b5579fdbfp+0,
    0x1.ae89f995ad3adp+0, 0x1.b33a2b84f15fbp+0, 0x1.b7f76f2fb5e47p+0, 0x1.bcc1e904bc1d2p+0,
    0x1.c199bdd85529cp+0, 0x1.c67f12e57d14bp+0, 0x1.cb720dcef9069p+0, 0x1.d072d4a07897cp+0,
    0x1.d5818dcfba487p+0, 0x1.da9e603db3285p+0, 0x1.dfc97337b9b5fp+0, 0x1.e502ee78b3ff6p+0,
    0x1.ea4afa2a490dap+0, 0x1.efa1bee615a27p+0, 0x1.f50765b6e4540p+0, 0x1.fa7c1819e90d8p+0,
};

// exp(x) for x <= 0, table-driven (P. T. P. Tang, "Table-driven implementation
// of the exponential function in IEEE floating-point arithmetic", ACM TOMS 15,
// 1989): x = (64 m + j) ln2 / 64 + r, |r| <= ln2 / 128, exp(x) = 2^m 2^(j/64)
// (1 + r + r^2/2 + .. + r^6/720).  Within 1.02 ulp: half an ulp each of the table
// and of the last rounding, 0.01 of r and of the polynomial, 1e-4 of its truncation
// (without r^6/720 the truncation is 0.3 ulp and results were up to 1.27 ulp off;
// tests/test_fp64_forms.py compares with 40 digits).  tab: the table in shared
// memory.  Results below the normal range take the library function.
__device__ __forceinline__ double exp_neg(double x, const double *tab) {
    if (!(x > -700.0)) return exp(x);
    constexpr double kMagic = 6755399441055744.0;  // 1.5 2^52: the sum's low bits are round(x 64 / ln2)
    const double t = fma(x, 0x1.71547652b82fep+6, kMagic);
    const int k = __double2loint(t);
    const double kd = t - kMagic;
    double r = fma(kd, -0x1.62e42fee00000p-7, x);
    r = fma(kd, -0x1.a39ef35793c76p-39, r);
    double q = fma(r, 1.0 / 720.0, 1.0 / 120.0);
    q = fma(q, r, 1.0 / 24.0);
    q = fma(q, r, 1.0 / 6.0);
    q = fma(q, r, 0.5);
    q = fma(q, r * r, r);
    const double s = tab[k & 63];
    const double v = fma(s, q, s);
    return __hiloint2double(__double2hiint(v) + ((k >> 6) << 20), __double2loint(v));
}

// One density on the axis.  Gaussian kinds: v = ((a - n) - f) r with the mean
// at index coordinate n + f and r = h / (sigma sqrt 2), so the unnormalised
// density is exp(q - v^2), q = v^2 at the midpoint nearest the mean (a constant
// the normalisation removes, which keeps narrow densities from underflowing).
// Supports (uniform, truncated) are decided on the rounded midpoints.
struct Dens1 {
    int kind;
    double mu, sg, tlo, thi;
    double nk, f, r, q;
    int32_t b, e;  // the points evaluated; the others' density is 0
};

__device__ __forceinline__ bool finite_key(unsigned long long k) {  // an end of the outputs' range (ordered key)
    const unsigned long long u = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return isfinite(__longlong_as_double((long long)u));
}

__device__ __forceinline__ Dens1 dens_of(const P1 &p, const Geo1 &G, const unsigned long long *__restrict__ ext,
                                         int64_t k) {
    Dens1 D;
    D.kind = p.kind[k];
    D.mu = p.mu[k];
    D.sg = p.sigma[k];
    D.tlo = p.lo ? p.lo[k] : 0.0;
    D.thi = p.hi ? p.hi[k] : 0.0;
    const double c = (D.mu - G.lo) / G.h - 0.5;
    D.nk = floor(c);
    D.f = c - D.nk;
    D.r = (G.h / D.sg) * 0.70710678118654752440;
    const double an = fmin(fmax(floor(c + 0.5), 0.0), (double)(G.n - 1));
    const double v0 = ((an - D.nk) - D.f) * D.r;
    D.q = v0 * v0;
    D.b = 0;
    D.e = (int32_t)G.n;
    if (D.kind == VUP_GAUSS && finite_key(ext[0]) && finite_key(ext[1])) {
        // exp(q - v^2) is 0 in FP64 below q - v^2 = -745.2: such points add nothing to
        // any sum, however large their output (a bound of FP32's range, right for the
        // histogram, lost 84 % of E[y^4] of y = exp(80 x) at sigma = 0.05).  0.8 and
        // 2^-46 q allow for the rounding of q - v^2, a cell and 2^-50 for that of the
        // window.  (With an output that is not finite every point is evaluated: 0 times
        // it is not a number.)
        const double h0 = sqrt(D.q + (746.0 + 0x1p-46 * D.q)) / D.r;
        const double hw = h0 + 1.0 + 0x1p-50 * (h0 + fabs(c));
        const double b = floor(c - hw), e = ceil(c + hw) + 1.0;
        if (b > 0.0) D.b = (int32_t)fmin(b, (double)G.n);
        if (e < (double)G.n) D.e = (int32_t)fmax(e, 0.0);
        if (D.b >= D.e || !(hw > 0.0)) {  // (not a number: evaluate everything)
            D.b = 0;
            D.e = (int32_t)G.n;
        }
    }
    return D;
}

// Density at point a and v there (0 for the uniform kind).
__device__ __forceinline__ double dens_at(const Dens1 &D, const Geo1 &G, int32_t a, const double *tab, double &v) {
    v = 0.0;
    if (D.kind != VUP_GAUSS) {
        const double x = __dadd_rn(G.lo, __dmul_rn((double)a + 0.5, G.h));
        if (D.kind == VUP_UNIFORM) return fabs(__dsub_rn(x, D.mu)) <= __dmul_rn(0.5, D.sg) ? 1.0 : 0.0;
        if (!(D.tlo <= x && x <= D.thi)) {
            return 0.0;
        }
    }
    v = (((double)a - D.nk) - D.f) * D.r;
    return exp_neg(fma(-v, v, D.q), tab);
}

// The NS sums of every thread over the block and the cluster, in a fixed
// order, to all threads of all CTAs (out[0..NS) in shared memory).  Warp w adds
// the sums w, w + kWarps, ..: across the warps' lanes first, then a shuffle
// tree; a lane per sum then adds the CTAs'.
template <int NS>
__device__ __forceinline__ void cluster_sums(cg::cluster_group &cl, const double (&v)[NS], double *s_all, double *s_blk,
                                             double *out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NS; ++i) s_all[i * kThreads + threadIdx.x] = v[i];
    __syncthreads();
    for (int i = warp; i < NS; i += kWarps) {
        double t = s_all[i * kThreads + lane];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) t += s_all[i * kThreads + 32 * w + lane];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) s_blk[i] = t;
    }
    cl.sync();
    if (threadIdx.x < NS) {
        double t = 0.0;
        for (int b = 0; b < (int)cl.num_blocks(); ++b) t += cl.map_shared_rank(s_blk, b)[threadIdx.x];
        out[threadIdx.x] = t;
    }
    __syncthreads();
}

template <bool kIpsa>
__global__ void __launch_bounds__(kThreads) k_1d(P1 p, Geo1 G, const unsigned long long *__restrict__ ext,
                                                 const double *__restrict__ y,
                                                 const int32_t *__restrict__ perm,
                                                 const int32_t *__restrict__ offsets, int B, int J,
                                                 double *__restrict__ raw, double *__restrict__ central,
                                                 float *__restrict__ hist, const double *__restrict__ grad,
                                                 float *__restrict__ dmu, float *__restrict__ dsg,
                                                 int *__restrict__ dstatus) {
    constexpr int kSums = kIpsa ? 15 : 5;
    extern __shared__ double s_g[];  // this CTA's points' densities
    __shared__ double s_all[kSums * kThreads], s_blk[kSums], s_blk2[3], s_tab[64], S[kSums], C[3], s_inv[2];
    __shared__ Dens1 s_dens;
    cg::cluster_group cl = cg::this_cluster();
    const int n_cta = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int64_t k = blockIdx.x / n_cta;
    if (threadIdx.x < 64) s_tab[threadIdx.x] = kExpTab[threadIdx.x];
    if (threadIdx.x == 64) s_dens = dens_of(p, G, ext, k);  // one warp's FP64 work, not every warp's
    __syncthreads();
    const Dens1 D = s_dens;
    const int32_t len = D.e - D.b, per = (len + n_cta - 1) / n_cta;
    const int32_t a0 = D.b + min(len, rank * per), a1 = D.b + min(len, (rank + 1) * per);
    double s[kSums];
#pragma unroll
    for (int i = 0; i < kSums; ++i) s[i] = 0.0;
    for (int32_t a = a0 + threadIdx.x; a < a1; a += kThreads) {
        double v;
        const double g = dens_at(D, G, a, s_tab, v);
        if (!kIpsa) s_g[a - a0] = g;
        const double yv = y[a], y2 = yv * yv, g2 = g * y2;
        s[0] += g;
        s[1] = fma(g, yv, s[1]);
        s[2] += g2;
        s[3] = fma(g2, yv, s[3]);
        s[4] = fma(g2, y2, s[4]);
        if constexpr (kIpsa) {
            const double gv = g * v, gw = gv * v, gv2 = gv * y2, gw2 = gw * y2;
            s[5] += gv;
            s[6] += gw;
            s[7] = fma(gv, yv, s[7]);
            s[8] += gv2;
            s[9] = fma(gv2, yv, s[9]);
            s[10] = fma(gv2, y2, s[10]);
            s[11] = fma(gw, yv, s[11]);
            s[12] += gw2;
            s[13] = fma(gw2, yv, s[13]);
            s[14] = fma(gw2, y2, s[14]);
        }
    }
    cluster_sums<kSums>(cl, s, s_all, s_blk, S);
    const double Z = S[0];
    const bool empty = !(Z > 0.0);  // the same in every CTA of the cluster
    const bool lead = rank == 0 && threadIdx.x == 0;
    if (empty && lead) atomicCAS(dstatus, 0, VUP_DSTAT_EMPTY);
    if constexpr (kIpsa) {
        if (!empty && lead) {
            // u = v sqrt 2
            const double Eu = S[5] / Z * 1.41421356237309504880, Eu2 = S[6] / Z * 2.0;
            const bool diff = D.kind != VUP_UNIFORM;
            double gm = 0.0, gs = 0.0;
            for (int j = 0; j < J; ++j) {
                const double M = S[1 + j] / Z;
                const double S1 = S[7 + j] / Z * 1.41421356237309504880, S2 = S[11 + j] / Z * 2.0;
                const double dm = diff ? (S1 - Eu * M) / D.sg : 0.0;
                const double ds = diff ? (S2 - Eu2 * M) / D.sg : 0.0;
                if (grad) {
                    gm += grad[k * J + j] * dm;
                    gs += grad[k * J + j] * ds;
                } else {
                    dmu[k * J + j] = (float)dm;
                    dsg[k * J + j] = (float)ds;
                }
            }
            if (grad) {
                dmu[k] = (float)gm;
                dsg[k] = (float)gs;
            }
        }
    } else {
        if (!empty && raw && rank == 0 && threadIdx.x < J) raw[k * J + threadIdx.x] = S[1 + threadIdx.x] / Z;
        if (threadIdx.x >= 32 && threadIdx.x < 34) s_inv[threadIdx.x - 32] = (threadIdx.x == 32 ? 1.0 : S[1]) / Z;
        __syncthreads();
        const double invZ = s_inv[0], mean = s_inv[1];
        if (central) {  // (every CTA takes part in the cluster's sums)
            double c[3] = {0.0, 0.0, 0.0};
            for (int32_t a = a0 + threadIdx.x; a < a1; a += kThreads) {
                const double d = y[a] - mean, d2 = d * d, q = s_g[a - a0] * d2;
                c[0] += q;
                c[1] = fma(q, d, c[1]);
                c[2] = fma(q, d2, c[2]);
            }
            cluster_sums<3>(cl, c, s_all, s_blk2, C);
            if (!empty && rank == 0 && threadIdx.x < J)
                central[k * J + threadIdx.x] = threadIdx.x == 0 ? mean : C[threadIdx.x - 1] / Z;
        }
        if (hist && !empty) {
            // eight lanes per bin (a sum of q points costs q / 8 + 3 FP64 operations
            // for four bins at once), the bins dealt to the cluster's lanes; a point's
            // density comes from the CTA that holds it
            const int sub = threadIdx.x & 7, slot = threadIdx.x >> 3;
            const float inv_per = 1.0f / (float)max(per, 1);
            for (int b0 = rank * (kThreads / 8); b0 < B; b0 += n_cta * (kThreads / 8)) {
                const int b = b0 + slot;
                const int32_t t1 = b < B ? offsets[b + 1] : 0;
                double t = 0.0;
#pragma unroll 4
                for (int32_t q = (b < B ? offsets[b] : 0) + sub; q < t1; q += 8) {
                    const int32_t i = perm[q] - D.b;
                    if (i >= 0 && i < len) {
                        int o = min((int)((float)i * inv_per), n_cta - 1);  // owner i / per, one off at most
                        o += i >= (o + 1) * per ? 1 : (i < o * per ? -1 : 0);
                        t += *cl.map_shared_rank(s_g + (i - o * per), o);
                    }
                }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (sub == 0 && b < B) hist[k * B + b] = (float)(t * invZ);
            }
        }
    }
    cl.sync();  // no CTA leaves while another reads its shared memory
}

// CTAs per density: enough that the densities' CTAs fill the SMs four times
// over (their work differs with sigma) and that four CTAs' points fit one SM's
// shared memory; not more, as a CTA's block sums cost about 10 points' FP64 work
// per thread.
int cluster_for(int64_t K, int64_t n) {
    const int64_t want = ceil_div64(4 * (int64_t)vup_num_sms(), K);
    int c = 1;
    while (c < kMaxCluster && c < want && n / (2 * c) >= kThreads) c *= 2;
    while (c < kMaxCluster && ceil_div64(n, c) > 6144) c *= 2;
    return c;
}

template <bool kIpsa, typename... Args>
vup_status launch_1d(vup_grid g, int64_t K, cudaStream_t s, Args... args) {
    const int c = cluster_for(K, g->n[0]);
    const size_t smem = kIpsa ? 0 : sizeof(double) * (size_t)ceil_div64(g->n[0], c);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(K * c));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)c;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (smem > 40 * 1024)
        VUP_CHECK_CUDA(smem_allow(k_1d<kIpsa>));
    VUP_CHECK_CUDA(cudaLaunchKernelEx(&cfg, k_1d<kIpsa>, args...));
    return VUP_OK;
}

}  // namespace

vup_status vup_propagate_1d(vup_grid g, const vup_densities *d, double *raw, double *central, float *hist,
                            cudaStream_t s) {
    const P1 p{d->kind, d->mu, d->sigma, d->lo, d->hi};
    const Geo1 G{g->n[0], g->lo[0], (g->hi[0] - g->lo[0]) / (double)g->n[0]};
    VUP_PROF("vup_1d_fp64", s, 1);
    return launch_1d<false>(g, d->K, s, p, G, (const unsigned long long *)g->ext, (const double *)g->y, (const int32_t *)g->perm,
                            (const int32_t *)g->offsets, g->B, g->J, raw, central, hist, (const double *)nullptr,
                            (float *)nullptr, (float *)nullptr, g->dstatus);
}

vup_status vup_ipsa_1d(vup_grid g, const vup_densities *d, const double *grad, float *dmu, float *dsg,
                       cudaStream_t s) {
    const P1 p{d->kind, d->mu, d->sigma, d->lo, d->hi};
    const Geo1 G{g->n[0], g->lo[0], (g->hi[0] - g->lo[0]) / (double)g->n[0]};
    VUP_PROF("ipsa_1d_fp64", s, 1);
    return launch_1d<true>(g, d->K, s, p, G, (const unsigned long long *)g->ext, (const double *)g->y, (const int32_t *)g->perm,
                           (const int32_t *)g->offsets, g->B, g->J, (double *)nullptr, (double *)nullptr,
                           (float *)nullptr, grad, dmu, dsg, g->dstatus);
}
