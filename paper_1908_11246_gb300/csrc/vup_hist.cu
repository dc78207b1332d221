// Output probability vectors (Eq. 4 / Eq. 5, Eq. VUP): H[k, b] = sum of the
// normalised input probabilities of the grid points whose model value falls in
// bin b.  The one-hot model matrix of Eq. MUP is applied as a segmented
// reduction over the grid points pre-sorted by bin ("sort and sum").
//
// Layout: a warp serves 128 densities, four per lane; every lane walks the
// same sorted point stream, so control flow is uniform and one 16-byte gather
// per lane (128 consecutive shared-memory words per warp, conflict-free)
// yields four distribution-points.  Points are grouped in runs that share the sort key
// and every axis index but the gathered one: inside a run only the gathered
// axis' factor is read, from a shared-memory tile; the product with the other
// axes' factors is applied once per run.  Those factors are loaded four runs
// ahead: the run-end word of run r carries the rest index of run r + 4.  The
// point stream is staged into shared memory with bulk asynchronous copies
// (cp.async.bulk + mbarrier) and read four points per broadcast load.
//
// The gathered axis is cut into P parts so that one part's 64-density tile
// fits in shared memory; the stream is sorted by (part, bin) and every part
// is chunked separately.  Each warp owns a chunk; bins cut by chunk
// boundaries are written as partials, and a reduction kernel sums partials
// and parts in a fixed order (deterministic).  On 2-D grids two layouts exist
// (either axis gathered); the device uses the one with fewer runs.
#include "vup_internal.cuh"
#include "vup_async.cuh"

#include <algorithm>
#include <vector>

namespace {

constexpr int kHistWarps = 20;
constexpr int kChunksPerWarp = 4;                    // chunks per warp in the smallest group
constexpr int kGroupChunks = kHistWarps * kChunksPerWarp;  // chunks per part come in multiples of this
constexpr int kKT = 128;                     // densities per k-tile (four per lane)
constexpr int kWin = 128;                    // sorted-point words per staging buffer
constexpr int kMaxPartRows = 392;            // gathered-axis rows per shared-memory tile
constexpr int kRowShift = 9;                 // log2 of a tile row's bytes (kKT floats)
constexpr uint32_t kOffMask = 0x1ffu << kRowShift;  // row byte offset (rows < 512)
constexpr uint32_t kRunEnd = 1u << 30, kBinEnd = 1u << 31;
constexpr uint32_t kFlags = kRunEnd | kBinEnd;
constexpr uint32_t kSpin = 1u << 26;
constexpr int kPF = 16;                      // runs prefetched per block (global fallback)
constexpr int kHistCtr = 5;                  // hist_sel[5..7]: the item counters of the three streams' walks
constexpr int kRecBinsH = 8;                 // bins per record group (the layout builder's kRecBins)

struct LayoutArgs {
    const uint32_t *hpt;
    const int32_t *perm;   // sorted position -> flat index of the layout (global fallback)
    const int32_t *run_start, *run_rest, *run_bin;
    const int32_t *chunk_pt, *chunk_run, *chunk_bin;
    const int32_t *koff;   // key offsets [P * B + 1]
    const int2 *key_chunks;  // [P * B] first / last chunk of each key (-1 if empty)
    const uint2 *ipt;      // interval stream (word pairs)
    const int32_t *iv_rest, *chunk_iv;
    const uint4 *rec;      // record stream (two uint4 per record)
    const int32_t *rec_rest, *rec_goff;
    const int2 *rec_gch;   // first / last chunk holding each group
    const int32_t *n_rec, *n_iv;
    const int32_t *rec_chunk, *rec_chunk_grp;
    const float *g_last;   // factor table of the gathered axis  [n_last][K_pad]
    const float *g0, *g1;  // rest-axis factor tables (g1 only for 3-D)
    int64_t n_last, part_rows;
    int64_t n1;            // size of the second rest axis (3-D)
    int64_t n0;            // rows of g0 (the first rest axis)
    int P;
    int ax_last, ax0, ax1; // the axes behind g_last, g0 and g1
    // members of the gathered axis' classes (CSR), null when it is not folded: its
    // rows of g_last are then summed as a tile is filled
    const int32_t *cls_start, *cls_members;
};

// (n_last, part_rows, n0, n1, P and the factor tables of L0 / L1 are the unfolded
// grid's; pick() replaces them by the merged grid's, known on the device)
struct HistArgs {
    LayoutArgs L0, L1;
    const FoldGeom *fold;
    const float *ftab, *ftab_fold;  // factor tables and merged factor tables, axis d at off / foff[d] rows
    int64_t off[3], foff[3];
    const int32_t *fold_start, *fold_members;  // class members per axis, as laid out by the layout build
    const int32_t *sel;   // device: chosen layout, stream (1 = intervals)
    const DensStats *ds;
    int ndim;
    int64_t K, K_pad;
    int B;
    int C;                // chunks per part
    int sets;             // batched form: work items per part and density tile (each a range of its chunks)
    int C_rec;            // record chunks per part
    int GB;               // record groups per part: ceil(B / kRecBins)
    int points_only;      // 1: point stream whatever the layout choice says
    float *hist;          // [K][B]
    float *part;          // [P * C][2][K_pad]
    float *direct;        // [P][K][B] (P > 1)
    int *dstatus;
};

// The chosen layout on the merged grid.
__device__ __forceinline__ LayoutArgs pick(const HistArgs &A) {
    const int l = A.sel[0] ? 1 : 0;
    LayoutArgs H = l ? A.L1 : A.L0;
    const FoldGeom *F = A.fold;
    H.n_last = F->n_last[l];
    H.part_rows = F->part_rows[l];
    H.P = F->P[l];
    if (F->any) {
        if (F->folded[H.ax_last]) {
            H.cls_start = A.fold_start + A.off[H.ax_last] + H.ax_last;
            H.cls_members = A.fold_members + A.off[H.ax_last];
        }
        if (F->folded[H.ax0]) H.g0 = A.ftab_fold + A.foff[H.ax0] * A.K_pad;
        H.n0 = F->n[H.ax0];
        if (A.ndim == 3) {
            if (F->folded[H.ax1]) H.g1 = A.ftab_fold + A.foff[H.ax1] * A.K_pad;
            H.n1 = F->n[H.ax1];
        }
    }
    return H;
}

using namespace vup_async;

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Bulk copy of `bytes` (multiple of 16, both addresses 16-byte aligned)
// completing on `bar`.
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// Shared memory of k_hist_smem: the part's gathered-axis factor tile
// [rows + 1][64] (the extra row is zero; foreign points of a chunk's first
// and last group point at it), per warp 2 staging buffers of kWin point
// words, 2 mbarriers per warp.
__host__ __device__ inline size_t hist_tile_bytes(int64_t rows) { return (size_t)((rows + 1) * kKT * 4); }
__host__ __device__ inline size_t hist_warp_bytes() { return (size_t)2 * kWin * 4; }
// Kernel variants: 0 point stream, 1 interval stream, 2 record stream, 3
// record stream with 16 warps of up to 128 registers (more of its five
// gathers and four accumulators in flight per warp; measured faster when the
// rest-factor table stays in L2, slower when its rows come from HBM and more
// warps hide the latency), 4 and 5 point and record stream of a 3-D grid with
// both rest-axis factor tables staged in shared memory.  The others run 20
// warps of 96 registers.  Each fills the register file of the one CTA per SM that the
// tile allows.
__host__ __device__ constexpr int hist_warps(int mode) { return (mode == 2 || mode == 3 || mode == 5) ? 16 : kHistWarps; }
__host__ __device__ constexpr int hist_stream_of(int mode) { return (mode == 3 || mode == 5) ? 2 : (mode == 4 ? 0 : mode); }
__host__ __device__ constexpr bool hist_staged(int mode) { return mode == 4 || mode == 5; }
__host__ __device__ inline size_t hist_smem_bytes(int64_t rows, int warps = kHistWarps) {
    return hist_tile_bytes(rows) + warps * hist_warp_bytes() + warps * 2 * sizeof(uint64_t);
}

// Store the finished sums of key `key` for this lane's four densities (global
// fallback kernel: the normalisers are applied here).
struct Flusher {
    const HistArgs &A;
    const LayoutArgs &H;
    int c, p;
    int32_t p0, p1, first_key;
    int64_t k;
    float4 invZ;
    __device__ __forceinline__ void operator()(int32_t key, float4 v) const {
        const float4 val = make_float4(v.x * invZ.x, v.y * invZ.y, v.z * invZ.z, v.w * invZ.w);
        const bool shared = H.koff[key] < p0 || H.koff[key + 1] > p1;
        if (shared) {
            const int side = (key == first_key) ? 0 : 1;
            *reinterpret_cast<float4 *>(A.part + ((int64_t)c * 2 + side) * A.K_pad + k) = val;
        } else {
            *reinterpret_cast<float4 *>(A.direct + (int64_t)key * A.K_pad + k) = val;
        }
    }
};

__device__ __forceinline__ float inv_z(const HistArgs &A, int64_t k) {
    if (k >= A.K) return 0.f;
    double z = 1.0;
    for (int d = 0; d < A.ndim; ++d) z *= A.ds[k * A.ndim + d].invZ;
    return (float)z;
}

__device__ __forceinline__ float4 load_inv_z(const HistArgs &A, int64_t k) {
    return make_float4(inv_z(A, k), inv_z(A, k + 1), inv_z(A, k + 2), inv_z(A, k + 3));
}

// Four densities' values per lane, handled as two packed FP32 pairs: the
// .f32x2 forms round each half exactly as the scalar operation does, so the
// sums are bit-identical to four scalar FMAs / subtractions, in half the
// instructions.
__device__ __forceinline__ uint64_t pk2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 up2(uint64_t r) {
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
    return v;
}
__device__ __forceinline__ float4 from_pairs(uint64_t lo, uint64_t hi) {
    const float2 l = up2(lo), h = up2(hi);
    return make_float4(l.x, l.y, h.x, h.y);
}
__device__ __forceinline__ float4 ld4(const float *q) { return *reinterpret_cast<const float4 *>(q); }
__device__ __forceinline__ float4 mul4(float4 a, float4 b) {
    uint64_t lo, hi;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(lo) : "l"(pk2(a.x, a.y)), "l"(pk2(b.x, b.y)));
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(hi) : "l"(pk2(a.z, a.w)), "l"(pk2(b.z, b.w)));
    return from_pairs(lo, hi);
}
__device__ __forceinline__ float4 sub4(float4 a, float4 b) {
    uint64_t lo, hi;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(lo) : "l"(pk2(a.x, a.y)), "l"(pk2(b.x, b.y)));
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(hi) : "l"(pk2(a.z, a.w)), "l"(pk2(b.z, b.w)));
    return from_pairs(lo, hi);
}
__device__ __forceinline__ void add4(float4 &a, float4 b) {
    uint64_t lo = pk2(a.x, a.y), hi = pk2(a.z, a.w);
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(lo) : "l"(pk2(b.x, b.y)));
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(hi) : "l"(pk2(b.z, b.w)));
    a = from_pairs(lo, hi);
}
__device__ __forceinline__ void fma4(float4 &a, float4 w, float4 b) {
    uint64_t lo = pk2(a.x, a.y), hi = pk2(a.z, a.w);
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(lo) : "l"(pk2(w.x, w.y)), "l"(pk2(b.x, b.y)));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(hi) : "l"(pk2(w.z, w.w)), "l"(pk2(b.z, b.w)));
    a = from_pairs(lo, hi);
}

// Sums of four densities per lane as FP32 TwoSum pairs.
struct PairSum4 {
    float4 h, l;
    __device__ __forceinline__ void clear() { h = l = make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ __forceinline__ void add(float4 x) {
        two_sum_acc(h.x, l.x, x.x);
        two_sum_acc(h.y, l.y, x.y);
        two_sum_acc(h.z, l.z, x.z);
        two_sum_acc(h.w, l.w, x.w);
    }
    // v z, the product unrounded
    __device__ __forceinline__ void add_scaled(float4 v, float4 z) {
        one(h.x, l.x, v.x, z.x);
        one(h.y, l.y, v.y, z.y);
        one(h.z, l.z, v.z, z.z);
        one(h.w, l.w, v.w, z.w);
    }
    __device__ __forceinline__ float4 value() const {
        return make_float4(h.x + l.x, h.y + l.y, h.z + l.z, h.w + l.w);
    }
    static __device__ __forceinline__ void one(float &h, float &l, float v, float z) {
        const float s = fmaf(v, z, h);
        const float b = s - h;
        l += (h - (s - b)) + fmaf(v, z, -b);
        h = s;
    }
};

// Factor of one class of a folded axis (four densities): its members' factors
// summed in index order as FP32 TwoSum pairs, rounded once.
__device__ __forceinline__ float4 class_factor(const float *__restrict__ col, int64_t K_pad,
                                               const int32_t *__restrict__ members, int32_t m0, int32_t m1) {
    PairSum4 t;
    t.clear();
    for (int32_t m = m0; m < m1; m += 4) {
        float4 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] = m + q < m1 ? ld4(col + (int64_t)(members[m + q] & (kFoldLast - 1)) * K_pad)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 4; ++q) t.add(v[q]);
    }
    return t.value();
}

// One warp's rows of a merged tile: the members m0 .. m1 - 1 of the rows' classes
// in class order (each class' last one flagged), whose factors (src: this lane's
// four densities of row 0 of the gathered axis' factor table) are summed per
// class.  Every row goes to dst
// (SCALED: times the normalisers iz, else its scaled value into the sum that
// tot receives, [h, l][lane]); eight rows' loads are in flight per warp (16, in
// line or not, and packed pair arithmetic measured slower: 121 - 144 us against
// 113 for the walk of 1024 x 1024 points x 16384 densities).
template <bool SCALED, int AHEAD>
__device__ __forceinline__ void tile_rows_in(const float *__restrict__ src, int64_t K_pad,
                                              const int32_t *__restrict__ members, int32_t m0, int32_t m1, float4 iz,
                                              float *dst, float4 *tot) {
    const int lane = threadIdx.x & 31;
    PairSum4 t;
    t.clear();
    PairSum4 c;
    c.clear();
    // lane u holds the u-th entry of a batch of 32
    int32_t e = members && m0 + lane < m1 ? members[m0 + lane] : 0;
    for (int32_t m = m0; m < m1; m += 32) {
        const int32_t e_next = members && m + 32 + lane < m1 ? members[m + 32 + lane] : 0;
        const int n = min(32, m1 - m);
        for (int u0 = 0; u0 < n; u0 += AHEAD) {
            float4 v[AHEAD];
            int32_t r[AHEAD];
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) {
                r[u] = members ? __shfl_sync(0xffffffffu, e, u0 + u) : ((m + u0 + u) | kFoldLast);
                v[u] = u0 + u < n ? ld4(src + (int64_t)(r[u] & (kFoldLast - 1)) * K_pad)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) {
                if (u0 + u < n) {
                    float4 x = v[u];
                    if (members) {
                        c.add(x);
                        x = c.value();
                    }
                    if (r[u] & kFoldLast) {
                        c.clear();
                        if (!SCALED) t.add_scaled(x, iz);
                        *reinterpret_cast<float4 *>(dst) = SCALED ? mul4(x, iz) : x;
                        dst += kKT;
                    }
                }
            }
        }
        e = e_next;
    }
    tot[lane] = t.h;
    tot[32 + lane] = t.l;
}

// One warp's rows of an unmerged tile, n rows from src (this lane's four
// densities), the copies all in flight (each lane reads back its own); dst and
// tot as above.
template <bool SCALED>
__device__ __forceinline__ void plain_rows_in(const float *__restrict__ src, int64_t K_pad, int32_t n, float4 iz, float *dst,
                                  float4 *tot) {
    for (int32_t a = 0; a < n; ++a) cp_async16(dst + (int64_t)a * kKT, src + a * K_pad);
    cp_async_commit();
    cp_async_wait_all();
    PairSum4 t;
    t.clear();
    for (int32_t a = 0; a < n; ++a, dst += kKT) {
        const float4 x = ld4(dst);
        if (SCALED) *reinterpret_cast<float4 *>(dst) = mul4(x, iz);
        else t.add_scaled(x, iz);
    }
    const int lane = threadIdx.x & 31;
    tot[lane] = t.h;
    tot[32 + lane] = t.l;
}

// Per-item context, kept in shared memory: the chosen layout, the output
// pointers and sizes.  Warps read it on demand, so none of it occupies
// registers across the point loop.
struct ItemCtx {
    LayoutArgs H;
    float *part;   // [P * C][2][K_pad] partial sums of keys cut by chunk bounds
    float *direct; // [P * B][K_pad] sums of keys held by one chunk
    int64_t K, K_pad;
    int B, C, C_rec, GB;
    int64_t rest_n0;  // (3-D, staged) rows of the first rest axis' factors, before the second's
    int64_t pre_rows;  // rows of a prefix tile (debug build's bound)
    int *dstatus;
};

// Store the finished sums of one key for a lane's four densities (16 bytes,
// density-contiguous: one coalesced 512-byte row per warp): keys cut by the
// chunk bounds go to the chunk's partials (side 0 = its first key), the
// others to the key's row of the direct sums.  A one-part histogram also
// goes through the direct rows: scattered 4-byte stores into the [K][B]
// output from the point loop measured slower than the coalesced rows plus
// the finishing copy.  Out of line: it runs once per key, and keeping it
// out of the point loop keeps that loop's code small.
__device__ __noinline__ void flush_key(const ItemCtx *X, int c, int p, int64_t k, int32_t key, float4 v,
                                       bool shared, bool first) {
    float *dst = shared ? X->part + ((int64_t)c * 2 + (first ? 0 : 1)) * X->K_pad + k
                        : X->direct + (int64_t)key * X->K_pad + k;
    *reinterpret_cast<float4 *>(dst) = v;
}

// Interval stream of chunk c (part p): interval i adds f_i (P[b_i] - P[a_i])
// to its key's sum for the lane's four densities, P being the part's prefix
// sums in the shared-memory tile and f_i its rest-axis factor.  Every
// interval loads its own rest factor four intervals ahead into one of four
// registers (the interval's index mod 4), so the loop runs in steps of four
// intervals (two 16-byte broadcast loads of word pairs) and rotates nothing.
template <int NF>
__device__ __forceinline__ bool iv_chunk(const ItemCtx &X, int c, int p, int64_t k, const float *ws, uint32_t *win,
                                         uint64_t *mbar, uint32_t &wseq, volatile int *abort) {
    const LayoutArgs &H = X.H;
    const int lane = threadIdx.x & 31;
    const int32_t p0 = H.chunk_pt[c], p1 = H.chunk_pt[c + 1];
    if (p0 >= p1) return true;
    const int32_t i0 = H.chunk_iv[c], i1 = H.chunk_iv[c + 1];
    const int32_t r0 = H.chunk_run[c], r1 = H.chunk_run[c + 1];
    const int32_t first_key = H.chunk_bin[2 * c], last_key = H.chunk_bin[2 * c + 1];
    const bool sh_first = H.koff[first_key] < p0 || H.koff[first_key + 1] > p1;
    const bool sh_last = H.koff[last_key] < p0 || H.koff[last_key + 1] > p1;

    // words [w0, w1): intervals from i0 rounded down to a multiple of four
    const int32_t ib = i0 & ~3;
    const int32_t w0 = 2 * ib, w1 = 2 * i1;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(H.ipt);
    const int32_t wb0 = w0 & ~(kWin - 1);
    if (lane == 0) {
        const int b0 = wseq & 1;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // earlier reads of both buffers
        bulk_copy(win + b0 * kWin, src + wb0, kWin * 4, &mbar[b0]);
        if (wb0 + kWin < w1) bulk_copy(win + (b0 ^ 1) * kWin, src + wb0 + kWin, kWin * 4, &mbar[b0 ^ 1]);
    }
    __syncwarp();

    // rest-factor rows: this lane's four densities of row `row` (byte stride)
    const uint32_t stride = (uint32_t)(X.K_pad * 4);
    const char *g0b = reinterpret_cast<const char *>(H.g0 + k);
    const char *g1b = NF == 2 ? reinterpret_cast<const char *>(H.g1 + k) : nullptr;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    auto row4 = [&](const char *base, uint32_t row) -> float4 {
        return *reinterpret_cast<const float4 *>(base + (uint64_t)row * stride);
    };
    // factor of interval i + 4 from interval i's code: 9 low bits below the row
    // field and 12 bits above it (2-D: the rest index; 3-D: a0 low, a1 high)
    // (debug build: rows outside the factor tables are recorded and read as row 0)
    auto rest2 = [&](uint32_t a0, uint32_t a1) -> float4 {
        if (!VUP_DBG_IN(a0, H.n0, X.dstatus)) a0 = 0;
        if (!VUP_DBG_IN(a1, H.n1, X.dstatus)) a1 = 0;
        return mul4(row4(g0b, a0), row4(g1b, a1));
    };
    auto rest1 = [&](uint32_t a0) -> float4 {
        if (!VUP_DBG_IN(a0, H.n0, X.dstatus)) a0 = 0;
        return row4(g0b, a0);
    };
    auto coded_factor = [&](uint32_t u) -> float4 {
        if (NF == 2) return rest2(u & 0x1ffu, (u >> 18) & 0xfffu);
        return rest1((u & 0x1ffu) | ((u >> 9) & (0xfffu << 9)));
    };
    auto first_factor = [&](int32_t i) -> float4 {
        if (i < i0 || i >= i1) return zero4;
        const int32_t rest = H.iv_rest[i];
        if (NF == 2) {
            const int32_t a0 = rest / (int32_t)H.n1;
            return rest2((uint32_t)a0, (uint32_t)(rest - a0 * (int32_t)H.n1));
        }
        return rest1((uint32_t)rest);
    };
    float4 f0 = first_factor(ib), f1 = first_factor(ib + 1), f2 = first_factor(ib + 2), f3 = first_factor(ib + 3);

    float4 bacc = zero4;
    int32_t r = r0, cur_key = first_key;
    const uint32_t wsl = smem_u32(ws) + lane * 16;
    auto gather = [&](uint32_t addr) -> float4 {
        float4 v;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                     : "r"(addr));
        return v;
    };
    auto flush = [&](int32_t key, float4 v) {
        const bool first = key == first_key;
        flush_key(&X, c, p, k, key, v, first ? sh_first : (key == last_key && sh_last), first);
    };
    auto step = [&](uint32_t x, uint32_t y, float4 &f) {
        uint32_t xo = x, yo = y & kOffMask;  // (debug build: rows past the tile are recorded, read as row 0)
        if (!VUP_DBG_IN(xo >> kRowShift, X.pre_rows, X.dstatus)) xo = 0;
        if (!VUP_DBG_IN(yo >> kRowShift, X.pre_rows, X.dstatus)) yo = 0;
        const float4 pa = gather(wsl + xo), pb = gather(wsl + yo);
        fma4(bacc, f, sub4(pb, pa));
        f = coded_factor(y);
        if (y & kBinEnd) {
            if (VUP_DBG_IN(cur_key, (int64_t)H.P * X.B, X.dstatus)) flush(cur_key, bacc);
            bacc = zero4;
            cur_key = r + 1 < r1 ? H.run_bin[r + 1] : -1;
        }
        r += (y >> 30) & 1u;  // run end
    };
    // foreign intervals read row 0 twice (difference 0) and carry no flags;
    // those before the chunk keep their rest codes (they load the chunk's first factors)
    constexpr uint32_t kCodes = ~(kOffMask | kFlags);
    auto masked = [&](uint32_t &x, uint32_t &y, int32_t i) {
        if (i < i0) {
            x = 0u;
            y &= kCodes;
        } else if (i >= i1) {
            x = 0u;
            y = 0u;
        }
    };

    for (int32_t wbase = wb0; wbase < w1; wbase += kWin, ++wseq) {
        const int b = wseq & 1;
        for (uint32_t i = 0; !mbar_try_wait(&mbar[b], (wseq >> 1) & 1); ++i) {
            if (i > kSpin || *abort) {  // a staged copy never landed: record and stop
                *abort = 1;
                atomicCAS(X.dstatus, 0, VUP_DSTAT_TIMEOUT);
                return false;
            }
        }
        const uint32_t *wv = win + b * kWin;
        const int lo = (w0 > wbase ? w0 : wbase) - wbase;
        const int hi = (w1 < wbase + kWin ? w1 : wbase + kWin) - wbase;
        for (int q = lo; q < hi; q += 8) {
            uint4 u0 = *reinterpret_cast<const uint4 *>(wv + q), u1 = *reinterpret_cast<const uint4 *>(wv + q + 4);
            const int32_t iq = (wbase + q) >> 1;
            if (iq < i0 || iq + 4 > i1) {
                masked(u0.x, u0.y, iq);
                masked(u0.z, u0.w, iq + 1);
                masked(u1.x, u1.y, iq + 2);
                masked(u1.z, u1.w, iq + 3);
            }
            step(u0.x, u0.y, f0);
            step(u0.z, u0.w, f1);
            step(u1.x, u1.y, f2);
            step(u1.z, u1.w, f3);
        }
        __syncwarp();
        if (lane == 0 && wbase + 2 * kWin < w1) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bulk_copy(win + b * kWin, src + wbase + 2 * kWin, kWin * 4, &mbar[b]);
        }
    }
    if (cur_key >= 0) flush(cur_key, bacc);
    return true;
}

// Record stream, chunk c of part p: record t adds s_t f_t (P[B_j+1] - P[B_j])
// to bin 8q + j, j = 0..7: a gather of P[B_0] and four more for each half of
// the group that holds a bin, one rest-factor load four records ahead, s_t
// its sign; a group's eight sums are stored when its last record passes (groups
// cut by the chunk bounds -- only its first and last -- go to the chunk's
// partial rows, as keys do on the other streams).
constexpr uint32_t kRecNegFlag = 1u << 30;
constexpr uint32_t kRecEndFlag = 1u << 31;

// Store a record group's eight sums (a lane's four densities each): whole
// groups to their direct rows, cut ones to the chunk's partial rows (side 0:
// its first group).  Out of line, like flush_key: it runs once per group.
__device__ __noinline__ void flush_group(const ItemCtx *X, int c, int p, int64_t k, int32_t gr, bool shared,
                                         bool first, float4 a0, float4 a1, float4 a2, float4 a3, float4 a4,
                                         float4 a5, float4 a6, float4 a7) {
    const int b0 = (gr - p * X->GB) * kRecBinsH;
    const int64_t K_pad = X->K_pad;
    float *row = shared ? X->part + ((int64_t)c * 2 + (first ? 0 : 1)) * kRecBinsH * K_pad + k
                        : X->direct + ((int64_t)p * X->B + b0) * K_pad + k;
    const float4 a[kRecBinsH] = {a0, a1, a2, a3, a4, a5, a6, a7};
#pragma unroll
    for (int j = 0; j < kRecBinsH; ++j)
        if (shared || b0 + j < X->B) *reinterpret_cast<float4 *>(row + j * K_pad) = a[j];
}
// RS: the rest-axis factor rows are read from shared memory (w0s, w1s).
template <int NF, bool RS>
__device__ __forceinline__ bool rec_chunk_walk(const ItemCtx &X, int c, int p, int64_t k, const float *ws,
                                               const float *w0s, const float *w1s, uint32_t *win, uint64_t *mbar, uint32_t &wseq, volatile int *abort) {
    const LayoutArgs &H = X.H;
    const int lane = threadIdx.x & 31;
    const int32_t r0 = H.rec_chunk[c], r1 = H.rec_chunk[c + 1];
    if (r0 >= r1) return true;
    const int32_t first_grp = H.rec_chunk_grp[2 * c], last_grp = H.rec_chunk_grp[2 * c + 1];
    // a group is cut when it starts before or ends after the chunk
    const bool sh_first = H.rec_goff[first_grp] < r0 || H.rec_goff[first_grp + 1] > r1;
    const bool sh_last = H.rec_goff[last_grp] < r0 || H.rec_goff[last_grp + 1] > r1;
    const bool last_ends = (H.rec[2 * (int64_t)(r1 - 1) + 1].x & kRecEndFlag) != 0;
    // words [w0, w1): records from r0 rounded down to a multiple of four
    const int32_t rb = r0 & ~3;
    const int64_t w0 = 8 * (int64_t)rb, w1 = 8 * (int64_t)r1;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(H.rec);
    const int64_t wb0 = w0 & ~(int64_t)(kWin - 1);
    if (lane == 0) {
        const int b0 = wseq & 1;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // earlier reads of both buffers
        bulk_copy(win + b0 * kWin, src + wb0, kWin * 4, &mbar[b0]);
        if (wb0 + kWin < w1) bulk_copy(win + (b0 ^ 1) * kWin, src + wb0 + kWin, kWin * 4, &mbar[b0 ^ 1]);
    }
    __syncwarp();

    const uint32_t stride = (uint32_t)(X.K_pad * 4);
    const char *g0b = reinterpret_cast<const char *>(H.g0 + k);
    const char *g1b = NF == 2 ? reinterpret_cast<const char *>(H.g1 + k) : nullptr;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    auto row4 = [&](const char *base, uint32_t row) -> float4 {
        return *reinterpret_cast<const float4 *>(base + (uint64_t)row * stride);
    };
    // rest factor from a record's code (2-D: the rest index; 3-D: a0 | a1 << 15)
    // (debug build: rows outside the factor tables are recorded and read as row 0)
    auto rest2 = [&](uint32_t a0, uint32_t a1) -> float4 {
        if (!VUP_DBG_IN(a0, H.n0, X.dstatus)) a0 = 0;
        if (!VUP_DBG_IN(a1, H.n1, X.dstatus)) a1 = 0;
        if (RS) return mul4(ld4(w0s + a0 * kKT), ld4(w1s + a1 * kKT));
        return mul4(row4(g0b, a0), row4(g1b, a1));
    };
    auto rest1 = [&](uint32_t a0) -> float4 {
        if (!VUP_DBG_IN(a0, H.n0, X.dstatus)) a0 = 0;
        return row4(g0b, a0);
    };
    auto coded_factor = [&](uint32_t u) -> float4 {
        if (NF == 2) return rest2(u & 0x7fffu, u >> 15);
        return rest1(u);
    };
    auto first_factor = [&](int32_t t) -> float4 {
        if (t < r0 || t >= r1) return zero4;
        const int32_t rest = H.rec_rest[t];
        if (NF == 2) {
            const int32_t a0 = rest / (int32_t)H.n1;
            return rest2((uint32_t)a0, (uint32_t)(rest - a0 * (int32_t)H.n1));
        }
        return rest1((uint32_t)rest);
    };
    float4 f0 = first_factor(rb), f1 = first_factor(rb + 1), f2 = first_factor(rb + 2), f3 = first_factor(rb + 3);

    float4 acc[kRecBinsH];
#pragma unroll
    for (int j = 0; j < kRecBinsH; ++j) acc[j] = zero4;
    // a group's eight sums: whole groups to their direct rows, cut ones to the chunk's partials
    auto flush = [&](int32_t gr) {
        const bool first = gr == first_grp;
        if (VUP_DBG_IN(gr - p * X.GB, X.GB, X.dstatus))  // (debug build: a group outside the part is skipped)
            flush_group(&X, c, p, k, gr, first ? sh_first : (gr == last_grp && sh_last), first, acc[0], acc[1], acc[2],
                    acc[3], acc[4], acc[5], acc[6], acc[7]);
#pragma unroll
        for (int j = 0; j < kRecBinsH; ++j) acc[j] = zero4;
    };
    const uint32_t wsl = smem_u32(ws) + lane * 16;
    auto gather = [&](uint32_t addr) -> float4 {
        float4 v;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                     : "r"(addr));
        return v;
    };
    auto step = [&](const uint4 u, const uint4 v, float4 &f) {
        // boundary rows B_0..B_8 (16 bits each); bins with B_j+1 == B_j are absent
        uint32_t rw[kRecBinsH + 1] = {u.x & 0xffffu, u.x >> 16, u.y & 0xffffu, u.y >> 16, u.z & 0xffffu,
                                      u.z >> 16,     u.w & 0xffffu, u.w >> 16, v.x & 0xffffu};
#ifdef VUP_DEBUG
        // (debug build: a boundary row past the tile makes the record empty)
        bool rows_ok = true;
#pragma unroll
        for (int j = 0; j <= kRecBinsH; ++j) rows_ok = rows_ok && VUP_DBG_IN(rw[j], X.pre_rows, X.dstatus);
        if (!rows_ok)
#pragma unroll
            for (int j = 0; j <= kRecBinsH; ++j) rw[j] = 0;
#endif
        const float4 fs = (v.x & kRecNegFlag) ? make_float4(-f.x, -f.y, -f.z, -f.w) : f;
        // each half (3-D: quarter, a line there holds 2.5 bins of a group where a
        // 2-D one holds 6) of the group is skipped when it holds no bin (its
        // boundaries then all equal its first)
        constexpr int kH = RS ? 2 : kRecBinsH / 2;
        float4 prev = gather(wsl + (rw[0] << kRowShift));
#pragma unroll
        for (int h = 0; h < kRecBinsH / kH; ++h) {
            if (rw[kH * h + kH] != rw[kH * h]) {
#pragma unroll
                for (int j = kH * h; j < kH * h + kH; ++j) {
                    const float4 nx = gather(wsl + (rw[j + 1] << kRowShift));
                    fma4(acc[j], fs, sub4(nx, prev));
                    prev = nx;
                }
            }
        }
        f = coded_factor(v.y);
        if (__builtin_expect((v.x & kRecEndFlag) != 0, 0)) flush((int32_t)v.z);
    };
    // foreign records: every boundary row 0 (differences 0), no group end;
    // those before the chunk keep their rest codes (they load its first factors)
    auto masked = [&](uint4 &u, uint4 &v, int32_t t) {
        if (t < r0) {
            u = make_uint4(0u, 0u, 0u, 0u);
            v = make_uint4(0u, v.y, 0u, 0u);
        } else if (t >= r1) {
            u = make_uint4(0u, 0u, 0u, 0u);
            v = make_uint4(0u, 0u, 0u, 0u);
        }
    };

    for (int64_t wbase = wb0; wbase < w1; wbase += kWin, ++wseq) {
        const int b = wseq & 1;
        for (uint32_t i = 0; !mbar_try_wait(&mbar[b], (wseq >> 1) & 1); ++i) {
            if (i > kSpin || *abort) {  // a staged copy never landed: record and stop
                *abort = 1;
                atomicCAS(X.dstatus, 0, VUP_DSTAT_TIMEOUT);
                return false;
            }
        }
        const uint4 *wq = reinterpret_cast<const uint4 *>(win + b * kWin);
        const int lo = (int)((w0 > wbase ? w0 : wbase) - wbase);
        const int hi = (int)((w1 < wbase + kWin ? w1 : wbase + kWin) - wbase);
        for (int qq = lo; qq < hi; qq += 32) {
            const int32_t t0 = (int32_t)((wbase + qq) >> 3);
            const bool edge = t0 < r0 || t0 + 4 > r1;
            auto one = [&](int m, float4 &f) {
                uint4 u = wq[qq / 4 + 2 * m], v = wq[qq / 4 + 2 * m + 1];
                if (__builtin_expect(edge, 0)) masked(u, v, t0 + m);
                step(u, v, f);
            };
            one(0, f0);
            one(1, f1);
            one(2, f2);
            one(3, f3);
        }
        __syncwarp();
        if (lane == 0 && wbase + 2 * kWin < w1) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bulk_copy(win + b * kWin, src + wbase + 2 * kWin, kWin * 4, &mbar[b]);
        }
    }
    if (!last_ends) flush(last_grp);  // the chunk ends inside its last group
    return true;
}

// One work item: part p, range cg of G of the part's chunks (drawn by the
// warps one at a time) and the 128 densities from k0 of the instance *Ap (kernel parameter or global
// memory).  Called by every thread of the CTA; `wseq` counts the staging
// windows this warp has consumed so far (it keeps the per-warp mbarrier
// phases consistent across items).
template <int NF, int MODE>
__device__ __forceinline__ void hist_item(const HistArgs *Ap, int p, int cg, int G, int64_t k0, uint8_t *sm,
                                          int64_t tile_rows, uint32_t &wseq, volatile int *abort, ItemCtx &X,
                                          float4 *s_invz, int *next_chunk) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t k = k0 + 4 * lane;
    float *ws = reinterpret_cast<float *>(sm);
    const size_t tb = hist_tile_bytes(tile_rows);
    uint32_t *win = reinterpret_cast<uint32_t *>(sm + tb + (size_t)warp * hist_warp_bytes());
    constexpr int kWarps = hist_warps(MODE);
    uint64_t *mbar = reinterpret_cast<uint64_t *>(sm + tb + kWarps * hist_warp_bytes()) + 2 * warp;

    // the previous item's readers of the tile and the context are done first
    __syncthreads();
    if (*abort) return;  // a wait of an earlier item expired (uniform: read after the barrier)
    if (threadIdx.x == 0) {
        const HistArgs &A = *Ap;
        *next_chunk = 0;
        X.H = pick(A);
        X.part = A.part;
        X.direct = A.direct;
        X.K = A.K;
        X.K_pad = A.K_pad;
        X.B = A.B;
        X.C = A.C;
        X.C_rec = A.C_rec;
        X.GB = A.GB;
        X.pre_rows = X.H.part_rows + 1;
        X.dstatus = A.dstatus;
        X.rest_n0 = X.H.n0;
    }
    if (threadIdx.x < kKT) reinterpret_cast<float *>(s_invz)[threadIdx.x] = inv_z(*Ap, k0 + threadIdx.x);
    __syncthreads();
    const LayoutArgs &H = X.H;
    if (p >= H.P) return;  // uniform
    // this part's rows of the gathered-axis factor table (16-byte asynchronous
    // copies) + a zero row, then every column scaled by its density's
    // normaliser 1 / prod_d Z_d
    const int64_t row0 = (int64_t)p * H.part_rows;
    const int64_t nrows = min(H.part_rows, H.n_last - row0);
    // every warp fills its share of the rows; the interval and record
    // streams then turn the columns into exclusive prefix sums P[0..nrows]
    // (each P the TwoSum pair of the rows before it, rounded once to FP32), so
    // that rows a .. b - 1 sum to P[b] - P[a]: the warps' totals first (kept in
    // the idle staging buffers), then each warp again from the totals before
    // it.  (Prefix tiles from a kernel of their own cost 60 us at 1024 rows x
    // 16384 densities, or five times that beside the contraction, whose
    // operands take the L2 bandwidth; the scan here costs an item 3 us.)
    const float4 iz4 = s_invz[lane];
    const int32_t a0 = (int32_t)(nrows * warp / kWarps), a1 = (int32_t)(nrows * (warp + 1) / kWarps);
    PairSum4 t;
    t.clear();
    {
        float *q = ws + (int64_t)a0 * kKT + 4 * lane;
        if (H.cls_start) {
            tile_rows_in<hist_stream_of(MODE) == 0, 8>(H.g_last + k, X.K_pad, H.cls_members, H.cls_start[row0 + a0],
                                                       H.cls_start[row0 + a1], iz4, q, reinterpret_cast<float4 *>(win));
        } else {
            plain_rows_in<hist_stream_of(MODE) == 0>(H.g_last + (row0 + a0) * X.K_pad + k, X.K_pad, a1 - a0, iz4, q,
                                                     reinterpret_cast<float4 *>(win));
        }
    }
    if (hist_staged(MODE)) {
        // the k-tile's rows of both rest-axis factor tables (unnormalised)
        float *rs = reinterpret_cast<float *>(sm + hist_smem_bytes(tile_rows, kWarps));
        const int64_t n0 = X.rest_n0, n1 = H.n1, K_pad = X.K_pad;
        for (int64_t e = threadIdx.x; e < (n0 + n1) * (kKT / 4); e += blockDim.x) {
            const int64_t a = e / (kKT / 4), cc = e % (kKT / 4);
            const float *src = a < n0 ? H.g0 + a * K_pad : H.g1 + (a - n0) * K_pad;
            cp_async16(rs + a * kKT + cc * 4, src + k0 + cc * 4);
        }
        cp_async_commit();
    }
    if (hist_stream_of(MODE) == 0) {
        if (threadIdx.x < kKT) ws[nrows * kKT + threadIdx.x] = 0.f;
    } else {
        __syncthreads();
        t.clear();
        for (int w = 0; w < warp; ++w) {
            const float4 *o = reinterpret_cast<const float4 *>(sm + tb + (size_t)w * hist_warp_bytes());
            t.add(o[lane]);
            add4(t.l, o[32 + lane]);
        }
        float *q = ws + (int64_t)a0 * kKT + 4 * lane;
        for (int32_t a = a0; a < a1; ++a, q += kKT) {
            const float4 x = ld4(q);
            *reinterpret_cast<float4 *>(q) = t.value();
            t.add_scaled(x, iz4);
        }
        if (warp == kWarps - 1) *reinterpret_cast<float4 *>(q) = t.value();
        // the staging buffers are next written by bulk copies (async proxy)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (hist_staged(MODE)) cp_async_wait_all();
    __syncthreads();

    // the item's chunks are handed out one at a time (at least kChunksPerWarp per warp
    // on average), so a warp that drew short chunks takes another instead of
    // idling at the next item's barrier
    auto run_chunk = [&](const int wc) -> bool {
        const int c = p * X.C + wc;
        const int32_t p0 = H.chunk_pt[c], p1 = H.chunk_pt[c + 1];
        if (p0 >= p1) return true;
        const int32_t r0 = H.chunk_run[c], r1 = H.chunk_run[c + 1];
        // keys cut by the chunk bounds can only be its first and last key
        const int32_t first_key = H.chunk_bin[2 * c], last_key = H.chunk_bin[2 * c + 1];
        const bool sh_first = H.koff[first_key] < p0 || H.koff[first_key + 1] > p1;
        const bool sh_last = H.koff[last_key] < p0 || H.koff[last_key + 1] > p1;
        auto flush = [&](int32_t key, float4 v) {
            const bool first = key == first_key;
            flush_key(&X, c, p, k, key, v, first ? sh_first : (key == last_key && sh_last), first);
        };

        // staging of the sorted point stream: window i of this item lands in
        // buffer (wseq + i) & 1
        const uint32_t *hpt = H.hpt;
        const int32_t wb0 = p0 & ~(kWin - 1);
        if (lane == 0) {
            const int b0 = wseq & 1;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // earlier items' reads of both buffers
            bulk_copy(win + b0 * kWin, hpt + wb0, kWin * 4, &mbar[b0]);
            if (wb0 + kWin < p1) bulk_copy(win + (b0 ^ 1) * kWin, hpt + wb0 + kWin, kWin * 4, &mbar[b0 ^ 1]);
        }
        __syncwarp();

        // rest-axis factors (four densities) of runs r .. r + 3, rotated through registers
        const int64_t K_pad = X.K_pad;
        const float *g0k = H.g0 + k;
        const float *g1k = NF == 2 ? H.g1 + k : nullptr;
        const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
        // 3-D: the product of the two rest axes' rows; with the rows staged in
        // shared memory (MODE 4) the first axis' row is kept in registers while
        // consecutive runs share it (95% of them on the 3-D workload: runs of
        // a bin are ordered by line)
        constexpr bool rs = NF == 2 && MODE == 4;
        const float *w0s = reinterpret_cast<const float *>(sm + hist_smem_bytes(tile_rows, kWarps)) + 4 * lane;
        const float *w1s = w0s + X.rest_n0 * kKT;
        uint32_t a0c = 0xffffffffu;
        float4 w0c = zero4;
        auto rest_rows = [&](uint32_t a0, uint32_t a1) -> float4 {
            // (debug build: rows outside the factor tables are recorded and read as row 0)
            if (!VUP_DBG_IN(a0, H.n0, X.dstatus)) a0 = 0;
            if (!VUP_DBG_IN(a1, H.n1, X.dstatus)) a1 = 0;
            if (rs) {
                if (a0 != a0c) {  // uniform: every lane follows the same run
                    w0c = ld4(w0s + a0 * kKT);
                    a0c = a0;
                }
                return mul4(w0c, ld4(w1s + a1 * kKT));
            }
            return mul4(ld4(g0k + (int64_t)a0 * K_pad), ld4(g1k + (int64_t)a1 * K_pad));
        };
        auto rest_factor = [&](int32_t r) -> float4 {
            if (r >= r1) return zero4;
            const int32_t rest = H.run_rest[r];
            if (NF == 2) {
                const int32_t a0 = rest / (int32_t)H.n1, a1 = rest - a0 * (int32_t)H.n1;
                return rest_rows((uint32_t)a0, (uint32_t)a1);
            }
            return ld4(g0k + (VUP_DBG_IN(rest, H.n0, X.dstatus) ? rest : 0) * K_pad);
        };
        // fc = factor of the current run, f1..f3 those of the next three runs
        // (MODE 4: shared-memory factors, no look-ahead: fc only)
        float4 fc = rest_factor(r0), f1 = zero4, f2 = zero4, f3 = zero4;
        if (!rs) {
            f1 = rest_factor(r0 + 1);
            f2 = rest_factor(r0 + 2);
            f3 = rest_factor(r0 + 3);
        }
        // factor of run r + 4 (MODE 4: r + 1), decoded from run r's end word: 9
        // low bits below the row field and 12 bits above it
        auto coded_factor = [&](uint32_t u) -> float4 {
            if (NF == 2) return rest_rows(u & 0x1ffu, (u >> 18) & 0xfffu);
            const uint32_t idx = (u & 0x1ffu) | (((u >> 18) & 0xfffu) << 9);
            return ld4(g0k + (int64_t)(VUP_DBG_IN(idx, H.n0, X.dstatus) ? idx : 0u) * K_pad);
        };

        // every point's factor is multiplied by its run's rest-axis factor fc as it
        // is added (one FMA per density, the same count as a plain add), so a run
        // end only advances the factor pipeline
        int32_t r = r0, cur_key = first_key;
        float4 bacc = zero4;
        const uint32_t wsl = smem_u32(ws) + lane * 16;
        const uint32_t null_word = (uint32_t)nrows << kRowShift;  // zero row, no flags

        auto run_end = [&](uint32_t u) {
            if (u & kBinEnd) {
                if (VUP_DBG_IN(cur_key, (int64_t)H.P * X.B, X.dstatus)) flush(cur_key, bacc);
                bacc = zero4;
                cur_key = r + 1 < r1 ? H.run_bin[r + 1] : -1;
            }
            if (rs) {
                fc = r + 1 < r1 ? coded_factor(u) : zero4;
            } else {
                fc = f1;
                f1 = f2;
                f2 = f3;
                f3 = coded_factor(u);
            }
            ++r;
        };
        auto gather = [&](uint32_t addr) -> float4 {
            float4 v;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                         : "r"(addr));
            return v;
        };
        // words without flags carry nothing but the row byte offset (run codes sit
        // on run-end words only), so the common path needs no masking
#ifdef VUP_DEBUG
        // (debug build: a row offset past the tile is recorded and read as the zero row 0)
        auto dbg_word = [&](uint32_t w) -> uint32_t {
            if ((w & kFlags) == 0)
                return VUP_DBG_IN(w >> kRowShift, nrows + 1, X.dstatus) && (w & ~kOffMask) == 0 ? w : 0u;
            return VUP_DBG_IN((w & kOffMask) >> kRowShift, nrows + 1, X.dstatus) ? w : (w & ~kOffMask);
        };
#endif
        auto group = [&](uint4 v) {
#ifdef VUP_DEBUG
            v = make_uint4(dbg_word(v.x), dbg_word(v.y), dbg_word(v.z), dbg_word(v.w));
#endif
            if (((v.x | v.y | v.z | v.w) & kFlags) == 0) {
                const float4 a0 = gather(wsl + v.x), a1 = gather(wsl + v.y), a2 = gather(wsl + v.z),
                             a3 = gather(wsl + v.w);
                fma4(bacc, fc, a0);
                fma4(bacc, fc, a1);
                fma4(bacc, fc, a2);
                fma4(bacc, fc, a3);
            } else {
                const float4 a0 = gather(wsl + (v.x & kOffMask)), a1 = gather(wsl + (v.y & kOffMask)),
                             a2 = gather(wsl + (v.z & kOffMask)), a3 = gather(wsl + (v.w & kOffMask));
                fma4(bacc, fc, a0);
                if (v.x & kFlags) run_end(v.x);
                fma4(bacc, fc, a1);
                if (v.y & kFlags) run_end(v.y);
                fma4(bacc, fc, a2);
                if (v.z & kFlags) run_end(v.z);
                fma4(bacc, fc, a3);
                if (v.w & kFlags) run_end(v.w);
            }
        };
        // a group cut by the chunk bounds: foreign points read the zero row
        auto masked = [&](uint4 v, int pa, int lo, int hi) {
            if (pa + 0 < lo || pa + 0 >= hi) v.x = null_word;
            if (pa + 1 < lo || pa + 1 >= hi) v.y = null_word;
            if (pa + 2 < lo || pa + 2 >= hi) v.z = null_word;
            if (pa + 3 < lo || pa + 3 >= hi) v.w = null_word;
            return v;
        };

        for (int32_t wbase = wb0; wbase < p1; wbase += kWin, ++wseq) {
            const int b = wseq & 1;
            for (uint32_t i = 0; !mbar_try_wait(&mbar[b], (wseq >> 1) & 1); ++i) {
                if (i > kSpin || *abort) {  // a staged copy never landed: record and stop
                    *abort = 1;
                    atomicCAS(X.dstatus, 0, VUP_DSTAT_TIMEOUT);
                    return false;
                }
            }
            const uint32_t *wv = win + b * kWin;
            const int lo = (p0 > wbase ? p0 : wbase) - wbase;
            const int hi = (p1 < wbase + kWin ? p1 : wbase + kWin) - wbase;
            const int ga = (lo + 3) & ~3, gb = hi & ~3;   // whole groups [ga, gb)
            if (lo & 3) {
                const int pa = lo & ~3;
                group(masked(*reinterpret_cast<const uint4 *>(wv + pa), pa, lo, hi));
            }
    #pragma unroll 2
            for (int pa = ga; pa < gb; pa += 4) group(*reinterpret_cast<const uint4 *>(wv + pa));
            if ((hi & 3) && gb >= ga) group(masked(*reinterpret_cast<const uint4 *>(wv + gb), gb, lo, hi));
            __syncwarp();
            if (lane == 0 && wbase + 2 * kWin < p1) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                bulk_copy(win + b * kWin, hpt + wbase + 2 * kWin, kWin * 4, &mbar[b]);
            }
        }
        if (cur_key >= 0) flush(cur_key, bacc);
        return true;
    };
    if constexpr (hist_stream_of(MODE) == 2) {
        // this item's range of the part's record chunks, handed out one at a time
        const int c_lo = (int)((int64_t)cg * X.C_rec / G), c_hi = (int)((int64_t)(cg + 1) * X.C_rec / G);
        for (;;) {
            int ci = 0;
            if (lane == 0) ci = atomicAdd(next_chunk, 1);
            ci = __shfl_sync(0xffffffffu, ci, 0);
            if (c_lo + ci >= c_hi) break;
            const float *w0s = reinterpret_cast<const float *>(sm + hist_smem_bytes(tile_rows, kWarps)) + 4 * lane;
            if (!rec_chunk_walk<NF, hist_staged(MODE)>(X, p * X.C_rec + c_lo + ci, p, k, ws, w0s,
                                                       w0s + X.rest_n0 * kKT, win, mbar, wseq, abort))
                return;
        }
    } else {
        for (;;) {
            int ci = 0;
            if (lane == 0) ci = atomicAdd(next_chunk, 1);
            ci = __shfl_sync(0xffffffffu, ci, 0);
            const int wc = (int)((int64_t)cg * X.C / G) + ci;
            if (wc >= (int)((int64_t)(cg + 1) * X.C / G)) break;
            bool ok;
            if constexpr (MODE == 1) ok = iv_chunk<NF>(X, p * X.C + wc, p, k, ws, win, mbar, wseq, abort);
            else ok = run_chunk(wc);
            if (!ok) return;
        }
    }
}

__device__ __forceinline__ uint64_t *hist_mbar(uint8_t *sm, int64_t tile_rows, int warps) {
    return reinterpret_cast<uint64_t *>(sm + hist_tile_bytes(tile_rows) + warps * hist_warp_bytes()) +
           2 * (threadIdx.x >> 5);
}
__device__ __forceinline__ void hist_init_mbar(uint8_t *sm, int64_t tile_rows, int warps) {
    if ((threadIdx.x & 31) == 0) {
        uint64_t *mbar = hist_mbar(sm, tile_rows, warps);
        mbar_init(&mbar[0], 1);
        mbar_init(&mbar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
}

// Stream of an instance's histogram: 1 = intervals (the layout's choice,
// unless the caller asked for points).
__device__ __forceinline__ int hist_stream(const HistArgs &A) { return A.points_only ? 0 : A.sel[1]; }

// Work items per (part, density tile) of a walk over n elements (points,
// intervals or records) per part in C chunks: the split G that ends first by
//   ceil(items / CTAs) (tile + max(n thr / G, ceil(C / G / warps) n / C thr warps / 2))
// SM cycles: the tile's copy (about 10 cycles per 512-byte row after a 3000-cycle
// start), the walk at its measured rate thr per element and 128 densities, or,
// where an item has fewer chunks than warps, at half a warp's share of it
// (latency).  Few density tiles are cut into up to C items (a 200 x 328 grid
// with 225 densities ran on 2 CTAs), many into as few as fill the last wave.
// One warp evaluates 32 candidates at a time; every CTA finds the same G.
__device__ __forceinline__ int hist_split(int64_t n, int C, int64_t tiles, int64_t rows, int warps, float thr,
                                          int ctas) {
    const int lane = threadIdx.x & 31;
    float best = 3.0e38f;
    int bg = 1;
    for (int g = 1 + lane; g <= C; g += 32) {
        const float waves = (float)((tiles * g + ctas - 1) / ctas);
        const float ch = (float)(((C + g - 1) / g + warps - 1) / warps);
        const float walk = (float)n * thr;
        const float t = waves * (3000.f + 10.f * (float)rows +
                                 fmaxf(walk / (float)g, ch * walk / (float)C * 0.5f * (float)warps));
        if (t < best) {
            best = t;
            bg = g;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ot = __shfl_xor_sync(0xffffffffu, best, o);
        const int og = __shfl_xor_sync(0xffffffffu, bg, o);
        if (ot < best || (ot == best && og < bg)) {
            best = ot;
            bg = og;
        }
    }
    return bg;
}
// Measured SM cycles per element and 128 densities of each stream's walk.
__host__ __device__ constexpr float hist_rate(int mode) {
    return hist_stream_of(mode) == 2 ? 55.f : (mode == 1 ? 19.f : 6.f);
}

// Persistent CTAs, one per SM (the tile fills its shared memory), drawing the
// items it = (k-tile * P + part) * G + range in order from a counter, so that
// CTAs running together share k-tiles (rest-factor rows stay in L2) and an SM
// takes the next item as it frees up (item costs vary; a static split of
// items over the CTAs measured 12 % slower on the 3-D workload).  The counters
// are zeroed by the merged-table kernel, which runs before the walks of every
// call.  Each stream is its own kernel (their register allocations stay
// apart); the host launches every stream's and the CTAs of those the device
// did not choose return at once (a CTA per item instead cost 32 us for each of
// them at 65536 densities of a 2048 x 2048 grid).
template <int NF, int MODE>
__global__ void __launch_bounds__(hist_warps(MODE) * 32, 1)
    k_hist_smem(const __grid_constant__ HistArgs A, int64_t tile_rows, int nkt, int *__restrict__ next_item) {
    pdl_trigger();
    pdl_wait();
    if (hist_stream(A) != hist_stream_of(MODE)) return;  // uniform
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ ItemCtx X;
    __shared__ float4 s_invz[kKT / 4];  // (the type: a lane reads four as one 16-byte load)
    __shared__ int abort, next_chunk, s_item, s_G;
    if (threadIdx.x == 0) abort = 0;
    hist_init_mbar(sm, tile_rows, hist_warps(MODE));
    const int P = A.fold->P[A.sel[0] ? 1 : 0];
    if (threadIdx.x < 32) {
        const LayoutArgs &L = A.sel[0] ? A.L1 : A.L0;
        const int64_t n = hist_stream_of(MODE) == 2 ? L.n_rec[0] : (MODE == 1 ? L.n_iv[0] : A.fold->N);
        const int C = hist_stream_of(MODE) == 2 ? A.C_rec : A.C;
        const int G = hist_split(n / P, C, (int64_t)nkt * P, A.fold->part_rows[A.sel[0] ? 1 : 0], hist_warps(MODE),
                                 hist_rate(MODE), gridDim.x);
        if (threadIdx.x == 0) s_G = G;
    }
    uint32_t wseq = 0;
    for (;;) {
        __syncthreads();  // the previous item's readers of s_item are done
        if (threadIdx.x == 0) s_item = atomicAdd(next_item, 1);
        __syncthreads();
        const int G = s_G, it = s_item;
        if (it >= (int64_t)nkt * P * G || abort) return;
        const int cg = it % G, pk = it / G;
        const int p = pk % P, kt = pk / P;
        hist_item<NF, MODE>(&A, p, cg, G, (int64_t)kt * kKT, sm, tile_rows, wseq, &abort, X, s_invz, &next_chunk);
    }
}

// Batched form: one persistent launch per stream over the work items of
// many instances (each with its own grid, densities and outputs), longest
// items first; items of instances on the other stream are skipped.
struct HistItem {
    int32_t inst, p, cg, kt;
};

// Per-stream item lists of a batch: the items of the instances whose
// device-chosen stream s is served by launch s, in the plan's (longest
// first) order, so that no launch walks past the other streams' items.  One
// CTA: the instances' streams to shared memory (global reads past
// kSplitStaged instances), then the items in blocks of kSplitThreads, each
// block compacted in order by warp ballots and per-warp counts.
constexpr int kSplitThreads = 1024;
constexpr int kSplitStaged = 32768;
__global__ void __launch_bounds__(kSplitThreads) k_hist_split_items(const HistArgs *__restrict__ insts, int n_inst,
                                                                    const HistItem *__restrict__ items, int n_items,
                                                                    int32_t *__restrict__ lists,
                                                                    int32_t *__restrict__ counts) {
    extern __shared__ uint8_t s_stream[];  // [n_inst] when staged
    __shared__ int s_warp[3][kSplitThreads / 32];
    __shared__ int s_base[3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool staged = n_inst <= kSplitStaged;
    if (staged)
        for (int i = tid; i < n_inst; i += blockDim.x) s_stream[i] = (uint8_t)min(hist_stream(insts[i]), 3);
    if (tid < 3) s_base[tid] = 0;
    __syncthreads();
    for (int base = 0; base < n_items; base += kSplitThreads) {
        const int it = base + tid;
        int st = 3;  // 3: no launch serves it
        if (it < n_items) {
            const int inst = items[it].inst;
            st = staged ? (int)s_stream[inst] : min(hist_stream(insts[inst]), 3);
        }
        unsigned m[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) m[q] = __ballot_sync(0xffffffffu, st == q);
        if (lane < 3) s_warp[lane][warp] = __popc(m[lane]);
        __syncthreads();
        if (st < 3) {
            int off = s_base[st] + __popc(m[st] & ((1u << lane) - 1u));
            for (int w = 0; w < warp; ++w) off += s_warp[st][w];
            lists[(int64_t)st * n_items + off] = it;
        }
        __syncthreads();
        if (tid < 3) {
            int t = 0;
            for (int w = 0; w < kSplitThreads / 32; ++w) t += s_warp[tid][w];
            s_base[tid] += t;
        }
        __syncthreads();
    }
    if (tid < 3) counts[tid] = s_base[tid];
}

template <int NF, int MODE>
__global__ void __launch_bounds__(hist_warps(MODE) * 32, 1) k_hist_batched(const HistArgs *__restrict__ insts,
                                                                     const HistItem *__restrict__ items,
                                                                     const int32_t *__restrict__ list,
                                                                     const int32_t *__restrict__ count,
                                                                     int64_t tile_rows,
                                                                     int *__restrict__ next_item) {
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ ItemCtx X;
    __shared__ float4 s_invz[kKT / 4];  // (the type: a lane reads four as one 16-byte load)
    __shared__ int abort, next_chunk, s_it;
    if (threadIdx.x == 0) abort = 0;
    hist_init_mbar(sm, tile_rows, hist_warps(MODE));
    uint32_t wseq = 0;
    // this stream's items are handed out one at a time in their (longest
    // first) order
    const int n_items = *count;
    for (;;) {
        __syncthreads();  // every thread has read the previous s_it
        if (threadIdx.x == 0) s_it = atomicAdd(next_item, 1);
        __syncthreads();
        const int it = s_it;
        if (it >= n_items) break;
        const HistItem w = items[list[it]];
        hist_item<NF, MODE>(insts + w.inst, w.p, w.cg, insts[w.inst].sets, (int64_t)w.kt * kKT, sm, tile_rows, wseq,
                            &abort, X, s_invz, &next_chunk);
    }
}

// Fallback when a part's tile does not fit shared memory (or 3-D rest indices
// exceed the run-end encoding): factors are gathered from global memory
// (L1-cached), rest-axis factors prefetched in register blocks.
__global__ void __launch_bounds__(kHistWarps * 32, 1) k_hist_global(HistArgs A, int G) {
    const LayoutArgs H = pick(A);
    const int p = blockIdx.x / G, cg = blockIdx.x - p * G;
    if (p >= H.P) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t k = (int64_t)blockIdx.y * kKT + 4 * lane;
    const int group = A.C / G;  // chunks of a block: cg * group + j * kHistWarps + warp
    for (int j = 0; j < group / kHistWarps; ++j) {
        const int c = p * A.C + cg * group + j * kHistWarps + warp;
        const int32_t p0 = H.chunk_pt[c], p1 = H.chunk_pt[c + 1];
        if (p0 >= p1) continue;
        const int32_t r0 = H.chunk_run[c], r1 = H.chunk_run[c + 1];
        const Flusher flush{A, H, c, p, p0, p1, H.chunk_bin[2 * c], k, load_inv_z(A, k)};
        // the gathered-axis index comes from the sorted order itself (the point
        // words' row field only covers shared-memory tiles)
        const float *wl = H.g_last + k;
        const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
        auto wrest = [&](int32_t r) -> float4 {
            if (r >= r1) return zero4;
            const int32_t rest = H.run_rest[r];
            if (A.ndim == 3) {
                const int64_t a0 = rest / H.n1, a1 = rest - a0 * H.n1;
                return mul4(ld4(H.g0 + a0 * A.K_pad + k), ld4(H.g1 + a1 * A.K_pad + k));
            }
            return ld4(H.g0 + (int64_t)rest * A.K_pad + k);
        };
        int32_t cur_key = H.run_bin[r0];
        float4 bacc = zero4;
        for (int32_t rb = r0; rb < r1; rb += kPF) {
            float4 w[kPF];
    #pragma unroll
            for (int u = 0; u < kPF; ++u) w[u] = wrest(rb + u);
            for (int u = 0; u < kPF; ++u) {
                const int32_t r = rb + u;
                if (r >= r1) break;
                float4 acc = zero4;
                for (int32_t q = H.run_start[r]; q < H.run_start[r + 1]; ++q) {
                    const int64_t a = H.perm[q] % H.n_last;
                    add4(acc, H.cls_start ? class_factor(wl, A.K_pad, H.cls_members, H.cls_start[a], H.cls_start[a + 1])
                                          : ld4(wl + a * A.K_pad));
                }
                fma4(bacc, w[u], acc);
                const int32_t nk = r + 1 < r1 ? H.run_bin[r + 1] : -1;
                if (nk != cur_key) {
                    flush(cur_key, bacc);
                    bacc = zero4;
                    cur_key = nk;
                }
            }
        }
    }
}

// Finish H[k, b]: for every part, the key (part, b) is either empty, summed
// whole by the single chunk that holds it (direct row), or cut by chunk
// boundaries and summed from the partials of the chunks overlapping it (in
// chunk order); parts are added in order.  Two tiles of 128 densities x 8
// bins per 256 threads: warp w takes bin w, each lane four consecutive
// densities of each tile (the two tiles' loads in flight together), so the
// direct rows and partials are read as coalesced 512-byte rows; the tiles go
// to the [K][B] output through shared memory (8 consecutive bins, one
// 32-byte sector, per row).
constexpr int kFinK = 128, kFinB = 8;
constexpr int kFinNK = 2;     // density tiles per CTA: their loads are in flight together
constexpr int kFinMaxP = 96;  // >= parts of any axis: ceil(32767 / kMaxPartRows) = 84
__device__ __forceinline__ void hist_finish_tiles(const HistArgs &A, int64_t kt0, int bt) {
    __shared__ float tile[kFinNK][kFinB][kFinK + 1];
    __shared__ int2 s_cc[kFinMaxP][kFinB];
    const LayoutArgs &H = A.sel[0] ? A.L1 : A.L0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int P = A.fold->P[A.sel[0] ? 1 : 0];
    const bool recs = !A.points_only && A.sel[1] == 2;  // record stream: every non-empty group wrote its rows
    // the chunk range of every (part, bin) key of the bin tile; on the record
    // stream that of the part's group of the bin
    for (int e = threadIdx.x; e < P * kFinB; e += blockDim.x) {
        const int p = e / kFinB, bb = e - p * kFinB, b = bt * kFinB + bb;
        s_cc[p][bb] = b >= A.B ? make_int2(-1, -1)
                      : recs   ? H.rec_gch[p * A.GB + b / kRecBinsH]
                               : H.key_chunks[p * A.B + b];
    }
    __syncthreads();
    const int b = bt * kFinB + warp;
    int64_t kq[kFinNK];  // this lane's first density in each tile
    bool live[kFinNK];   // the tile holds densities
#pragma unroll
    for (int t = 0; t < kFinNK; ++t) {
        live[t] = (kt0 + t) * kFinK < A.K;
        kq[t] = (kt0 + t) * kFinK + 4 * lane;
    }
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 total[kFinNK];
#pragma unroll
    for (int t = 0; t < kFinNK; ++t) total[t] = zero;
    if (b < A.B) {
        // four parts at a time: their direct rows (of every tile) in flight
        // together, then added in part order (cut keys from their chunks'
        // partials)
        for (int p0 = 0; p0 < P; p0 += 4) {
            float4 v[4][kFinNK];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int p = p0 + q;
                const int2 cc = p < P ? s_cc[p][warp] : make_int2(-1, -1);
                const float *row = A.direct + ((int64_t)p * A.B + b) * A.K_pad;
#pragma unroll
                for (int t = 0; t < kFinNK; ++t)
                    v[q][t] = (cc.x >= 0 && cc.x == cc.y && live[t]) ? *reinterpret_cast<const float4 *>(row + kq[t])
                                                                     : zero;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int p = p0 + q;
                if (p >= P) break;
                const int2 cc = s_cc[p][warp];
                if (cc.x < 0) continue;
                if (cc.x == cc.y) {
#pragma unroll
                    for (int t = 0; t < kFinNK; ++t) add4(total[t], v[q][t]);
                    continue;
                }
                // the partials of the chunks holding the key, two chunks'
                // loads (of every tile) in flight together, added in chunk order
                float4 sum[kFinNK];
#pragma unroll
                for (int t = 0; t < kFinNK; ++t) sum[t] = zero;
                const int32_t gr = p * A.GB + b / kRecBinsH, key = p * A.B + b;
                for (int c0 = cc.x; c0 <= cc.y; c0 += 2) {
                    float4 pv[2][kFinNK];
                    bool use[2];
#pragma unroll
                    for (int q2 = 0; q2 < 2; ++q2) {
                        const int c = c0 + q2;
                        use[q2] = false;
#pragma unroll
                        for (int t = 0; t < kFinNK; ++t) pv[q2][t] = zero;
                        if (c > cc.y) continue;
                        const float *row;
                        if (recs) {
                            if (H.rec_chunk[c] >= H.rec_chunk[c + 1]) continue;
                            const int side = H.rec_chunk_grp[2 * c] == gr ? 0 : 1;
                            row = A.part + (((int64_t)c * 2 + side) * kRecBinsH + b % kRecBinsH) * A.K_pad;
                        } else {
                            if (H.chunk_pt[c] >= H.chunk_pt[c + 1]) continue;
                            const int side = H.chunk_bin[2 * c] == key ? 0 : 1;
                            row = A.part + ((int64_t)c * 2 + side) * A.K_pad;
                        }
#pragma unroll
                        for (int t = 0; t < kFinNK; ++t)
                            if (live[t]) pv[q2][t] = *reinterpret_cast<const float4 *>(row + kq[t]);
                        use[q2] = true;
                    }
#pragma unroll
                    for (int q2 = 0; q2 < 2; ++q2)
                        if (use[q2])
#pragma unroll
                            for (int t = 0; t < kFinNK; ++t) add4(sum[t], pv[q2][t]);
                }
#pragma unroll
                for (int t = 0; t < kFinNK; ++t) add4(total[t], sum[t]);
            }
        }
    }
#pragma unroll
    for (int t = 0; t < kFinNK; ++t) {
        float *row = tile[t][warp] + 4 * lane;
        row[0] = total[t].x;
        row[1] = total[t].y;
        row[2] = total[t].z;
        row[3] = total[t].w;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kFinNK * kFinK * kFinB; e += blockDim.x) {
        const int t = e / (kFinK * kFinB), r = e - t * (kFinK * kFinB);
        const int kk = r / kFinB, bb = r - kk * kFinB;
        const int64_t kr = (kt0 + t) * kFinK + kk;
        const int bo = bt * kFinB + bb;
        if (kr < A.K && bo < A.B) A.hist[kr * A.B + bo] = tile[t][bb][kk];
    }
}

__global__ void __launch_bounds__(256, 3) k_hist_finish(const __grid_constant__ HistArgs A) {
    pdl_trigger();
    pdl_wait();
    hist_finish_tiles(A, (int64_t)blockIdx.x * kFinNK, blockIdx.y);
}

// Batched finish: items[i] = (instance, density tile, bin tile).
__global__ void __launch_bounds__(256, 3) k_hist_finish_batched(const HistArgs *__restrict__ insts, const int4 *__restrict__ items) {
    const int4 it = items[blockIdx.x];
    hist_finish_tiles(insts[it.x], (int64_t)it.y * kFinNK, it.z);
}

// ---- posterior sums ------------------------------------------------------------
// One point-stream pass for everything the posterior means need: per bin the
// sums of W and of W x_d for every axis d.  A CTA takes 64 densities: a tile
// row holds, per lane, the factors of its two densities and the same times the
// gathered axis' coordinate (a merged row: summed over its members), so one
// 16-byte gather per point gives both; a run's two sums S0 = sum w and S1 =
// sum w x are multiplied at its end by the rest axes' factors (H += f S0, the
// gathered axis' sum += f S1, a rest axis' sum += f_x S0 with f_x its factor
// times its coordinate).  Separate passes per axis gathered every point once for each
// (three times on 2-D grids) and re-read the weighted tables: 1024 x 1024
// points, K = 8192: 4.88 ms, 1.14 with equal slices merged, 0.57 in one pass.
struct PostArgs {
    HistArgs h;              // the histogram's arguments (tables, layout, scratch sizes)
    const float *xs;         // coordinates of every axis, axis d from off[d]
    const float *fx;         // rest factors times coordinate (merged), axis d at off[d] rows
    float *part, *direct;    // [cut row or key][1 + ndim][kb] of the densities k0 .. k0 + kb - 1
    int64_t k0, kb;
    float *hist, *post;      // [K][B] (or null), [K][B][ndim]
};
constexpr int kPostKT = 64;
// The sums of a walk, (1 + ndim) floats per cut row or key and density, are kept for
// as many densities as this many bytes hold (at least 128); the walk and its finish
// run once per such block (1024 x 1024 points, 256 bins: 25 KB per density, one
// block up to 21000 densities; 6 parts of 5000 bins: 0.37 MB, blocks of 1408).
constexpr size_t kPostSums = (size_t)512 << 20;
__device__ __forceinline__ float2 ld2(const float *q) { return *reinterpret_cast<const float2 *>(q); }

// Rest factors f_x (and, of folded axes, the merged f into ftab_fold).
__global__ void __launch_bounds__(128) k_post_tables(const __grid_constant__ PostArgs A, float *__restrict__ fx,
                                                     float *__restrict__ f_merged, int *__restrict__ ctr) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *ctr = 0;
    const HistArgs &h = A.h;
    const int64_t K_pad = h.K_pad, kb = (K_pad + 511) / 512;
    const int gathered = h.ndim == 2 && h.sel[0] ? 0 : h.ndim - 1;
    for (int d = 0; d < h.ndim; ++d) {
        if (d == gathered) continue;
        const bool folded = h.fold->folded[d] != 0;
        const int64_t rows = h.fold->n[d], off = h.off[d];
        for (int64_t u = blockIdx.x; u < rows * kb; u += gridDim.x) {
            const int64_t c = u / kb, k = (u - c * kb) * 512 + 4 * threadIdx.x;
            if (k >= K_pad) continue;
            const int32_t *st = h.fold_start + off + d + c, *mem = h.fold_members + off;
            const int32_t m0 = folded ? st[0] : 0, m1 = folded ? st[1] : 1;
            PairSum4 f, x;
            f.clear();
            x.clear();
            for (int32_t m = m0; m < m1; ++m) {
                const int64_t a = folded ? mem[m] & (kFoldLast - 1) : c;
                const float4 v = ld4(h.ftab + (off + a) * K_pad + k);
                const float xa = A.xs[off + a];
                f.add(v);
                x.add(make_float4(v.x * xa, v.y * xa, v.z * xa, v.w * xa));
            }
            *reinterpret_cast<float4 *>(fx + (off + c) * K_pad + k) = x.value();
            if (folded) *reinterpret_cast<float4 *>(f_merged + (h.foff[d] + c) * K_pad + k) = f.value();
        }
    }
}

// Midpoint coordinates of every axis, rounded once to FP32.
struct AxisGeom {
    int ndim;
    int64_t n[3];
    double lo[3], h[3];
};
__global__ void k_axis_coords(AxisGeom G, float *__restrict__ xs) {
    int64_t off = 0;
    for (int d = 0; d < G.ndim; ++d) {
        for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < G.n[d]; a += (int64_t)gridDim.x * blockDim.x)
            xs[off + a] = (float)__dadd_rn(G.lo[d], __dmul_rn((double)a + 0.5, G.h[d]));
        off += G.n[d];
    }
}

// Rest factors of one run for a lane's two densities: f, and f with one rest
// axis' factor weighted by its coordinate.
template <int NF>
struct RunFactors {
    float2 f, fx[NF];
};

// AHEAD: how many runs ahead a run-end word's rest code points (the layout's).
template <int NF, int AHEAD>
__global__ void __launch_bounds__(kHistWarps * 32, 1)
    k_post_walk(const __grid_constant__ PostArgs A, int64_t tile_rows, int nkt, int *__restrict__ next_item) {
    constexpr int NO = 2 + NF;  // sums per key: W, W x of the gathered axis, of the rest axes
    extern __shared__ __align__(128) uint8_t sm[];
    __shared__ LayoutArgs H;
    __shared__ float s_iz[kPostKT];
    __shared__ int abort, next_chunk, s_item, s_G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t K_pad = A.h.K_pad;
    const int C = A.h.C;
    int *dstatus = A.h.dstatus;
    if (threadIdx.x == 0) {
        abort = 0;
        H = pick(A.h);
    }
    hist_init_mbar(sm, tile_rows, kHistWarps);
    uint64_t *mbar = hist_mbar(sm, tile_rows, kHistWarps);
    float *ws = reinterpret_cast<float *>(sm);
    uint32_t *win = reinterpret_cast<uint32_t *>(sm + hist_tile_bytes(tile_rows) + (size_t)warp * hist_warp_bytes());
    __syncthreads();
    const int P = H.P;
    if (warp == 0) {
        const int G = hist_split(A.h.fold->N / P, C, (int64_t)nkt * P, H.part_rows, kHistWarps, hist_rate(0), gridDim.x);
        if (lane == 0) s_G = G;
    }
    uint32_t wseq = 0;
    for (;;) {
        __syncthreads();  // the previous item's readers of the tile and of s_item are done
        if (threadIdx.x == 0) {
            s_item = atomicAdd(next_item, 1);
            next_chunk = 0;
        }
        __syncthreads();
        const int G = s_G, it = s_item;
        if (it >= (int64_t)nkt * P * G || abort) return;  // uniform
        const int cg = it % G, pk = it / G, p = pk % P;
        const int64_t k0 = A.k0 + (int64_t)(pk / P) * kPostKT, k = k0 + 2 * lane;
        if (threadIdx.x < kPostKT) s_iz[threadIdx.x] = inv_z(A.h, k0 + threadIdx.x);
        __syncthreads();
        const int64_t row0 = (int64_t)p * H.part_rows;
        const int32_t nrows = (int32_t)min(H.part_rows, H.n_last - row0);
        {
            // this warp's rows: (w, w', w x, w' x) of the lane's two densities, class members summed
            const float2 iz = make_float2(s_iz[2 * lane], s_iz[2 * lane + 1]);
            const float *xs = A.xs + A.h.off[H.ax_last], *src = H.g_last + k;
            const int32_t a0 = nrows * warp / kHistWarps, a1 = nrows * (warp + 1) / kHistWarps;
            const int32_t *members = H.cls_start ? H.cls_members : nullptr;
            const int32_t m0 = members ? H.cls_start[row0 + a0] : (int32_t)row0 + a0;
            const int32_t m1 = members ? H.cls_start[row0 + a1] : (int32_t)row0 + a1;
            float *dst = ws + (int64_t)a0 * kKT + 4 * lane;
            PairSum4 c;
            c.clear();
            for (int32_t m = m0; m < m1; m += 8) {
                float2 v[8];
                float x[8];
                int32_t r[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    r[u] = m + u < m1 ? (members ? members[m + u] : (m + u) | kFoldLast) : 0;
                    const int64_t a = r[u] & (kFoldLast - 1);
                    v[u] = m + u < m1 ? ld2(src + a * K_pad) : make_float2(0.f, 0.f);
                    x[u] = m + u < m1 ? xs[a] : 0.f;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    c.add(make_float4(v[u].x, v[u].y, v[u].x * x[u], v[u].y * x[u]));
                    if (r[u] & kFoldLast) {
                        const float4 t = c.value();
                        *reinterpret_cast<float4 *>(dst) = make_float4(t.x * iz.x, t.y * iz.y, t.z * iz.x, t.w * iz.y);
                        dst += kKT;
                        c.clear();
                    }
                }
            }
            if (threadIdx.x < kKT) ws[(int64_t)nrows * kKT + threadIdx.x] = 0.f;
        }
        __syncthreads();

        const float *g0k = H.g0 + k, *x0k = A.fx + A.h.off[H.ax0] * K_pad + k;
        const float *g1k = NF == 2 ? H.g1 + k : nullptr, *x1k = NF == 2 ? A.fx + A.h.off[H.ax1] * K_pad + k : nullptr;
        auto factors = [&](uint32_t a0, uint32_t a1) -> RunFactors<NF> {
            // (debug build: rows outside the factor tables are recorded and read as row 0)
            if (!VUP_DBG_IN(a0, H.n0, dstatus)) a0 = 0;
            if (NF == 2 && !VUP_DBG_IN(a1, H.n1, dstatus)) a1 = 0;
            RunFactors<NF> R;
            R.f = ld2(g0k + (int64_t)a0 * K_pad);
            R.fx[0] = ld2(x0k + (int64_t)a0 * K_pad);
            if constexpr (NF == 2) {
                const float2 q = ld2(g1k + (int64_t)a1 * K_pad), qx = ld2(x1k + (int64_t)a1 * K_pad);
                R.fx[1] = make_float2(R.f.x * qx.x, R.f.y * qx.y);
                R.fx[0] = make_float2(R.fx[0].x * q.x, R.fx[0].y * q.y);
                R.f = make_float2(R.f.x * q.x, R.f.y * q.y);
            }
            return R;
        };
        auto coded = [&](uint32_t u) -> RunFactors<NF> {
            const uint32_t lo = u & 0x1ffu, hi = (u >> 18) & 0xfffu;
            return NF == 2 ? factors(lo, hi) : factors(lo | (hi << 9), 0u);
        };
        const uint32_t wsl = smem_u32(ws) + lane * 16;
        const uint32_t null_word = (uint32_t)nrows << kRowShift;  // zero row, no flags
        auto gather = [&](uint32_t word) -> float4 {
            uint32_t o = word & kOffMask;
            if (!VUP_DBG_IN(o >> kRowShift, nrows + 1, dstatus)) o = null_word;
            float4 v;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                         : "r"(wsl + o));
            return v;
        };
        const int c_end = (int)((int64_t)(cg + 1) * C / G);
        for (;;) {
            int ci = 0;
            if (lane == 0) ci = atomicAdd(&next_chunk, 1);
            ci = __shfl_sync(0xffffffffu, ci, 0) + (int)((int64_t)cg * C / G);
            if (ci >= c_end) break;
            const int c = p * C + ci;
            const int32_t p0 = H.chunk_pt[c], p1 = H.chunk_pt[c + 1];
            if (p0 >= p1) continue;
            const int32_t r0 = H.chunk_run[c], r1 = H.chunk_run[c + 1];
            // keys cut by the chunk bounds can only be its first and last key
            const int32_t first_key = H.chunk_bin[2 * c], last_key = H.chunk_bin[2 * c + 1];
            const bool sh_first = H.koff[first_key] < p0 || H.koff[first_key + 1] > p1;
            const bool sh_last = H.koff[last_key] < p0 || H.koff[last_key + 1] > p1;
            const int32_t wb0 = p0 & ~(kWin - 1);
            if (lane == 0) {
                const int b0 = wseq & 1;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // earlier reads of both buffers
                bulk_copy(win + b0 * kWin, H.hpt + wb0, kWin * 4, &mbar[b0]);
                if (wb0 + kWin < p1) bulk_copy(win + (b0 ^ 1) * kWin, H.hpt + wb0 + kWin, kWin * 4, &mbar[b0 ^ 1]);
            }
            __syncwarp();
            RunFactors<NF> pf[AHEAD];  // of the current run and the next ones
#pragma unroll
            for (int q = 0; q < AHEAD; ++q) {
                const int32_t rest = r0 + q < r1 ? H.run_rest[r0 + q] : 0;
                const int32_t a0 = NF == 2 ? rest / (int32_t)H.n1 : rest;
                pf[q] = factors((uint32_t)a0, NF == 2 ? (uint32_t)(rest - a0 * (int32_t)H.n1) : 0u);
            }
            int32_t r = r0, cur_key = first_key;
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f);  // S0, S1 of the current run
            float2 acc[NO];
#pragma unroll
            for (int o = 0; o < NO; ++o) acc[o] = make_float2(0.f, 0.f);
            auto flush = [&]() {
                const bool first = cur_key == first_key;
                const bool shared = first ? sh_first : (cur_key == last_key && sh_last);
                float *dst = (shared ? A.part + ((int64_t)c * 2 + (first ? 0 : 1)) * NO * A.kb
                                     : A.direct + (int64_t)cur_key * NO * A.kb) + (k - A.k0);
                if (VUP_DBG_IN(cur_key, (int64_t)P * A.h.B, dstatus))
#pragma unroll
                    for (int o = 0; o < NO; ++o) *reinterpret_cast<float2 *>(dst + o * A.kb) = acc[o];
#pragma unroll
                for (int o = 0; o < NO; ++o) acc[o] = make_float2(0.f, 0.f);
            };
            auto fold_run = [&]() {
                acc[0].x = fmaf(pf[0].f.x, s.x, acc[0].x);
                acc[0].y = fmaf(pf[0].f.y, s.y, acc[0].y);
                acc[1].x = fmaf(pf[0].f.x, s.z, acc[1].x);
                acc[1].y = fmaf(pf[0].f.y, s.w, acc[1].y);
#pragma unroll
                for (int o = 0; o < NF; ++o) {
                    acc[2 + o].x = fmaf(pf[0].fx[o].x, s.x, acc[2 + o].x);
                    acc[2 + o].y = fmaf(pf[0].fx[o].y, s.y, acc[2 + o].y);
                }
                s = make_float4(0.f, 0.f, 0.f, 0.f);
            };
            auto run_end = [&](uint32_t u) {
                fold_run();
                if (u & kBinEnd) {
                    flush();
                    cur_key = r + 1 < r1 ? H.run_bin[r + 1] : -1;
                }
#pragma unroll
                for (int q = 0; q + 1 < AHEAD; ++q) pf[q] = pf[q + 1];
                pf[AHEAD - 1] = coded(u);
                ++r;
            };
            auto group = [&](const uint4 v) {
                const float4 a0 = gather(v.x), a1 = gather(v.y), a2 = gather(v.z), a3 = gather(v.w);
                if (((v.x | v.y | v.z | v.w) & kFlags) == 0) {
                    add4(s, a0);
                    add4(s, a1);
                    add4(s, a2);
                    add4(s, a3);
                } else {
                    add4(s, a0);
                    if (v.x & kFlags) run_end(v.x);
                    add4(s, a1);
                    if (v.y & kFlags) run_end(v.y);
                    add4(s, a2);
                    if (v.z & kFlags) run_end(v.z);
                    add4(s, a3);
                    if (v.w & kFlags) run_end(v.w);
                }
            };
            for (int32_t wbase = wb0; wbase < p1; wbase += kWin, ++wseq) {
                const int b = wseq & 1;
                for (uint32_t i = 0; !mbar_try_wait(&mbar[b], (wseq >> 1) & 1); ++i) {
                    if (i > kSpin || *(volatile int *)&abort) {  // a staged copy never landed: record and stop
                        *(volatile int *)&abort = 1;
                        atomicCAS(dstatus, 0, VUP_DSTAT_TIMEOUT);
                        break;
                    }
                }
                if (*(volatile int *)&abort) break;
                const uint32_t *wv = win + b * kWin;
                const int lo = (p0 > wbase ? p0 : wbase) - wbase;
                const int hi = (p1 < wbase + kWin ? p1 : wbase + kWin) - wbase;
                for (int pa = lo & ~3; pa < hi; pa += 4) {
                    uint4 v = *reinterpret_cast<const uint4 *>(wv + pa);
                    if (pa < lo || pa + 4 > hi) {  // cut by the chunk bounds: foreign points read the zero row
                        if (pa + 0 < lo || pa + 0 >= hi) v.x = null_word;
                        if (pa + 1 < lo || pa + 1 >= hi) v.y = null_word;
                        if (pa + 2 < lo || pa + 2 >= hi) v.z = null_word;
                        if (pa + 3 < lo || pa + 3 >= hi) v.w = null_word;
                    }
                    group(v);
                }
                __syncwarp();
                if (lane == 0 && wbase + 2 * kWin < p1) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    bulk_copy(win + b * kWin, H.hpt + wbase + 2 * kWin, kWin * 4, &mbar[b]);
                }
            }
            if (*(volatile int *)&abort) break;
            if (cur_key >= 0) flush();  // (its last run ended with the chunk)
        }
    }
}

// H and the posterior means from the walk's sums (parts in order, cut keys from
// their chunks' partials in chunk order, as the histogram's finish): 128
// densities x 8 bins per CTA, a warp per bin.
template <int NO>
__global__ void __launch_bounds__(256) k_post_finish(const __grid_constant__ PostArgs A) {
    __shared__ float tile[NO][8][128 + 1];
    const HistArgs &h = A.h;
    const LayoutArgs &H = h.sel[0] ? h.L1 : h.L0;
    constexpr int nd = NO - 1;
    const int P = h.fold->P[h.sel[0] ? 1 : 0];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = blockIdx.y * 8 + warp;
    const int64_t k0 = A.k0 + (int64_t)blockIdx.x * 128, k = k0 + 4 * lane;
    float4 t[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) t[o] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t kb = A.kb;
    const float *direct = A.direct + (k - A.k0), *part = A.part + (k - A.k0);
    if (b < h.B)
        for (int p = 0; p < P; ++p) {
            const int32_t key = p * h.B + b;
            const int2 cc = H.key_chunks[key];
            if (cc.x < 0) continue;
            if (cc.x == cc.y) {
                const float *row = direct + (int64_t)key * NO * kb;
#pragma unroll
                for (int o = 0; o < NO; ++o) add4(t[o], ld4(row + o * kb));
                continue;
            }
            // a key cut by many chunks (few bins) is a chain of dependent loads: four
            // chunks at a time, added in chunk order (an empty chunk's row is not; 1495 x
            // 1786 points, 20 bins, K = 569: 84 us one at a time, 64 so)
            for (int c0 = cc.x; c0 <= cc.y; c0 += 4) {
                float4 v[4][NO];
                bool live[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int c = min(c0 + u, cc.y);
                    const int side = H.chunk_bin[2 * c] == key ? 0 : 1;
                    live[u] = c0 + u <= cc.y && H.chunk_pt[c] < H.chunk_pt[c + 1];
                    const float *row = part + ((int64_t)c * 2 + side) * NO * kb;
#pragma unroll
                    for (int o = 0; o < NO; ++o) v[u][o] = ld4(row + o * kb);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (live[u])
#pragma unroll
                        for (int o = 0; o < NO; ++o) add4(t[o], v[u][o]);
            }
        }
#pragma unroll
    for (int o = 0; o < NO; ++o) {
        float *q = tile[o][warp] + 4 * lane;
        q[0] = t[o].x;
        q[1] = t[o].y;
        q[2] = t[o].z;
        q[3] = t[o].w;
    }
    __syncthreads();
    // sum o > 0 belongs to an axis: 1 the gathered one, then the rest axes
    const int bb = threadIdx.x & 7;
    const int64_t bo = (int64_t)blockIdx.y * 8 + bb;
    for (int kk = threadIdx.x >> 3; kk < 128; kk += 32) {
        if (k0 + kk >= h.K || bo >= h.B) continue;
        const int64_t e = (k0 + kk) * h.B + bo;
        const float m = tile[0][bb][kk];
        if (A.hist) A.hist[e] = m;
        for (int d = 0; d < nd; ++d) {
            const int o = d == H.ax_last ? 1 : (d == H.ax0 ? 2 : 3);
            A.post[e * nd + d] = m > 0.f ? tile[o][bb][kk] / m : 0.f;
        }
    }
}

}  // namespace

// Chunks per part: groups of kGroupChunks chunks, as many groups (1..16) as
// give chunks of about 1536 points when the gathered axis is cut into P
// parts.  A launch then picks how many groups one CTA serves.
int vup_hist_chunks_for(int64_t N, int P) {
    const double per_group = (double)kGroupChunks * 1536.0;
    int64_t S = (int64_t)llround((double)N / ((double)std::max(P, 1) * per_group));
    S = std::max<int64_t>(1, std::min<int64_t>(16, S));
    return (int)(S * kGroupChunks);
}

// Record chunks per part: a quarter of the point chunks (records are several
// times fewer than intervals), in whole groups of kGroupChunks.
int vup_hist_rec_chunks_for(int n_chunks) {
    return kGroupChunks * std::max(1, n_chunks / kGroupChunks / 4);
}

// Parts of a gathered axis of n_last rows (one 64-density tile each) for a
// bin count; one part when the (part, bin) key space would exceed the sort.
int vup_hist_parts_for(int64_t n_last, int n_bins) {
    int P = (int)ceil_div64(n_last, kMaxPartRows);
    if ((int64_t)P * n_bins > 32768) P = 1;
    return P;
}

// Arguments of the histogram kernels for one grid; `rows` receives the
// largest shared-memory tile (rows of one part of a gathered axis).
static HistArgs hist_args_for(vup_grid g, int64_t K, float *hist, int64_t &rows, int &P_max,
                              const float *ftab = nullptr) {
    const int64_t K_pad = ceil_div64(K, 128) * 128;
    const int nd = g->ndim;
    const float *ft = ftab ? ftab : (const float *)g->ftab.p;
    auto tab = [&](int axis) {
        int64_t off = 0;
        for (int q = 0; q < axis; ++q) off += g->n[q] * K_pad;
        return ft + off;
    };
    HistArgs A{};
    A.sets = 1;
    rows = 0;
    P_max = 1;
    for (int l = 0; l < 2; ++l) {
        const auto &HL = g->hl[l < g->n_layouts ? l : 0];
        LayoutArgs &La = l == 0 ? A.L0 : A.L1;
        La.hpt = HL.hpt;
        La.perm = HL.perm;
        La.run_start = HL.run_start;
        La.run_rest = HL.run_rest;
        La.run_bin = HL.run_bin;
        La.chunk_pt = HL.chunk_pt;
        La.chunk_run = HL.chunk_run;
        La.chunk_bin = HL.chunk_bin;
        La.koff = HL.koff;
        La.key_chunks = HL.key_chunks;
        La.ipt = HL.ipt;
        La.iv_rest = HL.iv_rest;
        La.chunk_iv = HL.chunk_iv;
        La.n_rec = HL.n_rec;
        La.n_iv = HL.n_iv;
        La.rec = (const uint4 *)g->hl[0].rec.p;  // the built layout's arrays
        La.rec_rest = (const int32_t *)g->hl[0].rec_rest.p;
        La.rec_goff = (const int32_t *)g->hl[0].rec_goff.p;
        La.rec_gch = (const int2 *)g->hl[0].rec_gch.p;
        La.rec_chunk = g->hl[0].rec_chunk;
        La.rec_chunk_grp = g->hl[0].rec_chunk_grp;
        La.g_last = tab(HL.last_axis);
        if (nd == 3) {
            La.g0 = tab(0);
            La.g1 = tab(1);
            La.n1 = g->n[1];
            La.n0 = g->n[0];
        } else {
            La.g0 = tab(HL.last_axis == 1 ? 0 : 1);
            La.g1 = nullptr;
            La.n1 = 1;
            La.n0 = g->n[HL.last_axis == 1 ? 0 : 1];
        }
        La.n_last = HL.n_last;
        La.part_rows = HL.part_rows;
        La.P = HL.P;
        La.ax_last = HL.last_axis;
        La.ax0 = nd == 3 ? 0 : 1 - HL.last_axis;
        La.ax1 = nd == 3 ? 1 : La.ax0;
        rows = std::max(rows, HL.part_rows);
        P_max = std::max(P_max, HL.P);
    }
    A.fold = g->fold;
    A.ftab = ft;
    A.ftab_fold = (const float *)g->ftab_fold.p;
    A.fold_start = g->fold_start;
    A.fold_members = g->fold_members;
    for (int d = 0; d < nd; ++d) {
        A.off[d] = d ? A.off[d - 1] + g->n[d - 1] : 0;
        A.foff[d] = fold_row(nd, g->n, d);
    }
    A.sel = g->hist_sel;
    A.GB = (int)ceil_div64(g->B, kRecBinsH);
    A.C_rec = g->n_chunks_rec;
    A.ds = (const DensStats *)g->dstats.p;
    A.ndim = nd;
    A.K = K;
    A.K_pad = K_pad;
    A.B = g->B;
    A.C = g->n_chunks;
    A.hist = hist;
    A.part = (float *)g->hist_part.p;
    A.direct = (float *)g->hist_direct.p;
    A.dstatus = g->dstatus;
    return A;
}

// Merged factor tables (FoldGeom) of the folded rest axes of the chosen layout
// (the gathered axis' classes are summed where its tiles are made).  HBM
// bound: it reads a folded axis' factors once and writes 5/8 of that at most;
// a grid-stride walk over (axis, class, 512 densities), so that a grid without
// folded axes costs an empty launch.
struct FoldTabArgs {
    const FoldGeom *fold;
    const int32_t *sel;
    const int32_t *start, *members;
    const float *ftab;
    float *out;
    int64_t n[3], K_pad;
    int ndim;
    int *ctr;  // the walks' item counters, zeroed here (or null)
};
__device__ __forceinline__ void fold_table_rows(const FoldTabArgs &T, int64_t first, int64_t step) {
    const int64_t kb = (T.K_pad + 511) / 512;
    const int gathered = T.ndim == 2 && T.sel[0] ? 0 : T.ndim - 1;
    int64_t off = 0;
    for (int d = 0; d < T.ndim; ++d) {
        if (T.fold->folded[d] && d != gathered) {
            const int64_t rows = T.fold->n[d], foff = fold_row(T.ndim, T.n, d);
            for (int64_t u = first; u < rows * kb; u += step) {
                const int64_t c = u / kb, k = (u - c * kb) * 512 + 4 * threadIdx.x;
                if (k >= T.K_pad) continue;
                const int32_t *st = T.start + off + d + c;
                *reinterpret_cast<float4 *>(T.out + (foff + c) * T.K_pad + k) =
                    class_factor(T.ftab + off * T.K_pad + k, T.K_pad, T.members + off, st[0], st[1]);
            }
        }
        off += T.n[d];
    }
}
__global__ void __launch_bounds__(128) k_fold_tables(const __grid_constant__ FoldTabArgs T) {
    if (blockIdx.x == 0 && threadIdx.x < 3) T.ctr[threadIdx.x] = 0;
    if (!T.fold->any) return;
    fold_table_rows(T, blockIdx.x, gridDim.x);
}
// Batched form: block y serves the y-th instance with a histogram.
__global__ void __launch_bounds__(128) k_fold_tables_batched(const FoldTabArgs *__restrict__ jobs) {
    const FoldTabArgs &T = jobs[blockIdx.y];
    if (!T.fold->any) return;
    fold_table_rows(T, blockIdx.x, gridDim.x);
}

static FoldTabArgs fold_tab_args(vup_grid g, int64_t K) {
    FoldTabArgs T{};
    T.fold = g->fold;
    T.sel = g->hist_sel;
    T.start = g->fold_start;
    T.members = g->fold_members;
    T.ftab = (const float *)g->ftab.p;
    T.out = (float *)g->ftab_fold.p;
    T.K_pad = ceil_div64(K, 128) * 128;
    T.ndim = g->ndim;
    for (int d = 0; d < 3; ++d) T.n[d] = d < g->ndim ? g->n[d] : 0;
    return T;
}

vup_status vup_reserve_fold(vup_grid g, int64_t K) {
    const int64_t rows = fold_row(g->ndim, g->n, g->ndim);
    return devbuf_reserve(g->ftab_fold, sizeof(float) * (size_t)rows * (size_t)(ceil_div64(K, 128) * 128));
}

vup_status vup_fold_tables(vup_grid g, int64_t K, cudaStream_t s, const float *ftab) {
    FoldTabArgs T = fold_tab_args(g, K);
    if (ftab) T.ftab = ftab;
    T.ctr = g->hist_sel + kHistCtr;
    const int64_t rows = fold_row(g->ndim, g->n, g->ndim);
    const int64_t blocks = std::min<int64_t>(rows * ceil_div64(T.K_pad, 512), (int64_t)vup_num_sms() * 16);
    VUP_PROF("hist_fold_tables", s, 1);
    k_fold_tables<<<(unsigned)blocks, 128, 0, s>>>(T);
    VUP_CHECK_LAUNCH();
    return VUP_OK;
}

bool vup_hist_rest_staged(const vup_grid_s *g) {
    if (g->ndim != 3 || g->hl[0].last_axis != 2 || g->n[0] > 512 || g->n[1] > 4096) return false;
    const size_t rest_bytes = (size_t)(g->n[0] + g->n[1]) * kKT * sizeof(float);
    return hist_smem_bytes(g->hl[0].part_rows, hist_warps(4)) + rest_bytes <= kSmemMost;
}

vup_status vup_hist_fused(vup_grid g, int64_t K, float *hist, cudaStream_t s, const float *ftab,
                          bool points_only, cudaEvent_t keys_ready, bool tables_ready) {
    const int nd = g->ndim;
    int64_t rows;
    int P_max;
    HistArgs A = hist_args_for(g, K, hist, rows, P_max, ftab);
    const size_t smem = hist_smem_bytes(rows);
    // run-end words encode the rest index in 21 bits (3-D: a0 < 512, a1 < 4096)
    const bool coded = nd == 2 || (g->n[0] <= 512 && g->n[1] <= 4096);
    const bool in_smem = smem <= kSmemMost && coded;
    // 3-D point stream: both rest-axis factor tiles in shared memory when they fit beside the tile
    const size_t rest_bytes = nd == 3 ? (size_t)(g->n[0] + g->n[1]) * kKT * sizeof(float) : 0;
    const bool rest_staged = in_smem && vup_hist_rest_staged(g);
    // the global-memory fallback walks points whatever the device chose
    points_only = points_only || !in_smem;
    A.points_only = points_only ? 1 : 0;
    const int nkt = (int)ceil_div64(K, kKT), sms = vup_num_sms();
    if (!tables_ready) {
        vup_status st = vup_fold_tables(g, K, s, ftab);
        if (st != VUP_OK) return st;
    }
    {
        VUP_PROF("hist_segmented", s, in_smem && !points_only ? 3 : 1);
        if (in_smem) {
            // (at most one item per part, density tile and chunk)
            const int64_t most = (int64_t)P_max * nkt * std::max(A.C, A.C_rec);
            const unsigned ctas = (unsigned)std::min<int64_t>(sms, most);
            auto launch = [&](auto kern, int mode) -> vup_status {
                const size_t sm_bytes =
                    hist_smem_bytes(rows, hist_warps(mode)) + (hist_staged(mode) ? rest_bytes : 0);
                VUP_CHECK_CUDA(smem_allow(kern));
                VUP_CHECK_CUDA(launch_pdl(kern, dim3(ctas), dim3(hist_warps(mode) * 32), sm_bytes, s, A, rows, nkt,
                                          (int *)g->hist_sel + kHistCtr + hist_stream_of(mode)));
                return VUP_OK;
            };
            vup_status st;
            if (!points_only) {  // the record stream first: it needs no key sort
                // 16 warps when the rest-factor rows (of either layout) fit well in L2
                int64_t rest_rows = 0;
                for (int l = 0; l < g->n_layouts; ++l) rest_rows = std::max(rest_rows, g->N / g->hl[l].n_last);
                if (nd == 3) rest_rows = g->n[0] + g->n[1];
                const bool l2_rest = (double)rest_rows * A.K_pad * 4.0 <= 96.0 * 1024 * 1024;
                if (rest_staged) st = launch(k_hist_smem<2, 5>, 5);
                else if (l2_rest) st = nd == 3 ? launch(k_hist_smem<2, 3>, 3) : launch(k_hist_smem<1, 3>, 3);
                else st = nd == 3 ? launch(k_hist_smem<2, 2>, 2) : launch(k_hist_smem<1, 2>, 2);
                if (st != VUP_OK) return st;
            }
            if (keys_ready) VUP_CHECK_CUDA(cudaStreamWaitEvent(s, keys_ready, 0));
            st = nd == 3 ? (rest_staged ? launch(k_hist_smem<2, 4>, 4) : launch(k_hist_smem<2, 0>, 0))
                         : launch(k_hist_smem<1, 0>, 0);
            if (st != VUP_OK) return st;
            if (!points_only) {
                st = nd == 3 ? launch(k_hist_smem<2, 1>, 1) : launch(k_hist_smem<1, 1>, 1);
                if (st != VUP_OK) return st;
            }
        } else {
            // G groups of C / G chunks per part, G dividing C / kGroupChunks, for the
            // fewest idle SM slots in the last wave
            const int S = A.C / kGroupChunks;
            int G = S;
            double best = -1.0;
            for (int gg = S; gg >= 1; --gg) {
                if (S % gg) continue;
                const int64_t items = (int64_t)P_max * gg * nkt;
                const double eff = (double)items / (double)(ceil_div64(items, sms) * sms);
                if (eff > best + 0.02) {
                    best = eff;
                    G = gg;
                }
            }
            if (keys_ready) VUP_CHECK_CUDA(cudaStreamWaitEvent(s, keys_ready, 0));
            dim3 grd((unsigned)(P_max * G), (unsigned)nkt);
            k_hist_global<<<grd, kHistWarps * 32, 0, s>>>(A, G);
            VUP_CHECK_LAUNCH();
        }
    }
    VUP_PROF("hist_fixup", s, 1);
    dim3 fg((unsigned)ceil_div64(K, kFinK * kFinNK), (unsigned)ceil_div64(g->B, kFinB));
    VUP_CHECK_CUDA(launch_pdl(k_hist_finish, fg, dim3(32 * kFinB), 0, s, A));
    return VUP_OK;
}

bool vup_hist_tile_fits(vup_grid g) {
    const bool coded = g->ndim == 2 || (g->n[0] <= 512 && g->n[1] <= 4096);
    for (int l = 0; l < g->n_layouts; ++l)
        if (hist_smem_bytes(g->hl[l].part_rows) > kSmemMost) return false;
    return coded;
}

// H (or null) and posterior means of a 2-D / 3-D grid whose tiles fit shared
// memory, from the densities' factor tables and the point stream.
vup_status vup_post_fused(vup_grid g, int64_t K, float *hist, float *post, cudaStream_t s) {
    int64_t rows;
    int P_max;
    PostArgs A{};
    A.h = hist_args_for(g, K, nullptr, rows, P_max);
    A.h.points_only = 1;
    const int nd = g->ndim, no = 1 + nd;
    const int64_t K_pad = A.h.K_pad;
    int64_t axis_rows = 0;
    for (int d = 0; d < nd; ++d) axis_rows += g->n[d];
    // scratch: f_x tables, then the cut rows and the keys' rows; the coordinates
    const size_t f_fx = (size_t)axis_rows * K_pad, f_part = (size_t)P_max * A.h.C * 2 * no;
    const size_t f_dir = (size_t)P_max * A.h.B * no;  // (both per density)
    A.kb = std::min<int64_t>(K_pad, std::max<int64_t>(1, (int64_t)(kPostSums / (sizeof(float) * 128 * (f_part + f_dir)))) * 128);
    vup_status st;
    if ((st = devbuf_reserve(g->post_tmp, sizeof(float) * (f_fx + (f_part + f_dir) * A.kb))) != VUP_OK) return st;
    if ((st = devbuf_reserve(g->post_x, sizeof(float) * (size_t)axis_rows)) != VUP_OK) return st;
    float *fx = (float *)g->post_tmp.p, *xs = (float *)g->post_x.p;
    A.xs = xs;
    A.fx = fx;
    A.part = fx + f_fx;
    A.direct = A.part + f_part * A.kb;
    A.hist = hist;
    A.post = post;
    AxisGeom G{};
    G.ndim = nd;
    int64_t n_max = 1;
    for (int d = 0; d < nd; ++d) {
        G.n[d] = g->n[d];
        G.lo[d] = g->lo[d];
        G.h[d] = (g->hi[d] - g->lo[d]) / (double)g->n[d];
        n_max = std::max(n_max, g->n[d]);
    }
    int *ctr = g->hist_sel + kHistCtr;
    {
        VUP_PROF("posterior_axis_weights", s, 2);
        k_axis_coords<<<(unsigned)ceil_div64(n_max, 128), 128, 0, s>>>(G, xs);
        VUP_CHECK_LAUNCH();
        const int64_t blocks = std::min<int64_t>(axis_rows * ceil_div64(K_pad, 512), (int64_t)vup_num_sms() * 16);
        k_post_tables<<<(unsigned)blocks, 128, 0, s>>>(A, fx, (float *)g->ftab_fold.p, ctr);
        VUP_CHECK_LAUNCH();
    }
    for (A.k0 = 0; A.k0 < K; A.k0 += A.kb) {
        const int64_t nk = std::min(A.kb, K - A.k0);
        if (A.k0) VUP_CHECK_CUDA(cudaMemsetAsync(ctr, 0, sizeof(int), s));  // (the tables' kernel zeroed it for the first)
        {
            VUP_PROF("hist_segmented", s, 1);
            const int nkt = (int)ceil_div64(nk, kPostKT);
            const size_t smem = hist_smem_bytes(rows);
            const unsigned ctas = (unsigned)std::min<int64_t>(vup_num_sms(), (int64_t)P_max * nkt * A.h.C);
            auto launch = [&](auto kern) -> vup_status {
                VUP_CHECK_CUDA(smem_allow(kern));
                kern<<<ctas, kHistWarps * 32, smem, s>>>(A, rows, nkt, ctr);
                VUP_CHECK_LAUNCH();
                return VUP_OK;
            };
            st = nd == 2 ? launch(k_post_walk<1, 4>)
                         : (vup_hist_rest_staged(g) ? launch(k_post_walk<2, 1>) : launch(k_post_walk<2, 4>));
            if (st != VUP_OK) return st;
        }
        VUP_PROF("posterior_finish", s, 1);
        const dim3 fin((unsigned)ceil_div64(nk, 128), (unsigned)ceil_div64(g->B, 8));
        if (nd == 2) k_post_finish<3><<<fin, 256, 0, s>>>(A);
        else k_post_finish<4><<<fin, 256, 0, s>>>(A);
        VUP_CHECK_LAUNCH();
    }
    return VUP_OK;
}

// A 2-D grid whose every part fits the shared-memory tile.
bool vup_hist_batchable(vup_grid g) {
    if (g->ndim != 2) return false;
    for (int l = 0; l < g->n_layouts; ++l)
        if (hist_smem_bytes(g->hl[l].part_rows) > kSmemMost) return false;
    return true;
}

// Batched histograms of n 2-D instances: one persistent launch over every
// instance's (part, chunk group, density tile) items, longest first, and one
// finishing launch.
struct HistPlan {
    DevBuf fold;                      // FoldTabArgs of every instance that wants a histogram
    DevBuf args, items, fitems, ctr;  // ctr: next item of each stream's launch, then each stream's item count
    DevBuf lists;                     // [3][n_items] each stream's items (k_hist_split_items)
    int n_inst = 0, n_fold = 0, n_items = 0, n_fitems = 0;
    int64_t rows = 0;
};

// The most parts either layout of a grid has.
static int g_parts(const vup_grid_s *g) {
    int P = 1;
    for (int l = 0; l < g->n_layouts; ++l) P = std::max(P, g->hl[l].P);
    return P;
}

vup_status vup_hist_plan(int n, const vup_grid *gs, const int64_t *Ks, float *const *hists, void **out) {
    std::vector<HistArgs> args(n);
    std::vector<std::pair<int64_t, HistItem>> work;
    std::vector<int4> fin;
    int64_t rows_max = 0;
    // SM cycles of an instance's tile fill and of its walk per (part, density
    // tile), from the sizes (its stream and counts are the device's to choose): a
    // walk costs about a cycle per point and 128 densities on smooth models.  An
    // instance is cut so that no item's walk exceeds an SM's share of the whole
    // batch, nor falls below its fill: small batches fill the SMs, large ones keep one
    // item per tile.  32 instances of 32 - 1024 points a side 713 us with items of at
    // most a third of the share, 694 of the share, 694 of twice that or uncut; 10 of
    // at most 169: 127, 117, 116, 119; 16 of at most 621: 201, 185, 185, 219; 12 of at
    // most 202: 116, 116, 132, 157.
    std::vector<int64_t> fill(n), walk(n);
    double share = 0.0;
    for (int i = 0; i < n; ++i) {
        int64_t rows;
        int P_max;
        args[i] = hist_args_for(gs[i], Ks[i], hists[i], rows, P_max);
        fill[i] = 3000 + 30 * rows;
        walk[i] = gs[i]->N / P_max;
        if (hists[i]) share += (double)(fill[i] + walk[i]) * (double)P_max * (double)ceil_div64(Ks[i], kKT);
    }
    share /= vup_num_sms();
    for (int i = 0; i < n; ++i) {
        if (!hists[i]) continue;
        const int P_max = g_parts(gs[i]);
        const int64_t rows = std::max(args[i].L0.part_rows, args[i].L1.part_rows);
        rows_max = std::max(rows_max, rows);
        const int64_t most = std::max<int64_t>(1, args[i].C_rec / 8);  // at least eight record chunks
        const int G = (int)std::max<int64_t>(
            1, std::min(most, ceil_div64(walk[i], std::max((int64_t)share, fill[i]))));
        args[i].sets = G;
        const int64_t nkt = ceil_div64(Ks[i], kKT);
        const int64_t cost = fill[i] + walk[i] / G;
        for (int p = 0; p < P_max; ++p)
            for (int cg = 0; cg < G; ++cg)
                for (int64_t kt = 0; kt < nkt; ++kt) work.push_back({cost, HistItem{i, p, cg, (int32_t)kt}});
        for (int64_t kb = 0; kb < ceil_div64(Ks[i], kFinK * kFinNK); ++kb)
            for (int bt = 0; bt < (int)ceil_div64(gs[i]->B, kFinB); ++bt) fin.push_back(make_int4(i, (int)kb, bt, 0));
    }
    std::stable_sort(work.begin(), work.end(), [](const auto &a, const auto &b) { return a.first > b.first; });
    std::vector<HistItem> items(work.size());
    for (size_t q = 0; q < work.size(); ++q) items[q] = work[q].second;
    HistPlan *P = new HistPlan();
    P->n_inst = n;
    P->n_items = (int)items.size();
    P->n_fitems = (int)fin.size();
    P->rows = rows_max;
    vup_status st;
    // merged tables only where a histogram is asked for: the other instances' layouts
    // need not exist, nor their tables hold this K
    std::vector<FoldTabArgs> folds;
    for (int i = 0; i < n; ++i)
        if (hists[i]) folds.push_back(fold_tab_args(gs[i], Ks[i]));
    P->n_fold = (int)folds.size();
    if ((st = devbuf_reserve(P->args, sizeof(HistArgs) * n)) != VUP_OK ||
        (st = devbuf_reserve(P->fold, sizeof(FoldTabArgs) * std::max<size_t>(1, folds.size()))) != VUP_OK ||
        (st = devbuf_reserve(P->items, sizeof(HistItem) * std::max<size_t>(1, items.size()))) != VUP_OK ||
        (st = devbuf_reserve(P->fitems, sizeof(int4) * std::max<size_t>(1, fin.size()))) != VUP_OK ||
        (st = devbuf_reserve(P->ctr, sizeof(int) * 6)) != VUP_OK ||
        (st = devbuf_reserve(P->lists, sizeof(int32_t) * 3 * std::max<size_t>(1, items.size()))) != VUP_OK) {
        devbuf_free(P->args);
        devbuf_free(P->fold);
        devbuf_free(P->items);
        devbuf_free(P->fitems);
        devbuf_free(P->ctr);
        devbuf_free(P->lists);
        delete P;
        return st;
    }
    VUP_CHECK_CUDA(cudaMemcpy(P->args.p, args.data(), sizeof(HistArgs) * n, cudaMemcpyHostToDevice));
    VUP_CHECK_CUDA(cudaMemcpy(P->fold.p, folds.data(), sizeof(FoldTabArgs) * folds.size(), cudaMemcpyHostToDevice));
    VUP_CHECK_CUDA(cudaMemcpy(P->items.p, items.data(), sizeof(HistItem) * items.size(), cudaMemcpyHostToDevice));
    VUP_CHECK_CUDA(cudaMemcpy(P->fitems.p, fin.data(), sizeof(int4) * fin.size(), cudaMemcpyHostToDevice));
    // the largest tile any plan may use, so that graphs of earlier plans stay launchable
    VUP_CHECK_CUDA(smem_allow(k_hist_batched<1, 0>));
    VUP_CHECK_CUDA(smem_allow(k_hist_batched<1, 1>));
    VUP_CHECK_CUDA(smem_allow(k_hist_batched<1, 2>));
    *out = P;
    return VUP_OK;
}

void vup_hist_plan_free(void *plan) {
    HistPlan *P = (HistPlan *)plan;
    if (!P) return;
    devbuf_free(P->args);
    devbuf_free(P->fold);
    devbuf_free(P->items);
    devbuf_free(P->fitems);
    devbuf_free(P->ctr);
    devbuf_free(P->lists);
    delete P;
}

vup_status vup_hist_batched(void *plan, cudaStream_t s) {
    const HistPlan *P = (const HistPlan *)plan;
    if (P->n_items == 0) return VUP_OK;
    const size_t smem = hist_smem_bytes(P->rows);
    if (smem > kSmemMost) return VUP_ERR_UNSUPPORTED;
    {
        VUP_PROF("hist_segmented_batched", s, 5);
        for (int i0 = 0; i0 < P->n_fold; i0 += 65535) {  // (the grid's y limit)
            const unsigned ny = (unsigned)std::min(65535, P->n_fold - i0);
            k_fold_tables_batched<<<dim3(32, ny), 128, 0, s>>>((const FoldTabArgs *)P->fold.p + i0);
            VUP_CHECK_LAUNCH();
        }
        const int grid = std::max(1, std::min(P->n_items, vup_num_sms()));
        int *ctr = (int *)P->ctr.p, *counts = ctr + 3;
        const int32_t *lists = (const int32_t *)P->lists.p;
        const HistArgs *args = (const HistArgs *)P->args.p;
        const HistItem *items = (const HistItem *)P->items.p;
        VUP_CHECK_CUDA(cudaMemsetAsync(ctr, 0, 3 * sizeof(int), s));
        const size_t split_smem = P->n_inst <= kSplitStaged ? (size_t)P->n_inst : 0;
        k_hist_split_items<<<1, kSplitThreads, split_smem, s>>>(args, P->n_inst, items, P->n_items,
                                                                (int32_t *)P->lists.p, counts);
        VUP_CHECK_LAUNCH();
        k_hist_batched<1, 0><<<grid, kHistWarps * 32, smem, s>>>(args, items, lists, counts, P->rows, ctr);
        VUP_CHECK_LAUNCH();
        k_hist_batched<1, 1><<<grid, kHistWarps * 32, smem, s>>>(args, items, lists + P->n_items, counts + 1,
                                                                 P->rows, ctr + 1);
        VUP_CHECK_LAUNCH();
        k_hist_batched<1, 2><<<grid, hist_warps(2) * 32, hist_smem_bytes(P->rows, hist_warps(2)), s>>>(
            args, items, lists + 2 * (size_t)P->n_items, counts + 2, P->rows, ctr + 2);
        VUP_CHECK_LAUNCH();
    }
    VUP_PROF("hist_fixup_batched", s, 1);
    k_hist_finish_batched<<<P->n_fitems, 32 * kFinB, 0, s>>>((const HistArgs *)P->args.p,
                                                             (const int4 *)P->fitems.p);
    VUP_CHECK_LAUNCH();
    return VUP_OK;
}
