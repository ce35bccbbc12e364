// The map of Eq. (1)-(2) over a cluster tree of the pixels (tree.cuh says which pairs are summed
// where and why the result is the all-pairs sum to the working precision).
//
//   k_tree_crit      per sample and per tile of 64 samples, what the near/far decision reads
//   k_tree_leaf_geo  finest clusters (T x T pixel blocks): centre, frame, extent, near radius
//   k_tree_up_geo    parents (2 x 2 children), level by level
//   k_tree_nodes_*   per level from the coarsest: the level's samples summed at the p^2 nodes of every
//                    cluster, plus the parent's interpolant at the same nodes
//   k_tree_pixels_*  per finest cluster: the interpolant at its pixels plus the near samples pixel by
//                    pixel
// Sums over chunks of samples go to separate partial arrays, added in a fixed order by the reader, so
// maps are reproducible.
//
// FP32 maps, 8 x 8 nodes, near radius 3.5 half-sizes, leaves of 16 x 16 pixels: N_side 512 with 2e5 samples
// 309 -> 7.1 ms (6.3e11 pairs; 3e9 pair terms at nodes, 6e8 at pixels), N_side 64 with 10,240 samples
// 3.1 -> 0.47 ms; error against FP64 2.6e-8 of the rms (direct kernels 6.9e-8), largest 3e-7 (9e-7).  The
// node kernels are bound by FP32 issue (45-55% of the cycles, FMA pipe 35-57%) at the 16 warps per SM that their
// registers allow, the pixel kernel by its FP64 near pairs and by the tests that find them (issue 41%, FP64
// unit 21%).
#include "tree.cuh"

#include <algorithm>

namespace isw {

namespace {

struct TreeNodeArgs {
    TreeSamples S;
    const TreeRec *rec;
    const TreeGeo *geo, *pgeo;   // this level, the parent level (NULL at the coarsest)
    int nb, pnb;
    TreeWork W, Wp;              // items of this level, chunks of the parent's
    double *F;                   // [ncl + pool][64]
    const double *Fp;            // the parent level's
    unsigned long long *queue;
};

// Samples per chunk, at least.  Strings put up to 30 times the mean number of samples on a few clusters;
// cut by the planned chunks N_side 100 with 3e4 samples takes 1.1 ms, with the same number of chunks for
// every cluster (50, to spread the heavy ones) 1.9.  Doubled until the pool holds all chunks; with 1024 and 256
// N_side 64 with 10,240 samples takes 0.55 ms instead of 0.47 (256 and 64: the same).
constexpr int kNodeTarget = 512, kPixTarget = 128;

// Samples staged for one cluster, relative to its centre, each value twice as the (v, v) operand of a
// packed instruction over two targets: with D = n0 - Xhat and target n = n0 + m, d = D + m and
//   |d|^2 = K + 2 D.m + |m|^2,  Xdot.d = P + Xdot.m,  X'.d = Q + X'.m,  B = B0 + Xdot.m
// from the per-sample K = |D|^2, P = Xdot.D, Q = X'.D and B0 = 1 + n0.Xdot (free of cancellation), so
// a pair costs 18 FP32 operations instead of the 25 of the form that subtracts float pairs, and needs
// neither the far-field form nor a test of B.  |m| < 0.36 |D| on a cluster whose samples are far, so
// every sum keeps its relative accuracy.
// Entry (9 x 16 B, an odd stride: the staging threads' stores meet no bank conflict):
//   (2Dx, 2Dy) (2Dz, K) (Xdot x, y) (Xdot z, P) (-X' x, y) (-X' z, -Q) (B0, f) (c, -)
constexpr int kNodeRec = 9;
// Pixels may be close to their samples or in their beams: (c, rho^2 | 1 - |Xdot|), the low parts of D
// (its high parts are the 2D / 2) and W = n0 + Xdot/|Xdot|, as (Dx, Dy) (Dz, Wx) (Wy, Wz).
constexpr int kPixRec = 11;

struct __align__(16) TreeSmem32 {
    ulonglong2 rec[kTreeBatch * kPixRec];   // also the tables of the interpolation, before or after
    TreeScanSmem scan;
    TreeGeo geo, pgeo;
    double coef[kNN], tmp[kNN];
    int64_t item;
};

// The interpolant with coefficients coef (FP64, shared) at (x, y) in [-1, 1]^2: everything but the
// mean in FP32, the mean added in FP64.
__device__ __forceinline__ double interp32(const double *coef, const float *cf, float x, float y)
{
    float tx[kNP];
    tx[0] = 1.f;
    tx[1] = x;
#pragma unroll
    for (int i = 2; i < kNP; ++i) tx[i] = fmaf(2.f * x, tx[i - 1], -tx[i - 2]);
    float v = 0.f, t0 = 1.f, t1 = y;
#pragma unroll
    for (int j = 0; j < kNP; ++j) {
        const float4 a = reinterpret_cast<const float4 *>(cf)[2 * j], b = reinterpret_cast<const float4 *>(cf)[2 * j + 1];
        const float r = fmaf(b.w, tx[7], fmaf(b.z, tx[6], fmaf(b.y, tx[5], fmaf(b.x, tx[4],
                        fmaf(a.w, tx[3], fmaf(a.z, tx[2], fmaf(a.y, tx[1], a.x)))))));
        v = fmaf(r, t0, v);
        const float t2 = fmaf(2.f * y, t1, -t0);
        t0 = t1;
        t1 = t2;
    }
    return coef[0] + (double)v;
}

// coefficients in float with the mean taken out (interp32 adds it in FP64)
__device__ __forceinline__ void coefs_to_float(const double *coef, float *cf)
{
    for (int k = threadIdx.x; k < kNN; k += blockDim.x) cf[k] = k == 0 ? 0.f : (float)coef[k];
    __syncthreads();
}

// One sample relative to the centre of g, into its shared entry.
template <int REC>
__device__ __forceinline__ void stage_sample(const float4 (&q)[4], const TreeGeo &g, ulonglong2 *dst)
{
    float D[3], Dl[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {   // (n0 hi + lo) - (Xhat hi + lo) as a float pair
        const float nh = comp(g.c, c), xh = comp(q[0], c), t = nh - xh, bb = t - nh;
        const float e = ((nh - (t - bb)) - (xh + bb)) + (comp(g.l, c) - comp(q[1], c));
        D[c] = t + e;
        Dl[c] = e - (D[c] - t);
    }
    const float P = fmaf(q[2].z, D[2], fmaf(q[2].y, D[1], q[2].x * D[0]));
    const float Q = fmaf(q[3].z, D[2], fmaf(q[3].y, D[1], q[3].x * D[0]));
    const float K = fmaf(D[2], D[2], fmaf(D[1], D[1], D[0] * D[0]));
    const float om = q[2].w, v = 1.f - om, iv = v > 0.f ? 1.f / v : 0.f;
    const float wx = fmaf(q[2].x, iv, g.c.x), wy = fmaf(q[2].y, iv, g.c.y), wz = fmaf(q[2].z, iv, g.c.z);
    const float B0 = fmaf(0.5f * v, fmaf(wz, wz, fmaf(wy, wy, wx * wx)), om);   // 1 - v + v |n0 + Xdot/v|^2 / 2
    dst[0] = make_ulonglong2(dup2(2.f * D[0]), dup2(2.f * D[1]));
    dst[1] = make_ulonglong2(dup2(2.f * D[2]), dup2(K));
    dst[2] = make_ulonglong2(dup2(q[2].x), dup2(q[2].y));
    dst[3] = make_ulonglong2(dup2(q[2].z), dup2(P));
    dst[4] = make_ulonglong2(dup2(-q[3].x), dup2(-q[3].y));
    dst[5] = make_ulonglong2(dup2(-q[3].z), dup2(-Q));
    dst[6] = make_ulonglong2(dup2(B0), dup2(q[1].w));
    dst[7] = make_ulonglong2(dup2(q[0].w), f2_pack(q[3].w, om));
    if (REC > 9) {
        dst[8] = make_ulonglong2(dup2(Dl[0]), dup2(Dl[1]));
        dst[9] = make_ulonglong2(dup2(Dl[2]), dup2(wx));
        dst[10] = make_ulonglong2(dup2(wy), dup2(wz));
    }
}

// Stages count records of the scan's list in batches, one sample per thread; the next batch's records
// are in flight while eval(entries, first list entry, batch size) runs.  Whole block.
template <int REC, typename Eval>
__device__ __forceinline__ void tree_batches(TreeSmem32 &sm, const TreeRec *__restrict__ recs, int count, Eval &&eval)
{
    const int tid = threadIdx.x;
    float4 q[4];
    auto fetch = [&](int b0) {
        if (b0 + tid < count) {
            const float4 *src = recs[sm.scan.list[b0 + tid] & kTreeIndex].v;
#pragma unroll
            for (int k = 0; k < 4; ++k) q[k] = src[k];
        }
    };
    fetch(0);
#pragma unroll 1
    for (int b0 = 0; b0 < count; b0 += kTreeBatch) {
        if (b0 + tid < count) stage_sample<REC>(q, sm.geo, sm.rec + tid * REC);
        fetch(b0 + kTreeBatch);
        __syncthreads();
        eval(sm.rec, b0, count - b0 < kTreeBatch ? count - b0 : kTreeBatch);
        __syncthreads();
    }
}

// The samples of one level at the nodes of its clusters.  A half-warp holds the 64 nodes of the
// cluster, four per lane as two f32x2 pairs, and takes every eighth sample of a batch (two samples per
// warp at a time: one 16-byte shared load then feeds four nodes of two samples; with two nodes per
// lane of one sample the loads bound the loop).  The eight half-warps are added up at the end.
template <bool ROOT>
__global__ void __launch_bounds__(kTreeNT, 4) k_tree_nodes_f32(TreeNodeArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TreeSmem32 &sm = *reinterpret_cast<TreeSmem32 *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, half = lane >> 4, hl = lane & 15;
    const int np = *a.W.npool;
    TreeQueue queue{a.queue, 0ull};
    for (int64_t item = queue.first(&sm.item); item < a.W.ncl + np; item = queue.next(&sm.item)) {
        int kc, nch;
        int64_t at;
        const int64_t cl = tree_item(a.W, item, np, kc, nch, at);
        if (cl < 0) continue;
        const int64_t pcl = ROOT ? 0 : tree_parent(cl, a.nb, a.pnb);
        if (!ROOT) {
            load_geo(&sm.pgeo, a.pgeo + pcl);
        }
        load_geo(&sm.geo, a.geo + cl);
        __syncthreads();
        const float4 self = sm.geo.c, parent = ROOT ? self : sm.pgeo.c;
        if (tree_empty(self)) continue;
        uint64_t m[2][3], mm[2];   // node offsets from the centre, |m|^2
#pragma unroll
        for (int pp = 0; pp < 2; ++pp) {
            float o[2][3];
            node_offset(sm.geo, 32 * pp + hl, o[0]);
            node_offset(sm.geo, 32 * pp + 16 + hl, o[1]);
#pragma unroll
            for (int c = 0; c < 3; ++c) m[pp][c] = f2_pack(o[0][c], o[1][c]);
            mm[pp] = f2_fma(m[pp][2], m[pp][2], f2_fma(m[pp][1], m[pp][1], f2_mul(m[pp][0], m[pp][0])));
        }
        float ahi[4] = {0.f, 0.f, 0.f, 0.f}, alo[4] = {0.f, 0.f, 0.f, 0.f};
        auto consume = [&](int count) {
            tree_batches<kNodeRec>(sm, a.rec, count, [&](const ulonglong2 *mr, int b0, int cnt) {
                uint64_t part[2] = {0ull, 0ull};
#pragma unroll 1
                for (int s0 = 2 * w; s0 < cnt; s0 += 2 * (kTreeNT / 32)) {
                    const bool on = s0 + half < cnt;
                    const ulonglong2 *r = mr + kNodeRec * (on ? s0 + half : s0);
                    const ulonglong2 r0 = r[0], r1 = r[1], r2 = r[2], r3 = r[3], r4 = r[4], r5 = r[5], r6 = r[6];
                    const uint64_t c = on ? r[7].x : 0ull;   // no second sample: zero weight
#pragma unroll
                    for (int pp = 0; pp < 2; ++pp) {
                        const uint64_t Q = f2_fma(m[pp][2], r1.x, f2_fma(m[pp][1], r0.y, f2_fma(m[pp][0], r0.x, f2_add(mm[pp], r1.y))));
                        const uint64_t g = f2_fma(m[pp][2], r3.x, f2_fma(m[pp][1], r2.y, f2_mul(m[pp][0], r2.x)));
                        const uint64_t Qdn = f2_fma(m[pp][2], r5.x, f2_fma(m[pp][1], r4.y, f2_fma(m[pp][0], r4.x, r5.y)));
                        const uint64_t B = f2_add(g, r6.x), Pd = f2_add(g, r3.y), A = f2_sub(r6.y, Qdn);
                        const uint64_t num = f2_fma(A, Qdn, f2_mul(B, Pd));
                        float u0, u1;
                        f2_unpack(f2_mul(B, Q), u0, u1);
                        part[pp] = f2_fma(f2_mul(c, num), f2_pack(rcp_approx(u0), rcp_approx(u1)), part[pp]);
                    }
                }
#pragma unroll
                for (int pp = 0; pp < 2; ++pp) {
                    float p0, p1;
                    f2_unpack(part[pp], p0, p1);
                    fold(ahi[2 * pp], alo[2 * pp], p0);
                    fold(ahi[2 * pp + 1], alo[2 * pp + 1], p1);
                }
            });
        };
        tree_scan<ROOT, false>(a.S, kc, nch, self, parent, 0.f, 0.f, 0.f, sm.scan, consume);
        double (*red)[kNN] = reinterpret_cast<double (*)[kNN]>(sm.rec);   // the batches are done
#pragma unroll
        for (int q = 0; q < 4; ++q) red[2 * w + half][16 * q + hl] = widen(ahi[q]) + widen(alo[q]);
        __syncthreads();
        double v = 0.0;
        if (tid < kNN) {
#pragma unroll
            for (int i = 0; i < kTreeNT / 16; ++i) v += red[i][tid];
        }
        if (!ROOT && kc == 0 && !tree_wide(parent)) {   // the parent's interpolant at this cluster's nodes
            cheb_coefs<kNP>(a.Fp, a.Wp, pcl, sm.coef, sm.tmp);
            float *cf = reinterpret_cast<float *>(sm.rec + kTreeNT / 16 * kNN / 2);
            coefs_to_float(sm.coef, cf);
            if (tid < kNN) {
                float d[3], x, y;
                node_offset(sm.geo, tid, d);
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    d[c] += (comp(sm.geo.c, c) - comp(sm.pgeo.c, c)) + (comp(sm.geo.l, c) - comp(sm.pgeo.l, c));
                local_xy(sm.pgeo, d[0], d[1], d[2], x, y);
                v += interp32(sm.coef, cf, x, y);
            }
        }
        if (tid < kNN) a.F[at * kNN + tid] = v;
        __syncthreads();
    }
}

struct TreePixArgs {
    TreeSamples S;
    const TreeRec *rec;
    const Seg64 *s64;
    const TreeGeo *geo;          // finest clusters
    const double *nv;            // pixel table, T * T slots per cluster
    int64_t ldn;
    const int64_t *outidx;
    TreeWork W, Wf;              // items of the pixel stage, chunks of the finest level's node sums
    const double *F;
    double *theta;
    double *partial;             // [pool][T * T]
    int accumulate;
    float b_min;
    DevStatus *st;
    unsigned long long *queue;
};

// FP64 pairs of one warp's 64 pixels: queued as (record, pixel) and evaluated 32 at a time, one per
// lane.  Evaluated where they are found, a warp spent the FP64 unit's 64 cycles per instruction on
// one or two lanes, and the tiles that hold a string took 1.5 ms at N_side 64.
struct TreeNearQueue {
    uint32_t src[64];
    double val[32];
    double acc[64];
    uint8_t pix[64];
};
struct __align__(16) TreeSmemPix {
    TreeSmem32 s;
    TreeNearQueue q[kTreeNT / 32];
};

// Evaluate the first cnt <= 32 entries of the warp's queue and add them to the pixels' sums in queue
// order (entries of one pixel by the lowest lane that holds it).
__device__ __noinline__ void near_flush(TreeNearQueue &q, int cnt, const Seg64 *__restrict__ s64,
                                        const double *__restrict__ nv, int64_t ldn, int64_t kw, unsigned &zerocnt)
{
    const int lane = threadIdx.x & 31;
    const bool on = lane < cnt;
    const int px = on ? q.pix[lane] : 64 + lane;
    double v = 0.0;
    if (on) {
        const Seg64 g = s64[q.src[lane]];
        const int64_t k = kw + px;
        v = pair64(nv[k], nv[ldn + k], nv[2 * ldn + k], g, zerocnt);
    }
    q.val[lane] = v;
    __syncwarp();
    const unsigned peers = __match_any_sync(0xffffffffu, px);
    if (on && (peers & ((1u << lane) - 1u)) == 0u) {
        double s = q.acc[px];
        for (unsigned m = peers; m; m &= m - 1u) s += q.val[__ffs(m) - 1];
        q.acc[px] = s;
    }
    __syncwarp();
}

// The pixels of the finest clusters: a half-warp holds 64 of them, four per lane as two f32x2 pairs, and
// every warp takes all near samples, one per half-warp at a time.  A sample that may come within
// max(rho, R / 2) of some pixel takes d from float pairs; pairs with |d| < rho or B < b_min / 1000 go to
// the warp's FP64 queue.
__global__ void __launch_bounds__(kTreeNT, 4) k_tree_pixels_f32(TreePixArgs a)
{
    constexpr int TILE = kLeaf * kLeaf;
    static_assert(TILE == 2 * kTreeNT, "64 pixels per warp");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TreeSmem32 &sm = reinterpret_cast<TreeSmemPix *>(smem_raw)->s;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, half = lane >> 4, hl = lane & 15;
    TreeNearQueue &nq = reinterpret_cast<TreeSmemPix *>(smem_raw)->q[w];
    const uint64_t half2 = f2_pack(0.5f, 0.5f);
    unsigned nearcnt = 0, zerocnt = 0;
    const int np = *a.W.npool;
    TreeQueue queue{a.queue, 0ull};
    for (int64_t item = queue.first(&sm.item); item < a.W.ncl + np; item = queue.next(&sm.item)) {
        int kc, nch;
        int64_t at;
        const int64_t cl = tree_item(a.W, item, np, kc, nch, at);
        if (cl < 0) continue;
        load_geo(&sm.geo, a.geo + cl);
        nq.acc[lane] = 0.0;
        nq.acc[32 + lane] = 0.0;
        __syncthreads();
        const float4 self = sm.geo.c;
        if (tree_empty(self)) continue;
        float ahi[4] = {0.f, 0.f, 0.f, 0.f}, alo[4] = {0.f, 0.f, 0.f, 0.f};
        unsigned valid = 0;
        int qlen = 0;
        uint64_t m[2][3], ml[2][3], mm[2];   // offsets from the centre as float pairs, |m|^2
        const int64_t kw = cl * TILE + w * 64;   // pixel 16 q + hl of the warp is the lane's q-th
        {
            // two pixels per lane, the other two from the lane of the other half-warp that has the same ones
            float h[2][3], l[2][3], oh[2][3], ol[2][3];
            unsigned own = 0;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int64_t k = kw + 16 * (2 * half + u) + hl;
                if (a.outidx[k] >= 0) own |= 1u << (2 * half + u);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    split_float(a.nv[c * a.ldn + k] - sm.geo.n0[c], h[u][c], l[u][c]);
                    oh[u][c] = __shfl_xor_sync(0xffffffffu, h[u][c], 16);
                    ol[u][c] = __shfl_xor_sync(0xffffffffu, l[u][c], 16);
                }
            }
            valid = own | __shfl_xor_sync(0xffffffffu, own, 16);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                m[0][c] = half ? f2_pack(oh[0][c], oh[1][c]) : f2_pack(h[0][c], h[1][c]);
                m[1][c] = half ? f2_pack(h[0][c], h[1][c]) : f2_pack(oh[0][c], oh[1][c]);
                ml[0][c] = half ? f2_pack(ol[0][c], ol[1][c]) : f2_pack(l[0][c], l[1][c]);
                ml[1][c] = half ? f2_pack(l[0][c], l[1][c]) : f2_pack(ol[0][c], ol[1][c]);
            }
#pragma unroll
            for (int pp = 0; pp < 2; ++pp)
                mm[pp] = f2_fma(m[pp][2], m[pp][2], f2_fma(m[pp][1], m[pp][1], f2_mul(m[pp][0], m[pp][0])));
        }
        double far[2] = {0.0, 0.0};   // of the lane's pixels 2 half and 2 half + 1
        if (kc == 0 && !tree_wide(self)) {
            cheb_coefs<kNP>(a.F, a.Wf, cl, sm.coef, sm.tmp);
            float *cf = reinterpret_cast<float *>(sm.rec);
            coefs_to_float(sm.coef, cf);
            float d[2][3];
#pragma unroll
            for (int c = 0; c < 3; ++c) f2_unpack(half ? m[1][c] : m[0][c], d[0][c], d[1][c]);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                float x, y;
                local_xy(sm.geo, d[u][0], d[u][1], d[u][2], x, y);
                far[u] = interp32(sm.coef, cf, x, y);
            }
            __syncthreads();   // the coefficients' buffer is the first batch's
        }
        const float b_tiny = a.b_min * 1e-3f;
        auto consume = [&](int count) {
            tree_batches<kPixRec>(sm, a.rec, count, [&](const ulonglong2 *mr, int b0, int cnt) {
                uint64_t part[2] = {0ull, 0ull};
#pragma unroll 1
                for (int s0 = 0; s0 < cnt; s0 += 2) {
                    const bool on = s0 + half < cnt;
                    const int s = on ? s0 + half : s0;
                    const ulonglong2 *r = mr + kPixRec * s;
                    const ulonglong2 r0 = r[0], r1 = r[1], r2 = r[2], r3 = r[3], r4 = r[4], r5 = r[5], r6 = r[6], r7 = r[7];
                    const uint64_t c = on ? r7.x : 0ull;   // no second sample: zero weight
                    const uint32_t src = sm.scan.list[b0 + s];
                    if (!__any_sync(0xffffffffu, (src & (kTreeBeam | kTreeClose)) != 0u)) {
#pragma unroll
                        for (int pp = 0; pp < 2; ++pp) {
                            const uint64_t Q = f2_fma(m[pp][2], r1.x, f2_fma(m[pp][1], r0.y, f2_fma(m[pp][0], r0.x, f2_add(mm[pp], r1.y))));
                            const uint64_t g = f2_fma(m[pp][2], r3.x, f2_fma(m[pp][1], r2.y, f2_mul(m[pp][0], r2.x)));
                            const uint64_t Qdn = f2_fma(m[pp][2], r5.x, f2_fma(m[pp][1], r4.y, f2_fma(m[pp][0], r4.x, r5.y)));
                            const uint64_t B = f2_add(g, r6.x), Pd = f2_add(g, r3.y), A = f2_sub(r6.y, Qdn);
                            const uint64_t num = f2_fma(A, Qdn, f2_mul(B, Pd));
                            float u0, u1;
                            f2_unpack(f2_mul(B, Q), u0, u1);
                            part[pp] = f2_fma(f2_mul(c, num), f2_pack(rcp_approx(u0), rcp_approx(u1)), part[pp]);
                        }
                        continue;
                    }
                    const ulonglong2 r8 = r[8], r9 = r[9], r10 = r[10];
                    float rho2, om;
                    f2_unpack(r7.y, rho2, om);
                    const uint64_t om2 = dup2(om), hv2 = dup2(fmaf(-0.5f, om, 0.5f));   // 1 - v, v / 2
                    unsigned near = 0;
#pragma unroll
                    for (int pp = 0; pp < 2; ++pp) {
                        const uint64_t dx = f2_add(f2_fma(half2, r0.x, m[pp][0]), f2_add(ml[pp][0], r8.x));
                        const uint64_t dy = f2_add(f2_fma(half2, r0.y, m[pp][1]), f2_add(ml[pp][1], r8.y));
                        const uint64_t dz = f2_add(f2_fma(half2, r1.x, m[pp][2]), f2_add(ml[pp][2], r9.x));
                        const uint64_t Q = f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx)));
                        const uint64_t Pd = f2_fma(r3.x, dz, f2_fma(r2.y, dy, f2_mul(r2.x, dx)));
                        const uint64_t Qdn = f2_fma(r5.x, dz, f2_fma(r4.y, dy, f2_mul(r4.x, dx)));
                        const uint64_t A = f2_sub(r6.y, Qdn);
                        const uint64_t wx = f2_add(r9.y, m[pp][0]), wy = f2_add(r10.x, m[pp][1]), wz = f2_add(r10.y, m[pp][2]);
                        const uint64_t B = f2_fma(hv2, f2_fma(wz, wz, f2_fma(wy, wy, f2_mul(wx, wx))), om2);
                        const uint64_t num = f2_fma(A, Qdn, f2_mul(B, Pd));
                        float u0, u1, q0, q1, c0, c1;
                        f2_unpack(f2_mul(B, Q), u0, u1);
                        f2_unpack(Q, q0, q1);
                        f2_unpack(B, c0, c1);
                        u0 = rcp_approx(u0);
                        u1 = rcp_approx(u1);
                        if (q0 < rho2 || c0 < b_tiny) {
                            near |= 1u << (2 * pp);
                            u0 = 0.f;   // queued: zero weight here
                        }
                        if (q1 < rho2 || c1 < b_tiny) {
                            near |= 2u << (2 * pp);
                            u1 = 0.f;
                        }
                        part[pp] = f2_fma(f2_mul(c, num), f2_pack(u0, u1), part[pp]);
                    }
                    if (!__any_sync(0xffffffffu, near != 0u)) continue;
                    near &= on ? valid : 0u;
                    const unsigned below = (1u << lane) - 1u;
#pragma unroll 1
                    for (int q = 0; q < 4; ++q) {
                        const bool hit = near >> q & 1u;
                        const unsigned m = __ballot_sync(0xffffffffu, hit);
                        if (!m) continue;
                        if (hit) {
                            const int p = qlen + __popc(m & below);
                            nq.src[p] = src & kTreeIndex;
                            nq.pix[p] = (uint8_t)(16 * q + hl);
                            ++nearcnt;
                        }
                        qlen += __popc(m);
                        __syncwarp();
                        if (qlen >= 32) {
                            near_flush(nq, 32, a.s64, a.nv, a.ldn, kw, zerocnt);
                            const uint32_t ms = nq.src[32 + lane];
                            const uint8_t mp = nq.pix[32 + lane];
                            __syncwarp();
                            nq.src[lane] = ms;
                            nq.pix[lane] = mp;
                            qlen -= 32;
                            __syncwarp();
                        }
                    }
                }
#pragma unroll
                for (int pp = 0; pp < 2; ++pp) {
                    float p0, p1;
                    f2_unpack(part[pp], p0, p1);
                    fold(ahi[2 * pp], alo[2 * pp], p0);
                    fold(ahi[2 * pp + 1], alo[2 * pp + 1], p1);
                }
            });
        };
        const float R = target_radius(sm.geo);
        tree_scan<false, true>(a.S, kc, nch, self, self, R, 1.5f * R, a.b_min, sm.scan, consume);
        if (qlen > 0) near_flush(nq, qlen, a.s64, a.nv, a.ldn, kw, zerocnt);
        float sh[2] = {0.f, 0.f}, sl[2] = {0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 4; ++q) {   // both half-warps' sums of a pixel; half q / 2 writes it
            const float bh = __shfl_xor_sync(0xffffffffu, ahi[q], 16), bl = __shfl_xor_sync(0xffffffffu, alo[q], 16);
            float h = ahi[q], l = alo[q] + bl;
            fold(h, l, bh);
            if (half == q / 2) {
                sh[q & 1] = h;
                sl[q & 1] = l;
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int q = 2 * half + u;
            const double v = ((widen(sh[u]) + widen(sl[u])) + nq.acc[16 * q + hl]) + far[u];
            const int64_t k = kw + 16 * q + hl;
            if (nch == 1) {
                const int64_t oi = a.outidx[k];
                if (oi >= 0) a.theta[oi] = a.accumulate ? a.theta[oi] + v : v;
            } else {
                a.partial[item * TILE + w * 64 + 16 * q + hl] = v;   // pool entry of the chunk
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        nearcnt += __shfl_xor_sync(0xffffffffu, nearcnt, o);
        zerocnt += __shfl_xor_sync(0xffffffffu, zerocnt, o);
    }
    if (lane == 0 && (nearcnt | zerocnt)) {
        atomicAdd(&a.st->near_pairs, (unsigned long long)nearcnt);
        atomicAdd(&a.st->zero_pairs, (unsigned long long)zerocnt);
    }
}

// ------------------------------------------------------------------------------------
// FP64 maps: 16 x 16 nodes, leaves of 32 x 32 pixels.  The FP64 unit (two FMA lanes per clock and SM)
// is all that counts, so every thread simply holds its nodes or pixels and reads one staged sample at
// a time.  N_side 64 with 10,240 samples 18.3 -> 10.5 ms (a leaf of 32 pixels spans 0.5 rad there and four
// tenths of the pairs stay near), N_side 128 with 25,087 170 -> 41 ms.  Error against the oracle 1.2e-16
// to 1.9e-16 of the rms (direct kernel 0.5e-16 to 1.2e-16), largest 1.9e-15 (1.0e-15).
// ------------------------------------------------------------------------------------
constexpr int kNP64 = 16, kNN64 = kNP64 * kNP64, kLeaf64 = 32;
constexpr int kNodeTarget64 = 32, kPixTarget64 = 12;

// A staged Far64 record.
struct __align__(16) Stage64 {
    double v[16];
};
static_assert(sizeof(Far64) <= sizeof(Stage64) && sizeof(Far64) % 16 == 0, "stage layout");

// the interpolant with the shared coefficients at (x, y) in [-1, 1]^2: Clenshaw's recurrence in y, rows
// added from the highest order down
__device__ __forceinline__ double interp64(const double *coef, double x, double y)
{
    double tx[kNP64];
    tx[0] = 1.0;
    tx[1] = x;
#pragma unroll
    for (int i = 2; i < kNP64; ++i) tx[i] = fma(2.0 * x, tx[i - 1], -tx[i - 2]);
    const double y2 = 2.0 * y;
    double b1 = 0.0, b2 = 0.0, r = 0.0;
#pragma unroll 1
    for (int j = kNP64 - 1; j >= 0; --j) {
        r = 0.0;
#pragma unroll
        for (int i = kNP64 - 1; i >= 0; --i) r = fma(coef[j * kNP64 + i], tx[i], r);
        if (j > 0) {
            const double t = fma(y2, b1, r - b2);
            b2 = b1;
            b1 = t;
        }
    }
    return fma(y, b1, r - b2);
}

// [-1, 1]^2 coordinates in frame g of the direction at offset (dx, dy, dz) from its centre
__device__ __forceinline__ void local_xy64(const TreeGeo &g, double dx, double dy, double dz, double &x, double &y)
{
    const double s = 1.0 / (2.0 - 0.5 * (dx * dx + dy * dy + dz * dz));
    x = (dx * g.e1[0] + dy * g.e1[1] + dz * g.e1[2]) * (s / g.a1);
    y = (dx * g.e2[0] + dy * g.e2[1] + dz * g.e2[2]) * (s / g.a2);
}

// Values of cluster cl at its nodes, kept as (hi, lo) pairs [slot][2][256] -> the value of a middle node as a
// pair and the Chebyshev coefficients of the differences from it (shared).  The differences are a fraction of
// the values, so the interpolation's rounding stays below that of the value itself.
__device__ __forceinline__ void cheb_coefs64(const double *__restrict__ F, const TreeWork &W, int64_t cl, double *coef,
                                             double *tmp, double &rhi, double &rlo)
{
    const int nch = W.nch[cl];
    const int64_t at = nch == 1 ? cl : W.ncl + W.pbase[cl];
    for (int k = threadIdx.x; k < kNN64; k += kTreeNT) {
        double hi = 0.0, lo = 0.0;
        for (int c = 0; c < nch; ++c) {
            const double *f = F + (at + c) * 2 * kNN64 + k;
            fold64(hi, lo, f[0]);
            lo += f[kNN64];
        }
        coef[k] = hi;
        tmp[k] = lo;
    }
    __syncthreads();
    constexpr int kMid = kNN64 / 2 + kNP64 / 2;
    rhi = coef[kMid];
    rlo = tmp[kMid];
    double d[kNN64 / kTreeNT];
#pragma unroll
    for (int q = 0; q < kNN64 / kTreeNT; ++q) {
        const int k = q * kTreeNT + threadIdx.x;
        d[q] = (coef[k] - rhi) + (tmp[k] - rlo);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kNN64 / kTreeNT; ++q) coef[q * kTreeNT + threadIdx.x] = d[q];
    __syncthreads();
    cheb_transform<kNP64>(coef, tmp);
}

// Copies the staged batch: eval(batch start, size) runs with sm.rec filled; whole block.
template <typename Smem, typename Stage, typename Eval>
__device__ __forceinline__ void tree_batches64(Smem &sm, int count, Stage &&stage, Eval &&eval)
{
#pragma unroll 1
    for (int b0 = 0; b0 < count; b0 += kTreeBatch) {
        if (b0 + (int)threadIdx.x < count) stage(sm.scan.list[b0 + threadIdx.x], sm.rec[threadIdx.x]);
        __syncthreads();
        eval(count - b0 < kTreeBatch ? count - b0 : kTreeBatch);
        __syncthreads();
    }
}

// Far-field pair term (17 FP64 operations, see k_map_f64)
__device__ __forceinline__ double far_term64(const Far64 &r, double nx, double ny, double nz, double acc)
{
    const double hs = fma(nz, r.mxh[2], fma(ny, r.mxh[1], fma(nx, r.mxh[0], r.sg)));
    const double B = fma(nz, r.xd[2], fma(ny, r.xd[1], fma(nx, r.xd[0], 1.0)));
    const double A2 = fma(nz, r.xp[2], fma(ny, r.xp[1], fma(nx, r.xp[0], r.af)));
    const double B2 = fma(r.sx, B, r.be);
    const double num = fma(-A2, A2, fma(B2, B2, -r.K));
    return fma(num, rcp64(B * hs), acc);
}

struct TreeNodeArgs64 {
    TreeNodeArgs n;
    const Seg64 *s64;
};

// Node (xi, eta) of a cluster is n0 + (xi e1 + eta e2 - r^2 n0) / w with r^2 = xi^2 + eta^2 and w = (1 + r^2) / 2,
// so w times anything linear in n is a polynomial in xi plus one in eta:
//   w (a + v.m) = [a/2 + xi v.e1 + xi^2 (a/2 - v.n0)] + [eta v.e2 + eta^2 (a/2 - v.n0)],
// and w |d|^2 likewise (|m|^2 w = 2 r^2).  The pair term is a quotient of degree 2 over degree 2 in such forms: w
// cancels.  With the 2 x 16 values of the five forms |d|^2, B, c Xdot.d, A and c X'.d in tables per sample, a
// node costs five additions and 12 FP64 operations in all (18 to 21 from the node's offset), the tables
// one per node.  Offsets and not directions: the rounding of a direction moves a node by 5e-17, and the
// interpolant's values by that times the slope (2e-16 of the rms).
constexpr int kForms64 = 5, kTabBatch = 16;
struct __align__(16) NodeCoef64 {
    double v[kForms64][4], pad[2];   // constant, xi, eta, square; odd multiple of 16 bytes
};
struct __align__(16) NodeForms64 {
    double v[kForms64 + 1];
};
struct __align__(16) TreeNodeSmem64 {
    NodeCoef64 rec[kTreeBatch];
    NodeForms64 tab[kTabBatch][2 * kNP64];
    TreeScanSmem scan;
    TreeGeo geo, pgeo;
    double coef[kNN64], tmp[kNN64];
    int64_t item;
};

// Two nodes per thread.  Bound by the FP64 unit (85% busy); N_side 128 with 25,087 samples, both levels: 20.6 ms
// from the nodes' offsets, 15.9 ms from tables.
template <bool ROOT>
__global__ void __launch_bounds__(kTreeNT) k_tree_nodes_f64(TreeNodeArgs64 A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TreeNodeSmem64 &sm = *reinterpret_cast<TreeNodeSmem64 *>(smem_raw);
    const TreeNodeArgs &a = A.n;
    const int tid = threadIdx.x, lane = tid & 31;
    const int np = *a.W.npool;
    TreeQueue queue{a.queue, 0ull};
    for (int64_t item = queue.first(&sm.item); item < a.W.ncl + np; item = queue.next(&sm.item)) {
        int kc, nch;
        int64_t at;
        const int64_t cl = tree_item(a.W, item, np, kc, nch, at);
        if (cl < 0) continue;
        const int64_t pcl = ROOT ? 0 : tree_parent(cl, a.nb, a.pnb);
        if (!ROOT) load_geo(&sm.pgeo, a.pgeo + pcl);
        load_geo(&sm.geo, a.geo + cl);
        __syncthreads();
        const float4 self = sm.geo.c, parent = ROOT ? self : sm.pgeo.c;
        if (tree_empty(self)) continue;
        double hi[2] = {0.0, 0.0}, lo[2] = {0.0, 0.0};
        const double xt = ((lane & 8) == 0 ? sm.geo.a1 : sm.geo.a2) * cheb_at<kNP64>(1, lane & 7), x2 = xt * xt;
        auto stage = [&](uint32_t e, NodeCoef64 &d) {
            const Seg64 &s = A.s64[e];
            const double *n0 = sm.geo.n0, *e1 = sm.geo.e1, *e2 = sm.geo.e2;
            double D[3], P = 0.0, Q = 0.0, K = 0.0, B0 = 1.0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                D[c] = (n0[c] - s.xh[c]) - s.xl[c];
                P = fma(s.xd[c], D[c], P);
                Q = fma(s.xp[c], D[c], Q);
                K = fma(D[c], D[c], K);
                B0 = fma(s.xd[c], n0[c], B0);
            }
            const double f = s.xp[0] * s.xh[0] + s.xp[1] * s.xh[1] + s.xp[2] * s.xh[2];   // X'.Xhat
            auto dot = [](const double *u, const double *v) { return fma(u[2], v[2], fma(u[1], v[1], u[0] * v[0])); };
            auto put = [&](int k, double con, double x, double y, double sq) {
                d.v[k][0] = con;
                d.v[k][1] = x;
                d.v[k][2] = y;
                d.v[k][3] = sq;
            };
            put(0, 0.5 * K, 2.0 * dot(D, e1), 2.0 * dot(D, e2), 2.0 + fma(-2.0, dot(D, n0), 0.5 * K));
            const double p0 = dot(s.xd, n0), p1 = dot(s.xd, e1), p2 = dot(s.xd, e2);
            put(1, 0.5 * B0, p1, p2, fma(0.5, B0, -p0));
            put(2, s.c * (0.5 * P), s.c * p1, s.c * p2, s.c * fma(0.5, P, -p0));
            const double q0 = dot(s.xp, n0), q1 = dot(s.xp, e1), q2 = dot(s.xp, e2), A0 = f + Q;
            put(3, 0.5 * A0, q1, q2, fma(0.5, A0, -q0));
            put(4, s.c * (0.5 * Q), s.c * q1, s.c * q2, s.c * fma(0.5, Q, -q0));
        };
        auto eval = [&](int cnt) {
            double part[2] = {0.0, 0.0};
#pragma unroll 1
            for (int b0 = 0; b0 < cnt; b0 += kTabBatch) {
                const int nb = cnt - b0 < kTabBatch ? cnt - b0 : kTabBatch;
                if (b0 > 0) __syncthreads();
#pragma unroll 1
                for (int s = tid >> 4; s < nb; s += kTreeNT / 16) {   // entries for xt and -xt
                    const NodeCoef64 &c = sm.rec[b0 + s];
                    const bool xi = (lane & 8) == 0;
                    NodeForms64 *t = sm.tab[s] + (xi ? 0 : kNP64);
#pragma unroll
                    for (int k = 0; k < kForms64; ++k) {
                        const double2 u = *reinterpret_cast<const double2 *>(&c.v[k][0]), v = *reinterpret_cast<const double2 *>(&c.v[k][2]);
                        const double even = fma(x2, v.y, xi ? u.x : 0.0), lin = xi ? u.y : v.x;
                        t[lane & 7].v[k] = fma(xt, lin, even);
                        t[kNP64 - 1 - (lane & 7)].v[k] = fma(-xt, lin, even);
                    }
                }
                __syncthreads();
#pragma unroll 2
                for (int s = 0; s < nb; ++s) {
                    const NodeForms64 F = sm.tab[s][tid % kNP64];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const NodeForms64 G = sm.tab[s][kNP64 + q * (kTreeNT / kNP64) + tid / kNP64];
                        const double Q = F.v[0] + G.v[0], B = F.v[1] + G.v[1], Pd = F.v[2] + G.v[2];
                        const double An = F.v[3] + G.v[3], Qd = F.v[4] + G.v[4];
                        part[q] = fma(fma(B, Pd, -(An * Qd)), rcp64(B * Q), part[q]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) fold64(hi[q], lo[q], part[q]);
        };
        tree_scan<ROOT, false>(a.S, kc, nch, self, parent, 0.f, 0.f, 0.f, sm.scan,
                               [&](int count) { tree_batches64(sm, count, stage, eval); });
        if (!ROOT && kc == 0 && !tree_wide(parent)) {
            double rhi, rlo;
            cheb_coefs64(a.Fp, a.Wp, pcl, sm.coef, sm.tmp, rhi, rlo);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int k = q * kTreeNT + tid;
                const double xi = sm.geo.a1 * cheb_at<kNP64>(1, k % kNP64), eta = sm.geo.a2 * cheb_at<kNP64>(1, k / kNP64);
                const double r2 = xi * xi + eta * eta, s = 2.0 / (1.0 + r2);
                double m[3], x, y;
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    m[c] = (sm.geo.n0[c] - sm.pgeo.n0[c]) + s * (xi * sm.geo.e1[c] + eta * sm.geo.e2[c] - r2 * sm.geo.n0[c]);
                local_xy64(sm.pgeo, m[0], m[1], m[2], x, y);
                fold64(hi[q], lo[q], rhi);
                fold64(hi[q], lo[q], interp64(sm.coef, x, y));
                lo[q] += rlo;
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            a.F[at * 2 * kNN64 + q * kTreeNT + tid] = hi[q];
            a.F[(at * 2 + 1) * kNN64 + q * kTreeNT + tid] = lo[q];
        }
        __syncthreads();
    }
}

struct TreePixArgs64 {
    TreePixArgs p;
    const Far64 *far64;
    float d_far;
    int64_t nside;   // full-sky maps
    int nb;
    int parts;       // items of a cluster (and chunk): 1, or 4 with a block per warp each
};

// Ring form of the far-field pair term.  A pixel of a ring (z, s = sin theta) at azimuth phi has n / s =
// (cos phi, sin phi, z / s), so a linear form over s is a function of the ring plus one of the azimuth, and the
// quotient of degree 2 over degree 2 does not change.  On an equatorial leaf pixel (x, y) has ring x + y and
// azimuth x - y: tables of 63 + 63 values per sample leave 11 FP64 operations per pixel of 17.  A polar pixel
// has its own azimuth and takes two operations per form in the place of three (14).  The tables cost 0.8 per
// pixel.
// |d|^2 / (2 s) = [(z - zX)^2 + (s - sX)^2] / (2 s) + sX |u - uX|^2 / 2 with azimuth directions u and uX: a sum
// of squares, so that it keeps its relative accuracy next to the sample, where 1 - n.Xhat cancels (error of
// a map 3.1e-16 of the rms with that, 1.9e-16 with the squares); a block of polar pixels away from the sample
// takes - uX.u for the last square.
constexpr int kRings = 2 * kLeaf64 - 1, kTabPix = 4;
struct __align__(16) RingForms {
    double v[6];   // sigma |d|^2 / 2, B, s A - s f/2 (see Far64), -s e/2, -K; the first for the other azimuth part
};
struct __align__(16) AzForms {
    double v[4];   // the first three's azimuth parts
};
// A block of pixels: two slots of every lane of a warp
constexpr int kPix64 = kLeaf64 * kLeaf64 / kTreeNT, kBlocks64 = kPix64 / 2;

struct __align__(16) TreePixSmem64 {
    Stage64 rec[kTreeBatch];
    union {
        double n[3][kLeaf64 * kLeaf64];   // lists and patches: directions
        struct {
            double2 u[kLeaf64 * kLeaf64];   // (cos phi, sin phi)
            RingForms F[kTabPix][kRings + 1];
            AzForms G[kTabPix][kRings + 1];
        } sky;
    };
    double ring[5][kRings + 1], az[2][kRings + 1];   // z, s, 1/s, z/s, 1/s^2; cos, sin
    float4 cap[kTreeNT / 32][kBlocks64];
    TreeScanSmem scan;
    TreeGeo geo;
    double coef[kNN64], tmp[kNN64];
    int64_t item;
};

// Ring of the table, 0 .. 2 T - 2, and place of the azimuth: even ones first, a warp's pixels then lie in
// neighbouring entries
__device__ __forceinline__ int az_place(int l) { return (l >> 1) + (l & 1) * kLeaf64; }

// Eight pixels per thread, one cluster per item, or a quarter of one with fewer than two (cluster, sample
// tile) pairs for every CTA slot (N_side 64 with 1,000 samples 2.6 -> 2.2 ms, N_side 16 with 250 1.2 -> 0.6;
// with 2,500 samples at N_side 64 the quarters' tables cost more, 3.4 -> 4.4): four blocks of 8 x 8 pixels per warp (full sky) or of 64
// consecutive slots.  Bound by the FP64 unit.  N_side 64 with 10,240 samples 10.2 ms with 17 operations for every
// pixel -> 8.4 ms, N_side 128 with 30,001 33.5 -> 26.7 ms.  Samples that the cluster's test flags are tested again per block: with |d| >= d_far and
// B >= b_min on the block they too take the far-field form (its squares cancel to a factor 1/B of the rounding),
// else the pair term from the double-double Xhat (29 operations).
template <bool SKY>
__global__ void __launch_bounds__(kTreeNT, 3) k_tree_pixels_f64(TreePixArgs64 A)
{
    constexpr int TILE = kLeaf64 * kLeaf64, P = kPix64;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TreePixSmem64 &sm = *reinterpret_cast<TreePixSmem64 *>(smem_raw);
    const TreePixArgs &a = A.p;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int np = *a.W.npool;
    unsigned zerocnt = 0;
    TreeQueue queue{a.queue, 0ull};
    const int per = kBlocks64 / A.parts;   // blocks per warp of an item
    for (int64_t it = queue.first(&sm.item); it < (a.W.ncl + np) * A.parts; it = queue.next(&sm.item)) {
        int kc, nch;
        int64_t at;
        const int64_t item = it / A.parts;
        const int pb = (int)(it - item * A.parts) * per;   // first block
        const int64_t cl = tree_item(a.W, item, np, kc, nch, at);
        if (cl < 0) continue;
        if (!SKY && tree_empty(a.geo[cl].c)) continue;
        load_geo(&sm.geo, a.geo + cl);
        const int64_t k0 = cl * TILE;
        int slot[P], place[P];   // slot in the cluster; SKY: ring and azimuth entries
        unsigned valid = 0, eq = 0, live = 0;   // live: blocks of this item that have pixels
        if (SKY) {
            const int64_t N = A.nside, f = cl / ((int64_t)A.nb * A.nb), rem = cl - f * A.nb * A.nb;
            const int64_t y0 = rem / A.nb * kLeaf64, x0 = rem % A.nb * kLeaf64;
            const int64_t jr0 = (f < 4 ? 2 : f < 8 ? 3 : 4) * N - x0 - y0 - 1;   // HEALPix ring of entry r: jr0 - r
            if (tid < kRings) {
                const int64_t jr = jr0 - tid, i = jr < N ? jr : jr > 3 * N ? 4 * N - jr : N;
                const double N3 = 3.0 * (double)N;
                double z, st;
                if (jr < N || jr > 3 * N) {
                    const double q = (double)(i * i) / (N3 * (double)N);
                    z = jr < N ? 1.0 - q : q - 1.0;
                    st = sqrt((double)(6 * N * N - i * i)) * (double)i / (N3 * (double)N);
                } else {
                    z = (double)(4 * N - 2 * jr) / N3;
                    st = sqrt((double)((2 * jr - N) * (7 * N - 2 * jr))) / N3;
                }
                if (!(i > 0)) z = 0.0, st = 1.0;   // past the pole: padding only
                const double iw = 1.0 / st;
                sm.ring[0][tid] = z;
                sm.ring[1][tid] = st;
                sm.ring[2][tid] = iw;
                sm.ring[3][tid] = z * iw;
                sm.ring[4][tid] = iw * iw;
            } else if (tid >= 64 && tid - 64 < kRings) {
                const int l = tid - 64;
                const int64_t jp = f < 4 ? 2 * f + 1 : f < 8 ? 2 * (f - 4) : 2 * (f - 8) + 1;
                double sp, cp;
                sincospi_frac(jp * N + x0 - y0 + l - (kLeaf64 - 1), 4 * N, sp, cp);
                sm.az[0][az_place(l)] = cp;
                sm.az[1][az_place(l)] = sp;
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const int blk = w * kBlocks64 + q / 2, lx = blk % 4 * 8 + (lane & 7), ly = blk / 4 * 8 + q % 2 * 4 + (lane >> 3);
                slot[q] = diag_index_square(lx, ly, kLeaf64);
                place[q] = (lx + ly) | az_place(lx - ly + kLeaf64 - 1) << 8;
                const int64_t jr = jr0 - lx - ly;
                if (__all_sync(0xffffffffu, jr >= N && jr <= 3 * N)) eq |= 1u << q;
                if (a.outidx[k0 + slot[q]] >= 0) valid |= 1u << q;
                const double iw = sm.ring[2][lx + ly];
                sm.sky.u[q * kTreeNT + tid] = make_double2(a.nv[k0 + slot[q]] * iw, a.nv[a.ldn + k0 + slot[q]] * iw);
            }
        } else {
#pragma unroll
            for (int q = 0; q < P; ++q) {
                slot[q] = (w * P + q) * 32 + lane;
                place[q] = 0;
                if (a.outidx[k0 + slot[q]] >= 0) valid |= 1u << q;
#pragma unroll
                for (int c = 0; c < 3; ++c) sm.n[c][q * kTreeNT + tid] = a.nv[c * a.ldn + k0 + slot[q]];
            }
        }
        // balls of the blocks (radius < 0: no pixel)
#pragma unroll
        for (int p = 0; p < kBlocks64; ++p) {
            float4 x[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int64_t k = k0 + slot[2 * p + u];
                x[u] = make_float4((float)a.nv[k], (float)a.nv[a.ldn + k], (float)a.nv[2 * a.ldn + k],
                                   valid >> (2 * p + u) & 1 ? 0.f : -1.f);
            }
            const TreeCap c = warp_ball(x);
            if (lane == 0) sm.cap[w][p] = c.a;
            if (c.a.w >= 0.f && p >= pb && p < pb + per) live |= 1u << p;
        }
        __syncthreads();
        const float4 self = sm.geo.c;
        double hi[P], lo[P];
#pragma unroll
        for (int q = 0; q < P; ++q) hi[q] = lo[q] = 0.0;
        auto stage = [&](uint32_t e, Stage64 &d) {
            const double2 *src = reinterpret_cast<const double2 *>(A.far64 + (e & kTreeIndex));
#pragma unroll
            for (int k = 0; k < (int)sizeof(Far64) / 16; ++k) reinterpret_cast<double2 *>(d.v)[k] = src[k];
            if (SKY) {   // sigma sX, sigma / (2 sX)
                const double sX = sqrt(fma(d.v[1], d.v[1], d.v[0] * d.v[0]));
                d.v[14] = copysign(sX, d.v[3]);
                d.v[15] = sX > 0.0 ? 0.5 / d.v[14] : 0.0;
            }
        };
        // the far-field form at one block
        auto far_block = [&](const Stage64 &rec, int p, int ts, bool close, double &p0, double &p1) {
            double *const part[2] = {&p0, &p1};
            const Far64 &r = *reinterpret_cast<const Far64 *>(rec.v);
            if (SKY) {
                const bool e2 = (eq >> (2 * p) & 3) == 3;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int q = 2 * p + u;
                    const RingForms &F = sm.sky.F[ts][place[q] & 0xff];
                    double hs, B, A2;
                    if (e2) {
                        const AzForms &G = sm.sky.G[ts][place[q] >> 8];
                        hs = F.v[0] + G.v[0];
                        B = F.v[1] + G.v[1];
                        A2 = F.v[2] + G.v[2];
                    } else {
                        const double2 n = sm.sky.u[q * kTreeNT + tid];
                        if (close) {
                            const double *v = rec.v;
                            const double x = fma(v[14], n.x, v[0]), y = fma(v[14], n.y, v[1]);
                            hs = fma(v[15], fma(y, y, x * x), F.v[0]);
                        } else {
                            hs = fma(n.y, r.mxh[1], fma(n.x, r.mxh[0], F.v[5]));
                        }
                        B = fma(n.y, r.xd[1], fma(n.x, r.xd[0], F.v[1]));
                        A2 = fma(n.y, r.xp[1], fma(n.x, r.xp[0], F.v[2]));
                    }
                    const double B2 = fma(r.sx, B, F.v[3]);
                    *part[u] = fma(fma(-A2, A2, fma(B2, B2, F.v[4])), rcp64(B * hs), *part[u]);
                }
            } else {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int i = (2 * p + u) * kTreeNT + tid;
                    *part[u] = far_term64(r, sm.n[0][i], sm.n[1][i], sm.n[2][i], *part[u]);
                }
            }
        };
        auto near_block = [&](const Seg64 &g, int p, double &p0, double &p1) {
            double *const part[2] = {&p0, &p1};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int q = 2 * p + u;
                const int64_t k = k0 + slot[q];
                const double nx = a.nv[k], ny = a.nv[a.ldn + k], nz = a.nv[2 * a.ldn + k];
                const double dx = (nx - g.xh[0]) - g.xl[0], dy = (ny - g.xh[1]) - g.xl[1], dz = (nz - g.xh[2]) - g.xl[2];
                const double Q = fma(dz, dz, fma(dy, dy, dx * dx));
                const double Pd = fma(g.xd[2], dz, fma(g.xd[1], dy, g.xd[0] * dx));
                const double Qd = fma(g.xp[2], dz, fma(g.xp[1], dy, g.xp[0] * dx));
                // A and B from n itself: 1 + Xdot.Xhat + Xdot.d would round a small B twice
                const double An = nx * g.xp[0] + ny * g.xp[1] + nz * g.xp[2];
                const double B = 1.0 + (nx * g.xd[0] + ny * g.xd[1] + nz * g.xd[2]);
                const double num = B * Pd - An * Qd, den = B * Q;
                // the estimate of the reciprocal needs a normal value
                const int ex = __double2hiint(den) & 0x7ff00000;
                if (ex > 0x39b00000 && ex < 0x46000000) {
                    *part[u] = fma(g.c * num, rcp64(den), *part[u]);
                } else if (Q == 0.0) {
                    if (valid >> q & 1) ++zerocnt;
                } else {
                    *part[u] += g.c * num / den;
                }
            }
        };
        // whether a flagged sample may take the far-field form on block p
        auto far_on = [&](const float4 xh, const float4 bm, int p) {
            const float4 c = sm.cap[w][p];
            float x = c.x - xh.x, y = c.y - xh.y, z = c.z - xh.z;
            const float d = sqrtf(x * x + y * y + z * z) - c.w;
            x = c.x - bm.x, y = c.y - bm.y, z = c.z - bm.z;
            const float h = fmaxf(sqrtf(x * x + y * y + z * z) - c.w, 0.f);
            return (d >= A.d_far && fmaf(0.5f * (1.f - bm.w) * h, h, bm.w) >= a.b_min);
        };
        int l0 = 0;   // list position of the batch
        auto eval = [&](int cnt) {
            double part[P];
#pragma unroll
            for (int q = 0; q < P; ++q) part[q] = 0.0;
#pragma unroll 1
            for (int b0 = 0; b0 < cnt; b0 += kTabPix) {
                const int nb = cnt - b0 < kTabPix ? cnt - b0 : kTabPix;
                if (SKY) {
                    if (b0 > 0) __syncthreads();
                    if (tid < kRings) {
                        const double z = sm.ring[0][tid], st = sm.ring[1][tid], iw = sm.ring[2][tid], zw = sm.ring[3][tid],
                                     iw2 = sm.ring[4][tid];
                        for (int s = 0; s < nb; ++s) {
                            const Far64 &r = *reinterpret_cast<const Far64 *>(sm.rec[b0 + s].v);
                            RingForms &F = sm.sky.F[s][tid];
                            const double S = sm.rec[b0 + s].v[14], x = fma(r.sg, z, r.mxh[2]), y = fma(r.sg, st, -S);
                            const double h = fma(y, y, x * x) * (0.5 * r.sg * iw);
                            F.v[0] = h;
                            F.v[5] = h + S;
                            F.v[1] = fma(r.xd[2], zw, iw);
                            F.v[2] = fma(r.xp[2], zw, r.af * iw);
                            F.v[3] = r.be * iw;
                            F.v[4] = -r.K * iw2;
                        }
                    } else if (tid >= 64 && tid - 64 < kRings) {
                        const double c = sm.az[0][tid - 64], d = sm.az[1][tid - 64];
                        for (int s = 0; s < nb; ++s) {
                            const Far64 &r = *reinterpret_cast<const Far64 *>(sm.rec[b0 + s].v);
                            AzForms &G = sm.sky.G[s][tid - 64];
                            const double *v = sm.rec[b0 + s].v;
                            const double x = fma(v[14], c, v[0]), y = fma(v[14], d, v[1]);
                            G.v[0] = v[15] * fma(y, y, x * x);
                            G.v[1] = fma(r.xd[1], d, r.xd[0] * c);
                            G.v[2] = fma(r.xp[1], d, r.xp[0] * c);
                        }
                    }
                    __syncthreads();
                }
#pragma unroll 1
                for (int s = 0; s < nb; ++s) {
                    const uint32_t e = sm.scan.list[l0 + b0 + s];
                    const Stage64 &r = sm.rec[b0 + s];
                    if (!(e & (kTreeClose | kTreeBeam))) {
#pragma unroll
                        for (int p = 0; p < kBlocks64; ++p)
                            if (live >> p & 1u) far_block(r, p, s, false, part[2 * p], part[2 * p + 1]);
                        continue;
                    }
                    const float4 xh = a.S.crit[e & kTreeIndex].a, bm = a.S.crit[e & kTreeIndex].b;
#pragma unroll
                    for (int p = 0; p < kBlocks64; ++p) {
                        if (!(live >> p & 1u)) continue;
                        if (far_on(xh, bm, p)) far_block(r, p, s, true, part[2 * p], part[2 * p + 1]);
                        else near_block(a.s64[e & kTreeIndex], p, part[2 * p], part[2 * p + 1]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < P; ++q) fold64(hi[q], lo[q], part[q]);
        };
        const float R = target_radius(sm.geo);
        tree_scan<false, true>(a.S, kc, nch, self, self, R, A.d_far + R, a.b_min, sm.scan, [&](int count) {
            l0 = 0;
            tree_batches64(sm, count, stage, [&](int cnt) {
                eval(cnt);
                l0 += kTreeBatch;
            });
        });
        double rhi = 0.0, rlo = 0.0;
        const bool inner = kc == 0 && !tree_wide(self);
        if (inner) cheb_coefs64(a.F, a.Wf, cl, sm.coef, sm.tmp, rhi, rlo);
#pragma unroll
        for (int q = 0; q < P; ++q) {
            if (q / 2 < pb || q / 2 >= pb + per) continue;
            const int64_t k = k0 + slot[q];
            if (inner && live >> q / 2 & 1u) {
                double x, y;
                local_xy64(sm.geo, a.nv[k] - sm.geo.n0[0], a.nv[a.ldn + k] - sm.geo.n0[1], a.nv[2 * a.ldn + k] - sm.geo.n0[2], x, y);
                fold64(hi[q], lo[q], rhi);
                fold64(hi[q], lo[q], interp64(sm.coef, x, y));
                lo[q] += rlo;
            }
            const double v = hi[q] + lo[q];
            if (nch == 1) {
                const int64_t oi = a.outidx[k];
                if (oi >= 0) a.theta[oi] = a.accumulate ? a.theta[oi] + v : v;
            } else {
                a.partial[item * TILE + slot[q]] = v;   // pool entry of the chunk
            }
        }
        __syncthreads();
    }
    for (int o = 16; o > 0; o >>= 1) zerocnt += __shfl_xor_sync(0xffffffffu, zerocnt, o);
    if (lane == 0 && zerocnt) atomicAdd(&a.st->zero_pairs, (unsigned long long)zerocnt);
}

}  // namespace

int tree_leaf(int prec) { return prec == ISW_F64 ? kLeaf64 : kLeaf; }

TreePlan tree_plan(int prec, int64_t N, int nface, int64_t npix, int64_t n, int num_sms)
{
    TreePlan p{};
    const bool f64 = prec == ISW_F64;
    p.prec = prec;
    p.leaf = tree_leaf(prec);
    p.nn = f64 ? 2 * kNN64 : kNN;   // doubles per cluster
    p.n_pad = (n + kTreeS - 1) / kTreeS * kTreeS;
    p.nst = p.n_pad / kTreeS;
    p.nslots = f64 ? std::min(slots_of((const void *)&k_tree_nodes_f64<false>, sizeof(TreeNodeSmem64), num_sms),
                              slots_of((const void *)&k_tree_nodes_f64<true>, sizeof(TreeNodeSmem64), num_sms))
                   : slots_of((const void *)&k_tree_nodes_f32<false>, sizeof(TreeSmem32), num_sms);
    p.pslots = f64 ? std::min(slots_of((const void *)&k_tree_pixels_f64<false>, sizeof(TreePixSmem64), num_sms),
                              slots_of((const void *)&k_tree_pixels_f64<true>, sizeof(TreePixSmem64), num_sms))
                   : slots_of((const void *)&k_tree_pixels_f32, sizeof(TreeSmemPix), num_sms);
    int64_t all = 0;
    int64_t nb = nface > 0 ? (N + p.leaf - 1) / p.leaf : 0;
    int64_t ncl = nface > 0 ? nface * nb * nb : (npix + p.leaf * p.leaf - 1) / (p.leaf * p.leaf);
    for (;;) {
        const int L = p.levels++;
        p.nb[L] = (int)nb;
        p.ncl[L] = ncl;
        all += ncl;
        if ((nface > 0 ? nb <= 2 : ncl <= 48) || p.levels == kTreeLevels) break;
        nb = (nb + 1) / 2;
        ncl = nface > 0 ? nface * nb * nb : (ncl + 3) / 4;
    }
    all += p.ncl[0];
    p.pool = (f64 ? 16 : 8) * p.nslots;
    p.ppool = (f64 ? 16 : 8) * p.pslots;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += up256(bytes);
        return o;
    };
    p.off_queue = take(kTreeZero);   // zeroed per call
    p.off_crit = take((size_t)p.n_pad * sizeof(TreeCrit));
    p.off_vcrit = take((size_t)p.n_pad * sizeof(TreeCrit));
    p.off_caps = take((size_t)2 * p.nst * sizeof(TreeCap));
    p.off_sup = take((size_t)2 * ((p.nst + kTreeSuper - 1) / kTreeSuper) * sizeof(TreeCap));
    p.off_vidx = take((size_t)p.n_pad * sizeof(uint32_t));
    p.off_inv = take((size_t)n * sizeof(uint32_t));
    p.off_rec = f64 ? 0 : take((size_t)p.n_pad * sizeof(TreeRec));
    p.off_work = take((size_t)3 * all * sizeof(int));
    p.off_pool = take(((size_t)p.levels * p.pool + p.ppool) * sizeof(int2));
    p.off_partial = take((size_t)p.ppool * p.leaf * p.leaf * sizeof(double));
    for (int L = 0; L < p.levels; ++L) {
        p.off_geo[L] = take((size_t)p.ncl[L] * sizeof(TreeGeo));
        p.off_F[L] = take((size_t)(p.ncl[L] + p.pool) * p.nn * sizeof(double));
    }
    p.bytes = at;
    return p;
}

cudaError_t launch_map_tree(const TreePlan &p, const TreeMapArgs &m, cudaStream_t s)
{
    const bool f64 = p.prec == ISW_F64;
    const double kappa = f64 ? kKappa64 : kKappa32;
    unsigned char *b = (unsigned char *)m.scratch;
    TreeCrit *crit = (TreeCrit *)(b + p.off_crit), *vcrit = (TreeCrit *)(b + p.off_vcrit);
    TreeCap *caps = (TreeCap *)(b + p.off_caps), *sup = (TreeCap *)(b + p.off_sup);
    uint32_t *vidx = (uint32_t *)(b + p.off_vidx), *inv = (uint32_t *)(b + p.off_inv);
    TreeRec *rec = f64 ? nullptr : (TreeRec *)(b + p.off_rec);
    unsigned long long *queue = (unsigned long long *)(b + p.off_queue), *total = queue + kTreeLevels + 1;
    int *npool = (int *)(total + (kTreeLevels + 1) * kTargets);
    cudaError_t e = cudaMemsetAsync(queue, 0, kTreeZero, s);
    if (e != cudaSuccess) return e;
    const unsigned tb = (unsigned)((p.nst * 32 + 255) / 256);
    k_tree_crit<<<tb, 256, 0, s>>>(m.s32, m.s64, m.perm, m.n, p.nst, crit, caps, rec, inv);
    k_tree_vcrit<<<tb, 256, 0, s>>>(crit, m.s32, m.perm + m.n, inv, m.n, p.nst, vcrit, caps + p.nst, vidx);
    const int64_t nsup = (p.nst + kTreeSuper - 1) / kTreeSuper;
    k_tree_super<<<dim3((unsigned)((nsup + 3) / 4), 2), 128, 0, s>>>(caps, p.nst, nsup, sup);
    const TreeSamples S{crit, vcrit, caps, caps + p.nst, sup, sup + nsup, vidx, p.nst};
    TreeGeo *leaf_geo = (TreeGeo *)(b + p.off_geo[0]);
    if (f64)
        launch_leaf_geo<kLeaf64>(m.nv, m.ldn, m.outidx, m.order, m.theta_pix, kappa, p.ncl[0], leaf_geo, s);
    else
        launch_leaf_geo<kLeaf>(m.nv, m.ldn, m.outidx, m.order, m.theta_pix, kappa, p.ncl[0], leaf_geo, s);
    for (int L = 1; L < p.levels; ++L)
        launch_up_geo((const TreeGeo *)(b + p.off_geo[L - 1]), p.nb[L - 1], p.ncl[L - 1], (TreeGeo *)(b + p.off_geo[L]), p.nb[L], p.ncl[L], kappa, s);
    // stages 0 .. levels - 1: node sums of the level; stage `levels`: the pixels
    TreeStages g{};
    g.n = p.levels + 1;
    int2 *entries = (int2 *)(b + p.off_pool);
    for (int st = 0; st <= p.levels; ++st) {
        const bool pix = st == p.levels;
        const int L = pix ? 0 : st;
        g.first[st + 1] = g.first[st] + p.ncl[L];
        g.geo[st] = (const TreeGeo *)(b + p.off_geo[L]);
        g.nb[st] = p.nb[L];
        if (st + 1 < p.levels) {
            g.pgeo[st] = (const TreeGeo *)(b + p.off_geo[st + 1]);
            g.pnb[st] = p.nb[st + 1];
        }
        g.pool[st] = pix ? p.ppool : p.pool;
        g.target[st] = f64 ? (pix ? kPixTarget64 : kNodeTarget64) : (pix ? kPixTarget : kNodeTarget);
        g.entries[st] = entries + (size_t)st * p.pool;
    }
    const int64_t all = g.first[g.n];
    int *est = (int *)(b + p.off_work), *nch = est + all, *pbase = nch + all;
    k_tree_count<<<(unsigned)((all + 3) / 4), 128, 0, s>>>(g, S, m.n, est, total);
    k_tree_plan<<<(unsigned)((all + 127) / 128), 128, 0, s>>>(g, est, total, nch, pbase, npool);
    auto work = [&](int st) {
        return TreeWork{nch + g.first[st], pbase + g.first[st], g.entries[st], npool + st, g.first[st + 1] - g.first[st]};
    };
    for (int L = p.levels - 1; L >= 0; --L) {
        const bool root = L == p.levels - 1;
        TreeNodeArgs64 A{};
        TreeNodeArgs &a = A.n;
        a.S = S;
        a.rec = rec;
        a.geo = (const TreeGeo *)(b + p.off_geo[L]);
        a.nb = p.nb[L];
        a.W = work(L);
        a.F = (double *)(b + p.off_F[L]);
        if (!root) {
            a.pgeo = (const TreeGeo *)(b + p.off_geo[L + 1]);
            a.pnb = p.nb[L + 1];
            a.Fp = (const double *)(b + p.off_F[L + 1]);
            a.Wp = work(L + 1);
        }
        a.queue = queue + L;
        A.s64 = m.s64;
        const int64_t items = p.ncl[L] + p.pool;
        const dim3 grid((unsigned)(items < p.nslots ? items : p.nslots));
        if (f64) {
            const void *fn = root ? (const void *)&k_tree_nodes_f64<true> : (const void *)&k_tree_nodes_f64<false>;
            void *args[] = {(void *)&A};
            cudaLaunchKernel(fn, grid, dim3(kTreeNT), args, sizeof(TreeNodeSmem64), s);
        } else {
            const void *fn = root ? (const void *)&k_tree_nodes_f32<true> : (const void *)&k_tree_nodes_f32<false>;
            void *args[] = {(void *)&a};
            cudaLaunchKernel(fn, grid, dim3(kTreeNT), args, sizeof(TreeSmem32), s);
        }
    }
    TreePixArgs64 A{};
    TreePixArgs &a = A.p;
    a.S = S;
    a.rec = rec;
    a.s64 = m.s64;
    a.geo = leaf_geo;
    a.nv = m.nv;
    a.ldn = m.ldn;
    a.outidx = m.outidx;
    a.W = work(p.levels);
    a.Wf = work(0);
    a.F = (const double *)(b + p.off_F[0]);
    a.theta = m.theta;
    a.partial = (double *)(b + p.off_partial);
    a.accumulate = m.accumulate;
    a.b_min = m.b_min;
    a.st = m.st;
    a.queue = queue + kTreeLevels;
    A.far64 = m.far64;
    A.d_far = m.d_far;
    A.nside = m.nside;
    A.nb = p.nb[0];
    A.parts = p.ncl[0] * p.nst < 2 * (int64_t)p.pslots ? kBlocks64 : 1;
    const int64_t items = (p.ncl[0] + p.ppool) * (f64 ? A.parts : 1);
    const unsigned grid = (unsigned)(items < p.pslots ? items : p.pslots);
    if (f64 && m.nside > 0) k_tree_pixels_f64<true><<<grid, kTreeNT, sizeof(TreePixSmem64), s>>>(A);
    else if (f64) k_tree_pixels_f64<false><<<grid, kTreeNT, sizeof(TreePixSmem64), s>>>(A);
    else k_tree_pixels_f32<<<grid, kTreeNT, sizeof(TreeSmemPix), s>>>(a);
    k_tree_reduce<<<(unsigned)p.pslots, 256, 0, s>>>(a.W, p.leaf * p.leaf, a.partial, m.outidx, m.theta, m.accumulate);
    return cudaSuccess;
}

}  // namespace isw
