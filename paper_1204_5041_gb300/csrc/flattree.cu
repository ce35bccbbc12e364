// Flat-sky patch maps over a tree of square pixel clusters.  In the plane z = xi + i eta the pair term is
// w.d / |d|^2 = Re[ W / (z - z_s) ], W = w1 + i w2: analytic away from the sample, so the samples far from
// a cluster (centre z0, half-diagonal R, |z_s - z0| >= kappa R) act on it as one Taylor series
//   sum_s W_s / (z - z_s) = sum_k a_k ((z - z0) / R)^k,   a_k = -sum_s (W_s u_s) (R u_s)^k,  u_s = 1 / (z_s - z0),
// with an error kappa^-K of their terms after K of them: kappa = 3.5 with K = 16 in FP32 (2e-9, for
// samples at the near radius and the cluster's corners) and K = 32 in FP64 (4e-18).  A sample goes to
// the first level, from the whole patch down, at which it is far, and to the pixels of the leaves
// (32 x 32, 16 x 16 below 512 pixels a side) to which it is near at every level.  A sample costs 6 K operations per cluster; the
// selection of samples and the planning of chunks are those of tree.cuh, with positions in the plane and
// no beams.
//   k_flat_keys    spatial order of the samples
//   k_flat_crit    sorted records, decision data, tile balls
//   k_flat_series  coefficients of every cluster of a level, one sample per thread at a time
//   k_flat_pixels  the series of the leaf and its ancestors, plus the near samples, at the leaf's pixels
// 1024 x 1024 pixels with 2e5 samples: 85.7 -> 1.3 ms (0.5 of them the near samples, 0.6 the series of six
// levels, bound by the latency of finding a cluster's samples); FP32 error 1e-8 of the rms (direct
// 2e-8), FP64 1e-16.
#include "flat.cuh"
#include "tree.cuh"

namespace isw {

namespace {

constexpr float kFlatKappa = 3.5f;
// Samples beyond this coordinate are placed at it for the decisions near or far (widths are at most 1e15): balls and
// distances in float would be infinite from 1.8e19 on, and a tile with an infinite ball lost its other samples.
constexpr double kFlatEdge = 1e18;
constexpr int kSeriesTarget = 2048, kFlatPixTarget = 512;   // samples per chunk, at least
template <bool F64>
struct FlatNum {
    using T = float;
    using Rec = Flat32;
    static constexpr int K = 16;
};
template <>
struct FlatNum<true> {
    using T = double;
    using Rec = Flat64;
    static constexpr int K = 32;
};

__device__ __forceinline__ uint32_t spread2(uint32_t x)   // 12 bits -> even positions
{
    x &= 0xfffu;
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
    return x;
}

// Morton code of the position over twice the patch (samples beyond it in the border cells)
__global__ void k_flat_keys(const Flat64 *__restrict__ r64, int64_t n, double width, uint32_t *__restrict__ key,
                            uint32_t *__restrict__ idx)
{
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        const Flat64 g = r64[s];
        const float x = (float)(g.xs / (2.0 * width)) + 0.5f, y = (float)(g.ys / (2.0 * width)) + 0.5f;
        const uint32_t qx = (uint32_t)fminf(fmaxf(x * 4096.f, 0.f), 4095.f), qy = (uint32_t)fminf(fmaxf(y * 4096.f, 0.f), 4095.f);
        key[s] = spread2(qx) | (spread2(qy) << 1);
        idx[s] = (uint32_t)s;
    }
}

// One warp per tile of 64 samples in spatial order.  A sample of zero weight (behind the patch plane, or
// padding) is skipped.
__global__ void __launch_bounds__(256) k_flat_crit(const Flat32 *__restrict__ r32, const Flat64 *__restrict__ r64,
                                                   const uint32_t *__restrict__ perm, int64_t n, int64_t ntile, bool f64,
                                                   Flat32 *__restrict__ s32, Flat64 *__restrict__ s64,
                                                   TreeCrit *__restrict__ crit, TreeCap *__restrict__ caps)
{
    const int lane = threadIdx.x & 31;
    const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (t >= ntile) return;
    float4 x[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t s = t * kTreeS + 32 * h + lane;
        TreeCrit cr;
        cr.a = make_float4(0.f, 0.f, 0.f, 0.f);
        cr.b = make_float4(0.f, 0.f, 0.f, kCritSkip);
        x[h] = make_float4(0.f, 0.f, 0.f, -1.f);
        if (s < n) {
            const uint32_t src = perm[s];
            const Flat64 g = r64[src];
            if (f64) s64[s] = g;
            else s32[s] = r32[src];
            if (g.w1 != 0.0 || g.w2 != 0.0) {
                // a sample close to the patch plane is anywhere; its square is to stay finite
                cr.a.x = (float)fmin(fmax(g.xs, -kFlatEdge), kFlatEdge);
                cr.a.y = (float)fmin(fmax(g.ys, -kFlatEdge), kFlatEdge);
                cr.b = make_float4(1e6f, 0.f, 0.f, 0.f);   // never near by beam
                x[h] = cr.a;
            }
        }
        crit[s] = cr;
    }
    const TreeCap c = warp_ball(x);
    if (lane == 0) caps[t] = c;
}

struct FlatTreeArgs {
    TreeSamples S;
    const Flat32 *s32;
    const Flat64 *s64;
    TreePlane plane;
    double pitch;
    int level, nb, pnb;              // series: the level and its and its parent's clusters per side
    TreeWork W;
    double *A;                       // series: [ncl + pool][K][2]
    // pixels: every level's series
    int levels;
    const double *series[kTreeLevels];
    TreeWork Ws[kTreeLevels];
    int nbs[kTreeLevels];
    double *theta, *partial;
    int accumulate;
    unsigned long long *queue;
};

struct __align__(16) FlatSmem {
    Flat64 rec[kTreeBatch];
    TreeScanSmem scan;
    double a[kTreeLevels * 32 * 2];
    int64_t item;
};

// (x, e) <- the sum of the pairs (x, e) and (y, f) as a pair
__device__ __forceinline__ void pair_sum(float &x, float &e, float y, float f)
{
    const float s = x + y, bb = s - x;
    e += f + ((x - (s - bb)) + (y - bb));
    x = s;
}

template <bool F64, bool ROOT>
__global__ void __launch_bounds__(kTreeNT) k_flat_series(FlatTreeArgs a)
{
    using T = typename FlatNum<F64>::T;
    constexpr int K = FlatNum<F64>::K;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FlatSmem &sm = *reinterpret_cast<FlatSmem *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int np = *a.W.npool;
    const int64_t size = (int64_t)a.plane.leaf << a.level;
    const double R = 0.70710678118654752 * (double)size * a.pitch;
    TreeQueue queue{a.queue, 0ull};
    for (int64_t item = queue.first(&sm.item); item < a.W.ncl + np; item = queue.next(&sm.item)) {
        int kc, nch;
        int64_t at;
        const int64_t cl = tree_item(a.W, item, np, kc, nch, at);
        if (cl < 0) continue;
        const float4 self = plane_ball(a.plane, a.level, cl, a.nb);
        const float4 parent = ROOT ? self : plane_ball(a.plane, a.level + 1, tree_parent(cl, a.nb, a.pnb), a.pnb);
        const double zx = plane_centre(cl % a.nb, size, a.plane.M, a.pitch), zy = plane_centre(cl / a.nb, size, a.plane.M, a.pitch);
        T ar[K], ai[K];
#pragma unroll
        for (int k = 0; k < K; ++k) ar[k] = ai[k] = (T)0;
        auto consume = [&](int count) {
            for (int i = tid; i < count; i += kTreeNT) {
                const uint32_t e = sm.scan.list[i] & kTreeIndex;
                T dx, dy, w1, w2;
                if constexpr (F64) {
                    const Flat64 g = a.s64[e];
                    dx = g.xs - zx;
                    dy = g.ys - zy;
                    w1 = g.w1;
                    w2 = g.w2;
                } else {
                    const Flat32 g = a.s32[e];
                    const float xh = (float)zx, yh = (float)zy;
                    dx = (g.a.x - xh) + (g.a.z - (float)(zx - (double)xh));
                    dy = (g.a.y - yh) + (g.a.w - (float)(zy - (double)yh));
                    w1 = g.b.x;
                    w2 = g.b.y;
                }
                const T inv = (T)1 / (dx * dx + dy * dy);
                T ux = dx * inv, uy = -dy * inv;                              // 1 / (z_s - z0)
                if (inv < (T)(F64 ? 1e-300 : 1e-37)) {   // the square overflows; the weight grows like the distance
                    const T sx = dx * (T)0x1p-66, sy = dy * (T)0x1p-66, si = (T)1 / (sx * sx + sy * sy);
                    ux = sx * si * (T)0x1p-66;
                    uy = -sy * si * (T)0x1p-66;
                }
                T tx = -(w1 * ux - w2 * uy), ty = -(w1 * uy + w2 * ux);       // -W u
                const T vx = (T)R * ux, vy = (T)R * uy;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    ar[k] += tx;
                    ai[k] += ty;
                    const T nx = tx * vx - ty * vy;
                    ty = tx * vy + ty * vx;
                    tx = nx;
                }
            }
            __syncthreads();
        };
        tree_scan<ROOT, false, 1>(a.S, kc, nch, self, parent, 0.f, 0.f, 0.f, sm.scan, consume);
        // block sum of the 2K values: compensated pairs over the warp (FP32), then over the warps
#pragma unroll
        for (int k = 0; k < 2 * K; ++k) {
            T x = k & 1 ? ai[k >> 1] : ar[k >> 1];
            double v;
            if constexpr (F64) {
                for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                v = x;
            } else {
                float e = 0.f;
                for (int o = 16; o > 0; o >>= 1) {
                    const float y = __shfl_xor_sync(0xffffffffu, x, o), f = __shfl_xor_sync(0xffffffffu, e, o);
                    pair_sum(x, e, y, f);
                }
                v = (double)x + (double)e;
            }
            if (lane == 0) sm.a[w * 2 * K + k] = v;
        }
        __syncthreads();
        if (tid < 2 * K) {
            double v = sm.a[tid];
#pragma unroll
            for (int i = 1; i < kTreeNT / 32; ++i) v += sm.a[i * 2 * K + tid];
            a.A[at * 2 * K + tid] = v;
        }
        __syncthreads();
    }
}

// P = leaf^2 / 128 pixels per thread, slots in rows.
template <bool F64, int LEAF>
__global__ void __launch_bounds__(kTreeNT) k_flat_pixels(FlatTreeArgs a)
{
    using Rec = typename FlatNum<F64>::Rec;
    constexpr int K = FlatNum<F64>::K, TILE = LEAF * LEAF, P = TILE / kTreeNT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FlatSmem &sm = *reinterpret_cast<FlatSmem *>(smem_raw);
    Rec *rec = reinterpret_cast<Rec *>(sm.rec);
    const int tid = threadIdx.x;
    const int np = *a.W.npool;
    const int64_t M = a.plane.M;
    TreeQueue queue{a.queue, 0ull};
    for (int64_t item = queue.first(&sm.item); item < a.W.ncl + np; item = queue.next(&sm.item)) {
        int kc, nch;
        int64_t at;
        const int64_t cl = tree_item(a.W, item, np, kc, nch, at);
        if (cl < 0) continue;
        const int bx = (int)(cl % a.nb), by = (int)(cl / a.nb);
        const float4 self = plane_ball(a.plane, 0, cl, a.nb);
        double px[P], py[P], s64[P], s64lo[P], far[P];
        float xh[P], yh[P], xl[P], yl[P], ahi[P], alo[P];
        int64_t oi[P];
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const int l = q * kTreeNT + tid;
            const int64_t i = (int64_t)bx * LEAF + l % LEAF, j = (int64_t)by * LEAF + l / LEAF;
            s64[q] = s64lo[q] = far[q] = 0.0;
            ahi[q] = alo[q] = 0.f;
            oi[q] = i < M && j < M ? j * M + i : -1;
            px[q] = dmul(dsub(dadd((double)i, 0.5), dmul(0.5, (double)M)), a.pitch);
            py[q] = dmul(dsub(dadd((double)j, 0.5), dmul(0.5, (double)M)), a.pitch);
            xh[q] = __double2float_rn(px[q]);
            yh[q] = __double2float_rn(py[q]);
            xl[q] = __double2float_rn(px[q] - (double)xh[q]);
            yl[q] = __double2float_rn(py[q] - (double)yh[q]);
        }
        if (kc == 0) {
            // the series of the leaf and its ancestors, chunks added up
            for (int k = tid; k < a.levels * 2 * K; k += kTreeNT) {
                const int L = k / (2 * K), c = k % (2 * K);
                const int64_t cc = (int64_t)(by >> L) * a.nbs[L] + (bx >> L);
                const int n = a.Ws[L].nch[cc];
                const int64_t first = n == 1 ? cc : a.Ws[L].ncl + a.Ws[L].pbase[cc];
                double v = 0.0;
                for (int i = 0; i < n; ++i) v += a.series[L][(first + i) * 2 * K + c];
                sm.a[k] = v;
            }
            __syncthreads();
            for (int L = a.levels - 1; L >= 0; --L) {
                const int64_t size = (int64_t)LEAF << L;
                const double iR = 1.0 / (0.70710678118654752 * (double)size * a.pitch);
                const double zx = plane_centre(bx >> L, size, M, a.pitch), zy = plane_centre(by >> L, size, M, a.pitch);
                const double *c = sm.a + L * 2 * K;
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    if constexpr (F64) {
                        const double x = (px[q] - zx) * iR, y = (py[q] - zy) * iR;
                        double vr = 0.0, vi = 0.0;
                        for (int k = K - 1; k >= 1; --k) {
                            const double r = fma(vr, x, fma(-vi, y, c[2 * k]));
                            vi = fma(vr, y, fma(vi, x, c[2 * k + 1]));
                            vr = r;
                        }
                        fold64(s64[q], s64lo[q], fma(vr, x, -vi * y));
                        fold64(s64[q], s64lo[q], c[0]);
                    } else {
                        const float x = (float)((px[q] - zx) * iR), y = (float)((py[q] - zy) * iR);
                        float vr = 0.f, vi = 0.f;
                        for (int k = K - 1; k >= 1; --k) {
                            const float r = fmaf(vr, x, fmaf(-vi, y, (float)c[2 * k]));
                            vi = fmaf(vr, y, fmaf(vi, x, (float)c[2 * k + 1]));
                            vr = r;
                        }
                        far[q] += c[0] + (double)fmaf(vr, x, -vi * y);
                    }
                }
            }
        }
        auto consume = [&](int count) {
            for (int b0 = 0; b0 < count; b0 += kTreeBatch) {
                const int cnt = count - b0 < kTreeBatch ? count - b0 : kTreeBatch;
                if (tid < cnt) {
                    const uint32_t e = sm.scan.list[b0 + tid] & kTreeIndex;
                    if constexpr (F64) rec[tid] = a.s64[e];
                    else rec[tid] = a.s32[e];
                }
                __syncthreads();
                if constexpr (F64) {
                    double part[P];
#pragma unroll
                    for (int q = 0; q < P; ++q) part[q] = 0.0;
                    for (int s = 0; s < cnt; ++s) {
                        const Flat64 r = rec[s];
#pragma unroll
                        for (int q = 0; q < P; ++q) {
                            const double dx = dsub(px[q], r.xs), dy = dsub(py[q], r.ys);
                            const double Q = dadd(dmul(dx, dx), dmul(dy, dy));
                            part[q] += Q > 0.0 ? ddiv(dadd(dmul(r.w1, dx), dmul(r.w2, dy)), Q) : 0.0;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < P; ++q) fold64(s64[q], s64lo[q], part[q]);
                } else {
                    float part[P];
#pragma unroll
                    for (int q = 0; q < P; ++q) part[q] = 0.f;
#pragma unroll 2
                    for (int s = 0; s < cnt; ++s) {
                        const float4 ra = rec[s].a, rb = rec[s].b;
#pragma unroll
                        for (int q = 0; q < P; ++q) {
                            const float dx = (xh[q] - ra.x) + (xl[q] - ra.z);
                            const float dy = (yh[q] - ra.y) + (yl[q] - ra.w);
                            // d = 0 exactly makes the numerator 0: the floor keeps 0 * (1/Q) finite
                            const float Q = fmaxf(fmaf(dy, dy, dx * dx), 1e-30f);
                            part[q] = fmaf(fmaf(rb.y, dy, rb.x * dx), rcp_approx(Q), part[q]);
                        }
                    }
#pragma unroll
                    for (int q = 0; q < P; ++q) fold(ahi[q], alo[q], part[q]);
                }
                __syncthreads();
            }
        };
        tree_scan<false, true, 1>(a.S, kc, nch, self, self, 0.f, 0.f, 0.f, sm.scan, consume);
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const double v = F64 ? s64[q] + s64lo[q] : ((double)ahi[q] + (double)alo[q]) + far[q];
            if (nch == 1) {
                if (oi[q] >= 0) a.theta[oi[q]] = a.accumulate ? a.theta[oi[q]] + v : v;
            } else {
                a.partial[item * TILE + q * kTreeNT + tid] = v;   // pool entry of the chunk
            }
        }
    }
}

// theta of the leaves that were cut into chunks
__global__ void __launch_bounds__(256) k_flat_reduce(TreeWork W, const double *__restrict__ partial, int leaf, int nb,
                                                     int64_t M, double *__restrict__ theta, int accumulate)
{
    const int np = *W.npool, tile = leaf * leaf, parts = tile / 256;
    for (int k = blockIdx.x; k < np * parts; k += gridDim.x) {
        const int e = k / parts, l = k % parts * 256 + threadIdx.x;
        const int2 it = W.pool[e];
        if (it.y != 0) continue;
        const int64_t i = (int64_t)(it.x % nb) * leaf + l % leaf, j = (int64_t)(it.x / nb) * leaf + l / leaf;
        const int nch = W.nch[it.x];
        double hi = 0.0, lo = 0.0;
        for (int c = 0; c < nch; ++c) fold64(hi, lo, partial[(int64_t)(e + c) * tile + l]);
        if (i < M && j < M) theta[j * M + i] = accumulate ? theta[j * M + i] + (hi + lo) : hi + lo;
    }
}

const void *pixel_kernel(bool f64, int leaf)
{
    if (leaf == 32) return f64 ? (const void *)&k_flat_pixels<true, 32> : (const void *)&k_flat_pixels<false, 32>;
    return f64 ? (const void *)&k_flat_pixels<true, 16> : (const void *)&k_flat_pixels<false, 16>;
}

}  // namespace

FlatTreePlan flat_tree_plan(bool f64, int64_t M, int64_t n, int num_sms)
{
    FlatTreePlan p{};
    p.f64 = f64;
    p.n_pad = (n + kTreeS - 1) / kTreeS * kTreeS;
    p.nst = p.n_pad / kTreeS;
    const void *fs = f64 ? (const void *)&k_flat_series<true, false> : (const void *)&k_flat_series<false, false>;
    // leaves of 32 pixels once there are 256 of them: the near samples of a 16-pixel leaf (a hundred or so)
    // are too few for its set-up (1024 x 1024 pixels, 2e5 samples: 2.3 ms against 1.3)
    p.leaf = M >= 512 ? 32 : 16;
    const void *fp = pixel_kernel(f64, p.leaf);
    int a = 0, b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, fs, kTreeNT, sizeof(FlatSmem));
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fp, kTreeNT, sizeof(FlatSmem));
    p.nslots = (a > 0 ? a : 1) * num_sms;
    p.pslots = (b > 0 ? b : 1) * num_sms;
    p.pool = 8 * p.nslots;
    p.ppool = 8 * p.pslots;
    int64_t nb = (M + p.leaf - 1) / p.leaf, all = nb * nb;
    for (;;) {
        p.nb[p.levels++] = (int)nb;
        all += nb * nb;
        if (nb == 1 || p.levels == kTreeLevels) break;
        nb = (nb + 1) / 2;
    }
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += up256(bytes);
        return o;
    };
    const size_t K2 = 2 * (f64 ? FlatNum<true>::K : FlatNum<false>::K) * sizeof(double);
    p.off_queue = take(kTreeZero);
    p.off_crit = take((size_t)p.n_pad * sizeof(TreeCrit));
    p.off_caps = take((size_t)p.nst * sizeof(TreeCap));
    p.off_sup = take((size_t)((p.nst + kTreeSuper - 1) / kTreeSuper) * sizeof(TreeCap));
    p.off_rec = take((size_t)p.n_pad * (f64 ? sizeof(Flat64) : sizeof(Flat32)));
    p.off_sort = take(sort_scratch_bytes(n, 1));
    p.off_work = take((size_t)3 * all * sizeof(int));
    p.off_pool = take(((size_t)p.levels * p.pool + p.ppool) * sizeof(int2));
    p.off_partial = take((size_t)p.ppool * p.leaf * p.leaf * sizeof(double));
    for (int L = 0; L < p.levels; ++L) p.off_A[L] = take(((size_t)p.nb[L] * p.nb[L] + p.pool) * K2);
    p.bytes = at;
    return p;
}

cudaError_t launch_map_flat_tree(const FlatTreePlan &p, const void *r32, const void *r64, int64_t n, int64_t M, double width,
                                 double *theta, int accumulate, void *scratch, cudaStream_t s)
{
    unsigned char *b = (unsigned char *)scratch;
    unsigned long long *queue = (unsigned long long *)(b + p.off_queue), *total = queue + kTreeLevels + 1;
    int *npool = (int *)(total + (kTreeLevels + 1) * kTargets);
    cudaError_t e = cudaMemsetAsync(queue, 0, kTreeZero, s);
    if (e != cudaSuccess) return e;
    TreeCrit *crit = (TreeCrit *)(b + p.off_crit);
    TreeCap *caps = (TreeCap *)(b + p.off_caps), *sup = (TreeCap *)(b + p.off_sup);
    uint32_t *keys = (uint32_t *)(b + p.off_sort);
    Flat32 *s32 = (Flat32 *)(b + p.off_rec);
    Flat64 *s64 = (Flat64 *)(b + p.off_rec);
    const int64_t kb = (n + 255) / 256;
    k_flat_keys<<<(unsigned)(kb < 152 * 32 ? kb : 152 * 32), 256, 0, s>>>((const Flat64 *)r64, n, width, keys, keys + 2 * n);
    const uint32_t *perm = launch_sort_keys(n, 1, keys, s);
    k_flat_crit<<<(unsigned)((p.nst * 32 + 255) / 256), 256, 0, s>>>((const Flat32 *)r32, (const Flat64 *)r64, perm, n, p.nst,
                                                                      p.f64, s32, s64, crit, caps);
    const int64_t nsup = (p.nst + kTreeSuper - 1) / kTreeSuper;
    k_tree_super<<<dim3((unsigned)((nsup + 3) / 4), 1), 128, 0, s>>>(caps, p.nst, nsup, sup);
    const TreeSamples S{crit, nullptr, caps, nullptr, sup, nullptr, nullptr, p.nst};
    const double pitch = width / (double)M;
    TreeStages g{};
    g.n = p.levels + 1;
    g.plane = TreePlane{(float)pitch, kFlatKappa, M, p.leaf};
    int2 *entries = (int2 *)(b + p.off_pool);
    for (int st = 0; st <= p.levels; ++st) {
        const bool pix = st == p.levels;
        const int L = pix ? 0 : st;
        g.first[st + 1] = g.first[st] + (int64_t)p.nb[L] * p.nb[L];
        g.plane_level[st] = L;
        g.nb[st] = p.nb[L];
        if (st + 1 < p.levels) g.pnb[st] = p.nb[st + 1];
        g.pool[st] = pix ? p.ppool : p.pool;
        g.target[st] = pix ? kFlatPixTarget : kSeriesTarget;
        g.entries[st] = entries + (size_t)st * p.pool;
    }
    const int64_t all = g.first[g.n];
    int *est = (int *)(b + p.off_work), *nch = est + all, *pbase = nch + all;
    k_tree_count<<<(unsigned)((all + 3) / 4), 128, 0, s>>>(g, S, n, est, total);
    k_tree_plan<<<(unsigned)((all + 127) / 128), 128, 0, s>>>(g, est, total, nch, pbase, npool);
    FlatTreeArgs a{};
    a.S = S;
    a.s32 = s32;
    a.s64 = s64;
    a.plane = g.plane;
    a.pitch = pitch;
    a.levels = p.levels;
    a.theta = theta;
    a.partial = (double *)(b + p.off_partial);
    a.accumulate = accumulate;
    auto work = [&](int st) {
        return TreeWork{nch + g.first[st], pbase + g.first[st], g.entries[st], npool + st, g.first[st + 1] - g.first[st]};
    };
    for (int L = p.levels - 1; L >= 0; --L) {
        const bool root = L == p.levels - 1;
        a.level = L;
        a.nb = p.nb[L];
        a.pnb = root ? 0 : p.nb[L + 1];
        a.W = work(L);
        a.A = (double *)(b + p.off_A[L]);
        a.queue = queue + L;
        const int64_t items = a.W.ncl + p.pool;
        const void *fn = p.f64 ? (root ? (const void *)&k_flat_series<true, true> : (const void *)&k_flat_series<true, false>)
                               : (root ? (const void *)&k_flat_series<false, true> : (const void *)&k_flat_series<false, false>);
        void *args[] = {(void *)&a};
        cudaLaunchKernel(fn, dim3((unsigned)(items < p.nslots ? items : p.nslots)), dim3(kTreeNT), args, sizeof(FlatSmem), s);
        a.series[L] = a.A;
        a.Ws[L] = a.W;
        a.nbs[L] = p.nb[L];
    }
    a.nb = p.nb[0];
    a.W = work(p.levels);
    a.queue = queue + kTreeLevels;
    const int64_t items = a.W.ncl + p.ppool;
    const unsigned grid = (unsigned)(items < p.pslots ? items : p.pslots);
    void *args[] = {(void *)&a};
    cudaLaunchKernel(pixel_kernel(p.f64, p.leaf), dim3(grid), dim3(kTreeNT), args, sizeof(FlatSmem), s);
    k_flat_reduce<<<(unsigned)p.pslots, 256, 0, s>>>(a.W, a.partial, p.leaf, p.nb[0], M, theta, accumulate);
    return cudaSuccess;
}

}  // namespace isw
