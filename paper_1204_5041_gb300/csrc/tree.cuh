// Cluster tree over the pixels of a map (device side shared by tree.cu and treeadj.cu).
//
// The pair term of Eq. (1)-(2) is a smooth function of the direction n away from two places: n
// near the sample (1 - n.Xhat -> 0) and n in its beam (B = 1 + n.Xdot -> 0).  In the stereographic
// coordinates (xi, eta) about a cluster centre n0,
//   n = (2 xi e1 + 2 eta e2 + (1 - xi^2 - eta^2) n0) / (1 + xi^2 + eta^2),
// every factor of the pair term is a polynomial over 1 + xi^2 + eta^2, those denominators cancel,
// and the term is a rational function whose only poles are
//   (xi - xi_s)^2 + (eta - eta_s)^2 = 0        at distance |z_s|^2 = (1 - n0.Xhat) / (1 + n0.Xhat),
//   (xi - xi_b)^2 + (eta - eta_b)^2 = -beta^2  with |z_b|^2 + beta^2 = (1 + n0.Xdot) / (1 - n0.Xdot).
// So when n0.Xhat and -n0.Xdot are both below one threshold, i.e. the chord |n0 - Xhat| and the
// "beam chord" sqrt(2 (1 + n0.Xdot)) both exceed the cluster's near radius D, the sum of such
// samples over the cluster's square [-a, a]^2 is its polynomial interpolant in p x p Chebyshev
// points to within ~rho^-p, rho = (kappa - 1) + sqrt((kappa - 1)^2 + 1) for D = the chord of
// stereographic radius kappa a.  The pair terms are then evaluated at p^2 nodes instead of at every
// pixel of the cluster.
//
// Every (sample, pixel) pair is accounted for exactly once: at the first level, from the coarsest
// down, at which the sample is far from the pixel's cluster, or, if it is near at the finest level
// too, directly at the pixel.  Near at a cluster implies near at its parent (D_parent >= D_child +
// the distance of the two centres, both chords being 1-Lipschitz in n0), so that a level takes the
// samples that are near at the parent and far at itself.  The decision is one function of
// explicitly rounded operations, so every kernel takes the same one.
#pragma once

#include "isw_internal.cuh"
#include "kernels.cuh"
#include "pipeline.cuh"

namespace isw {

// Per sample: a = (Xhat, near-field radius rho), b = (-Xdot/|Xdot|, 1 - |Xdot|); a sample to be
// skipped (zero weight or padding) has b.w = kCritSkip.
constexpr float kCritSkip = 4.f;
struct __align__(16) TreeCrit {
    float4 a, b;
};
// Per tile of kTreeS samples, in the order that the tile is cut from: a ball (centre, radius; < 0 when
// the tile has no sample to sum) that holds the tile's Xhat vectors, enlarged by the largest rho
// (position order), or its Xdot vectors (velocity order).
struct __align__(16) TreeCap {
    float4 a;
};
// The samples in two orders.  Position order (Morton code of Xhat) is the order of the records; the
// velocity order (Morton code of Xdot) finds the samples whose beam meets a cluster: -Xdot near n0 has
// little to do with where the sample is, and in position order nearly every tile of a loop's samples
// holds some beam (N_side 512 with 2e5 samples: the tests of samples in such tiles took 1-2 ms a level).
struct TreeSamples {
    const TreeCrit *crit, *vcrit;
    const TreeCap *caps, *vcaps;
    const TreeCap *sup, *vsup; // the same balls over kTreeSuper consecutive tiles
    const uint32_t *vidx;      // record of a velocity-order entry
    int64_t nst;               // tiles of either order
};
// FP32 evaluation record (64 B): Xhat hi (3), c | Xhat lo (3), f = X'.Xhat | Xdot (3), 1 - |Xdot| | X' (3),
// rho^2.
struct __align__(16) TreeRec {
    float4 v[4];
};
// Cluster geometry: centre and tangent frame, half-sizes of the rectangle in stereographic
// coordinates that holds the cluster's pixels (or its children's rectangles), and the float centre
// with the near radius D that decides near and far.
struct __align__(16) TreeGeo {
    double n0[3], e1[3], e2[3], a1, a2;
    double pad;
    float4 c;    // n0, D
    float4 l;    // n0 - (float)n0
    float4 f1;   // e1, 1 / a1
    float4 f2;   // e2, 1 / a2
};

// Near radius of a cluster wider than a hemisphere (stereographic half-size above 1; scattered pixels of a short
// list): above every chord, so all samples are near to it, and its interpolant is not used.  Its frame and
// extents stand for nothing: its mean direction may be zero, a pixel may be the centre's antipode, where the
// coordinates are infinite.
constexpr float kWideRadius = 4.f;
__device__ __forceinline__ bool tree_wide(const float4 &c) { return c.w >= kWideRadius; }
// Near radius of a cluster without pixels (the end of a list whose last entries are no pixel indices): a mark,
// above every real radius.  Such a cluster has a finite frame that stands for nothing, takes no samples, and its
// parents leave it out.
constexpr float kEmptyRadius = 8.f;
__device__ __forceinline__ bool tree_empty(const float4 &c) { return c.w >= kEmptyRadius; }

// Work of one stage (a level's node sums, or the pixels): clusters with many samples are cut into
// chunks, listed in the pool; the others are one item each.
struct TreeWork {
    const int *nch;        // chunks of a cluster
    const int *pbase;      // first pool entry of a cluster with nch > 1
    const int2 *pool;      // (cluster, chunk)
    const int *npool;      // pool entries in use
    int64_t ncl;
};

// Parent of cluster c: 2 x 2 blocks of a face's nb x nb clusters (pnb x pnb parents), or, for a list of
// pixels in spatial order (nb = 0), four consecutive clusters.
__device__ __forceinline__ int64_t tree_parent(int64_t c, int nb, int pnb)
{
    if (nb == 0) return c >> 2;
    const int64_t f = c / ((int64_t)nb * nb), rem = c - f * nb * nb;
    return (f * pnb + rem / nb / 2) * pnb + rem % nb / 2;
}

constexpr int kTreeS = 64;        // samples per tile of the scan
constexpr int kTreeNT = 128;      // threads per CTA of the evaluation kernels
constexpr int kTreeBatch = 128;   // samples per staged batch, one per thread
constexpr int kTreeGroup = 32;    // candidate tiles tested sample by sample at a time
constexpr int kTreeSuper = 32;    // tiles per super tile
constexpr int kTreeList = kTreeGroup * kTreeS + kTreeBatch;

// cos(pi m / 32): Chebyshev points x_k = cos(pi (2k + 1) / (2p)) and values T_i(x_k) for p = 8, 16
__device__ __constant__ const double kCos32[64] = {
    1.0, 0.99518472667219688624, 0.98078528040323044913, 0.95694033573220886494,
    0.92387953251128675613, 0.88192126434835502971, 0.83146961230254523708, 0.77301045336273696081,
    0.7071067811865475244, 0.63439328416364549822, 0.55557023301960222474, 0.47139673682599764856,
    0.38268343236508977173, 0.29028467725446236764, 0.19509032201612826785, 0.098017140329560601994,
    0.0, -0.098017140329560601994, -0.19509032201612826785, -0.29028467725446236764,
    -0.38268343236508977173, -0.47139673682599764856, -0.55557023301960222474, -0.63439328416364549822,
    -0.7071067811865475244, -0.77301045336273696081, -0.83146961230254523708, -0.88192126434835502971,
    -0.92387953251128675613, -0.95694033573220886494, -0.98078528040323044913, -0.99518472667219688624,
    -1.0, -0.99518472667219688624, -0.98078528040323044913, -0.95694033573220886494,
    -0.92387953251128675613, -0.88192126434835502971, -0.83146961230254523708, -0.77301045336273696081,
    -0.7071067811865475244, -0.63439328416364549822, -0.55557023301960222474, -0.47139673682599764856,
    -0.38268343236508977173, -0.29028467725446236764, -0.19509032201612826785, -0.098017140329560601994,
    0.0, 0.098017140329560601994, 0.19509032201612826785, 0.29028467725446236764,
    0.38268343236508977173, 0.47139673682599764856, 0.55557023301960222474, 0.63439328416364549822,
    0.7071067811865475244, 0.77301045336273696081, 0.83146961230254523708, 0.88192126434835502971,
    0.92387953251128675613, 0.95694033573220886494, 0.98078528040323044913, 0.99518472667219688624};

// T_i at the k-th of NP Chebyshev points (i = 1: the point itself)
template <int NP>
__device__ __forceinline__ double cheb_at(int i, int k)
{
    static_assert(32 % (2 * NP) == 0 || NP == 16, "kCos32 holds multiples of pi / 32");
    return kCos32[(i * (2 * k + 1) * (16 / NP)) & 63];
}

// The near decision, by position and by beam: explicitly rounded operations, the same result in
// every kernel.
__device__ __forceinline__ bool tree_near_pos(const float4 &a, const float4 &c)
{
    const float dx = __fsub_rn(c.x, a.x), dy = __fsub_rn(c.y, a.y), dz = __fsub_rn(c.z, a.z);
    const float d2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
    const float r = __fadd_rn(c.w, a.w);
    return d2 < __fmul_rn(r, r);
}
// 2 B at the centre, and the decision from it
__device__ __forceinline__ float tree_beam2(const float4 &b, const float4 &c)
{
    const float wx = __fsub_rn(c.x, b.x), wy = __fsub_rn(c.y, b.y), wz = __fsub_rn(c.z, b.z);
    const float w2 = __fmaf_rn(wz, wz, __fmaf_rn(wy, wy, __fmul_rn(wx, wx)));
    // 2 B = 2 (1 - v) + v |n0 + Xdot/v|^2 without cancellation
    return __fmaf_rn(__fsub_rn(1.f, b.w), w2, __fmul_rn(2.f, b.w));
}
__device__ __forceinline__ bool tree_near_beam(const float4 &b, const float4 &c)
{
    return tree_beam2(b, c) < __fmul_rn(c.w, c.w);
}

// Whether a tile may hold a sample that is near, with margins.
__device__ __forceinline__ bool tree_tile_pos(const TreeCap &t, const float4 &c)
{
    const float dx = c.x - t.a.x, dy = c.y - t.a.y, dz = c.z - t.a.z;
    const float r = c.w + t.a.w + 1e-5f;
    return t.a.w >= 0.f && dx * dx + dy * dy + dz * dz < r * r * 1.0001f;
}
__device__ __forceinline__ bool tree_tile_beam(const TreeCap &t, const float4 &c)
{
    const float b = 1.f + (c.x * t.a.x + c.y * t.a.y + c.z * t.a.z) - t.a.w;   // lower bound of B
    return t.a.w >= 0.f && 2.f * b < c.w * c.w + 1e-5f;
}

struct TreeScanSmem {
    uint32_t list[kTreeList];
    uint32_t cand[kTreeGroup * kTreeSuper];   // candidate tiles
    uint32_t sup[kTreeNT];                    // candidate super tiles
    int wcnt[kTreeNT / 32];
    int tcnt[kTreeGroup];
};

// List entries: the record and, for LEAF, what the evaluation has to watch for at the cluster's pixels
// (all within chord R of the centre): kTreeBeam when some B may be below b_min, kTreeClose when the
// centre is within `close` + rho.
constexpr uint32_t kTreeBeam = 0x80000000u, kTreeClose = 0x40000000u, kTreeIndex = 0x3fffffffu;

// Exclusive prefix of 32 counts (tcnt, in warp order) and their total, for every thread.
__device__ __forceinline__ int tree_prefix(const int *tcnt, int &total)
{
    const int lane = threadIdx.x & 31;
    const int own = tcnt[lane];
    int incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - own;
}

// Tests the samples of up to kTreeGroup tiles (tile(i), i < n) and appends those of the cluster to
// sm.list after the `held` entries there; whole block, returns the new length.
template <bool ROOT, bool LEAF, typename Tile>
__device__ __forceinline__ int tree_select(const TreeSamples &S, int pass, const float4 self, const float4 outer,
                                           float close, float beam2, int n, int held, TreeScanSmem &sm, Tile &&tile)
{
    constexpr int W = kTreeNT / 32, NR = kTreeGroup / W;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const TreeCrit *crit = pass ? S.vcrit : S.crit;
    unsigned mk[NR][2];
    uint32_t fl = 0;   // two flag bits per tested sample
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        const int idx = i * W + w;
        mk[i][0] = mk[i][1] = 0u;
        if (idx < n) {
            const int64_t s = (int64_t)tile(idx) * kTreeS + lane;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 a = crit[s + 32 * h].a, b = crit[s + 32 * h].b;
                bool sel = b.w < kCritSkip;
                if (!ROOT) {
                    const bool pos = tree_near_pos(a, outer);
                    sel = sel && (pass ? !pos && tree_near_beam(b, outer) : pos);
                }
                if (!LEAF) {
                    sel = sel && !tree_near_pos(a, self) && !tree_near_beam(b, self);
                } else {
                    if (tree_beam2(b, self) < beam2) fl |= 1u << (4 * i + 2 * h);
                    float4 c = self;
                    c.w = close + 1e-6f;   // tree_near_pos adds rho
                    if (tree_near_pos(a, c)) fl |= 2u << (4 * i + 2 * h);
                }
                mk[i][h] = __ballot_sync(0xffffffffu, sel);
            }
        }
        if (lane == 0) sm.tcnt[idx] = __popc(mk[i][0]) + __popc(mk[i][1]);
    }
    __syncthreads();
    int total;
    const int excl = tree_prefix(sm.tcnt, total);
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        const int idx = i * W + w;
        int pos = held + __shfl_sync(0xffffffffu, excl, idx);
        if ((mk[i][0] | mk[i][1]) == 0u) continue;
        const int64_t s = (int64_t)tile(idx) * kTreeS + lane;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (mk[i][h] >> lane & 1u)
                sm.list[pos + __popc(mk[i][h] & below)] =
                    (pass ? S.vidx[s + 32 * h] : (uint32_t)s + 32 * h) |
                    (LEAF ? (fl >> (4 * i + 2 * h) & 1u) << 31 | (fl >> (4 * i + 2 * h + 1) & 1u) << 30 : 0u);
            pos += __popc(mk[i][h]);
        }
    }
    __syncthreads();
    return held + total;
}

// Selects, in a fixed order, the samples of the tiles kc, kc + split, ... that belong to one cluster
// (every split-th tile: strings are dense on a few clusters and consecutive in either order, so chunks
// of consecutive tiles would leave all near samples of such a cluster in one chunk).  ROOT: all
// samples far from it; LEAF: those near it; otherwise those near the parent and far from it.  The
// position order gives all samples (ROOT) or those near by position, the velocity order those near by
// beam only (PASSES = 1 leaves those out: flat sky).  consume(n) is called by the whole block with n entries in sm.list: a multiple of
// kTreeBatch, except for the last call.  Super tiles are tested first, 128 at a time, then the tiles of
// 32 candidates, then the samples of 32 tiles; entries left over wait, so that batches stay full.
template <bool ROOT, bool LEAF, int PASSES = 2, typename Consume>
__device__ __forceinline__ void tree_scan(const TreeSamples &S, int kc, int split, const float4 self,
                                          const float4 parent, float R, float close, float b_min, TreeScanSmem &sm,
                                          Consume &&consume)
{
    constexpr int W = kTreeNT / 32, NR = kTreeGroup / W;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned below = (1u << lane) - 1u;
    const float4 outer = LEAF ? self : parent;
    const float rb = sqrtf(2.f * b_min) * 1.001f + R + 1e-5f, beam2 = rb * rb;
    int held = 0;
    auto drain = [&]() {   // full batches
        if (held < kTreeBatch) return;
        const int full = held & ~(kTreeBatch - 1);
        consume(full);
        __syncthreads();
        const int rem = held - full;
        uint32_t v = 0;
        if (tid < rem) v = sm.list[full + tid];
        __syncthreads();
        if (tid < rem) sm.list[tid] = v;
        held = rem;
        __syncthreads();
    };
    if (ROOT) {
        const int64_t j1 = (S.nst - kc + split - 1) / split;   // tile j of the chunk is tile kc + j split
#pragma unroll 1
        for (int64_t g0 = 0; g0 < j1; g0 += kTreeGroup) {
            const int n = (int)(j1 - g0 < kTreeGroup ? j1 - g0 : kTreeGroup);
            held = tree_select<true, false>(S, 0, self, self, close, beam2, n, held, sm,
                                            [&](int i) { return kc + (g0 + i) * split; });
            drain();
        }
    } else {
        const int nsup = (int)((S.nst + kTreeSuper - 1) / kTreeSuper);
#pragma unroll 1
        for (int pass = 0; pass < PASSES; ++pass) {
            const TreeCap *caps = pass ? S.vcaps : S.caps, *sup = pass ? S.vsup : S.sup;
#pragma unroll 1
            for (int u0 = 0; u0 < nsup; u0 += kTreeNT) {
                bool in = false;
                if (u0 + tid < nsup) {
                    const TreeCap cap = sup[u0 + tid];
                    in = pass ? tree_tile_beam(cap, outer) : tree_tile_pos(cap, outer);
                }
                const unsigned m = __ballot_sync(0xffffffffu, in);
                if (lane == 0) sm.wcnt[w] = __popc(m);
                __syncthreads();
                int ns = 0, at = 0;
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    if (i == w) at = ns;
                    ns += sm.wcnt[i];
                }
                if (in) sm.sup[at + __popc(m & below)] = u0 + tid;
                __syncthreads();
#pragma unroll 1
                for (int v0 = 0; v0 < ns; v0 += kTreeGroup) {
                    unsigned mk[NR];
#pragma unroll
                    for (int i = 0; i < NR; ++i) {
                        const int idx = v0 + i * W + w;
                        bool hit = false;
                        if (idx < ns) {
                            const uint32_t t = sm.sup[idx] * kTreeSuper + lane;
                            if (t < (uint32_t)S.nst && (split == 1 || t % (uint32_t)split == (uint32_t)kc)) {
                                const TreeCap cap = caps[t];
                                hit = pass ? tree_tile_beam(cap, outer) : tree_tile_pos(cap, outer);
                            }
                        }
                        mk[i] = __ballot_sync(0xffffffffu, hit);
                        if (lane == 0) sm.tcnt[i * W + w] = __popc(mk[i]);
                    }
                    __syncthreads();
                    int ncand;
                    const int excl = tree_prefix(sm.tcnt, ncand);
#pragma unroll
                    for (int i = 0; i < NR; ++i) {
                        const int pos = __shfl_sync(0xffffffffu, excl, i * W + w);
                        if (mk[i] >> lane & 1u)
                            sm.cand[pos + __popc(mk[i] & below)] = sm.sup[v0 + i * W + w] * kTreeSuper + lane;
                    }
                    __syncthreads();
#pragma unroll 1
                    for (int g0 = 0; g0 < ncand; g0 += kTreeGroup) {
                        const int n = ncand - g0 < kTreeGroup ? ncand - g0 : kTreeGroup;
                        held = tree_select<false, LEAF>(S, pass, self, outer, close, beam2, n, held, sm,
                                                        [&](int i) { return sm.cand[g0 + i]; });
                        drain();
                    }
                }
            }
        }
    }
    if (held > 0) consume(held);
    __syncthreads();
}

// Item -> (cluster, chunk): pool entries first (the heavy clusters), then one item per cluster, -1 for
// a cluster whose chunks are in the pool.  `at` is the slot of the item's sums.
__device__ __forceinline__ int64_t tree_item(const TreeWork &W, int64_t item, int np, int &kc, int &nch, int64_t &at)
{
    if (item < np) {
        const int2 e = W.pool[item];
        kc = e.y;
        nch = W.nch[e.x];
        at = W.ncl + item;
        return e.x;
    }
    const int64_t c = item - np;
    kc = 0;
    nch = W.nch[c];
    at = c;
    return nch == 1 ? c : -1;
}

// Dynamic distribution with the next item's number already on its way: the counter is read by thread 0
// when an item starts and handed over when it ends.
struct TreeQueue {
    unsigned long long *counter;
    unsigned long long nx;
    __device__ __forceinline__ int64_t first(int64_t *slot)
    {
        if (threadIdx.x == 0) *slot = (int64_t)atomicAdd(counter, 1ull);
        __syncthreads();
        const int64_t item = *slot;
        if (threadIdx.x == 0) nx = atomicAdd(counter, 1ull);
        __syncthreads();
        return item;
    }
    __device__ __forceinline__ int64_t next(int64_t *slot)
    {
        if (threadIdx.x == 0) *slot = (int64_t)nx;
        __syncthreads();
        const int64_t item = *slot;
        if (threadIdx.x == 0) nx = atomicAdd(counter, 1ull);
        __syncthreads();
        return item;
    }
};

// Node values (node k = j NP + i) -> Chebyshev coefficients, in place in shared memory; whole block.
template <int NP>
__device__ __forceinline__ void cheb_transform(double *coef, double *tmp)
{
    constexpr int NN = NP * NP;
    for (int k = threadIdx.x; k < NN; k += blockDim.x) {   // along xi
        const int j = k / NP, m = k % NP;
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < NP; ++i) v = fma(coef[j * NP + i], cheb_at<NP>(m, i), v);
        tmp[k] = v * (m == 0 ? 1.0 / NP : 2.0 / NP);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < NN; k += blockDim.x) {
        const int q = k / NP, m = k % NP;
        double v = 0.0;
#pragma unroll
        for (int j = 0; j < NP; ++j) v = fma(tmp[j * NP + m], cheb_at<NP>(q, j), v);
        coef[k] = v * (q == 0 ? 1.0 / NP : 2.0 / NP);
    }
    __syncthreads();
}

// Values of cluster cl at its NP x NP nodes (the sum of its chunks) -> their Chebyshev coefficients in
// shared memory (coef, tmp: NP * NP doubles); whole block.
template <int NP>
__device__ __forceinline__ void cheb_coefs(const double *__restrict__ F, const TreeWork &W, int64_t cl, double *coef,
                                           double *tmp)
{
    constexpr int NN = NP * NP;
    const int nch = W.nch[cl];
    const int64_t at = nch == 1 ? cl : W.ncl + W.pbase[cl];
    for (int k = threadIdx.x; k < NN; k += blockDim.x) {
        double v = 0.0;
        for (int c = 0; c < nch; ++c) v += F[(at + c) * NN + k];
        coef[k] = v;
    }
    __syncthreads();
    cheb_transform<NP>(coef, tmp);
}

namespace {

// Conversions in integer instructions: a conversion takes a slot of the FP64 unit (two per clock and SM), and the
// FP32 kernels' few FP64 operations per pixel bound them where clusters have few samples.
// (float)x truncated; below the normal range 0; finite values
__device__ __forceinline__ float trunc_float(double x)
{
    const int hi = __double2hiint(x), e = (hi >> 20 & 0x7ff) - 896;
    const unsigned m = (unsigned)(hi & 0xfffff) << 3 | (unsigned)__double2loint(x) >> 29;
    return e <= 0 ? 0.f : __int_as_float((int)((unsigned)hi & 0x80000000u | (unsigned)e << 23 | m));
}
// x as a float pair, h truncated to 24 bits
__device__ __forceinline__ void split_float(double x, float &h, float &l)
{
    const double t = __hiloint2double(__double2hiint(x), __double2loint(x) & (int)0xe0000000);
    h = trunc_float(t);
    l = trunc_float(x - t);
}
// (double)x; below the normal range 0
__device__ __forceinline__ double widen(float x)
{
    const unsigned b = (unsigned)__float_as_int(x), e = b >> 23 & 0xff;
    const unsigned hi = (b & 0x80000000u) | (e == 0xff ? 0x7ffu : e + 896) << 20 | (b & 0x7fffff) >> 3;
    return e == 0 ? 0.0 : __hiloint2double((int)hi, (int)(b << 29));
}

__device__ __forceinline__ float warp_sum(float v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v)
{
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// ball around the mean of the lane's two points (w = enlargement, < 0: no point); radius < 0 when empty
__device__ __forceinline__ TreeCap warp_ball(const float4 (&x)[2])
{
    float sx = 0.f, sy = 0.f, sz = 0.f, cnt = 0.f, r = -1.f;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (x[h].w >= 0.f) {
            sx += x[h].x;
            sy += x[h].y;
            sz += x[h].z;
            cnt += 1.f;
        }
    cnt = fmaxf(warp_sum(cnt), 1.f);
    sx = warp_sum(sx) / cnt;
    sy = warp_sum(sy) / cnt;
    sz = warp_sum(sz) / cnt;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (x[h].w >= 0.f) {
            const float dx = x[h].x - sx, dy = x[h].y - sy, dz = x[h].z - sz;
            r = fmaxf(r, sqrtf(dx * dx + dy * dy + dz * dz) * 1.0001f + 1e-6f + x[h].w);
        }
    TreeCap c;
    c.a = make_float4(sx, sy, sz, warp_max(r));
    return c;
}

// Balls over kTreeSuper tiles, one warp each: around the mean of the tiles' centres.  Position order in
// blockIdx.y = 0, velocity order in 1 (caps and sup hold both, nst and nsup apart).
__global__ void __launch_bounds__(128) k_tree_super(const TreeCap *__restrict__ caps, int64_t nst, int64_t nsup,
                                                    TreeCap *__restrict__ sup)
{
    const int lane = threadIdx.x & 31;
    const int64_t u = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (u >= nsup) return;
    const int64_t t = u * kTreeSuper + lane;
    float4 a = make_float4(0.f, 0.f, 0.f, -1.f);
    if (t < nst) a = caps[blockIdx.y * nst + t].a;
    const float on = a.w >= 0.f ? 1.f : 0.f, cnt = fmaxf(warp_sum(on), 1.f);
    const float sx = warp_sum(on * a.x) / cnt, sy = warp_sum(on * a.y) / cnt, sz = warp_sum(on * a.z) / cnt;
    const float dx = a.x - sx, dy = a.y - sy, dz = a.z - sz;
    const float r = warp_max(on > 0.f ? sqrtf(dx * dx + dy * dy + dz * dz) * 1.0001f + 1e-6f + a.w : -1.f);
    TreeCap c;
    c.a = make_float4(sx, sy, sz, r);
    if (lane == 0) sup[blockIdx.y * nsup + u] = c;
}

// Clusters of a flat patch, leaf x 2^level pixels square, and their balls: the centre in the plane (third
// coordinate 0) and the near radius kappa times the half-diagonal.
struct TreePlane {
    float pitch, kappa;        // pitch 0: not a plane
    int64_t M;
    int leaf;
};
__device__ __forceinline__ double plane_centre(int64_t b, int64_t size, int64_t M, double pitch)
{
    return ((double)(b * size) + 0.5 * (double)size - 0.5 * (double)M) * pitch;
}
__device__ __forceinline__ float4 plane_ball(const TreePlane &p, int level, int64_t c, int nb)
{
    const int64_t size = (int64_t)p.leaf << level;
    const float h = 0.70710678f * (float)size * p.pitch;
    return make_float4((float)plane_centre(c % nb, size, p.M, (double)p.pitch),
                       (float)plane_centre(c / nb, size, p.M, (double)p.pitch), 0.f, p.kappa * h);
}

// The stages to plan: node sums of the levels, then the pixels.
constexpr int kTargets = 8;             // chunk sizes tried: target, 2 target, ...
// work counters, totals per chunk size and pool lengths of the stages
constexpr size_t kTreeZero =
    (kTreeLevels + 1) * ((1 + kTargets) * sizeof(unsigned long long) + sizeof(int));
struct TreeStages {
    int n;
    int64_t first[kTreeLevels + 2];     // prefix of the stages' cluster counts
    const TreeGeo *geo[kTreeLevels + 1], *pgeo[kTreeLevels + 1];   // the clusters, their parents (nodes only)
    TreePlane plane;                    // flat sky: the clusters' balls instead of geo
    int plane_level[kTreeLevels + 1];
    int nb[kTreeLevels + 1], pnb[kTreeLevels + 1];
    int pool[kTreeLevels + 1];          // pool entries
    int target[kTreeLevels + 1];        // smallest chunk
    int2 *entries[kTreeLevels + 1];
};

// Share of a tile's samples that lies within the near chord of a cluster, from the tile's ball (a
// linear ramp across the ball): position tiles by distance, beam tiles by B.
__device__ __forceinline__ float tile_share(const TreeCap &t, const float4 &c, int pass)
{
    if (t.a.w < 0.f) return 0.f;
    float x;
    if (pass) {
        const float b = 1.f + (c.x * t.a.x + c.y * t.a.y + c.z * t.a.z);
        x = 0.5f * c.w * c.w - b;
    } else {
        const float dx = c.x - t.a.x, dy = c.y - t.a.y, dz = c.z - t.a.z;
        x = c.w - sqrtf(dx * dx + dy * dy + dz * dz);
    }
    return fminf(fmaxf(0.5f + 0.5f * x / (t.a.w + 1e-6f), 0.f), 1.f);
}

// Estimate of every cluster's samples from the tile balls; all of them at the root.  And, for each chunk
// size, the pool entries that it would take.  One warp per (stage, cluster).
__global__ void __launch_bounds__(128) k_tree_count(TreeStages g, TreeSamples S, int64_t n, int *__restrict__ est,
                                                    unsigned long long *__restrict__ total)
{
    const int lane = threadIdx.x & 31;
    const int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (k >= g.first[g.n]) return;
    int st = 0;
    while (k >= g.first[st + 1]) ++st;
    const int64_t c = k - g.first[st];
    const bool leaf = st == g.n - 1;
    int64_t v = n;
    if (g.plane.pitch == 0.f && tree_empty(g.geo[st][c].c)) {
        v = 0;
    } else if (leaf || g.pnb[st] != 0 || g.pgeo[st]) {
        float4 self, outer;
        if (g.plane.pitch > 0.f) {
            self = plane_ball(g.plane, g.plane_level[st], c, g.nb[st]);
            outer = leaf ? self : plane_ball(g.plane, g.plane_level[st] + 1, tree_parent(c, g.nb[st], g.pnb[st]), g.pnb[st]);
        } else {
            self = g.geo[st][c].c;
            outer = leaf ? self : g.pgeo[st][tree_parent(c, g.nb[st], g.pnb[st])].c;
        }
        float share = 0.f;
        const int nsup = (int)((S.nst + kTreeSuper - 1) / kTreeSuper);
        for (int pass = 0; pass < (S.vsup ? 2 : 1); ++pass) {
            const TreeCap *sup = pass ? S.vsup : S.sup, *caps = pass ? S.vcaps : S.caps;
            for (int u0 = 0; u0 < nsup; u0 += 32) {
                bool in = false;
                if (u0 + lane < nsup) {
                    const TreeCap cap = sup[u0 + lane];
                    in = pass ? tree_tile_beam(cap, outer) : tree_tile_pos(cap, outer);
                }
                unsigned m = __ballot_sync(0xffffffffu, in);
                for (; m; m &= m - 1u) {
                    const int64_t t = (int64_t)(u0 + __ffs(m) - 1) * kTreeSuper + lane;
                    if (t < S.nst) {
                        const TreeCap cap = caps[t];
                        const float f = tile_share(cap, outer, pass);
                        share += leaf || pass ? f : fmaxf(f - tile_share(cap, self, pass), 0.f);
                    }
                }
            }
        }
        v = (int64_t)(warp_sum(share) * (float)kTreeS);
        if (v > n) v = n;
    }
    if (lane == 0) est[k] = (int)v;
    if (lane < kTargets) {
        const int64_t T = (int64_t)g.target[st] << lane;
        if (v >= T) atomicAdd(total + st * kTargets + lane, (unsigned long long)(1 + v / T));
    }
}

// Chunks per cluster: with the smallest chunk size whose entries fit the pool (none: no cluster is
// cut).  Where a cluster's entries lie in the pool depends on the order of the atomics; what they hold
// does not.
__global__ void __launch_bounds__(128) k_tree_plan(TreeStages g, const int *__restrict__ est,
                                                   const unsigned long long *__restrict__ total, int *__restrict__ nch,
                                                   int *__restrict__ pbase, int *__restrict__ npool)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= g.first[g.n]) return;
    int st = 0;
    while (k >= g.first[st + 1]) ++st;
    int j = 0;
    while (j < kTargets && total[st * kTargets + j] > (unsigned long long)g.pool[st]) ++j;
    const int64_t T = (int64_t)g.target[st] << j;
    const int m = j == kTargets || est[k] < T ? 1 : (int)(1 + est[k] / T);
    int b = 0;
    if (m > 1) {
        b = atomicAdd(npool + st, m);
        for (int i = 0; i < m; ++i) g.entries[st][b + i] = make_int2((int)(k - g.first[st]), i);
    }
    nch[k] = m;
    pbase[k] = b;
}

// theta of the clusters that were cut into chunks: their partial sums added in chunk order, one pixel per
// thread.  With few clusters a warp takes 32 pixels of one, since the FP64 additions of clusters with many
// chunks are the bound (N_side 64 in FP64, 48 clusters of 150 chunks: 375 us by 256 pixels, 103 us by 32); with
// more clusters than warps it takes a cluster, most of which have one chunk (N_side 1024: 44 us by 32 pixels, 34 us
// so).
__global__ void __launch_bounds__(256) k_tree_reduce(TreeWork W, int tile, const double *__restrict__ partial,
                                                     const int64_t *__restrict__ outidx, double *__restrict__ theta,
                                                     int accumulate)
{
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x / 32);
    const int parts = W.ncl < warps ? tile / 32 : 1, share = tile / parts;
    for (int64_t i = threadIdx.x / 32 * (int64_t)gridDim.x + blockIdx.x; i < W.ncl * parts; i += warps) {
        const int64_t cl = i / parts;
        const int nch = W.nch[cl];
        if (nch == 1) continue;
        const int l0 = (int)(i - cl * parts) * share;
        for (int l = l0 + (threadIdx.x & 31); l < l0 + share; l += 32) {
            const int64_t oi = outidx[cl * tile + l];
            const double *src = partial + (int64_t)W.pbase[cl] * tile + l;
            double hi = 0.0, lo = 0.0;
            int c = 0;
            for (; c + 8 <= nch; c += 8) {
                double v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = src[(int64_t)(c + k) * tile];
#pragma unroll
                for (int k = 0; k < 8; ++k) fold64(hi, lo, v[k]);
            }
            for (; c < nch; ++c) fold64(hi, lo, src[(int64_t)c * tile]);
            if (oi >= 0) theta[oi] = accumulate ? theta[oi] + (hi + lo) : hi + lo;
        }
    }
}

constexpr int kNP = 8, kNN = kNP * kNP;   // FP32: 8 x 8 nodes
constexpr int kLeaf = 16;                 // and 16 x 16 pixel leaves
// Near radius in stereographic half-sizes.  FP32 (8 x 8 nodes): 4 gives 2.2e-8 of the rms at N_side 100 and 10.1 ms at N_side 512
// with 2e5 samples, 3.5 2.6e-8 and 9.2 ms, 3 5.1e-8 and 8.5 ms.
// FP64 (16 x 16 nodes): in 80-bit arithmetic, with clusters set next to the strings, the truncation is
// 9e-16 of the rms at 4 and 1e-17 at 5; 4.5 keeps it below the rounding of the sums.
constexpr double kKappa32 = 3.5, kKappa64 = 4.5;

__device__ __forceinline__ double near_radius(double kappa, double a)
{
    // chord of stereographic radius kappa a
    const double z = kappa * a;
    return 2.0 * z / sqrt(1.0 + z * z);
}

// One warp per tile of 64 records (position order): decision data, evaluation records, caps, and the
// record of every input sample.
__global__ void __launch_bounds__(256) k_tree_crit(const Seg32 *__restrict__ s32, const Seg64 *__restrict__ s64,
                                                   const uint32_t *__restrict__ perm, int64_t n, int64_t ntile,
                                                   TreeCrit *__restrict__ crit, TreeCap *__restrict__ caps,
                                                   TreeRec *__restrict__ rec, uint32_t *__restrict__ inv)
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
        const Seg32 f = s32[s];
        if (s < n) {
            inv[perm[s]] = (uint32_t)s;
            if (f.b.w >= 0.f) {
                cr.a = make_float4(f.a.x, f.a.y, f.a.z, sqrtf(f.b.w) * 1.0001f);
                cr.b = make_float4(-f.k.x, -f.k.y, -f.k.z, (float)s64[s].om);
                x[h] = cr.a;
            }
        }
        crit[s] = cr;
        if (rec) {
            float4 *dst = rec[s].v;
            dst[0] = f.a;
            dst[1] = make_float4(f.b.x, f.b.y, f.b.z, f.e.w);
            dst[2] = make_float4(f.d.x, f.d.y, f.d.z, f.k.w);
            dst[3] = make_float4(f.e.x, f.e.y, f.e.z, f.b.w);
        }
    }
    const TreeCap c = warp_ball(x);
    if (lane == 0) caps[t] = c;
}

// One warp per tile of 64 samples in velocity order.
__global__ void __launch_bounds__(256) k_tree_vcrit(const TreeCrit *__restrict__ crit, const Seg32 *__restrict__ s32,
                                                    const uint32_t *__restrict__ vperm,
                                                    const uint32_t *__restrict__ inv, int64_t n, int64_t ntile,
                                                    TreeCrit *__restrict__ vcrit, TreeCap *__restrict__ vcaps,
                                                    uint32_t *__restrict__ vidx)
{
    const int lane = threadIdx.x & 31;
    const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (t >= ntile) return;
    float4 x[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t k = t * kTreeS + 32 * h + lane;
        TreeCrit cr;
        cr.a = make_float4(0.f, 0.f, 0.f, 0.f);
        cr.b = make_float4(0.f, 0.f, 0.f, kCritSkip);
        x[h] = make_float4(0.f, 0.f, 0.f, -1.f);
        uint32_t r = 0;
        if (k < n) {
            r = inv[vperm[k]];
            cr = crit[r];
            if (cr.b.w < kCritSkip) {
                const float4 d = s32[r].d;
                x[h] = make_float4(d.x, d.y, d.z, 0.f);
            }
        }
        vcrit[k] = cr;
        vidx[k] = r;
    }
    const TreeCap c = warp_ball(x);
    if (lane == 0) vcaps[t] = c;
}

// frame from a centre direction and a rough tangent; extents are filled in by the caller
__device__ __forceinline__ void make_frame(double cx, double cy, double cz, double tx, double ty, double tz,
                                           TreeGeo &g)
{
    const double c2 = cx * cx + cy * cy + cz * cz;
    if (!(c2 > 0.0)) cx = cy = 0.0, cz = 1.0;   // no mean direction: any will do
    const double r = c2 > 0.0 ? 1.0 / sqrt(c2) : 1.0;
    g.n0[0] = cx * r;
    g.n0[1] = cy * r;
    g.n0[2] = cz * r;
    double t = tx * g.n0[0] + ty * g.n0[1] + tz * g.n0[2];
    double ux = tx - t * g.n0[0], uy = ty - t * g.n0[1], uz = tz - t * g.n0[2];
    double u2 = ux * ux + uy * uy + uz * uz;
    if (!(u2 > 1e-12 * (tx * tx + ty * ty + tz * tz)) || !(u2 > 0.0)) {   // no tangent: any will do
        ux = fabs(g.n0[2]) < 0.9 ? -g.n0[1] : 0.0;
        uy = fabs(g.n0[2]) < 0.9 ? g.n0[0] : -g.n0[2];
        uz = fabs(g.n0[2]) < 0.9 ? 0.0 : g.n0[1];
        u2 = ux * ux + uy * uy + uz * uz;
    }
    const double ru = 1.0 / sqrt(u2);
    g.e1[0] = ux * ru;
    g.e1[1] = uy * ru;
    g.e1[2] = uz * ru;
    // once more against the rounding of the first projection
    t = g.e1[0] * g.n0[0] + g.e1[1] * g.n0[1] + g.e1[2] * g.n0[2];
    for (int c = 0; c < 3; ++c) g.e1[c] -= t * g.n0[c];
    const double rv = 1.0 / sqrt(g.e1[0] * g.e1[0] + g.e1[1] * g.e1[1] + g.e1[2] * g.e1[2]);
    for (int c = 0; c < 3; ++c) g.e1[c] *= rv;
    g.e2[0] = g.n0[1] * g.e1[2] - g.n0[2] * g.e1[1];
    g.e2[1] = g.n0[2] * g.e1[0] - g.n0[0] * g.e1[2];
    g.e2[2] = g.n0[0] * g.e1[1] - g.n0[1] * g.e1[0];
}

// A direction at angle theta from the centre has 2 - d^2 / 2 = 1 + cos(theta); the corners of a rectangle of
// half-sizes 1 have 2/3.
constexpr float kWideDen = 0.6f, kWideExtent = 1e3f;

// the float copies of a finished geometry, with the near radius D or the marks
__device__ __forceinline__ void finish_geo(TreeGeo &g, double D, bool empty)
{
    if (empty) {
        D = kEmptyRadius;
    } else if (!(fmax(g.a1, g.a2) <= 1.0) || !(D < kWideRadius)) {
        D = kWideRadius;
        g.a1 = g.a2 = kWideExtent;
    }
    g.pad = 0.0;
    g.c = make_float4((float)g.n0[0], (float)g.n0[1], (float)g.n0[2], (float)D);
    g.l = make_float4((float)(g.n0[0] - (double)g.c.x), (float)(g.n0[1] - (double)g.c.y),
                      (float)(g.n0[2] - (double)g.c.z), 0.f);
    g.f1 = make_float4((float)g.e1[0], (float)g.e1[1], (float)g.e1[2], (float)(1.0 / g.a1));
    g.f2 = make_float4((float)g.e2[0], (float)g.e2[1], (float)g.e2[2], (float)(1.0 / g.a2));
}

// Finest clusters, W warps each and G clusters per CTA; the frames of a CTA's clusters are made by as many lanes
// of one warp.  Sums in float are enough: they only choose the centre and frame, and the extents are measured
// from the pixels afterwards.
template <int T, int W, int G>
__global__ void __launch_bounds__(32 * W * G) k_tree_leaf_geo(const double *__restrict__ nv, int64_t ldn,
                                                              const int64_t *__restrict__ outidx, int order, double theta_pix,
                                                              double kappa, int64_t ncl, TreeGeo *__restrict__ geo)
{
    __shared__ float red[G][W][7];
    __shared__ TreeGeo gs[G];
    const int tid = threadIdx.x, lane = tid & 31, w = tid / 32 % W, own = tid / (32 * W);
    const int64_t t = blockIdx.x * (int64_t)G + own;
    if (t < ncl) {
        float s[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int l = 32 * w + lane; l < T * T; l += 32 * W) {
            const int64_t k = t * T * T + l;
            if (outidx[k] < 0) continue;
            int lx = T / 2, ly;
            if (order == kSlotsDiag) diag_slot_square(l, T, lx, ly);
            else if (order == kSlotsRows) lx = l % T;
            // a list has no axis of its own: the frame is then any
            const float f = order == kSlotsList ? 0.f : (float)lx - 0.5f * (float)(T - 1);
            for (int c = 0; c < 3; ++c) {
                const float v = trunc_float(nv[c * ldn + k]);
                s[c] += v;
                s[3 + c] += f * v;
            }
            s[6] = 1.f;   // has pixels
        }
        for (int c = 0; c < 7; ++c) {
            s[c] = warp_sum(s[c]);
            if (lane == 0) red[own][w][c] = s[c];
        }
    }
    __syncthreads();
    const int64_t t1 = blockIdx.x * (int64_t)G + tid;   // the cluster whose frame this thread makes
    const bool maker = tid < G && t1 < ncl;
    bool empty = false;
    if (maker) {
        double a[7];
        for (int c = 0; c < 7; ++c) {
            a[c] = 0.0;
            for (int i = 0; i < W; ++i) a[c] += red[tid][i][c];
        }
        empty = a[6] == 0.0;
        make_frame(a[0], a[1], a[2], a[3], a[4], a[5], gs[tid]);
    }
    __syncthreads();
    if (t < ncl) {
        const TreeGeo &g = gs[own];
        const float e1x = trunc_float(g.e1[0]), e1y = trunc_float(g.e1[1]), e1z = trunc_float(g.e1[2]);
        const float e2x = trunc_float(g.e2[0]), e2y = trunc_float(g.e2[1]), e2z = trunc_float(g.e2[2]);
        float m1 = 0.f, m2 = 0.f;
        for (int l = 32 * w + lane; l < T * T; l += 32 * W) {
            const int64_t k = t * T * T + l;
            if (outidx[k] < 0) continue;
            const float dx = trunc_float(nv[k] - g.n0[0]), dy = trunc_float(nv[ldn + k] - g.n0[1]),
                        dz = trunc_float(nv[2 * ldn + k] - g.n0[2]);
            const float den = 2.f - 0.5f * (dx * dx + dy * dy + dz * dz), s = 1.f / den;
            m1 = fmaxf(m1, fabsf(dx * e1x + dy * e1y + dz * e1z) * s);
            m2 = fmaxf(m2, fabsf(dx * e2x + dy * e2y + dz * e2z) * s);
            if (!(den > kWideDen)) m1 = kWideExtent;
        }
        m1 = warp_max(m1);
        m2 = warp_max(m2);
        if (lane == 0) {
            red[own][w][0] = m1;
            red[own][w][1] = m2;
        }
    }
    __syncthreads();
    if (maker) {
        TreeGeo &g = gs[tid];
        float m1 = 0.f, m2 = 0.f;
        for (int i = 0; i < W; ++i) {
            m1 = fmaxf(m1, red[tid][i][0]);
            m2 = fmaxf(m2, red[tid][i][1]);
        }
        // margin for the float arithmetic; a single pixel still gets a square of a quarter pixel
        g.a1 = fmax((double)m1 * 1.00001, 0.125 * theta_pix);
        g.a2 = fmax((double)m2 * 1.00001, 0.125 * theta_pix);
        finish_geo(g, near_radius(kappa, fmax(g.a1, g.a2)) * 1.00001 + 1e-7, empty);
        geo[t1] = g;
    }
}
// With 16 clusters for every SM the FP64 unit bounds a CTA per cluster, whose frame is the work of one thread:
// a warp per cluster and 16 per CTA take 270 us at N_side 1024 (49,152 clusters) instead of 719.  With fewer the
// latency of a CTA counts: at N_side 64 (192 clusters) 12 us with a CTA each, 17 with 16 per CTA.
template <int T>
void launch_leaf_geo(const double *nv, int64_t ldn, const int64_t *outidx, int order, double theta_pix, double kappa, int64_t ncl,
                     TreeGeo *geo, cudaStream_t s)
{
    constexpr int W = T * T / 128;
    if (ncl < 16 * 152)
        k_tree_leaf_geo<T, W, 1><<<(unsigned)ncl, 32 * W, 0, s>>>(nv, ldn, outidx, order, theta_pix, kappa, ncl, geo);
    else
        k_tree_leaf_geo<T, 1, 16><<<(unsigned)((ncl + 15) / 16), 512, 0, s>>>(nv, ldn, outidx, order, theta_pix, kappa, ncl, geo);
}

// Four lanes per parent cluster (tree_parent of the child level), a lane per child: points of the child's
// rectangle (corners and edge midpoints).  Offsets from the parent's centre are differences of FP64 centres plus a
// float offset, so they keep their relative accuracy for small clusters.  Children without pixels are left out
// (a list's invalid entries sort last, so they are the last ones), and a parent of none but those is one itself.
// With a warp per parent every lane
// repeated the frame's FP64 work (N_side 1024, five levels: 178 us, so 50 us).
__global__ void __launch_bounds__(128) k_tree_up_geo(const TreeGeo *__restrict__ child, int cnb, int64_t cncl,
                                                     TreeGeo *__restrict__ geo, int nb, int64_t ncl, double kappa)
{
    const int c = threadIdx.x & 3;
    const int64_t p = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 2, t = p < ncl ? p : ncl - 1;
    int64_t kid, kid0;
    bool has;
    if (nb == 0) {
        kid0 = 4 * t;
        kid = kid0 + c;
        has = kid < cncl;
    } else {
        const int64_t f = t / ((int64_t)nb * nb);
        const int by = (int)(t - f * nb * nb) / nb, bx = (int)(t - f * nb * nb) % nb;
        const int i = 2 * bx + (c & 1), j = 2 * by + (c >> 1);
        has = i < cnb && j < cnb;
        kid = (f * cnb + j) * cnb + i;
        kid0 = (f * cnb + 2 * by) * cnb + 2 * bx;
    }
    const TreeGeo k = child[has ? kid : kid0];
    has = has && !tree_empty(k.c);
    const float on = has ? 1.f : 0.f;
    auto sum4 = [](float v) {
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        return v + __shfl_xor_sync(0xffffffffu, v, 2);
    };
    auto max4 = [](float v) {
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
        return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
    };
    const float cx = sum4(on * k.c.x), cy = sum4(on * k.c.y), cz = sum4(on * k.c.z);
    const float ux = sum4(on * k.f1.x), uy = sum4(on * k.f1.y), uz = sum4(on * k.f1.z);
    const bool empty = sum4(on) == 0.f;
    TreeGeo g;
    make_frame(cx, cy, cz, ux, uy, uz, g);
    const float d0 = (float)(k.n0[0] - g.n0[0]), d1 = (float)(k.n0[1] - g.n0[1]), d2 = (float)(k.n0[2] - g.n0[2]);
    const float a1 = (float)k.a1, a2 = (float)k.a2;
    const float g1x = (float)g.e1[0], g1y = (float)g.e1[1], g1z = (float)g.e1[2];
    const float g2x = (float)g.e2[0], g2y = (float)g.e2[1], g2z = (float)g.e2[2];
    float m1 = 0.f, m2 = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int pt = q < 4 ? q : q + 1;   // 3 x 3 points without the middle one
        const float xi = (float)(pt % 3 - 1) * a1, eta = (float)(pt / 3 - 1) * a2;
        const float r2 = xi * xi + eta * eta, s = 2.f / (1.f + r2);
        const float x = d0 + s * (xi * k.f1.x + eta * k.f2.x - r2 * k.c.x);
        const float y = d1 + s * (xi * k.f1.y + eta * k.f2.y - r2 * k.c.y);
        const float z = d2 + s * (xi * k.f1.z + eta * k.f2.z - r2 * k.c.z);
        const float den = 2.f - 0.5f * (x * x + y * y + z * z), ps = 1.f / den;
        m1 = fmaxf(m1, fabsf(x * g1x + y * g1y + z * g1z) * ps);
        m2 = fmaxf(m2, fabsf(x * g2x + y * g2y + z * g2z) * ps);
        if (!(den > kWideDen)) m1 = kWideExtent;
    }
    m1 = max4(has ? m1 : 0.f);
    m2 = max4(has ? m2 : 0.f);
    g.a1 = empty ? 1.0 : (double)m1 * 1.002;
    g.a2 = empty ? 1.0 : (double)m2 * 1.002;
    // near at a child implies near here
    const float cd = max4(has ? (k.c.w + sqrtf(d0 * d0 + d1 * d1 + d2 * d2)) * 1.00003f + 2e-6f : 0.f);
    const double D = fmax(near_radius(kappa, fmax(g.a1, g.a2)) * 1.00001 + 1e-7, (double)cd);
    if (c == 0 && p < ncl) {
        finish_geo(g, D, empty);
        geo[p] = g;
    }
}
void launch_up_geo(const TreeGeo *child, int cnb, int64_t cncl, TreeGeo *geo, int nb, int64_t ncl, double kappa, cudaStream_t s)
{
    k_tree_up_geo<<<(unsigned)((ncl + 31) / 32), 128, 0, s>>>(child, cnb, cncl, geo, nb, ncl, kappa);
}

__device__ __forceinline__ void load_geo(TreeGeo *dst, const TreeGeo *src)
{
    constexpr int W = sizeof(TreeGeo) / 4;
    static_assert(sizeof(TreeGeo) % 4 == 0 && W <= kTreeNT, "geometry copy");
    if ((int)threadIdx.x < W) reinterpret_cast<uint32_t *>(dst)[threadIdx.x] = reinterpret_cast<const uint32_t *>(src)[threadIdx.x];
}

__device__ __forceinline__ float comp(const float4 &v, int c) { return c == 0 ? v.x : (c == 1 ? v.y : v.z); }

// Coordinates in [-1, 1]^2 of direction n0 + d (float offset d from the centre)
__device__ __forceinline__ void local_xy(const TreeGeo &g, float dx, float dy, float dz, float &x, float &y)
{
    const float s = __fdividef(1.f, 2.f - 0.5f * fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
    x = fmaf(dz, g.f1.z, fmaf(dy, g.f1.y, dx * g.f1.x)) * (s * g.f1.w);
    y = fmaf(dz, g.f2.z, fmaf(dy, g.f2.y, dx * g.f2.x)) * (s * g.f2.w);
}

// chord from the centre to the farthest point of the cluster's rectangle
__device__ __forceinline__ float target_radius(const TreeGeo &g)
{
    const float r2 = (float)(g.a1 * g.a1 + g.a2 * g.a2);
    return 2.f * sqrtf(r2 / (1.f + r2)) * 1.0001f + 1e-7f;
}

__device__ __forceinline__ uint64_t dup2(float v) { return f2_pack(v, v); }

// offset from the centre of the node at (xi, eta)
__device__ __forceinline__ void node_offset(const TreeGeo &g, int k, float (&m)[3])
{
    const float xi = (float)(g.a1 * cheb_at<kNP>(1, k % kNP)), eta = (float)(g.a2 * cheb_at<kNP>(1, k / kNP));
    const float r2 = fmaf(xi, xi, eta * eta), s = 2.f / (1.f + r2);
#pragma unroll
    for (int c = 0; c < 3; ++c) m[c] = s * fmaf(xi, comp(g.f1, c), fmaf(eta, comp(g.f2, c), -r2 * comp(g.c, c)));
}

size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

int slots_of(const void *fn, size_t smem, int num_sms)
{
    int nb = 0;
    if (smem > 48 * 1024) cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, kTreeNT, smem);
    return (nb > 0 ? nb : 1) * num_sms;
}

}  // namespace

}  // namespace isw
