// FP32 adjoint of the map over the cluster tree of the pixels (tree.cuh): the derivative sums of a sample
// (adjoint.cu) are smooth in n wherever its pair term is, so for a cluster far from the sample
//   sum_p g_p D(n_p) = sum_nodes G_node D(node),   G_node = sum_p g_p L_node(n_p),
// the transpose of the map's interpolation.
//   k_adj_up       G at the 8 x 8 nodes of every cluster, leaves from the pixels, parents from their
//                  children's nodes; also the offsets of nodes and pixels from their centre
//   k_adj_tree     one thread per sample: depth-first from the root clusters, each sample summed at the
//                  nodes of the first cluster far from it, or at the pixels of the leaves it is near to
//   k_adj_finish   the partial sums of a sample added in a fixed order, gradient rows assembled in FP64
// A CTA holds 128 samples that are neighbours, so that its threads agree on near and far: in position order
// for clusters near by position (and the roots), in velocity order for those near by beam only (a string's
// samples beam in many directions: in position order a third of the clusters would be visited for one or
// two lanes each).  The subtrees of the roots are dealt to up to kAdjParts items per CTA of samples, with
// separate partial sums.
// Bound by the FP32 sums of these pairs (40 operations each).  N_side 256, 50,176 samples: per sample ~1e4
// nodes and pixels instead of 786,432 pixels, 4.1 ms against 43.7 ms pair by pair.
#include "adjoint.cuh"
#include "tree.cuh"

#include <algorithm>

namespace isw {

namespace {

constexpr int kAdjParts = 8, kSums = kAcc;   // most shares of the root clusters
// Near radius in half-sizes: a sample's own gradient sees the truncation that the map averages over
// samples.  Median error of dL/dXdot per sample against FP64: 1.7e-7 at 3.5, 1.4e-7 at 4 (direct kernel
// 1.4e-7); 3.9 ms at 3.5, 4.3 ms at 4.
constexpr double kKappaAdj = 4.0;
constexpr int kPairs = kNN / 2, kPixPairs = kLeaf * kLeaf / 2;

// A pair of targets (nodes or pixels): offsets m from the centre, |m|^2 and weight, (v, v') pairs.
struct __align__(16) AdjPair {
    float4 a, b, c;   // (mx, mx', my, my') (mz, mz', |m|^2, |m'|^2) (g, g', -, -)
};
struct __align__(16) AdjLow {
    float4 a, b;      // low parts of m: (x, x', y, y') (z, z', -, -)
};

struct AdjUpArgs {
    const TreeGeo *geo, *cgeo;      // this level, its children
    int nb, cnb;
    int64_t ncl, cncl;
    const AdjPair *child;           // children's nodes
    AdjPair *node;                  // [ncl][32]
    // leaves
    const double *nv;
    int64_t ldn;
    const int64_t *outidx;
    const double *g;
    AdjPair *pix;                   // [ncl][128]
    AdjLow *low;
};

// One CTA of 128 threads per cluster, 256 points (pixels of the leaf, or the nodes of up to four
// children).  Moments m_ij = sum g T_i(x) T_j(y) in float over 32 points at a time, added in FP64, then the
// transposed Chebyshev transform.
template <bool LEAF>
__global__ void __launch_bounds__(128) k_adj_up(AdjUpArgs a)
{
    __shared__ TreeGeo geo;
    __shared__ float tx[256][kNP], ty[256][kNP];
    __shared__ double mom[2][kNN], tmp[kNN];
    const int tid = threadIdx.x;
    const int64_t cl = blockIdx.x;
    load_geo(&geo, a.geo + cl);
    __syncthreads();
    for (int q = 0; q < 2; ++q) {
        const int l = 128 * q + tid;
        float d[3] = {0.f, 0.f, 0.f}, g = 0.f;
        if (LEAF) {
            const int64_t k = cl * 256 + l, oi = a.outidx[k];
            float lo[3] = {0.f, 0.f, 0.f};
            if (oi >= 0) {
                for (int c = 0; c < 3; ++c) {
                    const double v = a.nv[c * a.ldn + k] - geo.n0[c];
                    d[c] = __double2float_rn(v);
                    lo[c] = __double2float_rn(v - (double)d[c]);
                }
                g = __double2float_rn(a.g[oi]);
            }
            float *p = reinterpret_cast<float *>(a.pix + k / 2) + (k & 1), *w = reinterpret_cast<float *>(a.low + k / 2) + (k & 1);
            p[0] = d[0];
            p[2] = d[1];
            p[4] = d[2];
            p[6] = fmaf(d[2], d[2], fmaf(d[1], d[1], d[0] * d[0]));
            p[8] = g;
            w[0] = lo[0];
            w[2] = lo[1];
            w[4] = lo[2];
        } else {
            int64_t kid;
            const int c = l >> 6, k = l & 63;
            bool has;
            if (a.nb == 0) {
                kid = 4 * cl + c;
                has = kid < a.cncl;
            } else {
                const int64_t f = cl / ((int64_t)a.nb * a.nb), rem = cl - f * a.nb * a.nb;
                const int64_t i = 2 * (rem % a.nb) + (c & 1), j = 2 * (rem / a.nb) + (c >> 1);
                has = i < a.cnb && j < a.cnb;
                kid = (f * a.cnb + j) * a.cnb + i;
            }
            if (has && !tree_empty(a.cgeo[kid].c)) {
                const float *p = reinterpret_cast<const float *>(a.child + kid * kPairs + k / 2) + (k & 1);
                const TreeGeo &cg = a.cgeo[kid];
                for (int q3 = 0; q3 < 3; ++q3) d[q3] = p[2 * q3] + (float)(cg.n0[q3] - geo.n0[q3]);
                g = p[8];
            }
        }
        float x, y;
        local_xy(geo, d[0], d[1], d[2], x, y);
        tx[l][0] = 1.f;
        tx[l][1] = x;
        ty[l][0] = g;
        ty[l][1] = g * y;
        for (int i = 2; i < kNP; ++i) {
            tx[l][i] = fmaf(2.f * x, tx[l][i - 1], -tx[l][i - 2]);
            ty[l][i] = fmaf(2.f * y, ty[l][i - 1], -ty[l][i - 2]);
        }
    }
    __syncthreads();
    {
        const int i = tid & 7, j = tid >> 3 & 7, half = tid >> 6;
        double v = 0.0;
        for (int p0 = 128 * half; p0 < 128 * half + 128; p0 += 32) {
            float s = 0.f;
#pragma unroll 8
            for (int p = p0; p < p0 + 32; ++p) s = fmaf(tx[p][i], ty[p][j], s);
            v += (double)s;
        }
        mom[half][j * kNP + i] = v;
    }
    __syncthreads();
    if (tid < kNN) {   // along xi: node (k, j) <- sum over i
        const int j = tid / kNP, k = tid % kNP;
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < kNP; ++i)
            v = fma((mom[0][j * kNP + i] + mom[1][j * kNP + i]) * (i == 0 ? 1.0 / kNP : 2.0 / kNP), cheb_at<kNP>(i, k), v);
        tmp[tid] = v;
    }
    __syncthreads();
    if (tid < kNN) {
        const int l = tid / kNP, k = tid % kNP;
        double v = 0.0;
#pragma unroll
        for (int j = 0; j < kNP; ++j) v = fma(tmp[j * kNP + k] * (j == 0 ? 1.0 / kNP : 2.0 / kNP), cheb_at<kNP>(j, l), v);
        float m[3];
        node_offset(geo, tid, m);
        float *p = reinterpret_cast<float *>(a.node + cl * kPairs + tid / 2) + (tid & 1);
        p[0] = m[0];
        p[2] = m[1];
        p[4] = m[2];
        p[6] = fmaf(m[2], m[2], fmaf(m[1], m[1], m[0] * m[0]));
        p[8] = (float)v;
    }
}

struct AdjTreeArgs {
    const TreeCrit *crit, *vcrit;
    const uint32_t *vidx;
    const TreeRec *rec;
    const Seg64 *s64;
    int levels;
    const TreeGeo *geo[kTreeLevels];
    const AdjPair *node[kTreeLevels];
    int nb[kTreeLevels];
    int64_t ncl[kTreeLevels];
    const AdjPair *pix;
    const AdjLow *low;
    const double *nv, *g;
    int64_t ldn;
    const int64_t *outidx;
    int64_t n_pad;                 // samples, padded to the tiles of 128
    int parts;
    double *partial;               // [2][parts][adj_rows][n_pad]
    float b_min;
    DevStatus *st;
    unsigned long long *queue;
};

// A sample relative to the centre of a cluster (see stage_sample in tree.cu), each value twice.
struct AdjRel {
    uint64_t D2[3], K, xd[3], P, xpn[3], Qn, B0, f;
};

// Queue of FP64 pairs (lane's sample, pixel) of a warp.
struct AdjQueue {
    uint32_t src[64];
    uint32_t pix[64];     // slot in the pixel table's leaf
    uint8_t who[64];
    double val[32];
};

struct __align__(16) AdjSmem {
    AdjPair tgt[kPixPairs];
    AdjLow low[kPixPairs];
    TreeGeo geo;
    double acc64[kSums][kTreeNT];
    AdjQueue q[kTreeNT / 32];
    int stack_level[4 * kTreeLevels + 8];
    int64_t stack_cl[4 * kTreeLevels + 8];
    int64_t item;
};

// The derivative sums of one sample over np pairs of targets, far form (the sample is not close to any of
// them): 34 FP32 operations and two reciprocals per target.  s: gq, ga, gT, ge, v, ge m (3), w m (3) and,
// for ten rows, gb Qd, u m (3).
template <bool NG9>
__device__ __forceinline__ void adj_sums(const AdjPair *__restrict__ t, int np, const AdjRel &r, float (&s)[15])
{
    constexpr int N = NG9 ? 15 : 11;
    uint64_t p[N];
#pragma unroll
    for (int k = 0; k < N; ++k) p[k] = 0ull;
#pragma unroll 2
    for (int i = 0; i < np; ++i) {
        const ulonglong2 ta = *reinterpret_cast<const ulonglong2 *>(&t[i].a), tb = *reinterpret_cast<const ulonglong2 *>(&t[i].b);
        const uint64_t g = *reinterpret_cast<const uint64_t *>(&t[i].c);
        const uint64_t mx = ta.x, my = ta.y, mz = tb.x;
        const uint64_t Q = f2_fma(mz, r.D2[2], f2_fma(my, r.D2[1], f2_fma(mx, r.D2[0], f2_add(tb.y, r.K))));
        const uint64_t h = f2_fma(mz, r.xd[2], f2_fma(my, r.xd[1], f2_mul(mx, r.xd[0])));
        const uint64_t Qdn = f2_fma(mz, r.xpn[2], f2_fma(my, r.xpn[1], f2_fma(mx, r.xpn[0], r.Qn)));   // -X'.d
        const uint64_t B = f2_add(h, r.B0), Pd = f2_add(h, r.P), A = f2_sub(r.f, Qdn);
        float q0, q1, b0, b1;
        f2_unpack(Q, q0, q1);
        f2_unpack(B, b0, b1);
        const uint64_t iQ = f2_pack(rcp_approx(q0), rcp_approx(q1)), iB = f2_pack(rcp_approx(b0), rcp_approx(b1));
        const uint64_t gq = f2_mul(g, iQ), gqb = f2_mul(gq, iB), ga = f2_mul(gqb, A);
        const uint64_t gT = f2_mul(gqb, f2_fma(A, Qdn, f2_mul(B, Pd))), ge = f2_mul(gT, iQ);
        const uint64_t t1n = f2_mul(Qdn, iB), vn = f2_mul(ga, t1n);   // -(X'.d)/B, -v
        const uint64_t w = f2_sub(gq, vn);
        p[0] = f2_add(p[0], gq);
        p[1] = f2_add(p[1], ga);
        p[2] = f2_add(p[2], gT);
        p[3] = f2_add(p[3], ge);
        p[4] = f2_add(p[4], vn);
        p[5] = f2_fma(ge, mx, p[5]);
        p[6] = f2_fma(ge, my, p[6]);
        p[7] = f2_fma(ge, mz, p[7]);
        p[8] = f2_fma(w, mx, p[8]);
        p[9] = f2_fma(w, my, p[9]);
        p[10] = f2_fma(w, mz, p[10]);
        if (NG9) {
            const uint64_t bq = f2_mul(gq, t1n), u = f2_sub(ga, bq);   // -g Qd/(BQ)
            p[11] = f2_add(p[11], bq);
            p[12] = f2_fma(u, mx, p[12]);
            p[13] = f2_fma(u, my, p[13]);
            p[14] = f2_fma(u, mz, p[14]);
        }
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
        float lo, hi;
        f2_unpack(p[k], lo, hi);
        s[k] = lo + hi;
    }
}

// Evaluate the first cnt <= 32 queued pairs in FP64 and add them to their samples' sums in queue order.
__device__ __noinline__ void adj_flush(AdjQueue &q, int cnt, const AdjTreeArgs &a, int64_t leaf0, double (*acc)[kTreeNT],
                                       unsigned &zerocnt)
{
    const int lane = threadIdx.x & 31, wbase = threadIdx.x & ~31;
    const bool on = lane < cnt;
    double t[kSums];
#pragma unroll
    for (int k = 0; k < kSums; ++k) t[k] = 0.0;
    const int who = on ? q.who[lane] : 32 + lane;
    if (on) {
        const Seg64 s = a.s64[q.src[lane]];
        const int64_t k = leaf0 + q.pix[lane];
        adj_pair64(a.nv[k], a.nv[a.ldn + k], a.nv[2 * a.ldn + k], a.g[a.outidx[k]], s, 10, t, zerocnt);
    }
    const unsigned peers = __match_any_sync(0xffffffffu, who);
    const bool lead = on && (peers & ((1u << lane) - 1u)) == 0u;
#pragma unroll 1
    for (int k = 0; k < kSums; ++k) {
        __syncwarp();
        double v = t[0];
#pragma unroll
        for (int j = 1; j < kSums; ++j) v = k == j ? t[j] : v;
        q.val[lane] = v;
        __syncwarp();
        if (lead) {
            double s = acc[k][wbase + who];
            for (unsigned m = peers; m; m &= m - 1u) s += q.val[__ffs(m) - 1];
            acc[k][wbase + who] = s;
        }
    }
    __syncwarp();
}

template <bool NG9>
__global__ void __launch_bounds__(kTreeNT) k_adj_tree(AdjTreeArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AdjSmem &sm = *reinterpret_cast<AdjSmem *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    AdjQueue &nq = sm.q[w];
    const int64_t ntile = a.n_pad / kTreeNT, n_items = 2 * ntile * a.parts;
    const int top = a.levels - 1;
    const uint64_t half2 = f2_pack(0.5f, 0.5f);
    const float b_tiny = a.b_min * 1e-3f;
    unsigned nearcnt = 0, zerocnt = 0;
    TreeQueue queue{a.queue, 0ull};
    for (int64_t item = queue.first(&sm.item); item < n_items; item = queue.next(&sm.item)) {
        const int pass = (int)(item / (ntile * a.parts));
        const int64_t tile = item / a.parts % ntile;
        const int part = (int)(item % a.parts);
        const int64_t idx = tile * kTreeNT + tid;
        const uint32_t src = pass ? a.vidx[idx] : (uint32_t)idx;
        const float4 ca = (pass ? a.vcrit : a.crit)[idx].a, cb = (pass ? a.vcrit : a.crit)[idx].b;
        const bool real = cb.w < kCritSkip;
        float4 q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) q[k] = a.rec[src].v[k];
        float ahi[kSums], alo[kSums];
#pragma unroll
        for (int k = 0; k < kSums; ++k) {
            ahi[k] = alo[k] = 0.f;
            sm.acc64[k][tid] = 0.0;
        }
        const float em1 = fmaf(q[2].z, q[0].z, fmaf(q[2].y, q[0].y, q[2].x * q[0].x));   // Xdot.Xhat
        // sums of one cluster -> the accumulators of adj_assemble, D and n0 put back
        auto add = [&](const float (&s)[15], const float (&D)[3], const TreeGeo &g) {
            fold(ahi[0], alo[0], fmaf(em1, s[0], -q[1].w * s[1]));
            fold(ahi[1], alo[1], s[0]);
            fold(ahi[2], alo[2], s[1]);
            fold(ahi[3], alo[3], s[2]);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                fold(ahi[4 + c], alo[4 + c], 2.f * fmaf(s[3], D[c], s[5 + c]));
                fold(ahi[7 + c], alo[7 + c], fmaf(s[0], D[c], fmaf(-s[4], comp(g.c, c), s[8 + c])));
                if (NG9) fold(ahi[10 + c], alo[10 + c], fmaf(s[1], D[c], fmaf(-s[11], comp(g.c, c), s[12 + c])));
            }
        };
        // the sample relative to the staged cluster's centre
        auto relate = [&](const TreeGeo &g, AdjRel &r, float (&D)[3], float (&Dl)[3], float (&W)[3]) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float nh = comp(g.c, c), xh = comp(q[0], c), t = nh - xh, bb = t - nh;
                const float e = ((nh - (t - bb)) - (xh + bb)) + (comp(g.l, c) - comp(q[1], c));
                D[c] = t + e;
                Dl[c] = e - (D[c] - t);
            }
            const float P = fmaf(q[2].z, D[2], fmaf(q[2].y, D[1], q[2].x * D[0]));
            const float Q = fmaf(q[3].z, D[2], fmaf(q[3].y, D[1], q[3].x * D[0]));
            const float K = fmaf(D[2], D[2], fmaf(D[1], D[1], D[0] * D[0]));
            const float om = q[2].w, v = 1.f - om, iv = v > 0.f ? 1.f / v : 0.f;
            W[0] = fmaf(q[2].x, iv, g.c.x);
            W[1] = fmaf(q[2].y, iv, g.c.y);
            W[2] = fmaf(q[2].z, iv, g.c.z);
            const float B0 = fmaf(0.5f * v, fmaf(W[2], W[2], fmaf(W[1], W[1], W[0] * W[0])), om);
#pragma unroll
            for (int c = 0; c < 3; ++c) r.D2[c] = dup2(2.f * D[c]);
            r.K = dup2(K);
            r.xd[0] = dup2(q[2].x);
            r.xd[1] = dup2(q[2].y);
            r.xd[2] = dup2(q[2].z);
            r.P = dup2(P);
            r.xpn[0] = dup2(-q[3].x);
            r.xpn[1] = dup2(-q[3].y);
            r.xpn[2] = dup2(-q[3].z);
            r.Qn = dup2(-Q);
            r.B0 = dup2(B0);
            r.f = dup2(q[1].w);
        };
        for (int64_t root = part; root < a.ncl[top]; root += a.parts) {
            int sp = 0;
            __syncthreads();
            if (tid == 0) {
                sm.stack_level[0] = top;
                sm.stack_cl[0] = root;
            }
            sp = 1;
            while (sp > 0) {
                __syncthreads();   // the stack's writes; the previous cluster's readers are done
                --sp;
                const int L = sm.stack_level[sp];
                const int64_t cl = sm.stack_cl[sp];
                load_geo(&sm.geo, a.geo[L] + cl);
                const float4 self = a.geo[L][cl].c;
                if (tree_empty(self)) continue;
                bool act = real;
                if (L < top) {
                    const float4 par = a.geo[L + 1][tree_parent(cl, a.nb[L], a.nb[L + 1])].c;
                    const bool pp = tree_near_pos(ca, par);
                    act = act && (pass ? !pp && tree_near_beam(cb, par) : pp);
                }
                const bool np = tree_near_pos(ca, self), nbm = tree_near_beam(cb, self);
                // summed here: far from it; the root's far samples belong to the position pass
                const bool far = act && !np && !nbm && (L < top || pass == 0);
                // down to where the sample is near by the pass's own criterion at the parent
                const bool deep = real && (pass ? nbm : np);
                const bool leaf = L == 0 && act && (np || nbm) && (L < top || (pass ? !np : np));
                const bool any_far = __syncthreads_or(far), any_deep = __syncthreads_or(L > 0 ? deep : leaf);
                if (any_far) {
                    const float4 *gsrc = reinterpret_cast<const float4 *>(a.node[L] + cl * kPairs);
                    for (int k = tid; k < kPairs * 3; k += kTreeNT) reinterpret_cast<float4 *>(sm.tgt)[k] = gsrc[k];
                    __syncthreads();
                    if (__any_sync(0xffffffffu, far)) {
                        AdjRel r;
                        float D[3], Dl[3], W[3], s[15];
                        relate(sm.geo, r, D, Dl, W);
                        adj_sums<NG9>(sm.tgt, kPairs, r, s);
                        if (far) add(s, D, sm.geo);
                    }
                }
                if (L > 0) {
                    if (any_deep) {   // children
                        const int cnb = a.nb[L - 1];
                        for (int c = 3; c >= 0; --c) {
                            int64_t kid;
                            bool has;
                            if (cnb == 0) {
                                kid = 4 * cl + c;
                                has = kid < a.ncl[L - 1];
                            } else {
                                const int64_t nb = a.nb[L], f = cl / (nb * nb), rem = cl - f * nb * nb;
                                const int64_t i = 2 * (rem % nb) + (c & 1), j = 2 * (rem / nb) + (c >> 1);
                                has = i < cnb && j < cnb;
                                kid = (f * cnb + j) * cnb + i;
                            }
                            if (has) {
                                if (tid == 0) {
                                    sm.stack_level[sp] = L - 1;
                                    sm.stack_cl[sp] = kid;
                                }
                                ++sp;
                            }
                        }
                    }
                    continue;
                }
                if (!any_deep) continue;
                // pixels of the leaf
                __syncthreads();
                {
                    const float4 *p = reinterpret_cast<const float4 *>(a.pix + cl * kPixPairs);
                    for (int k = tid; k < kPixPairs * 3; k += kTreeNT) reinterpret_cast<float4 *>(sm.tgt)[k] = p[k];
                    const float4 *l = reinterpret_cast<const float4 *>(a.low + cl * kPixPairs);
                    for (int k = tid; k < kPixPairs * 2; k += kTreeNT) reinterpret_cast<float4 *>(sm.low)[k] = l[k];
                }
                __syncthreads();
                if (!__any_sync(0xffffffffu, leaf)) continue;
                AdjRel r;
                float D[3], Dl[3], W[3], s[15];
                relate(sm.geo, r, D, Dl, W);
                const float R = target_radius(sm.geo);
                float4 ball = self;
                ball.w = 1.5f * R + 1e-6f;   // tree_near_pos adds rho
                const float rb = sqrtf(2.f * a.b_min) * 1.001f + R + 1e-5f;
                const bool close = leaf && (tree_near_pos(ca, ball) || tree_beam2(cb, self) < rb * rb);
                if (!__any_sync(0xffffffffu, close)) {
#pragma unroll 1
                    for (int p0 = 0; p0 < kPixPairs; p0 += 32) {
                        adj_sums<NG9>(sm.tgt + p0, 32, r, s);
                        if (leaf) add(s, D, sm.geo);
                    }
                    continue;
                }
                const float rho2 = q[3].w, om = q[2].w;
                const uint64_t om2 = dup2(om), hv2 = dup2(fmaf(-0.5f, om, 0.5f));
                const uint64_t W0 = dup2(W[0]), W1 = dup2(W[1]), W2 = dup2(W[2]);
                const uint64_t l0 = dup2(Dl[0]), l1 = dup2(Dl[1]), l2 = dup2(Dl[2]);
                int qlen = 0;
#pragma unroll 1
                for (int p0 = 0; p0 < kPixPairs; p0 += 32) {
                    // gq, ga, gT, v n0-weight, ge d (3), gq d + v m (3), gbQd n0-weight, gbA d + gbQd m (3)
                    uint64_t p[14];
#pragma unroll
                    for (int k = 0; k < 14; ++k) p[k] = 0ull;
#pragma unroll 1
                    for (int i = p0; i < p0 + 32; ++i) {
                        const ulonglong2 ta = *reinterpret_cast<const ulonglong2 *>(&sm.tgt[i].a),
                                         tb = *reinterpret_cast<const ulonglong2 *>(&sm.tgt[i].b);
                        uint64_t g = *reinterpret_cast<const uint64_t *>(&sm.tgt[i].c);
                        const ulonglong2 la = *reinterpret_cast<const ulonglong2 *>(&sm.low[i].a);
                        const uint64_t lz = *reinterpret_cast<const uint64_t *>(&sm.low[i].b);
                        const uint64_t mx = ta.x, my = ta.y, mz = tb.x;
                        const uint64_t dx = f2_add(f2_fma(half2, r.D2[0], mx), f2_add(la.x, l0));
                        const uint64_t dy = f2_add(f2_fma(half2, r.D2[1], my), f2_add(la.y, l1));
                        const uint64_t dz = f2_add(f2_fma(half2, r.D2[2], mz), f2_add(lz, l2));
                        const uint64_t Q = f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx)));
                        const uint64_t Pd = f2_fma(r.xd[2], dz, f2_fma(r.xd[1], dy, f2_mul(r.xd[0], dx)));
                        const uint64_t Qdn = f2_fma(r.xpn[2], dz, f2_fma(r.xpn[1], dy, f2_mul(r.xpn[0], dx)));
                        const uint64_t A = f2_sub(r.f, Qdn);
                        const uint64_t wx = f2_add(W0, mx), wy = f2_add(W1, my), wz = f2_add(W2, mz);
                        const uint64_t B = f2_fma(hv2, f2_fma(wz, wz, f2_fma(wy, wy, f2_mul(wx, wx))), om2);
                        float q0, q1, b0, b1, g0, g1;
                        f2_unpack(Q, q0, q1);
                        f2_unpack(B, b0, b1);
                        f2_unpack(g, g0, g1);
                        const bool n0 = q0 < rho2 || b0 < b_tiny, n1 = q1 < rho2 || b1 < b_tiny;
                        // near pairs: zero weight here, with the reciprocals kept finite
                        const uint64_t iQ = f2_pack(n0 ? 0.f : rcp_approx(q0), n1 ? 0.f : rcp_approx(q1)),
                                       iB = f2_pack(n0 ? 0.f : rcp_approx(b0), n1 ? 0.f : rcp_approx(b1));
                        const uint64_t gq = f2_mul(g, iQ), gqb = f2_mul(gq, iB), ga = f2_mul(gqb, A);
                        const uint64_t gT = f2_mul(gqb, f2_fma(A, Qdn, f2_mul(B, Pd))), ge = f2_mul(gT, iQ);
                        const uint64_t t1n = f2_mul(Qdn, iB), vn = f2_mul(ga, t1n);
                        p[0] = f2_add(p[0], gq);
                        p[1] = f2_add(p[1], ga);
                        p[2] = f2_add(p[2], gT);
                        p[3] = f2_add(p[3], vn);
                        p[4] = f2_fma(ge, dx, p[4]);
                        p[5] = f2_fma(ge, dy, p[5]);
                        p[6] = f2_fma(ge, dz, p[6]);
                        p[7] = f2_fma(gq, dx, f2_fma(f2_neg(vn), mx, p[7]));
                        p[8] = f2_fma(gq, dy, f2_fma(f2_neg(vn), my, p[8]));
                        p[9] = f2_fma(gq, dz, f2_fma(f2_neg(vn), mz, p[9]));
                        if (NG9) {
                            const uint64_t bqn = f2_mul(gq, t1n);   // -g Qd/(BQ)
                            p[10] = f2_add(p[10], bqn);
                            p[11] = f2_fma(ga, dx, f2_fma(f2_neg(bqn), mx, p[11]));
                            p[12] = f2_fma(ga, dy, f2_fma(f2_neg(bqn), my, p[12]));
                            p[13] = f2_fma(ga, dz, f2_fma(f2_neg(bqn), mz, p[13]));
                        }
                        if (__any_sync(0xffffffffu, leaf && (n0 || n1))) {
                            const unsigned below = (1u << lane) - 1u;
#pragma unroll 1
                            for (int u = 0; u < 2; ++u) {
                                const bool hit = leaf && (u ? n1 && g1 != 0.f : n0 && g0 != 0.f);
                                const unsigned m = __ballot_sync(0xffffffffu, hit);
                                if (!m) continue;
                                if (hit) {
                                    const int at = qlen + __popc(m & below);
                                    nq.src[at] = src;
                                    nq.pix[at] = 2 * i + u;
                                    nq.who[at] = (uint8_t)lane;
                                    ++nearcnt;
                                }
                                qlen += __popc(m);
                                __syncwarp();
                                if (qlen >= 32) {
                                    adj_flush(nq, 32, a, cl * 2 * kPixPairs, sm.acc64, zerocnt);
                                    const uint32_t ms = nq.src[32 + lane], mp = nq.pix[32 + lane];
                                    const uint8_t mw = nq.who[32 + lane];
                                    __syncwarp();
                                    nq.src[lane] = ms;
                                    nq.pix[lane] = mp;
                                    nq.who[lane] = mw;
                                    qlen -= 32;
                                    __syncwarp();
                                }
                            }
                        }
                    }
                    if (leaf) {
                        float v[14];
#pragma unroll
                        for (int k = 0; k < 14; ++k) {
                            float lo, hi;
                            f2_unpack(p[k], lo, hi);
                            v[k] = lo + hi;
                        }
                        fold(ahi[0], alo[0], fmaf(em1, v[0], -q[1].w * v[1]));
                        fold(ahi[1], alo[1], v[0]);
                        fold(ahi[2], alo[2], v[1]);
                        fold(ahi[3], alo[3], v[2]);
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            fold(ahi[4 + c], alo[4 + c], 2.f * v[4 + c]);
                            fold(ahi[7 + c], alo[7 + c], fmaf(-v[3], comp(sm.geo.c, c), v[7 + c]));
                            if (NG9) fold(ahi[10 + c], alo[10 + c], fmaf(-v[10], comp(sm.geo.c, c), v[11 + c]));
                        }
                    }
                }
                if (qlen > 0) adj_flush(nq, qlen, a, cl * 2 * kPixPairs, sm.acc64, zerocnt);
            }
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < adj_rows(NG9); ++k)
            a.partial[((int64_t)(pass * a.parts + part) * adj_rows(NG9) + k) * a.n_pad + idx] =
                ((double)ahi[k] + (double)alo[k]) + sm.acc64[k][tid];
        __syncthreads();
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

// vpos[record] = velocity-order position
__global__ void k_adj_vpos(const uint32_t *__restrict__ vidx, int64_t n, uint32_t *__restrict__ vpos)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        vpos[vidx[k]] = (uint32_t)k;
}

// One thread per record: its sums over passes and parts in order, then the gradient rows at the sample's
// place in the input.
__global__ void __launch_bounds__(128) k_adj_finish(const double *__restrict__ partial, int parts, int64_t n, int64_t n_pad,
                                                    const uint32_t *__restrict__ vpos, const uint32_t *__restrict__ perm,
                                                    const Seg64 *__restrict__ s64, int ngrad, double *__restrict__ grad,
                                                    int64_t ld)
{
    const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n) return;
    double acc[kSums];
    const int64_t vp = vpos[s];
    const int nk = adj_rows(ngrad >= 9);
#pragma unroll
    for (int k = 0; k < kSums; ++k) {
        double hi = 0.0, lo = 0.0;
        if (k < nk)
            for (int c = 0; c < 2 * parts; ++c)
                fold64(hi, lo, partial[((int64_t)c * nk + k) * n_pad + (c < parts ? s : vp)]);
        acc[k] = hi + lo;
    }
    double out[10];
    adj_assemble(s64[s], acc, ngrad, out);
    const int64_t dst = perm[s];
    for (int k = 0; k < ngrad; ++k) grad[k * ld + dst] = out[k];
}

}  // namespace

AdjTreePlan adj_tree_plan(int64_t N, int nface, int64_t npix, int64_t n, int ngrad, int num_sms)
{
    AdjTreePlan p{};
    p.map = tree_plan(ISW_F32C, N, nface, npix, n, num_sms);
    p.n_pad = (n + kTreeNT - 1) / kTreeNT * kTreeNT;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += up256(bytes);
        return o;
    };
    const int64_t nst = p.n_pad / kTreeS;
    p.off_queue = take(sizeof(unsigned long long));
    p.off_crit = take((size_t)p.n_pad * sizeof(TreeCrit));
    p.off_vcrit = take((size_t)p.n_pad * sizeof(TreeCrit));
    p.off_caps = take((size_t)2 * nst * sizeof(TreeCap));
    p.off_vidx = take((size_t)p.n_pad * sizeof(uint32_t));
    p.off_inv = take((size_t)p.n_pad * sizeof(uint32_t));   // record of a sample, then velocity position of a record
    p.off_rec = take((size_t)p.n_pad * sizeof(TreeRec));
    for (int L = 0; L < p.map.levels; ++L) {
        p.off_geo[L] = take((size_t)p.map.ncl[L] * sizeof(TreeGeo));
        p.off_node[L] = take((size_t)p.map.ncl[L] * kPairs * sizeof(AdjPair));
    }
    p.off_pix = take((size_t)p.map.ncl[0] * kPixPairs * sizeof(AdjPair));
    p.off_low = take((size_t)p.map.ncl[0] * kPixPairs * sizeof(AdjLow));
    int nb = 0;
    cudaFuncSetAttribute((const void *)&k_adj_tree<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(AdjSmem));
    cudaFuncSetAttribute((const void *)&k_adj_tree<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(AdjSmem));
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void *)&k_adj_tree<true>, kTreeNT, sizeof(AdjSmem));
    p.slots = (nb > 0 ? nb : 1) * num_sms;
    // as many shares as give every resident CTA 16 items: partial sums are 80 or 104 bytes per sample, pass and
    // share, so with eight at any size 2e6 samples took 3.3 GB
    const int64_t tiles = 2 * (p.n_pad / kTreeNT), want = 16 * (int64_t)p.slots;
    p.parts = (int)std::min<int64_t>(kAdjParts, (want + tiles - 1) / tiles);
    p.off_partial = take((size_t)2 * p.parts * adj_rows(ngrad >= 9) * p.n_pad * sizeof(double));
    p.bytes = at;
    return p;
}

cudaError_t launch_adjoint_tree(const AdjTreePlan &p, const AdjTreeCall &m, cudaStream_t s)
{
    unsigned char *b = (unsigned char *)m.scratch;
    unsigned long long *queue = (unsigned long long *)(b + p.off_queue);
    cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    TreeCrit *crit = (TreeCrit *)(b + p.off_crit), *vcrit = (TreeCrit *)(b + p.off_vcrit);
    TreeCap *caps = (TreeCap *)(b + p.off_caps);
    uint32_t *vidx = (uint32_t *)(b + p.off_vidx), *inv = (uint32_t *)(b + p.off_inv);
    TreeRec *rec = (TreeRec *)(b + p.off_rec);
    const int64_t nst = p.n_pad / kTreeS;
    const unsigned tb = (unsigned)((nst * 32 + 255) / 256);
    k_tree_crit<<<tb, 256, 0, s>>>(m.s32, m.s64, m.perm, m.n, nst, crit, caps, rec, inv);
    k_tree_vcrit<<<tb, 256, 0, s>>>(crit, m.s32, m.perm + m.n, inv, m.n, nst, vcrit, caps + nst, vidx);
    k_adj_vpos<<<(unsigned)((m.n + 255) / 256), 256, 0, s>>>(vidx, m.n, inv);
    const TreePlan &t = p.map;
    AdjTreeArgs a{};
    for (int L = 0; L < t.levels; ++L) {
        TreeGeo *geo = (TreeGeo *)(b + p.off_geo[L]);
        AdjPair *node = (AdjPair *)(b + p.off_node[L]);
        AdjUpArgs u{};
        u.geo = geo;
        u.ncl = t.ncl[L];
        u.nb = t.nb[L];
        u.node = node;
        if (L == 0) {
            launch_leaf_geo<kLeaf>(m.nv, m.ldn, m.outidx, m.order, m.theta_pix, kKappaAdj, t.ncl[0], geo, s);
            u.nv = m.nv;
            u.ldn = m.ldn;
            u.outidx = m.outidx;
            u.g = m.g;
            u.pix = (AdjPair *)(b + p.off_pix);
            u.low = (AdjLow *)(b + p.off_low);
            k_adj_up<true><<<(unsigned)t.ncl[0], 128, 0, s>>>(u);
        } else {
            launch_up_geo(a.geo[L - 1], t.nb[L - 1], t.ncl[L - 1], geo, t.nb[L], t.ncl[L], kKappaAdj, s);
            u.cgeo = a.geo[L - 1];
            u.cnb = t.nb[L - 1];
            u.cncl = t.ncl[L - 1];
            u.child = a.node[L - 1];
            k_adj_up<false><<<(unsigned)t.ncl[L], 128, 0, s>>>(u);
        }
        a.geo[L] = geo;
        a.node[L] = node;
        a.nb[L] = t.nb[L];
        a.ncl[L] = t.ncl[L];
    }
    a.crit = crit;
    a.vcrit = vcrit;
    a.vidx = vidx;
    a.rec = rec;
    a.s64 = m.s64;
    a.levels = t.levels;
    a.pix = (const AdjPair *)(b + p.off_pix);
    a.low = (const AdjLow *)(b + p.off_low);
    a.nv = m.nv;
    a.g = m.g;
    a.ldn = m.ldn;
    a.outidx = m.outidx;
    a.n_pad = p.n_pad;
    a.parts = p.parts;
    a.partial = (double *)(b + p.off_partial);
    a.b_min = m.b_min;
    a.st = m.st;
    a.queue = queue;
    const int64_t items = 2 * (p.n_pad / kTreeNT) * p.parts;
    const void *fn = m.ngrad >= 9 ? (const void *)&k_adj_tree<true> : (const void *)&k_adj_tree<false>;
    void *args[] = {(void *)&a};
    cudaLaunchKernel(fn, dim3((unsigned)(items < p.slots ? items : p.slots)), dim3(kTreeNT), args, sizeof(AdjSmem), s);
    k_adj_finish<<<(unsigned)((m.n + 127) / 128), 128, 0, s>>>(a.partial, p.parts, m.n, p.n_pad, inv, m.perm, m.s64, m.ngrad, m.grad,
                                                               m.ld_g);
    return cudaSuccess;
}

}  // namespace isw
