// FP64 adjoint of the map over the cluster tree of the pixels (tree.cuh): as in treeadj.cu the weights of a
// cluster are moved to its nodes (16 x 16), and a sample sums them there when it is far from the cluster, else
// the pixels of the leaves (32 x 32) that it is near to.
//   k_adj_up64     node weights of a level, from the pixels or from the children's nodes; the leaves' pixels
//                  packed in blocks
//   k_adj_tree64   one warp per sample and part of the root clusters: depth first, far clusters collected and
//                  summed 32 at a time, near leaves pixel by pixel
//   k_adj_finish64 the parts in order, gradient rows
// The lanes hold the targets and not the samples, so every decision is the warp's and no lane idles; the FP64
// unit (two FMA lanes per clock and SM) is the bound (86% busy; 30 operations a node, 38 a pixel, about 50 a
// pixel close to the sample), and targets come from L1 at a fiftieth of its rate.  N_side 64 with 5,120
// samples 22.5 -> 13.2 ms, N_side 128 with 20,000 440 -> 86 ms.  Median error of a sample's gradient against
// extended precision: dL/dX 6e-16 to 1.2e-15 (direct kernel 6e-16 to 1.8e-15), dL/dXdot 1.6e-16 to 7e-16
// (1.4e-16 to 5e-16).
#include "adjoint.cuh"
#include "tree.cuh"

namespace isw {

namespace {

constexpr int kNP64 = 16, kNN64 = kNP64 * kNP64, kLeaf64 = 32, kPts = 1024;
constexpr int kAdjMaxParts = 8, kSums = kAcc, kWarps = kTreeNT / 32;
static_assert(kPts == kLeaf64 * kLeaf64 && kPts == 4 * kNN64, "points of a cluster");

struct __align__(16) AdjPix64 {
    double2 a, b;   // (nx, ny) (nz, weight; 0: no pixel)
};

struct AdjUp64Args {
    const TreeGeo *geo, *cgeo;   // this level, its children
    int nb, cnb;
    int64_t ncl, cncl;
    const double *child;         // children's node weights
    double *node;                // [ncl][256]
    const double *nv;            // leaves
    int64_t ldn;
    const int64_t *outidx;
    const double *g;
    int blocks;                  // slots in the order of diag_slot_square: packed as 8 x 4 blocks
    AdjPix64 *pix;               // [ncl][1024]
};

// Offset of node k of cluster g from its centre
__device__ __forceinline__ void node_offset64(const TreeGeo &g, int k, double (&m)[3])
{
    const double xi = g.a1 * cheb_at<kNP64>(1, k % kNP64), eta = g.a2 * cheb_at<kNP64>(1, k / kNP64);
    const double r2 = xi * xi + eta * eta, s = 2.0 / (1.0 + r2);
#pragma unroll
    for (int c = 0; c < 3; ++c) m[c] = s * (xi * g.e1[c] + eta * g.e2[c] - r2 * g.n0[c]);
}

// One CTA of 256 threads per cluster, 1024 points (pixels of the leaf, or the nodes of up to four children),
// 64 at a time.  Moments M_ij = sum g T_i(x) T_j(y), a thread each, then the transposed Chebyshev transform:
// weight of node (k, l) = sum_ij c_i c_j T_i(x_k) T_j(x_l) M_ij with c_0 = 1/16, c_i = 2/16.
template <bool LEAF>
__global__ void __launch_bounds__(kNN64) k_adj_up64(AdjUp64Args a)
{
    constexpr int C = 64;
    __shared__ TreeGeo geo;
    __shared__ double tx[C][kNP64 + 1], ty[C][kNP64 + 1], mom[kNN64], tmp[kNN64];
    const int tid = threadIdx.x;
    const int64_t cl = blockIdx.x;
    load_geo(&geo, a.geo + cl);
    __syncthreads();
    double M = 0.0;
    for (int p0 = 0; p0 < kPts; p0 += C) {
        if (tid < C) {
            const int l = p0 + tid;
            double d[3] = {0.0, 0.0, 0.0}, g = 0.0;
            if (LEAF) {
                int slot = l;
                if (a.blocks) {
                    const int blk = l >> 5, lane = l & 31;
                    slot = diag_index_square(blk % 4 * 8 + (lane & 7), blk / 4 * 4 + (lane >> 3), kLeaf64);
                }
                const int64_t k = cl * kPts + slot, oi = a.outidx[k];
                const double n[3] = {a.nv[k], a.nv[a.ldn + k], a.nv[2 * a.ldn + k]};
                if (oi >= 0) {
                    for (int c = 0; c < 3; ++c) d[c] = n[c] - geo.n0[c];
                    g = a.g[oi];
                }
                AdjPix64 &o = a.pix[cl * kPts + l];
                o.a = make_double2(n[0], n[1]);
                o.b = make_double2(n[2], g);
            } else {
                const int c = l >> 8, k = l & 255;
                int64_t kid;
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
                    const TreeGeo &cg = a.cgeo[kid];
                    node_offset64(cg, k, d);
                    for (int q = 0; q < 3; ++q) d[q] += cg.n0[q] - geo.n0[q];
                    g = a.child[kid * kNN64 + k];
                }
            }
            const double s = 1.0 / (2.0 - 0.5 * (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]));
            const double x = (d[0] * geo.e1[0] + d[1] * geo.e1[1] + d[2] * geo.e1[2]) * (s / geo.a1);
            const double y = (d[0] * geo.e2[0] + d[1] * geo.e2[1] + d[2] * geo.e2[2]) * (s / geo.a2);
            double u0 = 1.0, u1 = x, v0 = g, v1 = g * y;
            for (int i = 0; i < kNP64; ++i) {
                tx[tid][i] = u0;
                ty[tid][i] = v0;
                const double u2 = fma(2.0 * x, u1, -u0), v2 = fma(2.0 * y, v1, -v0);
                u0 = u1, u1 = u2, v0 = v1, v1 = v2;
            }
        }
        __syncthreads();
        double s0 = 0.0, s1 = 0.0;
#pragma unroll 8
        for (int p = 0; p < C; p += 2) {
            s0 = fma(tx[p][tid % kNP64], ty[p][tid / kNP64], s0);
            s1 = fma(tx[p + 1][tid % kNP64], ty[p + 1][tid / kNP64], s1);
        }
        M += s0 + s1;
        __syncthreads();
    }
    const int k = tid % kNP64, l = tid / kNP64;
    mom[tid] = M * (k == 0 ? 1.0 / kNP64 : 2.0 / kNP64);
    __syncthreads();
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < kNP64; ++i) v = fma(mom[l * kNP64 + i], cheb_at<kNP64>(i, k), v);
    tmp[tid] = v * (l == 0 ? 1.0 / kNP64 : 2.0 / kNP64);
    __syncthreads();
    v = 0.0;
#pragma unroll
    for (int j = 0; j < kNP64; ++j) v = fma(tmp[j * kNP64 + k], cheb_at<kNP64>(j, l), v);
    a.node[cl * kNN64 + tid] = v;
}

struct AdjTree64Args {
    const TreeCrit *crit;
    const Seg64 *s64;
    int levels, parts;
    const TreeGeo *geo[kTreeLevels];
    const double *node[kTreeLevels];
    int nb[kTreeLevels];
    int64_t ncl[kTreeLevels];
    const AdjPix64 *pix;
    int64_t n;
    double *partial;   // [parts][adj_rows][n]
    float b_min, d_far;
    DevStatus *st;
    unsigned long long *queue;
};

// A sample at a far cluster: the five forms of k_tree_nodes_f64 times w = (1 + r^2) / 2, each constant + xi +
// eta + square coefficient, in the order |d|^2, B, Xdot.d, A, X'.d
struct __align__(16) AdjFar64 {
    double v[5][4], pad[2];
};
struct AdjWarp64 {
    AdjFar64 far[32];
    int64_t fcl[32], stack_cl[4 * kTreeLevels];
    int flv[32], stack_lv[4 * kTreeLevels];
};

// The five forms at this lane's table entry
__device__ __forceinline__ double form64(const double *c, double x, bool xi)
{
    const double2 u = *reinterpret_cast<const double2 *>(c), v = *reinterpret_cast<const double2 *>(c + 2);
    return fma(x, fma(x, v.y, xi ? u.y : v.x), xi ? u.x : 0.0);
}

template <bool NG9>
__global__ void __launch_bounds__(kTreeNT, 3) k_adj_tree64(AdjTree64Args a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AdjWarp64 &sm = reinterpret_cast<AdjWarp64 *>(smem_raw)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int top = a.levels - 1;
    const int64_t n_items = a.n * a.parts;
    // a pixel's far form takes d from the rounded direction, and a pixel on the line of sight has none: not below 1/16
    const double d_far = fmax((double)a.d_far, 0.0625), d_far2 = d_far * d_far, b_min = (double)a.b_min;
    unsigned zerocnt = 0;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(a.queue, 1ull);
        item = __shfl_sync(0xffffffffu, item, 0);
        if ((int64_t)item >= n_items) break;
        const int part = (int)((int64_t)item / a.n);
        const int64_t s = (int64_t)item - part * a.n;
        const float4 ca = a.crit[s].a, cb = a.crit[s].b;
        const Seg64 &sg = a.s64[s];
        double acc[kSums];
#pragma unroll
        for (int k = 0; k < kSums; ++k) acc[k] = 0.0;
        const double xh[3] = {sg.xh[0] + sg.xl[0], sg.xh[1] + sg.xl[1], sg.xh[2] + sg.xl[2]};
        const double e1 = 1.0 + (sg.xd[0] * xh[0] + sg.xd[1] * xh[1] + sg.xd[2] * xh[2]);   // 1 + Xdot.Xhat
        const double f1 = sg.xp[0] * xh[0] + sg.xp[1] * xh[1] + sg.xp[2] * xh[2];           // X'.Xhat

        // the sums of the collected far clusters
        auto far_flush = [&](int cnt) {
            __syncwarp();
            if (lane < cnt) {
                const TreeGeo &g = a.geo[sm.flv[lane]][sm.fcl[lane]];
                AdjFar64 &d = sm.far[lane];
                double D[3], P = 0.0, Q = 0.0, K = 0.0, B0 = 1.0;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    D[c] = (g.n0[c] - sg.xh[c]) - sg.xl[c];
                    P = fma(sg.xd[c], D[c], P);
                    Q = fma(sg.xp[c], D[c], Q);
                    K = fma(D[c], D[c], K);
                    B0 = fma(sg.xd[c], g.n0[c], B0);
                }
                auto dot = [](const double *u, const double *v) { return fma(u[2], v[2], fma(u[1], v[1], u[0] * v[0])); };
                auto put = [&](int k, double con, double x, double y, double sq) {
                    d.v[k][0] = con;
                    d.v[k][1] = x;
                    d.v[k][2] = y;
                    d.v[k][3] = sq;
                };
                put(0, 0.5 * K, 2.0 * dot(D, g.e1), 2.0 * dot(D, g.e2), 2.0 + fma(-2.0, dot(D, g.n0), 0.5 * K));
                const double p0 = dot(sg.xd, g.n0), p1 = dot(sg.xd, g.e1), p2 = dot(sg.xd, g.e2);
                put(1, 0.5 * B0, p1, p2, fma(0.5, B0, -p0));
                put(2, 0.5 * P, p1, p2, fma(0.5, P, -p0));
                const double q0 = dot(sg.xp, g.n0), q1 = dot(sg.xp, g.e1), q2 = dot(sg.xp, g.e2), A0 = f1 + Q;
                put(3, 0.5 * A0, q1, q2, fma(0.5, A0, -q0));
                put(4, 0.5 * Q, q1, q2, fma(0.5, Q, -q0));
            }
            __syncwarp();
#pragma unroll 1
            for (int i = 0; i < cnt; ++i) {
                const TreeGeo &g = a.geo[sm.flv[i]][sm.fcl[i]];
                const double *w8 = a.node[sm.flv[i]] + sm.fcl[i] * kNN64;
                const double ch = cheb_at<kNP64>(1, lane % kNP64), xi = g.a1 * ch, et = g.a2 * ch;
                double F[5], G[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    F[k] = form64(sm.far[i].v[k], xi, true);
                    G[k] = form64(sm.far[i].v[k], et, false);
                }
                const double wf = fma(0.5 * xi, xi, 0.5);
                double S2 = 0.0, S3 = 0.0, S4 = 0.0, E0 = 0.0, Ey = 0.0, Ew = 0.0, U0 = 0.0, Uy = 0.0, Uw = 0.0;
                double T0 = 0.0, Ty = 0.0, Tw = 0.0;
#pragma unroll 2
                for (int t = 0; t < kNN64 / 32; ++t) {
                    const int j = 2 * t + (lane >> 4);
                    const double gw = w8[t * 32 + lane];
                    const double eta = __shfl_sync(0xffffffffu, et, j);
                    const double Q = F[0] + __shfl_sync(0xffffffffu, G[0], j), B = F[1] + __shfl_sync(0xffffffffu, G[1], j);
                    const double Pd = F[2] + __shfl_sync(0xffffffffu, G[2], j), A = F[3] + __shfl_sync(0xffffffffu, G[3], j);
                    const double Qd = F[4] + __shfl_sync(0xffffffffu, G[4], j);
                    const double w = fma(0.5 * eta, eta, wf);
                    const double i2 = rcp64(B * Q), gi = gw * i2, iQ = B * i2;
                    const double gA = gi * A, gq = gw * iQ, gT = gi * fma(B, Pd, -(A * Qd)), ge = gT * iQ;
                    const double u = fma(gA, Qd * (Q * i2), gq);
                    S2 = fma(gq, w, S2);
                    S3 = fma(gA, w, S3);
                    S4 += gT;
                    E0 += ge;
                    Ey = fma(ge, eta, Ey);
                    Ew = fma(ge, w, Ew);
                    U0 += u;
                    Uy = fma(u, eta, Uy);
                    Uw = fma(u, w, Uw);
                    if (NG9) {
                        const double v = fma(gi, Qd, gA);
                        T0 += v;
                        Ty = fma(v, eta, Ty);
                        Tw = fma(v, w, Tw);
                    }
                }
                // w d = w D + xi e1 + eta e2 - r^2 n0 and w n = w n0 + ..., r^2 = 2 w - 1
                acc[0] += (e1 - 1.0) * S2 - f1 * S3;
                acc[1] += S2;
                acc[2] += S3;
                acc[3] += S4;
                const double Er = fma(2.0, Ew, -E0), Ur = fma(2.0, Uw, -U0) - (Uw - S2), Tr = NG9 ? fma(2.0, Tw, -T0) - (Tw - S3) : 0.0;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const double D = (g.n0[c] - sg.xh[c]) - sg.xl[c];
                    acc[4 + c] += 2.0 * fma(-g.n0[c], Er, fma(g.e2[c], Ey, fma(g.e1[c], xi * E0, D * Ew)));
                    acc[7 + c] += fma(-g.n0[c], Ur, fma(g.e2[c], Uy, fma(g.e1[c], xi * U0, D * S2)));
                    if (NG9) acc[10 + c] += fma(-g.n0[c], Tr, fma(g.e2[c], Ty, fma(g.e1[c], xi * T0, D * S3)));
                }
            }
            __syncwarp();
        };

        // the pixels of a near leaf
        auto near_leaf = [&](int64_t cl) {
            const AdjPix64 *px = a.pix + cl * kPts;
            double S2 = 0.0, S3 = 0.0, S4 = 0.0, V1[3] = {0.0, 0.0, 0.0}, V2[3] = {0.0, 0.0, 0.0};
            double V3[3] = {0.0, 0.0, 0.0};
#pragma unroll 2
            for (int t = 0; t < kPts / 32; ++t) {
                const double2 pa = px[t * 32 + lane].a, pb = px[t * 32 + lane].b;
                const double g = pb.y;
                const double dx = pa.x - xh[0], dy = pa.y - xh[1], dz = pb.x - xh[2];
                const double Q = fma(dz, dz, fma(dy, dy, dx * dx));
                const double B = fma(pb.x, sg.xd[2], fma(pa.y, sg.xd[1], fma(pa.x, sg.xd[0], 1.0)));
                const bool close = g != 0.0 && (Q < d_far2 || B < b_min);
                if (__any_sync(0xffffffffu, close)) {
                    if (g != 0.0) adj_pair64(pa.x, pa.y, pb.x, g, sg, NG9 ? 9 : 6, acc, zerocnt);
                    continue;
                }
                const double A = fma(pb.x, sg.xp[2], fma(pa.y, sg.xp[1], pa.x * sg.xp[0]));
                const double Qd = A - f1;
                const double i2 = g != 0.0 ? rcp64(B * Q) : 0.0, gi = g * i2, iQ = B * i2;
                const double gA = gi * A, gq = g * iQ, gT = gi * fma(B, B - e1, -(A * Qd)), ge = gT * iQ;
                const double t1 = Qd * (Q * i2), u = fma(gA, t1, gq);
                S2 += gq;
                S3 += gA;
                S4 += gT;
                V1[0] = fma(ge, dx, V1[0]);
                V1[1] = fma(ge, dy, V1[1]);
                V1[2] = fma(ge, dz, V1[2]);
                V2[0] = fma(u, pa.x, V2[0]);
                V2[1] = fma(u, pa.y, V2[1]);
                V2[2] = fma(u, pb.x, V2[2]);
                if (NG9) {
                    const double v = fma(gi, Qd, gA);
                    V3[0] = fma(v, pa.x, V3[0]);
                    V3[1] = fma(v, pa.y, V3[1]);
                    V3[2] = fma(v, pb.x, V3[2]);
                }
            }
            acc[0] += (e1 - 1.0) * S2 - f1 * S3;
            acc[1] += S2;
            acc[2] += S3;
            acc[3] += S4;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                acc[4 + c] += 2.0 * V1[c];
                acc[7 + c] += fma(-xh[c], S2, V2[c]);
                if (NG9) acc[10 + c] += fma(-xh[c], S3, V3[c]);
            }
        };

        if (cb.w < kCritSkip) {
            int nfar = 0;
            for (int64_t root = part; root < a.ncl[top]; root += a.parts) {
                int sp = 1;
                __syncwarp();
                if (lane == 0) {
                    sm.stack_lv[0] = top;
                    sm.stack_cl[0] = root;
                }
                while (sp > 0) {
                    __syncwarp();
                    --sp;
                    const int L = sm.stack_lv[sp];
                    const int64_t cl = sm.stack_cl[sp];
                    const float4 self = a.geo[L][cl].c;
                    if (tree_empty(self)) continue;
                    if (!tree_near_pos(ca, self) && !tree_near_beam(cb, self)) {
                        if (lane == 0) {
                            sm.flv[nfar] = L;
                            sm.fcl[nfar] = cl;
                        }
                        if (++nfar == 32) {
                            far_flush(32);
                            nfar = 0;
                        }
                    } else if (L == 0) {
                        near_leaf(cl);
                    } else {
                        int64_t kid = 0;
                        bool has = false;
                        if (lane < 4) {
                            if (a.nb[L] == 0) {
                                kid = 4 * cl + lane;
                                has = kid < a.ncl[L - 1];
                            } else {
                                const int64_t nb = a.nb[L], cnb = a.nb[L - 1], f = cl / (nb * nb), rem = cl - f * nb * nb;
                                const int64_t i = 2 * (rem % nb) + (lane & 1), j = 2 * (rem / nb) + (lane >> 1);
                                has = i < cnb && j < cnb;
                                kid = (f * cnb + j) * cnb + i;
                            }
                        }
                        const unsigned m = __ballot_sync(0xffffffffu, has);
                        if (has) {
                            const int at = sp + __popc(m & ((1u << lane) - 1u));
                            sm.stack_lv[at] = L - 1;
                            sm.stack_cl[at] = kid;
                        }
                        sp += __popc(m);
                    }
                }
            }
            if (nfar > 0) far_flush(nfar);
        }
        double out = 0.0;
#pragma unroll
        for (int k = 0; k < adj_rows(NG9); ++k) {
            double v = acc[k];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == k) out = v;
        }
        if (lane < adj_rows(NG9)) a.partial[((int64_t)part * adj_rows(NG9) + lane) * a.n + s] = out;
    }
    for (int o = 16; o > 0; o >>= 1) zerocnt += __shfl_xor_sync(0xffffffffu, zerocnt, o);
    if (lane == 0 && zerocnt) atomicAdd(&a.st->zero_pairs, (unsigned long long)zerocnt);
}

// One thread per record: its parts in order, then the gradient rows at the sample's place in the input.
__global__ void __launch_bounds__(128) k_adj_finish64(const double *__restrict__ partial, int64_t n, int parts,
                                                      const uint32_t *__restrict__ perm, const Seg64 *__restrict__ s64, int ngrad,
                                                      double *__restrict__ grad, int64_t ld)
{
    const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n) return;
    double acc[kSums];
    const int nk = adj_rows(ngrad >= 9);
#pragma unroll
    for (int k = 0; k < kSums; ++k) {
        double hi = 0.0, lo = 0.0;
        if (k < nk)
            for (int c = 0; c < parts; ++c) fold64(hi, lo, partial[((int64_t)c * nk + k) * n + s]);
        acc[k] = hi + lo;
    }
    double out[10];
    adj_assemble(s64[s], acc, ngrad, out);
    const int64_t dst = perm[s];
    for (int k = 0; k < ngrad; ++k) grad[k * ld + dst] = out[k];
}

}  // namespace

AdjTreePlan adj_tree_plan64(int64_t N, int nface, int64_t npix, int64_t n, int ngrad, int num_sms)
{
    AdjTreePlan p{};
    p.map = tree_plan(ISW_F64, N, nface, npix, n, num_sms);
    p.n_pad = (n + kTreeNT - 1) / kTreeNT * kTreeNT;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += up256(bytes);
        return o;
    };
    const size_t smem = kWarps * sizeof(AdjWarp64);
    const int s0 = slots_of((const void *)&k_adj_tree64<false>, smem, num_sms), s1 = slots_of((const void *)&k_adj_tree64<true>, smem, num_sms);
    p.slots = s0 < s1 ? s0 : s1;
    // enough warps of work to level the end: eight for each that is resident
    const int64_t want = (int64_t)p.slots * kWarps * 8;
    p.parts = (int)(n < want ? (want + n - 1) / (n > 0 ? n : 1) : 1);
    if (p.parts > kAdjMaxParts) p.parts = kAdjMaxParts;
    p.off_queue = take(sizeof(unsigned long long));
    p.off_crit = take((size_t)p.n_pad * sizeof(TreeCrit));
    p.off_caps = take((size_t)(p.n_pad / kTreeS) * sizeof(TreeCap));
    p.off_inv = take((size_t)p.n_pad * sizeof(uint32_t));
    for (int L = 0; L < p.map.levels; ++L) {
        p.off_geo[L] = take((size_t)p.map.ncl[L] * sizeof(TreeGeo));
        p.off_node[L] = take((size_t)p.map.ncl[L] * kNN64 * sizeof(double));
    }
    p.off_pix = take((size_t)p.map.ncl[0] * kPts * sizeof(AdjPix64));
    p.off_partial = take((size_t)p.parts * adj_rows(ngrad >= 9) * n * sizeof(double));
    p.bytes = at;
    return p;
}

cudaError_t launch_adjoint_tree64(const AdjTreePlan &p, const AdjTreeCall &m, cudaStream_t s)
{
    unsigned char *b = (unsigned char *)m.scratch;
    unsigned long long *queue = (unsigned long long *)(b + p.off_queue);
    cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    TreeCrit *crit = (TreeCrit *)(b + p.off_crit);
    const int64_t nst = p.n_pad / kTreeS;
    k_tree_crit<<<(unsigned)((nst * 32 + 255) / 256), 256, 0, s>>>(m.s32, m.s64, m.perm, m.n, nst, crit, (TreeCap *)(b + p.off_caps),
                                                                   nullptr, (uint32_t *)(b + p.off_inv));
    const TreePlan &t = p.map;
    AdjTree64Args a{};
    for (int L = 0; L < t.levels; ++L) {
        TreeGeo *geo = (TreeGeo *)(b + p.off_geo[L]);
        double *node = (double *)(b + p.off_node[L]);
        AdjUp64Args u{};
        u.geo = geo;
        u.ncl = t.ncl[L];
        u.nb = t.nb[L];
        u.node = node;
        if (L == 0) {
            launch_leaf_geo<kLeaf64>(m.nv, m.ldn, m.outidx, m.order, m.theta_pix, kKappa64, t.ncl[0], geo, s);
            u.nv = m.nv;
            u.ldn = m.ldn;
            u.outidx = m.outidx;
            u.g = m.g;
            u.blocks = m.order == kSlotsDiag;
            u.pix = (AdjPix64 *)(b + p.off_pix);
            k_adj_up64<true><<<(unsigned)t.ncl[0], kNN64, 0, s>>>(u);
        } else {
            launch_up_geo(a.geo[L - 1], t.nb[L - 1], t.ncl[L - 1], geo, t.nb[L], t.ncl[L], kKappa64, s);
            u.cgeo = a.geo[L - 1];
            u.cnb = t.nb[L - 1];
            u.cncl = t.ncl[L - 1];
            u.child = a.node[L - 1];
            k_adj_up64<false><<<(unsigned)t.ncl[L], kNN64, 0, s>>>(u);
        }
        a.geo[L] = geo;
        a.node[L] = node;
        a.nb[L] = t.nb[L];
        a.ncl[L] = t.ncl[L];
    }
    a.crit = crit;
    a.s64 = m.s64;
    a.levels = t.levels;
    a.parts = p.parts;
    a.pix = (const AdjPix64 *)(b + p.off_pix);
    a.n = m.n;
    a.partial = (double *)(b + p.off_partial);
    a.b_min = m.b_min;
    a.d_far = m.d_far;
    a.st = m.st;
    a.queue = queue;
    const int64_t items = (m.n * p.parts + kWarps - 1) / kWarps;
    const void *fn = m.ngrad >= 9 ? (const void *)&k_adj_tree64<true> : (const void *)&k_adj_tree64<false>;
    void *args[] = {(void *)&a};
    cudaLaunchKernel(fn, dim3((unsigned)(items < p.slots ? items : p.slots)), dim3(kTreeNT), args, kWarps * sizeof(AdjWarp64), s);
    k_adj_finish64<<<(unsigned)((m.n + 127) / 128), 128, 0, s>>>(a.partial, m.n, p.parts, m.perm, m.s64, m.ngrad, m.grad, m.ld_g);
    return cudaSuccess;
}

}  // namespace isw
