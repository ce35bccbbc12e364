// Launchers of the library's kernels (one translation unit each), called by the C ABI layer.
#pragma once

#include "isw_internal.cuh"

namespace isw {

// api.cu: number of work chunks along the streamed axis for ntiles tiles of the other axis, nst
// streamed tiles and `slots` resident CTAs (near-equal waves; at least two streamed tiles per
// chunk; at most max_split chunks)
int choose_split(int64_t ntiles, int64_t nst, int slots, int max_split, int min_items = 0, int min_chunk = 256);
constexpr int kMapItemsPerSlot = 64;   // work items per CTA slot that the map's chunk count aims at
constexpr int kAdjItemsPerSlot = 64;   // the same for the adjoint's pixel chunks,
constexpr int kAdjMinChunk = 32;       // each chunk keeping at least this many pixel tiles

// probe.cu: FMA-pipe throughput (flop/s, FMA = 2) of the FP32 or FP64 pipe; sink is never written
int fma_probe(bool f64, int num_sms, double *sink, double *flops, cudaStream_t s);

// healpix.cu
int launch_pix2vec(int64_t N, int64_t pix0, int64_t npix, const int64_t *pix_list, double *out, int64_t ld,
                   DevStatus *st, cudaStream_t s);
void launch_pixel_table(int64_t N, int mode, int64_t pix0, int64_t npix, const int64_t *pix_list, int tx, int ty,
                        int64_t ntiles, double *nv, int64_t ldn, int64_t *outidx, float4 *caps, DevStatus *st,
                        cudaStream_t s, const uint32_t *perm = nullptr);

// A gnomonic patch: orthonormal frame (e1, e2, e3) with e3 the centre, M x M pixels of
// coordinate pitch width / M; pixel (i, j) at (xi, eta) = ((i + 1/2 - M/2), (j + 1/2 - M/2)) * pitch,
// direction (xi e1 + eta e2 + e3) / norm, output slot j M + i.
struct PatchSpec {
    double frame[9];
    int64_t M;
    double width;
};
// patch pixel table: compact tx x ty blocks of the M x M grid (caps as for the sphere)
void launch_patch_table(const PatchSpec &p, int tx, int ty, int64_t ntiles, double *nv, int64_t ldn,
                        int64_t *outidx, float4 *caps, cudaStream_t s);

// flat.cu: flat-sky patch map (pixel tiles 32 x flat_ty() of the patch table)
int flat_seg_tile();
int flat_tx();
int flat_ty();
size_t flat_record_bytes();   // FP32 + FP64 record bytes per sample
int flat_slots(bool f64, int num_sms);
void launch_flat_pack(const double *S, int64_t n, int64_t ld, const PatchSpec &p, double xo0, double xo1, double xo2,
                      double GU, int64_t n_pad, void *r32, void *r64, cudaStream_t s);
void launch_map_flat(bool f64, const void *r32, const void *r64, const int64_t *outidx, int64_t ntiles, int64_t nst,
                     int split, int64_t M, double pitch, double *theta, double *partial, int accumulate,
                     DevStatus *st, unsigned long long *queue, uint32_t wait_polls, int grid, cudaStream_t s);

// cl.cu: angular power spectrum (scratch: cl_scratch_bytes; alm: double[2][lmax+1][lmax+1])
int cl_max_nside();
size_t cl_scratch_bytes(int64_t N, int64_t lmax);
void launch_map_cl(int64_t N, const double *map, int64_t lmax, void *scratch, double *alm, double *cl, cudaStream_t s);

// lightcone.cu
void launch_lightcone(int mode, const double *nodes, int64_t n, int64_t ld, const double *P, int64_t nloops,
                      int64_t ldp, double t_box, double xo0, double xo1, double xo2, double t_obs, double tol,
                      int max_iter, double *out, int64_t ld_out, double *tau, int32_t *status, DevStatus *st,
                      cudaStream_t s);
// one launch over many shells: per-node shell lookup through shell_off (device copies)
void launch_lightcone_shells(const double *nodes, int64_t n, int64_t ld, const int64_t *shell_off, int64_t nshell,
                             const double *t_box, const int32_t *mode, const double *P, int64_t nloops, int64_t ldp,
                             double xo0, double xo1, double xo2, double t_obs, double tol, double *out,
                             int64_t ld_out, DevStatus *st, cudaStream_t s);

// lcadj.cu: adjoint of the light-cone solve.  runs (int[nloops], zeroed by the caller), first,
// last (int64[nloops]) are workspace of the Burden per-loop reduction; gl may be NULL in LINEAR mode.
void launch_lightcone_adjoint(int mode, const double *nodes, int64_t n, int64_t ld, const double *P, int64_t nloops,
                              int64_t ldp, double t_box, double xo0, double xo1, double xo2, const double *tau,
                              const double *gs, int64_t ldgs, int ngs, double *gn, int64_t ldgn, double *gl,
                              int64_t ldgl, int *runs, int64_t *first, int64_t *last, double *contrib, DevStatus *st,
                              cudaStream_t s);   // contrib: 15 n doubles (Burden mode) or NULL

// cone.cu: stacking with HEALPix cones
void launch_vec2pix(int64_t N, const double *v, int64_t n, int64_t ld, int64_t *pix, DevStatus *st, cudaStream_t s);
void launch_box_place(const double *nodes, int64_t ld, const int64_t *off_out, const int64_t *src_start,
                      int64_t nshell, const double *place, double *out, int64_t ld_out, int64_t n_out,
                      cudaStream_t s);
// scratch: incl int32[n], block_tot int64[cone_cut_scratch_blocks(n) + 1]
int64_t cone_cut_scratch_blocks(int64_t n);
void launch_cone_cut(const double *S, int64_t ld, int64_t n, const int64_t *off, int64_t nshell, int64_t nside_hz,
                     const int64_t *cone_pix, const double *r_lo, const double *r_hi, double xo0, double xo1,
                     double xo2, int32_t *incl, int64_t *block_tot, double *out, int64_t ld_out, int64_t *off_out,
                     int64_t *count, cudaStream_t s);

// sort.cu: spatial order of the samples (stable radix sort of the Morton code of Xhat); returns the
// device array perm[n] (record s holds sample perm[s]), inside scratch of sort_scratch_bytes(n, orders).
// With orders = 2 perm[n + k] is the k-th sample in the Morton order of Xdot.
size_t sort_scratch_bytes(int64_t n, int orders);
const uint32_t *launch_spatial_order(const double *S, int64_t n, int64_t ld, double xo0, double xo1, double xo2,
                                     void *scratch, int orders, cudaStream_t s);
int spatial_order_launches();
// stable sort of 24-bit keys already in the scratch: keys [orders][n], indices [orders][n] after twice as
// many words
const uint32_t *launch_sort_keys(int64_t n, int orders, void *scratch, cudaStream_t s);
// the same for the selected pixels (a range, or a list when pix_list is given): perm[npix] of positions
const uint32_t *launch_pixel_order(int64_t N, int64_t pix0, int64_t npix, const int64_t *pix_list, void *scratch,
                                   cudaStream_t s);

// pack.cu: per-sample records of the map kernels and per-tile caps
// perm (may be NULL): record s is built from sample perm[s] (else from sample s)
// far (may be NULL): far-field records for the FP32 pair kernel, pair-interleaved (n_pad even)
// mid (may be NULL): mid-range records for the FP32 near-field pass
// far64 (may be NULL): far-field records for the FP64 kernel
void launch_pack(const double *samples, int64_t n, int64_t ld, double xo0, double xo1, double xo2, double GU,
                 double theta_pix, double near_k, int64_t n_pad, const uint32_t *perm, Seg32 *s32, Seg64 *s64,
                 Far2 *far, Mid2 *mid, Far64 *far64, DevStatus *st, cudaStream_t s);
void launch_seg_caps(const Seg32 *s32, const Seg64 *s64, int64_t n, int64_t n_pad, int seg_tile, float b_min,
                     SegCap *caps, cudaStream_t s);

// map.cu
struct MapArgs {
    const double *nv;        // pixel table directions [3][ldn]
    int64_t ldn;
    const int64_t *outidx;   // pixel table output indices
    const float4 *pcaps;     // pixel tile caps
    int64_t ntiles;          // pixel tiles
    const Seg32 *s32;
    const Seg64 *s64;
    const Far2 *far;         // far-field records of sample pairs (FP32 kernels)
    const Mid2 *mid;         // mid-range records of samples (FP32 near-field pass)
    const Far64 *far64;      // far-field records of samples (FP64 kernel)
    const SegCap *scaps;
    int64_t nst;             // segment tiles
    int split;               // segment chunks
    float b_min;
    float d_far;             // tile pairs at least this chord apart use the far-field form
    double *theta;           // output (RING or list order)
    double *partial;         // [split][ntiles*tile] when split > 1
    int accumulate;
    DevStatus *st;
    int64_t tile_stride;     // 1; > 1 only when timing variants: every tile_stride-th pixel tile
    unsigned long long *queue;   // work counters (far pass or FP64 kernel, near pass), zero at launch
    uint32_t wait_polls;     // limit of the consumer waits (kWaitPolls by default)
};
struct Variant {
    int threads, ppt, seg_tile, tx, ty;
};
int num_f32_variants();
Variant f32_variant(int idx);
int f64_seg_tile();
Variant f64_variant();
// slots = resident CTAs on the whole GPU for the variant
int map_f32c_slots(int idx, int num_sms);
int map_f64_slots(int num_sms);
void launch_map_f32c(int idx, const MapArgs &a, int grid, cudaStream_t s);
void launch_map_f32c_near(int idx, const MapArgs &a, int num_sms, cudaStream_t s);
void launch_map_f64(const MapArgs &a, int grid, cudaStream_t s);
void launch_reduce_partials(const MapArgs &a, int tile_sz, cudaStream_t s);

// tree.cu: the map over a cluster tree of the pixels
constexpr int kTreeLevels = 20;
// Whether a call of default settings runs over the tree, by pairs (both sides timed from N_side 4 to 90, samples of
// strings and scattered ones; direct / tree in ms):
//   FP32 full sky  1e6: N_side 16 with 500 0.69 / 0.29 and 0.29 / 0.21, N_side 64 with 500 0.78 / 0.38 and
//                  0.21 / 0.22.  The direct kernel sums a string's near pairs lane by lane in FP64.
//   FP32 patch     5e7: 128 x 128 with 5,000 0.91 / 0.36 with a string in it, 0.21 / 0.25 with none near
//   FP32 list      3e8: where the pixels lie is not known here.  A compact list of 5,000 with 60,000 samples 1.55 / 0.68,
//                  pixels scattered over the sky 0.67 / 0.81; 20,000 with 15,000 1.23 / 0.53 and 0.57 / 0.63; from 50,000
//                  scattered pixels on 1.1 to 2.2 times as fast.
//   FP32 adjoint   8e8 (the latency of the deepest subtrees bounds small calls; 120 sky calls of loops at 6e8 to 8e8 were
//                  0.8 to 1.5 times as fast, at 8e8 to 1e9 0.98 to 1.7, at 3e8 from 0.57 on); lists 2e9: 12,288
//                  scattered pixels 4.97 / 4.64 and 4.96 / 5.16, 50,000 4.91 / 3.67, compact ones 4.48 / 2.54.
//   FP64 map       9e7: sky calls of loops at 6e7 to 8e7 0.80 to 1.7 times as fast, from 9e7 on 1.01 and more; lists 0.76 to 1.9 at 6e7,
//                  from 1.2e8 on 1.2 and more.  The leaves have 32 x 32 pixels, so at least four faces of half that.
//   FP64 patch     6e7: 64 x 64 with 14,649 3.57 / 1.52 to 3.56 / 3.60 by width (0.05 to 0.5) and sample layout.
//   FP64 adjoint   6e6, N_side 32: N_side 32 with 500 1.3 / 0.83; lists of 12,288 with 489 1.14 / 0.91.  Between N_side 32 and 45
//                  a face's four leaves are less than half full: N_side 33 and 36 with 15,360 33 / 42, 40 37 / 42, 44 40 / 41, 45 44 / 41.
// The list entries hold 30-bit record numbers.
enum TreeUse : int { kTreeSky = 0, kTreePatch = 1, kTreePixelList = 2, kTreeAdjointSky = 3, kTreeAdjointList = 4 };
inline bool tree_rule(int prec, TreeUse use, int64_t npix, int64_t n)
{
    const bool f64 = prec == ISW_F64, adj = use == kTreeAdjointSky || use == kTreeAdjointList;
    const int64_t pix = adj ? 12 * 1024 : f64 ? 4096 : 192;
    double pairs;
    if (adj) pairs = f64 ? 6e6 : use == kTreeAdjointSky ? 8e8 : 2e9;
    else if (f64) pairs = use == kTreePatch ? 6e7 : 9e7;
    else pairs = use == kTreeSky ? 1e6 : use == kTreePatch ? 5e7 : 3e8;
    const bool sparse = f64 && use == kTreeAdjointSky && npix > 12 * 32 * 32 && npix < 12 * 45 * 45;   // leaves
    return npix >= pix && (double)npix * (double)n >= pairs && n < (int64_t(1) << 30) && !sparse;
}
// slot order of the pixel tables: anti-diagonals (full sky), rows (patch), spatially sorted list
enum : int { kSlotsDiag = 0, kSlotsRows = 1, kSlotsList = 2 };
struct TreePlan {
    int prec;
    int leaf, nn, levels;                 // leaf side in pixels, doubles per cluster's node sums
    int nb[kTreeLevels];                  // clusters per face side, from the finest level (0: a list)
    int64_t ncl[kTreeLevels];             // clusters of the level
    int64_t n_pad, nst;                   // padded samples, sample tiles
    int nslots, pslots;                   // resident CTAs of the node and pixel kernels
    int pool, ppool;                      // chunk pool entries of a level and of the pixels
    size_t off_queue, off_crit, off_vcrit, off_caps, off_sup, off_vidx, off_inv, off_rec, off_work, off_pool, off_partial;
    size_t off_geo[kTreeLevels], off_F[kTreeLevels], bytes;   // scratch layout
};
struct TreeMapArgs {
    const double *nv;         // pixel table: leaf x leaf slots per finest cluster, clusters in (face, y, x) order
    int64_t ldn;
    const int64_t *outidx;
    int order;                // slots of a cluster
    int64_t nside;            // N_side of a full-sky map, else 0
    double theta_pix;
    const Seg32 *s32;
    const Seg64 *s64;
    const Far64 *far64;       // FP64 maps
    const uint32_t *perm;     // sample of each record, and of each velocity-order entry (perm + n)
    int64_t n;
    float b_min, d_far;
    double *theta;
    int accumulate;
    DevStatus *st;
    void *scratch;            // TreePlan::bytes
};
int tree_leaf(int prec);
// nface faces of N x N pixels, or (nface = 0) a list of npix
TreePlan tree_plan(int prec, int64_t N, int nface, int64_t npix, int64_t n, int num_sms);
cudaError_t launch_map_tree(const TreePlan &p, const TreeMapArgs &m, cudaStream_t s);
inline int tree_launches(const TreePlan &p) { return 2 * p.levels + 7; }

// flattree.cu: flat-sky patch maps over a tree of pixel clusters
struct FlatTreePlan {
    bool f64;
    int leaf, levels, nb[kTreeLevels];    // leaf side in pixels, clusters per side from the leaves
    int64_t n_pad, nst;
    int nslots, pslots, pool, ppool;
    size_t off_queue, off_crit, off_caps, off_sup, off_rec, off_sort, off_work, off_pool, off_partial, off_A[kTreeLevels], bytes;
};
// Whether a flat-sky patch runs over the tree (2,600 drawn patches of 32 to 1,176 pixels a side, 100 to 182,000 samples):
//   FP32  9e8 pairs, where the direct kernel's 3e11 to 4e11 pairs a second meet the 0.35 to 2 ms that the tree's 20
//         launches and its near samples take: at 9e8 to 1e9 0.9 to 1.5 times as fast, at 2e9 1.6 to 2.9 times;
//         at 1e8 0.3 to 0.8 times
//   FP64  3e7 from 192 pixels a side (1.4 to 4 times as fast), 5e7 below (median 1.6 to 4.5, down to 0.4 where the
//         whole patch lies on a string)
// Patches whose squared distances leave the range of float go to the direct kernels (d >= pitch of a far sample, d < 1e18).
inline bool flat_tree_rule(bool f64, int64_t M, int64_t n, double width)
{
    const double pairs = (double)M * (double)M * (double)n;
    return M >= 32 && pairs >= (!f64 ? 9e8 : M >= 192 ? 3e7 : 5e7) && n < (int64_t(1) << 30) && width >= 1e-15 * (double)M &&
           width <= 1e15;
}
FlatTreePlan flat_tree_plan(bool f64, int64_t M, int64_t n, int num_sms);
cudaError_t launch_map_flat_tree(const FlatTreePlan &p, const void *r32, const void *r64, int64_t n, int64_t M, double width,
                                 double *theta, int accumulate, void *scratch, cudaStream_t s);
inline int flat_tree_launches(const FlatTreePlan &p) { return p.levels + 16; }

// treeadj.cu: FP32 adjoint over the cluster tree
struct AdjTreePlan {
    TreePlan map;                         // levels and clusters
    int64_t n_pad;
    int slots, parts;                     // resident CTAs; shares of the root clusters
    size_t off_queue, off_crit, off_vcrit, off_caps, off_vidx, off_inv, off_rec, off_pix, off_low, off_partial, bytes;
    size_t off_geo[kTreeLevels], off_node[kTreeLevels];
};
struct AdjTreeCall {
    const double *nv;                     // pixel table as in TreeMapArgs
    int64_t ldn;
    const int64_t *outidx;
    int order;
    double theta_pix;
    const double *g;                      // dL/dTheta by output index
    const Seg32 *s32;                     // n_pad records
    const Seg64 *s64;
    const uint32_t *perm;
    int64_t n;
    float b_min, d_far;
    int ngrad;
    double *grad;
    int64_t ld_g;
    DevStatus *st;
    void *scratch;
};
AdjTreePlan adj_tree_plan64(int64_t N, int nface, int64_t npix, int64_t n, int ngrad, int num_sms);
cudaError_t launch_adjoint_tree64(const AdjTreePlan &p, const AdjTreeCall &m, cudaStream_t s);
AdjTreePlan adj_tree_plan(int64_t N, int nface, int64_t npix, int64_t n, int ngrad, int num_sms);
cudaError_t launch_adjoint_tree(const AdjTreePlan &p, const AdjTreeCall &m, cudaStream_t s);
inline int adj_tree_launches(const AdjTreePlan &p) { return 2 * p.map.levels + (p.map.prec == ISW_F64 ? 3 : 5); }

// adjoint.cu
struct AdjArgs {
    const Pix32 *p32;        // pixel records in tile order
    const Pix64 *p64;
    const PixF2 *pf2;        // far-field records of pixel pairs (FP32 kernel)
    const float4 *pcaps;     // pixel tile caps
    int64_t npix_tiles;
    const Seg32 *s32;
    const Seg64 *s64;
    const SegCap *scaps;     // caps of the adjoint's sample tiles
    int64_t nseg_tiles;
    int64_t n, n_pad;
    int split;               // pixel chunks
    int ngrad;               // 6 or 9
    float b_min, d_far;
    double *grad;            // [ngrad][ld_g]
    int64_t ld_g;
    double *partial;         // [split][ngrad][n_pad] when split > 1
    DevStatus *st;
    unsigned long long *queue;   // work counter, zero at launch
    uint32_t wait_polls;     // limit of the consumer waits (kWaitPolls by default)
};
int adj_seg_tile(int prec);
int adj_pix_tile(int prec);
int adj_slots(int prec, int ngrad, int num_sms);
void launch_pack_pixels(const double *nv, int64_t ldn, const int64_t *outidx, const double *g, int64_t tot,
                        Pix32 *p32, Pix64 *p64, PixF2 *pf2, cudaStream_t s);
void launch_adjoint(int prec, const AdjArgs &a, int grid, cudaStream_t s);

}  // namespace isw
