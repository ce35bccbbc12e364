// Spatial order of the samples for the FP32 map.  The sum of Eq. (1)-(2) does not depend on the
// order of the samples, but the tiling does: a segment tile of consecutive samples gets a
// bounding cap, and only tile pairs whose caps are far apart take the far-field form.  Samples
// that are adjacent in the input need not be adjacent on the sky (a string whose nodes are moved
// to the light cone with velocities of random direction scatters), so the records are written in
// the order of a 3-D Morton code of the unit vector Xhat quantised to 8 bits per axis.  The sort
// is a stable least-significant-digit radix sort of (key, index) in three passes of 8 bits, so
// the order, and with it the rounding of the map's sums, is reproducible.
// The cluster-tree maps need a second order of the same samples, by the Morton code of Xdot (tree.cuh);
// both are sorted by the same launches (blockIdx.y).
//   k_sort_keys     keys (invalid samples last), index = input position
//   k_sort_hist     per block of 1024 elements, the 256-bin histogram of the pass's digit
//   k_sort_scan     one block per digit: exclusive scan of the digit's counts over the blocks, and the
//                   digit's total (one block for all digits took 42 us a pass at 2e5 samples, now 3)
//   k_sort_scatter  the block's elements in input order, ranked within their digit by a warp
//                   match and per-warp counts, written to their positions (stable)
#include "isw_internal.cuh"
#include "kernels.cuh"

namespace isw {

namespace {
constexpr int kSortThreads = 256, kSortBlock = 1024, kRadix = 256, kSortWarps = kSortThreads / 32;
constexpr uint32_t kInvalidKey = 0xffffffu;

__device__ __forceinline__ uint32_t spread3(uint32_t x)   // bits b0..b7 -> positions 0, 3, 6, ...
{
    x &= 0xffu;
    x = (x | (x << 8)) & 0x00f00fu;
    x = (x | (x << 4)) & 0x0c30c3u;
    x = (x | (x << 2)) & 0x249249u;
    return x;
}

__device__ __forceinline__ uint32_t morton(double x, double y, double z)   // of a point in [-1, 1]^3
{
    const double r[3] = {x, y, z};
    uint32_t q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double u = floor((r[c] + 1.0) * 128.0);
        q[c] = (uint32_t)(u < 0.0 ? 0.0 : (u > 255.0 ? 255.0 : u));
    }
    return spread3(q[0]) | (spread3(q[1]) << 1) | (spread3(q[2]) << 2);
}

__global__ void k_sort_keys(const double *__restrict__ S, int64_t n, int64_t ld, double xo0, double xo1, double xo2,
                            uint32_t *__restrict__ key, uint32_t *__restrict__ idx)
{
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        uint32_t k = kInvalidKey;
        if (blockIdx.y == 0) {
            const double r[3] = {S[s] - xo0, S[ld + s] - xo1, S[2 * ld + s] - xo2};
            const double nrm = sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
            if (nrm > 0.0 && isfinite(nrm)) k = morton(r[0] / nrm, r[1] / nrm, r[2] / nrm);
        } else {
            const double v[3] = {S[3 * ld + s], S[4 * ld + s], S[5 * ld + s]};
            if (isfinite(v[0] + v[1] + v[2])) k = morton(v[0], v[1], v[2]);
        }
        key[blockIdx.y * n + s] = k;
        idx[blockIdx.y * n + s] = (uint32_t)s;
    }
}

__global__ void __launch_bounds__(kSortThreads) k_sort_hist(const uint32_t *__restrict__ key, int64_t n, int shift,
                                                            uint32_t *__restrict__ hist, int nblocks)
{
    __shared__ uint32_t h[kRadix];
    const int tid = threadIdx.x;
    const int64_t b = blockIdx.x;
    key += blockIdx.y * n;
    h[tid] = 0;
    __syncthreads();
    for (int i = tid; i < kSortBlock; i += kSortThreads) {
        const int64_t e = b * kSortBlock + i;
        if (e < n) atomicAdd(&h[(key[e] >> shift) & (kRadix - 1)], 1u);
    }
    __syncthreads();
    hist[((int64_t)blockIdx.y * kRadix + tid) * nblocks + b] = h[tid];
}

// Inclusive scan over the block's kSortThreads values; wtot is shared scratch of kSortWarps words.
__device__ __forceinline__ uint32_t block_scan(uint32_t x, uint32_t *wtot)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wtot[w] = x;
    __syncthreads();
    for (int i = 0; i < w; ++i) x += wtot[i];
    __syncthreads();
    return x;
}

// Row blockIdx.x (one digit) of array blockIdx.y: exclusive scan in place, total to tot.
__global__ void __launch_bounds__(kSortThreads) k_sort_scan(uint32_t *__restrict__ hist, int nblocks,
                                                            uint32_t *__restrict__ tot)
{
    __shared__ uint32_t wtot[kSortWarps];
    __shared__ uint32_t last;
    const int tid = threadIdx.x;
    uint32_t *row = hist + ((int64_t)blockIdx.y * kRadix + blockIdx.x) * nblocks;
    uint32_t carry = 0;
    for (int b0 = 0; b0 < nblocks; b0 += kSortThreads) {
        const int b = b0 + tid;
        const uint32_t v = b < nblocks ? row[b] : 0u;
        const uint32_t x = block_scan(v, wtot);
        if (b < nblocks) row[b] = carry + x - v;
        if (tid == kSortThreads - 1) last = x;
        __syncthreads();
        carry += last;
        __syncthreads();
    }
    if (tid == 0) tot[blockIdx.y * kRadix + blockIdx.x] = carry;
}

__global__ void __launch_bounds__(kSortThreads) k_sort_scatter(const uint32_t *__restrict__ key_in,
                                                               const uint32_t *__restrict__ idx_in, int64_t n,
                                                               int shift, const uint32_t *__restrict__ offs,
                                                               const uint32_t *__restrict__ tot, int nblocks,
                                                               uint32_t *__restrict__ key_out,
                                                               uint32_t *__restrict__ idx_out)
{
    __shared__ uint32_t wtot[kSortWarps];
    __shared__ uint32_t base[kRadix];                // next output position of each digit
    __shared__ uint32_t wcnt[kSortWarps][kRadix];    // elements of each digit per warp, this round
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t b = blockIdx.x;
    key_in += blockIdx.y * n;
    idx_in += blockIdx.y * n;
    key_out += blockIdx.y * n;
    idx_out += blockIdx.y * n;
    const uint32_t all = tot[blockIdx.y * kRadix + tid];
    base[tid] = block_scan(all, wtot) - all + offs[((int64_t)blockIdx.y * kRadix + tid) * nblocks + b];
    for (int r = 0; r < kSortBlock / kSortThreads; ++r) {
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) wcnt[w][tid] = 0u;
        __syncthreads();
        const int64_t e = b * kSortBlock + (int64_t)r * kSortThreads + tid;
        const bool valid = e < n;
        const uint32_t k = valid ? key_in[e] : 0u;
        const uint32_t d = valid ? (k >> shift) & (kRadix - 1) : (uint32_t)kRadix;   // sentinel never written
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const unsigned below = peers & ((1u << lane) - 1u);
        if (valid && below == 0u) wcnt[wid][d] = (uint32_t)__popc(peers);
        __syncthreads();
        if (valid) {
            uint32_t pos = base[d] + (uint32_t)__popc(below);
            for (int w = 0; w < wid; ++w) pos += wcnt[w][d];
            key_out[pos] = k;
            idx_out[pos] = idx_in[e];
        }
        __syncthreads();
        uint32_t add = 0u;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) add += wcnt[w][tid];
        base[tid] += add;
        __syncthreads();
    }
}
// Keys of pixels: the Morton code of the centre, from float coordinates (they only order the pixels).
__global__ void k_pixel_keys(int64_t N, int64_t pix0, int64_t npix, const int64_t *__restrict__ pix_list,
                             uint32_t *__restrict__ key, uint32_t *__restrict__ idx)
{
    const int64_t all = 12 * N * N, cap = 2 * N * (N - 1);
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < npix; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = pix_list ? pix_list[k] : pix0 + k;
        uint32_t v = kInvalidKey;
        if (p >= 0 && p < all) {
            float z, phi;
            if (p >= cap && p < all - cap) {
                const int64_t q = p - cap;
                z = (float)((4.0 * (double)N - 2.0 * (double)(q / (4 * N) + N)) / (3.0 * (double)N));
                phi = (float)(q % (4 * N)) / (float)(4 * N);
            } else {
                const int64_t q = p < cap ? p : all - 1 - p, i = (1 + isqrt64(1 + 2 * q)) / 2;
                const float t = (float)i / (float)N;
                z = 1.f - t * t / 3.f;
                phi = ((float)(q - 2 * i * (i - 1)) + 0.5f) / (float)(4 * i);
                if (p >= cap) {
                    z = -z;
                    phi = 1.f - phi;
                }
            }
            const float st = sqrtf(fmaxf(1.f - z * z, 0.f));
            float s, c;
            sincospif(2.f * phi, &s, &c);
            v = morton(st * c, st * s, z);
        }
        key[k] = v;
        idx[k] = (uint32_t)k;
    }
}

// Sorts the key arrays in the scratch (orders of n each); returns the sorted indices.
const uint32_t *sort_passes(int64_t n, int orders, uint32_t *p, cudaStream_t s)
{
    const int64_t nblocks = (n + kSortBlock - 1) / kSortBlock, m = orders * n;
    uint32_t *key[2] = {p, p + m}, *idx[2] = {p + 2 * m, p + 3 * m};
    uint32_t *hist = p + 4 * m, *tot = hist + (int64_t)orders * kRadix * nblocks;
    int cur = 0;
    const dim3 grid((unsigned)nblocks, orders);
    for (int shift = 0; shift < 24; shift += 8) {
        k_sort_hist<<<grid, kSortThreads, 0, s>>>(key[cur], n, shift, hist, (int)nblocks);
        k_sort_scan<<<dim3(kRadix, orders), kSortThreads, 0, s>>>(hist, (int)nblocks, tot);
        k_sort_scatter<<<grid, kSortThreads, 0, s>>>(key[cur], idx[cur], n, shift, hist, tot, (int)nblocks, key[cur ^ 1],
                                                     idx[cur ^ 1]);
        cur ^= 1;
    }
    return idx[cur];
}

unsigned key_blocks(int64_t n)
{
    const int64_t b = (n + 255) / 256;
    return (unsigned)(b < 152 * 32 ? b : 152 * 32);
}
}  // namespace

size_t sort_scratch_bytes(int64_t n, int orders)
{
    const int64_t nblocks = (n + kSortBlock - 1) / kSortBlock;
    return (size_t)orders * ((size_t)4 * n + (size_t)kRadix * (nblocks + 1)) * sizeof(uint32_t) + 4 * 256;
}

const uint32_t *launch_spatial_order(const double *S, int64_t n, int64_t ld, double xo0, double xo1, double xo2,
                                     void *scratch, int orders, cudaStream_t s)
{
    if (n <= 0) return nullptr;
    uint32_t *p = reinterpret_cast<uint32_t *>(scratch);
    k_sort_keys<<<dim3(key_blocks(n), orders), 256, 0, s>>>(S, n, ld, xo0, xo1, xo2, p, p + 2 * orders * n);
    return sort_passes(n, orders, p, s);
}

const uint32_t *launch_pixel_order(int64_t N, int64_t pix0, int64_t npix, const int64_t *pix_list, void *scratch,
                                   cudaStream_t s)
{
    uint32_t *p = reinterpret_cast<uint32_t *>(scratch);
    k_pixel_keys<<<key_blocks(npix), 256, 0, s>>>(N, pix0, npix, pix_list, p, p + 2 * npix);
    return sort_passes(npix, 1, p, s);
}

const uint32_t *launch_sort_keys(int64_t n, int orders, void *scratch, cudaStream_t s)
{
    return sort_passes(n, orders, reinterpret_cast<uint32_t *>(scratch), s);
}

int spatial_order_launches() { return 1 + 3 * 3; }

}  // namespace isw
