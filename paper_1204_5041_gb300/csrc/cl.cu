// Angular power spectrum of a full-sky RING map (Sec. IV, Fig. 4 of the paper): spherical-
// harmonic analysis with uniform pixel weights, a_lm = (4 pi / N_pix) sum_p Theta_p Y*_lm(n_p),
// then C_l = (|a_l0|^2 + 2 sum_{m>=1} |a_lm|^2) / (2l + 1).
//   k_fft_table  roots of unity of the largest transform
//   k_ring_fft   F_r(m) = sum_j Theta_rj exp(-i m phi_rj) for the north/south ring pair (i, 4N - i): both
//                rings have one length L and one first phase, so they go through one complex FFT as real
//                and imaginary part (in shared memory; L a power of two directly, other L by Bluestein's
//                chirp transform with the next power of two >= 2L - 1).  A direct sum per (pixel, m)
//                took 160 of the 198 ms of N_side 512, l_max 1536; this takes 1.
//   k_alm        a_lm = (4 pi / N_pix) sum_r lambda_lm(z_r) F_r(m): one block per m, each thread a
//                few north/south ring pairs (lambda_lm(-z) = (-1)^(l+m) lambda_lm(z)), the Legendre
//                recursion in l in the form p_l = z p_{l-1} - beta_l p_{l-2} with the normalisation
//                carried per l outside the sum over rings, and (mantissa, 2^256 power) scaling so that
//                lambda_mm near the poles does not underflow; eight values of l are reduced over the
//                block at a time, in a fixed order (deterministic)
//   k_cl         fixed order over m
// Cost: O(N_pix log N) for the ring sums and four FP64 operations per ring pair, l and m: the FP64 unit
// (0.53e12 FMA/s) bounds k_alm at 9 ms for N_side 512, l_max 1536.
#include "isw_internal.cuh"
#include "kernels.cuh"

namespace isw {

constexpr double kLScale = 1.157920892373162e77;   // 2^256
constexpr int kAlmThreads = 256, kAlmPairs = 8, kCoefChunk = 64, kFftThreads = 256;

struct RingGeom {
    double z, t0;   // z and the first pixel's phase in turns
    int64_t np, p0;
};

__device__ __forceinline__ RingGeom ring_geom(int64_t N, int64_t i)
{
    RingGeom g;
    const double N3 = 3.0 * (double)N * (double)N;
    if (i < N) {
        g.z = 1.0 - ((double)i * (double)i) / N3;
        g.np = 4 * i;
        g.p0 = 2 * i * (i - 1);
        g.t0 = 1.0 / (8.0 * (double)i);
    } else if (i <= 3 * N) {
        g.z = (4.0 * (double)N - 2.0 * (double)i) / (3.0 * (double)N);
        g.np = 4 * N;
        g.p0 = 2 * N * (N - 1) + (i - N) * 4 * N;
        g.t0 = ((i + N) & 1) ? 0.0 : 1.0 / (8.0 * (double)N);
    } else {
        const int64_t k = 4 * N - i;
        g.z = -(1.0 - ((double)k * (double)k) / N3);
        g.np = 4 * k;
        g.p0 = 12 * N * N - 2 * k * (k + 1);
        g.t0 = 1.0 / (8.0 * (double)k);
    }
    return g;
}

// w[k] = exp(-2 pi i k / M), k < M / 2
__global__ void k_fft_table(int M, double2 *__restrict__ w)
{
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < M / 2; k += gridDim.x * blockDim.x) {
        double s, c;
        sincospi(2.0 * (double)k / (double)M, &s, &c);
        w[k] = make_double2(c, -s);
    }
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// In place, block-wide: natural order in, bit-reversed order out; w has the roots of order Mw.
__device__ __forceinline__ void fft_dif(double2 *A, int M, const double2 *__restrict__ w, int Mw)
{
    for (int h = M / 2; h >= 1; h >>= 1) {
        const int st = Mw / (2 * h);
        for (int t = threadIdx.x; t < M / 2; t += blockDim.x) {
            const int j = t & (h - 1), i = 2 * t - j;
            const double2 u = A[i], v = A[i + h];
            A[i] = make_double2(u.x + v.x, u.y + v.y);
            A[i + h] = cmul(make_double2(u.x - v.x, u.y - v.y), w[j * st]);
        }
        __syncthreads();
    }
}

// The inverse (without 1 / M): bit-reversed order in, natural order out.
__device__ __forceinline__ void ifft_dit(double2 *A, int M, const double2 *__restrict__ w, int Mw)
{
    for (int h = 1; h < M; h <<= 1) {
        const int st = Mw / (2 * h);
        for (int t = threadIdx.x; t < M / 2; t += blockDim.x) {
            const int j = t & (h - 1), i = 2 * t - j;
            const double2 r = w[j * st], u = A[i], v = cmul(A[i + h], make_double2(r.x, -r.y));
            A[i] = make_double2(u.x + v.x, u.y + v.y);
            A[i + h] = make_double2(u.x - v.x, u.y - v.y);
        }
        __syncthreads();
    }
}

// exp(-i pi j^2 / L)
__device__ __forceinline__ double2 chirp(int64_t j, int64_t L)
{
    double s, c;
    sincospi((double)((j * j) % (2 * L)) / (double)L, &s, &c);
    return make_double2(c, -s);
}

// F: [mmax + 1][2N][4]: (north + south) re, im, (north - south) re, im of ring pair i - 1; scratch holds
// Mw double2 per block.
__global__ void __launch_bounds__(kFftThreads) k_ring_fft(int64_t N, const double *__restrict__ map, int64_t mmax,
                                                          const double2 *__restrict__ w, int Mw,
                                                          double2 *__restrict__ scratch, double4 *__restrict__ F)
{
    extern __shared__ __align__(16) double2 A[];
    const int tid = threadIdx.x;
    double2 *B = scratch + (int64_t)blockIdx.x * Mw;
    for (int64_t i = 2 * N - blockIdx.x; i >= 1; i -= gridDim.x) {   // the longest rings first
        const RingGeom gn = ring_geom(N, i), gs = ring_geom(N, 4 * N - i);
        const bool equator = i == 2 * N;
        const int L = (int)gn.np;
        const bool pow2 = (L & (L - 1)) == 0;
        int M = L;
        if (!pow2) {
            M = 4;
            while (M < 2 * L - 1) M <<= 1;
            // transform of the conjugate chirp, bit-reversed order, kept in the block's scratch
            for (int j = tid; j < M; j += kFftThreads) {
                const int k = j < M - j ? j : M - j;
                double2 v = make_double2(0.0, 0.0);
                if (k < L) {
                    v = chirp(k, L);
                    v.y = -v.y;
                }
                A[j] = v;
            }
            __syncthreads();
            fft_dif(A, M, w, Mw);
            for (int j = tid; j < M; j += kFftThreads) B[j] = A[j];
            __syncthreads();
        }
        for (int j = tid; j < M; j += kFftThreads) {
            double2 v = make_double2(0.0, 0.0);
            if (j < L) {
                v = make_double2(map[gn.p0 + j], equator ? 0.0 : map[gs.p0 + j]);
                if (!pow2) v = cmul(v, chirp(j, L));
            }
            A[j] = v;
        }
        __syncthreads();
        fft_dif(A, M, w, Mw);
        if (!pow2) {
            for (int j = tid; j < M; j += kFftThreads) A[j] = cmul(A[j], B[j]);
            __syncthreads();
            ifft_dit(A, M, w, Mw);
        }
        const int bits = 31 - __clz(M);
        auto value = [&](int k) -> double2 {   // sum_j z_j exp(-2 pi i j k / L)
            if (pow2) return A[(int)(__brev((unsigned)k) >> (32 - bits))];
            const double2 v = cmul(A[k], chirp(k, L));
            const double s = 1.0 / (double)M;
            return make_double2(v.x * s, v.y * s);
        };
        const int64_t turn = 2 * gn.np;   // phi_r0 = 2 pi t0 with t0 = 0 or 1 / (2 np)
        for (int64_t m = tid; m <= mmax; m += kFftThreads) {
            const int k = (int)(m % L);
            const double2 a = value(k), b = value(k == 0 ? 0 : L - k);
            // z = north + i south, both real: north(k) = (a + b*)/2, south(k) = (a - b*)/(2i)
            const double nr = 0.5 * (a.x + b.x), ni = 0.5 * (a.y - b.y);
            const double sr = 0.5 * (a.y + b.y), si = 0.5 * (b.x - a.x);
            double2 ph = make_double2(1.0, 0.0);
            if (gn.t0 != 0.0) {
                double s, c;
                sincospi((double)(m % turn) * (1.0 / (double)gn.np), &s, &c);
                ph = make_double2(c, -s);
            }
            const double2 e = cmul(make_double2(nr + sr, ni + si), ph), o = cmul(make_double2(nr - sr, ni - si), ph);
            F[m * (2 * N) + (i - 1)] = make_double4(e.x, e.y, o.x, o.y);
        }
        __syncthreads();
    }
}

// value * 2^(256 sc), normalised so that |value| stays in range
struct Scaled {
    double v;
    int sc;
};

// sin(theta)^m as a scaled value (repeated squaring with rescaling)
__device__ __forceinline__ Scaled pow_scaled(double x, int64_t m)
{
    Scaled r{1.0, 0}, b{x, 0};
    while (m > 0) {
        if (m & 1) {
            r.v *= b.v;
            r.sc += b.sc;
            while (r.v != 0.0 && fabs(r.v) < 1.0 / kLScale) { r.v *= kLScale; --r.sc; }
        }
        m >>= 1;
        if (m) {
            b.v *= b.v;
            b.sc *= 2;
            while (b.v != 0.0 && fabs(b.v) < 1.0 / kLScale) { b.v *= kLScale; --b.sc; }
        }
    }
    return r;
}

// Sums the 16 values of every lane over the warp; lane 2k (and 2k + 1) ends with value k.
__device__ __forceinline__ double warp_sum16(double (&v)[16])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = 8; n >= 1; n >>= 1) {
        const bool up = (lane & (2 * n)) != 0;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            const double send = up ? v[k] : v[k + n], keep = up ? v[k + n] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * n);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// alm: double[2][mmax+1][lmax+1]; one block per m.  lambda_lm = A_l p_l with A_l the running product of
// a_l = sqrt((4 l^2 - 1) / (l^2 - m^2)) since the chunk's start and
//   p_l = z p_{l-1} - beta_l p_{l-2},  beta_l = ((l-1)^2 - m^2) / ((2l-1)(2l-3)),
// so a ring costs two operations for the recursion and two for its sums; at the end of a chunk both p
// are multiplied by A.  The rings of a warp's q-th group are left out of the sums while all of them are
// below 2^-256 (m beyond l sin theta).
template <int Q>
__global__ void __launch_bounds__(kAlmThreads) k_alm(int64_t N, const double4 *__restrict__ F, int64_t lmax,
                                                    double omega, double *__restrict__ alm)
{
    __shared__ double s_beta[kCoefChunk], s_a[kCoefChunk], s_A[kCoefChunk];
    __shared__ double red[2][kAlmThreads / 32][16];
    const int64_t m = blockIdx.x, L1 = lmax + 1, npair = 2 * N;   // pairs (i, 4N - i), i = 1..2N; i = 2N alone
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nt = blockDim.x, nw = nt >> 5;
    // c_m = sqrt((2m+1)/(4 pi) prod_{k<=m} (2k-1)/(2k)) (no underflow: ~ m^(-1/4)); the product over the
    // lanes of a warp, in a fixed order
    double cm = 1.0;
    for (int64_t k = 1 + lane; k <= m; k += 32) cm *= (2.0 * k - 1.0) / (2.0 * k);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cm *= __shfl_xor_sync(0xffffffffu, cm, o);
    cm = sqrt(cm * (2.0 * m + 1.0) / (4.0 * kPi));
    if (m & 1) cm = -cm;
    double p1[Q], p2[Q], zz[Q], fr[2][Q], fi[2][Q];
    int sc[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int64_t pidx = tid + (int64_t)q * nt;
        p1[q] = p2[q] = zz[q] = 0.0;
        sc[q] = 1;   // > 0: unused slot, contributes nothing
        fr[0][q] = fr[1][q] = fi[0][q] = fi[1][q] = 0.0;
        if (pidx < npair) {
            const RingGeom g = ring_geom(N, pidx + 1);   // north ring (z >= 0)
            const double4 f = F[m * npair + pidx];
            zz[q] = g.z;
            fr[0][q] = f.x;
            fi[0][q] = f.y;
            fr[1][q] = f.z;
            fi[1][q] = f.w;
            const Scaled sm = pow_scaled(sqrt((1.0 - g.z) * (1.0 + g.z)), m);
            p1[q] = cm * sm.v;
            sc[q] = sm.sc;
            while (p1[q] != 0.0 && fabs(p1[q]) < 1.0 / kLScale) { p1[q] *= kLScale; --sc[q]; }
        }
    }
    int buf = 0;
    // chunk of kCoefChunk values of l from l0; index l0 itself is the start value when l0 == m
    for (int64_t l0 = m; l0 <= lmax; l0 += kCoefChunk) {
        if (tid < kCoefChunk) {
            const double ll = (double)(l0 + tid), mm = (double)m;
            s_beta[tid] = l0 + tid < m + 2 ? 0.0 : ((ll - 1.0) * (ll - 1.0) - mm * mm) / ((2.0 * ll - 1.0) * (2.0 * ll - 3.0));
            s_a[tid] = l0 + tid == m ? 1.0 : sqrt((4.0 * ll * ll - 1.0) / (ll * ll - mm * mm));
        }
        __syncthreads();
        if (tid < kCoefChunk) {   // running product, the same order in every thread
            double A = 1.0;
            for (int k = 0; k <= tid; ++k) A *= s_a[k];
            s_A[tid] = A;
        }
        __syncthreads();
        for (int b0 = 0; b0 < kCoefChunk && l0 + b0 <= lmax; b0 += 8) {
            double v[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = 0.0;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const bool live = __any_sync(0xffffffffu, sc[q] == 0);
                const bool on = sc[q] == 0;
                const double er = on ? fr[0][q] : 0.0, ei = on ? fi[0][q] : 0.0, gr = on ? fr[1][q] : 0.0,
                             gi = on ? fi[1][q] : 0.0;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (l0 + b0 + j > m) {
                        const double pn = fma(zz[q], p1[q], -(s_beta[b0 + j] * p2[q]));
                        p2[q] = p1[q];
                        p1[q] = pn;
                    }
                    if (live) {   // l0 - m and b0 are even: the parity of l + m is that of j
                        v[2 * j] = fma(p1[q], (j & 1) ? gr : er, v[2 * j]);
                        v[2 * j + 1] = fma(p1[q], (j & 1) ? gi : ei, v[2 * j + 1]);
                    }
                }
                // a value that has grown past 1 takes its power back (true lambda = p A 2^(256 sc))
                if (sc[q] < 0 && fabs(p1[q]) * s_A[b0 + 7] > 1.0) {
                    p1[q] *= 1.0 / kLScale;
                    p2[q] *= 1.0 / kLScale;
                    ++sc[q];
                }
            }
            const double t = warp_sum16(v);
            if (!(lane & 1)) red[buf][wid][lane >> 1] = t;
            __syncthreads();
            if (tid < 16 && l0 + b0 + tid / 2 <= lmax) {
                double s = 0.0;
                for (int k = 0; k < nw; ++k) s += red[buf][k][tid];
                alm[(tid & 1) * L1 * L1 + m * L1 + l0 + b0 + tid / 2] = omega * s_A[b0 + tid / 2] * s;
            }
            buf ^= 1;
        }
        __syncthreads();
        const double A = s_A[kCoefChunk - 1];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            p1[q] *= A;
            p2[q] *= A;
        }
        __syncthreads();
    }
}

// One warp per value of m mod 8 of a block of 32 values of l; the eight partial sums added in order.
__global__ void __launch_bounds__(256) k_cl(const double *__restrict__ alm, int64_t lmax, double *__restrict__ cl)
{
    __shared__ double part[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t L1 = lmax + 1, l = blockIdx.x * 32ll + lane;
    double s = 0.0;
    for (int64_t m = w; m <= blockIdx.x * 32ll + 31 && m <= lmax; m += 8) {
        if (l > lmax || m > l) continue;
        const double re = alm[m * L1 + l], im = alm[L1 * L1 + m * L1 + l];
        const double p = re * re + im * im;
        s += m == 0 ? p : 2.0 * p;
    }
    part[w][lane] = s;
    __syncthreads();
    if (w == 0 && l <= lmax) {
        for (int k = 1; k < 8; ++k) s += part[k][lane];
        cl[l] = s / (2.0 * l + 1.0);
    }
}

int cl_max_nside() { return kAlmPairs * kAlmThreads / 2; }

namespace {
// order of the largest transform: 4N when N is a power of two, else the chirp transform of the rings
int fft_order(int64_t N)
{
    int M = 4;
    const bool pow2 = (N & (N - 1)) == 0;
    // the polar rings of a power-of-two N go up to L = 4 (N - 1), not a power of two
    const int64_t need = pow2 ? (N > 1 ? 2 * 4 * (N - 1) - 1 : 4) : 2 * 4 * N - 1;
    while (M < need || M < (pow2 ? 4 * N : 4)) M <<= 1;
    return M;
}
int fft_blocks(int64_t N)
{
    const int64_t b = 152 * 3;
    return (int)(2 * N < b ? 2 * N : b);
}
size_t cl_f_bytes(int64_t N, int64_t lmax) { return (size_t)(lmax + 1) * 2 * N * sizeof(double4); }
}  // namespace

size_t cl_scratch_bytes(int64_t N, int64_t lmax)
{
    const size_t M = (size_t)fft_order(N);
    return cl_f_bytes(N, lmax) + (M / 2 + M * fft_blocks(N)) * sizeof(double2);
}

void launch_map_cl(int64_t N, const double *map, int64_t lmax, void *scratch, double *alm, double *cl, cudaStream_t s)
{
    const int M = fft_order(N);
    double4 *F = (double4 *)scratch;
    double2 *w = (double2 *)((unsigned char *)scratch + cl_f_bytes(N, lmax)), *B = w + M / 2;
    const size_t smem = (size_t)M * sizeof(double2);
    cudaFuncSetAttribute((const void *)&k_ring_fft, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_fft_table<<<(M / 2 + 255) / 256, 256, 0, s>>>(M, w);
    k_ring_fft<<<fft_blocks(N), kFftThreads, smem, s>>>(N, map, lmax, w, M, B, F);
    // only l >= m is written: clear the plane so the unused triangle reads as zero
    cudaMemsetAsync(alm, 0, (size_t)2 * (lmax + 1) * (lmax + 1) * sizeof(double), s);
    // up to four ring pairs per thread while 256 threads hold them all: fewer pairs per thread keep the
    // recursions of a small map spread over the warps
    const int64_t npair = 2 * N;
    const double omega = 4.0 * kPi / (12.0 * (double)N * (double)N);
    const unsigned grid = (unsigned)(lmax + 1);
    auto threads = [&](int Q) {
        int64_t t = ((npair + Q - 1) / Q + 31) / 32 * 32;
        return (unsigned)(t < kCoefChunk ? kCoefChunk : t);
    };
    if (npair <= 2 * kAlmThreads) k_alm<2><<<grid, threads(2), 0, s>>>(N, F, lmax, omega, alm);
    else if (npair <= 4 * kAlmThreads) k_alm<4><<<grid, threads(4), 0, s>>>(N, F, lmax, omega, alm);
    else k_alm<kAlmPairs><<<grid, threads(kAlmPairs), 0, s>>>(N, F, lmax, omega, alm);
    k_cl<<<(unsigned)(lmax / 32 + 1), 256, 0, s>>>(alm, lmax, cl);
}

}  // namespace isw
