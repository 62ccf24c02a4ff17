// Device building blocks shared by the single-frame and the batched PnP
// solves: fixed-order sums of partials, the radix-select order statistic, the
// percentile/variance block and the 5-tap Gaussian tile.
#pragma once

#include <cooperative_groups.h>

#include <cmath>

#include "pnp_ops.cuh"

namespace mpi {

constexpr int kVecThreads = 256;
// Elements per block of the CG vector kernels (and so the number of partial
// sums of r.r): small enough that a 128 x 128 problem spreads over 32 blocks.
constexpr int kVecPerBlock = 512;
constexpr int kStatThreads = 1024;
// Values per iteration in a solve's device record (mpi_pnp_iter_info).
constexpr int kInfoCols = 4;

// Sum of `n` partials in a fixed order, computed by the whole block and
// returned to every thread (deterministic: fixed strides, fixed tree).
template <int NT>
__device__ double sum_parts(const double *__restrict__ part, int n, double *sh /* NT/32 + 1 */)
{
    double a = 0.0;
    for (int k = threadIdx.x; k < n; k += NT) a += part[k];
    a = block_sum<double, NT>(a, sh);
    if (threadIdx.x == 0) sh[NT / 32] = a;
    __syncthreads();
    const double r = sh[NT / 32];
    __syncthreads();
    return r;
}

// ---------------------------------------------------------------------------
// Percentile trimming and noise estimate (Sec. 3.3 and the noise estimator of
// Algorithm 1): exact order statistics by an 8-pass radix select on the
// order-preserving integer image of the FP64 values.

__device__ __forceinline__ uint64_t f64_key(double v)
{
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double key_f64(uint64_t k)
{
    const uint64_t b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)b);
}

// Minimum over the block (order-independent), returned to every thread.
template <int NT>
__device__ __forceinline__ double block_min(double v, double *sh /* >= NT/32 + 1 */)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();  // sh may still be read by an earlier reduction
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = sh[0];
        for (int w = 1; w < NT / 32; ++w) m = fmin(m, sh[w]);
        sh[NT / 32] = m;
    }
    __syncthreads();
    const double r = sh[NT / 32];
    __syncthreads();
    return r;
}

// The percentile step runs on a cluster of up to kStatBlocks blocks per image
// (distributed shared memory, cluster barriers): FP64 additions and
// comparisons take a block's SM 19 clocks per warp, so one block alone is
// bound by them (80 us at 100 x 100 values), while on few values the 20
// barriers of a cluster cost more than they save.  Four iterations of a small
// reconstruction with one block / with eight: 60 x 50 values 1040 / 1070 us,
// 70 x 60 1120 / 1123 us, 80 x 70 1195 / 1175 us, 100 x 100 1463 / 1363 us.
constexpr int kStatBlocks = 8;
inline int stat_blocks(int64_t N) { return N <= 4096 ? 1 : kStatBlocks; }

// The sums run in the order of one block of kStatThreads threads (thread t
// over the values t, t + kStatThreads, ...; its warps in order): each block
// takes its share of that block's warps.
struct StatShared {
    unsigned hist[256];
    double part[kStatThreads / 32];  // this block's partial sums, minimum and count,
    double least;                    // read by the others
    unsigned long long cnt;
    double sh[kStatThreads / 32 + 1];
    unsigned long long sel[2]; // prefix, remaining rank
};

// The values of rank `rank` (0-based) among the N: an 8-pass radix select on
// the order-preserving integer image; every block ends with the same value.
__device__ inline double cluster_select(const double *__restrict__ x, int64_t N, int64_t rank, StatShared &S)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31;
    const int nb = cl.num_blocks();
    const int64_t first = (int64_t)cl.block_rank() * kStatThreads, stride = (int64_t)nb * kStatThreads;
    uint64_t prefix = 0, mask = 0;
    int64_t krem = rank;
    for (int shift = 56; shift >= 0; shift -= 8) {
        if (tid < 256) S.hist[tid] = 0;
        __syncthreads();
        for (int64_t i0 = first; i0 < N; i0 += stride) {
            const int64_t i = i0 + tid;
            unsigned digit = 256;  // no bin
            if (i < N) {
                const uint64_t key = f64_key(x[i]);
                if ((key & mask) == prefix) digit = (unsigned)((key >> shift) & 255u);
            }
            const unsigned peers = __match_any_sync(0xffffffffu, digit);
            if (digit < 256 && lane == __ffs(peers) - 1) atomicAdd(&S.hist[digit], (unsigned)__popc(peers));
        }
        cl.sync();
        if (tid < 32) {  // eight digits per lane: the digit that holds the rank
            unsigned long long c[8], sum = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                unsigned long long n = 0;
                for (int b = 0; b < nb; ++b) n += *cl.map_shared_rank(&S.hist[8 * lane + q], b);
                c[q] = n;
                sum += n;
            }
            unsigned long long pre = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, pre, o);
                if (lane >= o) pre += y;
            }
            pre -= sum;
            const unsigned long long k = (unsigned long long)krem;
            if ((k >= pre && k < pre + sum) || (lane == 31 && k >= pre + sum)) {
                int q = 0;
                while (q < 7 && pre + c[q] <= k) pre += c[q++];
                S.sel[0] = prefix | ((uint64_t)(8 * lane + q) << shift);
                S.sel[1] = k - pre;
            }
        }
        cl.sync();  // the counts are read; sel is written
        prefix = S.sel[0];
        krem = (int64_t)S.sel[1];
        mask |= (uint64_t)255 << shift;
    }
    return key_f64(prefix);
}

// Sum of f(i) over the N values in the order of one block, for every thread.
template <typename F>
__device__ inline double cluster_sum(int64_t N, F f, StatShared &S)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, share = kStatThreads / 32 / cl.num_blocks();
    if (warp < share) {
        double s = 0.0;
        for (int64_t i = ((int)cl.block_rank() * share + warp) * 32 + lane; i < N; i += kStatThreads) s += f(i);
        s = warp_sum(s);
        if (lane == 0) S.part[warp] = s;
    }
    cl.sync();
    if (warp == 0) {
        double t = *cl.map_shared_rank(&S.part[lane % share], lane / share);
        double a = 0.0;
        for (int w = 0; w < kStatThreads / 32; ++w) a += __shfl_sync(0xffffffffu, t, w);
        if (lane == 0) S.sh[kStatThreads / 32] = a;
    }
    cl.sync();  // (the partials are read)
    return S.sh[kStatThreads / 32];
}

// One cluster computes, for the N values x: the clip value P (the pct-th
// percentile, linear interpolation between order statistics; -inf when
// do_clip is 0), rho1 = max(x, P) rounded to R, the population variance of
// rho1 in two FP64 passes, and updates the PnP scalars: sigma, lambda = nu0
// sigma^2 on the first iteration, nu = lambda / sigma^2 (kept if sigma = 0).
// rr_part/nblk: partial sums of the final CG residual for info_row (sigma,
// nu, residual norm, clip value: kInfoCols values).
template <typename R>
__device__ void outer_stats_cluster(int64_t N, const double *__restrict__ x, int do_clip, double pct,
                                    bool first, double nu0, double *__restrict__ scal,
                                    const double *__restrict__ rr_part, int nblk,
                                    double *__restrict__ info_row, R *__restrict__ rho1)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ StatShared S;
    const int64_t i0 = (int64_t)cl.block_rank() * kStatThreads + threadIdx.x;
    const int64_t stride = (int64_t)cl.num_blocks() * kStatThreads;
    double P = -INFINITY;
    if (do_clip) {
        const double h = double(N - 1) * pct / 100.0;
        const int64_t lo = (int64_t)floor(h);
        const int64_t hi = min(lo + 1, N - 1);
        const double xlo = cluster_select(x, N, lo, S);
        // The next order statistic in one pass instead of a second select:
        // x(lo + 1) is xlo itself when more than lo + 1 values are <= xlo,
        // else the smallest value above xlo (exact, order-independent).
        double xhi = xlo;
        if (hi != lo) {
            long long le = 0;
            double gt = INFINITY;
            for (int64_t i = i0; i < N; i += stride) {
                const double v = x[i];
                if (v <= xlo) ++le;
                else gt = fmin(gt, v);
            }
            le = block_sum<long long, kStatThreads>(le, reinterpret_cast<long long *>(S.sh));
            gt = block_min<kStatThreads>(gt, S.sh);
            if (threadIdx.x == 0) {
                S.cnt = (unsigned long long)le;
                S.least = gt;
            }
            cl.sync();
            le = 0;
            for (int b = 0; b < (int)cl.num_blocks(); ++b) {
                le += (long long)*cl.map_shared_rank(&S.cnt, b);
                gt = fmin(gt, *cl.map_shared_rank(&S.least, b));
            }
            xhi = le > hi ? xlo : gt;
        }
        P = xlo + (h - double(lo)) * (xhi - xlo);
    }
    for (int64_t i = i0; i < N; i += stride) rho1[i] = R(fmax(x[i], P));
    const double mean = cluster_sum(N, [&](int64_t i) { return fmax(x[i], P); }, S) / double(N);
    const double q = cluster_sum(N, [&](int64_t i) {
        const double dv = fmax(x[i], P) - mean;
        return dv * dv;
    }, S);
    if (cl.block_rank() == 0 && threadIdx.x < 32) {
        double rr = 0.0;
        for (int b = threadIdx.x; b < nblk; b += 32) rr += rr_part[b];
        rr = warp_sum(rr);
        if (threadIdx.x == 0) {
            const double sigma = sqrt(q / double(N));
            if (first) scal[kScalLambda] = nu0 * sigma * sigma;
            if (sigma > 0.0) scal[kScalNu] = scal[kScalLambda] / (sigma * sigma);
            scal[kScalSigma] = sigma;
            scal[kScalPct] = P;
            if (info_row) {
                info_row[0] = sigma;
                info_row[1] = scal[kScalNu];
                info_row[2] = sqrt(rr);
                info_row[3] = P;
            }
        }
    }
    cl.sync();  // no block leaves while another reads its shared memory
}

// ---------------------------------------------------------------------------
// Built-in denoiser: separable 5-tap Gaussian (sigma = 1 px), reflect
// boundary (d c b a | a b c d).

__device__ __forceinline__ int reflect_index(int i, int n)
{
    const int p = 2 * n;
    i %= p;
    if (i < 0) i += p;
    return i >= n ? p - 1 - i : i;
}

constexpr int kGx = 32, kGy = 8;

// One 32 x 8 output tile of the separable 5-tap Gaussian (rows first, then
// columns; reflect boundary) for tile origin (i0, j0).
template <typename R>
__device__ void gauss5_tile(const R *__restrict__ in, R *__restrict__ out, int nx, int ny, int i0,
                            int j0, R w0, R w1, R w2)
{
    __shared__ R tmp[kGy + 4][kGx];
    const R w[5] = {w2, w1, w0, w1, w2};
    const int tx = threadIdx.x % kGx, ty = threadIdx.x / kGx;
    const int i = i0 + tx;
    const int ic = min(i, nx - 1);
    for (int rr = ty; rr < kGy + 4; rr += kGy) {
        const int jr = reflect_index(j0 - 2 + rr, ny);
        const R *row = in + (int64_t)jr * nx;
        R acc = R(0);
#pragma unroll
        for (int m = -2; m <= 2; ++m) acc += w[m + 2] * row[reflect_index(ic + m, nx)];
        tmp[rr][tx] = acc;
    }
    __syncthreads();
    const int j = j0 + ty;
    if (i < nx && j < ny) {
        R acc = R(0);
#pragma unroll
        for (int m = -2; m <= 2; ++m) acc += w[m + 2] * tmp[reflect_index(j + m, ny) - (j0 - 2)][tx];
        out[(int64_t)j * nx + i] = acc;
    }
}

// 5-tap Gaussian weights exp(-m^2/2)/sum for m = 0, 1, 2.
inline void gauss5_weights(double w[3])
{
    double tot = 0.0;
    for (int m = -2; m <= 2; ++m) tot += std::exp(-0.5 * m * m);
    for (int m = 0; m <= 2; ++m) w[m] = std::exp(-0.5 * m * m) / tot;
}

}  // namespace mpi
