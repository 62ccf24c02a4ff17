// Core Stage CG of a small problem as one cooperative launch (FP32 path).
//
// A step by launches is a chain of five to six dependent kernels of 3 to 10
// us on L2-resident vectors: what a small problem waits for is the chain, not
// the work.  Here one thread owns one node for the whole solve, with the
// residual and the direction of all its components in registers; a step is
// its phases with a grid barrier between them, and the stop test runs on the
// device (the host polls nothing).  The barrier's release and acquire order
// the blocks' vectors for one another, so these are read by ordinary loads
// (from L1 where a neighbour in the block has read the line: the two
// Laplacians read each node seven times in 3-D); their pointers must not be
// __restrict__, which would let them take the path for constant data.
//
// Measured on GB300: 48 x 48 x 24 / 65 536 samples, 20 steps with the setup
// 1.02 ms (by launches 1.33 ms); 100 x 100 / 1632 samples to the tolerance,
// 65 to 150 steps, 19 us a step (by launches 48 us).  Four (2-D) or five (3-D)
// barriers and the L2 latency of what crosses them bound a step.
#pragma once

#include "grid_common.cuh"

namespace mpi {

constexpr int kResThreads = 256;
constexpr int kResMinBlocks = 2;
constexpr int kResFlat = 2048;  // unknowns per partial sum of r.r

// Barrier of all blocks of a cooperative launch: `arrived` counts up for the
// life of the launch.  A wait gives up after kResSpin polls (seconds) and
// raises `failed`; the solve then returns NaN.
struct ResBarrier {
    unsigned long long arrived;
    int failed;
};
constexpr int kResSpin = 1 << 22;

#ifdef __CUDACC__

// The barrier in two halves.  All threads call both; work of a block's own
// may stand between them.  The block's writes before res_arrive are ordered
// before its arrival (bar.sync, then a release by thread 0), the others'
// after the wait (an acquire by thread 0, then bar.sync).  res_wait is false
// once a wait has given up.
__device__ __forceinline__ void res_arrive(ResBarrier *b)
{
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(&b->arrived) : "memory");
}
__device__ __forceinline__ bool res_wait(ResBarrier *b, unsigned long long &target, int *s_ok)
{
    target += gridDim.x;
    if (threadIdx.x == 0) {
        int ok = 1, n = 0;
        unsigned long long seen;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(&b->arrived) : "memory");
            if (seen >= target) break;
            if (++n > kResSpin) {
                atomicExch(&b->failed, 1);
                ok = 0;
                break;
            }
        }
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}
__device__ __forceinline__ bool res_barrier(ResBarrier *b, unsigned long long &target, int *s_ok)
{
    res_arrive(b);
    return res_wait(b, target, s_ok);
}

// The block's partial sums of v over groups of PT consecutive threads, as
// CsDot::block_total<PT> forms them; part[group] for the first n_part groups.
template <int PT>
__device__ __forceinline__ void res_partials(F2Sum v, F2Sum *w, double *part, int n_part)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        F2Sum t;
        t.hi = __shfl_xor_sync(0xffffffffu, v.hi, o);
        t.lo = __shfl_xor_sync(0xffffffffu, v.lo, o);
        v.add(t);
    }
    __syncthreads();  // (w may still be read)
    if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = v;
    __syncthreads();
    constexpr int G = kResThreads / PT, W = PT / 32;
    const int group = blockIdx.x * G + threadIdx.x;
    if (threadIdx.x < G && group < n_part) {
        F2Sum s = w[threadIdx.x * W];
#pragma unroll
        for (int k = 1; k < W; ++k) s.add(w[threadIdx.x * W + k]);
        part[group] = s.value();
    }
}

// Their sum as cs_sum_parts<PT> forms it, in thread 0.  (FP64 additions take
// a warp 19 clocks: warps without a partial leave them out.)
template <int PT>
__device__ __forceinline__ double res_sum(const double *part, int n, double *sh)
{
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x < PT && 32 * warp < n) {
        double a = 0.0;
        for (int k = threadIdx.x; k < n; k += PT) a += part[k];
        a = warp_sum(a);
        if ((threadIdx.x & 31) == 0) sh[warp] = a;
    }
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < PT / 32 && 32 * w < n; ++w) t += sh[w];
    return t;
}

// One solve.  Op: kNC components; kPhases phases of M^T M p (phase(k) by all
// threads, a barrier after each); combine(node, sum), the node's sums of the
// transpose; lap(f, node); store_p32(node, v), the FP32 copy of the direction
// that phase(0) reads; kPqThreads; scalars scale = 1/T and gamma.  p, l1, q:
// kNC N elements; pq_part, rr_part: their partial sums; bar zeroed before the
// launch.
//
// Every sum is taken in the order of the step by launches, so that both give
// the same bits (a solve to a tolerance on a badly conditioned system carries
// a last-bit difference into the fourth digit of the field): <p, q> over
// groups of kPqThreads nodes, r.r over blocks of kResFlat unknowns in memory
// order.  For the latter the first blocks also keep the residual in that
// order and update it from q, which the owners of the nodes leave in memory.
template <class Op>
__global__ void __launch_bounds__(kResThreads, kResMinBlocks)
k_cs_resident(const __grid_constant__ Op op, int N, const float2 *__restrict__ b, float2 *x, float2 *p, float2 *l1,
              float2 *qv, double rel_tol, int max_iter, double *pq_part, double *rr_part, CsScal *sc, ResBarrier *bar)
{
    constexpr int NC = Op::kNC, PT = Op::kPqThreads, U = kResFlat / kResThreads;
    __shared__ double sh[kResThreads / 32];
    __shared__ F2Sum sw[kResThreads / 32];
    __shared__ df s_coef;
    __shared__ int s_ok, s_stop, s_zero;
    __shared__ double s_rr, s_tol;
    unsigned long long target = 0;
    const int node = blockIdx.x * kResThreads + threadIdx.x;
    const bool in = node < N;
    const int n_pq = (N + PT - 1) / PT;
    const int64_t n = (int64_t)NC * N, flat0 = (int64_t)blockIdx.x * kResFlat + threadIdx.x;
    const int n_rr = (int)((n + kResFlat - 1) / kResFlat);
    const bool flat = int(blockIdx.x) < n_rr;
    bool ok = true;
    double rr = 0.0;  // thread 0's
    df r[NC], d[NC], rf[U];
    if (flat) {
        CsDot<df> acc{};
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t e = flat0 + u * kResThreads;
            rf[u] = e < n ? b[e] : make_float2(0.0f, 0.0f);
            if (e < n) acc.add(rf[u], rf[u]);
        }
        res_partials<kResThreads>(acc.s, sw, rr_part, n_rr);
    }
    if (in) {
        float v[NC];
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            const int64_t e = (int64_t)m * N + node;
            r[m] = d[m] = b[e];
            x[e] = make_float2(0.0f, 0.0f);
            p[e] = d[m];
            v[m] = cs_to_float(d[m]);
        }
        op.store_p32(node, v);
    }
    ok = res_barrier(bar, target, &s_ok);
    {
        const double v = res_sum<kResThreads>(rr_part, n_rr, sh);
        if (threadIdx.x == 0) {
            rr = s_rr = v;
            s_tol = rel_tol > 0.0 ? rel_tol * sqrt(v) : -1.0;
        }
    }
    int it = 0;
    for (; ok && it < max_iter; ++it) {
        if (in) {
#pragma unroll
            for (int m = 0; m < NC; ++m) l1[(int64_t)m * N + node] = op.lap(p + (int64_t)m * N, node);
        }
#pragma unroll 1
        for (int k = 0; k < Op::kPhases; ++k) {
            op.phase(k);
            ok = res_barrier(bar, target, &s_ok) && ok;
        }
        if (!ok) break;
        df q[NC];
        CsDot<df> pq_acc{};
        if (in) {
            SumAcc<float> sum[NC] = {};
            op.combine(node, sum);
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                q[m] = cs_sum_scale_add(sum[m], op.scale, df_mul(op.lap(l1 + (int64_t)m * N, node), op.gamma));
                qv[(int64_t)m * N + node] = q[m];
                pq_acc.add(d[m], q[m]);
            }
        }
        res_partials<PT>(pq_acc.s, sw, pq_part, n_pq);
        ok = res_barrier(bar, target, &s_ok) && ok;
        {
            const double pq = res_sum<PT>(pq_part, n_pq, sh);
            if (threadIdx.x == 0) {
                s_zero = pq == 0.0;
                s_coef = df_from_double(rr / pq);
            } else if (threadIdx.x == 32) {  // (beside the division)
                s_stop = s_rr == 0.0 || (s_tol >= 0.0 && sqrt(s_rr) <= s_tol);
            }
            __syncthreads();
        }
        if (!ok || s_stop || s_zero) break;
        const df al = s_coef, nal = df_neg(al);
        if (flat) {
            CsDot<df> acc{};
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t e = flat0 + u * kResThreads;
                if (e < n) {
                    rf[u] = df_axpy(rf[u], nal, qv[e]);
                    acc.add(rf[u], rf[u]);
                }
            }
            res_partials<kResThreads>(acc.s, sw, rr_part, n_rr);
        }
        res_arrive(bar);
        if (in) {
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                const int64_t e = (int64_t)m * N + node;
                x[e] = df_axpy(x[e], al, d[m]);
                r[m] = df_axpy(r[m], nal, q[m]);
            }
        }
        ok = res_wait(bar, target, &s_ok) && ok;
        {
            const double v = res_sum<kResThreads>(rr_part, n_rr, sh);
            if (threadIdx.x == 0) {
                s_coef = df_from_double(v / rr);
                rr = s_rr = v;
            }
            __syncthreads();
        }
        const df be = s_coef;
        if (in) {
            float v[NC];
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                d[m] = df_axpy(r[m], be, d[m]);
                p[(int64_t)m * N + node] = d[m];
                v[m] = cs_to_float(d[m]);
            }
            op.store_p32(node, v);
        }
        ok = res_barrier(bar, target, &s_ok) && ok;
    }
    if (!ok && in) {
#pragma unroll
        for (int m = 0; m < NC; ++m) x[(int64_t)m * N + node] = make_float2(nanf(""), 0.0f);
    }
    if (node == 0) {
        sc->rr = rr;
        sc->iters = it;
        sc->done = 1;
    }
}

// Runs the solve if the device holds all its blocks at once; taken says
// whether it did.  work: units of the first phase for a whole warp's lanes.
template <class Op>
int launch_resident(const Op &op, int64_t N, int64_t work, const float2 *b, const mpi_grid_opts &o, float2 *x, CsScal *sc,
                    cudaStream_t st, bool &taken)
{
    taken = false;
    auto kern = k_cs_resident<Op>;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kResThreads, 0) != cudaSuccess) return MPI_OK;
    const int64_t most = (int64_t)std::min(per_sm, kResMinBlocks) * device_sm_count();
    const int64_t n_rr = (Op::kNC * N + kResFlat - 1) / kResFlat, n_pq = (N + Op::kPqThreads - 1) / Op::kPqThreads;
    const int64_t need = std::max((N + kResThreads - 1) / kResThreads, n_rr);
    if (need > most) return MPI_OK;
    int grid = (int)std::min(most, std::max(need, work * 32 / kResThreads));
    Scratch scr(st);
    const size_t vb = sizeof(float2) * Op::kNC * N;
    const size_t o_p = scr.reserve(vb), o_l = scr.reserve(vb), o_q = scr.reserve(vb),
                 o_pq = scr.reserve(sizeof(double) * n_pq), o_rr = scr.reserve(sizeof(double) * n_rr),
                 o_bar = scr.reserve(sizeof(ResBarrier));
    MPI_TRY(scr.allocate());
    float2 *p = scr.at<float2>(o_p), *l1 = scr.at<float2>(o_l), *q = scr.at<float2>(o_q);
    double *pq_part = scr.at<double>(o_pq), *rr_part = scr.at<double>(o_rr), rel_tol = o.rel_tol;
    ResBarrier *bar = scr.at<ResBarrier>(o_bar);
    int n = (int)N, max_iter = o.max_iter;
    Op arg = op;
    MPI_TRY_CUDA(cudaMemsetAsync(bar, 0, sizeof(ResBarrier), st));
    void *args[] = {&arg, &n, &b, &x, &p, &l1, &q, &rel_tol, &max_iter, &pq_part, &rr_part, &sc, &bar};
    if (cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(kResThreads), args, 0, st) != cudaSuccess) {
        (void)cudaGetLastError();  // the launches do the same
        return MPI_OK;
    }
    note_launch();
    taken = true;
    return MPI_OK;
}

#endif

}  // namespace mpi
