// Core Stage CG of a small problem as one cooperative launch (FP32 path).
//
// A step by launches is a chain of five to six dependent kernels of 3 to 10
// us on L2-resident vectors: what a small problem waits for is the chain, not
// the work.  Here one thread owns one node for the whole solve, with the
// residual and the direction of all its components in registers; a step is
// its phases with a grid barrier between them, and the stop test runs on the
// device (the host polls nothing).  Blocks read one another's vectors
// through L2 (__ldcg).
#pragma once

#include "grid_common.cuh"

namespace mpi {

constexpr int kResThreads = 256;
constexpr int kResMinBlocks = 2;

// Barrier of all blocks of a cooperative launch: `arrived` counts up for the
// life of the launch.  A wait gives up after kResSpin polls (seconds) and
// raises `failed`; the solve then returns NaN.
struct ResBarrier {
    unsigned long long arrived;
    int failed;
};
constexpr int kResSpin = 1 << 22;

#ifdef __CUDACC__

// Loads of data that other blocks write during the launch (COH) or before it.
template <bool COH, typename T> __device__ __forceinline__ T ld_shared_by_blocks(const T *p)
{
    if constexpr (COH) return __ldcg(p);
    else return *p;
}

// All threads call it; false once a wait has given up.  The block's writes
// are ordered before its arrival (bar.sync, then a release by thread 0), the
// others' after the wait (an acquire by thread 0, then bar.sync).
__device__ __forceinline__ bool res_barrier(ResBarrier *b, unsigned long long &target, int *s_ok)
{
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(&b->arrived) : "memory");
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

// One solve.  Op: kNC components; kPhases phases of M^T M p (phase(k) by all
// threads, a barrier after each); combine(node, sum), the node's sums of the
// transpose; lap(f, node); store_p32(node, v), the FP32 copy of the direction
// that phase(0) reads; scalars scale = 1/T and gamma.  p, l1: kNC N elements;
// part: 2 gridDim.x doubles; bar zeroed before the launch.
template <class Op>
__global__ void __launch_bounds__(kResThreads, kResMinBlocks)
k_cs_resident(const __grid_constant__ Op op, int N, const float2 *__restrict__ b, float2 *x, float2 *p, float2 *l1,
              double rel_tol, int max_iter, double *part, CsScal *sc, ResBarrier *bar)
{
    constexpr int NC = Op::kNC;
    __shared__ double sh[kResThreads / 32];
    __shared__ df s_coef;
    __shared__ int s_ok, s_stop;
    unsigned long long target = 0;
    const int node = blockIdx.x * kResThreads + threadIdx.x;
    const bool in = node < N;
    bool ok = true;
    // Sum over all threads in a fixed order; a barrier.  The sum is known to
    // thread 0 of every block, which calls then(sum): FP64 arithmetic takes a
    // whole warp 19 clocks an instruction here, so one thread forms the
    // step's scalars.
    auto grid_sum = [&](const CsDot<df> &acc, int slot, auto then) {
        const double t = acc.template block_total<kResThreads>(sh);
        double *mine = part + slot * gridDim.x;
        if (threadIdx.x == 0) mine[blockIdx.x] = t;
        ok = res_barrier(bar, target, &s_ok) && ok;
        if (threadIdx.x < 32) {
            double a = 0.0;
            for (int k = threadIdx.x; k < int(gridDim.x); k += 32) a += __ldcg(mine + k);
            a = warp_sum(a);
            if (threadIdx.x == 0) then(a);
        }
        __syncthreads();
    };
    double rr = 0.0, tol = -1.0;  // thread 0's
    df r[NC], d[NC];
    CsDot<df> acc{};
    if (in) {
        float v[NC];
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            const int64_t e = (int64_t)m * N + node;
            r[m] = d[m] = b[e];
            x[e] = make_float2(0.0f, 0.0f);
            p[e] = d[m];
            acc.add(r[m], r[m]);
            v[m] = cs_to_float(d[m]);
        }
        op.store_p32(node, v);
    }
    grid_sum(acc, 0, [&](double v) {
        rr = v;
        tol = rel_tol > 0.0 ? rel_tol * sqrt(v) : -1.0;
    });
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
                pq_acc.add(d[m], q[m]);
            }
        }
        grid_sum(pq_acc, 1, [&](double pq) {
            s_stop = rr == 0.0 || pq == 0.0 || (tol >= 0.0 && sqrt(rr) <= tol);
            s_coef = df_from_double(rr / pq);
        });
        if (!ok || s_stop) break;
        const df al = s_coef, nal = df_neg(al);
        CsDot<df> rr_acc{};
        if (in) {
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                const int64_t e = (int64_t)m * N + node;
                x[e] = df_axpy(x[e], al, d[m]);
                r[m] = df_axpy(r[m], nal, q[m]);
                rr_acc.add(r[m], r[m]);
            }
        }
        grid_sum(rr_acc, 0, [&](double v) {
            s_coef = df_from_double(v / rr);
            rr = v;
        });
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
    const int64_t need = (N + kResThreads - 1) / kResThreads;
    if (need > most) return MPI_OK;
    int grid = (int)std::min(most, std::max(need, work * 32 / kResThreads));
    Scratch scr(st);
    const size_t vb = sizeof(float2) * Op::kNC * N;
    const size_t o_p = scr.reserve(vb), o_l = scr.reserve(vb), o_part = scr.reserve(sizeof(double) * 2 * grid),
                 o_bar = scr.reserve(sizeof(ResBarrier));
    MPI_TRY(scr.allocate());
    float2 *p = scr.at<float2>(o_p), *l1 = scr.at<float2>(o_l);
    double *part = scr.at<double>(o_part), rel_tol = o.rel_tol;
    ResBarrier *bar = scr.at<ResBarrier>(o_bar);
    int n = (int)N, max_iter = o.max_iter;
    Op arg = op;
    MPI_TRY_CUDA(cudaMemsetAsync(bar, 0, sizeof(ResBarrier), st));
    void *args[] = {&arg, &n, &b, &x, &p, &l1, &rel_tol, &max_iter, &part, &sc, &bar};
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
