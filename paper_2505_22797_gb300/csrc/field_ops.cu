// Gridded FP32 pair operators.
//
// A c at a sample is p^T Phi(r_t) W_t with the symmetric 2x2 field
//   Phi(r) = sum_x c_x K(beta G (x - r)),   W = beta G v,
// three convolutions of the image with the entries of K.  K is analytic in a
// strip of half-width pi around real arguments (coth has its poles at
// multiples of i pi), so Phi's spectrum falls off as exp(-pi |k|) per unit of
// z = |beta G r|: modes |k| <= 6.5 determine it to 1e-8.  The direct sums
// evaluate all N T pairs; here one application is
//   1. the image's DFT on the box of Q voxels per axis (zero padded, so the
//      circular convolution is the linear one on every used offset),
//   2. per entry of K: times the kernel's spectrum, inverse DFT on P nodes,
//   3. at each sample an 8 x 8-point Kaiser-Bessel interpolation (the
//      non-equispaced FFT's window, beta = 2.7 x 8, node pitch <= 0.43; its
//      transform is divided out of the kernel's spectrum): 1.3e-9 relative
//      error on dense images, 4e-9 on single voxels,
// O(N log N + 64 T) instead of O(N T).  A^T is the exact transpose (spread to
// the nodes, DFT, the same spectrum, inverse DFT at the voxels).  The sampled kernel is closed
// periodically by a smooth cut-off outside the offsets in use, so it has no
// step whose spectrum the division could amplify.
//
// Rounding: FP32 transforms leave errors of about one rounding of the
// largest modes, which for images are the few lowest ones.  So the modes |kx|, |ky| <
// kFieldLow are carried in pairs of floats from the image (or the nodes) to
// the nodes (or the voxels); one rounding of the columns between the two axes
// alone left 5e-9 in the lowest modes, which the CG of a solve turned into 2e-6
// of the image (now 4e-7, the direct sums' own error 1.7e-6); the kernel is sampled with correctly rounded functions, and
// the interpolation's outer sum and the product with W are carried in pairs.
//
// Samples beyond the node window (more than 12 z units outside the voxels)
// are summed directly by blocks of their own beside the interpolation and the
// spreading, in the pair kernels' form: there every pair of a diagonal G is in
// the asymptotic range.
#include <algorithm>
#include <climits>
#include <cmath>

#include "field_ops.cuh"
#include "grid_common.cuh"
#include "langevin.cuh"
#include "pair_kernels.cuh"

namespace mpi {

namespace {

constexpr int kWin = 8;              // interpolation points per axis
constexpr double kKbBeta = 21.6;     // Kaiser-Bessel parameter
constexpr double kKbI0 = 207500183.76013563;  // I0(kKbBeta)
constexpr double kPitch = 0.43;      // largest node pitch in z units
constexpr double kModeMax = 6.5;     // modes kept, radians per z unit
constexpr double kMargin = 12.2;     // window beyond the outermost voxel's edge, z units
constexpr double kCutScale = 1.45;   // width of the kernel's cut-off, z units
constexpr double kCutArg = 4.2;      // erfc(4.2)/2 = 1.4e-9: the cut-off acts beyond the used offsets
constexpr int kFieldMaxN = 4096;     // largest transform
constexpr int64_t kFieldMaxT = (int64_t)1 << 26;  // 112 bytes of scratch per sample
constexpr int kLowY = 2 * kFieldLow - 1;

constexpr int kTile = 16;                       // nodes per tile edge
constexpr int kPatch = kTile + kWin - 1;        // a tile's stencils reach 23 x 23 nodes
// Pitch of a patch row: the four rows that a warp updates together, two rows
// apart, start 0, 24, 16, 8 banks in.
constexpr int kPatchPitch = 28;
constexpr int kPatchSize = kPatch * kPatch;
constexpr int kFieldUnit = 224;                 // samples per spreading unit
constexpr int kSpreadThreads = 384;             // warp = (half of the unit, entry of K, row parity)
constexpr int kSpreadPerSm = 3;                 // blocks per SM (registers and shared memory)
constexpr int kRunMin = 128, kRunMax = 512;     // samples per run at least, runs at most
constexpr int kInterpThreads = 256;
// Outside sums of A^T: a thread takes kOutRows voxels of one column.
constexpr int kOutThreads = kSpreadThreads;
constexpr int kOutRows = 4;
// Outside sums of A: kFwdS samples per thread.
constexpr int kOutStage = kFieldMaxN / 2;       // voxels at a time in shared memory, a row at least (n < Q/2)
constexpr int kOutFold = 128;                   // columns summed plainly before a compensated add
constexpr int kOutPerSm = 768;                  // their threads per SM (four blocks at most)
constexpr int kOutRounds = 3;                   // units per such block at most, if a unit is not all rows

// Kaiser-Bessel window I0(beta sqrt(1 - (x/4)^2))/I0(beta) at x = f + 3 - a
// for the stencil's points a = 0..3 as polynomials in t = f - 1/2
// (interpolation at Chebyshev nodes, error 1e-10); point 7 - a takes -t.
__constant__ float kKb[4][11] = {
    {2.094581274e-5f, -0.0001943944819f, 0.0007884017967f, -0.001837328005f, 0.002709326105f, -0.002596430644f,
     0.001550771254f, -0.0004467888186f, -7.938607108e-5f, 0.0001165451474f, -3.114197027e-5f},
    {0.009922455796f, -0.0416071335f, 0.07374687558f, -0.0687373978f, 0.03111775652f, 0.0003281534653f,
     -0.007699716889f, 0.003092077999f, 0.0002645081479f, -0.0004992794498f, 8.127822694e-5f},
    {0.2148323554f, -0.457409045f, 0.3101820902f, 0.01196447209f, -0.1096105266f, 0.03469018205f, 0.01382287955f,
     -0.0091916326f, -0.000403235075f, 0.001190508892f, -0.0001062250978f},
    {0.8475298278f, -0.562987389f, -0.3847173893f, 0.3206552203f, 0.07578343971f, -0.08754925482f,
     -0.007671164434f, 0.01525333744f, 0.0002094549709f, -0.001796536138f, 5.123070011e-5f}};

// --- device helpers ---------------------------------------------------------

__device__ __forceinline__ float2 f2c(V2<float> a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ V2<float> v2(float2 a) { return V2<float>{a.x, a.y}; }

// sum += a b for FP32 a, b with the product's rounding error kept.
__device__ __forceinline__ void f2_fma(F2Sum &s, float a, float b)
{
    const float p = __fmul_rn(a, b);
    s.add(p);
    s.lo = __fadd_rn(s.lo, __fmaf_rn(a, b, -p));
}
__device__ __forceinline__ F2Sum f2_shfl_xor(F2Sum v, int o)
{
    F2Sum t;
    t.hi = __shfl_xor_sync(0xffffffffu, v.hi, o);
    t.lo = __shfl_xor_sync(0xffffffffu, v.lo, o);
    return t;
}
__device__ __forceinline__ F2Sum f2_warp(F2Sum v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v.add(f2_shfl_xor(v, o));
    return v;
}
struct SampleRec {
    bool in;
    float fx, fy;   // inside: fractions; outside: beta G r
    int ix, iy;     // first stencil node (window-relative)
    df Wx, Wy;      // beta G v
};

// Window-relative node coordinate of a position: pair r sc + of.
__device__ __forceinline__ bool node_coord(const FieldAxis &a, float r, int &i, float &f)
{
    df x = df_mul(make_float2(a.sc[0], a.sc[1]), make_float2(r, 0.0f));
    x = df_add(x, make_float2(a.of[0], a.of[1]));
    if (!(x.x >= a.xlo && x.x <= a.xhi)) return false;  // also NaN
    const float fl = floorf(x.x);
    float fr = (x.x - fl) + x.y;
    int k = int(fl);
    if (fr < 0.0f) { fr += 1.0f; k -= 1; }
    if (fr >= 1.0f) { fr -= 1.0f; k += 1; }
    i = k - (kWin / 2 - 1);
    f = fr;
    return true;
}

// B (a, b)^T for one row of beta G, as a pair.
__device__ __forceinline__ df row_times(const float (&B0)[2], const float (&B1)[2], float a, float b, bool diag_first,
                                        bool diag_second)
{
    const df u = df_mul(make_float2(B0[0], B0[1]), make_float2(a, 0.0f));
    const df w = df_mul(make_float2(B1[0], B1[1]), make_float2(b, 0.0f));
    if (diag_first) return u;
    if (diag_second) return w;
    return df_add(u, w);
}

__device__ __forceinline__ SampleRec make_sample(const FieldDev &d, const float *__restrict__ rp, const float *__restrict__ vp,
                                                 int64_t t)
{
    const float2 r = make_float2(rp[2 * t], rp[2 * t + 1]), v = make_float2(vp[2 * t], vp[2 * t + 1]);
    SampleRec q;
    const bool bx = node_coord(d.x, r.x, q.ix, q.fx);
    const bool by = node_coord(d.y, r.y, q.iy, q.fy);
    q.in = bx && by;
    const bool dg = d.diag != 0;
    q.Wx = row_times(d.B[0], d.B[1], v.x, v.y, dg, false);
    q.Wy = row_times(d.B[2], d.B[3], v.x, v.y, false, dg);
    if (!q.in) {
        const df X = row_times(d.B[0], d.B[1], r.x, r.y, dg, false);
        const df Y = row_times(d.B[2], d.B[3], r.x, r.y, false, dg);
        q.fx = X.x;
        q.fy = Y.x;
        q.ix = q.iy = 0;
    }
    return q;
}

// --- tables -----------------------------------------------------------------

__device__ float2 table_entry(int n, int t)
{
    double s, c;
    sincospi(-2.0 * double(t) / double(n), &s, &c);
    return make_float2(float(c), float(s));
}

// 1 / (the window's transform at mode k of P nodes).
__device__ double window_inv(int k, int P)
{
    const double h = kWin * 3.14159265358979323846 * double(k) / double(P);
    const double s = sqrt(kKbBeta * kKbBeta - h * h);
    return s * kKbI0 / (kWin * 0.5 * (exp(s) - exp(-s)));
}

// Outside samples (unordered plans) and, per out_samples of them, the row runs done.
__host__ __device__ __forceinline__ int out_counters(const FieldDev &d)
{
    return 1 + int((d.T + d.out_samples - 1) / d.out_samples);
}

// Entry t of the tables laid end to end.
__device__ void fill_table(const FieldDev &d, int t)
{
    if (t < d.x.P) { d.b.twPx[t] = table_entry(d.x.P, t); return; }
    t -= d.x.P;
    if (t < d.y.P) { d.b.twPy[t] = table_entry(d.y.P, t); return; }
    t -= d.y.P;
    if (t < d.x.Q) { d.b.twQx[t] = table_entry(d.x.Q, t); return; }
    t -= d.x.Q;
    if (t < d.y.Q) { d.b.twQy[t] = table_entry(d.y.Q, t); return; }
    t -= d.y.Q;
    if (t <= d.x.J) { d.b.iphx[t] = window_inv(t, d.x.P); return; }
    t -= d.x.J + 1;
    if (t <= d.y.J) { d.b.iphy[t] = window_inv(t, d.y.P) * d.scale; return; }
    t -= d.y.J + 1;
    if (t < d.x.n) {
        d.b.xcol[t] = V2<float>{float(d.X0[0] + t * d.cx[0]), float(d.X0[1] + t * d.cx[1])};
        return;
    }
    t -= d.x.n;
    if (t < d.y.n) {
        d.b.yrow[t] = V2<float>{float(d.Y0[0] + t * d.cy[0]), float(d.Y0[1] + t * d.cy[1])};
        return;
    }
    t -= d.y.n;
    if (d.b.ocount && t < out_counters(d)) d.b.ocount[t] = 0;
}
int table_entries(const FieldDev &d)
{
    return d.x.P + d.y.P + d.x.Q + d.y.Q + d.x.J + 1 + d.y.J + 1 + d.x.n + d.y.n + (d.b.ocount ? out_counters(d) : 0);
}

// --- ordering the samples by tile ----------------------------------------------
// A stable counting sort: each warp of k_field_setup / k_field_place owns a
// run of consecutive samples, hist[tile][warp] their counts, whose prefix
// sums place them in sample order within the tile.

__device__ __forceinline__ int sample_tile(const FieldDev &d, const SampleRec &q)
{
    return q.in ? (q.iy / kTile) * d.tx + q.ix / kTile : d.tx * d.ty;
}

// Tile of every sample of run `run` and the run's tile counts, by one warp;
// cnt: tx ty + 1 ints of shared memory.
__device__ void bin_run(const FieldDev &d, int run, int *cnt, const float *__restrict__ r, const float *__restrict__ v)
{
    const int nt = d.tx * d.ty + 1, lane = threadIdx.x & 31;
    for (int k = lane; k < nt; k += 32) cnt[k] = 0;
    __syncwarp();
    const int64_t t0 = int64_t(run) * d.run_len;
#pragma unroll 2
    for (int u = 0; u < d.run_len; u += 32) {
        const int64_t t = t0 + u + lane;
        int k = -1;
        if (t < d.T) {
            k = sample_tile(d, make_sample(d, r, v, t));
            d.b.key[t] = k;
        }
        const unsigned peers = __match_any_sync(0xffffffffu, k);
        if (k >= 0 && lane == __ffs(peers) - 1) cnt[k] += __popc(peers);
        __syncwarp();
    }
    for (int k = lane; k < nt; k += 32) d.b.hist[int64_t(k) * d.n_run + run] = cnt[k];
}

// pos[tile][run] = the tile's samples in earlier runs, tcnt[tile] its total;
// one warp.
__device__ void scan_tile(const FieldDev &d, int tile)
{
    const int lane = threadIdx.x & 31;
    const int *h = d.b.hist + int64_t(tile) * d.n_run;
    int *o = d.b.pos + int64_t(tile) * d.n_run;
    int base = 0;
    for (int q0 = 0; q0 < d.n_run; q0 += 32) {
        const int q = q0 + lane;
        const int c = q < d.n_run ? h[q] : 0;
        int x = c;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, s);
            if (lane >= s) x += y;
        }
        if (q < d.n_run) o[q] = base + x - c;
        base += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) d.b.tcnt[tile] = base;
}

// Exclusive scan over the block's threads; s_w: 32 ints.
__device__ __forceinline__ int scan_block(int v, int *s_w, int *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < nw ? s_w[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        s_w[lane] = w;
    }
    __syncthreads();
    *total = s_w[31];
    const int res = (warp ? s_w[warp - 1] : 0) + x - v;
    __syncthreads();
    return res;
}

// The tiles' first positions, the units (at most kFieldUnit samples of one
// tile) per tile and each unit's tile, by one block.
__device__ void make_units(const FieldDev &d, int *s_w)
{
    const int nt = d.tx * d.ty;
    const int per = (nt + int(blockDim.x)) / int(blockDim.x);  // the outside bin nt included
    const int k0 = min(nt + 1, int(threadIdx.x) * per), k1 = min(nt + 1, k0 + per);
    int s = 0, u = 0;
    for (int k = k0; k < k1; ++k) {
        const int c = d.b.tcnt[k];
        s += c;
        if (k < nt) u += (c + kFieldUnit - 1) / kFieldUnit;
    }
    int total;
    s = scan_block(s, s_w, &total);
    u = scan_block(u, s_w, &total);
    for (int k = k0; k < k1; ++k) {
        d.b.toff[k] = s;
        d.b.uoff[k] = u;
        const int c = d.b.tcnt[k];
        s += c;
        if (k < nt)
            for (int e = 0; e < (c + kFieldUnit - 1) / kFieldUnit; ++e) d.b.unit_tile[u++] = k;
    }
}

__device__ __forceinline__ float4 operand(const FieldDev &d, const float *__restrict__ s, int64_t t, const SampleRec &q)
{
    float ux = 0.0f, uy = 0.0f;
    for (int k = 0; k < d.n_ch; ++k) {
        const float sv = s[int64_t(k) * d.T + t];
        ux += sv * d.p[2 * k];
        uy += sv * d.p[2 * k + 1];
    }
    const float Wx = q.Wx.x, Wy = q.Wy.x;
    return q.in ? make_float4(ux * Wx, fmaf(ux, Wy, uy * Wx), uy * Wy, 0.0f) : make_float4(ux, uy, 0.0f, 0.0f);
}

// Places each run's samples: position = the tile's first + its samples in
// earlier runs + the rank within the run.
__global__ void __launch_bounds__(128) k_field_place(const __grid_constant__ FieldDev d, const float *r,
                                                     const float *v, const float *s)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nt = d.tx * d.ty + 1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int run = blockIdx.x * (blockDim.x >> 5) + warp;
    if (run >= d.n_run) return;
    int *next = reinterpret_cast<int *>(smem_raw) + warp * nt;
    for (int k = lane; k < nt; k += 32) next[k] = -1;
    __syncwarp();
    const int64_t t0 = int64_t(run) * d.run_len;
    for (int u = 0; u < d.run_len; u += 32) {
        const int64_t t = t0 + u + lane;
        const bool valid = t < d.T;
        const int k = valid ? d.b.key[t] : -1;
        SampleRec q{};
        if (valid) q = make_sample(d, r, v, t);
        const unsigned peers = __match_any_sync(0xffffffffu, k);
        const int lead = __ffs(peers) - 1;
        int first = 0;
        if (valid && lane == lead) {
            first = next[k];
            if (first < 0) first = d.b.toff[k] + d.b.pos[int64_t(k) * d.n_run + run];
            next[k] = first + __popc(peers);
        }
        first = __shfl_sync(0xffffffffu, first, lead);
        if (valid) {
            const int p = first + __popc(peers & ((1u << lane) - 1u));
            d.b.list[p] = int(t);
            d.b.rec[p] = make_float4(q.fx, q.fy, __int_as_float(q.in ? (q.iy << 16) | q.ix : -1), 0.0f);
            d.b.wv[p] = make_float4(q.Wx.x, q.Wy.x, q.Wx.y, q.Wy.y);
            if (s) d.b.q4[p] = operand(d, s, t, q);
        }
        __syncwarp();
    }
}

__global__ void __launch_bounds__(256) k_field_load(const __grid_constant__ FieldDev d, const float *s)
{
    chain_wait();
    const int64_t p = int64_t(blockIdx.x) * 256 + threadIdx.x;
    if (p >= d.T) return;
    const int64_t t = d.b.list[p];
    d.b.sd[p] = make_float2(s[t], d.n_ch > 1 ? s[d.T + t] : 0.0f);
}

// Tables (32 entries per block: FP64 functions, spread over the SMs) and, in
// the blocks behind them, the samples' tiles.
__global__ void __launch_bounds__(128) k_field_setup(const __grid_constant__ FieldDev d, int n_table, const float *r,
                                                     const float *v)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (int(blockIdx.x) < n_table) {
        if (threadIdx.x < 32) fill_table(d, blockIdx.x * 32 + threadIdx.x);
        return;
    }
    const int warp = threadIdx.x >> 5;
    const int run = (blockIdx.x - n_table) * (blockDim.x >> 5) + warp;
    if (run < d.n_run) bin_run(d, run, reinterpret_cast<int *>(smem_raw) + warp * (d.tx * d.ty + 1), r, v);
}

// --- the kernel's spectrum ----------------------------------------------------

// Weight of the kernel at an offset of `off` nodes: smooth, exactly 1 on the
// offsets in use, and 0 where a periodic image of those lies.
__device__ __forceinline__ float cut_weight(const FieldAxis &a, float off)
{
    const float e = (fabsf(off) - 0.5f * float(a.P)) * a.cut_inv;
    return e < -float(kCutArg) ? 1.0f : (e > float(kCutArg) ? 0.0f : 0.5f * erfcf(e));
}

// (a, d) by the closed form with correctly rounded functions
// (the approximate ones' common bias would scale every sum; a spectrum needs
// only some 1e5 evaluations).
__device__ __forceinline__ void kernel_scalars(float u, float &f1, float &f2)
{
    if (u < Lang<float>::near_u) {
        Lang<float>::ad_near(u, f1, f2);
        return;
    }
    const float z = sqrtf(u), iz = __frcp_rn(z), iz2 = __frcp_rn(u);
    const float q = expf(-2.0f * z), rr = __frcp_rn(1.0f - q);
    const float coth = (1.0f + q) * rr, csch2 = 4.0f * q * rr * rr;
    f1 = fmaf(coth, iz, -iz2);
    f2 = ((iz2 - csch2) - f1) * iz2;
}

// The spectra A, B of two real sequences from that of a + i b at k and -k.
__device__ __forceinline__ void unpack2(V2<float> u, V2<float> w, float2 &A, float2 &B)
{
    A = make_float2(0.5f * (u.x + w.x), 0.5f * (u.y - w.y));
    B = make_float2(0.5f * (u.y + w.y), 0.5f * (w.x - u.x));
}

// Modes -(kFieldLow - 1) .. kFieldLow - 1 of the block's three sequences of
// length P (before their transform) by direct sums.  In a transform a low mode
// meets few twiddle factors, whose rounding errors (3e-8) are then common to
// all rows and scale every result; in the sum they average out.
__device__ __forceinline__ void low_rows(const V2<float> *a, int P, const float2 *__restrict__ tw, V2<float> (*low)[3])
{
    const int nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    for (int q = threadIdx.x >> 5; q < kLowY; q += nw) {
        const int k = q - (kFieldLow - 1);
        const int mm = k < 0 ? P + k : k;
        int at = (lane * mm) % P;
        const int step = (32 * mm) % P;
        V2<float> s[3] = {};
#pragma unroll 4
        for (int e = lane; e < P; e += 32) {
            const float2 w = tw[at];
            at += step;
            at -= at >= P ? P : 0;
            const V2<float> *z = a + smem_fft_pad(e) * 3;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                s[c].x = fmaf(z[c].x, w.x, fmaf(-z[c].y, w.y, s[c].x));
                s[c].y = fmaf(z[c].x, w.y, fmaf(z[c].y, w.x, s[c].y));
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            s[c].x = warp_sum(s[c].x);
            s[c].y = warp_sum(s[c].y);
            if (lane == 0) low[q][c] = s[c];
        }
    }
}

// Stores the half spectra of two rows' entries from the three transformed
// sequences (xx + i xy of each row, yy of both): planes [3][rows][J + 1].
__device__ __forceinline__ void store_rows(const V2<float> *z, int P, int J1, int l0, int rows, const V2<float> (*low)[3],
                                           float2 *out)
{
    const int64_t plane = int64_t(rows) * J1;
    const bool two = l0 + 1 < rows;
    float2 *o = out + int64_t(l0) * J1;
    for (int k = threadIdx.x; k < J1; k += blockDim.x) {
        const V2<float> *u = z + smem_fft_pad(k) * 3, *w = z + smem_fft_pad(k ? P - k : 0) * 3;
        if (k < kFieldLow) u = low[kFieldLow - 1 + k], w = low[kFieldLow - 1 - k];
        float2 A, B;
        unpack2(u[0], w[0], A, B);
        o[k] = A;
        o[plane + k] = B;
        if (two) {
            unpack2(u[1], w[1], A, B);
            o[J1 + k] = A;
            o[plane + J1 + k] = B;
        }
        unpack2(u[2], w[2], A, B);
        o[2 * plane + k] = A;
        if (two) o[2 * plane + J1 + k] = B;
    }
}

// Rows l0, l0 + 1 (l <= Py/2) of the sampled kernel's entries and their half
// spectra.
__device__ void kernel_rows(const FieldDev &d, int l0, unsigned char *smem)
{
    const int P = d.x.P;
    V2<float> *a = reinterpret_cast<V2<float> *>(smem);
    V2<float> *b = a + (smem_fft_pad(P - 1) + 1) * 3;
    const int half = d.y.P / 2;
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const int ox = i > P / 2 ? i - P : i;
        float e[2][3];
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            const int l = l0 + rr;
            float xx = 0.0f, xy = 0.0f, yy = 0.0f;
            for (int im = 0; im < 4; ++im) {
                const float nx = float((im & 1) ? (ox >= 0 ? ox - P : ox + P) : ox), ny = float((im & 2) ? l - d.y.P : l);
                const float w = cut_weight(d.x, nx) * cut_weight(d.y, ny);
                if (w == 0.0f || l > half) continue;
                const float y0 = fmaf(nx, d.hx[0][0], fmaf(ny, d.hy[0][0], fmaf(nx, d.hx[0][1], ny * d.hy[0][1])));
                const float y1 = fmaf(ny, d.hy[1][0], fmaf(nx, d.hx[1][0], fmaf(nx, d.hx[1][1], ny * d.hy[1][1])));
                float f1, f2;
                kernel_scalars(fmaf(y0, y0, y1 * y1), f1, f2);
                xx += w * fmaf(f2 * y0, y0, f1);
                xy += w * (f2 * y0 * y1);
                yy += w * fmaf(f2 * y1, y1, f1);
            }
            e[rr][0] = xx;
            e[rr][1] = xy;
            e[rr][2] = yy;
        }
        V2<float> *o = a + smem_fft_pad(i) * 3;
        o[0] = V2<float>{e[0][0], e[0][1]};
        o[1] = V2<float>{e[1][0], e[1][1]};
        o[2] = V2<float>{e[0][2], e[1][2]};
    }
    __shared__ V2<float> s_low[kLowY][3];
    __syncthreads();
    low_rows(a, P, d.b.twPx, s_low);
    __syncthreads();
    const V2<float> *z = smem_fft<3, -1, float>(a, b, d.fPx, reinterpret_cast<const V2<float> *>(d.b.twPx));
    store_rows(z, P, d.x.J + 1, l0, half + 1, s_low, d.b.KR);
}

// The modes +-m of a sequence (get(e): (re, im) hi and lo, e < n_e) of period
// n by one warp: four terms in FP32, then in pairs (the rounding errors of
// many small sums average out, those of a few large ones do not).  Valid in
// every lane.
struct LowPair {
    F2Sum rp, ip, rm, im;  // mode m, mode -m
};
template <typename F>
__device__ __forceinline__ LowPair low_modes(int n_e, int n, int m, const float2 *__restrict__ tw, F get)
{
    const int lane = threadIdx.x & 31;
    int at = (lane * m) % n;
    const int step = (32 * m) % n;
    F2Sum xc{}, xd{}, yc{}, yd{};
#pragma unroll 1
    for (int e0 = lane; e0 < n_e; e0 += 128) {
        float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f), l = s;  // x c, x d, y c, y d of four terms
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = e0 + 32 * u;
            const float2 w = tw[at];
            at += step;
            at -= at >= n ? n : 0;
            if (e < n_e) {
                const float4 q = get(e);
                s.x = fmaf(q.x, w.x, s.x);
                s.y = fmaf(q.x, w.y, s.y);
                s.z = fmaf(q.y, w.x, s.z);
                s.w = fmaf(q.y, w.y, s.w);
                l.x = fmaf(q.z, w.x, l.x);
                l.y = fmaf(q.z, w.y, l.y);
                l.z = fmaf(q.w, w.x, l.z);
                l.w = fmaf(q.w, w.y, l.w);
            }
        }
        xc.add(s.x); xc.lo += l.x;
        xd.add(s.y); xd.lo += l.y;
        yc.add(s.z); yc.lo += l.z;
        yd.add(s.w); yd.lo += l.w;
    }
    xc = f2_warp(xc);
    xd = f2_warp(xd);
    yc = f2_warp(yc);
    yd = f2_warp(yd);
    LowPair r{xc, yc, xc, yc};
    r.rm.add(yd);
    r.ip.add(xd);
    yd.hi = -yd.hi, yd.lo = -yd.lo;
    xd.hi = -xd.hi, xd.lo = -xd.lo;
    r.rp.add(yd);
    r.im.add(xd);
    return r;
}

// The coefficients of a column's lowest modes, mode sums times the kernel's
// (pairs): out[ky + kFieldLow - 1].
template <typename F>
__device__ __forceinline__ void low_coefs(int n_e, int n, int ky, const float2 *__restrict__ tw, const float2 *__restrict__ K,
                                          float4 *out, F get)
{
    const LowPair s = low_modes(n_e, n, ky, tw, get);
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int sg = 0; sg < 2; ++sg) {
            const int q = kFieldLow - 1 + (sg ? -ky : ky);
            const F2Sum re = sg ? s.rm : s.rp, im = sg ? s.im : s.ip;
            const df r = df_mul(df_fast_two_sum(re.hi, re.lo), K[q]), i = df_mul(df_fast_two_sum(im.hi, im.lo), K[q]);
            out[q] = make_float4(r.x, i.x, r.y, i.y);
        }
    }
}

// Adds the lowest modes' part of element e: sum over ky of the pair
// coefficient co[ky] times exp(2 pi i ky e / n), as pairs.
__device__ __forceinline__ void low_add(const float4 *co, int e, int n, const float2 *__restrict__ tw, F2Sum &re, F2Sum &im)
{
    int at = 0;
#pragma unroll
    for (int k = 0; k < kFieldLow; ++k) {
        const float2 t = tw[at];  // exp(-2 pi i k e / n)
        at += e;
        at -= at >= n ? n : 0;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (k == 0 && s) continue;
            const float ty = s ? t.y : -t.y;
            const float4 v = co[kFieldLow - 1 + (s ? -k : k)];
            f2_fma(re, v.x, t.x);
            f2_fma(re, -v.y, ty);
            f2_fma(im, v.x, ty);
            f2_fma(im, v.y, t.x);
            re.lo += fmaf(v.z, t.x, -v.w * ty);
            im.lo += fmaf(v.z, ty, v.w * t.x);
        }
    }
}
// Columns of the kernel's spectrum: NC adjacent kx (group g) of entry m.  The
// spectrum of a real kernel that is even under (x, y) -> (-x, -y) is real;
// the rows l > Py/2 are the conjugates of rows Py - l.
template <int NC> __device__ void kernel_cols(const FieldDev &d, int g, int m, unsigned char *smem)
{
    const int P = d.y.P, J1 = d.x.J + 1, half = P / 2;
    V2<float> *a = reinterpret_cast<V2<float> *>(smem);
    V2<float> *b = a + (smem_fft_pad(P - 1) + 1) * NC;
    const int c = threadIdx.x % NC, j0 = threadIdx.x / NC, dj = blockDim.x / NC;
    const int kx = g * NC + c;
    const bool on = kx < J1;
    const float2 *KR = d.b.KR + int64_t(m) * (half + 1) * J1 + (on ? kx : 0);
#pragma unroll 4
    for (int l = j0; l < P; l += dj) {
        float2 q = KR[int64_t(l <= half ? l : P - l) * J1];
        if (l > half) q.y = -q.y;
        a[smem_fft_pad(l) * NC + c] = v2(on ? q : make_float2(0.0f, 0.0f));
    }
    __syncthreads();
    if (g * NC < kFieldLow) {
        const int nw = blockDim.x >> 5, w = threadIdx.x >> 5;
        for (int q = w; q < NC * kFieldLow; q += nw) {
            const int cc = q % NC, ky = q / NC, kk = g * NC + cc;
            if (kk >= kFieldLow) continue;
            const LowPair s = low_modes(P, P, ky, d.b.twPy, [&](int e) {
                const V2<float> z = a[smem_fft_pad(e) * NC + cc];
                return make_float4(z.x, z.y, 0.0f, 0.0f);
            });
            if ((threadIdx.x & 31) == 0) {
                const double f = d.b.iphx[kk] * d.b.iphy[ky];
                float2 *K = d.b.KL + (m * kFieldLow + kk) * kLowY + kFieldLow - 1;
                K[ky] = df_from_double(s.rp.value() * f);
                K[-ky] = df_from_double(s.rm.value() * f);
            }
        }
        __syncthreads();
    }
    const V2<float> *z = smem_fft<NC, -1, float>(a, b, d.fPy, reinterpret_cast<const V2<float> *>(d.b.twPy));
    const int J = d.y.J, JY = 2 * J + 1;
    const float fx = on ? float(d.b.iphx[kx]) : 0.0f;
    float *KH = d.b.KH + (int64_t(m) * d.n_grp + g) * JY * NC + c;
#pragma unroll 4
    for (int k = j0; k < JY; k += dj) {
        const int ky = k - J;
        KH[int64_t(k) * NC] = z[smem_fft_pad(ky < 0 ? ky + P : ky) * NC + c].x * (fx * float(d.b.iphy[abs(ky)]));
    }
}

// --- forward ------------------------------------------------------------------

// Half spectra of image rows j0, j0 + 1; the lowest modes in pairs.
template <typename CIN> __device__ void image_rows(const FieldDev &d, int j0, const CIN *__restrict__ c, unsigned char *smem)
{
    const int Q = d.x.Q, nx = d.x.n;
    V2<float> *a = reinterpret_cast<V2<float> *>(smem);
    V2<float> *b = a + smem_fft_pad(Q - 1) + 1;
    const bool two = j0 + 1 < d.y.n;
    const CIN *c0 = c + int64_t(j0) * nx, *c1 = c0 + (two ? nx : 0);
    for (int i = threadIdx.x; i < Q; i += blockDim.x) {
        V2<float> q{0.0f, 0.0f};
        if (i < nx) q = V2<float>{float(c0[i]), two ? float(c1[i]) : 0.0f};
        a[smem_fft_pad(i)] = q;
    }
    __syncthreads();
    const int nw = blockDim.x >> 5, w = threadIdx.x >> 5;
    for (int q = w; q < 2 * kFieldLow; q += nw) {
        const int kx = q >> 1, rr = q & 1;
        if (rr && !two) continue;
        const LowPair s = low_modes(nx, Q, kx, d.b.twQx, [&](int e) {
            const V2<float> z = a[smem_fft_pad(e)];
            return make_float4(rr ? z.y : z.x, 0.0f, 0.0f, 0.0f);
        });
        if ((threadIdx.x & 31) == 0) {
            const float2 r = df_fast_two_sum(s.rp.hi, s.rp.lo), i = df_fast_two_sum(s.ip.hi, s.ip.lo);
            d.b.CL[int64_t(j0 + rr) * kFieldLow + kx] = make_float4(r.x, i.x, r.y, i.y);
        }
    }
    __syncthreads();
    const V2<float> *z = smem_fft<1, -1, float>(a, b, d.fQx, reinterpret_cast<const V2<float> *>(d.b.twQx));
    const int H = Q / 2 + 1;
    float2 *o = d.b.CR + int64_t(j0) * H;
    for (int k = threadIdx.x; k < H; k += blockDim.x) {
        float2 A, B;
        unpack2(z[smem_fft_pad(k)], z[smem_fft_pad(k ? Q - k : 0)], A, B);
        o[k] = A;
        if (two) o[H + k] = B;
    }
}

template <typename CIN>
__global__ void __launch_bounds__(128) k_field_image(const __grid_constant__ FieldDev d, const CIN *c)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    image_rows(d, 2 * blockIdx.x, c, smem_raw);
}

// Appends the outside samples among kListPer per thread to olist, in any order
// (a sample's sum does not depend on its neighbours in the list).
constexpr int kListPer = 4;
__device__ void list_outside(const FieldDev &d, int64_t block, const float *__restrict__ r)
{
    const int lane = threadIdx.x & 31;
    const int64_t t0 = block * kListPer * blockDim.x + threadIdx.x;
    float x[kListPer], y[kListPer];
#pragma unroll
    for (int u = 0; u < kListPer; ++u) {
        const int64_t t = min(t0 + int64_t(u) * blockDim.x, d.T - 1);
        x[u] = r[2 * t];
        y[u] = r[2 * t + 1];
    }
#pragma unroll
    for (int u = 0; u < kListPer; ++u) {
        const int64_t t = t0 + int64_t(u) * blockDim.x;
        int k;
        float f;
        const bool bx = node_coord(d.x, x[u], k, f), by = node_coord(d.y, y[u], k, f);
        const bool out = t < d.T && !(bx && by);
        const unsigned mask = __ballot_sync(0xffffffffu, out);
        if (mask == 0) continue;
        int base = 0;
        if (lane == 0) base = atomicAdd(d.b.ocount, __popc(mask));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (out) d.b.olist[base + __popc(mask & ((1u << lane) - 1u))] = int(t);
    }
}

// The sampled kernel's rows and, behind them, what else needs only the
// tables: the image's rows (c) and the list of the outside samples, or the
// tiles' prefix sums.
__global__ void __launch_bounds__(512) k_field_rows(const __grid_constant__ FieldDev d, int n_kernel, const float *c,
                                                    const float *r)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = blockIdx.x;
    if (b < n_kernel) {
        kernel_rows(d, 2 * b, smem_raw);
    } else if (c) {
        const int k = b - n_kernel, n_image = (d.y.n + 1) / 2;
        if (k < n_image) image_rows(d, 2 * k, c, smem_raw);
        else list_outside(d, k - n_image, r);
    } else {
        const int tile = (b - n_kernel) * int(blockDim.x >> 5) + int(threadIdx.x >> 5);
        if (tile <= d.tx * d.ty) scan_tile(d, tile);
    }
}

// The kernel spectrum's columns and, in one more block, the units.
template <int NC>
__global__ void __launch_bounds__(512) k_field_kcols(const __grid_constant__ FieldDev d)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_w[32];
    const int g = blockIdx.x % d.n_grp, m = blockIdx.x / d.n_grp;
    if (m < 3) kernel_cols<NC>(d, g, m, smem_raw);
    else make_units(d, s_w);
}

// k modulo n (n >= 1, |k| < 2^16); mag = floor(2^32 / n) + 1.
__device__ __forceinline__ int fast_mod(int k, int n, unsigned mag, int lift)
{
    const unsigned u = unsigned(k + lift);  // lift: a multiple of n that makes it positive
    return int(u - __umulhi(u, mag) * unsigned(n));
}

enum { kInterpForward = 0, kInterpOrdered = 1 };

struct InterpArgs {
    const float *r, *v;   // unordered trajectory
    float *s;             // [n_ch][T]
    bool residual;        // ordered: the data minus A c
};

// One sample's outputs from its channels' sums o (pairs): s, or in an ordered
// plan the operand of A^T (residual: of the data minus the sums).
template <int MODE>
__device__ __forceinline__ void finish_sample(const FieldDev &d, const InterpArgs &A, int64_t t, const df (&o)[2],
                                              bool inside, float Wx, float Wy)
{
    if constexpr (MODE == kInterpForward) {
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (k < d.n_ch) A.s[int64_t(k) * d.T + t] = o[k].x + o[k].y;
    } else {
        const float2 data = A.residual ? d.b.sd[t] : make_float2(0.0f, 0.0f);
        float ux = 0.0f, uy = 0.0f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (k >= d.n_ch) break;
            const float sk = A.residual ? ((k ? data.y : data.x) - o[k].x) - o[k].y : o[k].x + o[k].y;
            ux += sk * d.p[2 * k];
            uy += sk * d.p[2 * k + 1];
        }
        d.b.q4[t] = inside ? make_float4(ux * Wx, fmaf(ux, Wy, uy * Wx), uy * Wy, 0.0f) : make_float4(ux, uy, 0.0f, 0.0f);
    }
}

// Columns [ib, ie) of one staged row for a general G: sa += c f1, (vx, vy) +=
// c f2 (y.W) y.  FAR: every pair is in the asymptotic range.
template <bool FAR>
__device__ __forceinline__ void outside_line(int ib, int ie, const V2<float> *__restrict__ xcol, const V2<float> *xc,
                                             const float (&ox)[kFwdS], const float (&oy)[kFwdS], const float (&Wx)[kFwdS],
                                             const float (&Wy)[kFwdS], float (&sa)[kFwdS], float (&vx)[kFwdS], float (&vy)[kFwdS])
{
#pragma unroll(FAR ? 4 : 2)
    for (int i = ib; i < ie; ++i) {
        const V2<float> x = xcol[i];
        const float c = xc[i].y;
#pragma unroll
        for (int s = 0; s < kFwdS; ++s) {
            const float yx = x.x + ox[s], yy = x.y + oy[s], u = fmx(yx, yx, yy * yy);
            float f1, f2;
            if constexpr (FAR) lang_vfar<float, false>(u, f1, f2);
            else lang_checked<float, false>(u, f1, f2);
            sa[s] = fmx(c, f1, sa[s]);
            const float f = c * f2 * fmx(yx, Wx[s], yy * Wy[s]);
            vx[s] = fmx(f, yx, vx[s]);
            vy[s] = fmx(f, yy, vy[s]);
        }
    }
}

// Sums O = sum_x c_x (f1 W + f2 (y.W) y) of the n_out outside samples, by the
// first out_blocks blocks of a launch: a unit is out_samples samples and a run
// of rows, a block takes every out_blocks-th; a sample's runs are added, in
// their order, by the block that ends the last of them.  Bound by the FP32 pipe
// as the pair sums, whose inner loop it is.  A at 128 x 128 / 65 536 samples, 50
// and 94 % of them outside: 0.39 and 0.55 ms (pair sums of all samples 0.48 ms;
// a block summing its samples one after another, as here before, 2.9 ms: bursts
// of outside samples lie in few blocks); 512 x 512, 84 %: 7.2 ms (6.8, 37.6).
template <int MODE, typename CIN>
__device__ __forceinline__ void outside_units(const FieldDev &d, const InterpArgs &A, const CIN *__restrict__ cin,
                                              int n_out, V2<float> *s_xc, int *s_last)
{
    const int first = int(d.T) - n_out;  // (of the ordered samples)
    const int per = kFwdS * blockDim.x;  // out_samples
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nx = d.x.n, ny = d.y.n, rs = kOutStage / nx;
    const int n_grp = (n_out + per - 1) / per;
    // rows per unit: of the lengths that give 1, 2, .. units per block the one
    // that ends first (each unit costs about a row more than its rows)
    int len = ny, best = INT_MAX;
    for (int q = 1; q <= kOutRounds; ++q) {
        const int want = min(ny, max(1, q * d.out_blocks / n_grp)), l = (ny + want - 1) / want;
        const int units = n_grp * ((ny + l - 1) / l), cost = (units + d.out_blocks - 1) / d.out_blocks * (l + 1);
        if (cost < best) best = cost, len = l;
    }
    const int runs = (ny + len - 1) / len;
#pragma unroll 1
    for (int u = blockIdx.x; u < n_grp * runs; u += d.out_blocks) {
        const int g = u / runs, run = u % runs;
        const int j0 = run * len, j1 = min(ny, j0 + len);
        const int k0 = g * per + warp * (32 * kFwdS) + lane;  // the thread's samples: k0 + 32 s
        const bool any = k0 - lane < n_out;                            // of the warp
        float Rx[kFwdS], Ry[kFwdS], Wx[kFwdS], Wy[kFwdS];
        float Sa[kFwdS], Vx[kFwdS], Vy[kFwdS], cSa[kFwdS], cVx[kFwdS], cVy[kFwdS];
#pragma unroll
        for (int s = 0; s < kFwdS; ++s) {
            const int k = min(k0 + 32 * s, n_out - 1);
            if constexpr (MODE == kInterpOrdered) {
                const float4 rc = d.b.rec[first + k], w = d.b.wv[first + k];
                Rx[s] = rc.x, Ry[s] = rc.y, Wx[s] = w.x, Wy[s] = w.y;
            } else {
                const SampleRec q = make_sample(d, A.r, A.v, d.b.olist[k]);
                Rx[s] = q.fx, Ry[s] = q.fy, Wx[s] = q.Wx.x, Wy[s] = q.Wy.x;
            }
            Sa[s] = Vx[s] = Vy[s] = cSa[s] = cVx[s] = cVy[s] = 0.0f;
        }
#pragma unroll 1
        for (int j = j0; j < j1; j += rs) {
            const int nr = min(rs, j1 - j);
            __syncthreads();
            for (int e = threadIdx.x; e < nr * nx; e += blockDim.x)
                s_xc[e] = V2<float>{d.b.xcol[e % nx].x, float(cin[int64_t(j) * nx + e])};
            __syncthreads();
            if (!any) continue;
#pragma unroll 1
            for (int r = 0; r < nr; ++r) {
                const V2<float> yr = d.b.yrow[j + r];
                const V2<float> *xc = s_xc + r * nx;
                float ox[kFwdS], oy[kFwdS], yy2[kFwdS], yyW[kFwdS];
#pragma unroll
                for (int s = 0; s < kFwdS; ++s) {
                    ox[s] = yr.x - Rx[s];
                    oy[s] = yr.y - Ry[s];
                    yy2[s] = oy[s] * oy[s];
                    yyW[s] = oy[s] * Wy[s];
                }
#pragma unroll 1
                for (int ib = 0; ib < nx; ib += kOutFold) {
                    const int ie = min(nx, ib + kOutFold);
                    float sa[kFwdS], vx[kFwdS], fy[kFwdS];
#pragma unroll
                    for (int s = 0; s < kFwdS; ++s) sa[s] = vx[s] = fy[s] = 0.0f;
                    if (d.diag) {
                        fwd_row_vfar<float>(ib, ie, xc, Rx, yy2, Wx, yyW, sa, vx, fy);
#pragma unroll
                        for (int s = 0; s < kFwdS; ++s) fy[s] *= oy[s];
                    } else {
                        // the columns' positions lie on a line: the closest
                        // point of its segment decides the form (for the
                        // warp, so only where its samples are always the
                        // same ones: not in the unordered list)
                        const V2<float> b0 = d.b.xcol[ib], b1 = d.b.xcol[ie - 1];
                        const float ex = b1.x - b0.x, ey = b1.y - b0.y, ee = fmx(ex, ex, ey * ey);
                        bool far = true;
#pragma unroll
                        for (int s = 0; s < kFwdS; ++s) {
                            const float ax = b0.x + ox[s], ay = b0.y + oy[s];
                            const float w = ee > 0.0f ? __saturatef(-fmx(ax, ex, ay * ey) / ee) : 0.0f;
                            const float px = fmx(w, ex, ax), py = fmx(w, ey, ay);
                            far = far && fmx(px, px, py * py) >= 1.02f * vfar_threshold<float, false>();
                        }
                        if (MODE == kInterpOrdered && __all_sync(0xffffffffu, far))
                            outside_line<true>(ib, ie, d.b.xcol, xc, ox, oy, Wx, Wy, sa, vx, fy);
                        else
                            outside_line<false>(ib, ie, d.b.xcol, xc, ox, oy, Wx, Wy, sa, vx, fy);
                    }
#pragma unroll
                    for (int s = 0; s < kFwdS; ++s) {
                        kahan_add(Sa[s], cSa[s], sa[s]);
                        kahan_add(Vx[s], cVx[s], vx[s]);
                        kahan_add(Vy[s], cVy[s], fy[s]);
                    }
                }
            }
        }
#pragma unroll
        for (int s = 0; s < kFwdS; ++s) {
            const int k = k0 + 32 * s;
            if (k >= n_out) continue;
            const float Ox = fmx(Sa[s], Wx[s], Vx[s]), Oy = fmx(Sa[s], Wy[s], Vy[s]);
            df o[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) o[c] = make_float2(fmx(d.p[2 * c], Ox, d.p[2 * c + 1] * Oy), 0.0f);
            if (runs > 1) {
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    if (c < d.n_ch) d.b.fpart[(int64_t(run) * d.n_ch + c) * n_out + k] = o[c].x;
            } else {
                finish_sample<MODE>(d, A, MODE == kInterpOrdered ? first + k : d.b.olist[k], o, false, 0.0f, 0.0f);
            }
        }
        if (runs == 1) continue;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) *s_last = atomicAdd(&d.b.ocount[1 + g], 1) == runs - 1;
        __syncthreads();
        if (*s_last == 0) continue;
        __threadfence();
        if (threadIdx.x == 0) d.b.ocount[1 + g] = 0;  // for the plan's next application
        const int k1 = min(n_out, (g + 1) * per);
        for (int k = g * per + threadIdx.x; k < k1; k += blockDim.x) {
            df o[2] = {make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (c >= d.n_ch) break;
                F2Sum t{};
#pragma unroll 8
                for (int q = 0; q < runs; ++q) t.add(__ldcg(&d.b.fpart[(int64_t(q) * d.n_ch + c) * n_out + k]));
                o[c] = df_fast_two_sum(t.hi, t.lo);
            }
            finish_sample<MODE>(d, A, MODE == kInterpOrdered ? first + k : d.b.olist[k], o, false, 0.0f, 0.0f);
        }
    }
}

// Columns of NC adjacent kx of entry m: DFT of the image rows' spectra along
// y, times the kernel's spectrum, inverse DFT on the Py nodes; the window's
// rows are kept.
template <int NC> __device__ __forceinline__ void cols_fwd(const FieldDev &d, unsigned char *smem_raw, float4 (*s_low)[kLowY])
{
    const int P = d.y.P, Q = d.y.Q, J1 = d.x.J + 1, ny = d.y.n, M = max(P, Q);
    V2<float> *a = reinterpret_cast<V2<float> *>(smem_raw);
    V2<float> *b = a + (smem_fft_pad(M - 1) + 1) * NC;
    const int g = blockIdx.x % d.n_grp, m = blockIdx.x / d.n_grp;
    const int c = threadIdx.x % NC, j0 = threadIdx.x / NC, dj = blockDim.x / NC;
    const int kx = g * NC + c;
    const bool on = kx < J1;
    {
        const int H = d.x.Q / 2 + 1;
        int k = on ? kx % d.x.Q : 0;
        const bool mir = k >= H;
        if (mir) k = d.x.Q - k;
        const float2 *CR = d.b.CR + k;
#pragma unroll 4
        for (int j = j0; j < Q; j += dj) {
            float2 q = make_float2(0.0f, 0.0f);
            if (j < ny && on) q = CR[int64_t(j) * H];
            a[smem_fft_pad(j) * NC + c] = V2<float>{q.x, mir ? -q.y : q.y};
        }
    }
    __syncthreads();
    const bool low = g * NC < kFieldLow;
    if (low) {
        const int nw = blockDim.x >> 5, w = threadIdx.x >> 5;
        for (int q = w; q < NC * kFieldLow; q += nw) {
            const int cc = q % NC, kk = g * NC + cc;
            if (kk < kFieldLow)
                low_coefs(ny, Q, q / NC, d.b.twQy, d.b.KL + (m * kFieldLow + kk) * kLowY, s_low[cc],
                          [&](int e) { return d.b.CL[int64_t(e) * kFieldLow + kk]; });
        }
    }
    V2<float> *z = smem_fft<NC, -1, float>(a, b, d.fQy, reinterpret_cast<const V2<float> *>(d.b.twQy));
    V2<float> *o = z == a ? b : a;
    const int J = d.y.J, JY = 2 * J + 1;
    const float *KH = d.b.KH + ((int64_t(m) * d.n_grp + g) * JY + J) * NC + c;
    const int lift = (J / Q + 1) * Q;
    const int skip = kx < kFieldLow ? kFieldLow : 0;  // modes carried in pairs
    for (int l = J + 1 + j0; l < P - J; l += dj) o[smem_fft_pad(l) * NC + c] = V2<float>{0.0f, 0.0f};
#pragma unroll 4
    for (int ky = j0 - J; ky <= J; ky += dj) {
        V2<float> q{0.0f, 0.0f};
        const V2<float> u = z[smem_fft_pad(fast_mod(ky, Q, d.magQy, lift)) * NC + c];
        const float h = KH[ky * NC];
        if (abs(ky) >= skip) q = V2<float>{u.x * h, u.y * h};
        o[smem_fft_pad(ky < 0 ? ky + P : ky) * NC + c] = q;
    }
    __syncthreads();
    z = smem_fft<NC, 1, float>(o, o == a ? b : a, d.fPy, reinterpret_cast<const V2<float> *>(d.b.twPy));
    if (!on) return;
    float2 *F = d.b.FC + int64_t(m) * d.y.w * J1 + kx;
    const int l0 = d.y.l0 < 0 ? d.y.l0 + P : d.y.l0;
#pragma unroll 2
    for (int i = j0; i < d.y.w; i += dj) {
        int l = l0 + i;
        l -= l >= P ? P : 0;
        V2<float> q = z[smem_fft_pad(l) * NC + c];
        if (low && kx < kFieldLow) {
            F2Sum re{}, im{};
            low_add(s_low[c], l, P, d.b.twPy, re, im);
            re.add(q.x);
            im.add(q.y);
            const df r = df_fast_two_sum(re.hi, re.lo), s = df_fast_two_sum(im.hi, im.lo);
            q = V2<float>{r.x, s.x};
            d.b.FL[(int64_t(m) * d.y.w + i) * kFieldLow + kx] = make_float2(r.y, s.y);
        }
        F[int64_t(i) * J1] = f2c(q);
    }
}

// The columns and then, in the first out_blocks blocks, the outside samples'
// sums: their loop needs no more registers or shared memory than the columns'
// transforms, and in-window scans pay one load for it.  (As blocks of their own
// in the interpolation's launch they cost A at 128 x 128 / 65 536 samples 2 to
// 3 us of 82, a product of a solve 4 us, with nothing outside.)
template <int NC, int MODE, typename CIN>
__global__ void __maxnreg__(80)
k_field_cols_fwd(const __grid_constant__ FieldDev d, const __grid_constant__ InterpArgs A, const CIN *cin)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float4 s_low[NC][kLowY];
    __shared__ int s_last;
    // (loaded ahead of the columns' barriers, used behind them)
    const int n = MODE == kInterpOrdered ? d.b.toff[d.tx * d.ty] : *d.b.ocount;
    if (int(blockIdx.x) < 3 * d.n_grp) cols_fwd<NC>(d, smem_raw, s_low);
    if (int(blockIdx.x) >= d.out_blocks) return;
    const int n_out = MODE == kInterpOrdered ? int(d.T) - n : n;
    if (n_out > 0) outside_units<MODE, CIN>(d, A, cin, n_out, reinterpret_cast<V2<float> *>(smem_raw), &s_last);
}

// Node values of window rows 2b, 2b + 1 from their half spectra: xx + i xy of
// each row and yy of both as three complex sequences.
__global__ void __launch_bounds__(512) k_field_rows_inv(const __grid_constant__ FieldDev d)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float4 s_low[3][kFieldLow];  // (re, im) of both rows' lowest modes
    __shared__ float4 s_lo[3][kFieldLow];   // what those round off
    const int P = d.x.P, J = d.x.J, J1 = J + 1;
    V2<float> *a = reinterpret_cast<V2<float> *>(smem_raw);
    V2<float> *b = a + (smem_fft_pad(P - 1) + 1) * 3;
    const int i0 = 2 * blockIdx.x;
    const bool two = i0 + 1 < d.y.w;
    const int64_t plane = int64_t(d.y.w) * J1;
    const float2 *F = d.b.FC + int64_t(i0) * J1;
    for (int k = threadIdx.x; k <= P / 2; k += blockDim.x) {
        const float2 z0 = make_float2(0.0f, 0.0f);
        float2 A[3] = {z0, z0, z0}, B[3] = {z0, z0, z0};
        if (k <= J) {
            A[0] = F[k];
            B[0] = F[plane + k];
            A[2] = F[2 * plane + k];
            if (two) {
                A[1] = F[J1 + k];
                B[1] = F[plane + J1 + k];
                B[2] = F[2 * plane + J1 + k];
            }
        }
        V2<float> *o = a + smem_fft_pad(k) * 3, *n = a + smem_fft_pad(P - k) * 3;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (k < kFieldLow) {  // added at the end (the mean of a real row is real)
                const float f = k ? 2.0f : 1.0f;
                s_low[c][k] = make_float4(f * A[c].x, k ? f * A[c].y : 0.0f, f * B[c].x, k ? f * B[c].y : 0.0f);
                // entry c of A: xx of row 0, xx of row 1, yy of row 0; of B: xy, xy, yy of row 1
                const int64_t lp = int64_t(d.y.w) * kFieldLow, r0 = int64_t(i0) * kFieldLow + k, r1 = r0 + (two ? kFieldLow : 0);
                const float2 *L = d.b.FL;
                const float2 la = L[c == 0 ? r0 : c == 1 ? r1 : 2 * lp + r0];
                const float2 lb = L[c == 0 ? lp + r0 : c == 1 ? lp + r1 : 2 * lp + r1];
                s_lo[c][k] = make_float4(f * la.x, k ? f * la.y : 0.0f, f * lb.x, k ? f * lb.y : 0.0f);
                A[c] = B[c] = z0;
            }
            o[c] = V2<float>{A[c].x - B[c].y, A[c].y + B[c].x};
            if (k > 0 && 2 * k < P) n[c] = V2<float>{A[c].x + B[c].y, B[c].x - A[c].y};
        }
    }
    __syncthreads();
    const V2<float> *z = smem_fft<3, 1, float>(a, b, d.fPx, reinterpret_cast<const V2<float> *>(d.b.twPx));
    const int l0 = d.x.l0 < 0 ? d.x.l0 + P : d.x.l0;
    float4 *N = d.b.FN + int64_t(i0) * d.x.w;
    for (int i = threadIdx.x; i < d.x.w; i += blockDim.x) {
        int l = l0 + i;
        l -= l >= P ? P : 0;
        V2<float> q[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) q[c] = z[smem_fft_pad(l) * 3 + c];
        V2<float> h[3] = {};
        int at = l * (kFieldLow - 1) % P;
#pragma unroll
        for (int k = kFieldLow - 1; k >= 0; --k) {  // the mean last: one rounding at full size
            const float2 w = d.b.twPx[at];          // exp(-2 pi i k l / P)
            at -= l;
            at += at < 0 ? P : 0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float4 s = s_low[c][k], u = s_lo[c][k];
                if (k) {
                    h[c].x = fmaf(s.x, w.x, fmaf(s.y, w.y, h[c].x));
                    h[c].y = fmaf(s.z, w.x, fmaf(s.w, w.y, h[c].y));
                    q[c].x = fmaf(u.x, w.x, fmaf(u.y, w.y, q[c].x));
                    q[c].y = fmaf(u.z, w.x, fmaf(u.w, w.y, q[c].y));
                } else {
                    q[c].x = ((q[c].x + u.x) + h[c].x) + s.x;
                    q[c].y = ((q[c].y + u.z) + h[c].y) + s.z;
                }
            }
        }
        N[i] = make_float4(q[0].x, q[0].y, q[2].x, 0.0f);
        if (two) N[d.x.w + i] = make_float4(q[1].x, q[1].y, q[2].y, 0.0f);
    }
}

// The field at the samples and its product with W.  A warp takes 32 samples,
// eight lanes at a time per sample: lane a holds the stencil's column a (its
// eight rows are eight independent 16-byte loads; the eight lanes of a row
// read 128 consecutive bytes), sums its column in FP32 and adds over the
// lanes in pairs of floats.
template <int MODE>
__global__ void __launch_bounds__(kInterpThreads, 4)
k_field_interp(const __grid_constant__ FieldDev d, const __grid_constant__ InterpArgs A)
{
    chain_wait();
    const int lane = threadIdx.x & 31;
    const int64_t t = int64_t(blockIdx.x) * kInterpThreads + threadIdx.x;
    const bool valid = t < d.T;
    SampleRec q{};
    if (valid) {
        if constexpr (MODE == kInterpOrdered) {
            const float4 rc = d.b.rec[t], w = d.b.wv[t];
            const int xy = __float_as_int(rc.z);
            q.in = xy >= 0;
            q.fx = rc.x;
            q.fy = rc.y;
            q.ix = q.in ? xy & 0xffff : 0;
            q.iy = q.in ? xy >> 16 : 0;
            q.Wx = make_float2(w.x, w.z);
            q.Wy = make_float2(w.y, w.w);
        } else {
            q = make_sample(d, A.r, A.v, t);
        }
    }
    const bool in = valid && q.in;
    // this lane's stencil point as a polynomial
    float co[11];
    {
        const int a = lane & 7;
#pragma unroll
        for (int k = 0; k < 11; ++k) co[k] = a < 4 ? kKb[a][k] : ((k & 1) ? -kKb[7 - a][k] : kKb[7 - a][k]);
    }
    df phi[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    const unsigned inmask = __ballot_sync(0xffffffffu, in);
    if (inmask) {
#pragma unroll 2
        for (int g = 0; g < 8; ++g) {
            const int src = 4 * g + (lane >> 3);
            const float fx = __shfl_sync(0xffffffffu, q.fx, src), fy = __shfl_sync(0xffffffffu, q.fy, src);
            const int ix = __shfl_sync(0xffffffffu, q.ix, src), iy = __shfl_sync(0xffffffffu, q.iy, src);
            const bool on = (inmask >> src) & 1u;
            const float tx = (on ? fx : 0.5f) - 0.5f, ty = (on ? fy : 0.5f) - 0.5f;
            float wx = co[10], wl = co[10];
#pragma unroll
            for (int k = 9; k >= 0; --k) {
                wx = fmaf(wx, tx, co[k]);
                wl = fmaf(wl, ty, co[k]);
            }
            const float4 *F = d.b.FN + int64_t(on ? iy : 0) * d.x.w + (on ? ix : 0) + (lane & 7);
            float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
            float4 f[8];
#pragma unroll
            for (int b = 0; b < 8; ++b) f[b] = F[int64_t(b) * d.x.w];
            // outermost points first: the small terms are added while the sum is small
            constexpr int ord[8] = {0, 7, 1, 6, 2, 5, 3, 4};
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                const int b = ord[o];
                const float wy = __shfl_sync(0xffffffffu, wl, (lane & 24) + b);
                s0 = fmaf(wy, f[b].x, s0);
                s1 = fmaf(wy, f[b].y, s1);
                s2 = fmaf(wy, f[b].z, s2);
            }
            // Products as pairs, then the sums over the eight lanes: the lane
            // bits 0 and 1 also choose which entry a lane goes on with (0: xx,
            // 1: xy, 2: yy, 3: none), so three levels take four additions.
            F2Sum p0{}, p1{}, p2{};
            p0.hi = s0 * wx; p0.lo = fmaf(s0, wx, -p0.hi);
            p1.hi = s1 * wx; p1.lo = fmaf(s1, wx, -p1.hi);
            p2.hi = s2 * wx; p2.lo = fmaf(s2, wx, -p2.hi);
            const bool up = lane & 2;  // keeps yy, sends xx and xy
            F2Sum a = up ? p2 : p0, e = up ? F2Sum{} : p1;
            const F2Sum sa = up ? p0 : p2, se = up ? p1 : F2Sum{};
            a.add(f2_shfl_xor(sa, 2));
            e.add(f2_shfl_xor(se, 2));
            F2Sum v = (lane & 1) ? e : a;
            v.add(f2_shfl_xor((lane & 1) ? a : e, 1));
            v.add(f2_shfl_xor(v, 4));
            const int back = 8 * (lane & 3);
            const float h0 = __shfl_sync(0xffffffffu, v.hi, back), l0 = __shfl_sync(0xffffffffu, v.lo, back);
            const float h1 = __shfl_sync(0xffffffffu, v.hi, back + 1), l1 = __shfl_sync(0xffffffffu, v.lo, back + 1);
            const float h2 = __shfl_sync(0xffffffffu, v.hi, back + 2), l2 = __shfl_sync(0xffffffffu, v.lo, back + 2);
            if ((lane >> 2) == g) {
                phi[0] = df_fast_two_sum(h0, l0);
                phi[1] = df_fast_two_sum(h1, l1);
                phi[2] = df_fast_two_sum(h2, l2);
            }
        }
    }
    if (in) {
        const df Ox = df_add(df_mul(phi[0], q.Wx), df_mul(phi[1], q.Wy)), Oy = df_add(df_mul(phi[1], q.Wx), df_mul(phi[2], q.Wy));
        df o[2];
#pragma unroll
        for (int k = 0; k < 2; ++k)  // (a single channel's second is not stored)
            o[k] = df_add(df_mul(Ox, make_float2(d.p[2 * k], 0.0f)), df_mul(Oy, make_float2(d.p[2 * k + 1], 0.0f)));
        finish_sample<MODE>(d, A, t, o, true, q.Wx.x, q.Wy.x);
    }
}

// --- adjoint --------------------------------------------------------------------

// Chunks of the outside samples' partial images, of at least 128 samples (13 000
// on 64 x 64 voxels: 45 us, with 384 a chunk 70).
__device__ __forceinline__ int out_chunks_used(const FieldDev &d, int n_out)
{
    return n_out > 0 ? min(d.out_chunks, (n_out + 127) / 128) : 0;
}

// Partial image of the ordered outside samples c0 .. c1 - 1 on one tile of the
// voxels: a thread owns kOutRows voxels of one column, 32 staged samples at a
// time are summed plainly and added with compensation.  For a diagonal G two
// samples share packed FP32 arithmetic, as in the pair sums; for a general G
// their test against the warp's voxels chooses the form.  A^T at 128 x 128 /
// 65 536 samples, 94 % of them outside: 0.48 ms, before 0.81 ms (pair sums of
// all samples 0.42 ms); 512 x 512, 84 %: 5.7 ms (7.9, 6.0).
__device__ __forceinline__ void outside_image(const FieldDev &d, int tile, int c0, int c1, float *s_p, float *__restrict__ out)
{
    static_assert(6 * kOutThreads <= 6 * kPatch * kPatchPitch, "staged samples");
    const int nx = d.x.n, ny = d.y.n, lane = threadIdx.x & 31;
    const int n_q = nx * ((ny + kOutRows - 1) / kOutRows);
    const int q0 = tile * kOutThreads + int(threadIdx.x), qc = min(q0, n_q - 1);
    const int i = qc % nx, jb = qc / nx * kOutRows;
    const V2<float> xc = d.b.xcol[i];
    float Yx[kOutRows], Yy[kOutRows], acc[kOutRows], comp[kOutRows];
#pragma unroll
    for (int k = 0; k < kOutRows; ++k) {
        const V2<float> yr = d.b.yrow[min(jb + k, ny - 1)];
        Yx[k] = yr.x, Yy[k] = yr.y;
        acc[k] = comp[k] = 0.0f;
    }
    float lo[2] = {xc.x + Yx[0], xc.y + Yy[0]}, hi[2] = {lo[0], lo[1]};  // general G: the warp's voxels
    if (!d.diag) {
#pragma unroll
        for (int k = 1; k < kOutRows; ++k) {
            const float e[2] = {xc.x + Yx[k], xc.y + Yy[k]};
#pragma unroll
            for (int a = 0; a < 2; ++a) lo[a] = min(lo[a], e[a]), hi[a] = max(hi[a], e[a]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                lo[a] = min(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
                hi[a] = max(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
            }
    }
#pragma unroll 1
    for (int cb = c0; cb < c1; cb += kOutThreads) {
        const int nb = min(kOutThreads, c1 - cb), nb2 = (nb + 1) & ~1;
        __syncthreads();
        if (int(threadIdx.x) < nb2) {
            const int k = threadIdx.x, t = cb + min(k, nb - 1);
            const float4 rc = d.b.rec[t], w = d.b.wv[t];
            const float4 u = k < nb ? d.b.q4[t] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);  // (an odd count: one without weight)
            const float uW = u.x * w.x + u.y * w.y, Sxx = w.x * u.x, Sxy = w.x * u.y + w.y * u.x, Syy = w.y * u.y;
            if (d.diag) {  // pairs: (-x, -y), (uW, Sxx), (Sxy, Syy), each entry (even, odd)
                float *q = s_p + 12 * (k >> 1) + (k & 1);
                q[0] = -rc.x;
                q[2] = -rc.y;
                q[4] = uW;
                q[6] = Sxx;
                q[8] = Sxy;
                q[10] = Syy;
            } else {
                float *q = s_p + 6 * k;
                q[0] = rc.x;
                q[1] = rc.y;
                q[2] = uW;
                q[3] = Sxx;
                q[4] = Sxy;
                q[5] = Syy;
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int k0 = 0; k0 < nb2; k0 += 32) {
            const int kn = min(32, nb2 - k0);
            float blk[kOutRows];
#pragma unroll
            for (int k = 0; k < kOutRows; ++k) blk[k] = 0.0f;
            if (d.diag) {
                const float4 *pk = reinterpret_cast<const float4 *>(s_p) + 3 * (k0 >> 1);
                float2 yr2[kOutRows], blk2[kOutRows];
#pragma unroll
                for (int k = 0; k < kOutRows; ++k) yr2[k] = make_float2(Yy[k], Yy[k]), blk2[k] = make_float2(0.0f, 0.0f);
#pragma unroll 2
                for (int h = 0; h < (kn >> 1); ++h)
                    adj_pair2_vfar_diag<false>(pk[3 * h], pk[3 * h + 1], pk[3 * h + 2], make_float2(xc.x, xc.x), yr2, blk2);
#pragma unroll
                for (int k = 0; k < kOutRows; ++k) blk[k] = blk2[k].x + blk2[k].y;
            } else {
                bool far = true;
                if (lane < kn) {
                    const float *q = s_p + 6 * (k0 + lane);
                    const float gx = max(0.0f, max(lo[0] - q[0], q[0] - hi[0])), gy = max(0.0f, max(lo[1] - q[1], q[1] - hi[1]));
                    far = fmx(gy, gy, gx * gx) >= vfar_threshold<float, false>();
                }
                const unsigned mask = __ballot_sync(0xffffffffu, far);
#pragma unroll 1
                for (int k = 0; k < kn; ++k) {
                    const float *q = s_p + 6 * (k0 + k);
                    const V2<float> rr{q[0], q[1]};
                    const V4<float> S{q[2], q[3], q[4], q[5]};
                    if ((mask >> k) & 1u) adj_sample<float, false, false, 2>(rr, S, xc, Yx, Yy, blk);
                    else adj_sample<float, false, false, 0>(rr, S, xc, Yx, Yy, blk);
                }
            }
#pragma unroll
            for (int k = 0; k < kOutRows; ++k) kahan_add(acc[k], comp[k], blk[k]);
        }
    }
    if (q0 >= n_q) return;
#pragma unroll
    for (int k = 0; k < kOutRows; ++k)
        if (jb + k < ny) out[int64_t(jb + k) * nx + i] = acc[k];
}

// One spreading unit u, by one block: the patch of the unit's tile, summed over
// its samples in order.  A warp owns one entry of K on the patch rows of one
// parity: a sample's stencil has four such rows of eight points, one per lane,
// so no two lanes share a node and the order of the additions is the samples'
// order.  The unit's two halves go to two copies of the patch, added at the
// end: twice the independent chains of load, FMA and store.  What bounds it is
// the shared-memory pipe: per sample and warp one load and one store of the
// patch, and a quarter of three 16-byte loads (weights and addresses of four
// samples, fetched one step ahead).
constexpr int kUnitPitch = kFieldUnit + 4;
__device__ __forceinline__ void spread_unit(const FieldDev &d, int u, float (*s_patch)[3][kPatch * kPatchPitch])
{
    __shared__ __align__(16) float s_wx[kWin][kUnitPitch];
    __shared__ __align__(16) float s_c[3][kWin][kUnitPitch];  // entry x row weight, rows by parity
    __shared__ __align__(16) int s_at[kUnitPitch];
    const int tile = d.b.unit_tile[u];
    const int u0 = d.b.uoff[tile], nu = d.b.uoff[tile + 1] - u0;
    const int t0 = d.b.toff[tile], t1 = d.b.toff[tile + 1];
    const int len = (t1 - t0 + nu - 1) / nu;  // the tile's units share its samples evenly
    const int q0 = t0 + (u - u0) * len;
    const int n = max(0, min(len, t1 - q0)), n4 = (n + 3) & ~3;
    for (int k = threadIdx.x; k < 6 * kPatch * kPatchPitch; k += kSpreadThreads) (&s_patch[0][0][0])[k] = 0.0f;
    const int ox = (tile % d.tx) * kTile, oy = (tile / d.tx) * kTile;
    for (int k = threadIdx.x; k < n4; k += kSpreadThreads) {
        float wx[kWin] = {}, wy[kWin] = {};
        float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        int ix = 0, iy = 0;
        if (k < n) {
            const float4 rc = d.b.rec[q0 + k];
            q = d.b.q4[q0 + k];
            const int xy = __float_as_int(rc.z);
            iy = (xy >> 16) - oy;
            ix = (xy & 0xffff) - ox;
            const float tx = rc.x - 0.5f, tx2 = tx * tx, ty = rc.y - 0.5f, ty2 = ty * ty;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                float ex = kKb[a][10], dx = kKb[a][9], ey = ex, dy = dx;
#pragma unroll
                for (int j = 8; j >= 0; j -= 2) ex = fmaf(ex, tx2, kKb[a][j]), ey = fmaf(ey, ty2, kKb[a][j]);
#pragma unroll
                for (int j = 7; j >= 1; j -= 2) dx = fmaf(dx, tx2, kKb[a][j]), dy = fmaf(dy, ty2, kKb[a][j]);
                wx[a] = fmaf(dx, tx, ex);
                wx[7 - a] = fmaf(-dx, tx, ex);
                wy[a] = fmaf(dy, ty, ey);
                wy[7 - a] = fmaf(-dy, ty, ey);
            }
        }
        const int odd = iy & 1;
        s_at[k] = (iy * kPatchPitch + ix) | (odd << 16);
#pragma unroll
        for (int a = 0; a < kWin; ++a) {
            s_wx[a][k] = wx[a];
            // row iy + b has parity (iy + b) & 1: slot p holds b = p ^ (iy & 1)
            const float w = odd ? wy[a ^ 1] : wy[a];
            s_c[0][a][k] = q.x * w;
            s_c[1][a][k] = q.y * w;
            s_c[2][a][k] = q.z * w;
        }
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = warp / 6, mid = (n4 / 4 + 1) / 2 * 4;
    const int k0 = half ? mid : 0, k1 = half ? n4 : mid;
    if (k0 < k1) {
        const int m = (warp % 6) >> 1, par = warp & 1;
        const int col = lane & 7, p = 2 * (lane >> 3) + par;
        const float4 *wp = reinterpret_cast<const float4 *>(s_wx[col]), *cp = reinterpret_cast<const float4 *>(s_c[m][p]);
        const int4 *ap = reinterpret_cast<const int4 *>(s_at);
        // this lane's offset in the stencil for an even / odd first row
        float *P0 = s_patch[half][m] + p * kPatchPitch + col, *P1 = s_patch[half][m] + (p ^ 1) * kPatchPitch + col;
        auto add = [&](int at, float c, float w) {
            float *o = ((at >> 16) ? P1 : P0) + (at & 0xffff);
            *o = fmaf(c, w, *o);
            __syncwarp();
        };
        int4 at = ap[k0 >> 2];
        float4 w = wp[k0 >> 2], c = cp[k0 >> 2];
        for (int k = k0; k < k1; k += 4) {
            const int nx = min(k + 4, k1 - 4) >> 2;
            const int4 at2 = ap[nx];
            const float4 w2 = wp[nx], c2 = cp[nx];
            add(at.x, c.x, w.x);
            add(at.y, c.y, w.y);
            add(at.z, c.z, w.z);
            add(at.w, c.w, w.w);
            at = at2;
            w = w2;
            c = c2;
        }
    }
    __syncthreads();
    float *out = d.b.upart + int64_t(u) * 3 * kPatchSize;
    for (int k = threadIdx.x; k < 3 * kPatchSize; k += kSpreadThreads) {
        const int mm = k / kPatchSize, e = k % kPatchSize;
        const int at = (e / kPatch) * kPatchPitch + e % kPatch;
        out[k] = s_patch[0][mm][at] + s_patch[1][mm][at];
    }
}

// The units, one per block, then the outside samples' partial images by the
// blocks from the last one down (units leave most of them free: their number is
// only bounded by n_unit_max).
__global__ void __launch_bounds__(kSpreadThreads, kSpreadPerSm) k_field_spread(const __grid_constant__ FieldDev d)
{
    chain_wait();
    __shared__ __align__(16) float s_patch[2][3][kPatch * kPatchPitch];
    const int nt = d.tx * d.ty;
    const int first = d.b.toff[nt], n_unit = d.b.uoff[nt];
    if (int(blockIdx.x) < n_unit) spread_unit(d, blockIdx.x, s_patch);
    const int n_out = int(d.T) - first;
    if (n_out <= 0) return;
    const int used = out_chunks_used(d, n_out), len = (n_out + used - 1) / used;
#pragma unroll 1
    for (int job = int(gridDim.x) - 1 - int(blockIdx.x); job < used * d.out_tiles; job += gridDim.x) {
        const int chunk = job / d.out_tiles, tile = job % d.out_tiles;
        const int c0 = first + chunk * len, c1 = min(int(d.T), c0 + len);
        outside_image(d, tile, c0, c1, &s_patch[0][0][0], d.b.opart + int64_t(chunk) * d.x.n * d.y.n);
    }
}

// Half spectra of node rows 2b, 2b + 1: a node is the sum of the patches of
// the up to four tiles that reach it, in a fixed order, in pairs of floats (a
// tile where the trajectory dwells has thousands of units, whose plain FP32
// sum would leave 1e-6).  Bound by the latency of those loads: the tiles' first
// units, then four of a tile, are in flight at once (A^T at 128 x 128 / 65 536
// samples 92.7 us, one unit after another 95.5; plain FP32 sums of one unit
// after another 93.0).
constexpr int kUnitsAtOnce = 4;
__global__ void __launch_bounds__(512) k_field_rows_fwd(const __grid_constant__ FieldDev d)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P = d.x.P, J1 = d.x.J + 1, wx = d.x.w;
    V2<float> *a = reinterpret_cast<V2<float> *>(smem_raw);
    V2<float> *b = a + (smem_fft_pad(P - 1) + 1) * 3;
    const int i0 = 2 * blockIdx.x;
    const int l0 = d.x.l0 < 0 ? d.x.l0 + P : d.x.l0;
    const int ty1 = min(i0 / kTile, d.ty - 1);
    const int ty0 = max(0, (i0 - kPatch + kTile) / kTile);
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        F2Sum g[2][3] = {};
        if (i < wx) {
            const int tx1 = min(i / kTile, d.tx - 1), tx0 = max(0, (i - kPatch + kTile) / kTile);
            auto load = [&](const float *e, bool two, float (&q)[2][3]) {
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    q[0][m] = e[m * kPatchSize];
                    q[1][m] = two ? e[m * kPatchSize + kPatch] : 0.0f;
                }
            };
            auto add = [&](const float (&q)[2][3]) {
#pragma unroll
                for (int m = 0; m < 3; ++m) g[0][m].add(q[0][m]), g[1][m].add(q[1][m]);
            };
            // the four tiles' first units at once, then what more they have
            int u0[4], u1[4];
            float q[4][2][3];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int ty = ty0 + (k >> 1), tx = tx0 + (k & 1), tile = ty * d.tx + tx;
                const bool on = ty <= ty1 && tx <= tx1;
                u0[k] = on ? d.b.uoff[tile] : 0;
                u1[k] = on ? d.b.uoff[tile + 1] : 0;
            }
            auto patch = [&](int k, int u) {
                const int pr = i0 - (ty0 + (k >> 1)) * kTile;  // patch row of the first node row
                return d.b.upart + int64_t(u) * 3 * kPatchSize + pr * kPatch + i - (tx0 + (k & 1)) * kTile;
            };
            const bool two[2] = {i0 - ty0 * kTile + 1 < kPatch, i0 - ty0 * kTile + 1 < kPatch + kTile};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (u0[k] < u1[k]) {
                    load(patch(k, u0[k]), two[k >> 1], q[k]);
                } else {
#pragma unroll
                    for (int m = 0; m < 3; ++m) q[k][0][m] = q[k][1][m] = 0.0f;
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) add(q[k]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                for (int u = u0[k] + 1; u < u1[k]; u += kUnitsAtOnce) {
#pragma unroll
                    for (int e = 0; e < kUnitsAtOnce; ++e) load(patch(k, min(u + e, u1[k] - 1)), two[k >> 1], q[e]);
#pragma unroll
                    for (int e = 0; e < kUnitsAtOnce; ++e)
                        if (u + e < u1[k]) add(q[e]);
                }
            }
        }
        int l = l0 + i;
        l -= l >= P ? P : 0;
        V2<float> *o = a + smem_fft_pad(l) * 3;
        o[0] = V2<float>{g[0][0].hi + g[0][0].lo, g[0][1].hi + g[0][1].lo};
        o[1] = V2<float>{g[1][0].hi + g[1][0].lo, g[1][1].hi + g[1][1].lo};
        o[2] = V2<float>{g[0][2].hi + g[0][2].lo, g[1][2].hi + g[1][2].lo};
    }
    __shared__ V2<float> s_low[kLowY][3];
    __syncthreads();
    low_rows(a, P, d.b.twPx, s_low);
    __syncthreads();
    const V2<float> *z = smem_fft<3, -1, float>(a, b, d.fPx, reinterpret_cast<const V2<float> *>(d.b.twPx));
    store_rows(z, P, J1, i0, d.y.w, s_low, d.b.FC);
}

// Columns of NC adjacent kx of entry m: DFT along y of the window's rows,
// times the kernel's spectrum, inverse DFT at the voxel rows.
template <int NC>
__global__ void __launch_bounds__(512) k_field_cols_adj(const __grid_constant__ FieldDev d)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float4 s_low[NC][kLowY];
    const int P = d.y.P, Q = d.y.Q, J1 = d.x.J + 1, ny = d.y.n, M = max(P, Q), wy = d.y.w;
    V2<float> *a = reinterpret_cast<V2<float> *>(smem_raw);
    V2<float> *b = a + (smem_fft_pad(M - 1) + 1) * NC;
    const int g = blockIdx.x % d.n_grp, m = blockIdx.x / d.n_grp;
    const int c = threadIdx.x % NC, j0 = threadIdx.x / NC, dj = blockDim.x / NC;
    const int kx = g * NC + c;
    const bool on = kx < J1;
    {
        const float2 *F = d.b.FC + int64_t(m) * wy * J1 + (on ? kx : 0);
        const int l0 = d.y.l0 < 0 ? d.y.l0 + P : d.y.l0;
#pragma unroll 4
        for (int i = j0; i < P; i += dj) {
            float2 q = make_float2(0.0f, 0.0f);
            if (i < wy && on) q = F[int64_t(i) * J1];
            int l = l0 + i;
            l -= l >= P ? P : 0;
            a[smem_fft_pad(l) * NC + c] = v2(q);
        }
    }
    __syncthreads();
    const bool low = g * NC < kFieldLow;
    if (low) {
        const int nw = blockDim.x >> 5, w = threadIdx.x >> 5;
        for (int q = w; q < NC * kFieldLow; q += nw) {
            const int cc = q % NC, kk = g * NC + cc;
            if (kk < kFieldLow)
                low_coefs(P, P, q / NC, d.b.twPy, d.b.KL + (m * kFieldLow + kk) * kLowY, s_low[cc], [&](int e) {
                    const V2<float> z = a[smem_fft_pad(e) * NC + cc];
                    return make_float4(z.x, z.y, 0.0f, 0.0f);
                });
        }
        __syncthreads();
    }
    V2<float> *z = smem_fft<NC, -1, float>(a, b, d.fPy, reinterpret_cast<const V2<float> *>(d.b.twPy));
    V2<float> *o = z == a ? b : a;
    const int J = d.y.J, JY = 2 * J + 1;
    const float *KH = d.b.KH + ((int64_t(m) * d.n_grp + g) * JY + J) * NC + c;
    const int skip = kx < kFieldLow ? kFieldLow : 0;  // modes carried in pairs
#pragma unroll 2
    for (int k = j0; k < Q; k += dj) {
        V2<float> s{0.0f, 0.0f};
        // modes ky = k mod Q
        for (int ky = k - int(__umulhi(unsigned(J + k), d.magQy)) * Q; ky <= J; ky += Q) {
            if (abs(ky) < skip) continue;
            const V2<float> u = z[smem_fft_pad(ky < 0 ? ky + P : ky) * NC + c];
            const float h = KH[ky * NC];
            s.x = fmaf(u.x, h, s.x);
            s.y = fmaf(u.y, h, s.y);
        }
        o[smem_fft_pad(k) * NC + c] = s;
    }
    __syncthreads();
    z = smem_fft<NC, 1, float>(o, o == a ? b : a, d.fQy, reinterpret_cast<const V2<float> *>(d.b.twQy));
    if (!on) return;
    float2 *AC = d.b.AC + int64_t(m) * ny * J1 + kx;
    for (int j = j0; j < ny; j += dj) {
        const V2<float> q = z[smem_fft_pad(j) * NC + c];
        if (low && kx < kFieldLow) {
            F2Sum re{q.x, 0.0f}, im{q.y, 0.0f};
            low_add(s_low[c], j, Q, d.b.twQy, re, im);
            const float2 r = df_fast_two_sum(re.hi, re.lo), i = df_fast_two_sum(im.hi, im.lo);
            d.b.AL[(int64_t(m) * ny + j) * kFieldLow + kx] = make_float4(r.x, i.x, r.y, i.y);
        } else {
            AC[int64_t(j) * J1] = f2c(q);
        }
    }
}

// Voxel rows 2b, 2b + 1: the three entries' half spectra added and folded to
// the Qx modes of the voxel grid, inverse DFT (the modes kx < kFieldLow
// added in pairs), plus the outside samples' partial images.
template <typename OUT, bool CG>
__global__ void __launch_bounds__(128) k_field_out(const __grid_constant__ FieldDev d, OUT *__restrict__ out,
                                                   const double *p, const double *nu_dev,
                                                   double *__restrict__ dot_part)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double s_red[4];
    __shared__ float4 s_low[2][kFieldLow];
    const int Q = d.x.Q, nx = d.x.n, ny = d.y.n, J = d.x.J, J1 = J + 1;
    V2<float> *a = reinterpret_cast<V2<float> *>(smem_raw);
    V2<float> *b = a + smem_fft_pad(Q - 1) + 1;
    const int j0 = 2 * blockIdx.x;
    const bool two = j0 + 1 < ny;
    const int64_t plane = int64_t(ny) * J1;
    const float2 *A0 = d.b.AC + int64_t(j0) * J1, *A1 = A0 + (two ? J1 : 0);
    for (int k = threadIdx.x; k < Q; k += blockDim.x) {
        V2<float> z{0.0f, 0.0f};
        for (int kx = k - ((J + k) / Q) * Q; kx <= J; kx += Q) {
            const int ka = abs(kx);
            if (ka < kFieldLow) continue;
            const float2 u0 = A0[ka], u1 = A0[plane + ka], u2 = A0[2 * plane + ka];
            const float2 w0 = A1[ka], w1 = A1[plane + ka], w2 = A1[2 * plane + ka];
            const float ar = u0.x + u1.x + u2.x, br = w0.x + w1.x + w2.x;
            float ai = u0.y + u1.y + u2.y, bi = w0.y + w1.y + w2.y;
            if (kx < 0) ai = -ai, bi = -bi;
            z.x += ar - bi;
            z.y += ai + br;
        }
        a[smem_fft_pad(k)] = z;
    }
    if (threadIdx.x < 2 * kFieldLow) {
        const int rr = threadIdx.x / kFieldLow, k = threadIdx.x % kFieldLow;
        const int j = j0 + (two ? rr : 0);
        F2Sum re{}, im{};
        for (int m = 0; m < 3; ++m) {
            const float4 v = d.b.AL[(int64_t(m) * ny + j) * kFieldLow + k];
            re.add(v.x);
            im.add(v.y);
            re.lo += v.z;
            im.lo += v.w;
        }
        const float2 r = df_fast_two_sum(re.hi, re.lo), i = df_fast_two_sum(im.hi, im.lo);
        // a mode and its conjugate: twice the real part (the mean counts once)
        s_low[rr][k] = k ? make_float4(2.0f * r.x, 2.0f * i.x, 2.0f * r.y, 2.0f * i.y) : make_float4(r.x, 0.0f, r.y, 0.0f);
    }
    __syncthreads();
    const V2<float> *z = smem_fft<1, 1, float>(a, b, d.fQx, reinterpret_cast<const V2<float> *>(d.b.twQx));
    const int n_out = int(d.T) - d.b.toff[d.tx * d.ty];
    const int used = out_chunks_used(d, n_out);
    const int64_t N = int64_t(nx) * ny;
    double dot = 0.0;
    const double nu = CG ? *nu_dev : 0.0;
    for (int t = threadIdx.x; t < 2 * nx; t += blockDim.x) {
        const int rr = t >= nx ? 1 : 0, i = t - rr * nx;
        if (rr && !two) break;
        const V2<float> q = z[smem_fft_pad(i)];
        F2Sum s{rr ? q.y : q.x, 0.0f};
        int at = 0;
#pragma unroll
        for (int k = 0; k < kFieldLow; ++k) {
            const float2 w = d.b.twQx[at];  // exp(-2 pi i k i / Q)
            at += i;
            at -= at >= Q ? Q : 0;
            const float4 v = s_low[rr][k];
            f2_fma(s, v.x, w.x);
            if (k) f2_fma(s, v.y, w.y);
            s.lo += fmaf(v.z, w.x, v.w * w.y);
        }
        const int64_t e = int64_t(j0 + rr) * nx + i;
        for (int c = 0; c < used; c += 8) {  // (eight loads in flight)
            float q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) q[k] = c + k < used ? d.b.opart[int64_t(c + k) * N + e] : 0.0f;
#pragma unroll
            for (int k = 0; k < 8; ++k) s.add(q[k]);
        }
        if constexpr (CG) {
            const double pe = p[e], val = s.value() + nu * pe;
            dot += pe * val;
            out[e] = OUT(val);
        } else if constexpr (sizeof(OUT) == 4) {
            out[e] = s.hi + s.lo;
        } else {
            out[e] = s.value();
        }
    }
    if constexpr (CG) {
        dot = block_sum<double, 128>(dot, s_red);
        if (threadIdx.x == 0) dot_part[blockIdx.x] = dot;
    }
}

// --- host -----------------------------------------------------------------------

size_t up256(size_t b) { return (b + 255) & ~size_t(255); }

// The transforms' lengths, 2^a 3^b 5^c, in ascending order with their passes:
// made once, so that a call plans an axis in 0.2 us (factoring every candidate
// took 4 to 15, also for calls that then take the pair sums).
struct FftLengths {
    struct Length {
        int n, np;
    } l[256];  // (134 up to 4096)
    int count = 0;
    FftLengths()
    {
        for (int n = 4; n <= kFieldMaxN && count < 256; ++n)
            if (const int np = smem_fft_plan(n).np) l[count++] = {n, np};
    }
    const Length *begin() const { return l; }
    const Length *end() const { return l + count; }
    const Length *from(int64_t n) const  // the first of at least n
    {
        return std::lower_bound(begin(), end(), n, [](const Length &a, int64_t b) { return a.n < b; });
    }
};
const FftLengths &fft_lengths()
{
    static const FftLengths list;
    return list;
}

// The length in [n, 5/4 n + 8] that costs least: elements times passes, and
// a fixed part for the load and the store.
int good_length(int64_t n, double &cost)
{
    const FftLengths &lengths = fft_lengths();
    int best = 0;
    for (auto k = lengths.from(n); k != lengths.end() && k->n <= n + n / 4 + 8; ++k) {
        const double c = double(k->n) * (4.0 + k->np);
        if (best == 0 || c < cost) best = k->n, cost = c;
    }
    return best;
}

void split(double v, float (&o)[2])
{
    o[0] = float(v);
    o[1] = float(v - double(o[0]));
}

// pitch: |beta G e| h, one voxel's step in z units.
bool plan_axis(int n, double pitch, double p0, double h, FieldAxis &a)
{
    const double extra = 5.5 * kPitch;  // the stencil beyond the window
    const double D = n - 0.5 + (kMargin + extra) / pitch;
    const double qmin = 2.0 * D + 2.0 * kCutArg * kCutScale / pitch;
    if (!(qmin <= kFieldMaxN) || !(qmin * pitch / kPitch <= kFieldMaxN)) return false;
    a.n = n;
    a.Q = 0;
    // A longer period needs more nodes: the pair that costs least (the
    // transforms over the nodes outweigh those over the voxels).
    const int64_t q0 = std::max<int64_t>(4, (int64_t)std::ceil(qmin));
    const FftLengths &lengths = fft_lengths();
    double best = 0.0;
    for (auto k = lengths.from(q0); k != lengths.end() && k->n <= q0 + q0 / 5 + 4; ++k) {
        const int q = k->n, npq = k->np;
        const double pmin = q * pitch / kPitch;
        if (!(pmin <= kFieldMaxN)) break;
        double cp = 0.0;
        const int p = good_length((int64_t)std::ceil(pmin), cp);
        if (p == 0) break;
        const double c = cp + 0.3 * double(q) * (4.0 + npq);
        if (a.Q == 0 || c < best) best = c, a.Q = q, a.P = p;
    }
    if (a.Q == 0) return false;
    const double step = double(a.P) / a.Q;  // nodes per voxel
    const double lo = (-0.5 - kMargin / pitch) * step, hi = (n - 0.5 + kMargin / pitch) * step;
    a.l0 = (int)std::floor(lo) - kWin / 2;
    a.w = (int)std::floor(hi) + kWin / 2 + 3 - a.l0;
    a.J = std::min((int)(kModeMax * a.Q * pitch / (2.0 * 3.14159265358979323846)), (a.P - 1) / 2 - 1);
    a.xlo = float(lo - a.l0);
    a.xhi = float(hi - a.l0);
    split(step / h, a.sc);
    split((-p0 / h - 0.5) * step - a.l0, a.of);
    // half the nodes between the largest offset in use and its nearest image
    const double cut = 0.5 * a.P - std::max<double>(a.l0 + a.w, (n - 1) * step - a.l0);
    a.cut_inv = float(kCutArg / cut);
    return a.J >= kFieldLow && a.w + kWin <= a.P && a.w < 32768 && cut / kCutArg * (pitch / step) > 1.0;
}

int cols_nc(const FieldDev &d) { return std::max(d.y.P, d.y.Q) <= 2048 ? 4 : 2; }
// One radix-8 butterfly per thread and pass, up to 512 threads (384 at 4 x 768
// points; 512 or 256 threads were 10 and 7 % slower over a whole A).
int fft_threads(int nc, int n)
{
    const int b = (nc * n + 7) / 8, per = (b + 511) / 512;
    return std::max(128, ((b + per - 1) / per + 31) / 32 * 32);
}
int cols_threads(const FieldDev &d) { return fft_threads(cols_nc(d), std::max(d.y.P, d.y.Q)); }
size_t rows_smem(const FieldDev &d) { return 2 * sizeof(float2) * smem_fft_elems(std::max(d.x.P, d.x.Q), 3); }
size_t cols_smem(const FieldDev &d)
{
    return std::max(2 * sizeof(float2) * smem_fft_elems(std::max(d.y.P, d.y.Q), cols_nc(d)), sizeof(float2) * kOutStage);
}
size_t image_smem(const FieldDev &d) { return 2 * sizeof(float2) * smem_fft_elems(d.x.Q, 1); }
// Warps per block of the ordering kernels: each has its own tile counters.
int order_warps(const FieldDev &d) { return std::max(1, std::min<int>(4, 48 * 1024 / (4 * (d.tx * d.ty + 1)))); }
size_t order_smem(const FieldDev &d) { return sizeof(int) * size_t(d.tx * d.ty + 1) * order_warps(d); }

// Shared memory above 48 KB is granted per kernel; asked for outside any
// stream capture (field_prepare), so the launches only launch.
int allow_all(const FieldDev &d, bool forward, bool adjoint)
{
    const bool four = cols_nc(d) == 4;
    MPI_TRY(allow_smem(k_field_rows, rows_smem(d)));
    MPI_TRY(allow_smem(four ? k_field_kcols<4> : k_field_kcols<2>, cols_smem(d)));
    if (forward) {
        MPI_TRY(allow_smem(k_field_image<double>, image_smem(d)));
        MPI_TRY(allow_smem(four ? k_field_cols_fwd<4, kInterpForward, float> : k_field_cols_fwd<2, kInterpForward, float>,
                           cols_smem(d)));
        MPI_TRY(allow_smem(four ? k_field_cols_fwd<4, kInterpOrdered, double> : k_field_cols_fwd<2, kInterpOrdered, double>,
                           cols_smem(d)));
        MPI_TRY(allow_smem(k_field_rows_inv, rows_smem(d)));
    }
    if (adjoint) {
        MPI_TRY(allow_smem(k_field_setup, order_smem(d)));
        MPI_TRY(allow_smem(k_field_place, order_smem(d)));
        MPI_TRY(allow_smem(k_field_rows_fwd, rows_smem(d)));
        MPI_TRY(allow_smem(four ? k_field_cols_adj<4> : k_field_cols_adj<2>, cols_smem(d)));
        MPI_TRY(allow_smem(k_field_out<float, false>, image_smem(d)));
        MPI_TRY(allow_smem(k_field_out<double, false>, image_smem(d)));
        MPI_TRY(allow_smem(k_field_out<double, true>, image_smem(d)));
    }
    return MPI_OK;
}

// The plan's buffers: `keep` holds what a prepared plan needs between
// applications, `work` what one preparation or application uses.
void lay_out(FieldPlan &plan, char *keep, char *work, size_t &keep_bytes, size_t &work_bytes)
{
    FieldDev &d = plan.d;
    FieldBuf &b = d.b;
    size_t tot[2] = {0, 0};
    auto take = [&](int which, auto *&ptr, size_t n) {
        char *base = which ? work : keep;
        ptr = base ? reinterpret_cast<std::remove_reference_t<decltype(ptr)>>(base + tot[which]) : nullptr;
        tot[which] += up256(sizeof(*ptr) * n);
    };
    const size_t J1 = d.x.J + 1, T1 = size_t(d.T), ny = d.y.n, nt = size_t(d.tx) * d.ty, nh = (nt + 1) * d.n_run;
    take(0, b.twPx, d.x.P); take(0, b.twPy, d.y.P); take(0, b.twQy, d.y.Q); take(0, b.twQx, d.x.Q);
    take(0, b.iphx, J1); take(0, b.iphy, d.y.J + 1);
    take(0, b.xcol, d.x.n); take(0, b.yrow, ny);
    take(0, b.KH, size_t(3) * d.n_grp * cols_nc(d) * (2 * d.y.J + 1));
    take(0, b.KL, 3 * kFieldLow * kLowY);
    take(1, b.KR, 3 * size_t(d.y.P / 2 + 1) * J1);
    take(1, b.FC, size_t(3) * d.y.w * J1);
    if (plan.forward) {
        take(1, b.CR, ny * (d.x.Q / 2 + 1));
        take(1, b.CL, ny * kFieldLow);
        take(1, b.FL, size_t(3) * d.y.w * kFieldLow);
        // (the outside samples' partial sums are done before the nodes are formed)
        const size_t n_part = size_t(d.n_ch) * kOutRounds * d.out_blocks * d.out_samples;
        take(1, b.FN, std::max(size_t(d.y.w) * d.x.w, (n_part + 3) / 4));
        b.fpart = reinterpret_cast<float *>(b.FN);
        take(0, b.ocount, out_counters(d));
        if (!plan.adjoint) take(1, b.olist, T1);
    }
    if (plan.adjoint) {
        take(1, b.key, T1); take(1, b.hist, nh); take(1, b.pos, nh); take(1, b.tcnt, nt + 1);
        take(0, b.list, T1); take(0, b.toff, nt + 1); take(0, b.uoff, nt + 1); take(0, b.unit_tile, d.n_unit_max);
        take(0, b.rec, T1); take(0, b.wv, T1);
        if (plan.forward) take(0, b.sd, T1);
        take(1, b.q4, T1);
        take(1, b.upart, size_t(3) * kPatchSize * d.n_unit_max);
        take(1, b.opart, size_t(d.out_chunks) * d.x.n * ny);
        take(1, b.AC, 3 * ny * J1);
        take(1, b.AL, 3 * ny * kFieldLow);
    }
    keep_bytes = tot[0];
    work_bytes = tot[1];
}

}  // namespace

int field_plan(const ModelH &m, const GridH &g, int64_t T, bool forward, bool adjoint, FieldPlan &plan)
{
    FieldDev &d = plan.d;
    d = FieldDev{};
    const double bx0 = m.beta * m.G[0], bx1 = m.beta * m.G[2], by0 = m.beta * m.G[1], by1 = m.beta * m.G[3];
    if (T < 1 || T > kFieldMaxT) return MPI_ERR_UNSUPPORTED;
    if (!plan_axis(g.nx, std::hypot(bx0, bx1) * std::fabs(g.dx), g.x0, g.dx, d.x) ||
        !plan_axis(g.ny, std::hypot(by0, by1) * std::fabs(g.dy), g.y0, g.dy, d.y))
        return MPI_ERR_UNSUPPORTED;
    d.fPx = smem_fft_plan(d.x.P);
    d.fPy = smem_fft_plan(d.y.P);
    d.fQx = smem_fft_plan(d.x.Q);
    d.fQy = smem_fft_plan(d.y.Q);
    d.T = T;
    d.tx = (d.x.w + kTile - 1) / kTile;
    d.ty = (d.y.w + kTile - 1) / kTile;
    d.run_len = (int)(std::max<int64_t>(kRunMin, (T + kRunMax - 1) / kRunMax) + 31) / 32 * 32;
    d.n_run = (int)((T + d.run_len - 1) / d.run_len);
    const int nt = d.tx * d.ty;
    d.n_unit_max = (int)(T / kFieldUnit + std::min<int64_t>(nt, T));
    const int64_t columns = (int64_t)g.nx * ((g.ny + kOutRows - 1) / kOutRows);
    d.out_tiles = (int)((columns + kOutThreads - 1) / kOutThreads);
    const int at_once = kSpreadPerSm * device_sm_count();
    d.out_chunks = std::max(1, std::min(64, (8 * d.out_tiles <= at_once ? 1 : 3) * at_once / d.out_tiles));
    d.out_blocks = std::max(1, std::min(4, kOutPerSm / cols_threads(d))) * device_sm_count();
    d.out_samples = kFwdS * cols_threads(d);
    d.n_ch = m.n_ch;
    d.diag = m.G[1] == 0.0 && m.G[2] == 0.0;
    for (int k = 0; k < 4; ++k) {
        d.p[k] = float(m.p[k]);
        split(m.beta * m.G[k], d.B[k]);
    }
    d.cx[0] = bx0 * g.dx;
    d.cx[1] = bx1 * g.dx;
    d.cy[0] = by0 * g.dy;
    d.cy[1] = by1 * g.dy;
    for (int k = 0; k < 2; ++k) {
        split(d.cx[k] * d.x.Q / d.x.P, d.hx[k]);
        split(d.cy[k] * d.y.Q / d.y.P, d.hy[k]);
    }
    d.scale = 1.0 / (double(d.x.P) * d.y.P);
    const double x = g.x0 + 0.5 * g.dx, y = g.y0 + 0.5 * g.dy;
    d.X0[0] = bx0 * x;
    d.X0[1] = bx1 * x;
    d.Y0[0] = by0 * y;
    d.Y0[1] = by1 * y;
    const int nc = cols_nc(d);
    d.n_grp = (d.x.J + nc) / nc;
    d.magQy = unsigned((int64_t(1) << 32) / d.y.Q + 1);
    if (std::max({rows_smem(d), cols_smem(d), order_smem(d)}) > 227 * 1024 - 2048)
        return MPI_ERR_UNSUPPORTED;
    plan.forward = forward;
    plan.adjoint = adjoint;
    lay_out(plan, nullptr, nullptr, plan.keep_bytes, plan.work_bytes);
    return MPI_OK;
}

void field_carve(FieldPlan &plan, void *keep, void *work)
{
    size_t k, w;
    lay_out(plan, static_cast<char *>(keep), static_cast<char *>(work), k, w);
}

int field_prepare(const FieldPlan &plan, const float *c, const float *r, const float *v, cudaStream_t st)
{
    const FieldDev &d = plan.d;
    MPI_TRY(allow_all(d, plan.forward, plan.adjoint));
    const int n_table = (table_entries(d) + 31) / 32, ow = order_warps(d);
    const int n_bin = plan.adjoint ? (d.n_run + ow - 1) / ow : 0;
    const size_t osm = plan.adjoint ? order_smem(d) : 0;
    launch_chained(k_field_setup, n_table + n_bin, 32 * ow, osm, st, d, n_table, r, v);
    MPI_CHECK_LAUNCH();
    const int kr = (d.y.P / 2 + 2) / 2, tr = fft_threads(3, d.x.P);
    const int more = c ? (d.y.n + 1) / 2 : plan.adjoint ? (d.tx * d.ty + 1 + tr / 32 - 1) / (tr / 32) : 0;
    const int list = c ? (int)((d.T + tr * kListPer - 1) / (tr * kListPer)) : 0;
    launch_chained(k_field_rows, kr + more + list, tr, rows_smem(d), st, d, kr, c, r);
    MPI_CHECK_LAUNCH();
    auto cols = cols_nc(d) == 4 ? k_field_kcols<4> : k_field_kcols<2>;
    launch_chained(cols, 3 * d.n_grp + (plan.adjoint ? 1 : 0), fft_threads(cols_nc(d), d.y.P), cols_smem(d), st, d);
    MPI_CHECK_LAUNCH();
    return MPI_OK;
}

int field_order(const FieldPlan &plan, const float *r, const float *v, const float *s, cudaStream_t st)
{
    const FieldDev &d = plan.d;
    const int ow = order_warps(d);
    launch_chained(k_field_place, (d.n_run + ow - 1) / ow, 32 * ow, order_smem(d), st, d, r, v, s);
    MPI_CHECK_LAUNCH();
    return MPI_OK;
}

int field_load(const FieldPlan &plan, const float *s, cudaStream_t st)
{
    launch_chained(k_field_load, (unsigned)((plan.d.T + 255) / 256), 256, 0, st, plan.d, s);
    MPI_CHECK_LAUNCH();
    return MPI_OK;
}

namespace {

// Image rows' spectra -> node values; the outside samples' sums.
template <int MODE, typename CIN>
int field_nodes(const FieldDev &d, const InterpArgs &A, const CIN *c, cudaStream_t st)
{
    auto cols = cols_nc(d) == 4 ? k_field_cols_fwd<4, MODE, CIN> : k_field_cols_fwd<2, MODE, CIN>;
    launch_chained(cols, std::max(3 * d.n_grp, d.out_blocks), cols_threads(d), cols_smem(d), st, d, A, c);
    MPI_CHECK_LAUNCH();
    launch_chained(k_field_rows_inv, (d.y.w + 1) / 2, fft_threads(3, d.x.P), rows_smem(d), st, d);
    MPI_CHECK_LAUNCH();
    return MPI_OK;
}

unsigned interp_blocks(const FieldDev &d) { return unsigned((d.T + kInterpThreads - 1) / kInterpThreads); }

}  // namespace

int field_forward(const FieldPlan &plan, const float *c, const float *r, const float *v, float *s, cudaStream_t st)
{
    ProfScope prof(kProfForward, st);
    MPI_TRY(field_prepare(plan, c, r, v, st));
    const InterpArgs A{r, v, s, false};
    MPI_TRY((field_nodes<kInterpForward>(plan.d, A, c, st)));
    launch_chained(k_field_interp<kInterpForward>, interp_blocks(plan.d), kInterpThreads, 0, st, plan.d, A);
    MPI_CHECK_LAUNCH();
    return MPI_OK;
}

template <typename CIN>
int field_forward_ordered(const FieldPlan &plan, const CIN *c, bool residual, cudaStream_t st)
{
    const FieldDev &d = plan.d;
    ProfScope prof(kProfForward, st);
    launch_chained(k_field_image<CIN>, (d.y.n + 1) / 2, 128, image_smem(d), st, d, c);
    MPI_CHECK_LAUNCH();
    const InterpArgs A{nullptr, nullptr, nullptr, residual};
    MPI_TRY((field_nodes<kInterpOrdered>(d, A, c, st)));
    launch_chained(k_field_interp<kInterpOrdered>, interp_blocks(d), kInterpThreads, 0, st, d, A);
    MPI_CHECK_LAUNCH();
    return MPI_OK;
}

int field_dot_blocks(int ny) { return (ny + 1) / 2; }

template <typename OUT>
int field_adjoint(const FieldPlan &plan, OUT *out, const double *cg_p, const double *nu_dev, double *dot_part,
                  cudaStream_t st)
{
    const FieldDev &d = plan.d;
    ProfScope prof(kProfAdjoint, st);
    launch_chained(k_field_spread, std::max(d.n_unit_max, kSpreadPerSm * device_sm_count()), kSpreadThreads, 0, st, d);
    MPI_CHECK_LAUNCH();
    launch_chained(k_field_rows_fwd, (d.y.w + 1) / 2, fft_threads(3, d.x.P), rows_smem(d), st, d);
    MPI_CHECK_LAUNCH();
    auto cols = cols_nc(d) == 4 ? k_field_cols_adj<4> : k_field_cols_adj<2>;
    launch_chained(cols, 3 * d.n_grp, cols_threads(d), cols_smem(d), st, d);
    MPI_CHECK_LAUNCH();
    const unsigned nb = (unsigned)field_dot_blocks(d.y.n);
    if constexpr (sizeof(OUT) == sizeof(double)) {
        if (cg_p) {
            launch_chained(k_field_out<double, true>, nb, 128, image_smem(d), st, d, out, cg_p, nu_dev, dot_part);
            MPI_CHECK_LAUNCH();
            return MPI_OK;
        }
    } else if (cg_p) {
        set_error("internal: CG epilogue needs FP64 output");
        return MPI_ERR_INVALID;
    }
    launch_chained(k_field_out<OUT, false>, nb, 128, image_smem(d), st, d, out, nullptr, nullptr, nullptr);
    MPI_CHECK_LAUNCH();
    return MPI_OK;
}

bool field_worth(const GridH &g, int64_t T) { return double(T) * g.nx * g.ny >= 1.5e7; }

// What the direct sums and the gridded operators take, in microseconds,
// fitted to GB300 timings of both at 24 x 24 to 256 x 256 voxels and 8e6 to
// 5e8 pairs (fields of view of 24 and 48 mm, three trajectories, fields along
// the axes and turned; 306 cases).  Choosing by the fit loses 1 % on average
// against the faster of the two, at most half of a call's time near the line;
// a fixed rate for the direct sums lost 13 %.
//
// A pair of the direct A^T costs by its regime, decided per sample for a
// warp's box of 16 x 16 voxels: the share of the samples within 12 z units of
// a box follows from the grid.
static double near_share(const FieldDev &d)
{
    const double px = std::hypot(d.cx[0], d.cx[1]), py = std::hypot(d.cy[0], d.cy[1]);
    return std::min(1.0, (16.0 + 24.0 / px) / d.x.n) * std::min(1.0, (16.0 + 24.0 / py) / d.y.n);
}
static double nodes_768(const FieldDev &d) { return double(d.x.P) * d.y.P / (768.0 * 768.0); }

bool field_route(const FieldPlan &plan)
{
    const FieldDev &d = plan.d;
    const double T = double(d.T), pairs = 1e-6 * T * d.x.n * d.y.n, nodes = nodes_768(d);
    if (plan.adjoint)
        return 56.0 + 35.0 * nodes + 278e-6 * T < 40.0 + pairs * ((d.diag ? 0.40 : 0.64) + 2.1 * near_share(d));
    return 53.0 + 29.0 * nodes + 44e-6 * T < 40.0 + pairs * (d.diag ? 0.51 : 1.07);
}

// A solve prepares once and applies A^T A products times in a replayed graph
// (shared: direct sums whose launches serve many frames).  15 products at
// 128 x 128 / 4000 samples: direct 2.63 ms, gridded 1.66 ms; 48 x 48 / 16 000:
// 2.48 and 1.75 ms; 64 x 64 / 8000: 1.64 and 1.62 ms; 64 x 64 / 4000: 1.16 and
// 1.60 ms.
static bool field_route_solve(const FieldPlan &plan, int64_t products, bool shared)
{
    const FieldDev &d = plan.d;
    const double T = double(d.T), pairs = 1e-6 * T * d.x.n * d.y.n, nodes = nodes_768(d);
    const double direct = (shared ? 0.0 : 55.0) + pairs * ((d.diag ? 0.77 : 1.7) + 3.0 * near_share(d));
    const double field = 82.0 + 8.0 * nodes * nodes + 100e-6 * T;
    return double(products) * (direct - field) > 60.0 + 60.0 * nodes + 400e-6 * T;
}

bool field_solve_plan(const ModelH &m, const GridH &g, int64_t T, int n_iter, int n_cg, bool shared, FieldPlan &plan)
{
    return T > 0 && field_worth(g, T) && field_plan(m, g, T, true, true, plan) == MPI_OK &&
           field_route_solve(plan, (int64_t)n_iter * (n_cg + 1), shared);
}

template int field_forward_ordered<double>(const FieldPlan &, const double *, bool, cudaStream_t);
template int field_adjoint<float>(const FieldPlan &, float *, const double *, const double *, double *, cudaStream_t);
template int field_adjoint<double>(const FieldPlan &, double *, const double *, const double *, double *, cudaStream_t);

}  // namespace mpi
