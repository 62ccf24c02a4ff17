// Internal interface of the gridded pair operators: A and A^T in FP32 as
// convolutions on a regular grid with local interpolation at the samples
// (field_ops.cu), for problems where the direct pair sums (pair_kernels.cuh)
// cost more.
#pragma once

#include "pair_ops.cuh"
#include "smem_fft.cuh"

namespace mpi {

constexpr int kFieldLow = 4;  // modes |kx|, |ky| < kFieldLow are carried in pairs of floats

// One axis of a gridded problem (z units: multiples of 1/beta G).
struct FieldAxis {
    int n;        // voxels
    int Q;        // period of the box in voxels
    int P;        // nodes of the interpolation grid per period
    int J;        // modes |k| <= J are kept
    int l0, w;    // node window [l0, l0 + w) that the samples' 8-point stencils reach
    float xlo, xhi;    // samples inside: window-relative coordinate in [xlo, xhi]
    float sc[2], of[2];  // window-relative node coordinate = r sc + of (pairs)
    float cut_inv;       // kernel cut-off erfc((|offset| - P/2) cut_inv)/2, offsets in nodes
};

// Device buffers of one gridded problem (carved from one scratch block).
struct FieldBuf {
    float2 *twPx, *twPy, *twQx, *twQy;  // exp(-2 pi i t / n)
    double *iphx, *iphy;     // 1 / window transform, k = 0 .. J (iphy: times 1/(Px Py))
    V2<float> *xcol, *yrow;  // voxel positions (samples outside the window)
    float2 *KR;      // kernel rows' half spectra [3][Py/2 + 1][Jx + 1]
    float *KH;       // kernel spectrum, scaled: [3][groups of adjacent kx][2 Jy + 1][kx in the group]
    float2 *KL;      // its lowest modes in pairs [3][kFieldLow][2 kFieldLow - 1]
    float2 *CR;      // image rows' half spectra [ny][Qx/2 + 1]
    float4 *CL;      // their lowest modes in pairs [ny][kFieldLow]
    float2 *FC;      // column-transformed half spectra [3][wy][Jx + 1]
    float2 *FL;      // what FC rounds off of its lowest modes [3][wy][kFieldLow]
    float4 *FN;      // node values (xx, xy, yy, 0) [wy][wx]
    // samples by tile (A^T and the solves)
    int *key, *hist, *pos, *tcnt;
    int *list, *toff, *uoff, *unit_tile;
    float4 *rec;     // inside: (fx, fy, node column | row << 16, 0); outside: (beta G r)
    float4 *wv;      // beta G v as pairs (hi x, hi y, lo x, lo y)
    float4 *q4;      // inside: (ux Wx, ux Wy + uy Wx, uy Wy, 0); outside: (ux, uy, 0, 0)
    float2 *sd;      // the data of a solve, both channels, in the samples' order
    float *upart;    // unit patches
    float *opart;    // outside samples' partial images
    int *ocount;     // outside samples (unordered), and per group of them the runs of rows done
    int *olist;      // the outside samples (unordered)
    float *fpart;    // their partial sums by runs of rows (in FN's memory)
    float2 *AC;      // [3][ny][Jx + 1]
    float4 *AL;      // [3][ny][kFieldLow]
};

// Everything a kernel needs to know about one gridded problem.
struct FieldDev {
    FieldAxis x, y;
    SmemFft fPx, fPy, fQx, fQy;
    FieldBuf b;
    int64_t T;
    int tx, ty;       // tiles of the node window
    int run_len, n_run;  // ordering: samples per run, runs
    int n_grp;           // groups of adjacent kx in the column transforms
    unsigned magQy;      // floor(2^32 / Qy) + 1
    int n_unit_max;
    int out_tiles, out_chunks;  // outside samples, A^T: voxel tiles, partial images
    int out_blocks, out_samples;  // and A: blocks of the column launch that sum them, samples per block
    int n_ch, diag;
    float p[4];
    float B[4][2];    // beta G as pairs
    double X0[2], Y0[2];  // beta G (x_0, 0), beta G (0, y_0) of the first voxel
    double cx[2], cy[2];  // beta G (dx, 0), beta G (0, dy): one voxel's step in z units
    float hx[2][2], hy[2][2];  // one node's step in z units, as pairs
    double scale;         // 1 / (Px Py)
};

// Whether a problem is large enough to plan (host, microseconds).
bool field_worth(const GridH &g, int64_t T);

struct FieldPlan {
    FieldDev d;
    size_t keep_bytes = 0, work_bytes = 0;
    bool forward = false, adjoint = false;  // which buffers it lays out
};
// Fills plan.d's sizes and the bytes of scratch it needs (adjoint: also for
// the sample order); MPI_ERR_UNSUPPORTED when the box or its transforms would
// be too large.  field_carve points the buffers into the scratch: keep_bytes
// hold a prepared plan, work_bytes serve one preparation or application (plans
// used one after another on one stream may share them).  Both 256-aligned.
int field_plan(const ModelH &m, const GridH &g, int64_t T, bool forward, bool adjoint, FieldPlan &plan);
void field_carve(FieldPlan &plan, void *keep, void *work);
// Whether one call on this plan costs less than the direct sums.
bool field_route(const FieldPlan &plan);
// The plan (both directions) of a PnP solve with A, if it costs less than the
// direct sums over the solve's n_iter (n_cg + 1) products A^T A (shared: sums
// whose launches serve many frames).
bool field_solve_plan(const ModelH &m, const GridH &g, int64_t T, int n_iter, int n_cg, bool shared, FieldPlan &plan);

// Tables and the kernel spectrum; with an adjoint plan also the first half of the sample order (r, v); c: the
// rows of an image for the forward operator (plans without adjoint).
int field_prepare(const FieldPlan &plan, const float *c, const float *r, const float *v, cudaStream_t st);
// The second half of the sample order, after field_prepare; with s
// ([n_ch][T]) also loads it as the operand of field_adjoint.
int field_order(const FieldPlan &plan, const float *r, const float *v, const float *s, cudaStream_t st);
// Keeps s ([n_ch][T]) as the data of a solve (plans with both directions).
int field_load(const FieldPlan &plan, const float *s, cudaStream_t st);
// One call: s = A c on the unordered trajectory (a forward plan, not prepared).
int field_forward(const FieldPlan &plan, const float *c, const float *r, const float *v, float *s, cudaStream_t st);
// The operand of field_adjoint set to A c on the ordered samples, or with
// residual to the solve's data minus A c.
template <typename CIN>
int field_forward_ordered(const FieldPlan &plan, const CIN *c, bool residual, cudaStream_t st);
// out = A^T of the loaded operand (OUT float or double); with cg_p: out +=
// nu cg_p (OUT double) and field_dot_blocks partial sums of <cg_p, out>.
template <typename OUT>
int field_adjoint(const FieldPlan &plan, OUT *out, const double *cg_p, const double *nu_dev, double *dot_part,
                  cudaStream_t st);
int field_dot_blocks(int ny);
}  // namespace mpi
