// Forward kernels: x*f for a shared pid list (matrix form), for one pid per
// point (pointwise form), alpha_s, and the host-buffer pipeline.
//
// PDFFlow Sec. 2.1: the query is a flavour set plus equal-length arrays of x
// and Q; the answer is one interpolated value per point and flavour.
#include <math.h>
#include <stdlib.h>

#include <algorithm>

#include "pdf_internal.h"
#include "sort_acc.cuh"
#include "warp_eval.cuh"

using namespace pdfgpu;

namespace {

constexpr int kBlock = 256;

// Matrix form.  A warp's task is 32 consecutive points and one group of `per`
// consecutive columns (all of them, one group, in long queries), taken
// grid-stride; the work of a task is eval_points (warp_eval.cuh).  With all
// columns in one group the rows of 32 points leave as one contiguous run.
// STAGE: the block first copies the coordinate tables into shared memory.
// TAPE: each point's adjoint tape record is written as well; AS: alpha_s at
// the point's Q^2 goes to as_out[i] (a point whose x alone is out of the
// domain still gets its alpha_s, as alphasQ2 would give it).
template <bool Q_IS_Q, bool TAPE, bool AS, bool STAGE, bool WHOLE>
__global__ void __launch_bounds__(kBlock, WHOLE ? 3 : 2) k_xfxq2(const __grid_constant__ GridDev g,
                                                     const __grid_constant__ Cols cols, int npid, int per, int groups,
                                                     int member, const double *__restrict__ x,
                                                     const double *__restrict__ q, int64_t n,
                                                     double *__restrict__ out, double *__restrict__ tape,
                                                     double *__restrict__ as_out, int tab_bytes, int warp_bytes)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const CoordTabs T = STAGE ? stage_tabs(g, smem) : grid_tabs(g);
    __syncthreads();
    const int lane = lane_id(), wid = threadIdx.x >> 5;
    unsigned char *mine = smem + tab_bytes + (size_t)wid * warp_bytes;
    WarpBufs B{reinterpret_cast<uint4 *>(mine), reinterpret_cast<int64_t *>(mine + warp_bytes - kQueue * 8), 0};
    const size_t patches = (size_t)member * g.nqc * g.nxc * g.nflav;
    Query Y{cols.c, npid, 0, npid, g.coef + patches * 16,
            g.fcoef ? reinterpret_cast<const unsigned char *>(g.fcoef) + patches * 128 : nullptr,
            x, q, n, out, tape, as_out};
    const int64_t tasks = (n + 31) / 32 * groups;
    const int64_t stride = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + wid; t < tasks; t += stride) {
        int64_t base = t * 32;
        if (!WHOLE) {
            const int64_t blk = t / groups;
            Y.a0 = (int)(t - blk * groups) * per;
            Y.a1 = min(npid, Y.a0 + per);
            base = blk * 32;
        }
        eval_points<Q_IS_Q, TAPE, AS, WHOLE>(g, T, Y, B, base, lane);
        if (!WHOLE && B.qn) drain_queue(g, T, Y, Q_IS_Q, B, lane);
    }
    if (WHOLE)
        while (B.qn) drain_queue(g, T, Y, Q_IS_Q, B, lane);
    if (lane == 0) bulk_wait_all();
}

// One point of the pointwise form in FP64.
__device__ __forceinline__ void slow_point_pw(const GridDev &g, const double *cm, const unsigned char *fm, int col,
                                              double xi, double qi, int64_t i, double *out, double *tape,
                                              double *dtape, int *dbins, int nbins)
{
    bool bad = !(x_ok(dbits(xi)) && q2_ok(dbits(qi)));
    flag_status(g, bad);
    if (bad) {
        xi = 0.5;
        qi = 10.0;
    }
    const Axis X = axis_x(g, xi), Q = axis_q2(g, qi);
    const bool oor = out_of_range(g, X, Q);
    flag_status(g, oor, PDF_S_RANGE);
    bad |= oor;
    if (tape) tape_put(tape, i, X, Q, bad);
    const size_t p = ((size_t)Q.cell * g.nxc + X.cell) * g.nflav + (col >= 0 ? col : 0);
    const double *C = cm + p * 16;
    double v = 0.0;
    if (dtape) {
        double dtx = 0.0, dtq = 0.0;
        if (col >= 0) {
            v = patch(C, X, Q);
            patch_d(C, fm ? fm + p * 128 : nullptr, X, Q, &dtx, &dtq);
            const ChainFactors f = chain_factors(g, X.cell, Q.cell, xi, qi);
            dtx *= f.x;
            dtq *= f.q;
        }
        reinterpret_cast<double2 *>(dtape)[i] = make_double2(dtx, dtq);
        dbins[i] = sorted_bin(g, X, Q, bad, col, half_pair(X, Q), nbins);
    } else if (col >= 0) {
        v = patch_any<true>(g, C, X, Q);
    }
    out[i] = bad ? dnan() : v;
}

// Pointwise form: one flavour per point.  DT (with TAPE): also keep each point's
// derivatives in x and Q^2, computed with the value from the same rows
// (quad_patch_d) and taken through the chain rule here, where the FP64 pipe is
// idle, in dtape[i] = (dP/dx, dP/dQ^2) (zeros for an absent pid), and the
// point's bin in the pointwise sorted adjoint in dbins[i] (-1 for none).
// Five blocks of 128 threads per SM, at 96 registers (with both tapes 160 bytes
// of them spilled, 104 with one, 100 plain): 1351 us per pointwise fit step; two
// blocks of 256 1364, six of 128, which spill more, 1385.  With the rules of
// fix_limit 1360.
constexpr int kPwBlock = 128;

template <bool TAPE, bool DT, bool STAGE>
__global__ void __launch_bounds__(kPwBlock, 5) k_xfxq2_pw(const __grid_constant__ GridDev g, int member,
                                                        const int *__restrict__ pid,
                                                        const double *__restrict__ x,
                                                        const double *__restrict__ q2,
                                                        int64_t n, double *__restrict__ out,
                                                        double *__restrict__ tape, double *__restrict__ dtape,
                                                        int *__restrict__ dbins, int nbins, int tab_bytes)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const CoordTabs T = STAGE ? stage_tabs(g, smem) : grid_tabs(g);
    __syncthreads();
    const int lane = lane_id(), wid = threadIdx.x >> 5;
    unsigned char *mine = smem + tab_bytes + (size_t)wid * (kWarpBuf + kQueue * 8);
    WarpBufs B{reinterpret_cast<uint4 *>(mine), reinterpret_cast<int64_t *>(mine + kWarpBuf), 0};
    const size_t patches = (size_t)member * g.nqc * g.nxc * g.nflav;
    const double *cm = g.coef + patches * 16;
    const unsigned char *fm = g.fcoef ? reinterpret_cast<const unsigned char *>(g.fcoef) + patches * 128 : nullptr;
    auto drain = [&]() {
        const Queued e = next_queued(B, lane);
        const int64_t i = e.i;
        if (i >= 0 && e.sub == 0)
            slow_point_pw(g, cm, fm, pid_col(g, pid[i]), x[i], q2[i], i, out, tape, dtape, dbins, nbins);
        __syncwarp();
    };
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = ((int64_t)blockIdx.x * (blockDim.x >> 5) + wid) * 32; base < n; base += stride) {
        const int64_t i = base + lane;
        const bool live = i < n;
        const double xi = live ? x[i] : 0.5, qi = live ? q2[i] : 10.0;
        const int col = live ? pid_col(g, pid[i]) : -1;
        // inside the knots, so inside the domain (32 points outside: no coordinates)
        bool fast = live && in_x(g, dbits(xi)) && in_q2(g, dbits(qi)) && fm;
        if (__any_sync(kAll, fast)) {
            const FixAxis X = fix_axis_x(g, T, dbits(xi)), Q = fix_axis_q2(g, T, dbits(qi));
            fast = fast && X.ok && Q.ok;
            const uint32_t patch0 =
                fast ? (uint32_t)(Q.cell * g.nxc + X.cell) * (uint32_t)g.nflav + (col >= 0 ? col : 0) : 0u;
            uint32_t off[4];
            quad_offsets(patch0 * 128u, lane, off);
            Dig W[4][4];
            quad_weights(B.buf, lane, fast ? X.t : kFixHalf, fast ? Q.t : kFixHalf, W);
            int c[4][8], last;
            quad_load(fm, off, c);
            const int64_t s = quad_patch(c, W, quad_pos(lane), last);
            fast &= col < 0 || !fix_needs_fp64(last, fix_limit(X.t, Q.t));
            if (fast) {
                out[i] = col >= 0 ? fix_value(s, last) : 0.0;
                if (TAPE) tape_put(tape, i, X, Q);
            }
            if (DT) {
                int64_t dx, dq;
                quad_patch_d(c, W, B.buf, lane, quad_pos(lane), dx, dq);
                double dtx = col >= 0 ? fix_value(dx, last) : 0.0, dtq = col >= 0 ? fix_value(dq, last) : 0.0;
                const bool knot = fast && col >= 0 && (fix_at_knot(X.t) || fix_at_knot(Q.t));
                if (__any_sync(kAll, knot) && knot) {            // rare: the derivatives at a knot in FP64 (patch_d)
                    Axis AX, AQ;
                    AX.in = AQ.in = true;
                    AX.below = AQ.below = false;
                    make_basis(AX, fix_t(X.t), g.extrap);
                    make_basis(AQ, fix_t(Q.t), g.extrap);
                    patch_vd(cm + (size_t)patch0 * 16, AX, AQ, &dtx, &dtq);
                }
                if (fast) {
                    const ChainFactors f = chain_factors(g, X.cell, Q.cell, xi, qi);
                    reinterpret_cast<double2 *>(dtape)[i] = make_double2(dtx * f.x, dtq * f.q);
                    const int halves = (upper_half(X.t) ? 1 : 0) | (upper_half(Q.t) ? 2 : 0);
                    dbins[i] = col < 0 ? -1 : checked_index(g.status, (int)patch0 * 4 + halves, nbins);   // sorted_bin's
                }
            }
        }
        push_queue(B, live && !fast, i, lane);
        if (B.qn >= 32) drain();
    }
    if (B.qn) drain();
}

// alpha_s, one point per lane (fix_alphas): 1e7 points 286 -> 93 us (FP64
// pipe 82 % busy before; now 56 % of the issue slots, the logarithm and the table
// look-ups in shared memory); points outside the Q range or the
// domain are queued per warp and evaluated 32 at a time.
// STAGE: the block's copy of the Q tables and of the cubics (as chunks of 16
// bytes, the first of all cells before the second) in shared memory.
__host__ __device__ inline int alphas_tab_bytes(const GridDev &g)
{
    return (g.nqc * 56 + kGuideRun * 8 + kLogTab * 12 + g.nqg * 2 + 127) & ~127;
}

template <bool Q_IS_Q, bool STAGE>
__global__ void __launch_bounds__(kBlock) k_alphas(const __grid_constant__ GridDev g, const double *__restrict__ q,
                                                   int64_t n, double *__restrict__ out)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int64_t squeue[kBlock / 32][kQueue];
    uint4 *rows = reinterpret_cast<uint4 *>(smem);
    FixCell *cells = reinterpret_cast<FixCell *>(rows + 2 * g.nqc);
    int64_t *logs = reinterpret_cast<int64_t *>(cells + g.nqc);
    uint64_t *keys = reinterpret_cast<uint64_t *>(logs + kLogTab);
    uint32_t *invs = reinterpret_cast<uint32_t *>(keys + g.nqc + kGuideRun);
    uint16_t *guide = reinterpret_cast<uint16_t *>(invs + kLogTab);
    if (STAGE) {
        for (int k = threadIdx.x; k < 2 * g.nqc; k += blockDim.x)
            rows[(k & 1) * g.nqc + (k >> 1)] = reinterpret_cast<const uint4 *>(g.facoef)[k];
        for (int k = threadIdx.x; k < g.nqc; k += blockDim.x) cells[k] = g.qfix[k];
        for (int k = threadIdx.x; k < g.nqc + kGuideRun; k += blockDim.x) keys[k] = g.qbits[k];
        for (int k = threadIdx.x; k < g.nqg; k += blockDim.x) guide[k] = g.qguide[k];
        for (int k = threadIdx.x; k < kLogTab; k += blockDim.x) {
            logs[k] = g.flog[k];
            invs[k] = g.finv[k];
        }
        __syncthreads();
    }
    const CoordTabs T = STAGE ? CoordTabs{invs, logs, nullptr, keys, nullptr, guide, nullptr, cells} : grid_tabs(g);
    const int lane = lane_id(), wid = threadIdx.x >> 5;
    WarpBufs B{nullptr, squeue[wid], 0};
    auto drain = [&]() {
        const Queued e = next_queued(B, lane);
        const int64_t i = e.i;
        if (i >= 0 && e.sub == 0) {
            double qi = q[i];
            if (Q_IS_Q) qi = qi * qi;
            const bool bad = !q2_ok(dbits(qi));
            flag_status(g, bad);
            bool oor;
            const double v = alphas_at(g, axis_q2(g, T, bad ? 10.0 : qi), &oor);
            flag_status(g, oor && !bad, PDF_S_RANGE);
            out[i] = bad ? dnan() : v;
        }
        __syncwarp();
    };
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = ((int64_t)blockIdx.x * (blockDim.x >> 5) + wid) * 32; base < n; base += stride) {
        const int64_t i = base + lane;
        const bool live = i < n;
        double qi = live ? q[i] : 10.0;
        if (Q_IS_Q) qi = qi * qi;
        const FixAxis Q = fix_axis_q2(g, T, dbits(qi));
        bool fast = live && Q.ok;                    // inside the knots, so inside the domain
        int c[8];
        if (STAGE) {
            const uint4 a = rows[Q.cell], b = rows[g.nqc + Q.cell];
            c[0] = a.x, c[1] = a.y, c[2] = a.z, c[3] = a.w, c[4] = b.x, c[5] = b.y, c[6] = b.z, c[7] = b.w;
        } else {
            fix_ld(reinterpret_cast<const unsigned char *>(g.facoef) + (size_t)Q.cell * 32, c);
        }
        bool none;
        const double v = fix_alphas(c, Q.t, none);
        fast &= !none;
        if (fast) out[i] = v;
        push_queue(B, live && !fast, i, lane);
        if (B.qn >= 32) drain();
    }
    if (B.qn) drain();
}

// alpha_s and d alpha_s / d Q^2 = (da/dtq) / dW / Q^2 (zero across a frozen edge).
__global__ void __launch_bounds__(kBlock) k_alphas_grad(GridDev g, const double *__restrict__ q2, int64_t n,
                                                        double *__restrict__ out, double *__restrict__ dq2)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        double qi = q2[i];
        bool bad = !q2_ok(dbits(qi));
        flag_status(g, bad);
        if (bad) qi = 10.0;
        const Axis Q = axis_q2(g, qi);
        bool oor;
        const double v = alphas_at(g, Q, &oor);
        flag_status(g, oor, PDF_S_RANGE);
        bad |= oor;
        const D4 a = ld4(g.acoef + (size_t)Q.cell * 4);
        double d2 = Q.in ? 2.0 * Q.t : 1.0, d3 = Q.in ? 3.0 * Q.t * Q.t : 1.0;
        double dt = fma(d3, a.w, fma(d2, a.z, a.y));
        if (!Q.in && g.extrap == PDF_EXTRAP_FREEZE) dt = 0.0;
        if (!Q.in && g.extrap == PDF_EXTRAP_CONTINUATION) {
            // d/dt of the continuation from the edge values y0 = a(0), y1 = a(1)
            const double y0 = a.x, y1 = a.x + a.y + a.z + a.w;
            dt = (y0 > kContMin && y1 > kContMin) ? v * log(y1 / y0) : y1 - y0;
        }
        if (out) out[i] = bad ? dnan() : v;
        dq2[i] = bad ? dnan() : dt * g.qcell[Q.cell].y * __drcp_rn(qi);
    }
}

// The cells the kernels' knot searches give (x, Q^2 given as bit patterns;
// the guide table when the grid has one): a test hook.
__global__ void k_cells(GridDev g, const double *__restrict__ x, const double *__restrict__ q2, int64_t n,
                        int *__restrict__ xc, int *__restrict__ qc)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        xc[i] = axis_x(g, x[i]).cell;
        qc[i] = axis_q2(g, q2[i]).cell;
    }
}

__global__ void k_log(GridDev g, const double *__restrict__ in, int64_t n, double *__restrict__ out)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = dlog(g, in[i]);
}

// A tape is only written for the adjoint's grids (not under the power-law
// continuation, which has no adjoint) and must allow 32-byte loads.
int check_tape(const pdfgpu_grid *g, const double *tape)
{
    if (!tape) return PDF_OK;
    if (g->d.extrap == PDF_EXTRAP_CONTINUATION)
        return fail(PDF_E_ARG, "no adjoint tape under the power-law continuation (the adjoint needs linear, "
                               "freeze or error extrapolation)");
    if ((uintptr_t)tape % 32) return fail(PDF_E_ARG, "tape must be 32-byte aligned");
    return PDF_OK;
}

// The matrix form's launch.  A long query gives each warp all the columns of
// 32 points.  A short one splits the columns into groups until there are
// about kShortWarps warps per SM: below that the SMs wait for one warp's
// chain of loads, and the coordinates computed once per group are cheaper
// than idle SMs (1e5 points x 11 flavours with alpha_s: 22 us; 43 us in FP64).
constexpr int kShortWarps = 16;
// Points per SM from which copying the coordinate tables into shared memory
// pays (the copy is about 20 KB per block).
constexpr int64_t kStagePoints = 256;
constexpr size_t kStageMax = 48 * 1024;      // the tables of larger grids stay global

template <bool Q_IS_Q, bool TAPE, bool AS>
int launch_points(pdfgpu_grid *g, int32_t member, const Cols &cols, int n_pid, const double *x, const double *q,
                  int64_t n, double *out, double *tape, double *alphas, cudaStream_t s)
{
    using Kern = void (*)(const GridDev, const Cols, int, int, int, int, const double *, const double *, int64_t,
                          double *, double *, double *, int, int);
    const int64_t blocks32 = (n + 31) / 32;
    int groups = 1, per = n_pid;
    if (blocks32 < (int64_t)kShortWarps * g->sm_count) {
        groups = (int)std::min<int64_t>(n_pid, (int64_t)kShortWarps * g->sm_count / blocks32);
        per = (n_pid + groups - 1) / groups;
        groups = (n_pid + per - 1) / per;
    }
    int tab = coord_tab_bytes(g->d);
    const bool stage = n >= kStagePoints * g->sm_count && (size_t)tab <= kStageMax;
    if (!stage) tab = 0;
    const Kern k = groups > 1 ? (stage ? k_xfxq2<Q_IS_Q, TAPE, AS, true, false>
                                       : k_xfxq2<Q_IS_Q, TAPE, AS, false, false>)
                              : (stage ? k_xfxq2<Q_IS_Q, TAPE, AS, true, true>
                                       : k_xfxq2<Q_IS_Q, TAPE, AS, false, true>);
    const int warp_bytes = (groups > 1 ? kWarpBuf : std::max(kWarpBuf, 32 * 8 * n_pid)) + kQueue * 8;
    // 256-thread blocks share one copy of the tables; a short query or wide
    // rows take smaller blocks, which spread more evenly over the SMs
    int block = kBlock;
    while (block > 32 && ((size_t)tab + (size_t)(block / 32) * warp_bytes > 75 * 1024 ||
                          (!stage && blocks32 * groups < (int64_t)(block / 32) * 2 * g->sm_count)))
        block /= 2;
    const size_t smem = (size_t)tab + (size_t)(block / 32) * warp_bytes;
    int rc = allow_dynamic_smem((const void *)k, smem);
    if (rc) return rc;
    const int grid = wave_grid(g, (const void *)k, block, smem, blocks32 * groups * 32);
    k<<<grid, block, smem, s>>>(g->d, cols, n_pid, per, groups, member, x, q, n, out, tape, alphas, tab, warp_bytes);
    PDF_CUDA(cudaGetLastError());
    return PDF_OK;
}

int launch_matrix(pdfgpu_grid *g, int32_t member, const int32_t *pids, int32_t n_pid,
                  const double *x, const double *q, int64_t n, double *out, double *tape, cudaStream_t s,
                  bool q_is_q)
{
    clear_error();
    int rc = check_grid(g, true);
    if (rc) return rc;
    if (n < 0) return fail(PDF_E_ARG, "negative n");
    if (member < 0 || member >= g->d.nmem) return fail(PDF_E_ARG, "member out of range");
    Cols cols;
    rc = resolve_cols(g, pids, n_pid, &cols);
    if (rc) return rc;
    rc = check_tape(g, tape);
    if (rc) return rc;
    if (n == 0) return PDF_OK;
    if (!x || !q || !out) return fail(PDF_E_ARG, "null array");
    auto launch = tape     ? launch_points<false, true, false>
                  : q_is_q ? launch_points<true, false, false>
                           : launch_points<false, false, false>;
    return launch(g, member, cols, n_pid, x, q, n, out, tape, nullptr, s);
}

// x*f and alpha_s at the same points in one launch.
int launch_xf_alphas(pdfgpu_grid *g, int32_t member, const int32_t *pids, int32_t n_pid, const double *x,
                     const double *q2, int64_t n, double *out, double *alphas, cudaStream_t s)
{
    clear_error();
    int rc = check_grid(g, true);
    if (rc) return rc;
    if (!g->has_alphas) return fail(PDF_E_DESC, "grid has no alpha_s values");
    if (n < 0) return fail(PDF_E_ARG, "negative n");
    if (member < 0 || member >= g->d.nmem) return fail(PDF_E_ARG, "member out of range");
    Cols cols;
    rc = resolve_cols(g, pids, n_pid, &cols);
    if (rc) return rc;
    if (n == 0) return PDF_OK;
    if (!x || !q2 || !out || !alphas) return fail(PDF_E_ARG, "null array");
    return launch_points<false, false, true>(g, member, cols, n_pid, x, q2, n, out, nullptr, alphas, s);
}

int launch_alphas(pdfgpu_grid *g, const double *q, int64_t n, double *out, cudaStream_t s, bool q_is_q)
{
    clear_error();
    int rc = check_grid(g, false);
    if (rc) return rc;
    if (!g->has_alphas) return fail(PDF_E_DESC, "grid has no alpha_s values");
    if (n < 0) return fail(PDF_E_ARG, "negative n");
    if (n == 0) return PDF_OK;
    if (!q || !out) return fail(PDF_E_ARG, "null array");
    int tab = alphas_tab_bytes(g->d);
    const bool stage = n >= kStagePoints * g->sm_count && (size_t)tab <= 32 * 1024;
    if (!stage) tab = 0;
    auto k = q_is_q ? (stage ? k_alphas<true, true> : k_alphas<true, false>)
                    : (stage ? k_alphas<false, true> : k_alphas<false, false>);
    k<<<wave_grid(g, (const void *)k, kBlock, tab, n), kBlock, tab, s>>>(g->d, q, n, out);
    PDF_CUDA(cudaGetLastError());
    return PDF_OK;
}

int launch_pw(pdfgpu_grid *g, int32_t member, const int32_t *pid, const double *x, const double *q2, int64_t n,
              double *out, double *tape, double *dtape, cudaStream_t s)
{
    clear_error();
    int rc = check_grid(g, true);
    if (rc) return rc;
    if (n < 0) return fail(PDF_E_ARG, "negative n");
    if (member < 0 || member >= g->d.nmem) return fail(PDF_E_ARG, "member out of range");
    rc = check_tape(g, tape);
    if (rc) return rc;
    if (dtape && !tape) return fail(PDF_E_ARG, "a derivative tape goes with a tape");
    if (dtape && (uintptr_t)dtape % 16) return fail(PDF_E_ARG, "derivative tape must be 16-byte aligned");
    const int64_t nbins64 = (int64_t)g->d.nqc * g->d.nxc * g->d.nflav * 4;   // the pointwise adjoint's bins
    if (dtape && nbins64 >= (int64_t)1 << 30) return fail(PDF_E_RANGE, "grid too large for the derivative tape");
    if (n == 0) return PDF_OK;
    if (!pid || !x || !q2 || !out) return fail(PDF_E_ARG, "null array");
    int tab = coord_tab_bytes(g->d);
    const bool stage = n >= kStagePoints * g->sm_count && (size_t)tab <= kStageMax;
    if (!stage) tab = 0;
    auto k = dtape  ? (stage ? k_xfxq2_pw<true, true, true> : k_xfxq2_pw<true, true, false>)
             : tape ? (stage ? k_xfxq2_pw<true, false, true> : k_xfxq2_pw<true, false, false>)
                    : (stage ? k_xfxq2_pw<false, false, true> : k_xfxq2_pw<false, false, false>);
    const size_t smem = (size_t)tab + (kPwBlock / 32) * (kWarpBuf + kQueue * 8);
    rc = allow_dynamic_smem((const void *)k, smem);
    if (rc) return rc;
    int grid = wave_grid(g, (const void *)k, kPwBlock, smem, n);
    int *dbins = dtape ? reinterpret_cast<int *>(dtape + 2 * n) : nullptr;
    k<<<grid, kPwBlock, smem, s>>>(g->d, member, pid, x, q2, n, out, tape, dtape, dbins,
                                 (int)std::min<int64_t>(nbins64, (int64_t)1 << 30), tab);
    PDF_CUDA(cudaGetLastError());
    return PDF_OK;
}

}  // namespace

extern "C" int xfxQ2_alphasQ2(pdfgpu_grid_t g, int32_t member, const int32_t *pids, int32_t n_pid,
                              const double *x, const double *q2, int64_t n, double *out, double *alphas,
                              pdfgpu_stream_t stream)
{
    PDF_TRACE("xfxQ2_alphasQ2");
    return launch_xf_alphas(g, member, pids, n_pid, x, q2, n, out, alphas, (cudaStream_t)stream);
}

extern "C" int xfxQ2(pdfgpu_grid_t g, int32_t member, const int32_t *pids, int32_t n_pid,
                     const double *x, const double *q2, int64_t n, double *out, pdfgpu_stream_t stream)
{
    PDF_TRACE("xfxQ2");
    return launch_matrix(g, member, pids, n_pid, x, q2, n, out, nullptr, (cudaStream_t)stream, false);
}

extern "C" int xfxQ(pdfgpu_grid_t g, int32_t member, const int32_t *pids, int32_t n_pid,
                    const double *x, const double *q, int64_t n, double *out, pdfgpu_stream_t stream)
{
    PDF_TRACE("xfxQ");
    return launch_matrix(g, member, pids, n_pid, x, q, n, out, nullptr, (cudaStream_t)stream, true);
}

extern "C" int xfxQ2_pw(pdfgpu_grid_t g, int32_t member, const int32_t *pid, const double *x,
                        const double *q2, int64_t n, double *out, pdfgpu_stream_t stream)
{
    PDF_TRACE("xfxQ2_pw");
    return launch_pw(g, member, pid, x, q2, n, out, nullptr, nullptr, (cudaStream_t)stream);
}

extern "C" int xfxQ2_tape(pdfgpu_grid_t g, int32_t member, const int32_t *pids, int32_t n_pid,
                          const double *x, const double *q2, int64_t n, double *out, double *tape,
                          pdfgpu_stream_t stream)
{
    PDF_TRACE("xfxQ2_tape");
    if (!tape && n != 0) {
        clear_error();
        return fail(PDF_E_ARG, "null tape");
    }
    return launch_matrix(g, member, pids, n_pid, x, q2, n, out, tape, (cudaStream_t)stream, false);
}

extern "C" int xfxQ2_pw_tape(pdfgpu_grid_t g, int32_t member, const int32_t *pid, const double *x,
                             const double *q2, int64_t n, double *out, double *tape, double *dtape,
                             pdfgpu_stream_t stream)
{
    PDF_TRACE("xfxQ2_pw_tape");
    if (!tape && n != 0) {
        clear_error();
        return fail(PDF_E_ARG, "null tape");
    }
    return launch_pw(g, member, pid, x, q2, n, out, tape, dtape, (cudaStream_t)stream);
}

extern "C" int alphasQ2(pdfgpu_grid_t g, const double *q2, int64_t n, double *out, pdfgpu_stream_t stream)
{
    PDF_TRACE("alphasQ2");
    return launch_alphas(g, q2, n, out, (cudaStream_t)stream, false);
}

extern "C" int alphasQ(pdfgpu_grid_t g, const double *q, int64_t n, double *out, pdfgpu_stream_t stream)
{
    PDF_TRACE("alphasQ");
    return launch_alphas(g, q, n, out, (cudaStream_t)stream, true);
}

extern "C" int alphasQ2_grad(pdfgpu_grid_t g, const double *q2, int64_t n, double *out, double *dq2,
                             pdfgpu_stream_t stream)
{
    PDF_TRACE("alphasQ2_grad");
    clear_error();
    int rc = check_grid(g, false);
    if (rc) return rc;
    if (!g->has_alphas) return fail(PDF_E_DESC, "grid has no alpha_s values");
    if (n < 0) return fail(PDF_E_ARG, "negative n");
    if (n == 0) return PDF_OK;
    if (!q2 || !dq2) return fail(PDF_E_ARG, "null array");
    int grid = wave_grid(g, (const void *)k_alphas_grad, kBlock, 0, n);
    k_alphas_grad<<<grid, kBlock, 0, (cudaStream_t)stream>>>(g->d, q2, n, out, dq2);
    PDF_CUDA(cudaGetLastError());
    return PDF_OK;
}

extern "C" int pdf_debug_log(pdfgpu_grid_t g, const double *in, int64_t n, double *out,
                             pdfgpu_stream_t stream)
{
    PDF_TRACE("pdf_debug_log");
    clear_error();
    int rc = check_grid(g, false);
    if (rc) return rc;
    if (n < 0) return fail(PDF_E_ARG, "negative n");
    if (n == 0) return PDF_OK;
    if (!in || !out) return fail(PDF_E_ARG, "null array");
    int grid = wave_grid(g, (const void *)k_log, kBlock, 0, n);
    k_log<<<grid, kBlock, 0, (cudaStream_t)stream>>>(g->d, in, n, out);
    PDF_CUDA(cudaGetLastError());
    return PDF_OK;
}

extern "C" int pdf_debug_cells(pdfgpu_grid_t g, const double *x, const double *q2, int64_t n, int32_t *x_cell,
                               int32_t *q_cell, int32_t *guided, pdfgpu_stream_t stream)
{
    PDF_TRACE("pdf_debug_cells");
    clear_error();
    int rc = check_grid(g, false);
    if (rc) return rc;
    if (n < 0) return fail(PDF_E_ARG, "negative n");
    if (guided) {
        guided[0] = g->d.nxg > 0;
        guided[1] = g->d.nqg > 0;
    }
    if (n == 0) return PDF_OK;
    if (!x || !q2 || !x_cell || !q_cell) return fail(PDF_E_ARG, "null array");
    int grid = wave_grid(g, (const void *)k_cells, kBlock, 0, n);
    k_cells<<<grid, kBlock, 0, (cudaStream_t)stream>>>(g->d, x, q2, n, x_cell, q_cell);
    PDF_CUDA(cudaGetLastError());
    return PDF_OK;
}

// Host buffers: chunks of points flow through three device staging slots on
// three internal streams, so the copy-in of one chunk, the kernel of the
// next and the copy-out of a third overlap.
extern "C" int xfxQ2_host(pdfgpu_grid_t g, int32_t member, const int32_t *pids, int32_t n_pid,
                          const double *x, const double *q2, int64_t n, double *out)
{
    PDF_TRACE("xfxQ2_host");
    clear_error();
    int rc = check_grid(g, true);
    if (rc) return rc;
    if (n < 0) return fail(PDF_E_ARG, "negative n");
    if (n_pid < 1 || n_pid > PDF_MAX_PIDS) return fail(PDF_E_RANGE, "bad pid count");
    if (n == 0) return PDF_OK;
    if (!x || !q2 || !out) return fail(PDF_E_ARG, "null array");
    std::lock_guard<std::mutex> lock(g->host_mu);
    // points per chunk: small enough that the pipeline fills quickly (the
    // device-to-host copy of the outputs is the bound), large enough to fill
    // the GPU; $PDFGPU_HOST_CHUNK overrides it
    static const int64_t chunk_pts = [] {
        const char *e = getenv("PDFGPU_HOST_CHUNK");
        long long v = e ? atoll(e) : 0;
        return (int64_t)(v >= 4096 ? v : (1 << 18));
    }();
    const int64_t chunk = std::min<int64_t>(n, chunk_pts);
    if (g->stage_pts < chunk || g->stage_pid < n_pid) {
        for (int s = 0; s < 3; ++s)
            for (int k = 0; k < 3; ++k) {
                if (g->stage[s][k]) cudaFree(g->stage[s][k]);
                g->stage[s][k] = nullptr;
            }
        int64_t pts = std::max<int64_t>(chunk, g->stage_pts);
        int np = std::max(n_pid, g->stage_pid);
        for (int s = 0; s < 3; ++s) {
            if (dev_malloc((void **)&g->stage[s][0], pts * sizeof(double), "host-path staging") ||
                dev_malloc((void **)&g->stage[s][1], pts * sizeof(double), "host-path staging") ||
                dev_malloc((void **)&g->stage[s][2], pts * np * sizeof(double), "host-path staging"))
                return PDF_E_NOMEM;
        }
        g->stage_pts = pts;
        g->stage_pid = np;
    }
    for (int s = 0; s < 3; ++s)
        if (!g->hs[s]) PDF_CUDA(cudaStreamCreateWithFlags(&g->hs[s], cudaStreamNonBlocking));
    // on any failure, copies already queued are drained before returning, so
    // that none of them touches the caller's buffers after the call
    auto drain = [&](int code) {
        for (int s = 0; s < 3; ++s) cudaStreamSynchronize(g->hs[s]);
        return code;
    };
    int64_t nchunks = (n + chunk - 1) / chunk;
    for (int64_t c = 0; c < nchunks; ++c) {
        int s = (int)(c % 3);
        cudaStream_t st = g->hs[s];
        int64_t off = c * chunk, m = std::min(chunk, n - off);
        cudaError_t e = cudaMemcpyAsync(g->stage[s][0], x + off, m * sizeof(double), cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(g->stage[s][1], q2 + off, m * sizeof(double), cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return drain(cuda_fail(e, "host-to-device copy"));
        rc = launch_matrix(g, member, pids, n_pid, g->stage[s][0], g->stage[s][1], m, g->stage[s][2], nullptr, st, false);
        if (rc) return drain(rc);
        e = cudaMemcpyAsync(out + off * n_pid, g->stage[s][2], m * n_pid * sizeof(double), cudaMemcpyDeviceToHost,
                            st);
        if (e != cudaSuccess) return drain(cuda_fail(e, "device-to-host copy"));
    }
    for (int s = 0; s < 3; ++s) PDF_CUDA(cudaStreamSynchronize(g->hs[s]));
    return PDF_OK;
}
