// Luminosity of 32 events by one warp, sum_a f_a(x1) f_{-a}(x2) in fixed
// point (fix.cuh, warp_eval.cuh), shared by the luminosity and its VEGAS
// integral.
//
// The coordinates arrive as logarithms, so a knot search and two FP64
// operations give each local coordinate; the 2 F patches per event are the
// work.  The partons are taken one after the other (the weights of both would
// not leave room for two blocks per SM): the first parton's F values wait in
// shared memory, the second's are multiplied in as they come.
#pragma once

#include "warp_eval.cuh"

namespace pdfgpu {

// The coordinate tables of the logarithms (order keys and cells): a block's
// copies in shared memory, or the grid's.
struct LogTabs {
    const int64_t *ukey, *wkey;
    const double2 *xcell, *qcell;
};

__host__ __device__ inline int log_tab_bytes(const GridDev &g) { return ((g.nxc + g.nqc) * 24 + 127) & ~127; }

__device__ __forceinline__ LogTabs grid_log_tabs(const GridDev &g) { return {g.ukey, g.wkey, g.xcell, g.qcell}; }

__device__ __forceinline__ LogTabs stage_log_tabs(const GridDev &g, unsigned char *buf)
{
    double2 *xc = reinterpret_cast<double2 *>(buf), *qc = xc + g.nxc;
    int64_t *uk = reinterpret_cast<int64_t *>(qc + g.nqc), *wk = uk + g.nxc;
    for (int k = threadIdx.x; k < g.nxc; k += blockDim.x) {
        xc[k] = g.xcell[k];
        uk[k] = g.ukey[k];
    }
    for (int k = threadIdx.x; k < g.nqc; k += blockDim.x) {
        qc[k] = g.qcell[k];
        wk[k] = g.wkey[k];
    }
    return {uk, wk, xc, qc};
}

// The axes of axis_u and axis_w from these tables.
__device__ __forceinline__ Axis axis_u(const GridDev &g, const LogTabs &T, double u)
{
    return axis_log(g, T.ukey, T.xcell, g.nxc, g.xstep, g.ulo, g.uhi, u);
}
__device__ __forceinline__ Axis axis_w(const GridDev &g, const LogTabs &T, double w)
{
    return axis_log(g, T.wkey, T.qcell, g.nqc, g.qstep, g.wlo, g.whi, w);
}

// Whether both partons and the scale lie in the knot range.
__device__ __forceinline__ bool in_logs(const GridDev &g, double u1, double u2, double w)
{
    const int64_t a = dkey(u1), b = dkey(u2), c = dkey(w);
    return (a >= g.ulo) & (a <= g.uhi) & (b >= g.ulo) & (b <= g.uhi) & (c >= g.wlo) & (c <= g.whi);
}

// Cell and fixed-point coordinate (value 2^62) of a logarithm z inside the knot
// range.  The coordinate is the FP64 one of axis_u / axis_w.
__device__ __forceinline__ FixAxis fix_axis_log(const GridDev &g, const int64_t *keys, const double2 *cells, int ncell,
                                                int step, double z)
{
    FixAxis A;
    A.cell = checked_index(g.status, find_cell<int64_t>(keys, ncell, step, dkey(z)), ncell);
    A.ok = true;
    const double2 c = cells[A.cell];
    const int64_t t = __double2ll_rn((z - c.x) * c.y * 4611686018427387904.0 /* 2^62 */);
    A.t = min(max(t, (int64_t)0), (int64_t)1 << 62);
    return A;
}

// Bytes of one warp's buffers: weights, `row` doubles per event, queue.
__host__ __device__ inline int lumi_warp_bytes(int row) { return kWarpBuf + 32 * 8 * row + kQueue * 8; }

// One event per lane; lanes with `fast` false get nothing useful.  rows: 32 x
// `row` doubles of shared memory; parton 1's value of flavour a is left at
// [lane][a] and, with SAVE (row = 2 F), parton 2's of flavour b at [lane][F +
// b].  Returns the event's sum; `fast` is cleared where a patch needs FP64.
template <bool SAVE>
__device__ __forceinline__ double lumi_quads(const GridDev &g, const signed char *anti, const unsigned char *fm,
                                             uint4 *buf, double *rows, int row, int lane, const FixAxis &X1,
                                             const FixAxis &X2, const FixAxis &Q, bool &fast)
{
    const QuadPos pos = quad_pos(lane);
    const uint32_t cell_bytes = (uint32_t)g.nflav * 128u;
    double *mine = rows + lane * row;
    bool none = false;
    double s = 0.0;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        const FixAxis &X = side ? X2 : X1;
        uint32_t off[4];
        quad_offsets(fast ? (uint32_t)(Q.cell * g.nxc + X.cell) * cell_bytes : 0u, lane, off);
        Dig W[4][4];
        quad_weights(buf, lane, fast ? X.t : kFixHalf, fast ? Q.t : kFixHalf, W);
        const int limit = fix_limit(X.t, Q.t);
        for (int a = 0; a < g.nflav; ++a) {
            const int b = anti[a];
            double v = 0.0;
            const int col = side ? b : a;
            if (b >= 0) {                        // the same for the whole warp
                int c[4][8], last;
                quad_load(fm + col * 128, off, c);
                const int64_t p = quad_patch(c, W, pos, last);
                v = fix_value(p, last);
                none |= fix_needs_fp64(last, limit);
            }
            if (side == 0) {
                mine[a] = v;
                if (SAVE && b < 0) mine[g.nflav + a] = 0.0;
            } else if (b >= 0) {
                s = fma(mine[a], v, s);
                if (SAVE) mine[g.nflav + b] = v;
            }
        }
    }
    fast = fast && !none;
    return s;
}

}  // namespace pdfgpu
