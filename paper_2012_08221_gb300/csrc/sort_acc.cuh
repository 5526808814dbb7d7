// Device helpers shared by the adjoints that accumulate a grid gradient in
// the monomial basis of the interpolation patch (the grid gradients of
// bwd.cu and the luminosity adjoint of lumi.cu): per bin of sorted points a
// half-warp holds G[n][m] = sum over the bin's points of (weight) bq_n bx_m
// and maps it back to the 16 stencil values once per run of the bin; and
// the pointwise bin of a point, which the forward pass also writes into the
// derivative tape.
#pragma once

#include "pdf_common.cuh"

namespace pdfgpu {

// Maps a half-warp's 16 accumulators back to the 16 stencil values of their
// bin.  Lane 4n + m passes G[n][m] in g; lane 4j + i gets
// sum_{n,m} Mq[n][j] G[n][m] Mx[m][i], in two stages through the half-warp's
// 16 shared slots buf: T[j][m] = sum_n Mq[n][j] G[n][m] (lane 4j + m), then
// sum_m T[j][m] Mx[m][i] -- 8 FMAs per lane.
__device__ __forceinline__ double map_back(double g, double *buf, const double *__restrict__ Mq,
                                           const double *__restrict__ Mx, int sn, int sm, unsigned hmask)
{
    buf[4 * sn + sm] = g;
    __syncwarp(hmask);
    double t = 0.0;
#pragma unroll
    for (int n = 0; n < 4; ++n) t = fma(Mq[n * 4 + sn], buf[4 * n + sm], t);
    __syncwarp(hmask);
    buf[4 * sn + sm] = t;
    __syncwarp(hmask);
    double dv = 0.0;
#pragma unroll
    for (int m = 0; m < 4; ++m) dv = fma(buf[4 * sn + m], Mx[m * 4 + sm], dv);
    __syncwarp(hmask);
    return dv;
}

// The same for a list of accumulators, kMapCols at a time: the matrices' entries
// are loaded once, and the columns' chains run side by side (one after the
// other, a flush of 13 columns cost 13 round trips through shared memory and
// 104 loads while the other half-warp waited).  buf: kMapCols x 16 slots of
// the half-warp; emit(a, value) gets column a's stencil value of this lane.
constexpr int kMapCols = 4;

template <int N, typename Emit>
__device__ __forceinline__ void map_back_all(double (&acc)[N], int n, double *buf, const double *__restrict__ Mq,
                                             const double *__restrict__ Mx, int sn, int sm, unsigned hmask, Emit emit)
{
    double q[4], x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        q[k] = Mq[4 * k + sn];
        x[k] = Mx[4 * k + sm];
    }
#pragma unroll
    for (int a0 = 0; a0 < N; a0 += kMapCols) {
        if (a0 < n) {
            double t[kMapCols];
#pragma unroll
            for (int a = 0; a < kMapCols; ++a)
                if (a0 + a < N) buf[16 * a + 4 * sn + sm] = acc[a0 + a];
            __syncwarp(hmask);
#pragma unroll
            for (int a = 0; a < kMapCols; ++a) {
                t[a] = 0.0;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (a0 + a < N) t[a] = fma(q[k], buf[16 * a + 4 * k + sm], t[a]);
            }
            __syncwarp(hmask);
#pragma unroll
            for (int a = 0; a < kMapCols; ++a)
                if (a0 + a < N) buf[16 * a + 4 * sn + sm] = t[a];
            __syncwarp(hmask);
#pragma unroll
            for (int a = 0; a < kMapCols; ++a)
                if (a0 + a < N && a0 + a < n) {
                    double dv = 0.0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) dv = fma(buf[16 * a + 4 * sn + k], x[k], dv);
                    emit(a0 + a, dv);
                }
            __syncwarp(hmask);
        }
    }
#pragma unroll
    for (int a = 0; a < N; ++a) acc[a] = 0.0;
}

// Half of a cell a point lies in along each axis: bit 0 set when t_x > 1/2,
// bit 1 when t_q > 1/2.  In an upper half the accumulation runs in powers of
// s = 1 - t (and maps back with the cell's matrix in s), so that the weights
// that vanish at the near knot come out of small powers, not of cancelling
// ones: a bin holds the points of one cell (and flavour) and one half pair.
// (The tape records the same two bits, from the same t, for the counting
// pass.)
__device__ __forceinline__ int half_pair(const Axis &X, const Axis &Q)
{
    return (upper_half(X.t) ? 1 : 0) | (upper_half(Q.t) ? 2 : 0);
}

// The local coordinate the accumulation uses: t, or 1 - t in an upper half
// (exact: t lies in [1/2, 1] there; of a fixed-point t before it is rounded).
__device__ __forceinline__ double near_coord(int64_t t)
{
    return fix_t(upper_half(t) ? ((int64_t)1 << 62) - t : t);
}
__device__ __forceinline__ double near_coord(const Axis &A)
{
    if (A.f >= 0) return near_coord(A.f);
    return upper_half(A.t) ? 1.0 - A.t : A.t;
}

// Chain rule from the local coordinates to x and Q^2: d/dx = d/dt_x (1/dU) / x
// and d/dQ^2 = d/dt_q (1/dW) / Q^2, with one reciprocal of x Q^2 for both (1/x
// = Q^2 / (x Q^2), 1/Q^2 = x / (x Q^2)); where the product leaves the normal
// range the two reciprocals are taken apart.  Every adjoint and the derivative
// tape take their factors from here.
struct ChainFactors {
    double x, q;
};
__device__ __forceinline__ ChainFactors chain_factors(const GridDev &g, int xc, int qc, double x, double q2)
{
    const double xq = x * q2;
    double rx, rq;
    if (dbits(xq) - 0x0010000000000000ull < 0x7FE0000000000000ull) {   // normal and finite
        const double r = __drcp_rn(xq);
        rx = q2 * r;
        rq = x * r;
    } else {
        rx = __drcp_rn(x);
        rq = __drcp_rn(q2);
    }
    return {g.xcell[xc].y * rx, g.qcell[qc].y * rq};
}

// Bin of a point in the pointwise sorted accumulation, ((cell * F + flavour
// column) * 4 + half pair), or -1 for a point that adds nothing there: a
// domain error, outside the grid under the error option, an absent pid, or
// outside the knot range on either axis (see k_bwd_rec).  The counting pass
// and the record pass both take the bin from this one function, on the same
// tape values (or both read the one the forward pass wrote from them into
// the derivative tape), so that every record placed was counted.
__device__ __forceinline__ int sorted_bin(const GridDev &g, const Axis &X, const Axis &Q, bool bad, int col,
                                          int halves, int nbins)
{
    if (bad || col < 0 || !(X.in && Q.in)) return -1;
    return checked_index(g.status, ((Q.cell * g.nxc + X.cell) * g.nflav + col) * 4 + halves, nbins);
}

}  // namespace pdfgpu
