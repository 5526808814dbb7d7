// The library's host/device routines built for the CPU: the table builders of
// csrc/grid.cu and the knot search and fixed-point patches that its kernels
// inline, called from tests/fixed_host.py.
#include "grid.cu"

namespace {

// One axis: knots (ln z to FP64 as the library's tables hold it, and as long
// double), the cells' matrices in both forms and their fixed-point cells.
struct HostAxis {
    std::vector<double> U, M;
    std::vector<FixMatrix> F;
    std::vector<FixCell> C;

    HostAxis(const double *z, int n, bool linear)
        : U(n), M((size_t)(n - 1) * 16), F(n - 1), C(n - 1)
    {
        const LogTables &L = log_tables();
        const FixLogTables &T = fix_log_tables();
        std::vector<long double> UL(n);
        long double m[16], s[16], c[16];
        double ms[16];
        for (int k = 0; k < n; ++k) {
            U[k] = tlog(z[k], L.tab.data(), L.etab.data());
            UL[k] = logl((long double)z[k]);
        }
        for (int k = 0; k + 1 < n; ++k) {
            cell_matrix<double>(U.data(), n, k, &M[(size_t)k * 16], linear, ms);
            cell_matrix<long double>(UL.data(), n, k, m, linear, s);
            centre_matrix(m, c);
            F[k] = fix_matrix(c);
            C[k] = fix_cell(z[k], z[k + 1], T.inv.data(), T.log.data());
        }
    }
};

}  // namespace

// Cells that the guided search gives for n keys over the lower keys lo[ncell]
// of an axis whose last knot has the bits `last`.
extern "C" void host_cells(const uint64_t *lo, int ncell, uint64_t last, const uint64_t *key, int n, int *cell,
                           int *guided)
{
    std::vector<uint64_t> keys(lo, lo + ncell);
    std::vector<uint16_t> guide;
    int shift, run;
    build_guide(keys, last, guide, &shift, &run);
    search_table(keys);
    *guided = (int)guide.size();
    for (int i = 0; i < n; ++i)
        cell[i] = find_cell_guided(keys.data(), ncell, largest_pow2_below(ncell), guide.data(), (int)guide.size(),
                                   shift, run, lo[0], key[i]);
}

// n points on one subgrid of nq Q^2 knots (v [nq][nx]): per point the
// fixed-point value, the FP64 form's at the same coordinates, the two
// fixed-point derivatives in t (NaN where the kernels take FP64), the FP64
// form's value at coordinates from FP64 logarithms, and the coordinates (value
// 2^62; -1 in a cell without them).
extern "C" void host_eval(int nx, const double *x, int x_linear, int nq, const double *q2, int q_linear,
                          const double *v, int n, const double *px, const double *pq, double *out, int64_t *t)
{
    const HostAxis X(x, nx, x_linear), Q(q2, nq, q_linear);
    const FixLogTables &T = fix_log_tables();
    auto cell_of = [](const double *z, int m, double p) {
        return std::max((int)(std::upper_bound(z, z + m - 1, p) - z) - 1, 0);
    };
    for (int i = 0; i < n; ++i) {
        const int kx = cell_of(x, nx, px[i]), kq = cell_of(q2, nq, pq[i]);
        double s[4][4], C[4][4];
        unsigned mask = 0;
        for (int r = 0; r < 4; ++r)
            for (int c = 0; c < 4; ++c) {
                const int row = kq - 1 + r, col = kx - 1 + c;
                const bool ok = row >= 0 && row < nq && col >= 0 && col < nx;
                s[r][c] = ok ? v[(size_t)row * nx + col] : 0.0;
                mask |= ok ? 1u << (4 * r + c) : 0u;
            }
        const double *Mx = &X.M[(size_t)kx * 16], *Mq = &Q.M[(size_t)kq * 16];
        for (int r = 0; r < 4; ++r)
            for (int m = 0; m < 4; ++m) {
                C[r][m] = 0.0;
                for (int k = 0; k < 4; ++k) C[r][m] = fma(Mx[4 * m + k], s[r][k], C[r][m]);
            }
        double P[4][4];
        for (int k = 0; k < 4; ++k)
            for (int m = 0; m < 4; ++m) {
                P[k][m] = 0.0;
                for (int r = 0; r < 4; ++r) P[k][m] = fma(Mq[4 * k + r], C[r][m], P[k][m]);
            }
        uint32_t w[32];
        fix_patch(s, mask, X.F[kx], Q.F[kq], w);
        const bool cells = X.C[kx].K && Q.C[kq].K;
        t[2 * i] = cells ? fix_coord(fix_log(dbits(px[i]), T.inv.data(), T.log.data()), X.C[kx]) : -1;
        t[2 * i + 1] = cells ? fix_coord(fix_log(dbits(pq[i]), T.inv.data(), T.log.data()), Q.C[kq]) : -1;
        auto fp_coord = [](double z, const std::vector<double> &U, int k) {
            const LogTables &L = log_tables();
            return (tlog(z, L.tab.data(), L.etab.data()) - U[k]) * (1.0 / (U[k + 1] - U[k]));
        };
        const double tx = cells ? ldexp((double)t[2 * i], -62) : fp_coord(px[i], X.U, kx);
        const double tq = cells ? ldexp((double)t[2 * i + 1], -62) : fp_coord(pq[i], Q.U, kq);
        auto horner = [](double z, double a, double b, double c, double d) {
            return fma(z, fma(z, fma(z, d, c), b), a);
        };
        auto fp64 = [&](double zx, double zq) {
            double row[4];
            for (int k = 0; k < 4; ++k) row[k] = horner(zx, P[k][0], P[k][1], P[k][2], P[k][3]);
            return horner(zq, row[0], row[1], row[2], row[3]);
        };
        double *o = out + 5 * i;
        o[1] = fp64(tx, tq);
        o[4] = fp64(fp_coord(px[i], X.U, kx), fp_coord(pq[i], Q.U, kq));
        o[0] = o[2] = o[3] = NAN;
        const int last = (int)w[6];
        if (!cells || fix_needs_fp64(last, fix_limit(t[2 * i], t[2 * i + 1]))) continue;
        Dig wt[16];
        fix_weights(t[2 * i] - kFixHalf, t[2 * i + 1] - kFixHalf, wt);
        int64_t sum = 0, dx = 0, dq = 0;
        for (int k = 0; k < 4; ++k) {
            const int *c = (const int *)w + 8 * k;
            sum += fix_row(c, wt + 4 * k);
            dx += fix_row_dx(c, wt + 4 * k);
            if (k) dq += k * fix_row(c, wt + 4 * (k - 1));
        }
        const int e = (last & 127) - kFixBias - 59;
        o[0] = ldexp((double)sum, e);
        o[2] = ldexp((double)dx, e);
        o[3] = ldexp((double)dq, e);
    }
}

extern "C" void host_alphas(int nq, const double *q2, const double *a, int n, const double *pq, double *out, int64_t *t)
{
    const HostAxis Q(q2, nq, false);
    const FixLogTables &T = fix_log_tables();
    std::vector<long double> W(nq);
    for (int k = 0; k < nq; ++k) W[k] = logl((long double)q2[k]);
    for (int i = 0; i < n; ++i) {
        const int k = std::max((int)(std::upper_bound(q2, q2 + nq - 1, pq[i]) - q2) - 1, 0);
        uint32_t w[8];
        fix_cubic(W.data(), a, nq, k, false, w);
        t[i] = fix_coord(fix_log(dbits(pq[i]), T.inv.data(), T.log.data()), Q.C[k]);
        out[i] = NAN;
        if (!Q.C[k].K || fix_needs_fp64((int)w[6], kFixNone)) continue;
        Dig d[4];
        d[0] = {1 << 30, 0};
        d[1] = fix_split(t[i] - kFixHalf);
        d[2] = fix_split(fix_mul(d[1], d[1]));
        d[3] = fix_split(fix_mul(d[2], d[1]));
        out[i] = ldexp((double)fix_row((const int *)w, d), ((int)w[6] & 127) - kFixBias - 59);
    }
}
