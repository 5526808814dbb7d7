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
    keys.insert(keys.end(), kGuideRun, ~(uint64_t)0);
    *guided = (int)guide.size();
    for (int i = 0; i < n; ++i)
        cell[i] = find_cell_guided(keys.data(), ncell, largest_pow2_below(ncell), guide.data(), (int)guide.size(),
                                   shift, run, keys[0], key[i]);
}

