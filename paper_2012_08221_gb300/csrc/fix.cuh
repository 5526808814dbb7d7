// Fixed-point evaluation of the interpolant.
//
// The FP64 pipe of this GPU issues 2 FMAs per clock and SM; IMAD.WIDE (32 x
// 32 + 64 bits) issues 64 (pdf_probe_wide_multiply: 63, and 57 where all pairs
// of operands meet).  Inside the knot range a patch is therefore
// evaluated in 64-bit integers: the 16 monomial coefficients of the patch
// about the cell's centre, scaled by the power of two above the largest of
// them (a block exponent), against the 16 products of the powers of the two
// local coordinates tc = t - 1/2 in [-1/2, 1/2].  A 64-bit by 64-bit product
// costs three IMAD.WIDE (the low x low digit product is below the last bit
// kept), and sums need no normalisation.
//
// Formats.  A "Dig" is a 64-bit integer h 2^32 + l with SIGNED l, so that
// digit products are plain signed 32 x 32 multiplies.
//   coordinates and their products (weights)  value 2^62
//   coefficients                              value 2^(61 - E), |.| <= 2^61,
//                                             E: max |coefficient| < 2^E
//   sums of coefficient x weight              value 2^(59 - E)
//   logarithms                                value 2^60 modulo 16
// Errors: a sum is off by about 2^(E - 57) anywhere in the cell, what the build
// leaves by 2^(E - 57) on even cells and up to 2^(E - 53) at the limit of those
// it serves (kFixBuild), a logarithm by about 2^-59 absolute.  FP64 is off by several 2^-53 of the terms
// at the point, and its logarithm by 2^-53 |ln x| (2^-49 at 16 ... 32), which a
// cell's width magnifies.  What FP64 does better keeps FP64: values on the lower
// edges of a patch that is small there (fix_patch, fix_limit; knots come out to
// the last bit in either form), patches that the block exponent or the build
// cannot hold, cells too wide or too narrow (fix_cell in grid.cu), points
// outside the knots.  At a given t a weak patch (see kFixStrong) is still less
// accurate next to its lower edges than the FP64 form would be; at a given x and
// Q^2 it is more accurate.
// Integer sums do not depend on their order: every kernel gives the same bits
// however it splits a patch over lanes.
#pragma once

// Included by pdf_common.cuh, after the bit helpers it uses.

namespace pdfgpu {

struct Dig {
    int h, l;
};

// The two words of a 64-bit value.  On the device they are split off in PTX:
// from a plain cast the compiler remembers the 64-bit value and widens the
// products below to 64 x 64 bits (279 instructions per alpha_s, not 150).
PDF_HD int fix_hi(int64_t v)
{
#ifdef __CUDA_ARCH__
    int hi;
    asm("{.reg .b32 lo; mov.b64 {lo, %0}, %1;}" : "=r"(hi) : "l"(v));
    return hi;
#else
    return (int)(uint32_t)((uint64_t)v >> 32);
#endif
}
PDF_HD int fix_lo(int64_t v)
{
#ifdef __CUDA_ARCH__
    int lo;
    asm("{.reg .b32 hi; mov.b64 {%0, hi}, %1;}" : "=r"(lo) : "l"(v));
    return lo;
#else
    return (int)(uint32_t)(uint64_t)v;
#endif
}
// Bits [n, n + 32) of a value, 0 < n < 32 (one funnel shift).
PDF_HD int fix_bits(int64_t v, int n)
{
#ifdef __CUDA_ARCH__
    return (int)__funnelshift_r((unsigned)fix_lo(v), (unsigned)fix_hi(v), n);
#else
    return (int)(uint32_t)((uint64_t)v >> n);
#endif
}

PDF_HD Dig fix_split(int64_t v)
{
    const int lo = fix_lo(v);
    return {fix_hi(v) + (int)((uint32_t)lo >> 31), lo};
}

PDF_HD int64_t wide(int a, int b) { return (int64_t)a * (int64_t)b; }
PDF_HD int64_t wide(int a, int b, int64_t c) { return (int64_t)a * (int64_t)b + c; }
PDF_HD uint64_t wide(uint32_t a, uint32_t b) { return (uint64_t)a * (uint64_t)b; }
PDF_HD uint64_t wide(uint32_t a, uint32_t b, uint64_t c) { return (uint64_t)a * (uint64_t)b + c; }

// Product of two values of at most 1/2 (2^61), in the format of the factors.
PDF_HD int64_t fix_mul(Dig a, Dig b)
{
    const int64_t cr = wide(a.l, b.h, wide(a.h, b.l, (int64_t)1 << 29));
    return wide(2 * a.h, 2 * b.h) + fix_bits(cr, 30);
}

// ln 2 in 2^-92, in signed 32-bit digits.
constexpr int kLn2Top = 186065279, kLn2Mid = 2099050395, kLn2Low = -1130480839;

// ln of a positive normal double from its bits, value 2^60 modulo 2^64.
//   x = 2^e m; j = top 10 bits of m; inv = 1/c_j in 2^-31 (c_j the middle of
//   the table interval), r = m inv - 1 exact to 2^-62, |r| <= 2^-11;
//   ln(1 + r) = r - r^2/2 + r^3 (1/3 - r/4 + r^2/5)  (next term < 2^-68);
//   tab holds -ln(inv).  Host tables and kernels call this same routine, so
//   a point on a knot gets the knot's own logarithm.
PDF_HD int64_t fix_log(uint64_t bits, const uint32_t *inv, const int64_t *tab)
{
    const uint32_t hw = (uint32_t)fix_hi((int64_t)bits);
    const int e = (int)(hw >> 20) - 1023;
    const uint32_t j = (hw >> (20 - kLogBits)) & (kLogTab - 1);
    const uint32_t mh = (uint32_t)fix_bits((int64_t)bits, 21) | 0x80000000u, ml = (uint32_t)fix_lo((int64_t)bits) << 11;
    const uint32_t I = inv[j];
    const uint64_t P = wide(mh, I, (uint64_t)(uint32_t)fix_hi((int64_t)wide(ml, I)));
    const int64_t R = (int64_t)(P - ((uint64_t)1 << 62));       // r 2^62
    const int rh = fix_bits(R, 21), rl = fix_lo(R) & 0x1FFFFF, rs = fix_bits(R, 30);
    const int64_t sq = wide(rh, rh);                            // r^2 2^82
    const int64_t r2 = sq + (wide(rh, rl) >> 20);
    int z = fix_hi(wide(rs, 429496730, -((int64_t)536870912 << 32)));  // -1/4 + r/5, in 2^-31
    z = fix_hi(wide(rs, z, (int64_t)715827883 << 32));                 // 1/3 + r z
    const int c = fix_hi(wide(fix_hi(sq), rh));                        // r^3 2^59
    const int64_t tail = wide(c, z, 1 << 29) >> 30;                    // in 2^-60
    const int64_t head = (R - (r2 >> 21) + 2) >> 2;
    // e ln 2: the upper 32 bits of the constant times e, the lower ones, and 32 more
    const int64_t el = wide(e, kLn2Mid, (int64_t)((uint64_t)(uint32_t)(e * kLn2Top) << 32)) + fix_hi(wide(e, kLn2Low, (int64_t)1 << 31));
    return (int64_t)((uint64_t)head + (uint64_t)tab[j] + (uint64_t)el + (uint64_t)tail);
}

// One cell's logarithm of the lower knot and 2^126 / (width << s), with the
// normalising shift s in the low 6 bits (width << s in [2^62, 2^63)); K = 0
// marks a cell that the format cannot serve.
struct FixCell {
    int64_t U;
    uint64_t K;
};

// Local coordinate t of a logarithm in its cell, value 2^62.
PDF_HD int64_t fix_coord(int64_t u, const FixCell &c)
{
    int64_t v = (int64_t)((uint64_t)u - (uint64_t)c.U);
    v = v < 0 ? 0 : v;                      // a unit of the logarithm's error below the knot
    const uint64_t vv = (uint64_t)v << (c.K & 63);
    const uint32_t vh = (uint32_t)fix_hi((int64_t)vv), vl = (uint32_t)fix_lo((int64_t)vv);
    const uint32_t kh = (uint32_t)fix_hi((int64_t)c.K), kl = (uint32_t)fix_lo((int64_t)c.K);
    const uint64_t a = (uint32_t)fix_hi((int64_t)wide(vh, kl)), b = (uint32_t)fix_hi((int64_t)wide(vl, kh));
    return (int64_t)(wide(vh, kh, a) + b);
}

constexpr int64_t kFixHalf = (int64_t)1 << 61;

#ifdef __CUDACC__
// The same t as a double.
__device__ __forceinline__ double fix_t(int64_t t) { return __ll2double_rn(t) * 2.168404344971009e-19; /* 2^-62 */ }
#endif

// The 16 weights tq^n tx^m of a point (index 4 n + m) from tc = t - 1/2.
PDF_HD void fix_weights(int64_t tcx, int64_t tcq, Dig w[16])
{
    w[0] = {1 << 30, 0};
    w[1] = fix_split(tcx);
    w[2] = fix_split(fix_mul(w[1], w[1]));
    w[3] = fix_split(fix_mul(w[2], w[1]));
    w[4] = fix_split(tcq);
    w[8] = fix_split(fix_mul(w[4], w[4]));
    w[12] = fix_split(fix_mul(w[8], w[4]));
#pragma unroll
    for (int n = 4; n <= 12; n += 4)
#pragma unroll
        for (int m = 1; m < 4; ++m) w[n + m] = fix_split(fix_mul(w[n], w[m]));
}

// Sum of four coefficients (l, h pairs) against four weights: the high
// products, and the upper word of the cross products' rounded sum, which is
// below 2^63 in size (4 x 2^29 x 2^31 + 2^31 x 2^30 (1 + 1/2 + 1/4 + 1/8)).
PDF_HD int64_t fix_row(const int c[8], const Dig w[4])
{
    int64_t hh = 0, cr = (int64_t)1 << 31;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        hh = wide(c[2 * m + 1], w[m].h, hh);
        cr = wide(c[2 * m + 1], w[m].l, cr);
        cr = wide(c[2 * m], w[m].h, cr);
    }
    return hh + fix_hi(cr);
}

// The same row differentiated in t of the x axis, c1 w0 + 2 c2 w1 + 3 c3 w2
// (the weights w_m = tq^n tx^m serve for their own derivatives).
PDF_HD int64_t fix_row_dx(const int c[8], const Dig w[4])
{
    int64_t h3 = wide(c[7], w[2].h), r3 = wide(c[6], w[2].h, wide(c[7], w[2].l, (int64_t)1 << 31));
    const int64_t s3 = h3 + fix_hi(r3);
    const int64_t h2 = wide(c[5], w[1].h, h3), r2 = wide(c[4], w[1].h, wide(c[5], w[1].l, r3));
    const int64_t s2 = h2 + fix_hi(r2);              // c2 w1 + c3 w2
    const int64_t h1 = wide(c[3], w[0].h), r1 = wide(c[2], w[0].h, wide(c[3], w[0].l, (int64_t)1 << 31));
    return (h1 + fix_hi(r1)) + 2 * s2 + s3;
}

// Coordinates that round to a knot as doubles: there a derivative may be zero
// by exact cancellation, which FP64 from the knot's own expansion keeps.
PDF_HD bool fix_at_knot(int64_t t) { return t <= 0 || t >= ((int64_t)1 << 62) - 256; }

// Block exponent: the low 7 bits of a row's last coefficient are E + kFixBias.
// Bit 7 marks a patch that serves away from the cell's lower edges only
// (kFixWeak), kFixNone one that the format cannot hold.
constexpr int kFixBias = 80;
constexpr int kFixWeak = 128;
constexpr int kFixNone = 255;

// On a lower edge: t < 2^-20 on either axis.  There the FP64 form, which expands
// about the lower corner, gives the values on the knots to the last bit, and
// the fixed-point form's error follows the patch's largest coefficient: a weak
// patch (fix_patch) then takes FP64.  The limit is the least exponent byte that
// does so at the point.
constexpr int kFixEdge = 1 << 10;         // 2^-20 in the upper word of a t (value 2^62)
PDF_HD int fix_limit(int64_t tx, int64_t tq)
{
    return fix_hi(tx) < kFixEdge || fix_hi(tq) < kFixEdge ? kFixWeak : kFixNone;
}
PDF_HD bool fix_needs_fp64(int last, int limit) { return (last & 255) >= limit; }

#ifdef __CUDACC__
__device__ __forceinline__ double fix_value(int64_t s, int last)
{
    return __ll2double_rn(s) * __hiloint2double((last & 127) * (1 << 20) + ((1023 - 59 - kFixBias) << 20), 0);
}

// Eight 32-bit words (one row of a fixed-point patch) in one 32-byte load.
__device__ __forceinline__ void fix_ld(const unsigned char *p, int c[8])
{
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]), "=r"(c[4]), "=r"(c[5]), "=r"(c[6]), "=r"(c[7])
        : "l"(p));
}
#endif

// Lower corner (t = 0 on both axes) against the largest coefficient (below 2^E)
// and the stencil (below 2^Ev).  A fixed-point sum is off by 2^(E - 57) or so,
// at the corner by less than 2^(E - 57.5), which rounds to the knot's value
// while the corner is 2^(E - 5) at least; FP64 is off by 2^-53 of the largest
// term at the point, next to the corner of the corner's value.
//  - From 2^(E - 2) on fixed point is as good everywhere.
//  - Below, the patch is weak: FP64 on its lower edges.  Away from them the
//    argument decides: FP64's logarithm moves the value by 2^-53 |ln x| / width
//    of 2^E, more than 2^(E - 54) anywhere; fixed point's by 2^(E - 59) /
//    width.  Largest error of the value itself, FP64 / fixed point, cells of
//    0.1 at ln x = -5 with the corner 2^-k of the rest: k = 4 1e-13 / 1e-15, 6
//    8e-13 / 6e-15.  (The patch alone, at a given t: 8e-15 / 9e-16, 1e-14 /
//    5e-15.)
//  - 2^7 below (a flavour that sets in at a threshold knot), or with a stencil
//    2^12 above the corner, the patch keeps FP64.
// Of the 196 x 50 grid's patches 2.8 % are weak (by area), none is 2^7 below
// (0.005 % are 2^6 below).  A point that takes FP64 keeps its warp: one in a query of one pass per
// warp costs 2.5 us and more (1e5 points x 11 flavours 19.3 -> 21.7 us, 54000
// events 33 -> 37).  So the edge is narrow: with it at 2^-14 every second such
// query had a point there, with 2^-10 the matrix-form fit step took 3 % longer
// and the luminosity 2 %, with 2^-4 x*f 3.5 % and 400 batched requests 11 %.
constexpr int kFixStrong = 1;
constexpr int kFixCorner = 7;
constexpr int kFixStencil = 12;
PDF_HD int fix_exponent(double v) { return ((int)(dbits(v) >> 52) & 0x7FF) - 1022; }   // |v| < 2^this

// What the build leaves in a patch is at most about 2^(Ev - 60 + spreads) for
// stencil values below 2^Ev: with interval ratios 2^r on both axes that is 2^(2
// r), and smooth values have coefficients (2^E) that do not grow with it; steep
// ones have a stencil far above the cell.  Patches where it passes 2^(E - 54)
// keep FP64 (ratios from about 2^6 on; a cell 2^12 times its neighbours on both
// axes was off by 8e-12 of its values' size).  The limit lies where ordinary
// grids have nothing beyond it (196 x 50: 0.21 % of the area from 5 on, 0.007 %
// from 6, none from 7); with it at 4, 400 batched requests took 10 % longer and
// the luminosity 25 %.  kFixReach: the same against the corner's size, for a weak
// patch.
constexpr int kFixBuild = 6;
constexpr int kFixReach = 7;

// One coefficient (value 2^(61 - E)) as the table holds it: the last of a row
// carries the exponent byte.
PDF_HD int64_t fix_last(int64_t v, int e8) { return ((v - e8 + 128) & ~(int64_t)255) | e8; }

PDF_HD void fix_words(int64_t v, uint32_t *out)
{
    const Dig d = fix_split(v);
    out[0] = (uint32_t)d.l;
    out[1] = (uint32_t)d.h;
}

// c1 - (c2 - c3 / 2) / 2, all halved: minus the cubic without its constant term
// at tc = -1/2.
PDF_HD int64_t fix_lower(int64_t c1, int64_t c2, int64_t c3) { return (c1 - ((c2 - (c3 >> 1)) >> 1)) >> 1; }

// A cell's centred matrix in fixed point: row m holds its four entries times
// 2^(61 - k[m]), the sum of their sizes at most 2^k[m]; k[0] < 0 marks a cell
// whose entries are too large (very uneven knots), which keeps FP64.  Bit i of
// `used`: the stencil's entry i has weight in it (a straight line takes the two
// knots of its interval only).  spread = max over the rows of k[m] - m: an error
// in row m's coefficient counts 2^-m at the cell's edges.
struct FixMatrix {
    Dig d[4][4];
    int k[4];
    int spread;
    unsigned used;
};

// Sum over i of M[i] v_i / 2^61 (|v_i| <= 2^61), rounded down, and the next 8 bits
// in `rest`: one entry of a matrix product.  The low x low products count here
// (without them an entry was off by up to 8 units, and the build by 2^4 times
// what it leaves now).
PDF_HD int64_t fix_dot(const Dig M[4], Dig v0, Dig v1, Dig v2, Dig v3, int &rest)
{
    const Dig v[4] = {v0, v1, v2, v3};
    int64_t hh = 0, cr = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        hh = wide(M[i].h, v[i].h, hh);
        cr = wide(M[i].h, v[i].l, cr);
        cr = wide(M[i].l, v[i].h, cr) + fix_hi(wide(M[i].l, v[i].l));
    }
    rest = (int)((uint64_t)cr >> 21) & 255;
    return (int64_t)((uint64_t)hh << 3) + (cr >> 29);
}
// The entry times 2^s, 0 <= s < 8, rounded.
PDF_HD int64_t fix_entry(int64_t v, int rest, int s)
{
    return (int64_t)((uint64_t)v << s) + ((rest + (128 >> s)) >> (8 - s));
}

// A double as an integer times 2^-s, rounded; zero below.
PDF_HD int64_t fix_from(double v, int s)
{
    const uint64_t b = dbits(v);
    const int e = (int)(b >> 52) & 0x7FF, n = e - 1075 + s;
    const uint64_t m = e ? (b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull : 0;
    const uint64_t r = n >= 0 ? m << (n & 63) : n > -54 ? (m + ((uint64_t)1 << (-n - 1))) >> -n : 0;
    return (int64_t)b < 0 ? -(int64_t)r : (int64_t)r;
}

PDF_HD int fix_clz(uint64_t v)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}
PDF_HD int64_t fix_shift(int64_t v, int n)   // v 2^n, rounded
{
    if (n >= 0) return (int64_t)((uint64_t)v << (n & 63));
    return n > -63 ? (v + ((int64_t)1 << (-n - 1))) >> -n : 0;
}

// The fixed-point patch of a 4 x 4 stencil v (rows of Q, columns of x; ok bits
// 4 r + i of `mask`), from its cells' matrices: all in integers, so that the
// coefficients keep about 2^-58 of the stencil's largest value (an FP64 sum
// keeps 2^-53) and the FP64 pipe stays free.  The interpolation of a constant
// being the constant, the sums run over the differences to the lower corner.
// The first product keeps the bits that the matrix's row sum leaves room for
// (steep functions have entries far below it, and lost up to 5 of them).
// The values' common exponent is that of the entries with weight: a straight
// line's neighbours may be far larger than its own knots (2^30: values off by
// 1e-9 when they counted; FP64 never mixes them in).
PDF_HD void fix_patch(const double v[4][4], unsigned mask, const FixMatrix &X, const FixMatrix &Q, uint32_t out[32])
{
    unsigned used = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) used |= (Q.used >> r) & 1 ? X.used << (4 * r) : 0;
    int emax = 0;
    bool finite = true;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = (int)(dbits(v[r][i]) >> 52) & 0x7FF;
            if ((mask >> (4 * r + i)) & 1) finite = finite && e != 0x7FF;
            if ((mask & used) >> (4 * r + i) & 1) emax = e > emax ? e : emax;
        }
    mask &= used;
    const int Ev = emax - 1022;                      // |v| < 2^Ev
    bool ok = finite && X.k[0] >= 0 && Q.k[0] >= 0;
    const int64_t ref = fix_from(v[1][1], 60 - Ev);
    int64_t cx[4][4];
    int rest[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        Dig d[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            d[i] = fix_split((mask >> (4 * r + i)) & 1 ? fix_from(v[r][i], 60 - Ev) - ref : 0);
#pragma unroll
        for (int m = 0; m < 4; ++m) cx[r][m] = fix_dot(X.d[m], d[0], d[1], d[2], d[3], rest[r][m]);
    }
    int64_t C[4][4];
    int E = -100000, up[4];                          // up[m]: bits that column m gains before the second product
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        uint64_t any = 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) any |= (uint64_t)(cx[r][m] < 0 ? -cx[r][m] : cx[r][m]);
        const int most = m || X.k[0] + Q.k[0] > 7 ? 7 : X.k[0] + Q.k[0], room = fix_clz(any) - 4;
        up[m] = room < most ? room : most;
        up[m] = up[m] < 0 ? 0 : up[m];
        Dig c[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) c[r] = fix_split(fix_entry(cx[r][m], rest[r][m], up[m]));
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            int low;
            const int64_t down = fix_dot(Q.d[n], c[0], c[1], c[2], c[3], low);
            C[n][m] = fix_entry(down, low, 0);
            const int k = X.k[m] + Q.k[n] - up[m];
            const int64_t t = n + m ? C[n][m] : C[0][0] + (ref >> (k & 63));
            const int e = 4 - fix_clz((uint64_t)(t < 0 ? -t : t)) + k + Ev;
            if (t && e > E) E = e;
        }
    }
    int e8 = 0;
    if (emax == 0) {                                 // zeros (subnormal values keep FP64)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int i = 0; i < 4; ++i) ok = ok && (!((mask >> (4 * r + i)) & 1) || v[r][i] == 0.0);
    } else {
        const int ec = fix_exponent(v[1][1]), spread = X.spread + Q.spread;
        e8 = E + kFixBias;
        ok = ok && e8 >= 0 && e8 < 127 && E - ec <= kFixCorner && Ev - ec <= kFixStencil && Ev + spread - E <= kFixBuild;
        if (E - ec > kFixStrong || Ev + spread - ec > kFixReach) e8 |= kFixWeak;
    }
    if (!ok) e8 = kFixNone;
    const bool fill = ok && emax != 0;
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            C[n][m] = fill ? fix_shift(C[n][m], 1 - E + X.k[m] + Q.k[n] - up[m] + Ev) : 0;
            if (m == 3) C[n][m] = fix_last(C[n][m], e8);
        }
    // the constant term from the others as stored, so that the sum at the corner is the knot's value
    int64_t low[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) low[n] = fix_lower(C[n][1], C[n][2], C[n][3]);
    if (fill)
        C[0][0] = fix_shift(ref, 1 + Ev - E) + low[0] + fix_lower(C[1][0] - low[1], C[2][0] - low[2], C[3][0] - low[3]);
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int m = 0; m < 4; ++m) fix_words(C[n][m], out + 2 * (4 * n + m));
}

}  // namespace pdfgpu
