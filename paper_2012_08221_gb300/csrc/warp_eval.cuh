// Warp-level evaluation of x*f at 32 points in fixed point (fix.cuh).
//
// A patch is 128 bytes at a random place of a table of 10-20 MB, and the L1
// serves about one request per 1.7 clocks and SM whatever its size up to a
// 128-byte line.  One point per lane would be four 32-byte requests per patch
// (5.6 TB/s of coefficients in a bare gather); here the four lanes of a quad
// take the four rows of one point's patch, one 128-byte request (21.8 TB/s),
// for each of the quad's four points in turn, and add their row sums with a
// reduce-scatter of three exchanges that leaves each lane its own point's
// patch.  The weights of a point are computed by its own lane and reach the
// quad through a swizzled 4 KB buffer per warp.
// What bounds it now is no single unit: per flavour and 32 points 48 IMAD.WIDE
// (2 cycles each of a sub-core: 22 % of the time), about 75 other integer
// instructions and 2 FP64 instructions for the conversion of the result (issue
// slots 42 % busy); the L1's data path is 50 % busy, and the 24 warps that 80
// registers allow wait for the rows from L2 and for their own chains.  1e7
// points x 13 flavours of the 196 x 50 grid: 3656 us with FP64 Horner patches
// (FP64 pipe 95 % busy), 1392 us here (1369 without the rules of fix_limit, whose
// operand spills 12 bytes).
//
// Points outside the knots (or in cells or patches that the format does not
// hold) are collected in a queue per warp and evaluated 32 at a time in FP64,
// so that a few of them do not make every warp run both paths (1e6 points x 3
// flavours with 5 % outside under the continuation: 475 -> 103 us).  A query that
// mostly outside pays for both: it is slower than FP64 alone was from two thirds
// of the points outside on (1e6 points x 13 flavours 380 -> 451 us at 95 %, 382
// with all of them outside; alpha_s 36 -> 44; 1e6 events 735 -> 925 and 764).
#pragma once

#include "pdf_common.cuh"

namespace pdfgpu {

constexpr int kWarpBuf = 4096;            // bytes of the weights buffer of one warp
constexpr int kQueue = 64;                // slots of a warp's queue
constexpr unsigned kAll = 0xffffffffu;

// This thread's lane, as a value that the compiler keeps instead of reading the
// thread index again in every loop.
__device__ __forceinline__ int lane_id()
{
    int lane = threadIdx.x & 31;
    asm volatile("" : "+r"(lane));
    return lane;
}

__device__ __forceinline__ double dnan() { return __longlong_as_double(0x7FF8000000000000ll); }

// Bytes of a block's copies of the coordinate tables (0: they stay global).
__host__ __device__ inline int coord_tab_bytes(const GridDev &g)
{
    const int b = (g.nxc + g.nqc) * 24 + 2 * kGuideRun * 8 + kLogTab * 12 + (g.nxg + g.nqg) * 2;
    return (b + 127) & ~127;
}

// Where a block's copies of the tables lie in its buffer (16-byte aligned).
__device__ __forceinline__ CoordTabs staged_tabs(const GridDev &g, unsigned char *buf)
{
    FixCell *xf = reinterpret_cast<FixCell *>(buf), *qf = xf + g.nxc;
    int64_t *lg = reinterpret_cast<int64_t *>(qf + g.nqc);
    uint64_t *xb = reinterpret_cast<uint64_t *>(lg + kLogTab), *qb = xb + g.nxc + kGuideRun;
    uint32_t *iv = reinterpret_cast<uint32_t *>(qb + g.nqc + kGuideRun);
    uint16_t *xg = reinterpret_cast<uint16_t *>(iv + kLogTab), *qg = xg + g.nxg;
    return {iv, lg, xb, qb, xg, qg, xf, qf};
}

// Makes the copies (whole block); the caller synchronises the block afterwards.
__device__ __forceinline__ CoordTabs stage_tabs(const GridDev &g, unsigned char *buf)
{
    const CoordTabs T = staged_tabs(g, buf);
    uint32_t *iv = const_cast<uint32_t *>(T.inv);
    int64_t *lg = const_cast<int64_t *>(T.log);
    uint64_t *xb = const_cast<uint64_t *>(T.xbits), *qb = const_cast<uint64_t *>(T.qbits);
    uint16_t *xg = const_cast<uint16_t *>(T.xguide), *qg = const_cast<uint16_t *>(T.qguide);
    FixCell *xf = const_cast<FixCell *>(T.xfix), *qf = const_cast<FixCell *>(T.qfix);
    for (int k = threadIdx.x; k < kLogTab; k += blockDim.x) {
        lg[k] = g.flog[k];
        iv[k] = g.finv[k];
    }
    for (int k = threadIdx.x; k < g.nxc; k += blockDim.x) xf[k] = g.xfix[k];
    for (int k = threadIdx.x; k < g.nqc; k += blockDim.x) qf[k] = g.qfix[k];
    for (int k = threadIdx.x; k < g.nxc + kGuideRun; k += blockDim.x) xb[k] = g.xbits[k];
    for (int k = threadIdx.x; k < g.nqc + kGuideRun; k += blockDim.x) qb[k] = g.qbits[k];
    for (int k = threadIdx.x; k < g.nxg; k += blockDim.x) xg[k] = g.xguide[k];
    for (int k = threadIdx.x; k < g.nqg; k += blockDim.x) qg[k] = g.qguide[k];
    return T;
}

// Weights of the quad's four points for this lane's row, from every lane's
// own two coordinates.  16-byte chunk c of point p sits at slot
// 8 p + (c ^ swizzle(p)): stores and loads of 8 lanes meet 8 different banks.
__device__ __forceinline__ int weight_swizzle(int p) { return ((p & 3) << 1) | ((p >> 2) & 1); }

__device__ __forceinline__ void quad_weights(uint4 *buf, int lane, int64_t tx, int64_t tq, Dig W[4][4])
{
    Dig w[16];
    fix_weights(tx - kFixHalf, tq - kFixHalf, w);
    const int sw = weight_swizzle(lane);
#pragma unroll
    for (int c = 0; c < 8; ++c)
        buf[8 * lane + (c ^ sw)] = make_uint4(w[2 * c].h, w[2 * c].l, w[2 * c + 1].h, w[2 * c + 1].l);
    __syncwarp();
    const int r = lane & 3;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int p = (lane & ~3) | j, sp = weight_swizzle(p);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint4 v = buf[8 * p + ((2 * r + h) ^ sp)];
            W[j][2 * h] = {(int)v.x, (int)v.y};
            W[j][2 * h + 1] = {(int)v.z, (int)v.w};
        }
    }
    __syncwarp();
}

// Position of a lane in its quad, as two flags.
struct QuadPos {
    bool up, odd;
};
__device__ __forceinline__ QuadPos quad_pos(int lane) { return {(lane & 2) != 0, (lane & 1) != 0}; }

// Row sums of the quad's four points -> the patch of this lane's own point.
__device__ __forceinline__ int64_t quad_sum(const int64_t s[4], QuadPos r)
{
    int64_t a = r.up ? s[2] : s[0], b = r.up ? s[3] : s[1];
    const int64_t c = r.up ? s[0] : s[2], d = r.up ? s[1] : s[3];
    a += __shfl_xor_sync(kAll, c, 2);
    b += __shfl_xor_sync(kAll, d, 2);
    const int64_t k = r.odd ? b : a, t = r.odd ? a : b;
    return k + __shfl_xor_sync(kAll, t, 1);
}

// One patch per point of the warp: `off[j]` is the byte offset from `base` of
// this lane's row of point j of the quad.
__device__ __forceinline__ void quad_load(const unsigned char *base, const uint32_t off[4], int c[4][8])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) fix_ld(base + off[j], c[j]);
}

// The low word of the last coefficient of this lane's own patch (the block
// exponent; every row has it).
__device__ __forceinline__ int quad_last(const int c[4][8], QuadPos r)
{
    const int lo = r.odd ? c[1][6] : c[0][6], hi = r.odd ? c[3][6] : c[2][6];
    return r.up ? hi : lo;
}

// The fixed-point value of this lane's own point, and in `last` quad_last.
__device__ __forceinline__ int64_t quad_patch(const int c[4][8], const Dig W[4][4], QuadPos r, int &last)
{
    last = quad_last(c, r);
    int64_t s[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = fix_row(c[j], W[j]);
    return quad_sum(s, r);
}

// The two derivatives of the same patch.  A row's derivative in t_q takes the
// weights of the row before it, which are read again from the buffer that
// quad_weights left.
__device__ __forceinline__ void quad_patch_d(const int c[4][8], const Dig W[4][4], const uint4 *buf, int lane,
                                             QuadPos pos, int64_t &dx, int64_t &dq)
{
    const int r = lane & 3, prev = max(r - 1, 0);
    int64_t sx[4], sq[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        sx[j] = fix_row_dx(c[j], W[j]);
        const int p = (lane & ~3) | j, sp = weight_swizzle(p);
        Dig V[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint4 v = buf[8 * p + ((2 * prev + h) ^ sp)];
            V[2 * h] = {(int)v.x, (int)v.y};
            V[2 * h + 1] = {(int)v.z, (int)v.w};
        }
        const int64_t t = fix_row(c[j], V);
        sq[j] = (pos.odd ? t : 0) + (pos.up ? 2 * t : 0);        // r t
    }
    dx = quad_sum(sx, pos);
    dq = quad_sum(sq, pos);
}

// Byte offsets of this lane's rows of the quad's points, from each lane's own
// patch offset.
__device__ __forceinline__ void quad_offsets(uint32_t own, int lane, uint32_t off[4])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) off[j] = __shfl_sync(kAll, own, (lane & ~3) | j) + (lane & 3) * 32;
}

// alpha_s inside the Q range at a fixed-point coordinate, from the row of its
// cell; `none` is set where the cell's cubic needs FP64.
__device__ __forceinline__ double fix_alphas(const int c[8], int64_t t, bool &none)
{
    Dig w[4];
    w[0] = {1 << 30, 0};
    w[1] = fix_split(t - kFixHalf);
    w[2] = fix_split(fix_mul(w[1], w[1]));
    w[3] = fix_split(fix_mul(w[2], w[1]));
    none = fix_needs_fp64(c[6], kFixNone);
    return fix_value(fix_row(c, w), c[6]);
}
__device__ __forceinline__ double fix_alphas(const GridDev &g, int cell, int64_t t, bool &none)
{
    int c[8];
    fix_ld(reinterpret_cast<const unsigned char *>(g.facoef) + (size_t)cell * 32, c);
    return fix_alphas(c, t, none);
}

// alpha_s at any point of the Q axis; FP64 arithmetic where it has no
// fixed-point coordinate.
__device__ __forceinline__ double alphas_at(const GridDev &g, const Axis &Q, bool *oor)
{
    *oor = g.extrap == PDF_EXTRAP_ERROR && !Q.in;
    if (*oor) return dnan();
    if (Q.f >= 0) {
        bool none;
        const double a = fix_alphas(g, Q.cell, Q.f, none);
        if (!none) return a;
    }
    return alphas_any(g, ld4(g.acoef + (size_t)Q.cell * 4), Q);
}

// What an evaluation of 32 points reads and writes: a matrix-form query of
// `npid` columns scol[] of one member.  Outputs of flavours [a0, a1) go to
// out[i][a]; tape and alphas may be null (with the flags off).
struct Query {
    const signed char *scol;
    int npid, a0, a1;
    const double *cm;             // the member's FP64 patches
    const unsigned char *fm;      // its fixed-point patches
    const double *x, *q;
    int64_t n;
    double *out, *tape, *alphas;
};

// A warp's buffers in shared memory and the fill of its queue.
struct WarpBufs {
    uint4 *buf;        // kWarpBuf bytes at least: weights, then the staged output rows
    int64_t *queue;    // kQueue slots
    int qn;
};

// A lane's share of the queue: its point (-1: none), and which of the `count`
// lanes of that point it is.
struct Queued {
    int64_t i;
    int sub, count;
};

// One point in FP64: domain errors, points outside the knots, cells that the
// format does not serve; of a point in a cell that it serves only the patches
// that the format does not hold (its other flavours keep the bits that any
// other query gives them).
__device__ __forceinline__ void slow_point(const GridDev &g, const CoordTabs &T, const Query &Y, bool q_is_q, Queued e)
{
    const int64_t i = e.i;
    double xi = Y.x[i], qi = Y.q[i];
    if (q_is_q) qi = qi * qi;
    const bool qbad = !q2_ok(dbits(qi));
    bool bad = qbad || !x_ok(dbits(xi));
    flag_status(g, bad);
    if (bad) {
        xi = 0.5;
        if (!Y.alphas || qbad) qi = 10.0;
    }
    const Axis X = axis_x(g, T, xi), Q = axis_q2(g, T, qi);
    const bool fixed = !bad && Y.fm && X.f >= 0 && Q.f >= 0;
    if (Y.alphas && e.sub == 0) {
        bool oor;
        const double a = alphas_at(g, Q, &oor);
        Y.alphas[i] = qbad ? dnan() : a;
    }
    const bool oor = out_of_range(g, X, Q);
    flag_status(g, oor, PDF_S_RANGE);
    bad |= oor;
    if (Y.tape && e.sub == 0) tape_put(Y.tape, i, X, Q, bad);
    const int limit = fix_limit(X.f, Q.f);
    const size_t patch0 = ((size_t)Q.cell * g.nxc + X.cell) * g.nflav;
    const double *cell = Y.cm + patch0 * 16;
    for (int a = Y.a0 + e.sub; a < Y.a1; a += e.count) {
        int col = Y.scol[a];
        if (col >= 0) col = checked_index(g.status, col, g.nflav);
        if (fixed && (col < 0 || !fix_needs_fp64(reinterpret_cast<const int *>(Y.fm + (patch0 + col) * 128)[6], limit)))
            continue;
        const double v = col >= 0 ? patch_any<true>(g, cell + col * 16, X, Q) : 0.0;
        Y.out[i * Y.npid + a] = bad ? dnan() : v;
    }
}

// Appends the lanes' points to the queue (at most kQueue in all: a warp's
// pass adds each lane once and starts below 32).
__device__ __forceinline__ void push_queue(WarpBufs &B, bool mine, int64_t i, int lane)
{
    const unsigned m = __ballot_sync(kAll, mine);
    if (!m) return;
    if (mine) B.queue[B.qn + __popc(m & ((1u << lane) - 1))] = i;
    B.qn += __popc(m);
    __syncwarp();
}

// Takes up to 32 points off the queue; with fewer than 32 the lanes share
// them, a power of two of lanes to a point (the last points of a warp would
// else wait for one lane's whole list of patches: 1000 events of which 5 % lie
// outside the knots, 61 -> 37 us).
__device__ __forceinline__ Queued next_queued(WarpBufs &B, int lane)
{
    __syncwarp();
    const int m = min(B.qn, 32);
    const int shift = m > 1 ? 32 - __clz(m - 1) : 0;          // 2^shift slots for m points
    Queued e;
    e.count = 32 >> shift;
    e.sub = lane & (e.count - 1);
    const int slot = lane >> (5 - shift);
    e.i = slot < m ? B.queue[slot] : -1;
    const int64_t rest = lane + 32 < B.qn ? B.queue[lane + 32] : 0;
    __syncwarp();
    B.queue[lane] = rest;
    B.qn -= m;
    __syncwarp();
    return e;
}

// The queue's first 32 points in FP64, after the rows staged for them have
// been written; the lanes that share a point share its columns.
__device__ __forceinline__ void drain_queue(const GridDev &g, const CoordTabs &T, const Query &Y, bool q_is_q, WarpBufs &B,
                                            int lane)
{
    if (lane == 0) bulk_wait_all();
    const Queued e = next_queued(B, lane);
    if (e.i >= 0) slow_point(g, T, Y, q_is_q, e);
    __syncwarp();
}

// 32 points [base, base + 32) of a query by one warp.  WHOLE: all the columns
// (a0 = 0, a1 = npid), whose rows leave the warp as one contiguous run.
template <bool Q_IS_Q, bool TAPE, bool AS, bool WHOLE>
__device__ __forceinline__ void eval_points(const GridDev &g, const CoordTabs &T, const Query &Y, WarpBufs &B,
                                            int64_t base, int lane)
{
    const int64_t i = base + lane;
    const bool live = i < Y.n;
    const double xi = live ? Y.x[i] : 0.5;
    double qi = live ? Y.q[i] : 10.0;
    if (Q_IS_Q) qi = qi * qi;
    // inside the knots, so inside the domain (32 points outside: no coordinates)
    // 32 points outside the knots need no coordinates here.  In long queries the
    // test would make every pass wait for the points first (1e7 points x 13
    // flavours 1388 -> 1400 us, 400 batched requests 3130 -> 3214).
    if (!WHOLE && !__any_sync(kAll, in_x(g, dbits(xi)) && in_q2(g, dbits(qi)))) {
        push_queue(B, live, i, lane);
        return;
    }
    const FixAxis X = fix_axis_x(g, T, dbits(xi)), Q = fix_axis_q2(g, T, dbits(qi));
    const bool fast = live && X.ok && Q.ok && Y.fm;      // inside the knots, so inside the domain
    push_queue(B, live && !fast, i, lane);
    if (__any_sync(kAll, fast)) {
        if (TAPE && fast) tape_put(Y.tape, i, X, Q);
        bool none = false;                    // a patch or cubic that the format does not hold
        if (AS && fast) Y.alphas[i] = fix_alphas(g, Q.cell, Q.t, none);
        const uint32_t cell = fast ? (uint32_t)(Q.cell * g.nxc + X.cell) : 0u;
        uint32_t off[4];
        quad_offsets(cell * ((uint32_t)g.nflav * 128u), lane, off);
        warp_run_reuse(lane);                 // the previous run has left the buffer
        Dig W[4][4];
        quad_weights(B.buf, lane, fast ? X.t : kFixHalf, fast ? Q.t : kFixHalf, W);
        double *srow = reinterpret_cast<double *>(B.buf) + lane * Y.npid;
        const QuadPos pos = quad_pos(lane);
        const int limit = fix_limit(X.t, Q.t);
        for (int a = Y.a0; a < Y.a1; ++a) {
            int col = Y.scol[a];
            double v = 0.0;
            if (col >= 0) {                   // the same for the whole warp
                col = checked_index(g.status, col, g.nflav);
                int c[4][8], last;
                quad_load(Y.fm + col * 128, off, c);
                const int64_t s = quad_patch(c, W, pos, last);
                v = fix_value(s, last);
                none |= fix_needs_fp64(last, limit);
            }
            if (WHOLE) srow[a] = v;
            else if (fast) Y.out[i * Y.npid + a] = v;
        }
        if (WHOLE) {
            const int rows = (int)min((int64_t)32, Y.n - base);
            warp_run_store(Y.out + base * Y.npid, reinterpret_cast<double *>(B.buf), rows * Y.npid, lane);
        }
        push_queue(B, fast && none, i, lane);
    }
    if (B.qn >= 32) drain_queue(g, T, Y, Q_IS_Q, B, lane);
}

}  // namespace pdfgpu
