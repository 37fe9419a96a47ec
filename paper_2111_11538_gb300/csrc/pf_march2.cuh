// Warp-marching sweeps of the 2D Q1 operator (the V-cycle of pf_mg.cuh).
//
// A work item is a strip of 32 node columns (one per lane) over a chunk of
// rows; one warp marches it along y with everything in registers.  A row's
// operand is formed from its own lane's words, which are loaded while the row
// before is worked on, its sums and differences with the right neighbour come
// from one shuffle per component, a cell row is formed from two such rows,
// and the forces that a cell row leaves on the row above are carried to the
// next step.  Right-corner forces reach their node by one shuffle.  No block
// barrier: the warps of a block drift apart, so that one warp's loads overlap
// another's arithmetic, and the whole sweep costs one pass of latency and the
// grid barrier that follows it.  (Copying the words ahead into shared memory
// with 4-byte cp.async, three rows deep, was slower: each copy took 5.6
// shared-memory wavefronts where a load into a register takes one or two.)
//
// What it replaced: 32x16 node tiles staged through shared memory with three
// block barriers per tile, at 20 % issue (barrier and load latency) and, in
// FP64, with the coarse levels' few tiles on as few SMs.  Items here are 30
// (28 for two products) columns by a few rows, dealt to the blocks first and
// to their warps second, so that a 64^2 level still uses every SM.
#pragma once

namespace pfdev {

// A lane and the lanes of its right and left neighbour columns.  A grid of
// at most 32 columns is one strip of whole periodic rows (per: its last lane's
// neighbour is lane 0), without halo columns.
struct Lanes2 {
    int lane, nxt, prv;
    bool per;
    __device__ __forceinline__ Lanes2(int nx)
    {
        lane = threadIdx.x & 31;
        per = nx <= 32;
        nxt = per ? (lane + 1 >= nx ? 0 : lane + 1) : min(lane + 1, 31);
        prv = per ? (lane == 0 ? nx - 1 : lane - 1) : max(lane - 1, 0);
    }
};

// the row's displacement (FP32: its sum with the right neighbour's) and its
// difference to the right neighbour
template <typename T>
struct Row2 {
    T v[2], d[2];
};

template <typename T>
__device__ __forceinline__ void row2(const T (&v)[2], const Lanes2 &Ln, Row2<T> &R)
{
#pragma unroll
    for (int c = 0; c < 2; c++) {
        const T r = __shfl_sync(0xffffffffu, v[c], Ln.nxt);
        R.v[c] = sizeof(T) == 8 ? v[c] : v[c] + r;
        R.d[c] = r - v[c];
    }
}

// Corner-force coefficients of the cell between rows lo and hi (l4, m4: a
// quarter of its moduli): the force on its corner (sx, sy), s = -1 or +1, is
// sx ax + sy ay + sx sy axy per component.  This is cell_force2 /
// node_force2 with the sums along x and y taken apart.
// FP64 takes differences of neighbours first, as there: they are nearly exact
// where the field is smooth (the y gradient, the sum of both columns'
// differences, is 2 (hi.v - lo.v) + (hi.d - lo.d)).  The difference of the rows'
// sums, as many operations, costs digits: relative error of A u at 256^2, a
// smooth u, 5.1e-14 against 2.6e-15, at 2048^2 3.3e-12 against 2.1e-14.
// FP32, whose passes only precondition the FP64 residual, takes the rows' sums:
// the FP64 residual after a pass is the pass's own to 2 % up to 8192^2, the
// V-cycles are as many either way, and differences first take 2 to 3 % longer
// (a chain longer by one operation; 2048^2 0.471 and 0.481 ms per V-cycle).
template <typename T>
struct Cell2 {
    T ax0, sh, ay1, xy[2];          // ax = (ax0, sh), ay = (sh, ay1)
};

template <typename T>
__host__ __device__ __forceinline__ Cell2<T> cell2(T l4, T m4, const Row2<T> &lo, const Row2<T> &hi)
{
    const T gxu = lo.d[0] + hi.d[0], gxv = lo.d[1] + hi.d[1];
    const T xyu = hi.d[0] - lo.d[0], xyv = hi.d[1] - lo.d[1];
    const T dyu = hi.v[0] - lo.v[0], dyv = hi.v[1] - lo.v[1];
    const T gyu = sizeof(T) == 8 ? T(2) * dyu + xyu : dyu, gyv = sizeof(T) == 8 ? T(2) * dyv + xyv : dyv;
    const T lt = l4 * (gxu + gyv), m2 = m4 + m4;
    const T ch = (l4 + T(3) * m4) * T(1.0 / 3.0);
    Cell2<T> C;
    C.ax0 = lt + m2 * gxu;
    C.ay1 = lt + m2 * gyv;
    C.sh = m4 * (gyu + gxv);
    C.xy[0] = ch * xyu;
    C.xy[1] = ch * xyv;
    return C;
}

// the mean strain's part (ue: Voigt mean strain)
template <typename T>
__device__ __forceinline__ void cell2_mean(T l4, T m4, const T *ue, Cell2<T> &C)
{
    const T lt = T(2) * l4 * (ue[0] + ue[1]), m2 = T(4) * m4;
    C.ax0 += lt + m2 * ue[0];
    C.ay1 += lt + m2 * ue[1];
    C.sh += T(2) * m4 * ue[2];
}

// Left-corner (O subtracted) and right-corner (O added) sums of a node row:
// the row below a cell row ends with it (lower), the row above starts.
template <typename T>
struct Node2 {
    T E[2], O[2];
    __device__ __forceinline__ void start(const Cell2<T> &C)      // upper corners of the cell row below
    {
        E[0] = C.sh;
        E[1] = C.ay1;
        O[0] = C.ax0 + C.xy[0];
        O[1] = C.sh + C.xy[1];
    }
    __device__ __forceinline__ void finish(const Cell2<T> &C, const Lanes2 &Ln, T (&q)[2])   // lower corners of the cell row above
    {
        const T e[2] = {E[0] - C.sh, E[1] - C.ay1};
        const T o[2] = {O[0] + (C.ax0 - C.xy[0]), O[1] + (C.sh - C.xy[1])};
#pragma unroll
        for (int c = 0; c < 2; c++) q[c] = (e[c] - o[c]) + __shfl_sync(0xffffffffu, e[c] + o[c], Ln.prv);
    }
};

// The sweeps' part of the dynamic shared memory starts at byte OFF: the
// operation's record.
constexpr int M2_OP_BYTES = 320;
extern __shared__ __align__(16) unsigned char pcg_dyn[];

// Rows per work item of an nx x ny level for nbk blocks of nwb warps, with
// strips of OW columns and `extra` rows of start-up: the candidate with the
// least time by a simple count.  FP32 sweeps are bound by a warp's latency
// (items per warp, rounded up, times rows; a first row's copies cost about
// four rows' work); FP64 ones by the FP64 pipes, one per quarter of an SM, and
// by the loads between (a row of a lone warp takes as long as its FP64
// instructions, 64 cycles each): two items to a pipe, so that one's loads
// overlap another's arithmetic, but one in a job of one or two blocks, whose
// short chunks cost more rows of start-up than that gains.  One / two / four
// items per pipe, ms per step: 512^2 7.18 / 6.68 / 7.22, batches of 32 x 128^2
// 12.05 / 10.63 / 10.35, of 16 x 256^2 17.9 / 14.9 / 14.5, of 64 x 64^2 (two
// blocks each) 6.56 / 6.74 / 7.00; one in all, the batch of 32 was slower than
// the tiled sweeps (11.57).  Where two blocks share an SM (more than 2^18
// nodes) the count is still per block: 1024^2 73.6, counted per SM 90.4.
inline int m2_chunk(int nx, int ny, int nbk, int nwb, int OW, int extra, bool fp64)
{
    const long long ns = nx <= 32 ? 1 : (nx + OW - 1) / OW;
    const long long units = (nbk > 2 ? 8LL : 4LL) * nbk;
    int best = ny;
    long long bcost = -1;
    for (int zc = 1; zc <= ny; zc++) {
        const long long items = ns * ((ny + zc - 1) / zc);
        const long long cost = fp64 ? ((items + units - 1) / units) * (zc + extra)
                                    : ((items + (long long)nbk * nwb - 1) / ((long long)nbk * nwb)) * (zc + extra + 4);
        if (bcost < 0 || cost < bcost) {
            bcost = cost;
            best = zc;
        }
    }
    return best;
}

// One product: op.load(g, gx, gy, own, lanes, R) loads the words of node g
// (own: an output row), op.form(R, g, own, lanes, gx, v, keep, S) gives the operand
// v of the node (own: an output node; keep[3] is handed to the epilogue),
// op.mod(R, l, m) the moduli of the cell at the node and op.epi(g, v, q, keep,
// S) receives q = A v at every output node.  op.cell(C, S) gets every own cell
// before the mean strain op.ue is added (op.E); S collects what they sum and
// is returned.  Not inlined: a sweep then has the registers to itself.
template <typename T, int NT, size_t OFF, class OP>
__device__ __noinline__ typename OP::Sums m2_sweep(int nx, int ny, int zc, int bid, int nbk)
{
    const OP op = *reinterpret_cast<const OP *>(pcg_dyn + OFF);
    const Lanes2 Ln(nx);
    const int lane = Ln.lane, nw = (NT / 32) * nbk;
    typename OP::Sums S;
    const int ns = Ln.per ? 1 : (nx + 29) / 30, items = ns * ((ny + zc - 1) / zc);
    for (int item = (int)(threadIdx.x >> 5) * nbk + bid; item < items; item += nw) {
        const int x0 = (item % ns) * 30, y0 = (item / ns) * zc, y1 = min(y0 + zc, ny);
        const int gxr = Ln.per ? lane : x0 - 1 + lane, gx = wrapm(gxr, nx);
        const bool ownx = (Ln.per || (lane >= 1 && lane <= 30)) && gxr < nx;
        typename OP::Raw R;
        int gy = wrap(y0 - 1, ny);
        op.load(gx + nx * gy, gx, gy, false, Ln, R);
        Row2<T> lo;
        Node2<T> nd;
        T vl[2] = {T(0), T(0)}, kl[3] = {T(0), T(0), T(0)}, l4 = T(0), m4 = T(0);
        for (int y = y0 - 1; y <= y1; y++) {
            T v[2], k[3], ln, mn;
            op.form(R, gx + nx * gy, ownx && y >= y0 && y < y1, Ln, gx, v, k, S);
            op.mod(R, ln, mn);
            gy = gy + 1 == ny ? 0 : gy + 1;
            if (y < y1) op.load(gx + nx * gy, gx, gy, y + 1 < y1, Ln, R);
            Row2<T> hi;
            row2(v, Ln, hi);
            if (y >= y0) {
                Cell2<T> C = cell2(l4, m4, lo, hi);
                const bool own = ownx && y > y0;             // node row y - 1 and the cells at it
                if constexpr (OP::E) {
                    if (own) op.cell(C, S);
                    cell2_mean(l4, m4, op.ue, C);
                }
                if (y > y0) {
                    T q[2];
                    nd.finish(C, Ln, q);
                    if (own) op.epi(gx + nx * (y - 1), vl, q, kl, S);
                }
                nd.start(C);
            }
            lo = hi;
            l4 = T(0.25) * ln;
            m4 = T(0.25) * mn;
#pragma unroll
            for (int c = 0; c < 2; c++) vl[c] = v[c];
#pragma unroll
            for (int c = 0; c < 3; c++) kl[c] = k[c];
        }
    }
    return S;
}

// Two products, the second one row behind the first: op.form(R, lanes, gx, v, a)
// gives the first operand v and an auxiliary a[3]; op.mid(v, a, q, r, w)
// the intermediate r and second operand w from q = A v; op.epi(g, v, a, r,
// w, q, S) gets q = A w at every output node (28 columns per strip).
template <typename T, int NT, size_t OFF, class OP>
__device__ __noinline__ typename OP::Sums m2_sweep2(int nx, int ny, int zc, int bid, int nbk)
{
    const OP op = *reinterpret_cast<const OP *>(pcg_dyn + OFF);
    const Lanes2 Ln(nx);
    const int lane = Ln.lane, nw = (NT / 32) * nbk;
    typename OP::Sums S;
    const int ns = Ln.per ? 1 : (nx + 27) / 28, items = ns * ((ny + zc - 1) / zc);
    for (int item = (int)(threadIdx.x >> 5) * nbk + bid; item < items; item += nw) {
        const int x0 = (item % ns) * 28, y0 = (item / ns) * zc, y1 = min(y0 + zc, ny);
        const int gxr = Ln.per ? lane : x0 - 2 + lane, gx = wrapm(gxr, nx);
        const bool ownx = (Ln.per || (lane >= 2 && lane <= 29)) && gxr < nx;
        typename OP::Raw R;
        int gy = wrapm(y0 - 2, ny);
        op.load(gx + nx * gy, gx, gy, Ln, R);
        Row2<T> lo0, lo1;
        Node2<T> n0, n1;
        // row y - 1 of the first operand, row y - 2 of the second
        T v1[2] = {T(0), T(0)}, a1[3] = {T(0), T(0), T(0)}, l1 = T(0), m1 = T(0);
        T v2[2] = {T(0), T(0)}, a2[3] = {T(0), T(0), T(0)}, r2[2] = {T(0), T(0)}, w2[2] = {T(0), T(0)}, l2 = T(0), m2 = T(0);
        for (int y = y0 - 2; y <= y1 + 1; y++) {
            T v[2], a[3], ln, mn;
            op.form(R, Ln, gx, v, a);
            op.mod(R, ln, mn);
            gy = gy + 1 == ny ? 0 : gy + 1;
            if (y <= y1) op.load(gx + nx * gy, gx, gy, Ln, R);
            Row2<T> hi;
            row2(v, Ln, hi);
            T r[2] = {T(0), T(0)}, w[2] = {T(0), T(0)};
            if (y > y0 - 2) {
                const Cell2<T> C = cell2(l1, m1, lo0, hi);
                if (y >= y0) {
                    // second operand at row y - 1, its cells at row y - 2
                    T q[2];
                    n0.finish(C, Ln, q);
                    op.mid(v1, a1, q, r, w);
                    Row2<T> h1;
                    row2(w, Ln, h1);
                    if (y > y0) {
                        Cell2<T> C1 = cell2(l2, m2, lo1, h1);
                        const bool own = ownx && y > y0 + 1;
                        if constexpr (OP::E) {
                            if (own) op.cell(C1, S);
                            cell2_mean(l2, m2, op.ue, C1);
                        }
                        if (y > y0 + 1) {
                            T q1[2];
                            n1.finish(C1, Ln, q1);
                            if (own) op.epi(gx + nx * (y - 2), v2, a2, r2, w2, q1, S);
                        }
                        n1.start(C1);
                    }
                    lo1 = h1;
                }
                n0.start(C);
            }
            lo0 = hi;
#pragma unroll
            for (int c = 0; c < 2; c++) { v2[c] = v1[c]; r2[c] = r[c]; w2[c] = w[c]; v1[c] = v[c]; }
#pragma unroll
            for (int c = 0; c < 3; c++) { a2[c] = a1[c]; a1[c] = a[c]; }
            l2 = l1;
            m2 = m1;
            l1 = T(0.25) * ln;
            m1 = T(0.25) * mn;
        }
    }
    return S;
}

// a pair of neighbouring values, the first at an even index (through L1: the
// restriction reads every fine row from up to two coarse rows)
__device__ __forceinline__ void ld_pair(const float *p, float (&v)[2])
{
    const float2 a = __ldca(reinterpret_cast<const float2 *>(p));
    v[0] = a.x;
    v[1] = a.y;
}
__device__ __forceinline__ void ld_pair(const double *p, double (&v)[2])
{
    const double2 a = __ldca(reinterpret_cast<const double2 *>(p));
    v[0] = a.x;
    v[1] = a.y;
}

// The coarse correction at a fine node (bilinear prolongation of C's xpost;
// component 1 lies n values after component 0).  Each lane loads the two
// coarse rows' values at its own gx >> 1; an odd column takes the other half
// from its right neighbour's lane, the last lane of a strip with halo columns
// (an odd column) from loads of its own.
template <typename T>
struct Prolong2 {
    const T *x;
    int cnx, cny;
    struct Raw {
        T a[4], b[4];
    };
    __device__ __forceinline__ void load(int gx, int gy, const Lanes2 &Ln, Raw &R) const
    {
        const int ix = gx >> 1, iy = gy >> 1, iy1 = (gy & 1) ? (iy + 1 == cny ? 0 : iy + 1) : iy, n = cnx * cny;
#pragma unroll
        for (int c = 0; c < 2; c++) {
            R.a[2 * c] = __ldca(x + c * n + ix + cnx * iy);
            R.a[2 * c + 1] = __ldca(x + c * n + ix + cnx * iy1);
        }
        if (!Ln.per && Ln.lane == 31) {
            const int ix1 = ix + 1 == cnx ? 0 : ix + 1;
#pragma unroll
            for (int c = 0; c < 2; c++) {
                R.b[2 * c] = __ldca(x + c * n + ix1 + cnx * iy);
                R.b[2 * c + 1] = __ldca(x + c * n + ix1 + cnx * iy1);
            }
        }
    }
    __device__ __forceinline__ void add(const Raw &R, int gx, const Lanes2 &Ln, T (&v)[2]) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            // rows averaged (the same row twice on an even row)
            const T e = T(0.5) * (R.a[2 * c] + R.a[2 * c + 1]);
            T r = __shfl_sync(0xffffffffu, e, Ln.nxt);
            if (!Ln.per && Ln.lane == 31) r = T(0.5) * (R.b[2 * c] + R.b[2 * c + 1]);
            v[c] += (gx & 1) ? T(0.5) * (e + r) : e;
        }
    }
};

// The restriction (transpose of the bilinear prolongation) of the finer
// level's residual r at a coarse node: pairs (2 gx, 2 gx + 1) of the three
// fine rows around it; the value at 2 gx - 1 is the left lane's second
// entry, or a load of its own for the first lane of a
// strip with halo columns.
template <typename T>
struct Restrict2 {
    const T *r;
    int fnx, fny;
    struct Raw {
        T p[6][2], b[6];
    };
    __device__ __forceinline__ void load(int gx, int gy, const Lanes2 &Ln, Raw &R) const
    {
        const unsigned n = (unsigned)fnx * fny;
#pragma unroll
        for (int b = 0; b < 3; b++) {
            const T *row = r + fnx * wrap(2 * gy + b - 1, fny);
#pragma unroll
            for (int c = 0; c < 2; c++) {
                ld_pair(row + c * n + 2 * gx, R.p[2 * b + c]);
                if (!Ln.per && Ln.lane == 0) R.b[2 * b + c] = __ldca(row + c * n + (gx == 0 ? fnx - 1 : 2 * gx - 1));
            }
        }
    }
    __device__ __forceinline__ void get(const Raw &R, const Lanes2 &Ln, T (&f)[2]) const
    {
        f[0] = f[1] = T(0);
#pragma unroll
        for (int b = 0; b < 3; b++)
#pragma unroll
            for (int c = 0; c < 2; c++) {
                T am = __shfl_sync(0xffffffffu, R.p[2 * b + c][1], Ln.prv);
                if (!Ln.per && Ln.lane == 0) am = R.b[2 * b + c];
                const T s = R.p[2 * b + c][0] + T(0.5) * (am + R.p[2 * b + c][1]);
                f[c] += b == 1 ? s : T(0.5) * s;
            }
    }
};

// ---------------------------------------------------------------------------
// The sweeps of the V-cycle.  An operation is a plain record, filled in shared
// memory by one thread; component 1 of a vector lies n values after
// component 0 (unsigned: g + n reaches 2^32 on a grid of 2^31 nodes).  What a thread sums goes into Sums.
// ---------------------------------------------------------------------------
// gamma = r.u, delta = w.u and half the own cells' stresses (of u, without
// the mean strain)
template <typename T>
struct Sums2 {
    Acc<T> ru, wu, se[3];
};

// Finest level, first pre-smoothing step, with the CG update of the previous
// iteration (upd) at the output nodes:
//   p = u + beta p, s = w + beta s, x += alpha p, r -= alpha s
// (u: the previous V-cycle's result), then v = c2 D^-1 r, r1 = r - A v.
template <typename T>
struct OpFirst2 {
    static constexpr bool E = false;
    const T *lam, *mu, *dinv, *r, *w, *s, *u;
    T *p, *x[2], *sn, *rn, *xpre, *r1, *d1;
    T ta, tb, c2;
    unsigned n;
    bool upd, dir;              // dir: keep the direction for further smoothing steps
    typedef Acc<T> Sums;        // ||r||^2
    struct Raw {
        T l, m, di, r[2], w[2], s[2], u[2], p[2], x[2];
    };
    __device__ __forceinline__ void load(int g, int, int, bool own, const Lanes2 &, Raw &R) const
    {
        R.l = __ldcg(lam + g);
        R.m = __ldcg(mu + g);
        R.di = __ldcg(dinv + g);
#pragma unroll
        for (int c = 0; c < 2; c++) {
            R.r[c] = __ldcg(r + g + c * n);
            if (upd) {
                R.w[c] = __ldcg(w + g + c * n);
                R.s[c] = __ldcg(s + g + c * n);
                if (own) {
                    R.u[c] = __ldcg(u + g + c * n);
                    R.p[c] = __ldcg(p + g + c * n);
                    R.x[c] = __ldcg(x[c] + g);
                }
            }
        }
    }
    __device__ __forceinline__ void mod(const Raw &R, T &l, T &m) const { l = R.l; m = R.m; }
    __device__ __forceinline__ void form(const Raw &R, int g, bool own, const Lanes2 &, int, T (&v)[2], T (&k)[3], Sums &S) const
    {
        const T di = c2 * R.di;
        k[2] = T(0);
#pragma unroll
        for (int c = 0; c < 2; c++) {
            T f = R.r[c];
            if (upd) {
                const T si = R.w[c] + tb * R.s[c];
                f -= ta * si;
                if (own) {
                    const T pi = R.u[c] + tb * R.p[c];
                    p[g + c * n] = pi;
                    x[c][g] = R.x[c] + ta * pi;
                    sn[g + c * n] = si;
                    rn[g + c * n] = f;
                    S.fma_plain(f, f);
                }
            }
            v[c] = di * f;
            k[c] = f;
            if (own) {
                xpre[g + c * n] = v[c];
                if (dir) d1[g + c * n] = v[c];
            }
        }
    }
    __device__ __forceinline__ void epi(int g, const T (&)[2], const T (&q)[2], const T (&k)[3], Sums &) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) r1[g + c * n] = k[c] - q[c];
    }
};

// Chebyshev step: d = c1 d + c2 D^-1 r, x += d, r' = r - A d; last: the next
// step as well (x + d + n1 d + n2 D^-1 r'), into xo.
template <typename T>
struct OpCheb2 {
    static constexpr bool E = false;
    const T *lam, *mu, *dinv, *r, *d, *xi;
    T *xo, *rn, *dn;
    T c1, c2, n1, n2;
    unsigned n;
    bool last, dir;            // dir: the step has a previous direction d
    typedef Acc<T> Sums;
    struct Raw {
        T l, m, di, r[2], d[2], x[2];
    };
    __device__ __forceinline__ void load(int g, int, int, bool own, const Lanes2 &, Raw &R) const
    {
        R.l = __ldcg(lam + g);
        R.m = __ldcg(mu + g);
        R.di = __ldcg(dinv + g);
#pragma unroll
        for (int c = 0; c < 2; c++) {
            R.r[c] = __ldcg(r + g + c * n);
            R.d[c] = dir ? __ldcg(d + g + c * n) : T(0);
            if (own) R.x[c] = __ldcg(xi + g + c * n);
        }
    }
    __device__ __forceinline__ void mod(const Raw &R, T &l, T &m) const { l = R.l; m = R.m; }
    __device__ __forceinline__ void form(const Raw &R, int g, bool own, const Lanes2 &, int, T (&v)[2], T (&k)[3], Sums &) const
    {
        const T di = c2 * R.di, dl = n2 * R.di;
        k[2] = dl;
#pragma unroll
        for (int c = 0; c < 2; c++) {
            v[c] = di * R.r[c] + c1 * R.d[c];
            k[c] = R.r[c];
            if (own) {
                const T xn = R.x[c] + v[c];
                if (last) {
                    k[c] = xn + n1 * v[c] + dl * R.r[c];
                } else {
                    xo[g + c * n] = xn;
                    dn[g + c * n] = v[c];
                }
            }
        }
    }
    __device__ __forceinline__ void epi(int g, const T (&)[2], const T (&q)[2], const T (&k)[3], Sums &) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            if (last) xo[g + c * n] = k[c] - k[2] * q[c];
            else rn[g + c * n] = k[c] - q[c];
        }
    }
};

// First step of the coarsest level's solve: f = R r, v = c2 D^-1 f, r1 = f - A v.
template <typename T>
struct OpPre2 {
    static constexpr bool E = false;
    const T *lam, *mu, *dinv;
    Restrict2<T> Rs;
    T *f, *xpre, *r1, *d1;
    T c2;
    unsigned n;
    typedef Acc<T> Sums;
    struct Raw {
        T l, m, di;
        typename Restrict2<T>::Raw f;
    };
    __device__ __forceinline__ void load(int g, int gx, int gy, bool, const Lanes2 &Ln, Raw &R) const
    {
        R.l = __ldcg(lam + g);
        R.m = __ldcg(mu + g);
        R.di = __ldcg(dinv + g);
        Rs.load(gx, gy, Ln, R.f);
    }
    __device__ __forceinline__ void mod(const Raw &R, T &l, T &m) const { l = R.l; m = R.m; }
    __device__ __forceinline__ void form(const Raw &R, int g, bool own, const Lanes2 &Ln, int, T (&v)[2], T (&k)[3], Sums &) const
    {
        T ff[2];
        Rs.get(R.f, Ln, ff);
        const T di = c2 * R.di;
        k[2] = T(0);
#pragma unroll
        for (int c = 0; c < 2; c++) {
            k[c] = ff[c];
            v[c] = di * ff[c];
            if (own) { f[g + c * n] = ff[c]; xpre[g + c * n] = v[c]; d1[g + c * n] = v[c]; }
        }
    }
    __device__ __forceinline__ void epi(int g, const T (&)[2], const T (&q)[2], const T (&k)[3], Sums &) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) r1[g + c * n] = k[c] - q[c];
    }
};

// w = A u with the mean strain, gamma = r.u, delta = w.u and the own cells'
// stresses (one-level hierarchies; the others fuse it, OpFine2).
template <typename T>
struct OpApply2 {
    static constexpr bool E = true;
    const T *lam, *mu, *u, *r;
    T *w;
    T ue[3];
    unsigned n;
    typedef Sums2<T> Sums;
    struct Raw {
        T l, m, u[2], r[2];
    };
    __device__ __forceinline__ void load(int g, int, int, bool own, const Lanes2 &, Raw &R) const
    {
        R.l = __ldcg(lam + g);
        R.m = __ldcg(mu + g);
#pragma unroll
        for (int c = 0; c < 2; c++) {
            R.u[c] = __ldcg(u + g + c * n);
            if (own) R.r[c] = __ldcg(r + g + c * n);
        }
    }
    __device__ __forceinline__ void mod(const Raw &R, T &l, T &m) const { l = R.l; m = R.m; }
    __device__ __forceinline__ void form(const Raw &R, int, bool own, const Lanes2 &, int, T (&v)[2], T (&k)[3], Sums &S) const
    {
        k[2] = T(0);
#pragma unroll
        for (int c = 0; c < 2; c++) {
            v[c] = R.u[c];
            k[c] = T(0);
            if (own) S.ru.fma_plain(R.r[c], v[c]);
        }
    }
    __device__ __forceinline__ void cell(const Cell2<T> &C, Sums &S) const
    {
        S.se[0].add_plain(C.ax0);
        S.se[1].add_plain(C.ay1);
        S.se[2].add_plain(C.sh);
    }
    __device__ __forceinline__ void epi(int g, const T (&v)[2], const T (&q)[2], const T (&)[3], Sums &S) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            w[g + c * n] = q[c];
            S.wu.fma_plain(q[c], v[c]);
        }
    }
};

// Two-step pre-smoothing of a coarse level: f = R r, d0 = c20 D^-1 f, r1 = f -
// A d0, d1 = c11 d0 + c21 D^-1 r1, x = d0 + d1, r2 = r1 - A d1.
template <typename T>
struct OpPrePair2 {
    static constexpr bool E = false;
    const T *lam, *mu, *dinv;
    Restrict2<T> Rs;
    T *f, *xpre, *r2;
    T c20, c11, c21;
    unsigned n;
    typedef Acc<T> Sums;
    struct Raw {
        T l, m, di;
        typename Restrict2<T>::Raw f;
    };
    __device__ __forceinline__ void load(int g, int gx, int gy, const Lanes2 &Ln, Raw &R) const
    {
        R.l = __ldcg(lam + g);
        R.m = __ldcg(mu + g);
        R.di = __ldcg(dinv + g);
        Rs.load(gx, gy, Ln, R.f);
    }
    __device__ __forceinline__ void mod(const Raw &R, T &l, T &m) const { l = R.l; m = R.m; }
    __device__ __forceinline__ void form(const Raw &R, const Lanes2 &Ln, int, T (&v)[2], T (&a)[3]) const
    {
        T ff[2];
        Rs.get(R.f, Ln, ff);
        const T di = c20 * R.di;
        a[2] = c21 * R.di;
#pragma unroll
        for (int c = 0; c < 2; c++) { a[c] = ff[c]; v[c] = di * ff[c]; }
    }
    __device__ __forceinline__ void mid(const T (&v)[2], const T (&a)[3], const T (&q)[2], T (&r)[2], T (&w)[2]) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            r[c] = a[c] - q[c];
            w[c] = c11 * v[c] + a[2] * r[c];
        }
    }
    __device__ __forceinline__ void epi(int g, const T (&v)[2], const T (&a)[3], const T (&r)[2], const T (&w)[2],
                                        const T (&q)[2], Sums &) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            f[g + c * n] = a[c];
            xpre[g + c * n] = v[c] + w[c];
            r2[g + c * n] = r[c] - q[c];
        }
    }
};

// What a post-smoothing starts from: x_pre + P e and the right-hand side f.
template <typename T>
struct PostRaw2 {
    T l, m, di, f[2], x[2];
    typename Prolong2<T>::Raw e;
};
template <typename T, class OP>
__device__ __forceinline__ void post_load2(const OP &op, const T *f, int g, int gx, int gy, const Lanes2 &Ln, PostRaw2<T> &R)
{
    R.l = __ldcg(op.lam + g);
    R.m = __ldcg(op.mu + g);
    R.di = __ldcg(op.dinv + g);
#pragma unroll
    for (int c = 0; c < 2; c++) {
        R.f[c] = __ldcg(f + g + c * op.n);
        R.x[c] = __ldcg(op.xpre + g + c * op.n);
    }
    op.P.load(gx, gy, Ln, R.e);
}

// First post-smoothing step alone (FP64): x = x_pre + P e, r = f - A x; last
// (one-step smoothing): x + c2 D^-1 r into xpost, else x and r.
template <typename T>
struct OpPost2 {
    static constexpr bool E = false;
    const T *lam, *mu, *dinv, *f, *xpre;
    Prolong2<T> P;
    T *xpost, *r;
    T c2;
    unsigned n;
    bool last;
    typedef Acc<T> Sums;
    typedef PostRaw2<T> Raw;
    __device__ __forceinline__ void load(int g, int gx, int gy, bool, const Lanes2 &Ln, Raw &R) const { post_load2(*this, f, g, gx, gy, Ln, R); }
    __device__ __forceinline__ void mod(const Raw &R, T &l, T &m) const { l = R.l; m = R.m; }
    __device__ __forceinline__ void form(const Raw &R, int g, bool own, const Lanes2 &Ln, int gx, T (&v)[2], T (&k)[3], Sums &) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) v[c] = R.x[c];
        P.add(R.e, gx, Ln, v);
        k[2] = c2 * R.di;
#pragma unroll
        for (int c = 0; c < 2; c++) {
            k[c] = last ? v[c] + k[2] * R.f[c] : R.f[c];
            if (own && !last) xpost[g + c * n] = v[c];
        }
    }
    __device__ __forceinline__ void epi(int g, const T (&)[2], const T (&q)[2], const T (&k)[3], Sums &) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            if (last) xpost[g + c * n] = k[c] - k[2] * q[c];
            else r[g + c * n] = k[c] - q[c];
        }
    }
};

// Two-step post-smoothing of a coarse level from x = x_pre + P e.
template <typename T>
struct OpPostPair2 {
    static constexpr bool E = false;
    const T *lam, *mu, *dinv, *f, *xpre;
    Prolong2<T> P;
    T *xpost;
    T c20, c11, c21;
    unsigned n;
    typedef Acc<T> Sums;
    typedef PostRaw2<T> Raw;
    __device__ __forceinline__ void load(int g, int gx, int gy, const Lanes2 &Ln, Raw &R) const { post_load2(*this, f, g, gx, gy, Ln, R); }
    __device__ __forceinline__ void mod(const Raw &R, T &l, T &m) const { l = R.l; m = R.m; }
    __device__ __forceinline__ void form(const Raw &R, const Lanes2 &Ln, int gx, T (&v)[2], T (&a)[3]) const
    {
        a[2] = R.di;
#pragma unroll
        for (int c = 0; c < 2; c++) { a[c] = R.f[c]; v[c] = R.x[c]; }
        P.add(R.e, gx, Ln, v);
    }
    __device__ __forceinline__ void mid(const T (&)[2], const T (&a)[3], const T (&q)[2], T (&r)[2], T (&w)[2]) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            r[c] = a[c] - q[c];
            w[c] = c20 * a[2] * r[c];
        }
    }
    __device__ __forceinline__ void epi(int g, const T (&v)[2], const T (&a)[3], const T (&r)[2], const T (&w)[2],
                                        const T (&q)[2], Sums &) const
    {
        const T di = c21 * a[2];
#pragma unroll
        for (int c = 0; c < 2; c++) xpost[g + c * n] = v[c] + w[c] + (c11 * w[c] + di * (r[c] - q[c]));
    }
};

// Finest level, one-step post-smoothing and the CG's product of its result:
// x = x_pre + P e, u = x + c20 D^-1 (r - A x), w = A u with the mean strain,
// gamma = r.u, delta = w.u and the own cells' stresses.
template <typename T>
struct OpFine2 {
    static constexpr bool E = true;
    const T *lam, *mu, *dinv, *r, *xpre;
    Prolong2<T> P;
    T *u, *w;
    T c20;
    T ue[3];
    unsigned n;
    typedef Sums2<T> Sums;
    typedef PostRaw2<T> Raw;
    __device__ __forceinline__ void load(int g, int gx, int gy, const Lanes2 &Ln, Raw &R) const { post_load2(*this, r, g, gx, gy, Ln, R); }
    __device__ __forceinline__ void mod(const Raw &R, T &l, T &m) const { l = R.l; m = R.m; }
    __device__ __forceinline__ void form(const Raw &R, const Lanes2 &Ln, int gx, T (&v)[2], T (&a)[3]) const
    {
        a[2] = c20 * R.di;
#pragma unroll
        for (int c = 0; c < 2; c++) { a[c] = R.f[c]; v[c] = R.x[c]; }
        P.add(R.e, gx, Ln, v);
    }
    __device__ __forceinline__ void mid(const T (&v)[2], const T (&a)[3], const T (&q)[2], T (&r_)[2], T (&w_)[2]) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            r_[c] = T(0);
            w_[c] = v[c] + a[2] * (a[c] - q[c]);
        }
    }
    __device__ __forceinline__ void cell(const Cell2<T> &C, Sums &S) const
    {
        S.se[0].add_plain(C.ax0);
        S.se[1].add_plain(C.ay1);
        S.se[2].add_plain(C.sh);
    }
    __device__ __forceinline__ void epi(int g, const T (&)[2], const T (&a)[3], const T (&)[2], const T (&w_)[2],
                                        const T (&q)[2], Sums &S) const
    {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            u[g + c * n] = w_[c];
            w[g + c * n] = q[c];
            S.ru.fma_plain(a[c], w_[c]);
            S.wu.fma_plain(q[c], w_[c]);
        }
    }
};

}  // namespace pfdev
