// Warp-marching sweeps of the 3D Q1 operator in FP32 (the V-cycle of
// pf_mg3.cuh), the counterpart of pf_march2.cuh.
//
// A work item is a strip of 30 node columns (lanes 1..30 of a warp; lanes 0
// and 31 are halo) by M3_ROWS rows over a chunk of planes; one warp marches it
// along z with everything in registers.  Per plane it walks its node rows
// (and a halo row on each side): a row's operand is formed from its own
// lane's words, loaded while the row before is worked on, and kept as its sum
// and difference with the right neighbour (one shuffle per component); a cell
// row takes four such rows, two of this plane and two of the plane before,
// which stay in registers; what a cell row leaves on the plane above is
// carried to the next plane as left/right sums, and a finished node row takes
// its right-corner part by one shuffle per component.  No shared memory and no
// block barrier.
//
// What it replaced: 32x8 node tiles per plane with the corner forces of every
// cell passed through shared memory, two block barriers per plane and a
// second, nearly empty round of cells (297 cells on 256 threads).  Taking the
// sums along x, y and z apart costs about 160 flops per cell against 270, at
// the price of 32/30 x (M3_ROWS + 1) / M3_ROWS cells per node.  256^3, us per
// sweep before and after: w = A u with its sums 690 / 618, last smoothing of
// the finest level 1230 / 742, of the 128^3 level 380 / 224; first smoothing
// with the CG update 1360 / 302 (the update's own pass: 2.0 GB, 6.7 TB/s) +
// 514; restriction and first smoothing of the 128^3 level 560 / 333.  What
// bounds it is the issue of ~400 instructions per node row by 12 warps per SM
// (registers) and their latencies: words prefetched a plane ahead into L1
// gained nothing.
#pragma once

namespace pfdev {

struct Row3 {
    float e[3], d[3];
};

__device__ __forceinline__ void row3(const float (&v)[3], const Lanes2 &Ln, Row3 &R)
{
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float r = __shfl_sync(0xffffffffu, v[c], Ln.nxt);
        R.e[c] = v[c] + r;
        R.d[c] = r - v[c];
    }
}

// Corner-force coefficients of the cell between rows a, b of the lower and
// a1, b1 of the upper plane (l, m: 1/16 of its moduli): the force on corner
// (sx, sy, sz), s = -1 or +1, is sx ax + sy ay + sz az + sx sy xy + sy sz yz +
// sz sx zx + sx sy sz xyz per component; ax, ay, az are the rows of the
// symmetric s.  This is cell_force3 / corner_forces3 with the sums along each
// axis taken apart.
struct Cell3 {
    float s[6];                     // xx yy zz yz xz xy, a quarter of the average stress
    float xy[3], yz[3], zx[3], xyz[3];
};

__device__ __forceinline__ void cell3(float l, float m, const Row3 &a, const Row3 &b, const Row3 &a1, const Row3 &b1,
                                      Cell3 &C)
{
    float gx[3], gy[3], gz[3], hxy[3], hyz[3], hzx[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float sd0 = a.d[k] + b.d[k], dd0 = b.d[k] - a.d[k], se0 = a.e[k] + b.e[k], de0 = b.e[k] - a.e[k];
        const float sd1 = a1.d[k] + b1.d[k], dd1 = b1.d[k] - a1.d[k], se1 = a1.e[k] + b1.e[k], de1 = b1.e[k] - a1.e[k];
        gx[k] = sd0 + sd1;
        gy[k] = de0 + de1;
        gz[k] = se1 - se0;
        hxy[k] = dd0 + dd1;
        hyz[k] = de1 - de0;
        hzx[k] = sd1 - sd0;
        C.xyz[k] = dd1 - dd0;
    }
    const float lt = l * (gx[0] + gy[1] + gz[2]), m2 = m + m;
    C.s[0] = fmaf(m2, gx[0], lt);
    C.s[1] = fmaf(m2, gy[1], lt);
    C.s[2] = fmaf(m2, gz[2], lt);
    C.s[3] = m * (gz[1] + gy[2]);
    C.s[4] = m * (gz[0] + gx[2]);
    C.s[5] = m * (gy[0] + gx[1]);
    const float l3 = l * (1.0f / 3.0f), m3 = m * (1.0f / 3.0f), c9 = (l + 4.0f * m) * (1.0f / 9.0f);
    const float A = l3 * (hxy[1] + hzx[2]), B = l3 * (hxy[0] + hyz[2]), D = l3 * (hzx[0] + hyz[1]);
    const float P = hyz[0] + hzx[1], Q = hzx[1] + hxy[2], R = hxy[2] + hyz[0];
    C.xy[0] = fmaf(m, hxy[0], B);
    C.xy[1] = fmaf(m, hxy[1], A);
    C.xy[2] = m3 * (Q + R);
    C.yz[0] = m3 * (P + R);
    C.yz[1] = fmaf(m, hyz[1], D);
    C.yz[2] = fmaf(m, hyz[2], B);
    C.zx[0] = fmaf(m, hzx[0], D);
    C.zx[1] = m3 * (P + Q);
    C.zx[2] = fmaf(m, hzx[2], A);
#pragma unroll
    for (int k = 0; k < 3; k++) C.xyz[k] *= c9;
}

// the mean strain's part (ue: Voigt mean strain)
__device__ __forceinline__ void cell3_mean(float l, float m, const float *ue, Cell3 &C)
{
    const float lt = 4.0f * l * (ue[0] + ue[1] + ue[2]), m8 = 8.0f * m, m4 = 4.0f * m;
#pragma unroll
    for (int v = 0; v < 3; v++) C.s[v] += fmaf(m8, ue[v], lt);
#pragma unroll
    for (int v = 3; v < 6; v++) C.s[v] = fmaf(m4, ue[v], C.s[v]);
}

// Sums that a node row collects: E - O of its own lane plus E + O of the lane
// on its left.
struct Node3 {
    float E[3], O[3];
};

// what a cell row leaves on its four node rows: lower plane a0 (sy = -1), b0
// (sy = +1), upper plane a1, b1
__device__ __forceinline__ void cell3_rows(const Cell3 &C, Node3 &a0, Node3 &b0, Node3 &a1, Node3 &b1)
{
    constexpr int SX[3] = {0, 5, 4}, SY[3] = {5, 1, 3}, SZ[3] = {4, 3, 2};
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float ax = C.s[SX[k]], ay = C.s[SY[k]], az = C.s[SZ[k]];
        const float y0 = ay - C.yz[k], x0 = ax - C.zx[k], w0 = C.xy[k] - C.xyz[k];
        const float y1 = ay + C.yz[k], x1 = ax + C.zx[k], w1 = C.xy[k] + C.xyz[k];
        a0.E[k] = -az - y0; a0.O[k] = x0 - w0;
        b0.E[k] = y0 - az;  b0.O[k] = x0 + w0;
        a1.E[k] = az - y1;  a1.O[k] = x1 - w1;
        b1.E[k] = az + y1;  b1.O[k] = x1 + w1;
    }
}

__device__ __forceinline__ void add3(Node3 &a, const Node3 &b)
{
#pragma unroll
    for (int k = 0; k < 3; k++) { a.E[k] += b.E[k]; a.O[k] += b.O[k]; }
}

// Output rows per work item (four: 10 % slower at 256^3, spills).
constexpr int M3_ROWS = 2;

// Planes per work item of an nx x ny x nz level for nw warps: the candidate
// with the least (items per warp, rounded up) x (planes + 2).
inline int m3_chunk(int nx, int ny, int nz, int nw)
{
    const long long cols = (long long)(nx <= 32 ? 1 : (nx + 29) / 30) * ((ny + M3_ROWS - 1) / M3_ROWS);
    int best = nz;
    long long bcost = -1;
    for (int zc = 1; zc <= nz; zc++) {
        const long long items = cols * ((nz + zc - 1) / zc);
        const long long cost = ((items + nw - 1) / nw) * (zc + 2);
        if (bcost < 0 || cost < bcost) {
            bcost = cost;
            best = zc;
        }
    }
    return best;
}

// One sweep: op.load(R, r, own, gx, gy, gz, g, gm, Ln) loads the words of node
// g = (gx, gy, gz), row r of the item (0 and
// M3_ROWS + 1: halo rows) (own: an output row), and the
// moduli of the cell gm of the same column in the plane before; op.form(R, r,
// own, gx, gy, gz, g, Ln, v, k, S) gives the operand v of the node (own: an output
// node; k[4] is handed to the epilogue); op.epi(g, q, k, S) receives q = A v
// at every output node.  op.cell(C, S) gets every own cell before the mean
// strain op.ue is added (op.E).  S collects what they sum and is returned.
template <class OP>
__device__ __noinline__ typename OP::Sums m3_sweep(const OP *sop, int nx, int ny, int nz, int zc, int bid, int nbk)
{
    constexpr int MR = M3_ROWS, NR = MR + 2;          // output rows, rows formed
    const OP op = *sop;
    const Lanes2 Ln(nx);
    const int lane = Ln.lane, nw = (int)(blockDim.x >> 5) * nbk;
    typename OP::Sums S;
    const int ns = Ln.per ? 1 : (nx + 29) / 30, nyg = (ny + MR - 1) / MR, items = ns * nyg * ((nz + zc - 1) / zc);
    const int plane = nx * ny;
    for (int item = (int)(threadIdx.x >> 5) * nbk + bid; item < items; item += nw) {
        const int x0 = (item % ns) * 30, y0 = ((item / ns) % nyg) * MR, z0 = (item / (ns * nyg)) * zc, z1 = min(z0 + zc, nz);
        const int gxr = Ln.per ? lane : x0 - 1 + lane, gx = wrapm(gxr, nx);
        const bool ownx = (Ln.per || (lane >= 1 && lane <= 30)) && gxr < nx;
        int gy[NR];
#pragma unroll
        for (int r = 0; r < NR; r++) gy[r] = wrapm(y0 - 1 + r, ny);
        Row3 lo[NR];
        Node3 carry[MR];
        float kp[MR][4];
        typename OP::Raw R;
        int gz = wrapm(z0 - 1, nz), gzm = gz;
        op.load(R, 0, false, gx, gy[0], gz, gx + nx * gy[0] + plane * gz, gx + nx * gy[0] + plane * gzm, Ln);
        for (int z = z0 - 1; z <= z1; z++) {             // the plane that is formed
            const bool zown = z >= z0 && z < z1, cells = z >= z0, nodes = z > z0;
            const int gzn = gz + 1 == nz ? 0 : gz + 1;
            Row3 hp;                                     // row r - 1 of this plane
            Node3 b0, b1;                                // what cell row r - 2 left on node row r - 1
            float kq[4], lp = 0.f, mp = 0.f;             // keep of row r - 1, moduli of cell row r - 1
#pragma unroll
            for (int r = 0; r < NR; r++) {
                const int g = gx + nx * gy[r] + plane * gz;
                const bool own = ownx && zown && r >= 1 && r <= MR && y0 + r - 1 < ny;
                float v[3], k[4];
                op.form(R, r, own, gx, gy[r], gz, g, Ln, v, k, S);
                const float l = R.l * 0.0625f, m = R.m * 0.0625f;
                if (r < NR - 1) {
                    constexpr int last = NR - 1;
                    const int gyn = gy[r < last ? r + 1 : last];
                    op.load(R, r + 1, zown && r < MR, gx, gyn, gz, gx + nx * gyn + plane * gz, gx + nx * gyn + plane * gzm, Ln);
                } else if (z < z1) {
                    op.load(R, 0, false, gx, gy[0], gzn, gx + nx * gy[0] + plane * gzn, gx + nx * gy[0] + plane * gz, Ln);
                }
                Row3 h;
                row3(v, Ln, h);
                if (r >= 1) {
                    if (cells) {
                        Cell3 C;
                        cell3(lp, mp, lo[r - 1], lo[r], hp, h, C);
                        const bool ownc = ownx && nodes && r >= 2 && y0 + r - 2 < ny;   // cell row r - 1 at node row r - 1
                        if constexpr (OP::E) {
                            if (ownc) op.cell(C, S);
                            cell3_mean(lp, mp, op.ue, C);
                        }
                        Node3 a0, c0, a1, c1;
                        cell3_rows(C, a0, c0, a1, c1);
                        if (r >= 2) {
                            // node row r - 1: lower plane complete, upper plane carried on
                            if (nodes) {
                                add3(a0, b0);
                                add3(a0, carry[r - 2]);
                                float q[3];
#pragma unroll
                                for (int c = 0; c < 3; c++)
                                    q[c] = (a0.E[c] - a0.O[c]) + __shfl_sync(0xffffffffu, a0.E[c] + a0.O[c], Ln.prv);
                                if (ownc) op.epi(gx + nx * gy[r - 1] + plane * gzm, q, kp[r - 2], S);
                            }
                            add3(a1, b1);
                            carry[r - 2] = a1;
                        }
                        b0 = c0;
                        b1 = c1;
                    }
                    lo[r - 1] = hp;
                    if (r >= 2)
#pragma unroll
                        for (int c = 0; c < 4; c++) kp[r - 2][c] = kq[c];
                }
                hp = h;
#pragma unroll
                for (int c = 0; c < 4; c++) kq[c] = k[c];
                lp = l;
                mp = m;
            }
            lo[NR - 1] = hp;
            gzm = gz;
            gz = gzn;
        }
    }
    return S;
}

// gamma = r.u, delta = w.u and a quarter of the own cells' stresses
struct Sums3 {
    Acc<float> ru, wu, se[6];
};

// First smoothing step from zero: v = c2 D^-1 f, r1 = f - A v; dir: keep v, the
// direction and iterate of further steps, in d1.
struct OpSmooth3 {
    static constexpr bool E = false;
    typedef Acc<float> Sums;
    const float *lam, *mu, *dinv, *f;
    float *r1, *d1;
    float c2;
    unsigned n;                 // distance of a vector's components
    bool dir;
    struct Raw {
        float l, m, di, f[3];
    };
    __device__ __forceinline__ void load(Raw &R, int, bool, int, int, int, int g, int gm, const Lanes2 &) const
    {
        R.l = __ldcg(lam + gm);
        R.m = __ldcg(mu + gm);
        R.di = __ldcg(dinv + g);
#pragma unroll
        for (int c = 0; c < 3; c++) R.f[c] = __ldcg(f + ((unsigned)g + c * n));
    }
    __device__ __forceinline__ void form(const Raw &R, int, bool own, int, int, int, int g, const Lanes2 &, float (&v)[3],
                                         float (&k)[4], Sums &) const
    {
        const float di = c2 * R.di;
        k[3] = 0.f;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            v[c] = di * R.f[c];
            k[c] = R.f[c];
            if (own && dir) d1[(unsigned)g + c * n] = v[c];
        }
    }
    __device__ __forceinline__ void epi(int g, const float (&q)[3], const float (&k)[4], Sums &) const
    {
#pragma unroll
        for (int c = 0; c < 3; c++) r1[(unsigned)g + c * n] = k[c] - q[c];
    }
};

// Chebyshev step (as OpCheb2): x += d, r' = r - A d with d = c1 d + c2 D^-1 r;
// last: the next step as well, into xo.
struct OpCheb3 {
    static constexpr bool E = false;
    typedef Acc<float> Sums;
    const float *lam, *mu, *dinv, *r, *d, *xi;
    float *xo, *rn, *dn;
    float c1, c2, n1, n2;
    unsigned n;
    bool last, dir;             // dir: the step has a previous direction d
    struct Raw {
        float l, m, di, r[3], d[3], x[3];
    };
    __device__ __forceinline__ void load(Raw &R, int, bool own, int, int, int, int g, int gm, const Lanes2 &) const
    {
        R.l = __ldcg(lam + gm);
        R.m = __ldcg(mu + gm);
        R.di = __ldcg(dinv + g);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const unsigned o = (unsigned)g + c * n;
            R.r[c] = __ldcg(r + o);
            R.d[c] = dir ? __ldcg(d + o) : 0.f;
            if (own) R.x[c] = __ldcg(xi + o);
        }
    }
    __device__ __forceinline__ void form(const Raw &R, int, bool own, int, int, int, int g, const Lanes2 &, float (&v)[3],
                                         float (&k)[4], Sums &) const
    {
        const float di = c2 * R.di, dl = n2 * R.di;
        k[3] = dl;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const unsigned o = (unsigned)g + c * n;
            v[c] = di * R.r[c] + c1 * R.d[c];
            k[c] = R.r[c];
            if (own) {
                const float xn = R.x[c] + v[c];
                if (last) {
                    k[c] = xn + n1 * v[c] + dl * R.r[c];
                } else {
                    xo[o] = xn;
                    dn[o] = v[c];
                }
            }
        }
    }
    __device__ __forceinline__ void epi(int g, const float (&q)[3], const float (&k)[4], Sums &) const
    {
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const unsigned o = (unsigned)g + c * n;
            if (last) xo[o] = k[c] - k[3] * q[c];
            else rn[o] = k[c] - q[c];
        }
    }
};

// First post-smoothing step: x = x_pre + P e (trilinear), r = f - A x; last
// (one-step smoothing): x + c2 D^-1 r, the level's final correction, into
// xpost, else x and r.  With last, x_pre is one step from zero, c2 D^-1 f, and
// is formed again instead of being stored and read.  Coarse rows are loaded as the fine rows reach them
// (an item starts at an even row): row r even lies between two coarse rows,
// row r odd on one.
struct OpPost3 {
    static constexpr bool E = false;
    typedef Acc<float> Sums;
    const float *lam, *mu, *dinv, *f, *xpre, *xc;
    float *xpost, *rn;
    int cnx, cny, cnz;
    unsigned cn;
    float c2;
    unsigned n;
    bool last;
    struct Raw {
        float l, m, di, f[3], x[3], c0[3], c1[3], d0[3], d1[3];   // c: next coarse row (two planes), d: the first one's
        float cur[3];                                             // the current coarse row, interpolated in x and z
    };
    __device__ __forceinline__ void coarse(int gx, int cy, int gz, float (&a)[3], float (&b)[3]) const
    {
        const int iz = gz >> 1, iz1 = (gz & 1) ? (iz + 1 == cnz ? 0 : iz + 1) : iz;
        const unsigned o0 = (unsigned)((gx >> 1) + cnx * (cy + cny * iz)), o1 = (unsigned)((gx >> 1) + cnx * (cy + cny * iz1));
#pragma unroll
        for (int c = 0; c < 3; c++) {
            a[c] = __ldca(xc + o0 + c * cn);
            b[c] = __ldca(xc + o1 + c * cn);
        }
    }
    __device__ __forceinline__ void load(Raw &R, int r, bool own, int gx, int gy, int gz, int g, int gm, const Lanes2 &) const
    {
        R.l = __ldcg(lam + gm);
        R.m = __ldcg(mu + gm);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const unsigned o = (unsigned)g + c * n;
            if (!last) R.x[c] = __ldcg(xpre + o);
            if (own || last) R.f[c] = __ldcg(f + o);
        }
        if (last) R.di = __ldcg(dinv + g);
        if ((r & 1) == 0) {
            const int iy = gy >> 1;
            if (r == 0) coarse(gx, iy, gz, R.d0, R.d1);
            coarse(gx, iy + 1 == cny ? 0 : iy + 1, gz, R.c0, R.c1);
        }
    }
    __device__ __forceinline__ void interp(const float (&a)[3], const float (&b)[3], int gx, const Lanes2 &Ln, float (&t)[3]) const
    {
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float e = 0.5f * (a[c] + b[c]), o = __shfl_sync(0xffffffffu, e, Ln.nxt);
            t[c] = (gx & 1) ? 0.5f * (e + o) : e;
        }
    }
    __device__ __forceinline__ void form(Raw &R, int r, bool own, int gx, int, int, int g, const Lanes2 &Ln, float (&v)[3],
                                         float (&k)[4], Sums &) const
    {
        k[3] = c2 * R.di;
        if (last)
#pragma unroll
            for (int c = 0; c < 3; c++) R.x[c] = k[3] * R.f[c];
        if ((r & 1) == 0) {
            float nx_[3];
            if (r == 0) interp(R.d0, R.d1, gx, Ln, R.cur);
            interp(R.c0, R.c1, gx, Ln, nx_);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                v[c] = R.x[c] + 0.5f * (R.cur[c] + nx_[c]);
                R.cur[c] = nx_[c];
            }
        } else {
#pragma unroll
            for (int c = 0; c < 3; c++) v[c] = R.x[c] + R.cur[c];
        }
#pragma unroll
        for (int c = 0; c < 3; c++) {
            k[c] = last ? v[c] + k[3] * R.f[c] : R.f[c];
            if (own && !last) xpost[(unsigned)g + c * n] = v[c];
        }
    }
    __device__ __forceinline__ void epi(int g, const float (&q)[3], const float (&k)[4], Sums &) const
    {
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const unsigned o = (unsigned)g + c * n;
            if (last) xpost[o] = k[c] - k[3] * q[c];
            else rn[o] = k[c] - q[c];
        }
    }
};

// w = A u with the mean strain, gamma = r.u, delta = w.u and the own cells'
// stresses.
struct OpApply3 {
    static constexpr bool E = true;
    typedef Sums3 Sums;
    const float *lam, *mu, *u, *r;
    float *w;
    float ue[6];
    unsigned n;
    struct Raw {
        float l, m, u[3], r[3];
    };
    __device__ __forceinline__ void load(Raw &R, int, bool own, int, int, int, int g, int gm, const Lanes2 &) const
    {
        R.l = __ldcg(lam + gm);
        R.m = __ldcg(mu + gm);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const unsigned o = (unsigned)g + c * n;
            R.u[c] = __ldcg(u + o);
            if (own) R.r[c] = __ldcg(r + o);
        }
    }
    __device__ __forceinline__ void form(const Raw &R, int, bool own, int, int, int, int, const Lanes2 &, float (&v)[3],
                                         float (&k)[4], Sums &S) const
    {
        k[3] = 0.f;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            v[c] = R.u[c];
            k[c] = v[c];
            if (own) S.ru.fma_plain(R.r[c], v[c]);
        }
    }
    __device__ __forceinline__ void cell(const Cell3 &C, Sums &S) const
    {
#pragma unroll
        for (int v = 0; v < 6; v++) S.se[v].add_plain(C.s[v]);
    }
    __device__ __forceinline__ void epi(int g, const float (&q)[3], const float (&k)[4], Sums &S) const
    {
#pragma unroll
        for (int c = 0; c < 3; c++) {
            w[(unsigned)g + c * n] = q[c];
            S.wu.fma_plain(q[c], k[c]);
        }
    }
};

// Jacobi-preconditioned CG: u = D^-1 r, w = A u with the mean strain, and the
// sums of OpApply3 with ||r||^2.
struct SumsJ3 : Sums3 {
    Acc<float> rr;
};
struct OpJac3 {
    static constexpr bool E = true;
    typedef SumsJ3 Sums;
    const float *lam, *mu, *dinv, *r;
    float *w;
    float ue[6];
    unsigned n;
    struct Raw {
        float l, m, di, r[3];
    };
    __device__ __forceinline__ void load(Raw &R, int, bool, int, int, int, int g, int gm, const Lanes2 &) const
    {
        R.l = __ldcg(lam + gm);
        R.m = __ldcg(mu + gm);
        R.di = __ldcg(dinv + g);
#pragma unroll
        for (int c = 0; c < 3; c++) R.r[c] = __ldcg(r + ((unsigned)g + c * n));
    }
    __device__ __forceinline__ void form(const Raw &R, int, bool own, int, int, int, int, const Lanes2 &, float (&v)[3],
                                         float (&k)[4], Sums &S) const
    {
        k[3] = 0.f;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            v[c] = R.di * R.r[c];
            k[c] = v[c];
            if (own) {
                S.ru.fma_plain(R.r[c], v[c]);
                S.rr.fma_plain(R.r[c], R.r[c]);
            }
        }
    }
    __device__ __forceinline__ void cell(const Cell3 &C, Sums &S) const
    {
#pragma unroll
        for (int v = 0; v < 6; v++) S.se[v].add_plain(C.s[v]);
    }
    __device__ __forceinline__ void epi(int g, const float (&q)[3], const float (&k)[4], Sums &S) const
    {
#pragma unroll
        for (int c = 0; c < 3; c++) {
            w[(unsigned)g + c * n] = q[c];
            S.wu.fma_plain(q[c], k[c]);
        }
    }
};

}  // namespace pfdev
