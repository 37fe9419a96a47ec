// Geometric multigrid preconditioner of the 2D solve (K3/K4): u = M r is one
// V-cycle over a hierarchy of periodic Q1 grids, each coarse level with half
// the nodes per axis and the 2x2 average of its fine cells' moduli (the
// operator rediscretised, not the Galerkin product).  Smoothing is a
// Chebyshev iteration on D^-1 A over [b/30, b], where b is a bound on the
// largest eigenvalue of D^-1 A that holds for any cell moduli (the largest
// eigenvalue of diag(K_e)^-1 K_e of one element, set by the Poisson ratio);
// restriction is the transpose of bilinear prolongation.  With the same
// polynomial before and after the coarse correction and a polynomial coarse
// solve, the V-cycle is a fixed symmetric positive-definite operator, so it
// serves as a CG preconditioner.  The mean-strain dofs keep their Jacobi
// scaling (block-diagonal preconditioner).
//
// Levels beyond the block-run ones: a smoothing is one warp-marching sweep of
// the Q1 operator (pf_march2.cuh) and one grid barrier.  Operands that are
// pointwise in stored vectors are formed as the sweep reaches their row (the
// restricted residual, the prolonged correction, the CG update), two steps
// run in one sweep, and the last step of a smoothing, which needs no operator
// product, is applied in the epilogue of the step before it.  The coarse
// levels are run by the job's first block in its shared memory (whole levels,
// one pass per phase, block barriers).
#pragma once

namespace pfdev {

constexpr int MG_MAX_STEPS = 16;

template <typename T>
struct MGLevel {
    int nx, ny, nz;                // nodes (= cells) per axis, periodic (nz = 1 in 2D)
    T *lam, *mu;                   // cell moduli (level 0: the solve's own, read only)
    T *dinv;                       // inverse Jacobi diagonal (level 0: the solve's own)
    T *f[3];                       // right-hand side (levels >= 1; level 0 uses the CG residual)
    T *xpre[3];                    // iterate of the pre-smoothing (coarsest: of its solve)
    T *xpost[3];                   // iterate of the post-smoothing; the level's final correction
                                   // when it is done (finest level: u = M r)
    T *r[2][3], *d[2][3];          // [buffer][component]: residual, Chebyshev direction
};

template <typename T>
struct MGHier {
    int L;                         // levels
    int Lg;                        // levels [0, Lg) run on the whole grid, [Lg, L) by the job's first
                                   // block in shared memory (mg_block_words)
    int deg[MG_MAX_LEVELS];        // Chebyshev steps of each pre- and post-smoothing, per level
    int csteps;                    // Chebyshev steps of the coarsest solve (>= 2)
    T c1[MG_MAX_STEPS], c2[MG_MAX_STEPS];   // d_j = c1[j] d_{j-1} + c2[j] D^-1 r_j  (c1[0] = 0)
    T *dense;                      // 2D FP64: the block-run levels' map, (2 nodes)^2 values
    MGLevel<T> lv[MG_MAX_LEVELS];
};

__device__ __forceinline__ int mg_wrap(int a, int n, bool small) { return small ? wrapm(a, n) : wrap(a, n); }

// Shared memory of the block-run levels [Lg, L), in words of T: per level 11
// arrays of its node count (x, r, d, f by component, then the inverse
// diagonal and the cell moduli), then the scratch of the largest level: the
// operand (2 per node) and the cell forces (5 per cell).  The first
// block-run level has at most NB nodes and each next a quarter of the one
// before, so mg_block_words_cap(NB) bounds the total.
constexpr int MG_BLK_ARRAYS = 11, MG_BLK_SCRATCH = 7;

// node count up to which a level is run by one block: the shared arrays of
// such levels fit next to two resident 256-thread PCG blocks per SM
template <typename T>
__host__ __device__ constexpr long long mg_block_nodes() { return sizeof(T) == 4 ? 1024 : 256; }

template <typename T>
__host__ __device__ inline long long mg_block_words(const MGHier<T> &H)
{
    long long w = 0, nmax = 0;
    for (int k = H.Lg; k < H.L; k++) {
        const long long n = (long long)H.lv[k].nx * H.lv[k].ny;
        w += MG_BLK_ARRAYS * n;
        nmax = n > nmax ? n : nmax;
    }
    return nmax ? w + MG_BLK_SCRATCH * nmax : 0;
}

__host__ __device__ constexpr long long mg_block_words_cap(long long nb)
{
    return MG_BLK_ARRAYS * (nb * 4 / 3 + 1) + MG_BLK_SCRATCH * nb;
}

// A block-run level's arrays in shared memory.
template <typename T>
struct BLevel {
    int nx, ny, n;
    T *x[2], *r[2], *d[2], *f[2], *dinv, *lam, *mu;
};

template <typename T>
__device__ __forceinline__ BLevel<T> blevel(T *base, const MGHier<T> &H, int k)
{
    long long off = 0;
    for (int m = H.Lg; m < k; m++) off += MG_BLK_ARRAYS * (long long)H.lv[m].nx * H.lv[m].ny;
    BLevel<T> B;
    B.nx = H.lv[k].nx;
    B.ny = H.lv[k].ny;
    B.n = B.nx * B.ny;
    T *p = base + off;
    const int n = B.n;
    B.x[0] = p; B.x[1] = p + n; B.r[0] = p + 2 * n; B.r[1] = p + 3 * n; B.d[0] = p + 4 * n; B.d[1] = p + 5 * n;
    B.f[0] = p + 6 * n; B.f[1] = p + 7 * n; B.dinv = p + 8 * n; B.lam = p + 9 * n; B.mu = p + 10 * n;
    return B;
}

// the scratch after the block-run levels
template <typename T>
__device__ __forceinline__ T *bscratch(T *base, const MGHier<T> &H)
{
    long long off = 0;
    for (int m = H.Lg; m < H.L; m++) off += MG_BLK_ARRAYS * (long long)H.lv[m].nx * H.lv[m].ny;
    return base + off;
}

// One sweep of a block-run level, whole level at once: val(i, v) for every
// node (called once per node, so it may store), then the cell forces, then
// epi(i, v, q) with q = A v at every node; block barriers between phases.
template <typename T, class Val, class Epi>
__device__ __forceinline__ void blk_sweep(const BLevel<T> &B, T *scr, int nmax, Val &&val, Epi &&epi)
{
    const int n = B.n, nx = B.nx, ny = B.ny;
    T *v0 = scr, *v1 = scr + nmax, *cf = scr + 2 * nmax;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        T v[2];
        val(i, v);
        v0[i] = v[0];
        v1[i] = v[1];
    }
    __syncthreads();
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        const int cx = c % nx, cy = c / nx;
        const int cx1 = cx + 1 == nx ? 0 : cx + 1, cy1 = cy + 1 == ny ? 0 : cy + 1;
        const int nd[4] = {c, cx1 + nx * cy, cx + nx * cy1, cx1 + nx * cy1};
        T uc[4][2];
#pragma unroll
        for (int b = 0; b < 4; b++) {
            uc[b][0] = v0[nd[b]];
            uc[b][1] = v1[nd[b]];
        }
        T s3[3], fh[2];
        cell_force2<T>(B.lam[c], B.mu[c], uc, s3, fh);
        cf[c] = s3[0];
        cf[nmax + c] = s3[1];
        cf[2 * nmax + c] = s3[2];
        cf[3 * nmax + c] = fh[0];
        cf[4 * nmax + c] = fh[1];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int ix = i % nx, iy = i / nx;
        T q[2] = {T(0), T(0)};
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const int ex = (a & 1) ? (ix == 0 ? nx - 1 : ix - 1) : ix;
            const int ey = (a >> 1) ? (iy == 0 ? ny - 1 : iy - 1) : iy;
            const int c = ex + nx * ey;
            const T s3[3] = {cf[c], cf[nmax + c], cf[2 * nmax + c]};
            const T fh[2] = {cf[3 * nmax + c], cf[4 * nmax + c]};
            T f[2];
            node_force2<T>(a, s3, fh, f);
            q[0] += f[0];
            q[1] += f[1];
        }
        const T v[2] = {v0[i], v1[i]};
        epi(i, v, q);
    }
    __syncthreads();
}

// Coarse level C from fine level F (both in global memory): cell moduli =
// mean of the 2x2 fine cells, Jacobi diagonal from the four coarse cells
// around each node.  Threads t0, t0 + st, ... take the coarse nodes.
template <typename T>
__device__ void mg_coarsen(const MGLevel<T> &F, const MGLevel<T> &C, long long t0, long long st)
{
    const int n = C.nx * C.ny;
    auto avg = [&](const T *a, int cx, int cy) {
        const int i = 2 * cx + F.nx * (2 * cy);
        return T(0.25) * ((__ldcg(a + i) + __ldcg(a + i + 1)) + (__ldcg(a + i + F.nx) + __ldcg(a + i + F.nx + 1)));
    };
    for (long long i = t0; i < n; i += st) {
        const int cx = (int)(i % C.nx), cy = (int)(i / C.nx);
        C.lam[i] = avg(F.lam, cx, cy);
        C.mu[i] = avg(F.mu, cx, cy);
        T dg = T(0);
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const int ex = wrap(cx - (a & 1), C.nx), ey = wrap(cy - (a >> 1), C.ny);
            dg += avg(F.lam, ex, ey) * KdL<T, 2>() + avg(F.mu, ex, ey) * KdM<T, 2>();
        }
        C.dinv[i] = T(1) / dg;
    }
}

// The same into a block-run level's shared arrays, from a grid level
// (global, fl / fm / fnx) or the block-run level above (shared).
template <typename T>
__device__ void mg_coarsen_blk(const T *fl, const T *fm, int fnx, bool global, const BLevel<T> &C)
{
    for (int i = threadIdx.x; i < C.n; i += blockDim.x) {
        const int cx = i % C.nx, cy = i / C.nx, f = 2 * cx + fnx * (2 * cy);
        auto ld = [&](const T *a, int o) { return global ? __ldcg(a + o) : a[o]; };
        C.lam[i] = T(0.25) * ((ld(fl, f) + ld(fl, f + 1)) + (ld(fl, f + fnx) + ld(fl, f + fnx + 1)));
        C.mu[i] = T(0.25) * ((ld(fm, f) + ld(fm, f + 1)) + (ld(fm, f + fnx) + ld(fm, f + fnx + 1)));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < C.n; i += blockDim.x) {
        const int cx = i % C.nx, cy = i / C.nx;
        T dg = T(0);
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const int c = wrap(cx - (a & 1), C.nx) + C.nx * wrap(cy - (a >> 1), C.ny);
            dg += C.lam[c] * KdL<T, 2>() + C.mu[c] * KdM<T, 2>();
        }
        C.dinv[i] = T(1) / dg;
    }
    __syncthreads();
}

// Hierarchy set-up at the start of a solve (the cell moduli are written anew
// every step; they follow phi_g, which is held fixed, to rounding): the grid
// levels below Lg, with a barrier after each.  Returns false
// if a barrier timed out.
template <typename T>
__device__ bool mg_setup(const MGHier<T> &H, unsigned int *bc, unsigned int *bg, int *err, int bid, int nbk)
{
    const int Lgw = H.Lg < H.L ? H.Lg : H.L;
    const long long t0 = bid * (long long)blockDim.x + threadIdx.x, st = (long long)nbk * blockDim.x;
    for (int k = 1; k < Lgw; k++) {
        mg_coarsen<T>(H.lv[k - 1], H.lv[k], t0, st);
        if (!grid_sync(bc, bg, err, nbk)) return false;
    }
    return true;
}

// The shared arrays of the block-run levels, filled by the job's first
// block at the start of every CG pass (the residual sweep before it uses
// the same shared memory as scratch).
template <typename T>
__device__ void mg_setup_block(const MGHier<T> &H, T *sblk)
{
    const int Lgw = H.Lg < H.L ? H.Lg : H.L;
    for (int k = Lgw; k < H.L; k++) {
            const BLevel<T> C = blevel<T>(sblk, H, k);
            if (k == Lgw) {
                mg_coarsen_blk<T>(H.lv[k - 1].lam, H.lv[k - 1].mu, H.lv[k - 1].nx, true, C);
            } else {
                const BLevel<T> F = blevel<T>(sblk, H, k - 1);
                mg_coarsen_blk<T>(F.lam, F.mu, F.nx, false, C);
            }
    }
}

// Double-float arithmetic: a value is an unevaluated sum hi + lo of two
// FP32 numbers (~48 significant bits).  Sums use Knuth's TwoSum, products
// the FMA form of TwoProduct; results are renormalised with the fast
// two-sum (|a| >= |b|).  The mixed method's refinement residual b - A x is
// formed this way: FP64 runs at a small fraction of the FP32 rate here.
struct DF {
    float hi, lo;
};
__device__ __forceinline__ DF df_quick(float a, float b)
{
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ DF df_two_sum(float a, float b)
{
    const float s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ DF df_from(double x)
{
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ double df_val(DF a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ DF df_add(DF a, DF b)
{
    const DF s = df_two_sum(a.hi, b.hi), t = df_two_sum(a.lo, b.lo);
    const DF u = df_quick(s.hi, s.lo + t.hi);
    return df_quick(u.hi, u.lo + t.lo);
}
__device__ __forceinline__ DF df_neg(DF a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ DF df_sub(DF a, DF b) { return df_add(a, df_neg(b)); }
// exact scaling by a power of two
__device__ __forceinline__ DF df_scale(DF a, float p2) { return {a.hi * p2, a.lo * p2}; }
__device__ __forceinline__ DF df_mul_f(DF a, float b)
{
    const float p = a.hi * b;
    const float e = fmaf(a.hi, b, -p);
    return df_quick(p, fmaf(a.lo, b, e));
}
__device__ __forceinline__ DF df_mul(DF a, DF b)
{
    const float p = a.hi * b.hi;
    const float e = fmaf(a.hi, b.hi, -p);
    return df_quick(p, e + fmaf(a.hi, b.lo, a.lo * b.hi));
}

// plane-strain stress of a Voigt strain e (engineering shear) in
// double-float: l tr e + 2 m e on the normals, m e on the shear
__device__ __forceinline__ void voigt2_df(float l, float m, const DF (&e)[3], DF (&s)[3])
{
    const float m2 = 2.0f * m;                 // exact
    const DF tr = df_add(e[0], e[1]);
    s[0] = df_add(df_mul_f(tr, l), df_mul_f(e[0], m2));
    s[1] = df_add(df_mul_f(tr, l), df_mul_f(e[1], m2));
    s[2] = df_mul_f(e[2], m);
}

// cell_force2 in double-float: average stress of the cell's displacement
// plus the mean-strain stress, hourglass forces (l, m: the FP32 moduli)
__device__ __forceinline__ void cell_force2_df(float l, float m, const DF (&ue)[4][2], const DF (&xe)[3], DF (&s)[3],
                                               DF (&fh)[2], DF (&s_own)[3])
{
    const DF Gxu = df_scale(df_add(df_sub(ue[1][0], ue[0][0]), df_sub(ue[3][0], ue[2][0])), 0.5f);
    const DF Gyu = df_scale(df_add(df_sub(ue[2][0], ue[0][0]), df_sub(ue[3][0], ue[1][0])), 0.5f);
    const DF Gxv = df_scale(df_add(df_sub(ue[1][1], ue[0][1]), df_sub(ue[3][1], ue[2][1])), 0.5f);
    const DF Gyv = df_scale(df_add(df_sub(ue[2][1], ue[0][1]), df_sub(ue[3][1], ue[1][1])), 0.5f);
    const DF hu = df_sub(df_sub(ue[0][0], ue[1][0]), df_sub(ue[2][0], ue[3][0]));
    const DF hv = df_sub(df_sub(ue[0][1], ue[1][1]), df_sub(ue[2][1], ue[3][1]));
    const DF G[3] = {Gxu, Gyv, df_add(Gyu, Gxv)};   // Voigt strain, engineering shear
    voigt2_df(l, m, G, s_own);
    DF sx[3];
    voigt2_df(l, m, xe, sx);
#pragma unroll
    for (int v = 0; v < 3; v++) s[v] = df_add(s_own[v], sx[v]);
    // (l + 3 m) / 12, with l + 3 m exact as a double-float
    const float p3 = 3.0f * m;
    const DF l3m = df_add(DF{l, 0.0f}, DF{p3, fmaf(3.0f, m, -p3)});
    const DF c = df_mul(l3m, df_from(1.0 / 12.0));
    fh[0] = df_mul(c, hu);
    fh[1] = df_mul(c, hv);
}

// node_force2 in double-float
__device__ __forceinline__ void node_force2_df(int a, const DF (&s)[3], const DF (&fh)[2], DF (&f)[2])
{
    const float bx = (a & 1) ? 0.5f : -0.5f, by = (a >> 1) ? 0.5f : -0.5f;
    const bool gp = (a == 0 || a == 3);
    const DF g0 = gp ? fh[0] : df_neg(fh[0]), g1 = gp ? fh[1] : df_neg(fh[1]);
    f[0] = df_add(df_add(df_scale(s[0], bx), df_scale(s[2], by)), g0);
    f[1] = df_add(df_add(df_scale(s[1], by), df_scale(s[2], bx)), g1);
}

// Shared memory (in doubles) of setup_tiled for a TX x TY tile: the FP64
// operand on the tile halo and five values per halo cell.
template <int TX, int TY>
__host__ __device__ constexpr int setup_tiled_doubles() { return 2 * (TX + 2) * (TY + 2) + 5 * (TX + 1) * (TY + 1); }

// Byte offset of the sweeps' operation record in the dynamic shared
// memory: after the block-run levels' arrays and the set-up sweep's scratch
// (which share the start), rounded to 16 bytes.  The total is pcg_dyn_smem.
template <typename T, int TX, int TY>
__host__ __device__ constexpr size_t mg_march_offset()
{
    const size_t blk = sizeof(T) * (size_t)mg_block_words_cap(mg_block_nodes<T>());
    const size_t stp = sizeof(double) * (size_t)setup_tiled_doubles<TX, TY>();
    return ((blk > stp ? blk : stp) + 15) / 16 * 16;
}

// The set-up sweep of one CG pass, 2D, over node tiles: right-hand side
// b = sum_e Bbar^T sig*, Jacobi diagonal, r = b - A x (x: the FP64 solution
// in refinement mode, else the displacement; mean strain xe) with the
// operator applied in FP64 from per-cell average stress and hourglass forces
// computed once per tile (dscr: setup_tiled_doubles<TX, TY>() doubles of
// shared memory), and the per-node sums of the mean-strain rows: acc[0]
// ||b||^2, [1] ||r||^2, [2] sum lam, [3] sum mu, [4..6] sum sig*, [10..12]
// sum of the own cells' stress of x without the mean strain; in the mixed
// method the operator part is evaluated in double-float.  Also clears
// p, s and (when x is not used or in refinement mode) the iterate.  In
// refinement mode the first pass keeps b in A.b64; a residual-only pass
// (resid) reads it there and skips everything that does not change during
// a solve (b, the diagonal, sums [0] and [2, 10)).
template <typename T, int TX, int TY>
__device__ void setup_tiled(const PCGArgs<T, 2> &A, bool use_x, bool refine, bool resid, const double *xe,
                            double *dscr, Acc<double> (&acc)[16], int bid, int nbk)
{
    const Params &P = A.P;
    constexpr int HX = TX + 2, HY = TY + 2, CX = TX + 1, CY = TY + 1, HN = HX * HY, HC = CX * CY, NT = TX * TY;
    double *hu = dscr, *hc = dscr + 2 * HN;
    const int nx = P.nx, ny = P.ny;
    const int ntx = (nx + TX - 1) / TX, nty = (ny + TY - 1) / TY, ntiles = ntx * nty;
    const bool small = nx < HX || ny < HY;
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
    // the mixed method's refinement residual: double-float instead of FP64
    const bool dfp = refine && sizeof(T) == 4;
    DF *du = reinterpret_cast<DF *>(dscr), *dc = du + 2 * HN;      // same bytes as hu, hc
    const DF xed[3] = {df_from(xe[0]), df_from(xe[1]), df_from(xe[2])};
    for (int tile = bid; tile < ntiles; tile += nbk) {
        const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
        if (use_x && dfp) {
            for (int h = threadIdx.x; h < HN; h += NT) {
                const int g = mg_wrap(x0 - 1 + h % HX, nx, small) + nx * mg_wrap(y0 - 1 + h / HX, ny, small);
                du[h] = df_from(__ldcg(A.x64[0] + g));
                du[HN + h] = df_from(__ldcg(A.x64[1] + g));
            }
            __syncthreads();
            for (int h = threadIdx.x; h < HC; h += NT) {
                const int cx = h % CX, cy = h / CX;
                const int g = mg_wrap(x0 - 1 + cx, nx, small) + nx * mg_wrap(y0 - 1 + cy, ny, small);
                DF uc[4][2];
#pragma unroll
                for (int b = 0; b < 4; b++) {
                    const int hn = (cx + (b & 1)) + HX * (cy + (b >> 1));
                    uc[b][0] = du[hn];
                    uc[b][1] = du[HN + hn];
                }
                DF s3[3], fh[2], own[3];
                cell_force2_df((float)A.lam[g], (float)A.mu[g], uc, xed, s3, fh, own);
                dc[h] = s3[0];
                dc[HC + h] = s3[1];
                dc[2 * HC + h] = s3[2];
                dc[3 * HC + h] = fh[0];
                dc[4 * HC + h] = fh[1];
            }
            __syncthreads();
        } else if (use_x) {
            for (int h = threadIdx.x; h < HN; h += NT) {
                const int g = mg_wrap(x0 - 1 + h % HX, nx, small) + nx * mg_wrap(y0 - 1 + h / HX, ny, small);
                hu[h] = refine ? __ldcg(A.x64[0] + g) : (double)A.x[0][g];
                hu[HN + h] = refine ? __ldcg(A.x64[1] + g) : (double)A.x[1][g];
            }
            __syncthreads();
            for (int h = threadIdx.x; h < HC; h += NT) {
                const int cx = h % CX, cy = h / CX;
                const int g = mg_wrap(x0 - 1 + cx, nx, small) + nx * mg_wrap(y0 - 1 + cy, ny, small);
                double uc[4][2];
#pragma unroll
                for (int b = 0; b < 4; b++) {
                    const int hn = (cx + (b & 1)) + HX * (cy + (b >> 1));
                    uc[b][0] = hu[hn];
                    uc[b][1] = hu[HN + hn];
                }
                const double l = (double)A.lam[g], m = (double)A.mu[g];
                double s3[3], fh[2], sx[3];
                cell_force2<double>(l, m, uc, s3, fh);
                voigt_stress<double, 2>(l, m, xe, sx);
                hc[h] = s3[0] + sx[0];
                hc[HC + h] = s3[1] + sx[1];
                hc[2 * HC + h] = s3[2] + sx[2];
                hc[3 * HC + h] = fh[0];
                hc[4 * HC + h] = fh[1];
            }
            __syncthreads();
        }
        const int gx = x0 + tx, gy = y0 + ty;
        if (gx < nx && gy < ny) {
            const int n = gx + nx * gy, lx = tx + 1, ly = ty + 1;
            double b[2], ax[2] = {0.0, 0.0}, dgn = 1.0, so[3], deo[3] = {0.0, 0.0, 0.0}, lo, mo, unused[2], unused3[3];
            if (resid) {
                b[0] = __ldcg(A.b64[0] + n);
                b[1] = __ldcg(A.b64[1] + n);
                lo = (double)A.lam[n];
                mo = (double)A.mu[n];
            } else {
                node_setup<T, double, double, 2>(P, n, A.lam, A.mu, A.sig, A.x64, xe, false, b, unused, dgn, so, unused3,
                                                 lo, mo);
                if (refine) {
                    A.b64[0][n] = b[0];
                    A.b64[1][n] = b[1];
                }
            }
            double rv2[2] = {b[0], b[1]};
            if (use_x && dfp) {
                DF axd[2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll
                for (int a = 0; a < 4; a++) {
                    const int cl = (lx - (a & 1)) + CX * (ly - (a >> 1));
                    const DF s3[3] = {dc[cl], dc[HC + cl], dc[2 * HC + cl]};
                    const DF fh[2] = {dc[3 * HC + cl], dc[4 * HC + cl]};
                    DF f[2];
                    node_force2_df(a, s3, fh, f);
                    axd[0] = df_add(axd[0], f[0]);
                    axd[1] = df_add(axd[1], f[1]);
                }
#pragma unroll
                for (int d = 0; d < 2; d++) rv2[d] = df_val(df_sub(df_from(b[d]), axd[d]));
                // the own cell's stress of x without the mean strain
                const int c0 = lx + CX * ly;
                DF sx[3];
                voigt2_df((float)lo, (float)mo, xed, sx);
#pragma unroll
                for (int v = 0; v < 3; v++) deo[v] = df_val(df_sub(dc[v * HC + c0], sx[v]));
            } else if (use_x) {
#pragma unroll
                for (int a = 0; a < 4; a++) {
                    const int cl = (lx - (a & 1)) + CX * (ly - (a >> 1));
                    const double s3[3] = {hc[cl], hc[HC + cl], hc[2 * HC + cl]};
                    const double fh[2] = {hc[3 * HC + cl], hc[4 * HC + cl]};
                    double f[2];
                    node_force2<double>(a, s3, fh, f);
                    ax[0] += f[0];
                    ax[1] += f[1];
                }
                // the own cell's stress of x without the mean strain
                const int c0 = lx + CX * ly;
                double sx[3];
                voigt_stress<double, 2>(lo, mo, xe, sx);
                deo[0] = hc[c0] - sx[0];
                deo[1] = hc[HC + c0] - sx[1];
                deo[2] = hc[2 * HC + c0] - sx[2];
                rv2[0] = b[0] - ax[0];
                rv2[1] = b[1] - ax[1];
            }
            if (!resid) {
                A.dinv[n] = (T)(1.0 / dgn);
                acc[2].add(lo);
                acc[3].add(mo);
#pragma unroll
                for (int v = 0; v < 3; v++) acc[4 + v].add(so[v]);
            }
#pragma unroll
            for (int v = 0; v < 3; v++) acc[10 + v].add(deo[v]);
#pragma unroll
            for (int d = 0; d < 2; d++) {
                const double rv = rv2[d];
                if (refine && !use_x) A.x64[d][n] = 0.0;
                if (refine || !use_x) A.x[d][n] = T(0);
                A.p[d][n] = T(0);
                A.s[0][d][n] = T(0);
                A.r[0][d][n] = (T)rv;
                if (!resid) acc[0].addprod(b[d], b[d]);
                acc[1].addprod(rv, rv);
            }
        }
        __syncthreads();
    }
}

// One pass of MG-preconditioned CG (the Chronopoulos-Gear form of the
// Jacobi solve, with u = M r a V-cycle).  Per iteration i:
//   V-cycle on r_i, its first sweep also doing the update of iteration i-1
//   (p, s, x, r) and reducing ||r_i||^2 for the stopping test;
//   u_i = the V-cycle's result, w_i = A u_i, gamma_i = r_i.u_i, delta_i =
//   w_i.u_i and the mean-strain row in one sweep (FP32: with the finest
//   level's post-smoothing) and one reduction.
// Returns CTL_DONE or CTL_STOP, or -1 when a barrier timed out.
template <typename T, int TX, int TY>
__device__ int mg_pass(const PCGArgs<T, 2> &A, const MGHier<T> &H, PCGState &S, T *sblk, T &s_ta, T &s_tb, T *s_ue,
                       int &s_ctl, int bid, int nbk, int *err)
{
    constexpr int NV = 3, NT = TX * TY;
    const bool lead = threadIdx.x == 0;
    const int L = H.L, Lgw = H.Lg < H.L ? H.Lg : H.L, cs = H.csteps;
    const MGLevel<T> &L0 = H.lv[0];
    // the sweeps' place in the dynamic shared memory; the operation's record
    // there is filled by the lead thread (every sweep follows a barrier of the
    // whole block) and read by all
    constexpr size_t OFF = mg_march_offset<T, TX, TY>();
    unsigned char *s_op = pcg_dyn + OFF;

    // ---- grid levels --------------------------------------------------
    // Chebyshev step j on level k: d_j from buffer par, x += d_j, r_{j+1} =
    // r_j - A d_j into buffer 1 - par (post: of the post-smoothing, whose
    // iterate is xpost).  last: apply step j + 1 too (pointwise) and leave the
    // final correction in xpost.
    auto cheb = [&](int k, int j, int par, bool last, bool post) {
        const MGLevel<T> &V = H.lv[k];
        OpCheb2<T> &op = *reinterpret_cast<OpCheb2<T> *>(s_op);
        static_assert(sizeof(op) <= M2_OP_BYTES, "operation record");
        if (lead) {
            op.lam = V.lam; op.mu = V.mu; op.dinv = V.dinv; op.n = (unsigned)V.nx * V.ny;
            op.r = V.r[par][0]; op.d = V.d[par][0]; op.xi = post ? V.xpost[0] : V.xpre[0];
            op.xo = last || post ? V.xpost[0] : V.xpre[0];
            op.rn = V.r[1 - par][0]; op.dn = V.d[1 - par][0];
            op.c1 = H.c1[j]; op.c2 = H.c2[j]; op.n1 = H.c1[j + 1]; op.n2 = H.c2[j + 1];
            op.last = last;
            op.dir = j > 0;
        }
        __syncthreads();
        m2_sweep<T, NT, OFF, OpCheb2<T>>(V.nx, V.ny, A.zc1[k], bid, nbk);
    };
    auto restrict_of = [&](int k) {
        const MGLevel<T> &F = H.lv[k - 1];
        const int pf = H.deg[k - 1] & 1;
        Restrict2<T> R;
        R.r = F.r[pf][0];
        R.fnx = F.nx; R.fny = F.ny;
        return R;
    };
    auto prolong_of = [&](int k) {
        const MGLevel<T> &C = H.lv[k + 1];
        Prolong2<T> P;
        P.x = C.xpost[0];
        P.cnx = C.nx; P.cny = C.ny;
        return P;
    };
    // restriction (transpose of bilinear prolongation) of grid level k-1's
    // residual after its pre-smoothing, at node (gx, gy) of level k (the top
    // block-run level's right-hand side)
    auto restrict_g = [&](int k, int gx, int gy, T (&f)[2]) {
        const MGLevel<T> &F = H.lv[k - 1];
        const int pf = H.deg[k - 1] & 1;
        f[0] = T(0);
        f[1] = T(0);
#pragma unroll
        for (int b = -1; b <= 1; b++) {
            const int fy = wrap(2 * gy + b, F.ny);
            const T wy = b == 0 ? T(1) : T(0.5);
#pragma unroll
            for (int a = -1; a <= 1; a++) {
                const int i = wrap(2 * gx + a, F.nx) + F.nx * fy;
                const T w = wy * (a == 0 ? T(1) : T(0.5));
                f[0] += w * __ldcg(F.r[pf][0] + i);
                f[1] += w * __ldcg(F.r[pf][1] + i);
            }
        }
    };
    // FP64 sweeps are bound by the FP64 pipes: two one-product sweeps and a
    // barrier are cheaper there than one two-product sweep, which repeats two
    // more rows of each chunk (64^2: 18 against 10 us on the 32^2 level)
    constexpr bool PAIR = sizeof(T) == 4;
    // post-smoothing of a grid level k (k = 0: one step, FP64 only; else two)
    auto post = [&](int k, int cur) {
        const MGLevel<T> &V = H.lv[k];
        if constexpr (PAIR) {
            OpPostPair2<T> &op = *reinterpret_cast<OpPostPair2<T> *>(s_op);
            static_assert(sizeof(op) <= M2_OP_BYTES, "operation record");
            if (lead) {
                op.lam = V.lam; op.mu = V.mu; op.dinv = V.dinv; op.n = (unsigned)V.nx * V.ny;
                op.f = V.f[0]; op.xpre = V.xpre[0]; op.xpost = V.xpost[0];
                op.P = prolong_of(k);
                op.c20 = H.c2[0]; op.c11 = H.c1[1]; op.c21 = H.c2[1];
            }
            __syncthreads();
            m2_sweep2<T, NT, OFF, OpPostPair2<T>>(V.nx, V.ny, A.zc2[k], bid, nbk);
            return grid_sync(A.bar_count, A.bar_gen, err, nbk);
        } else {
            OpPost2<T> &op = *reinterpret_cast<OpPost2<T> *>(s_op);
            static_assert(sizeof(op) <= M2_OP_BYTES, "operation record");
            if (lead) {
                op.lam = V.lam; op.mu = V.mu; op.dinv = V.dinv; op.n = (unsigned)V.nx * V.ny;
                op.f = k == 0 ? A.r[cur][0] : V.f[0];
                op.xpre = V.xpre[0]; op.xpost = V.xpost[0]; op.r = V.r[0][0];
                op.P = prolong_of(k);
                op.c2 = H.c2[0];
                op.last = k == 0;
            }
            __syncthreads();
            m2_sweep<T, NT, OFF, OpPost2<T>>(V.nx, V.ny, A.zc1[k], bid, nbk);
            if (!grid_sync(A.bar_count, A.bar_gen, err, nbk)) return false;
            if (k == 0) return true;
            cheb(k, 0, 0, true, true);
            return grid_sync(A.bar_count, A.bar_gen, err, nbk);
        }
    };
    // pre-smoothing of grid level k >= 1 (two steps), or the coarsest solve
    // (csteps >= 3) if the coarsest level is a grid level
    auto pre = [&](int k) {
        const MGLevel<T> &V = H.lv[k];
        if (PAIR && k < L - 1) {
            OpPrePair2<T> &op = *reinterpret_cast<OpPrePair2<T> *>(s_op);
            static_assert(sizeof(op) <= M2_OP_BYTES, "operation record");
            if (lead) {
                op.lam = V.lam; op.mu = V.mu; op.dinv = V.dinv; op.n = (unsigned)V.nx * V.ny;
                op.f = V.f[0]; op.xpre = V.xpre[0]; op.r2 = V.r[0][0];
                op.Rs = restrict_of(k);
                op.c20 = H.c2[0]; op.c11 = H.c1[1]; op.c21 = H.c2[1];
            }
            __syncthreads();
            m2_sweep2<T, NT, OFF, OpPrePair2<T>>(V.nx, V.ny, A.zc2[k], bid, nbk);
            return grid_sync(A.bar_count, A.bar_gen, err, nbk);
        }
        OpPre2<T> &op = *reinterpret_cast<OpPre2<T> *>(s_op);
        static_assert(sizeof(op) <= M2_OP_BYTES, "operation record");
        if (lead) {
            op.lam = V.lam; op.mu = V.mu; op.dinv = V.dinv; op.n = (unsigned)V.nx * V.ny;
            op.f = V.f[0]; op.xpre = V.xpre[0]; op.r1 = V.r[1][0]; op.d1 = V.d[1][0];
            op.Rs = restrict_of(k);
            op.c2 = H.c2[0];
        }
        __syncthreads();
        m2_sweep<T, NT, OFF, OpPre2<T>>(V.nx, V.ny, A.zc1[k], bid, nbk);
        if (!grid_sync(A.bar_count, A.bar_gen, err, nbk)) return false;
        int par = 1;
        const bool co = k == L - 1;
        const int nk = co ? cs - 1 : H.deg[k];
        for (int j = 1; j < nk; j++) {
            cheb(k, j, par, co && j + 1 == nk, false);
            if (!grid_sync(A.bar_count, A.bar_gen, err, nbk)) return false;
            par ^= 1;
        }
        return true;
    };

    // ---- block-run levels (shared memory) ---------------------------------
    // (the marching sweeps on one block's warps took longer than these phases,
    // 29 against 23 us per V-cycle at 512^2: a chain of rows per warp is longer
    // than a phase over all nodes)
    const int nmax = Lgw < L ? H.lv[Lgw].nx * H.lv[Lgw].ny : 0;
    T *scr = bscratch<T>(sblk, H);
    auto bcheb = [&](int k, int j, bool last) {
        const BLevel<T> B = blevel<T>(sblk, H, k);
        const T c1 = H.c1[j], c2 = H.c2[j], n1 = H.c1[j + 1], n2 = H.c2[j + 1];
        blk_sweep<T>(
            B, scr, nmax,
            [&](int i, T (&v)[2]) {
                const T di = c2 * B.dinv[i];
#pragma unroll
                for (int c = 0; c < 2; c++) v[c] = di * B.r[c][i] + (j > 0 ? c1 * B.d[c][i] : T(0));
            },
            [&](int i, const T (&v)[2], const T (&q)[2]) {
                const T di = n2 * B.dinv[i];
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    const T x = B.x[c][i] + v[c];
                    const T rn = B.r[c][i] - q[c];
                    if (last) {
                        B.x[c][i] = x + (n1 * v[c] + di * rn);
                    } else {
                        B.x[c][i] = x;
                        B.r[c][i] = rn;
                        B.d[c][i] = v[c];
                    }
                }
            });
    };
    // (unit >= 0: from the unit vector of that entry in place of the
    // restricted residual)
    auto bpre = [&](int k, int unit) {
        const BLevel<T> B = blevel<T>(sblk, H, k);
        const T c2 = H.c2[0];
        const bool top = k == Lgw;
        blk_sweep<T>(
            B, scr, nmax,
            [&](int i, T (&v)[2]) {
                const int ix = i % B.nx, iy = i / B.nx;
                T f[2];
                if (top && unit >= 0) {
                    f[0] = i == unit ? T(1) : T(0);
                    f[1] = i + B.n == unit ? T(1) : T(0);
                } else if (top) {
                    restrict_g(k, ix, iy, f);
                } else {
                    const BLevel<T> F = blevel<T>(sblk, H, k - 1);
                    f[0] = T(0);
                    f[1] = T(0);
#pragma unroll
                    for (int b = -1; b <= 1; b++) {
                        const int fy = wrap(2 * iy + b, F.ny);
                        const T wy = b == 0 ? T(1) : T(0.5);
#pragma unroll
                        for (int a = -1; a <= 1; a++) {
                            const int fi = wrap(2 * ix + a, F.nx) + F.nx * fy;
                            const T w = wy * (a == 0 ? T(1) : T(0.5));
                            f[0] += w * F.r[0][fi];
                            f[1] += w * F.r[1][fi];
                        }
                    }
                }
                B.f[0][i] = f[0];
                B.f[1][i] = f[1];
                const T di = c2 * B.dinv[i];
                v[0] = di * f[0];
                v[1] = di * f[1];
            },
            [&](int i, const T (&v)[2], const T (&q)[2]) {
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    B.x[c][i] = v[c];
                    B.r[c][i] = B.f[c][i] - q[c];
                    B.d[c][i] = v[c];
                }
            });
        const bool co = k == L - 1;
        const int nk = co ? cs - 1 : H.deg[k];
        for (int j = 1; j < nk; j++) bcheb(k, j, co && j + 1 == nk);
    };
    auto bpost = [&](int k) {
        const int dk = H.deg[k];
        const BLevel<T> B = blevel<T>(sblk, H, k);
        const BLevel<T> C = blevel<T>(sblk, H, k + 1);
        blk_sweep<T>(
            B, scr, nmax,
            [&](int i, T (&v)[2]) {
                const int gx = i % B.nx, gy = i / B.nx;
                const int ox = gx & 1, oy = gy & 1, ix = gx >> 1, iy = gy >> 1;
                const T w = (ox && oy) ? T(0.25) : ((ox || oy) ? T(0.5) : T(1));
                const int ix1 = ox ? (ix + 1 == C.nx ? 0 : ix + 1) : ix, iy1 = oy ? (iy + 1 == C.ny ? 0 : iy + 1) : iy;
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    T e = C.x[c][ix + C.nx * iy];
                    if (ox) e += C.x[c][ix1 + C.nx * iy];
                    if (oy) e += C.x[c][ix + C.nx * iy1];
                    if (ox && oy) e += C.x[c][ix1 + C.nx * iy1];
                    v[c] = B.x[c][i] + w * e;
                }
            },
            [&](int i, const T (&v)[2], const T (&q)[2]) {
                const T di = H.c2[0] * B.dinv[i];
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    const T rn = B.f[c][i] - q[c];
                    B.x[c][i] = dk == 1 ? v[c] + di * rn : v[c];
                    B.r[c][i] = rn;
                }
            });
        for (int j = 0; j + 1 < dk; j++) bcheb(k, j, j + 2 == dk);
    };

    // FP64: the correction of the block-run levels is a fixed symmetric linear
    // map of their right-hand side.  While the first block runs them, the
    // other blocks, which would wait, each compute the map's column of one
    // unit vector; once all columns are there (after a few V-cycles of the
    // solve), the map is applied as a dense product spread over all warps (at
    // 64^2, 512 unknowns: 51 -> 4 us per V-cycle)
    const int nun = Lgw < L ? 2 * H.lv[Lgw].nx * H.lv[Lgw].ny : 0;
    int ncol = 0;
    auto bcycle = [&](int unit, T *dst) {
        for (int k = Lgw; k < L; k++) bpre(k, unit);
        for (int k = L - 2; k >= Lgw; k--) bpost(k);
        const BLevel<T> B = blevel<T>(sblk, H, Lgw);
        for (int i = threadIdx.x; i < 2 * B.n; i += blockDim.x) dst[i] = B.x[0][i];
        __syncthreads();
    };
    auto block64 = [&]() {
        if (ncol < nun) {
            if (bid == 0) bcycle(-1, H.lv[Lgw].xpost[0]);
            else if (ncol + bid - 1 < nun) bcycle(ncol + bid - 1, H.dense + (size_t)(ncol + bid - 1) * nun);
            ncol += nbk - 1;
            return;
        }
        T *f = bscratch<T>(sblk, H);
        const int nn = nun / 2, nx = H.lv[Lgw].nx, lane = threadIdx.x & 31;
        for (int i = threadIdx.x; i < nn; i += blockDim.x) {
            T v[2];
            restrict_g(Lgw, i % nx, i / nx, v);
            f[i] = v[0];
            f[nn + i] = v[1];
        }
        __syncthreads();
        for (int i = (threadIdx.x >> 5) * nbk + bid; i < nun; i += (NT / 32) * nbk) {
            const T *row = H.dense + (size_t)i * nun;
            T y = T(0);
            for (int j = lane; j < nun; j += 32) y = fma(__ldcg(row + j), f[j], y);
            y = warp_sum(y);
            if (lane == 0) H.lv[Lgw].xpost[0][i] = y;
        }
    };

    if ((bid == 0 || !PAIR) && Lgw < L) mg_setup_block<T>(H, sblk);

    int cur = 0;
    bool first = true;
    while (true) {
        if (lead) {
            if (!first) cg_scalar_update<NV>(S);
            s_ta = (T)S.alpha;
            s_tb = (T)S.beta;
            for (int vv = 0; vv < NV; vv++) s_ue[vv] = (T)S.UE[vv];
        }
        __syncthreads();
        const T ta = s_ta, tb = s_tb;
        const int nxt = first ? cur : 1 - cur;

        // ---- finest level, first pre-smoothing sweep; from the second
        // iteration on its own nodes also take the CG update
        Acc<T> racc[1];
        {
            OpFirst2<T> &op = *reinterpret_cast<OpFirst2<T> *>(s_op);
            static_assert(sizeof(op) <= M2_OP_BYTES, "operation record");
            if (lead) {
                op.lam = L0.lam; op.mu = L0.mu; op.dinv = L0.dinv; op.n = (unsigned)L0.nx * L0.ny;
                op.r = A.r[cur][0]; op.w = A.w[cur][0]; op.s = A.s[cur][0]; op.u = L0.xpost[0];
                op.p = A.p[0]; op.x[0] = A.x[0]; op.x[1] = A.x[1]; op.sn = A.s[nxt][0]; op.rn = A.r[nxt][0];
                op.xpre = L0.xpre[0]; op.r1 = L0.r[1][0]; op.d1 = L0.d[1][0];
                op.ta = ta; op.tb = tb; op.c2 = H.c2[0];
                op.upd = !first;
                op.dir = L == 1;
            }
            __syncthreads();
            racc[0] = m2_sweep<T, NT, OFF, OpFirst2<T>>(L0.nx, L0.ny, A.zc1[0], bid, nbk);
        }
        if (!first) {
            double *const tr = S.red;
            if (!reduce_barrier<Acc<T>, 1>(racc, A.partials, 1, A.bar_count, A.bar_gen, err, tr, bid, nbk)) return -1;
            if (lead) {
                double rnew = tr[0];
                for (int vv = 0; vv < NV; vv++) rnew += S.RE[vv] * S.RE[vv];
                S.it++;
                S.rho_final = rnew;
                int ctl = CTL_RUN;
                if (rnew <= S.target * S.target) ctl = CTL_DONE;
                else if (S.it_total + S.it >= A.maxit) ctl = CTL_STOP;
                s_ctl = ctl;
            }
            __syncthreads();
            cur = nxt;
            const int ctl = s_ctl;
            if (ctl != CTL_RUN) return ctl;
        } else if (!grid_sync(A.bar_count, A.bar_gen, err, nbk)) {
            return -1;
        }

        // ---- rest of the V-cycle (one-level hierarchies: the coarsest solve)
        if (L == 1) {
            int par = 1;
            for (int j = 1; j < cs - 1; j++) {
                cheb(0, j, par, j + 2 == cs, false);
                if (!grid_sync(A.bar_count, A.bar_gen, err, nbk)) return -1;
                par ^= 1;
            }
        }
        for (int k = 1; k < Lgw; k++)
            if (!pre(k)) return -1;
        if (Lgw < L) {
            if constexpr (PAIR) {
                if (bid == 0) bcycle(-1, H.lv[Lgw].xpost[0]);
            } else {
                block64();
            }
            if (!grid_sync(A.bar_count, A.bar_gen, err, nbk)) return -1;
        }
        for (int k = (Lgw < L - 1 ? Lgw : L - 1) - 1; k >= (PAIR ? 1 : 0); k--)
            if (!post(k, cur)) return -1;

        // ---- u = V-cycle result (FP32: with the finest level's one-step
        // post-smoothing in the same sweep), w = A u (+ mean strain), gamma, delta, mean-strain row
        Acc<T> acc[2 + NV];
        auto take = [&](const Sums2<T> &sums) {
            acc[0] = sums.ru;
            acc[1] = sums.wu;
            for (int v = 0; v < 3; v++) acc[2 + v].s = T(2) * sums.se[v].s;     // twice half of each cell's stress
        };
        if (PAIR && L > 1) {
            OpFine2<T> &op = *reinterpret_cast<OpFine2<T> *>(s_op);
            static_assert(sizeof(op) <= M2_OP_BYTES, "operation record");
            if (lead) {
                op.lam = L0.lam; op.mu = L0.mu; op.dinv = L0.dinv; op.n = (unsigned)L0.nx * L0.ny;
                op.r = A.r[cur][0]; op.xpre = L0.xpre[0]; op.u = L0.xpost[0]; op.w = A.w[cur][0];
                for (int v = 0; v < 3; v++) op.ue[v] = s_ue[v];
                op.P = prolong_of(0);
                op.c20 = H.c2[0];
            }
            __syncthreads();
            take(m2_sweep2<T, NT, OFF, OpFine2<T>>(L0.nx, L0.ny, A.zc2[0], bid, nbk));
        } else {
            OpApply2<T> &op = *reinterpret_cast<OpApply2<T> *>(s_op);
            static_assert(sizeof(op) <= M2_OP_BYTES, "operation record");
            if (lead) {
                op.lam = L0.lam; op.mu = L0.mu; op.n = (unsigned)L0.nx * L0.ny;
                op.u = L0.xpost[0]; op.r = A.r[cur][0]; op.w = A.w[cur][0];
                for (int v = 0; v < 3; v++) op.ue[v] = s_ue[v];
            }
            __syncthreads();
            take(m2_sweep<T, NT, OFF, OpApply2<T>>(L0.nx, L0.ny, A.zc1[0], bid, nbk));
        }
        double *const tt = S.red;
        if (!reduce_barrier<Acc<T>, 2 + NV>(acc, A.partials, 0, A.bar_count, A.bar_gen, err, tt, bid, nbk)) return -1;
        if (lead) {
            double s6[6];
            dmat_mul<2>(S.Sl, S.Sm, S.UE, s6);
            for (int vv = 0; vv < NV; vv++) S.WE[vv] = tt[2 + vv] + s6[vv];
            double gnew = tt[0], dnew = tt[1];
            for (int vv = 0; vv < NV; vv++) {
                gnew += S.RE[vv] * S.UE[vv];
                dnew += S.WE[vv] * S.UE[vv];
            }
            cg_take_gamma_delta(S, gnew, dnew, first);
        }
        first = false;
    }
}

}  // namespace pfdev
