// Persistent PCG for the mechanics (K3/K4); here the Jacobi-preconditioned
// loops and what they share with the multigrid ones (pf_mg.cuh, pf_mg3.cuh).
//
// The iteration is the Chronopoulos-Gear form of preconditioned CG: with
// u = M^-1 r, w = A u, gamma = r.u, delta = w.u,
//     beta_i  = gamma_i / gamma_{i-1}
//     alpha_i = gamma_i / (delta_i - beta_i gamma_i / alpha_{i-1})
//     p_i = u_i + beta_i p_{i-1},  s_i = w_i + beta_i s_{i-1}
//     x_{i+1} = x_i + alpha_i p_i,  r_{i+1} = r_i - alpha_i s_i
// which produces the iterates of standard PCG but needs all its inner
// products at one point per iteration.  In 2D and in 3D FP64 one sweep over
// node tiles does the vector updates, rebuilds u_{i+1} on the tile and its halo
// in shared memory from r_i, w_i, s_{i-1} (double-buffered in global memory),
// applies the Q1 operator to it and accumulates gamma, delta and ||r||^2: one
// grid barrier per iteration, after which every block sums the blocks'
// partials in the same fixed order.  In 3D FP32 the update is a pass of its
// own, in place, and a marching sweep (pf_march3.cuh) does the rest: two
// barriers.
//
// The few FP64 scalars of the iteration (alpha, beta, the mean-strain dofs)
// are computed by thread 0 of every block (identically, from the same
// reduced values) and broadcast through shared memory: FP64 runs at a small
// fraction of the FP32 rate on this GPU, so no other thread touches them.
#pragma once
#include <type_traits>

#include "pf_kernels.cuh"

namespace pfdev {

// Node tiles of the Jacobi PCG's sweep and of the 2D multigrid's set-up (one
// node per thread: the block has X*Y*Z threads); the shape is a launch option
// (pf_config.pcg_tile), picked per size class from measurements when left to
// the library.  The 32x16 tile runs one 512-thread block per SM: fewer blocks
// in each grid reduction and a smaller idle tail in the halo passes than two
// 256-thread blocks.  The marching sweeps (2D multigrid, 3D FP32) use no tile;
// in 2D the shape still sets their block size, in 3D FP32 nothing.
template <int D, int S> struct Tile;
template <> struct Tile<2, 0> { static constexpr int X = 32, Y = 8, Z = 1; };
template <> struct Tile<2, 1> { static constexpr int X = 32, Y = 16, Z = 1; };
template <> struct Tile<3, 0> { static constexpr int X = 16, Y = 4, Z = 4; };
template <> struct Tile<3, 1> { static constexpr int X = 32, Y = 4, Z = 2; };
constexpr int PCG_SHAPES = 2;

constexpr int MG_MAX_LEVELS = 12;
template <typename T> struct MGHier;

template <typename T, int D>
struct PCGArgs {
    Params P;
    const T *lam, *mu;
    const T *sig[6];
    T *x[3], *p[3];
    T *r[2][3], *w[2][3], *s[2][3];
    T *dinv;                       // inverse of the Jacobi diagonal, written by the set-up
    T *u[3];                       // refinement mode: FP32 displacement written at the end
    double *x64[3];                // refinement mode: FP64 solution
    int refine;                    // 1: FP64 outer residual around the FP32 iteration
    double eta;                    // refinement mode: relative target of one FP32 pass
    double *partials;
    double *emean;                 // refinement mode: FP64 mean strain between two passes, 6 doubles
    unsigned int *bar_count, *bar_gen;
    Scalars *sc;
    Diag *dg;
    double rtol;
    int maxit;
    int warm;
    int block0, nblocks;           // this job's blocks in the launch
    const MGHier<T> *mg;           // multigrid hierarchy (2D, k_pcg<..., MG = true> only)
    double *b64[3];                // MG refinement mode: the FP64 right-hand side, kept from the
                                   // first pass for the later ones
    int zc1[MG_MAX_LEVELS], zc2[MG_MAX_LEVELS];   // MG: rows (3D: planes) per work item of a level's
                                                  // one- and two-product sweeps (pf_march2.cuh, pf_march3.cuh)
};

// Grid barrier that also reduces K per-thread values: the warps of a block
// reduce them, one warp per value combines the warps' and writes the block's
// partial, and after the barrier every block sums all partials in the same
// fixed order, again one warp per value.  (The last block to arrive used to
// sum them before it released the others, one warp for all values: a second
// trip through L2 for every other block and K reductions in a row.)  After
// the call every thread may read the totals in out[], which stay until the
// block's next call.  FP32 values are reduced as error-free (hi, lo) pairs.
// `region` picks one of PCG_REGIONS sets of partials: a set may be written
// again only after another barrier has passed since it was read.  Waits are
// bounded (SPIN_LIMIT polls, then PF_ETIMEOUT in *err and false is returned).
// The scratch is sized for the largest block, 512 threads.
constexpr int PCG_REGIONS = 3, PCG_MAX_WARPS = 16;

template <typename AccT, int K>
__device__ __forceinline__ bool reduce_barrier(AccT (&acc)[K], double *partials, int region, unsigned int *count,
                                            unsigned int *gen, int *err, double *out, int bid, int nbk)
{
    constexpr bool pairs = std::is_same<AccT, Acc<float>>::value;
    __shared__ float sh[pairs ? K : 1][PCG_MAX_WARPS], sl[pairs ? K : 1][PCG_MAX_WARPS];
    __shared__ double sd[pairs ? 1 : K][PCG_MAX_WARPS];
    __shared__ int s_ok;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    double *const part = partials + (size_t)region * nbk * PSTRIDE;
#pragma unroll
    for (int k = 0; k < K; k++) {
        if constexpr (pairs) {
            float h = acc[k].s, l = acc[k].c;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float h2 = __shfl_xor_sync(0xffffffffu, h, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
                pair_add(h, l, h2, l2);
            }
            if (lane == 0) { sh[k][wid] = h; sl[k][wid] = l; }
        } else {
            const double v = warp_sum(acc[k].value());
            if (lane == 0) sd[k][wid] = v;
        }
    }
    __syncthreads();
    for (int k = wid; k < K; k += nw) {
        if constexpr (pairs) {
            float h = lane < nw ? sh[k][lane] : 0.f, l = lane < nw ? sl[k][lane] : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float h2 = __shfl_xor_sync(0xffffffffu, h, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
                pair_add(h, l, h2, l2);
            }
            if (lane == 0) reinterpret_cast<float2 *>(part + (size_t)bid * PSTRIDE)[k] = make_float2(h, l);
        } else {
            const double v = warp_sum(lane < nw ? sd[k][lane] : 0.0);
            if (lane == 0) part[(size_t)bid * PSTRIDE + k] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        s_ok = 1;
        const unsigned int g = ld_relaxed_gpu(gen);
        const unsigned int arrived = atom_add_acq_rel_gpu(count, 1u);
        if (arrived == (unsigned int)nbk - 1) {
            *count = 0u;
            red_add_release_gpu(gen, 1u);
        } else if (!wait_generation(gen, g, err, SPIN_LIMIT)) {
            s_ok = 0;
        }
    }
    __syncthreads();
    for (int k = wid; k < K; k += nw) {
        if constexpr (pairs) {
            float h = 0.f, l = 0.f;
            for (int b = lane; b < nbk; b += 32) {
                const float2 v = __ldcg(reinterpret_cast<const float2 *>(part + (size_t)b * PSTRIDE) + k);
                pair_add(h, l, v.x, v.y);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float h2 = __shfl_xor_sync(0xffffffffu, h, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
                pair_add(h, l, h2, l2);
            }
            if (lane == 0) out[k] = (double)h + (double)l;
        } else {
            double v = 0.0;
            for (int b = lane; b < nbk; b += 32) v += __ldcg(part + (size_t)b * PSTRIDE + k);
            v = warp_sum(v);
            if (lane == 0) out[k] = v;
        }
    }
    __syncthreads();
    return s_ok != 0;
}

// Plain grid barrier (no reduction).  Waits are bounded like reduce_barrier.
__device__ __forceinline__ bool grid_sync(unsigned int *count, unsigned int *gen, int *err, int nbk)
{
    __shared__ int s_gok;
    __syncthreads();
    if (threadIdx.x == 0) {
        s_gok = 1;
        const unsigned int g = ld_relaxed_gpu(gen);
        const unsigned int arrived = atom_add_acq_rel_gpu(count, 1u);
        if (arrived == (unsigned int)nbk - 1) {
            *count = 0u;
            red_add_release_gpu(gen, 1u);
        } else if (!wait_generation(gen, g, err, SPIN_LIMIT)) {
            s_gok = 0;
        }
    }
    __syncthreads();
    return s_gok != 0;
}

// q = sum over the 2^d cells around a node of (lam K_lam + mu K_mu) u_e, plus
// the mean-strain coupling B_a^T D_c UE, from shared-memory tiles.
// su: [D][HN] halo nodes, sl/sm: [HC] halo cells.  (lx, ly, lz): the node's
// halo-local coordinates.
template <typename T, int D, int HX, int HY, int CX, int CY>
__device__ __forceinline__ void apply_tile(const T *su, const T *sl, const T *sm, int HN, int lx, int ly, int lz,
                                           const T *ue, T (&q)[D], T (&eown)[Dims<D>::NV], T &lown, T &mown)
{
    constexpr int NN = Dims<D>::NN, NV = Dims<D>::NV;
#pragma unroll
    for (int d = 0; d < D; d++) q[d] = T(0);
#pragma unroll
    for (int a = 0; a < NN; a++) {
        const int ax = a & 1, ay = (a >> 1) & 1, az = D == 3 ? (a >> 2) & 1 : 0;
        // Halo nodes and halo cells both start one before the tile, so the
        // cell whose lower corner is halo node (cx, cy, cz) has cell-local
        // coordinates (cx, cy, cz); cell a of this node has its lower corner
        // at the node minus bits(a).
        const int cx = lx - ax, cy = ly - ay, cz = lz - az;
        const int cl = cx + CX * (cy + CY * (D == 3 ? cz : 0));
        const T l = sl[cl], m = sm[cl];
        T ul[NN][D];
#pragma unroll
        for (int b = 0; b < NN; b++) {
            const int bx = b & 1, by = (b >> 1) & 1, bz = D == 3 ? (b >> 2) & 1 : 0;
            const int hn = (cx + bx) + HX * ((cy + by) + HY * (D == 3 ? cz + bz : 0));
#pragma unroll
            for (int d = 0; d < D; d++) ul[b][d] = su[d * HN + hn];
        }
#pragma unroll
        for (int co = 0; co < D; co++) {
            T acc = T(0);
#pragma unroll
            for (int b = 0; b < NN; b++)
#pragma unroll
                for (int cc = 0; cc < D; cc++)
                    acc += (l * Kl<T, D>(a * D + co, b * D + cc) + m * Km<T, D>(a * D + co, b * D + cc)) * ul[b][cc];
            q[co] += acc;
        }
        T se[NV], bt[D];
        voigt_stress<T, D>(l, m, ue, se);
        bbar_t<T, D>(a, se, bt);
#pragma unroll
        for (int d = 0; d < D; d++) q[d] += bt[d];
        if (a == 0) {
            avg_strain<T, D>(ul, eown);
            lown = l;
            mown = m;
        }
    }
}

// 2D Q1 element with constant moduli, exact form of its stiffness: writing
// the bilinear displacement of a unit cell as its average gradient G plus
// the hourglass mode h = u00 - u10 - u01 + u11 (per component), the strain is
// G + h * (eta - 1/2, xi - 1/2) terms whose cross products with G integrate
// to zero, so  K_e u = Bbar^T D eps(G) + (lam + 3 mu)/12 * gamma h  with
// gamma = (+1, -1, -1, +1) over the cell's nodes.  cell_force2 returns the
// average stress (without any mean strain) and the two hourglass forces.
template <typename TC>
__device__ __forceinline__ void cell_force2(TC l, TC m, const TC (&ue)[4][2], TC (&s)[3], TC (&fh)[2])
{
    const TC Gxu = TC(0.5) * ((ue[1][0] - ue[0][0]) + (ue[3][0] - ue[2][0]));
    const TC Gyu = TC(0.5) * ((ue[2][0] - ue[0][0]) + (ue[3][0] - ue[1][0]));
    const TC Gxv = TC(0.5) * ((ue[1][1] - ue[0][1]) + (ue[3][1] - ue[2][1]));
    const TC Gyv = TC(0.5) * ((ue[2][1] - ue[0][1]) + (ue[3][1] - ue[1][1]));
    const TC hu = (ue[0][0] - ue[1][0]) - (ue[2][0] - ue[3][0]);
    const TC hv = (ue[0][1] - ue[1][1]) - (ue[2][1] - ue[3][1]);
    const TC tr = Gxu + Gyv;
    s[0] = l * tr + TC(2) * m * Gxu;
    s[1] = l * tr + TC(2) * m * Gyv;
    s[2] = m * (Gyu + Gxv);
    const TC c = (l + TC(3) * m) * TC(1.0 / 12.0);
    fh[0] = c * hu;
    fh[1] = c * hv;
}

// force on the node with local index a of a 2D cell from its average stress
// s (mean strain included) and hourglass forces fh
template <typename TC>
__device__ __forceinline__ void node_force2(int a, const TC *s, const TC *fh, TC (&f)[2])
{
    const TC bx = (a & 1) ? TC(0.5) : TC(-0.5), by = (a >> 1) ? TC(0.5) : TC(-0.5);
    const TC g = (a == 0 || a == 3) ? TC(1) : TC(-1);
    f[0] = bx * s[0] + by * s[2] + g * fh[0];
    f[1] = by * s[1] + bx * s[2] + g * fh[1];
}

// 3D Q1 hex with constant moduli, exact form of its stiffness (the
// counterpart of the 2D decomposition): per displacement component the
// trilinear field of a unit cell is its mean, its average gradient G and the
// modes h1 = xi eta, h2 = eta zeta, h3 = zeta xi, h4 = xi eta zeta (centred
// coordinates).  2x2x2 Gauss integration of the strain energy splits into
// Bbar^T D eps(G) and a quadratic form in the twelve h coefficients whose
// gradient (with respect to h) gives the hourglass forces; the cross terms
// integrate to zero.  cell_force3 returns, in c[20]: the average stress
// (Voigt xx yy zz yz xz xy, without the mean strain) in c[0..5] and the
// forces g[k][comp] = dE/dh_k,comp in c[6 + 3k + comp]; c[18..19] pad.
template <typename TC>
__device__ __forceinline__ void cell_force3(TC l, TC m, const TC (&ue)[8][3], TC (&c)[20])
{
    TC G[3][3], h[4][3];     // G[comp][dir], h[mode][comp]
#pragma unroll
    for (int k = 0; k < 3; k++) {
        // node b = bx + 2 by + 4 bz; pairs along x
        const TC e00 = ue[0][k] + ue[1][k], d00 = ue[1][k] - ue[0][k];
        const TC e01 = ue[2][k] + ue[3][k], d01 = ue[3][k] - ue[2][k];
        const TC e10 = ue[4][k] + ue[5][k], d10 = ue[5][k] - ue[4][k];
        const TC e11 = ue[6][k] + ue[7][k], d11 = ue[7][k] - ue[6][k];
        G[k][0] = TC(0.25) * ((d00 + d01) + (d10 + d11));
        G[k][1] = TC(0.25) * ((e01 + e11) - (e00 + e10));
        G[k][2] = TC(0.25) * ((e10 + e11) - (e00 + e01));
        h[0][k] = TC(0.5) * ((d01 + d11) - (d00 + d10));     // sx sy
        h[1][k] = TC(0.5) * ((e11 - e10) - (e01 - e00));     // sy sz
        h[2][k] = TC(0.5) * ((d10 + d11) - (d00 + d01));     // sz sx
        h[3][k] = (d11 - d10) - (d01 - d00);                 // sx sy sz
    }
    const TC tr = G[0][0] + G[1][1] + G[2][2];
    c[0] = l * tr + TC(2) * m * G[0][0];
    c[1] = l * tr + TC(2) * m * G[1][1];
    c[2] = l * tr + TC(2) * m * G[2][2];
    c[3] = m * (G[1][2] + G[2][1]);
    c[4] = m * (G[0][2] + G[2][0]);
    c[5] = m * (G[0][1] + G[1][0]);
    const TC A = h[0][1] + h[2][2], B = h[0][0] + h[1][2], C = h[2][0] + h[1][1];
    const TC Pq = h[1][0] + h[2][1], Q = h[2][1] + h[0][2], R = h[0][2] + h[1][0];
    const TC c12 = TC(1.0 / 12.0), m3 = TC(3) * m, c144 = (l + TC(4) * m) * TC(1.0 / 144.0);
    c[6] = (l * B + m3 * h[0][0]) * c12;       // mode 1, x
    c[7] = (l * A + m3 * h[0][1]) * c12;       // mode 1, y
    c[8] = m * (Q + R) * c12;                  // mode 1, z
    c[9] = m * (Pq + R) * c12;                 // mode 2, x
    c[10] = (l * C + m3 * h[1][1]) * c12;      // mode 2, y
    c[11] = (l * B + m3 * h[1][2]) * c12;      // mode 2, z
    c[12] = (l * C + m3 * h[2][0]) * c12;      // mode 3, x
    c[13] = m * (Pq + Q) * c12;                // mode 3, y
    c[14] = (l * A + m3 * h[2][2]) * c12;      // mode 3, z
    c[15] = c144 * h[3][0];
    c[16] = c144 * h[3][1];
    c[17] = c144 * h[3][2];
    c[18] = TC(0);
    c[19] = TC(0);
}

// force on the node at corner (ax, ay, az) of a 3D cell from its average
// stress s (mean strain included) and hourglass forces g = c + 6
template <typename TC>
__device__ __forceinline__ void node_force3(int ax, int ay, int az, const TC *s, const TC *g, TC (&f)[3])
{
    const TC sx = ax ? TC(1) : TC(-1), sy = ay ? TC(1) : TC(-1), sz = az ? TC(1) : TC(-1);
    const TC w1 = TC(0.5) * sx * sy, w2 = TC(0.5) * sy * sz, w3 = TC(0.5) * sz * sx, w4 = sx * sy * sz;
    f[0] = TC(0.25) * (sx * s[0] + sy * s[5] + sz * s[4]) + w1 * g[0] + w2 * g[3] + w3 * g[6] + w4 * g[9];
    f[1] = TC(0.25) * (sy * s[1] + sx * s[5] + sz * s[3]) + w1 * g[1] + w2 * g[4] + w3 * g[7] + w4 * g[10];
    f[2] = TC(0.25) * (sz * s[2] + sy * s[3] + sx * s[4]) + w1 * g[2] + w2 * g[5] + w3 * g[8] + w4 * g[11];
}

// Per-node part of the solve's set-up: right-hand side b = sum_e Bbar^T sig*,
// Jacobi diagonal, A x (element tables + mean-strain coupling XE) and the own
// cell's quantities.  TC is the arithmetic type, TV the type of x.
template <typename T, typename TC, typename TV, int D>
__device__ __forceinline__ void node_setup(const Params &P, long long n, const T *lam, const T *mu, const T *const *sig,
                                           TV *const *x, const TC *XE, bool use_x, TC (&b)[D], TC (&ax)[D], TC &dgn,
                                           TC (&sig_own)[Dims<D>::NV], TC (&de_own)[Dims<D>::NV], TC &l_own, TC &m_own)
{
    constexpr int NN = Dims<D>::NN, NV = Dims<D>::NV;
    int i, j, k;
    cell_coords<D>(P, n, i, j, k);
#pragma unroll
    for (int d = 0; d < D; d++) { b[d] = TC(0); ax[d] = TC(0); }
#pragma unroll
    for (int v = 0; v < NV; v++) de_own[v] = TC(0);
    dgn = TC(0);
#pragma unroll
    for (int a = 0; a < NN; a++) {
        const int ox = a & 1, oy = (a >> 1) & 1, oz = D == 3 ? (a >> 2) & 1 : 0;
        const int ci = i - ox, cj = j - oy, ck = k - oz;
        const long long c = lin<D>(P, ci, cj, ck);
        const TC l = (TC)lam[c], m = (TC)mu[c];
        dgn += l * KdL<TC, D>() + m * KdM<TC, D>();
        TC s[NV], bt[D];
#pragma unroll
        for (int v = 0; v < NV; v++) s[v] = (TC)sig[v][c];
        bbar_t<TC, D>(a, s, bt);
#pragma unroll
        for (int d = 0; d < D; d++) b[d] += bt[d];
        if (a == 0) {
#pragma unroll
            for (int v = 0; v < NV; v++) sig_own[v] = s[v];
            l_own = l;
            m_own = m;
        }
        if (use_x) {
            TC ue[NN][D];
#pragma unroll
            for (int bn = 0; bn < NN; bn++) {
                const int px = bn & 1, py = (bn >> 1) & 1, pz = D == 3 ? (bn >> 2) & 1 : 0;
                const long long mm = lin<D>(P, ci + px, cj + py, ck + pz);
#pragma unroll
                for (int d = 0; d < D; d++) ue[bn][d] = (TC)__ldcg(x[d] + mm);
            }
            if constexpr (D == 2) {
                TC s3[3], fh[2], sx[3], f[2];
                cell_force2<TC>(l, m, ue, s3, fh);
                if (a == 0)
#pragma unroll
                    for (int v = 0; v < 3; v++) de_own[v] = s3[v];
                voigt_stress<TC, 2>(l, m, XE, sx);
#pragma unroll
                for (int v = 0; v < 3; v++) s3[v] += sx[v];
                node_force2<TC>(a, s3, fh, f);
                ax[0] += f[0];
                ax[1] += f[1];
            } else {
                // the exact hex decomposition: average stress (plus the mean
                // strain) and hourglass forces of the cell, force on this node
                TC c[20], sx[6], f[3];
                cell_force3<TC>(l, m, ue, c);
                if (a == 0)
#pragma unroll
                    for (int v = 0; v < 6; v++) de_own[v] = c[v];
                voigt_stress<TC, 3>(l, m, XE, sx);
#pragma unroll
                for (int v = 0; v < 6; v++) c[v] += sx[v];
                node_force3<TC>(ox, oy, oz, c, c + 6, f);
#pragma unroll
                for (int d = 0; d < 3; d++) ax[d] += f[d];
            }
        }
    }
}

// Periodic 32-bit index of a tile-halo position.  Halo coordinates lie in
// [-1, n - 1 + tile], so one conditional wrap per axis suffices unless the
// grid is not larger than a tile (small), where a modulo is used.
template <int D>
__device__ __forceinline__ int hidx(const Params &P, int x, int y, int z, bool small)
{
    if (small) return (int)linm<D>(P, x, y, z);
    x += (x < 0) ? P.nx : 0;
    x -= (x >= P.nx) ? P.nx : 0;
    y += (y < 0) ? P.ny : 0;
    y -= (y >= P.ny) ? P.ny : 0;
    if constexpr (D == 3) {
        z += (z < 0) ? P.nz : 0;
        z -= (z >= P.nz) ? P.nz : 0;
        return x + P.nx * (y + P.ny * z);
    }
    return x + P.nx * y;
}

// FP64 state of the iteration, in shared memory and touched only by thread 0
// (so it costs the other threads no registers).
struct PCGState {
    double XE[6];      // mean strain of x (plain) / of the correction (refine)
    double E64[6];     // FP64 mean strain of the solution (refine)
    double DiagE[6], invDiagE[6], RE[6], UE[6], PE[6], SE[6], WE[6];
    double Sl, Sm, bnorm, rho_final, target, prev_res;
    double gamma, delta, gamma_prev, alpha_prev, alpha, beta;
    double inv_gamma, inv_gamma_prev, inv_alpha, inv_alpha_prev;   // FP64 divisions are slow here
    double tot0[10];   // first pass's set-up sums [0, 10) (fixed during a solve; MG refinement reuses them)
    double red[16];    // totals of the last reduction
    int it, it_total, conv;
    // refinement: the FP64 residual has met the tolerance, its square there, and
    // the mean-strain part of the correction added since
    int met;
    double rho_met, cE[6];
};

// Scalar part of one CG update, thread 0 only: beta and alpha from gamma and
// delta (one division here, 1/alpha = den / gamma reusing 1/gamma, and one
// for 1/gamma after the reduction), then the mean-strain dofs' p, s, x, r
// and their Jacobi-preconditioned u.
template <int NV>
__device__ __forceinline__ void cg_scalar_update(PCGState &S)
{
    S.beta = (S.it == 0) ? 0.0 : S.gamma * S.inv_gamma_prev;
    const double den = (S.it == 0) ? S.delta : S.delta - S.beta * S.gamma * S.inv_alpha_prev;
    S.alpha = S.gamma / den;
    S.inv_alpha = den * S.inv_gamma;
    for (int vv = 0; vv < NV; vv++) {
        S.PE[vv] = S.UE[vv] + S.beta * S.PE[vv];
        S.SE[vv] = S.WE[vv] + S.beta * S.SE[vv];
        S.XE[vv] += S.alpha * S.PE[vv];
        S.RE[vv] -= S.alpha * S.SE[vv];
        S.UE[vv] = S.RE[vv] * S.invDiagE[vv];
    }
}

// Thread 0 after the reduction of gamma and delta: shift the previous
// iteration's values (not on the first sweep of a pass).
__device__ __forceinline__ void cg_take_gamma_delta(PCGState &S, double gnew, double dnew, bool first)
{
    if (!first) {
        S.gamma_prev = S.gamma;
        S.alpha_prev = S.alpha;
        S.inv_gamma_prev = S.inv_gamma;
        S.inv_alpha_prev = S.inv_alpha;
    }
    S.gamma = gnew;
    S.delta = dnew;
    S.inv_gamma = 1.0 / gnew;
}

// Control words broadcast by thread 0.
enum { CTL_RUN = 0, CTL_DONE = 1, CTL_ZERO = 2, CTL_STOP = 3, CTL_UNDO = 4 };

}  // namespace pfdev

#include "pf_march2.cuh"
#include "pf_march3.cuh"
#include "pf_mg.cuh"
#include "pf_mg3.cuh"

namespace pfdev {

// The solve.  Plain mode (refine = 0): x = A.x (the displacement itself).
// Refinement mode (FP32 storage): the solution is kept in FP64 (A.x64 and the
// FP64 mean strain); every outer pass forms the true residual b - A x64 in
// FP64, solves for a correction with the FP32 iteration (A.x holds the
// correction), adds it in FP64, and stops when the FP64 residual meets rtol;
// the FP32 displacement A.u is written from x64 at the end.
// the hierarchy's place in shared memory, none without multigrid
template <typename T, bool MG> struct MGStore { MGHier<T> h; };
template <typename T> struct MGStore<T, false> {};

template <int D, int S>
constexpr int tile_threads() { return Tile<D, S>::X * Tile<D, S>::Y * Tile<D, S>::Z; }
static_assert(tile_threads<2, 1>() <= 32 * PCG_MAX_WARPS && tile_threads<3, 0>() <= 32 * PCG_MAX_WARPS &&
              MG3_THREADS <= 32 * PCG_MAX_WARPS, "warps of a block");

// The Jacobi loops' scalars after a sweep's reduction (tt: gamma, delta,
// ||r||^2, mean-strain row): counts the iteration, tests ||r|| <= target, takes
// gamma and delta; returns what to do next to every thread.
template <int D>
__device__ __forceinline__ int pcg_step(PCGState &S, const double *tt, bool was_first, double target, int maxit, int &s_ctl)
{
    constexpr int NV = Dims<D>::NV;
    if (threadIdx.x == 0) {
        double s6[6];
        dmat_mul<D>(S.Sl, S.Sm, S.UE, s6);
        for (int vv = 0; vv < NV; vv++) S.WE[vv] = tt[3 + vv] + s6[vv];
        double gnew = tt[0], dnew = tt[1], rnew = tt[2];
        for (int vv = 0; vv < NV; vv++) {
            gnew += S.RE[vv] * S.UE[vv];
            dnew += S.WE[vv] * S.UE[vv];
            rnew += S.RE[vv] * S.RE[vv];
        }
        int ctl = CTL_RUN;
        if (!was_first) {
            S.it++;
            S.rho_final = rnew;
            if (rnew <= target * target) ctl = CTL_DONE;      // ||r|| <= target without a square root
            else if (S.it_total + S.it >= maxit) ctl = CTL_STOP;
        }
        cg_take_gamma_delta(S, gnew, dnew, was_first);
        s_ctl = ctl;
    }
    __syncthreads();
    return s_ctl;
}

// Refinement, own nodes: the pass's correction (A.x, S.XE) added to the
// solution.  If the solution had met the tolerance, A.u (written at the end of
// the solve) and S.cE keep the correction for refine_undo.
template <typename T, int D>
__device__ __noinline__ void refine_add(const PCGArgs<T, D> &A, PCGState &S, int bid, int nbk)
{
    const long long N = A.P.N, t0 = bid * (long long)blockDim.x + threadIdx.x, st = (long long)nbk * blockDim.x;
    const bool keep = S.met != 0;
    for (int d = 0; d < D; d++) {
        const T *__restrict__ x = A.x[d];
        double *__restrict__ y = A.x64[d];
#pragma unroll 4
        for (long long n = t0; n < N; n += st) y[n] += (double)x[n];
        T *__restrict__ u = A.u[d];
        if (keep)
            for (long long n = t0; n < N; n += st) u[n] = x[n];
    }
    if (threadIdx.x == 0)
        for (int v = 0; v < Dims<D>::NV; v++) {
            S.cE[v] = S.XE[v];
            S.E64[v] += S.XE[v];
            if (bid == 0) A.emean[v] = S.E64[v];
        }
}
// ... and taken back (x64 to its rounding)
template <typename T, int D>
__device__ __noinline__ void refine_undo(const PCGArgs<T, D> &A, PCGState &S, int bid, int nbk)
{
    for (long long n = bid * (long long)blockDim.x + threadIdx.x; n < A.P.N; n += (long long)nbk * blockDim.x)
#pragma unroll
        for (int d = 0; d < D; d++) A.x64[d][n] -= (double)A.u[d][n];
    if (threadIdx.x == 0)
        for (int v = 0; v < Dims<D>::NV; v++) S.E64[v] -= S.cE[v];
}

// threads of a block: one per tile node; 3D in FP32 (pf_march3.cuh): MG3_THREADS
template <typename T, int D, int S, bool MG>
constexpr int pcg_threads() { return D == 3 && sizeof(T) == 4 ? MG3_THREADS : tile_threads<D, S>(); }

template <typename T, int D, int SH, bool MG>
__global__ void __launch_bounds__(pcg_threads<T, D, SH, MG>(), D == 3 && sizeof(T) == 4 ? 1 : 512 / tile_threads<D, SH>())
k_pcg(const PCGArgs<T, D> *jobs, int njobs)
{
    // this block's job, copied to shared memory
    __shared__ PCGArgs<T, D> sA;
    {
        const PCGArgs<T, D> *J = my_job(jobs, njobs);
        const int *src = reinterpret_cast<const int *>(J);
        int *dst = reinterpret_cast<int *>(&sA);
        for (int i = threadIdx.x; i < (int)(sizeof(PCGArgs<T, D>) / sizeof(int)); i += blockDim.x) dst[i] = src[i];
        __syncthreads();
    }
    const PCGArgs<T, D> &A = sA;
    const int bid = (int)blockIdx.x - A.block0, nbk = A.nblocks;
    constexpr int NV = Dims<D>::NV;
    constexpr int TX = Tile<D, SH>::X, TY = Tile<D, SH>::Y, TZ = Tile<D, SH>::Z;
    constexpr int HX = TX + 2, HY = TY + 2, HZ = D == 3 ? TZ + 2 : 1;
    constexpr int CX = TX + 1, CY = TY + 1, CZ = D == 3 ? TZ + 1 : 1;
    constexpr int HN = HX * HY * HZ, HC = CX * CY * CZ;
    constexpr int MAX_OUTER = 24;
    // 3D FP32: warp-marching sweeps (pf_march3.cuh)
    constexpr bool MARCH = D == 3 && sizeof(T) == 4;
    // the node and cell tiles of the plain sweep (the multigrid variants
    // keep theirs in the dynamic shared memory)
    __shared__ T su[MG || MARCH ? 1 : D * HN];
    __shared__ T sl[MG || MARCH ? 1 : HC], sm[MG || MARCH ? 1 : HC];
    // 2D: per-cell stress and hourglass forces, 5 values per cell (3D FP64
    // uses the element-matrix path and needs none)
    __shared__ __align__(16) T scell[D == 2 && !MG ? 5 * HC : 1];
    __shared__ T s_ta, s_tb, s_ue[6], s_xe[6];
    __shared__ int s_ctl;

    const Params &P = A.P;
    const long long N = P.N;
    int *err = &A.sc->status;
    const int ntx = (P.nx + TX - 1) / TX, nty = (P.ny + TY - 1) / TY, ntz = D == 3 ? (P.nz + TZ - 1) / TZ : 1;
    const int ntiles = ntx * nty * ntz;
    const int tx = threadIdx.x % TX, ty = (threadIdx.x / TX) % TY, tz = D == 3 ? threadIdx.x / (TX * TY) : 0;
    const long long t0 = bid * (long long)blockDim.x + threadIdx.x;
    const long long st = (long long)nbk * blockDim.x;
    const bool refine = A.refine != 0;
    const bool lead = threadIdx.x == 0;
    const bool small = P.nx < TX + 2 || P.ny < TY + 2 || (D == 3 && P.nz < TZ + 2);

    __shared__ PCGState S;
    double *XE = S.XE, *E64 = S.E64, *DiagE = S.DiagE, *RE = S.RE, *UE = S.UE, *PE = S.PE, *SE = S.SE;
    double &Sl = S.Sl, &Sm = S.Sm, &bnorm = S.bnorm, &rho_final = S.rho_final, &target = S.target;
    double &gamma = S.gamma, &delta = S.delta, &gamma_prev = S.gamma_prev, &alpha_prev = S.alpha_prev;
    double &alpha = S.alpha, &beta = S.beta;
    int &it = S.it, &it_total = S.it_total;
    bool conv = false;
    if (lead) {
        for (int v = 0; v < 6; v++) { XE[v] = 0.0; E64[v] = 0.0; }
        Sl = Sm = bnorm = rho_final = target = 0.0;
        gamma = delta = alpha = beta = 0.0;
        gamma_prev = alpha_prev = 1.0;
        S.inv_gamma = S.inv_gamma_prev = S.inv_alpha = S.inv_alpha_prev = 1.0;
        it = 0;
        it_total = 0;
        S.met = 0;
        if (A.warm)
            for (int v = 0; v < NV; v++) (refine ? E64 : XE)[v] = A.sc->E[v];
    }

    // MG: a copy of the hierarchy descriptor in shared memory (its pointers
    // are read all over a V-cycle); the coarse levels' moduli are rebuilt for
    // this solve; the block-run levels' arrays: dynamic shared memory
    // (pcg_dyn_smem)
    __shared__ MGStore<T, MG> sH;
    T *sblk = reinterpret_cast<T *>(pcg_dyn);
    if constexpr (MG) {
        const int *src = reinterpret_cast<const int *>(A.mg);
        int *dst = reinterpret_cast<int *>(&sH.h);
        for (int i = threadIdx.x; i < (int)(sizeof(MGHier<T>) / sizeof(int)); i += blockDim.x) dst[i] = src[i];
        __syncthreads();
        if constexpr (D == 2) {
            if (!mg_setup<T>(sH.h, A.bar_count, A.bar_gen, err, bid, nbk)) return;
        } else {
            if (!mg_setup3<T>(sH.h, A.bar_count, A.bar_gen, err, bid, nbk)) return;
        }
    }

    for (int outer = 0; outer < (refine ? MAX_OUTER : 1); outer++) {
        // ---------------- set-up: r0 = b - A x0, diagonal, cell sums --------
        const bool use_x = refine ? (A.warm || outer > 0) : (A.warm != 0);
        if (lead)
            for (int v = 0; v < NV; v++) s_xe[v] = (T)(refine ? 0.0 : XE[v]);
        __syncthreads();
        {
            // every thread needs the mean strain of x for A x: FP64 from the
            // previous pass (refine) or the FP32 copy broadcast above
            double xe64[6];
            T xeT[6];
            for (int v = 0; v < NV; v++) {
                xe64[v] = outer == 0 ? (A.warm ? A.sc->E[v] : 0.0) : __ldcg(A.emean + v);
                xeT[v] = s_xe[v];
            }
            Acc<double> acc[16];
            if constexpr (MG && D == 2) {
                // 2D multigrid variant: the tiled FP64 set-up (cells once per
                // tile) in the dynamic shared memory; later refinement passes
                // only form the residual
                setup_tiled<T, TX, TY>(A, use_x, refine, refine && outer > 0, xe64,
                                       reinterpret_cast<double *>(pcg_dyn), acc, bid, nbk);
            } else if constexpr (MG || MARCH) {
                // 3D multigrid variant and the mixed method: the z-marching sweep
                setup_march3<T, MG>(A, use_x, refine, MG && refine && outer > 0, xe64, reinterpret_cast<double *>(pcg_dyn), acc,
                                bid, nbk);
            } else
            for (long long n = t0; n < N; n += st) {
                double bv[D], rv[D];
                if (refine) {
                    double b[D], ax[D], dgn, so[NV], deo[NV], lo, mo;
                    node_setup<T, double, double, D>(P, n, A.lam, A.mu, A.sig, A.x64, xe64, use_x, b, ax, dgn, so, deo, lo, mo);
                    A.dinv[n] = (T)(1.0 / dgn);
#pragma unroll
                    for (int d = 0; d < D; d++) { bv[d] = b[d]; rv[d] = b[d] - ax[d]; }
                    acc[2].add(lo); acc[3].add(mo);
#pragma unroll
                    for (int v = 0; v < NV; v++) { acc[4 + v].add(so[v]); acc[10 + v].add(deo[v]); }
                    if (!use_x)
#pragma unroll
                        for (int d = 0; d < D; d++) A.x64[d][n] = 0.0;
                } else {
                    T b[D], ax[D], dgn, so[NV], deo[NV], lo, mo;
                    node_setup<T, T, T, D>(P, n, A.lam, A.mu, A.sig, A.x, xeT, use_x, b, ax, dgn, so, deo, lo, mo);
                    A.dinv[n] = T(1) / dgn;
#pragma unroll
                    for (int d = 0; d < D; d++) { bv[d] = (double)b[d]; rv[d] = (double)(b[d] - ax[d]); }
                    acc[2].add((double)lo); acc[3].add((double)mo);
#pragma unroll
                    for (int v = 0; v < NV; v++) { acc[4 + v].add((double)so[v]); acc[10 + v].add((double)deo[v]); }
                }
#pragma unroll
                for (int d = 0; d < D; d++) {
                    if (refine || !use_x) A.x[d][n] = T(0);
                    A.p[d][n] = T(0);
                    A.s[0][d][n] = T(0);
                    A.r[0][d][n] = (T)rv[d];
                    acc[0].addprod(bv[d], bv[d]);
                    acc[1].addprod(rv[d], rv[d]);
                }
            }
            double *const tot = S.red;
            if (!reduce_barrier<Acc<double>, 16>(acc, A.partials, 2, A.bar_count, A.bar_gen, err, tot, bid, nbk)) return;
            if (lead) {
                // a residual-only pass reuses the first pass's sums of b, the
                // moduli and the eigenstress
                if (MG && refine) {
                    if (outer == 0)
                        for (int k = 0; k < 10; k++) S.tot0[k] = tot[k];
                    else
                        for (int k = 0; k < 10; k++)
                            if (k != 1) tot[k] = S.tot0[k];
                }
                // scalars of the mean-strain dofs
                Sl = tot[2];
                Sm = tot[3];
                double AXE[6], unit[6], s6[6];
                for (int vv = 0; vv < NV; vv++) {
                    for (int w = 0; w < NV; w++) unit[w] = (w == vv) ? 1.0 : 0.0;
                    dmat_mul<D>(Sl, Sm, unit, s6);
                    DiagE[vv] = s6[vv];
                    S.invDiagE[vv] = 1.0 / s6[vv];
                }
                dmat_mul<D>(Sl, Sm, refine ? E64 : XE, AXE);
                double bbt = tot[0], rho = tot[1];
                for (int vv = 0; vv < NV; vv++) {
                    const double BE = tot[4 + vv] + (vv < D ? (double)N * (-P.prestress) : 0.0);
                    RE[vv] = BE - (use_x ? tot[10 + vv] + AXE[vv] : 0.0);
                    UE[vv] = RE[vv] * S.invDiagE[vv];
                    bbt += BE * BE;
                    rho += RE[vv] * RE[vv];
                    PE[vv] = 0.0;
                    SE[vv] = 0.0;
                    if (refine) XE[vv] = 0.0;
                }
                bnorm = sqrt(bbt);
                rho_final = rho;
                int ctl = CTL_RUN;
                // refinement goes on to half the tolerance: its passes end
                // anywhere below their targets, and a residual just under the
                // tolerance would leave an error several times the usual one.
                // A solution that meets the tolerance but not its half (met)
                // gets one more pass, and comes back if that pass's correction
                // takes the residual above the tolerance again
                const double res = sqrt(rho), tol = A.rtol * bnorm;
                if (bnorm == 0.0) ctl = CTL_ZERO;
                else if (res <= (refine ? 0.5 * tol : tol)) ctl = CTL_DONE;
                else if (refine && S.met && !(res <= tol)) ctl = CTL_UNDO;
                // refinement that no longer halves the FP64 residual has
                // reached what the FP32 passes can resolve: stop (not
                // converged unless the tolerance is met)
                else if (refine && outer > 0 && res > 0.5 * S.prev_res) ctl = res <= tol ? CTL_DONE : CTL_STOP;
                else if (refine && res <= tol) {
                    S.met = 1;
                    S.rho_met = rho;
                }
                if (ctl == CTL_UNDO) rho_final = S.rho_met;
                S.prev_res = res;
                // target of this pass: the requested tolerance, or in refinement
                // mode what an FP32 iteration can deliver on this correction
                // (eta); when the final tolerance is not far below that, the pass
                // aims for it directly, which saves a pass that would otherwise
                // start just above the tolerance: within a factor 100, but 10
                // with the Jacobi preconditioner on axes of more than 64 nodes.
                // (FP32 passes there do not always get down to 3e-5 of where they
                // start, and ran on to cg_maxit: of 30 core-shells of 224 x 138,
                // rtol 1e-10, 15 failed with 100 here, none with 10; 0.5 tol and
                // 100, before the solves went on to half the tolerance, 6.  The
                // iterations are as many; on small grids 10 costs a few per cent.)
                if (refine) {
                    const bool deep = MG || max(P.nx, max(P.ny, D == 3 ? P.nz : 1)) <= 64;
                    const double fin = 0.25 * tol, pass = A.eta * res;
                    target = fin >= (deep ? 0.01 : 0.1) * pass ? fin : pass;
                } else {
                    target = A.rtol * bnorm;
                }
                gamma = 0.0; delta = 0.0; gamma_prev = 1.0; alpha_prev = 1.0; alpha = 0.0; beta = 0.0;
                S.inv_gamma = S.inv_gamma_prev = S.inv_alpha = S.inv_alpha_prev = 1.0;
                it = 0;
                s_ctl = ctl;
            }
            __syncthreads();
        }
        const int ctl0 = s_ctl;
        if (ctl0 == CTL_ZERO) {
            for (long long n = t0; n < N; n += st)
                for (int d = 0; d < D; d++) {
                    A.x[d][n] = T(0);
                    if (refine) A.x64[d][n] = 0.0;
                }
            if (lead) {
                for (int vv = 0; vv < NV; vv++) { XE[vv] = 0.0; E64[vv] = 0.0; }
                rho_final = 0.0;
            }
            conv = true;
            break;
        }
        if (ctl0 == CTL_DONE) { conv = true; break; }
        if (ctl0 == CTL_STOP) { conv = false; break; }
        if (ctl0 == CTL_UNDO) {
            refine_undo<T, D>(A, S, bid, nbk);
            conv = true;
            break;
        }

        // ---------------- sweeps: the first builds w_0, then iterations -----
        if constexpr (MG) {
            int rc;
            if constexpr (D == 2)
                rc = mg_pass<T, TX, TY>(A, sH.h, S, sblk, s_ta, s_tb, s_ue, s_ctl, bid, nbk, err);
            else
                rc = mg_pass3<T>(A, sH.h, S, reinterpret_cast<T *>(pcg_dyn), s_ta, s_tb, s_ue, s_ctl, bid, nbk, err);
            if (rc < 0) return;
            if (lead) conv = rc == CTL_DONE;
        } else if constexpr (MARCH) {
            // The CG update in a pass of its own, in place (p = D^-1 r + beta
            // p, x += alpha p, s = w + beta s, r -= alpha s), then one
            // marching sweep forms u = D^-1 r, w = A u and the sums: per node
            // 19 words in the update, 10 and the halo rows in the sweep, and
            // a second grid barrier, against a halo of 2.5 nodes per node
            // that each formed from r, w and s on 16x4x4 tiles, with 20
            // values per cell through shared memory.  53x47x61, per
            // iteration: 37 us -> 26 us.
            __shared__ __align__(16) unsigned char s_jop[sizeof(OpJac3)];
            OpJac3 &op = *reinterpret_cast<OpJac3 *>(s_jop);
            bool first = true;
            int redpar = 0;
            while (true) {
                if (lead) {
                    if (!first) cg_scalar_update<NV>(S);
                    s_ta = (T)alpha;
                    s_tb = (T)beta;
                    op.lam = A.lam; op.mu = A.mu; op.dinv = A.dinv; op.r = A.r[0][0]; op.w = A.w[0][0];
                    op.n = (unsigned)N;
                    for (int vv = 0; vv < NV; vv++) op.ue[vv] = (T)UE[vv];
                }
                __syncthreads();
                if (!first) {
                    const T ta = s_ta, tb = s_tb;
                    for (long long n = t0; n < N; n += st) {
                        const T di = A.dinv[n];
#pragma unroll
                        for (int d = 0; d < D; d++) {
                            const T rv = A.r[0][d][n];
                            const T pi = di * rv + tb * A.p[d][n], si = __ldcg(A.w[0][d] + n) + tb * A.s[0][d][n];
                            A.p[d][n] = pi;
                            A.x[d][n] += ta * pi;
                            A.s[0][d][n] = si;
                            A.r[0][d][n] = rv - ta * si;
                        }
                    }
                    if (!grid_sync(A.bar_count, A.bar_gen, err, nbk)) return;
                }
                const SumsJ3 sums = m3_sweep(&op, P.nx, P.ny, P.nz, A.zc1[0], bid, nbk);
                Acc<T> acc[3 + NV];      // gamma, delta, ||r||^2, mean-strain row
                acc[0] = sums.ru;
                acc[1] = sums.wu;
                acc[2] = sums.rr;
                for (int v = 0; v < NV; v++) acc[3 + v].s = T(4) * sums.se[v].s;     // four times a quarter of each cell's stress
                double *const tt = S.red;
                if (!reduce_barrier<Acc<T>, 3 + NV>(acc, A.partials, redpar, A.bar_count, A.bar_gen, err, tt, bid, nbk)) return;
                redpar ^= 1;
                const int ctl = pcg_step<D>(S, tt, first, target, A.maxit, s_ctl);
                first = false;
                if (ctl == CTL_DONE || ctl == CTL_STOP) {
                    if (lead) conv = (ctl == CTL_DONE);
                    break;
                }
            }
        } else {
            bool first = true;
            int cur = 0, redpar = 0;
            while (true) {
                if (lead) {
                    if (!first) cg_scalar_update<NV>(S);
                    s_ta = (T)alpha;
                    s_tb = (T)beta;
                    for (int vv = 0; vv < NV; vv++) s_ue[vv] = (T)UE[vv];
                }
                __syncthreads();
                const T ta = s_ta, tb = s_tb;
                T ue[NV];
    #pragma unroll
                for (int vv = 0; vv < NV; vv++) ue[vv] = s_ue[vv];
                const int nxt = first ? cur : 1 - cur;
                Acc<T> acc[3 + NV];      // gamma, delta, ||r||^2, mean-strain row
                // Register double buffering across tiles: the loads of the next
                // tile's halo (r, w, s, diag), cells (lam, mu) and own node are
                // issued before the current tile is staged and computed, so their
                // latency overlaps that work.
                constexpr int NT = TX * TY * TZ;       // threads = tile nodes
                constexpr int HS = (HN + NT - 1) / NT, CS = (HC + NT - 1) / NT;
                struct Raw {
                    T r[HS][D], w[HS][D], s[HS][D], dg[HS];
                    T l[CS], m[CS];
                    T ro[D], wo[D], so[D], xo[D], po[D], dgo;
                };
                auto load_raw = [&](int tile, Raw &R) {
                    const int bx = tile % ntx, by = (tile / ntx) % nty, bz = D == 3 ? tile / (ntx * nty) : 0;
                    const int x0 = bx * TX, y0 = by * TY, z0 = bz * TZ;
    #pragma unroll
                    for (int k = 0; k < HS; k++) {
                        const int h = threadIdx.x + NT * k;
                        if (h < HN) {
                            const int lx = h % HX, ly = (h / HX) % HY, lz = D == 3 ? h / (HX * HY) : 0;
                            const int g = hidx<D>(P, x0 - 1 + lx, y0 - 1 + ly, z0 - 1 + lz, small);
                            R.dg[k] = __ldcg(A.dinv + g);
    #pragma unroll
                            for (int d = 0; d < D; d++) {
                                R.r[k][d] = __ldcg(A.r[cur][d] + g);
                                if (!first) {
                                    R.w[k][d] = __ldcg(A.w[cur][d] + g);
                                    R.s[k][d] = __ldcg(A.s[cur][d] + g);
                                }
                            }
                        }
                    }
    #pragma unroll
                    for (int k = 0; k < CS; k++) {
                        const int h = threadIdx.x + NT * k;
                        if (h < HC) {
                            const int lx = h % CX, ly = (h / CX) % CY, lz = D == 3 ? h / (CX * CY) : 0;
                            const int g = hidx<D>(P, x0 - 1 + lx, y0 - 1 + ly, z0 - 1 + lz, small);
                            R.l[k] = __ldg(A.lam + g);
                            R.m[k] = __ldg(A.mu + g);
                        }
                    }
                    const int gx = x0 + tx, gy = y0 + ty, gz = z0 + tz;
                    if (gx < P.nx && gy < P.ny && (D == 2 || gz < P.nz)) {
                        const int n = gx + P.nx * (gy + (D == 3 ? P.ny * gz : 0));
                        R.dgo = __ldcg(A.dinv + n);
    #pragma unroll
                        for (int d = 0; d < D; d++) {
                            R.ro[d] = __ldcg(A.r[cur][d] + n);
                            if (!first) {
                                R.wo[d] = __ldcg(A.w[cur][d] + n);
                                R.so[d] = __ldcg(A.s[cur][d] + n);
                                R.xo[d] = A.x[d][n];
                                R.po[d] = A.p[d][n];
                            }
                        }
                    }
                };
                Raw R;
                if (bid < ntiles) load_raw(bid, R);
                for (int tile = bid; tile < ntiles; tile += nbk) {
                    const int bx = tile % ntx, by = (tile / ntx) % nty, bz = D == 3 ? tile / (ntx * nty) : 0;
                    const int x0 = bx * TX, y0 = by * TY, z0 = bz * TZ;
                    // stage this tile: u_{i+1} = (r_i - alpha (w_i + beta s_{i-1})) / diag
                    // on the halo nodes, lam / mu on the halo cells
    #pragma unroll
                    for (int k = 0; k < HS; k++) {
                        const int h = threadIdx.x + NT * k;
                        if (h < HN) {
                            const T inv = R.dg[k];
    #pragma unroll
                            for (int d = 0; d < D; d++) {
                                T rv = R.r[k][d];
                                if (!first) rv -= ta * (R.w[k][d] + tb * R.s[k][d]);
                                su[d * HN + h] = rv * inv;
                            }
                        }
                    }
    #pragma unroll
                    for (int k = 0; k < CS; k++) {
                        const int h = threadIdx.x + NT * k;
                        if (h < HC) {
                            sl[h] = R.l[k];
                            sm[h] = R.m[k];
                        }
                    }
                    T ro[D], wo[D], so[D], xo[D], po[D];
                    const T dgo = R.dgo;
    #pragma unroll
                    for (int d = 0; d < D; d++) { ro[d] = R.ro[d]; wo[d] = R.wo[d]; so[d] = R.so[d]; xo[d] = R.xo[d]; po[d] = R.po[d]; }
                    // issue the next tile's loads; they complete while this one computes
                    if (tile + nbk < ntiles) load_raw(tile + nbk, R);
                    __syncthreads();
                    if constexpr (D == 2) {
                        // per halo cell: average stress (mean strain UE included)
                        // and hourglass forces, shared by the cell's four nodes
                        for (int h = threadIdx.x; h < HC; h += blockDim.x) {
                            const int cx = h % CX, cy = h / CX;
                            T uc[4][2];
    #pragma unroll
                            for (int b = 0; b < 4; b++) {
                                const int hn = (cx + (b & 1)) + HX * (cy + (b >> 1));
                                uc[b][0] = su[hn];
                                uc[b][1] = su[HN + hn];
                            }
                            const T l = sl[h], m = sm[h];
                            T s3[3], fh[2], sx[3];
                            cell_force2<T>(l, m, uc, s3, fh);
                            voigt_stress<T, 2>(l, m, ue, sx);
                            scell[h] = s3[0] + sx[0];
                            scell[HC + h] = s3[1] + sx[1];
                            scell[2 * HC + h] = s3[2] + sx[2];
                            scell[3 * HC + h] = fh[0];
                            scell[4 * HC + h] = fh[1];
                        }
                        __syncthreads();
                    }
                    const int gx = x0 + tx, gy = y0 + ty, gz = z0 + tz;
                    const bool active = gx < P.nx && gy < P.ny && (D == 2 || gz < P.nz);
                    if (active) {
                        const int n = gx + P.nx * (gy + (D == 3 ? P.ny * gz : 0));
                        const int lx = tx + 1, ly = ty + 1, lz = D == 3 ? tz + 1 : 0;
                        const int hn = lx + HX * (ly + HY * lz);
                        T un[D];
    #pragma unroll
                        for (int d = 0; d < D; d++) un[d] = su[d * HN + hn];
                        T rn[D];
                        if (!first) {
                            const T inv = dgo;
    #pragma unroll
                            for (int d = 0; d < D; d++) {
                                const T ri = ro[d];
                                const T si = wo[d] + tb * so[d];
                                const T pi = ri * inv + tb * po[d];
                                A.p[d][n] = pi;
                                A.x[d][n] = xo[d] + ta * pi;
                                A.s[nxt][d][n] = si;
                                rn[d] = ri - ta * si;
                                A.r[nxt][d][n] = rn[d];
                            }
                        } else {
    #pragma unroll
                            for (int d = 0; d < D; d++) rn[d] = ro[d];
                        }
                        T q[D], se[NV];
                        if constexpr (D == 2) {
                            q[0] = T(0);
                            q[1] = T(0);
    #pragma unroll
                            for (int a = 0; a < 4; a++) {
                                const int cl = (lx - (a & 1)) + CX * (ly - (a >> 1));
                                const T s3[3] = {scell[cl], scell[HC + cl], scell[2 * HC + cl]};
                                const T fh[2] = {scell[3 * HC + cl], scell[4 * HC + cl]};
                                T f[2];
                                node_force2<T>(a, s3, fh, f);
                                q[0] += f[0];
                                q[1] += f[1];
                            }
                            // own cell's average stress without the mean strain
                            const int c0 = lx + CX * ly;
                            T sx[3];
                            voigt_stress<T, 2>(sl[c0], sm[c0], ue, sx);
                            se[0] = scell[c0] - sx[0];
                            se[1] = scell[HC + c0] - sx[1];
                            se[2] = scell[2 * HC + c0] - sx[2];
                        } else {
                            T eo[NV], lo, mo;
                            apply_tile<T, D, HX, HY, CX, CY>(su, sl, sm, HN, lx, ly, lz, ue, q, eo, lo, mo);
                            voigt_stress<T, D>(lo, mo, eo, se);
                        }
    #pragma unroll
                        for (int d = 0; d < D; d++) {
                            A.w[nxt][d][n] = q[d];
                            acc[0].fma_plain(rn[d], un[d]);
                            acc[1].fma_plain(q[d], un[d]);
                            acc[2].fma_plain(rn[d], rn[d]);
                        }
    #pragma unroll
                        for (int vv = 0; vv < NV; vv++) acc[3 + vv].add_plain(se[vv]);
                    }
                    __syncthreads();
                }
                double *const tt = S.red;
                if (!reduce_barrier<Acc<T>, 3 + NV>(acc, A.partials, redpar, A.bar_count, A.bar_gen, err, tt, bid, nbk)) return;
                redpar ^= 1;
                const int ctl = pcg_step<D>(S, tt, first, target, A.maxit, s_ctl);
                if (!first) cur = nxt;
                first = false;
                if (ctl == CTL_DONE || ctl == CTL_STOP) {
                    if (lead) conv = (ctl == CTL_DONE);
                    break;
                }
            }
        }
        if (lead) it_total += it;
        if (!refine) break;
        // every warp has read s_ctl of the pass's last iteration before the
        // lead thread writes it again
        __syncthreads();
        if (lead) {
            // A pass that spent cg_maxit, and the last one, are followed by no
            // residual: what has met the tolerance stays as it was before
            // them, as it does before a pass that missed its target
            const bool last = it_total >= A.maxit || outer + 1 == MAX_OUTER;
            s_ctl = S.met && (last || !(rho_final <= target * target)) ? CTL_DONE : (last ? CTL_STOP : CTL_RUN);
            if (s_ctl == CTL_DONE) rho_final = S.rho_met;
        }
        __syncthreads();
        const int stop = s_ctl;
        if (stop == CTL_DONE) { conv = true; break; }
        // x64 += correction, then a grid-wide sync before the next pass reads
        // x64 around every node
        refine_add<T, D>(A, S, bid, nbk);
        if (!grid_sync(A.bar_count, A.bar_gen, err, nbk)) return;
        if (stop == CTL_STOP) { conv = false; break; }
    }
    if (refine) {
        for (long long n = t0; n < N; n += st)
#pragma unroll
            for (int d = 0; d < D; d++) A.u[d][n] = (T)A.x64[d][n];
    }
    if (bid == 0 && lead) {
        for (int vv = 0; vv < NV; vv++) A.sc->E[vv] = refine ? E64[vv] : XE[vv];
        A.sc->iters = it_total;
        A.sc->bnorm = bnorm;
        A.sc->relres = bnorm > 0.0 ? sqrt(rho_final) / bnorm : 0.0;
        if (!conv) atomicMax(err, 4);
        A.dg->cg_last = it_total;
        if (it_total > A.dg->cg_max) A.dg->cg_max = it_total;
        A.dg->cg_total += it_total;
    }
}


// Host side of one translation unit's PCG instantiations: occupancy query,
// cooperative launch and the upload of that unit's copy of the element
// tables (constant memory is per unit).  Dynamic shared memory: with MG, the
// arrays of the block-run levels (the bound for any hierarchy, so one
// attribute serves all), which the FP64 set-up sweep uses as scratch before
// them, and the operation record of the marching sweeps.
template <typename T, int D>
size_t pcg_dyn_smem(int shape, bool mg)
{
    if (D == 2 && mg) {
        // the block-run levels' arrays (or, before them in each pass, the
        // set-up sweep's FP64 scratch), then the sweeps' operation record
        return shape == 1 ? mg_march_offset<T, Tile<2, 1>::X, Tile<2, 1>::Y>() + M2_OP_BYTES
                          : mg_march_offset<T, Tile<2, 0>::X, Tile<2, 0>::Y>() + M2_OP_BYTES;
    }
    if (D == 3 && (mg || sizeof(T) == 4)) {
        // the FP64 V-cycle's sweeps (mg_sweep3z), or the set-up sweep's (FP64
        // or double-single, three raw streams)
        const size_t cells = sizeof(T) == 4 ? 0 : sizeof(T) * (size_t)mg_sweep3z_words<T>();
        const size_t stp = sizeof(double) * (size_t)mg_sweep3z_words<double, true>(3);
        static_assert(sizeof(DS) == sizeof(double) && V3S<DS>::WORDS == V3S<double>::WORDS,
                      "the double-single set-up sweep fits the FP64 one's shared memory");
        return cells > stp ? cells : stp;
    }
    return 0;
}

// the kernel variant of a tile shape, with or without the multigrid
// preconditioner (3D FP32 marches warps and has one)
template <typename T, int D>
const void *pcg_kernel(int shape, bool mg)
{
    if constexpr (D == 3 && sizeof(T) == 4)
        return mg ? (const void *)k_pcg<T, D, 0, true> : (const void *)k_pcg<T, D, 0, false>;
    else if (mg)
        return shape == 1 ? (const void *)k_pcg<T, D, 1, true> : (const void *)k_pcg<T, D, 0, true>;
    else
        return shape == 1 ? (const void *)k_pcg<T, D, 1, false> : (const void *)k_pcg<T, D, 0, false>;
}

template <typename T, int D>
cudaError_t pcg_occupancy_t(int shape, bool mg, int block, int *per_sm)
{
    const void *fn = pcg_kernel<T, D>(shape, mg);
    const size_t dyn = pcg_dyn_smem<T, D>(shape, mg);
    if (dyn) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        if (e != cudaSuccess) return e;
    }
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, fn, block, dyn);
}

template <typename T, int D>
cudaError_t pcg_launch_t(int shape, bool mg, const void *jobs, int njobs, int grid, int block, cudaStream_t s)
{
    const PCGArgs<T, D> *pj = (const PCGArgs<T, D> *)jobs;
    void *args[] = {(void *)&pj, (void *)&njobs};
    return cudaLaunchCooperativeKernel(pcg_kernel<T, D>(shape, mg), dim3(grid), dim3(block), args,
                                       pcg_dyn_smem<T, D>(shape, mg), s);
}

} // namespace pfdev
