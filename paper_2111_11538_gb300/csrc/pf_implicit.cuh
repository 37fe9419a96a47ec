// Backward-Euler step of the field relations (Sec. 2.4, closing paragraph:
// the relations are integrated in time by backward Euler and each step is
// solved by Newton's method): device kernels of the Jacobian-free
// Newton-Krylov solve that pf_lib.cu drives.
//
// The unknown of one step is y = (theta, x_O, x_H, x_H2O) at the new time
// level, stored as four blocks of N cells.  Its equations are
//   F(y) = y - y_n - dt R(y)                       (free rows),
//   F(y) = x_H - x_H,bc and x_H2O - 0              (supply cells: held values),
// with R the right-hand sides of the explicit update (the same fluxes, the
// same driving force, the same reaction; the coupling scalars tr eps_e and
// |dev eps_e|^2 of the mechanics solved at y_n, held over the step).
// Jacobian-vector products are exact (up to rounding): a Newton step's
// pointwise derivatives are taken once in forward mode and stored, and each
// product is the linearised stencil with them; the linear solves are restarted GMRES
// preconditioned by a fixed Chebyshev polynomial of each field's own
// diffusion block (see k_be_pc_*), in FP64 or FP32 (k_be_pc32_*); FP64
// everywhere else.
#pragma once

namespace pfdev {

struct BEArgs {
    int nx, ny, nz;
    long long N;
    double dt;
    CellConst<double> K;                 // model constants (dt unused: see dt above)
    const double *phig, *mob, *trE, *devE2;
    const unsigned char *mask;
};

template <int D>
__device__ __forceinline__ void be_neighbours(const BEArgs &a, long long c, long long (&nb)[2 * D])
{
    const int i = (int)(c % a.nx);
    const long long r = c / a.nx;
    const int j = (int)(r % a.ny);
    const int k = D == 3 ? (int)(r / a.ny) : 0;
    const long long base = c - i, pl = (long long)a.nx * a.ny;
    nb[0] = base + (i == 0 ? a.nx - 1 : i - 1);
    nb[1] = base + (i == a.nx - 1 ? 0 : i + 1);
    nb[2] = c + (long long)a.nx * ((j == 0 ? a.ny - 1 : j - 1) - j);
    nb[3] = c + (long long)a.nx * ((j == a.ny - 1 ? 0 : j + 1) - j);
    if constexpr (D == 3) {
        nb[4] = c + pl * ((k == 0 ? a.nz - 1 : k - 1) - k);
        nb[5] = c + pl * ((k == a.nz - 1 ? 0 : k + 1) - k);
    }
}

// Forward-mode derivative (value, directional derivative): the pointwise
// parts of R are evaluated in it, so that J z is exact (up to rounding)
// rather than a difference quotient, whose rounding error grows with the
// stiffness of dt R.
struct Dual {
    double v, d;
    __device__ __forceinline__ Dual() {}
    __device__ __forceinline__ Dual(double a) : v(a), d(0.0) {}
    __device__ __forceinline__ Dual(double a, double b) : v(a), d(b) {}
};
__device__ __forceinline__ Dual operator+(Dual a, Dual b) { return Dual(a.v + b.v, a.d + b.d); }
__device__ __forceinline__ Dual operator-(Dual a, Dual b) { return Dual(a.v - b.v, a.d - b.d); }
__device__ __forceinline__ Dual operator-(Dual a) { return Dual(-a.v, -a.d); }
__device__ __forceinline__ Dual operator*(Dual a, Dual b) { return Dual(a.v * b.v, a.d * b.v + a.v * b.d); }
__device__ __forceinline__ Dual operator/(Dual a, Dual b)
{
    const double q = a.v / b.v;
    return Dual(q, (a.d - q * b.d) / b.v);
}
__device__ __forceinline__ Dual &operator+=(Dual &a, Dual b) { a = a + b; return a; }
__device__ __forceinline__ bool be_nonzero(double a) { return a != 0.0; }
__device__ __forceinline__ bool be_nonzero(Dual a) { return a.v != 0.0; }

// The pointwise part of cell c's derived fields: m = c sum_a W_a f_a'(x_O)
// and M_O = D_O / (c sum_a W_a f_a'') at (theta, x_O) = (th, x).
template <typename S>
__device__ __forceinline__ void be_point_cell(const BEArgs &a, long long c, S th, S x, S &m, S &M, S &Wg)
{
    const CellConst<double> &K = a.K;
    S Wf, Ww;
    phase_weights<S>(th, S(a.phig[c]), Wf, Ww, Wg);
    const S m1 = Wf * f_fe1(x) + Ww * f_wu1(x) + Wg * f_ga1(x);
    const S m2 = Wf * f_fe2(x) + Ww * f_wu2(x) + Wg * f_ga2(x);
    m = S(K.c) * m1;
    const S DO = (S(1.0) - Wg) * S(K.DOs) + Wg * S(K.DOg);
    const S den = S(K.c) * m2;
    M = be_nonzero(den) ? DO / den : S(0.0);
}

// The driving force of theta at (th, xo), without the gradient term.
template <typename S>
__device__ __forceinline__ S be_force_cell(const BEArgs &a, long long c, S th, S xo)
{
    const CellConst<double> &K = a.K;
    const double tE = a.trE[c], s2 = a.devE2[c];
    const double hg0 = hfun(a.phig[c]), sol = 1.0 - hg0;
    const S hpt = hder(th);
    const S Af = S(K.c) * f_fe(xo) + S(0.5 * K.Ks * tE * tE + K.Gs * s2);
    const S Aw = S(K.c) * f_wu(xo) + S(0.5 * K.Ks * tE * tE + K.Gs * s2);
    const double Kmix = sol * K.Ks + hg0 * K.Kg;
    return S(sol) * hpt * (Af - Aw) + S(K.w2) * mder(th) - S(K.eig3 * sol * Kmix * tE) * hpt;
}

// mu_O = c sum_a W_a f_a'(x_O) - kappa_O Lap x_O, M_O, D_H, D_H2O (Sec. 2.2,
// 3.2, Table 1; phase interpolation of the diffusivities) of cell c; ld(b, i)
// gives field b (theta, x_O, x_H, x_H2O) at cell i.
template <int D, class LD>
__device__ __forceinline__ void be_derive_cell(const BEArgs &a, long long c, LD &&ld, double (&out)[4])
{
    const CellConst<double> &K = a.K;
    long long nb[2 * D];
    be_neighbours<D>(a, c, nb);
    const double x = ld(1, c);
    double lap = -2.0 * D * x;
#pragma unroll
    for (int q = 0; q < 2 * D; q++) lap += ld(1, nb[q]);
    double m, Wg;
    be_point_cell<double>(a, c, ld(0, c), x, m, out[1], Wg);
    out[0] = m - K.kappa * lap;
    out[2] = (1.0 - Wg) * K.DHs + Wg * K.DHg;
    out[3] = (1.0 - Wg) * K.DWs + Wg * K.DWg;
}

// R(y) of cell c (Sec. 2.4): ld as above, ldd(b, i) the derived field b
// (mu, M, D_H, D_H2O) at cell i.
template <int D, class LD, class LDD>
__device__ __forceinline__ void be_rates_cell(const BEArgs &a, long long c, LD &&ld, LDD &&ldd, double (&R)[4])
{
    const CellConst<double> &K = a.K;
    long long nb[2 * D];
    be_neighbours<D>(a, c, nb);
    const double th = ld(0, c), xo = ld(1, c), xh = ld(2, c), xw = ld(3, c);
    const double mu0 = ldd(0, c), M0 = ldd(1, c), DH0 = ldd(2, c), DW0 = ldd(3, c);
    double lapt = 0.0, dO = 0.0, dH = 0.0, dW = 0.0;
#pragma unroll
    for (int q = 0; q < 2 * D; q++) {
        const long long n = nb[q];
        lapt += ld(0, n) - th;
        dO += 0.5 * (M0 + ldd(1, n)) * (ldd(0, n) - mu0);
        dH += 0.5 * (DH0 + ldd(2, n)) * (ld(2, n) - xh);
        dW += 0.5 * (DW0 + ldd(3, n)) * (ld(3, n) - xw);
    }
    R[0] = K.Lh * a.mob[c] * (be_force_cell<double>(a, c, th, xo) - K.eps2 * lapt);
    double rr = mfun(a.phig[c]) * K.kf * xo * xh;
    if (xw >= 1.0) rr = 0.0;
    R[1] = dO - rr;
    R[2] = dH - 2.0 * rr;
    R[3] = dW + rr;
}

// derived fields of the state y: der = (mu, M, D_H, D_H2O)
template <int D>
__global__ void k_be_derive(const BEArgs a, const double *__restrict__ y, double *__restrict__ der)
{
    const long long N = a.N;
    auto ld = [&](int b, long long i) { return y[b * N + i]; };
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        double o[4];
        be_derive_cell<D>(a, c, ld, o);
#pragma unroll
        for (int b = 0; b < 4; b++) der[b * N + c] = o[b];
    }
}

// Non-negative double as an ordered integer (atomicMax of a maximum norm).
__device__ __forceinline__ void be_atomic_max(unsigned long long *m, double v)
{
    atomicMax(m, (unsigned long long)__double_as_longlong(v));
}

// R(y) from the state y and its derived fields der.  mode 0: out = F(y)
// (y0 = y_n) and *maxabs = max |F|; mode 1: out = R(y) on every row.
template <int D>
__global__ void k_be_rates(const BEArgs a, const double *__restrict__ y, const double *__restrict__ y0,
                           const double *__restrict__ der, double *__restrict__ out, int mode,
                           unsigned long long *maxabs)
{
    const long long N = a.N;
    auto ld = [&](int b, long long i) { return y[b * N + i]; };
    auto ldd = [&](int b, long long i) { return der[b * N + i]; };
    double mx = 0.0;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        double R[4];
        be_rates_cell<D>(a, c, ld, ldd, R);
        if (mode == 1) {
#pragma unroll
            for (int b = 0; b < 4; b++) out[b * N + c] = R[b];
        } else {
            const bool held = a.mask[c] != 0;
#pragma unroll
            for (int b = 0; b < 4; b++) {
                double f;
                if (held && b == 2) f = y[2 * N + c] - a.K.xHbc;
                else if (held && b == 3) f = y[3 * N + c];
                else f = y[b * N + c] - y0[b * N + c] - a.dt * R[b];
                out[b * N + c] = f;
                mx = fmax(mx, fabs(f));
            }
        }
    }
    if (mode == 0) {
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((threadIdx.x & 31) == 0) be_atomic_max(maxabs, mx);
    }
}

// Pointwise derivatives of a Newton step's state y, for the products with
// its Jacobian: lin = (dm/dtheta, dm/dx_O, dM/dtheta, dM/dx_O, L mob times
// dforce/dtheta and dforce/dx_O, d(reaction)/dx_O, d(reaction)/dx_H), 8 N
// values.  (D_H and D_H2O follow the fixed gas fraction.)
__global__ void k_be_lin(const BEArgs a, const double *__restrict__ y, double *__restrict__ lin)
{
    const long long N = a.N;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const double th = y[c], xo = y[N + c], xh = y[2 * N + c], xw = y[3 * N + c];
        const double Lm = a.K.Lh * a.mob[c];
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const Dual t(th, q == 0 ? 1.0 : 0.0), x(xo, q == 1 ? 1.0 : 0.0);
            Dual m, M, Wg;
            be_point_cell<Dual>(a, c, t, x, m, M, Wg);
            lin[q * N + c] = m.d;
            lin[(2 + q) * N + c] = M.d;
            lin[(4 + q) * N + c] = Lm * be_force_cell<Dual>(a, c, t, x).d;
        }
        const double k = xw >= 1.0 ? 0.0 : mfun(a.phig[c]) * a.K.kf;
        lin[6 * N + c] = k * xh;
        lin[7 * N + c] = k * xo;
    }
}

// Jacobian-vector product J z = z - dt R'(y) z (free rows), z (held rows), in
// two passes: the changes of mu and M along z (dv = (dmu, dM)), then the
// linearised fluxes and sources.  FP64 issue bounds both (GB300 takes 64
// cycles per warp instruction): ~100 operations per cell against the ~1000 of
// evaluating R in forward mode for every product.  256^2: 60.5 us -> 17 us.
template <int D>
__global__ void k_be_jpoint(const BEArgs a, const double *__restrict__ lin, const double *__restrict__ z,
                            double *__restrict__ dv)
{
    const long long N = a.N;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        long long nb[2 * D];
        be_neighbours<D>(a, c, nb);
        const double zt = z[c], zx = z[N + c];
        double lap = -2.0 * D * zx;
#pragma unroll
        for (int q = 0; q < 2 * D; q++) lap += z[N + nb[q]];
        dv[c] = fma(lin[c], zt, fma(lin[N + c], zx, -a.K.kappa * lap));
        dv[N + c] = fma(lin[2 * N + c], zt, lin[3 * N + c] * zx);
    }
}

template <int D>
__global__ void k_be_jvp(const BEArgs a, const double *__restrict__ der, const double *__restrict__ lin,
                         const double *__restrict__ z, const double *__restrict__ dv, double *__restrict__ out)
{
    const long long N = a.N;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        long long nb[2 * D];
        be_neighbours<D>(a, c, nb);
        const double zt = z[c], zx = z[N + c], zh = z[2 * N + c], zw = z[3 * N + c];
        const double mu0 = der[c], M0 = der[N + c], DH0 = der[2 * N + c], DW0 = der[3 * N + c];
        const double dmu0 = dv[c], dM0 = dv[N + c];
        double lapt = -2.0 * D * zt, fo = 0.0, fh = 0.0, fw = 0.0;     // f: twice the flux sums
#pragma unroll
        for (int q = 0; q < 2 * D; q++) {
            const long long n = nb[q];
            lapt += z[n];
            fo = fma(dM0 + dv[N + n], der[n] - mu0, fo);
            fo = fma(M0 + der[N + n], dv[n] - dmu0, fo);
            fh = fma(DH0 + der[2 * N + n], z[2 * N + n] - zh, fh);
            fw = fma(DW0 + der[3 * N + n], z[3 * N + n] - zw, fw);
        }
        const double r0 = fma(lin[4 * N + c], zt, fma(lin[5 * N + c], zx, -a.K.Lh * a.mob[c] * a.K.eps2 * lapt));
        const double rr = fma(lin[6 * N + c], zx, lin[7 * N + c] * zh);
        const bool held = a.mask[c] != 0;
        out[c] = zt - a.dt * r0;
        out[N + c] = zx - a.dt * fma(0.5, fo, -rr);
        out[2 * N + c] = held ? zh : zh - a.dt * fma(0.5, fh, -2.0 * rr);
        out[3 * N + c] = held ? zw : zw - a.dt * fma(0.5, fw, rr);
    }
}

// y = y_n with the held values on supply cells (the Newton start).
__global__ void k_be_init(const BEArgs a, const double *__restrict__ y0, double *__restrict__ y)
{
    const long long N = a.N;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const bool held = a.mask[c] != 0;
        y[c] = y0[c];
        y[N + c] = y0[N + c];
        y[2 * N + c] = held ? a.K.xHbc : y0[2 * N + c];
        y[3 * N + c] = held ? 0.0 : y0[3 * N + c];
    }
}

// ---------------------------------------------------------------------------
// Preconditioner: per field the diffusion block of I - dt dR/dy,
//   theta: d + dt L eps mob_c sum_n (d_c - d_n)      (the gradient term),
//   x_i:   d + dt sum_n (D_c + D_n) / 2 (d_c - d_n)   (O with D_O, H, H2O),
// identity on held rows, and K Chebyshev steps on it with Jacobi scaling
// from z = 0, on the interval [1 - s, 1 + s], s = max over rows of
// (offdiagonal sum) / diagonal, which contains the spectrum of the scaled
// block (Gershgorin; the theta block is similar to a symmetric matrix).
// ---------------------------------------------------------------------------
// per-row diagonal of the four blocks, and max over rows of s per block
template <int D>
__global__ void k_be_pc_diag(const BEArgs a, const double *__restrict__ der, double *__restrict__ dg,
                             unsigned long long *smax)
{
    const long long N = a.N;
    const double cth = -a.dt * a.K.Lh * a.K.eps2;       // dt L eps
    double m[4] = {0.0, 0.0, 0.0, 0.0};
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        long long nb[2 * D];
        be_neighbours<D>(a, c, nb);
        const bool held = a.mask[c] != 0;
        double s[4];
        s[0] = 2.0 * D * cth * a.mob[c];
        const double DOc = (1.0 - hfun(a.phig[c])) * a.K.DOs + hfun(a.phig[c]) * a.K.DOg;
        double so = 0.0, sh = 0.0, sw = 0.0;
#pragma unroll
        for (int q = 0; q < 2 * D; q++) {
            const long long n = nb[q];
            const double hn = hfun(a.phig[n]);
            so += 0.5 * (DOc + (1.0 - hn) * a.K.DOs + hn * a.K.DOg);
            sh += 0.5 * (der[2 * N + c] + der[2 * N + n]);
            sw += 0.5 * (der[3 * N + c] + der[3 * N + n]);
        }
        s[1] = a.dt * so;
        s[2] = held ? 0.0 : a.dt * sh;
        s[3] = held ? 0.0 : a.dt * sw;
#pragma unroll
        for (int b = 0; b < 4; b++) {
            dg[b * N + c] = 1.0 + s[b];
            m[b] = fmax(m[b], s[b] / (1.0 + s[b]));
        }
    }
#pragma unroll
    for (int b = 0; b < 4; b++) {
        for (int o = 16; o > 0; o >>= 1) m[b] = fmax(m[b], __shfl_xor_sync(0xffffffffu, m[b], o));
        if ((threadIdx.x & 31) == 0) be_atomic_max(smax + b, m[b]);
    }
}

// q = A d for the four blocks (A as above)
template <int D>
__global__ void k_be_pc_apply(const BEArgs a, const double *__restrict__ der, const double *__restrict__ d,
                              double *__restrict__ q)
{
    const long long N = a.N;
    const double cth = -a.dt * a.K.Lh * a.K.eps2;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        long long nb[2 * D];
        be_neighbours<D>(a, c, nb);
        const bool held = a.mask[c] != 0;
        const double hc = hfun(a.phig[c]);
        const double DOc = (1.0 - hc) * a.K.DOs + hc * a.K.DOg;
        double lt = 0.0, fo = 0.0, fh = 0.0, fw = 0.0;
#pragma unroll
        for (int k = 0; k < 2 * D; k++) {
            const long long n = nb[k];
            const double hn = hfun(a.phig[n]);
            lt += d[c] - d[n];
            fo += 0.5 * (DOc + (1.0 - hn) * a.K.DOs + hn * a.K.DOg) * (d[N + c] - d[N + n]);
            fh += 0.5 * (der[2 * N + c] + der[2 * N + n]) * (d[2 * N + c] - d[2 * N + n]);
            fw += 0.5 * (der[3 * N + c] + der[3 * N + n]) * (d[3 * N + c] - d[3 * N + n]);
        }
        q[c] = d[c] + cth * a.mob[c] * lt;
        q[N + c] = d[N + c] + a.dt * fo;
        q[2 * N + c] = held ? d[2 * N + c] : d[2 * N + c] + a.dt * fh;
        q[3 * N + c] = held ? d[3 * N + c] : d[3 * N + c] + a.dt * fw;
    }
}

struct BECheb {
    double c1[4], c2[4];   // d = c1 d + c2 D^-1 r, per block
};

// z = 0, r = v, d = D^-1 r / theta_b  (c2 carries 1 / theta_b)
__global__ void k_be_pc_init(long long N, const double *__restrict__ v, const double *__restrict__ dg,
                             double *__restrict__ z, double *__restrict__ r, double *__restrict__ d, BECheb cf)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < 4 * N; i += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(i / N);
        z[i] = 0.0;
        r[i] = v[i];
        d[i] = cf.c2[b] * v[i] / dg[i];
    }
}

// one Chebyshev step after q = A d: z += d, r -= q, d = c1 d + c2 D^-1 r;
// last: z += d only
__global__ void k_be_pc_step(long long N, const double *__restrict__ q, const double *__restrict__ dg,
                             double *__restrict__ z, double *__restrict__ r, double *__restrict__ d, BECheb cf,
                             int last)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < 4 * N; i += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(i / N);
        const double dd = d[i];
        z[i] += dd;
        if (!last) {
            const double rr = r[i] - q[i];
            r[i] = rr;
            d[i] = cf.c1[b] * dd + cf.c2[b] * rr / dg[i];
        }
    }
}

// ---------------------------------------------------------------------------
// The same preconditioner in FP32 (pf_implicit_opts.pc_precision =
// PF_MIXED; GB300 runs FP32 at 64 times its FP64 rate): the blocks'
// coefficients packed once per Newton step, one fused kernel per Chebyshev
// step (the stencil reads the previous direction and writes the next, so no
// q pass), the result handed back in FP64.  The Krylov vectors, the
// Jacobian-vector products and the Newton residual stay FP64; only the
// preconditioner, an approximate inverse by construction, rounds to FP32.
// ---------------------------------------------------------------------------
struct BEPc32 {
    float *cth;        // N: the theta block's dt L eps mob_c (with its sign)
    float *DO, *DH, *DW;   // N: the diffusivities of the three species blocks
    float *dginv;      // 4N: inverse diagonals
    float *z, *r, *d0, *d1, *r1;   // 4N each: iterate, residual (r1: ping-pong, 2D), directions (ping-pong)
};
struct BECheb32 {
    float c1[4], c2[4];
};

__device__ __forceinline__ void be_neighbours32(int nx, int ny, int nz, int c, int (&nb)[6])
{
    const int i = c % nx, r = c / nx;
    const int j = r % ny, k = r / ny;
    const int base = c - i, pl = nx * ny;
    nb[0] = base + (i == 0 ? nx - 1 : i - 1);
    nb[1] = base + (i == nx - 1 ? 0 : i + 1);
    nb[2] = c + nx * ((j == 0 ? ny - 1 : j - 1) - j);
    nb[3] = c + nx * ((j == ny - 1 ? 0 : j + 1) - j);
    nb[4] = c + pl * ((k == 0 ? nz - 1 : k - 1) - k);
    nb[5] = c + pl * ((k == nz - 1 ? 0 : k + 1) - k);
}

// the FP32 coefficients of the four blocks (after k_be_pc_diag)
__global__ void k_be_pc32_pack(const BEArgs a, const double *__restrict__ der, const double *__restrict__ dg,
                               BEPc32 P)
{
    const int N = (int)a.N;
    const double cth = -a.dt * a.K.Lh * a.K.eps2;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        const double hc = hfun(a.phig[c]);
        P.cth[c] = (float)(cth * a.mob[c]);
        P.DO[c] = (float)((1.0 - hc) * a.K.DOs + hc * a.K.DOg);
        P.DH[c] = (float)der[2 * (size_t)N + c];
        P.DW[c] = (float)der[3 * (size_t)N + c];
#pragma unroll
        for (int b = 0; b < 4; b++) P.dginv[(size_t)b * N + c] = (float)(1.0 / dg[(size_t)b * N + c]);
    }
}

// z = 0, r = v, d0 = c2 D^-1 r
__global__ void k_be_pc32_init(int N, const double *__restrict__ v, BEPc32 P, BECheb32 cf)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x)
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const size_t i = (size_t)b * N + c;
            const float rv = (float)v[i];
            P.z[i] = 0.0f;
            P.r[i] = rv;
            P.d0[i] = cf.c2[b] * rv * P.dginv[i];
        }
}

// one Chebyshev step in 3D: q = A din at cell c, then z += din, r -= q,
// dout = c1 din + c2 D^-1 r (2D: k_be_pc32_tile)
__global__ void k_be_pc32_step(int nx, int ny, int nz, int N, float dt, const unsigned char *__restrict__ mask,
                               BEPc32 P, const float *__restrict__ din, float *__restrict__ dout, BECheb32 cf)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
        int nb[6];
        be_neighbours32(nx, ny, nz, c, nb);
        const float d0c = din[c], d1c = din[N + c], d2c = din[2 * N + c], d3c = din[3 * N + c];
        const float DOc = P.DO[c], DHc = P.DH[c], DWc = P.DW[c];
        float lt = 0.0f, fo = 0.0f, fh = 0.0f, fw = 0.0f;
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const int n = nb[k];
            lt += d0c - din[n];
            fo += 0.5f * (DOc + P.DO[n]) * (d1c - din[N + n]);
            fh += 0.5f * (DHc + P.DH[n]) * (d2c - din[2 * N + n]);
            fw += 0.5f * (DWc + P.DW[n]) * (d3c - din[3 * N + n]);
        }
        const bool held = mask[c] != 0;
        float q[4], dc[4] = {d0c, d1c, d2c, d3c};
        q[0] = d0c + P.cth[c] * lt;
        q[1] = d1c + dt * fo;
        q[2] = held ? d2c : d2c + dt * fh;
        q[3] = held ? d3c : d3c + dt * fw;
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const size_t i = (size_t)b * N + c;
            P.z[i] += dc[b];
            const float rr = P.r[i] - q[b];
            P.r[i] = rr;
            dout[i] = cf.c1[b] * dc[b] + cf.c2[b] * rr * P.dginv[i];
        }
    }
}

// the last step (z += din) into the FP64 result
__global__ void k_be_pc32_final(int N, BEPc32 P, const float *__restrict__ din, double *__restrict__ zo)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x)
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const size_t i = (size_t)b * N + c;
            zo[i] = (double)(P.z[i] + din[i]);
        }
}

// The FP32 preconditioner in 2D, several Chebyshev steps per launch.  A step
// alone moves its 100 bytes per cell through L2 and costs a launch (256^2:
// 4.9 us + the gap, 31 steps).  Here a block keeps a 32x32 window of all four
// fields in registers (lane = column, warp = two rows) and takes nsteps <= H
// steps on it, each spoiling one more ring of cells, so that the
// (32 - 2H)^2 cells inside are the ones it owns; a step costs it one block
// barrier, x neighbours by shuffle and y neighbours through shared memory.
// Redundant cells (32^2 / (32 - 2H)^2) are FP32 work, which is cheap here.
// Windows wrap around the grid, of any size (a window wider than the grid
// holds periodic images).
//   first: r = f v (f: *vf, 1 if null), its owned cells written to vout (the
//   normalised Krylov vector, not v itself), z = 0, d = c2 D^-1 r;  else r, d
//   from rin, din and z from P.z.
//   last: zo = z + d after the steps, else r, d, z are stored for the next.
constexpr int BE_TILE = 32, BE_TILE_MAXH = 8;
struct BECheb32Set {
    BECheb32 k[BE_TILE_MAXH];
};
__global__ void __launch_bounds__(512, 1)
k_be_pc32_tile(int nx, int ny, int N, float dt, const unsigned char *__restrict__ mask, BEPc32 P, int H, int nsteps,
               BECheb32Set cs, const double *__restrict__ v, const double *__restrict__ vf, double *__restrict__ vout, BECheb32 cinit,
               const float *__restrict__ rin, const float *__restrict__ din, float *__restrict__ rout,
               float *__restrict__ dout, double *__restrict__ zo, int first, int last)
{
    __shared__ float sd[2][4][BE_TILE][BE_TILE];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int own = BE_TILE - 2 * H, ntx = (nx + own - 1) / own;
    const int ox = (int)(blockIdx.x % ntx) * own - H, oy = (int)(blockIdx.x / ntx) * own - H;
    auto modp = [](int a, int n) { a %= n; return a < 0 ? a + n : a; };
    const int gx = modp(ox + lane, nx);
    float r[2][4], d[2][4], z[2][4], dg[2][4], cth[2], hf[2], wx[2][3], wl[2][3], wy[3][3];
    size_t gi[2];
    bool mine[2];
    // face weights (D_c + D_n) / 2: right faces, left ones by shuffle, the
    // three y faces of the two rows
    {
        const float *const Ds[3] = {P.DO, P.DH, P.DW};
        const int gr = modp(gx + 1, nx);
        float D[4][3];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int gy = modp(oy + 2 * wid - 1 + q, ny);
#pragma unroll
            for (int f = 0; f < 3; f++) {
                D[q][f] = Ds[f][gx + (size_t)nx * gy];
                if (q == 1 || q == 2) wx[q - 1][f] = 0.5f * (D[q][f] + Ds[f][gr + (size_t)nx * gy]);
            }
        }
#pragma unroll
        for (int f = 0; f < 3; f++) {
#pragma unroll
            for (int q = 0; q < 3; q++) wy[q][f] = 0.5f * (D[q][f] + D[q + 1][f]);
#pragma unroll
            for (int q = 0; q < 2; q++) wl[q][f] = __shfl_up_sync(0xffffffffu, wx[q][f], 1);
        }
    }
    const double f = first && vf ? *vf : 1.0;
#pragma unroll
    for (int q = 0; q < 2; q++) {
        const int ey = 2 * wid + q, gy = modp(oy + ey, ny);
        gi[q] = gx + (size_t)nx * gy;
        mine[q] = lane >= H && lane < BE_TILE - H && ey >= H && ey < BE_TILE - H && ox + lane < nx && oy + ey < ny;
        cth[q] = P.cth[gi[q]];
        hf[q] = mask[gi[q]] ? 0.f : dt;
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const size_t i = (size_t)b * N + gi[q];
            dg[q][b] = P.dginv[i];
            if (first) {
                const double vv = v[i] * f;
                if (mine[q] && vout) vout[i] = vv;
                r[q][b] = (float)vv;
                z[q][b] = 0.f;
                d[q][b] = cinit.c2[b] * r[q][b] * dg[q][b];
            } else {
                r[q][b] = rin[i];
                d[q][b] = din[i];
                z[q][b] = mine[q] ? P.z[i] : 0.f;
            }
        }
    }
    for (int k = 0; k < nsteps; k++) {
        float (*sb)[BE_TILE][BE_TILE] = sd[k & 1];
#pragma unroll
        for (int q = 0; q < 2; q++)
#pragma unroll
            for (int b = 0; b < 4; b++) sb[b][2 * wid + q][lane] = d[q][b];
        __syncthreads();
        const int up = wid == 0 ? 0 : 2 * wid - 1, dn = wid == 15 ? BE_TILE - 1 : 2 * wid + 2;   // the outermost rows are spoilt anyway
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const float dc[2] = {d[0][b], d[1][b]}, du = sb[b][up][lane], dd = sb[b][dn][lane];
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const float l = __shfl_up_sync(0xffffffffu, dc[q], 1), rr_ = __shfl_down_sync(0xffffffffu, dc[q], 1);
                const float u = q == 0 ? du : dc[0], w = q == 0 ? dc[1] : dd, c = dc[q];
                float a;
                if (b == 0) {
                    a = fmaf(cth[q], (c - l) + (c - rr_) + (c - u) + (c - w), c);
                } else {
                    const float f = fmaf(wl[q][b - 1], c - l, fmaf(wx[q][b - 1], c - rr_,
                                    fmaf(wy[q][b - 1], c - u, wy[q + 1][b - 1] * (c - w))));
                    a = fmaf(b == 1 ? dt : hf[q], f, c);
                }
                z[q][b] += c;
                r[q][b] -= a;
                d[q][b] = fmaf(cs.k[k].c1[b], c, cs.k[k].c2[b] * r[q][b] * dg[q][b]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 2; q++)
        if (mine[q])
#pragma unroll
            for (int b = 0; b < 4; b++) {
                const size_t i = (size_t)b * N + gi[q];
                if (last) {
                    zo[i] = (double)(z[q][b] + d[q][b]);
                } else {
                    P.z[i] = z[q][b];
                    rout[i] = r[q][b];
                    dout[i] = d[q][b];
                }
            }
}

// ---------------------------------------------------------------------------
// Vector kernels of the Krylov solve (length L = 4N).
// ---------------------------------------------------------------------------
// Classical Gram-Schmidt, one launch per pass: every block owns `per`
// consecutive elements, which it works on in pieces of BE_CH held in shared
// memory; the last block to finish adds the blocks' partial sums in block
// order and leaves them in out.  FP64 issue bounds it: 1 or 2 instructions
// per element and vector.
//   GS 0: out[k] = V_k . w;
//   GS 1: w -= sum_k cin[k] V_k, out[k] = V_k . w (the second pass's
//         coefficients, on the piece just formed);
//   GS 2: w -= sum_k cin[k] V_k, out[0] = w . w, out[1] = 1 / |w| (1 if w = 0).
// The vectors stream from L2 and beyond (60 of 2.1 MB), so that what counts
// is the loads in flight: 16 bytes per lane, eight vectors (the update) or
// seven pieces (the products) at a time, 32 warps per SM.
// 256^2, restarts of 60, per iteration: three dot products of 24 us, two
// combinations of 15 us, three device-to-host copies with their waits and a
// scaling before; 26 + 41 + 22 us now at 40 vectors (8-byte loads and
// 16 warps per SM: 38 + 47 + 24).
constexpr int BE_CH = 1024, BE_GST = 512;
template <int GS>
__global__ void __launch_bounds__(BE_GST, 2) k_be_gs(long long L, long long per, const double *__restrict__ V, int nv,
                                                     double *w, const double *__restrict__ cin, double *part,
                                                     unsigned int *ticket, double *out)
{
    __shared__ __align__(16) double sw[BE_CH];
    __shared__ double sc[64], acc[64];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, t = threadIdx.x;
    constexpr int NW = BE_GST / 32;
    if (t < 64) {
        acc[t] = 0.0;
        sc[t] = GS > 0 && t < nv ? cin[t] : 0.0;
    }
    __syncthreads();
    // (L and per are multiples of 4: pieces have even lengths and 16-byte
    // boundaries)
    const long long i0 = blockIdx.x * per, i1 = min(i0 + per, L);
    double n2 = 0.0;
    double2 *const sw2 = reinterpret_cast<double2 *>(sw);
    for (long long p0 = i0; p0 < i1; p0 += BE_CH) {
        const int n = (int)min((long long)BE_CH, i1 - p0) / 2;      // pairs
        double2 *const w2 = reinterpret_cast<double2 *>(w + p0);
        if (t < n) {
            double2 x = w2[t];
            if constexpr (GS > 0) {
                const double2 *v = reinterpret_cast<const double2 *>(V + p0) + t;
                double2 s = make_double2(0.0, 0.0);
#pragma unroll 8
                for (int k = 0; k < nv; k++) {
                    const double2 a = v[(size_t)k * (L / 2)];
                    s.x = fma(sc[k], a.x, s.x);
                    s.y = fma(sc[k], a.y, s.y);
                }
                x.x -= s.x;
                x.y -= s.y;
                w2[t] = x;
            }
            if constexpr (GS == 2) n2 = fma(x.x, x.x, fma(x.y, x.y, n2));
            else sw2[t] = x;
        }
        if constexpr (GS < 2) {
            __syncthreads();
            for (int k = wid; k < nv; k += NW) {
                const double2 *v = reinterpret_cast<const double2 *>(V + (size_t)k * L + p0);
                double2 s = make_double2(0.0, 0.0), r = s;
                int q = lane;
                for (; q + 32 * 6 < n; q += 32 * 7) {
                    double2 a[7];
#pragma unroll
                    for (int u = 0; u < 7; u++) a[u] = v[q + 32 * u];
#pragma unroll
                    for (int u = 0; u < 7; u++) {
                        const double2 b = sw2[q + 32 * u];
                        double2 &z = (u & 1) ? r : s;
                        z.x = fma(a[u].x, b.x, z.x);
                        z.y = fma(a[u].y, b.y, z.y);
                    }
                }
                for (; q < n; q += 32) {
                    const double2 a = v[q], b = sw2[q];
                    s.x = fma(a.x, b.x, s.x);
                    s.y = fma(a.y, b.y, s.y);
                }
                double x = (s.x + s.y) + (r.x + r.y);
                for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                if (lane == 0) acc[k] += x;
            }
            __syncthreads();
        }
    }
    if constexpr (GS == 2) {
        for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        if (lane == 0) sw[wid] = n2;
        __syncthreads();
        if (t == 0) {
            double x = 0.0;
            for (int q = 0; q < NW; q++) x += sw[q];
            acc[0] = x;
        }
        __syncthreads();
    }
    const int nk = GS == 2 ? 1 : nv;
    if (t < nk) part[(size_t)t * gridDim.x + blockIdx.x] = acc[t];
    __threadfence();
    __syncthreads();
    if (t == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int k = wid; k < nk; k += NW) {
        double x = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) x += __ldcg(part + (size_t)k * gridDim.x + b);
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) {
            out[k] = x;
            if (GS == 2) out[1] = x > 0.0 ? 1.0 / sqrt(x) : 1.0;
        }
    }
    if (t == 0) *ticket = 0u;
}

// dst = *f v
__global__ void k_be_scale(long long L, const double *__restrict__ v, const double *__restrict__ f,
                           double *__restrict__ dst)
{
    const double c = *f;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < L; i += (long long)gridDim.x * blockDim.x)
        dst[i] = c * v[i];
}

// w += sum_k c[k] V_k (c in device memory, nv <= 64)
__global__ void k_be_comb(long long L, const double *__restrict__ V, int nv, const double *__restrict__ c,
                          double *__restrict__ w)
{
    __shared__ double sc[64];
    if (threadIdx.x < nv) sc[threadIdx.x] = c[threadIdx.x];
    __syncthreads();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < L; i += (long long)gridDim.x * blockDim.x) {
        double s = w[i];
        for (int k = 0; k < nv; k++) s = fma(sc[k], V[(size_t)k * L + i], s);
        w[i] = s;
    }
}

// dst = a x + b y
__global__ void k_be_axpby(long long L, double a, const double *__restrict__ x, double b, const double *__restrict__ y,
                           double *__restrict__ dst)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < L; i += (long long)gridDim.x * blockDim.x)
        dst[i] = a * x[i] + b * y[i];
}

// Newton update y -= delta; max |delta| and max |y| (after the update)
__global__ void k_be_newton(long long L, const double *__restrict__ delta, double *__restrict__ y,
                            unsigned long long *mx)
{
    double md = 0.0, my = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < L; i += (long long)gridDim.x * blockDim.x) {
        const double v = y[i] - delta[i];
        y[i] = v;
        md = fmax(md, fabs(delta[i]));
        my = fmax(my, fabs(v));
    }
    for (int o = 16; o > 0; o >>= 1) {
        md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
        my = fmax(my, __shfl_xor_sync(0xffffffffu, my, o));
    }
    if ((threadIdx.x & 31) == 0) {
        be_atomic_max(mx, md);
        be_atomic_max(mx + 1, my);
    }
}

// ---------------------------------------------------------------------------
// Gather / scatter between the field buffers and the state vector, and the
// balances of the finished step.
// ---------------------------------------------------------------------------
__global__ void k_be_gather(long long N, const double *__restrict__ th, const double *__restrict__ xo,
                            const double *__restrict__ xh, const double *__restrict__ xw, double *__restrict__ y)
{
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        y[c] = th[c];
        y[N + c] = xo[c];
        y[2 * N + c] = xh[c];
        y[3 * N + c] = xw[c];
    }
}

// new fields from y; per-block partial sums of x_O, x_H, x_H2O, of the water
// the held cells' own relations would hold (removed) and of the hydrogen
// added to reach x_H,bc (supplied): the free relation's value is
// y_n + dt R(y) (R in rates)
__global__ void k_be_finish(const BEArgs a, const double *__restrict__ y, const double *__restrict__ y0,
                            const double *__restrict__ rates, double *__restrict__ th, double *__restrict__ xo,
                            double *__restrict__ xh, double *__restrict__ xw, double *__restrict__ part)
{
    const long long N = a.N;
    double s[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        th[c] = y[c];
        xo[c] = y[N + c];
        xh[c] = y[2 * N + c];
        xw[c] = y[3 * N + c];
        s[0] += y[N + c];
        s[1] += y[2 * N + c];
        s[2] += y[3 * N + c];
        if (a.mask[c]) {
            s[3] += y0[3 * N + c] + a.dt * rates[3 * N + c];
            s[4] += a.K.xHbc - (y0[2 * N + c] + a.dt * rates[2 * N + c]);
        }
    }
    __shared__ double sh[5][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 5; k++) {
        double v = s[k];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) sh[k][wid] = v;
    }
    __syncthreads();
    if (wid == 0) {
#pragma unroll
        for (int k = 0; k < 5; k++) {
            double v = lane < (int)(blockDim.x >> 5) ? sh[k][lane] : 0.0;
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) part[(size_t)blockIdx.x * 5 + k] = v;
        }
    }
}

// the block partials of k_be_finish into the diagnostics (one warp, fixed order)
__global__ void k_be_diag(const double *__restrict__ part, int nb, Diag *dg)
{
    const int lane = threadIdx.x;
    double t[5];
#pragma unroll
    for (int k = 0; k < 5; k++) {
        double v = 0.0;
        for (int b = lane; b < nb; b += 32) v += part[(size_t)b * 5 + k];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        t[k] = v;
    }
    if (lane == 0) {
        dg->sumO_prev = dg->sumO;
        dg->sumO = t[0];
        dg->sumH = t[1];
        dg->sumW = t[2];
        dg->removedW += t[3];
        dg->suppliedH += t[4];
        if (!isfinite(t[0] + t[1] + t[2]) && dg->status == 0) dg->status = 5;
    }
}

}  // namespace pfdev
