"""Rounding of the marching sweeps' cell forces (cell2, cell3; host builds of
the device functions).  A displacement of size 1 that varies by 1e-3 between
neighbours is exact in the type, and so is every difference of neighbours up
to one rounding; every force coefficient is then a sum of at most 16 such
differences (three additions deep per axis, a product and up to three more
additions), so that its error stays below 16 eps times the moduli's sum times
the sum of the cell's neighbour differences.  A sum of displacements taken
before the difference leaves eps times the displacement, ~100 times that."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>
#include "pf_cg.cuh"
using namespace pfdev;
typedef long double LD;

template <typename T>
double two()
{
    std::mt19937 g(1);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    double worst = 0.0;
    for (int k = 0; k < 20000; k++) {
        T u[2][2][2];                     // [y][x][component]
        for (auto &y : u) for (auto &x : y) for (int c = 0; c < 2; c++) x[c] = (T)(1.0 - 2.0 * c + 1e-3 * U(g));
        const T l = (T)(1.5 + U(g)), m = (T)(1.5 + U(g));
        Row2<T> R[2];
        for (int y = 0; y < 2; y++)
            for (int c = 0; c < 2; c++) { R[y].v[c] = u[y][0][c]; R[y].d[c] = u[y][1][c] - u[y][0][c]; }
        const Cell2<T> C = cell2<T>(l, m, R[0], R[1]);
        LD gx[2], gy[2], xy[2], s = 0.0;
        for (int c = 0; c < 2; c++) {
            const LD a = u[0][0][c], b = u[0][1][c], d = u[1][0][c], e = u[1][1][c];
            gx[c] = (b - a) + (e - d);
            gy[c] = (d - a) + (e - b);
            xy[c] = (e - d) - (b - a);
            s += fabsl(b - a) + fabsl(e - d) + fabsl(d - a) + fabsl(e - b);
        }
        const LD L = l, M = m, lt = L * (gx[0] + gy[1]), ch = (L + 3 * M) / 3;
        const LD ref[5] = {lt + 2 * M * gx[0], M * (gy[0] + gx[1]), lt + 2 * M * gy[1], ch * xy[0], ch * xy[1]};
        const T got[5] = {C.ax0, C.sh, C.ay1, C.xy[0], C.xy[1]};
        for (int q = 0; q < 5; q++)
            worst = fmax(worst, (double)(fabsl(got[q] - ref[q]) / (s * (L + 2 * M))) / std::numeric_limits<T>::epsilon());
    }
    return worst;
}

double three()
{
    std::mt19937 g(2);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    double worst = 0.0;
    for (int k = 0; k < 20000; k++) {
        float u[2][2][2][3];              // [z][y][x][component]
        for (auto &z : u) for (auto &y : z) for (auto &x : y)
            for (int c = 0; c < 3; c++) x[c] = (float)(1.0 - 0.7 * c + 1e-3 * U(g));
        const float l = (float)(1.5 + U(g)), m = (float)(1.5 + U(g));
        Row3 R[2][2];
        for (int z = 0; z < 2; z++)
            for (int y = 0; y < 2; y++)
                for (int c = 0; c < 3; c++) { R[z][y].v[c] = u[z][y][0][c]; R[z][y].d[c] = u[z][y][1][c] - u[z][y][0][c]; }
        Cell3 C;
        cell3(l, m, R[0][0], R[0][1], R[1][0], R[1][1], C);
        LD G[3][3] = {}, h[3][3] = {}, h3[3] = {}, s = 0.0;    // G[axis][c]; h: xy, yz, zx
        for (int c = 0; c < 3; c++) {
            const LD lo = u[0][0][0][c];
            for (int z = 0; z < 2; z++)
                for (int y = 0; y < 2; y++)
                    for (int x = 0; x < 2; x++) {
                        const LD v = (LD)u[z][y][x][c] - lo;          // exact; the sums below have no constant part
                        const int sx = 2 * x - 1, sy = 2 * y - 1, sz = 2 * z - 1;
                        G[0][c] += sx * v; G[1][c] += sy * v; G[2][c] += sz * v;
                        h[0][c] += sx * sy * v; h[1][c] += sy * sz * v; h[2][c] += sz * sx * v;
                        h3[c] += sx * sy * sz * v;
                        s += fabsl(v);
                    }
        }
        const LD L = l, M = m, lt = L * (G[0][0] + G[1][1] + G[2][2]), l3 = L / 3, m3 = M / 3, c9 = (L + 4 * M) / 9;
        LD ref[18];
        float got[18];
        int n = 0;
        auto put = [&](LD a, float b) { ref[n] = a; got[n++] = b; };
        for (int v = 0; v < 3; v++) put(lt + 2 * M * G[v][v], C.s[v]);
        put(M * (G[2][1] + G[1][2]), C.s[3]);
        put(M * (G[2][0] + G[0][2]), C.s[4]);
        put(M * (G[1][0] + G[0][1]), C.s[5]);
        const LD *xy = h[0], *yz = h[1], *zx = h[2];
        const LD A = l3 * (xy[1] + zx[2]), B = l3 * (xy[0] + yz[2]), D = l3 * (zx[0] + yz[1]);
        const LD P = yz[0] + zx[1], Q = zx[1] + xy[2], W = xy[2] + yz[0];
        put(M * xy[0] + B, C.xy[0]); put(M * xy[1] + A, C.xy[1]); put(m3 * (Q + W), C.xy[2]);
        put(m3 * (P + W), C.yz[0]); put(M * yz[1] + D, C.yz[1]); put(M * yz[2] + B, C.yz[2]);
        put(M * zx[0] + D, C.zx[0]); put(m3 * (P + Q), C.zx[1]); put(M * zx[2] + A, C.zx[2]);
        for (int c = 0; c < 3; c++) put(c9 * h3[c], C.xyz[c]);
        for (int q = 0; q < n; q++)
            worst = fmax(worst, (double)(fabsl(got[q] - ref[q]) / (s * (L + 2 * M))) / std::numeric_limits<float>::epsilon());
    }
    return worst;
}

int main()
{
    printf("%.3f %.3f %.3f\n", two<float>(), two<double>(), three());
    return 0;
}
"""


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    d = tmp_path_factory.mktemp("rounding")
    src, exe = str(d / "r.cu"), str(d / "r")
    with open(src, "w") as fh:
        fh.write(SRC)
    subprocess.check_call(["nvcc", "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-I" + os.path.join(ROOT, "include"),
                           "-I" + os.path.join(ROOT, "paper_2111_11538_gb300", "csrc"), "-o", exe, src])
    return [float(x) for x in subprocess.check_output([exe], text=True).split()]


def test_cell_forces_take_differences_first(errors):
    assert max(errors) <= 16.0, errors
