"""Rounding of the FP64 2D marching sweeps' cell forces (cell2, a host build of
the device function).  A displacement of size 1 that varies by 1e-3 between
neighbours is exact in the type, and so is every difference of neighbours up
to one rounding; every force coefficient is then a sum of a few such
differences times moduli (fewer than 16 roundings in all), so that its error
stays below 16 eps times the moduli's sum times the sum of the cell's
neighbour differences.  A sum of displacements taken
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

int main()
{
    printf("%.3f\n", two<double>());
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
