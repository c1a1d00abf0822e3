"""Shared memory of the x passes, on the host: what a launch asks for holds what its kernel lays out.

The geometry is a host function of the kernels' own header; a small program compiled here walks it over line
lengths, rows per CTA and row pitches (the allocation-free step takes any pitch of its caller's).  A staged tile
lays out [16 bytes][G][sp] rows, then its states and end values; rows of chunks of 9 and 17 values are always staged
(there is no other kernel for them).
"""
import os
import shutil
import subprocess

import pytest

from paper_2604_19370_gb300 import build

PROGRAM = r"""
#include <stdio.h>
#include "wf_lines.cuh"
using namespace wf;

template <typename P, int PD, int M>
int check(int lo, int hi, int most) {
    int bad = 0;
    for (int N = lo; N <= hi; N += 1 + N / 16)
        for (int lines : {1, 9, 700})
            for (int extra : {0, 1, 5, 8, 1000, 16000, 65000, 131000, 524000})
                for (int G : {0, 1, 2, 4, 8}) {
                    LineArgs l = {};
                    l.N = N, l.M = M, l.C = line_chunks(N, M), l.J = 2, l.G = G;
                    l.nlines = lines, l.pitch = N + extra, l.narr = 2, l.b.S = 1;
                    PassArgs<P> a;
                    pass_args(l, N, a);
                    int nt = 0;
                    size_t smem = 0;
                    const char* what = nullptr;
                    if (!x_geometry<P, PD, M>(l, most, 72 * 1024, a, &nt, &smem)) what = "refused";
                    else {
                        const size_t rows = a.staged ? (size_t)a.G * a.sp : 0;
                        const size_t layout = 16 + (rows + (size_t)a.cells * PD + 4 * PD * a.G) * sizeof(P);
                        if (smem < layout || smem > 227 * 1024) what = "shared memory";
                        else if (M < 33 && !a.staged) what = "not staged";
                        else if (a.staged && (size_t)a.sp * sizeof(P) < (N * sizeof(P) + 15) / 16 * 16) what = "row stride";
                        else if (a.cells < a.C * a.G || nt > most) what = "threads";
                    }
                    if (what && bad++ < 5)
                        printf("%s: %d-byte values p %d chunk %d N %d lines %d pitch %d G %d\n", what, (int)sizeof(P), PD, M, N,
                               lines, N + extra, G);
                }
    return bad;
}

template <int PD>
int degree() {
    return check<float, PD, 9>(PD + 1, 144, 512) + check<float, PD, 17>(PD + 1, 1600, 512) +
           check<float, PD, 33>(PD + 1, 16384, 512) + check<float, PD, 33>(16385, 32768 + PD, 1024) +
           check<double, PD, 9>(PD + 1, 144, 512) + check<double, PD, 17>(PD + 1, 1088, 512) +
           check<double, PD, 33>(PD + 1, 16384, 512) + check<double, PD, 33>(16385, 32768 + PD, 1024);
}

int main() {
    const int bad = degree<1>() + degree<2>() + degree<3>();
    printf("%d\n", bad);
    return bad ? 1 : 0;
}
"""


def test_x_pass_shared_memory_covers_its_layout(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "geometry.cu", tmp_path / "geometry"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
