"""Shared memory of the FP64 quadrature, on the host: no SM takes more of its CTAs than an even spread gives it.

An SM has 228 KB, of which a CTA takes what it asks for and 1 KB for the system, and a CTA may ask for 227 KB.
"""
import os
import shutil
import subprocess

import pytest

from paper_2604_19370_gb300 import build

PROGRAM = r"""
#include <stdio.h>
#include "wf_quad.cuh"

int main() {
    int bad = 0;
    for (size_t need : {20000, 37000, 69000, 90000, 117000})
        for (int sms : {132, 148, 152})
            for (long ctas = 1; ctas < 3000; ++ctas) {
                const size_t smem = wf::even_smem(need, ctas, sms);
                const size_t fit = (ctas + sms - 1) / sms, held = 228 * 1024 / (smem + 1024);
                // as many as before where those were not too many, else as many as the even spread
                const size_t want = 228 * 1024 / (need + 1024) < fit ? 228 * 1024 / (need + 1024) : fit;
                if (smem < need || smem > 227 * 1024 || held != want)
                    if (bad++ < 5) printf("need %zu ctas %ld sms %d: %zu, %zu held, %zu wanted\n", need, ctas, sms, smem, held, want);
            }
    printf("%d\n", bad);
    return bad ? 1 : 0;
}
"""


def test_even_spread(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "even.cu", tmp_path / "even"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
