"""The table of time factors where its entries outnumber an int (a batch of 512 steps of more than four million instances):
every entry is formed, at its place.  The kernel is run by itself, on two instances and many steps (17 GB)."""
import subprocess

import pytest

from paper_1805_00007_gb300 import _build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#include <cstring>
#include "lbch_kernels.cuh"
using namespace lbch;
int main()
{
    const int steps = (1 << 30) + 5, n_inst = 2;
    const size_t n = (size_t)steps * n_inst;
    InstDev inst[2];
    memset(inst, 0, sizeof inst);
    inst[0].vel = VEL_REV_SHEAR;  // 1 until step 2^30, then -1
    inst[0].Tper = (double)(1 << 30);
    inst[1].vel = VEL_UNIFORM;    // 1
    Ctl ctl = {0, 0, 0};
    InstDev* d_inst;
    Ctl* d_ctl;
    double *T, got[12];
    if (cudaMalloc(&d_inst, sizeof inst) || cudaMalloc(&d_ctl, sizeof ctl) || cudaMalloc(&T, n * 8)) return 2;
    if (cudaMemcpy(d_inst, inst, sizeof inst, cudaMemcpyHostToDevice) || cudaMemcpy(d_ctl, &ctl, sizeof ctl, cudaMemcpyHostToDevice)) return 2;
    if (cudaMemset(T, 0xff, n * 8)) return 2;
    time_table_kernel<<<time_table_blocks(steps, n_inst), TIME_NT>>>(d_inst, n_inst, d_ctl, steps, T);
    if (cudaMemcpy(got, T + n - 12, sizeof got, cudaMemcpyDeviceToHost)) return 3;
    for (int k = 0; k < 12; k++) printf("%g ", got[k]);
    if (cudaMemcpy(got, T, sizeof got, cudaMemcpyDeviceToHost)) return 3;
    for (int k = 0; k < 12; k++) printf("%g ", got[k]);
    return 0;
}
"""


def test_more_entries_than_an_int_counts(tmp_path):
    src, exe = tmp_path / "table.cu", tmp_path / "table"
    src.write_text(SOURCE)
    subprocess.run([_build.nvcc(), *_build.COMPILE_FLAGS, "-I", _build.CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout
    assert [float(v) for v in out.split()] == [1, 1] + [-1, 1] * 5 + [1, 1] * 6
