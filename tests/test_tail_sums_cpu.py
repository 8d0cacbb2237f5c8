"""The 32-bit sums that lay out a wave of the cluster kernel, at row lengths whose
plain sums wrap (no graph of that size is made): the arithmetic of the kernel's
header, compiled for the host."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

from paper_2402_15253_gb300 import build as libbuild

PROGRAM = r"""
#include <cstdio>
#include "pico.h"
#include "peel_tail.cuh"
using namespace pico::peel;
int main()
{
    const int rows[] = {1, 2, 3, 4, 17, 35, 512};
    int bad = 0;
    for (unsigned budget : {kTailBudget, kTailLateBudget})
    for (long long d : {1ll, 129ll, (long long)budget - 1, (long long)budget, (long long)budget + 1,
                        125000000ll, 1073741824ll, 2147483646ll})
        for (int n : rows)
            for (long long other : {1ll, 4194304ll}) {
                // n rows of d arcs and 512 - n of `other`, summed as a tile is
                long long exact = 0;
                int sum = 0;
                for (int i = 0; i < 512; ++i) {
                    const long long x = i < n ? d : other;
                    exact += x;
                    sum = (int)((unsigned)sum + (unsigned)tail_row(x, budget));
                    bad += sum < 0;
                }
                bad += ((unsigned)sum > budget) != (exact > (long long)budget);
                if (exact <= (long long)budget) bad += sum != exact;
            }
    // without a budget rows count whole, in graphs whose arcs fit 32 bits
    bad += tail_row(kTailMaxGraph, kTailNoBudget) != kTailMaxGraph;
    printf("bad %d\n", bad);
    return bad != 0;
}
"""


def test_wave_sums(tmp_path):
    nvcc = libbuild._nvcc()
    if not (os.path.exists(nvcc) or shutil.which(nvcc)):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "sums.cu", tmp_path / "sums"
    src.write_text(PROGRAM)
    flags = [f for f in libbuild.NVCC_FLAGS if not f.startswith("-O")] + ["-Xcompiler", "-O1"]
    r = subprocess.run([nvcc, *libbuild.ARCH, *flags, str(src), "-o", str(exe)], capture_output=True,
                       text=True, cwd=ROOT)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
