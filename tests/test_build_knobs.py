"""Tuning knobs of the symmetric kernels: a setting whose units would not hold whole Kahan groups (its
pairs would be counted twice at small N) does not compile."""
import os
import shutil
import subprocess

import pytest

from paper_2602_20787_gb300 import build


@pytest.mark.parametrize("defs,ok", [([], True), (["-DSTEPS_KAHAN_GROUP=4"], True),
                                     (["-DSTEPS_KAHAN_GROUP=16", "-DSTEPS_SYM_MAX_STEP_SPLIT=2"], True),
                                     (["-DSTEPS_KAHAN_GROUP=16"], False), (["-DSTEPS_KAHAN_GROUP=32"], False),
                                     (["-DSTEPS_SYM_MAX_STEP_SPLIT=8"], False), (["-DSTEPS_SYM_MAX_STEP_SPLIT=3"], False)])
def test_units_hold_whole_groups(tmp_path, defs, ok):
    nvcc = build._nvcc()
    if not shutil.which(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "knobs.cu"
    src.write_text('#include "pair_sym.cuh"\n')
    run = subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-c", "-o", os.devnull, "-I" + build.CSRC, "-I" + build.INCLUDE,
                          *defs, str(src)], capture_output=True, text=True)
    assert (run.returncode == 0) == ok, run.stderr
