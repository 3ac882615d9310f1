"""The build-time choices of the FP32 row compile: two cells per lane instead of four
(-DKSS_F32_VEC=2, every storage with FP32 arithmetic and the runtimes that launch it) and the
scalar row (-DKSS_ROW_PAIRED=0).  nvcc cross-compiles sm_103a without a GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2603_13618_gb300 import build


@pytest.mark.parametrize("macro,srcs", [
    ("-DKSS_F32_VEC=2", ["launch_f32.cu", "launch_f16.cu", "kss_runtime.cu", "kss_adjoint.cu"]),
    ("-DKSS_ROW_PAIRED=0", ["launch_f32.cu", "kss_runtime.cu"])])
def test_row_choices_compile(macro, srcs, tmp_path):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no nvcc")
    procs = [subprocess.Popen([build.nvcc(), *build.flags([macro]), "-c",
                               os.path.join(build.CSRC, s), "-o", str(tmp_path / (s + ".o"))],
                              stdout=subprocess.PIPE, stderr=subprocess.PIPE, text=True)
             for s in srcs]
    for s, p in zip(srcs, procs):
        out, err = p.communicate(timeout=600)
        assert p.returncode == 0, f"{s} {macro}:\n{out}\n{err}"
