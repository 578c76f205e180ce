"""The kernel variants of the spectral solve (csrc/spectral_f*.cu instantiate
the templates of spectral_dev.cuh) compile for sm_103a, where nvcc is present:
every variant that the host side chooses from is an entry of the compiler's
report."""
import glob
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1712_08494_gb300", "csrc")


def test_kernel_variants_compile_for_sm103a(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    units = sorted(glob.glob(os.path.join(CSRC, "spectral_f*.cu")))
    wanted = {}  # kernel arguments named in each unit
    for u in units:
        wanted[u] = set(re.findall(r"k_spectral<([^>]*)>", open(u).read()))
    assert sum(len(w) for w in wanted.values()) == 6  # FP32, FP32 big, FP64, each with and without mixed lengths
    # the assembler without optimisation: its report lists the kernels, and the translation is what is tested
    runs = {u: subprocess.Popen([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                                 "--expt-relaxed-constexpr", "-Xptxas", "-O0,-v", "-I", CSRC, "-c", u, "-o",
                                 str(tmp_path / (os.path.basename(u) + ".o"))],
                                stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True) for u in units}
    for u, r in runs.items():
        log = r.communicate()[0]
        assert r.returncode == 0, log[-4000:]
        kernels = {k for k in re.findall(r"Compiling entry function '(\S+)'", log) if "k_spectral" in k}
        assert len(kernels) == len(wanted[u]), (u, kernels)
