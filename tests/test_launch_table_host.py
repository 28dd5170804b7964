"""The launch configurations with kernels, format by format and gauge by gauge, are
those of the table in lgt.h (launch_table_check.cu, compiled for the host)."""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_supported_configurations_are_the_documented_ones(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = tmp_path / "launch_table_check"
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
                           "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "paper_1305_3440_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"),
                           os.path.join(ROOT, "tests", "launch_table_check.cu"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr


def test_no_sweep_kernel_is_compiled_that_no_dispatch_reaches():
    """FP64 and FP32-pair sweep kernels exist in their configurations and in no other
    (an early return under `if constexpr` discards nothing after it)."""
    import re
    from paper_1305_3440_gb300 import build
    names = subprocess.run(["nm", "-C", build.build()], capture_output=True, text=True, check=True).stdout
    for kernel, want in (("k_sweep_f64", {0, 1, 2, 3, 16}), ("k_sweep_pair", {0, 1, 2, 3})):
        assert {int(c) for c in re.findall(kernel + r"<\d+, \d+, (\d+)>", names)} == want, kernel
