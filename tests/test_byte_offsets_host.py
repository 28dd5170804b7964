"""The fixed-link sweeps' byte offsets on the largest lattices they take, compiled for
the host with the undefined-behaviour sanitiser (byte_offsets_check.cu)."""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_byte_offsets_hold_up_to_the_largest_lattice(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = tmp_path / "byte_offsets_check"
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
                           "-Xcompiler", "-fsanitize=signed-integer-overflow,-fno-sanitize-recover=all",
                           "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "paper_1305_3440_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "byte_offsets_check.cu"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
