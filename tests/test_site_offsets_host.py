"""The fixed-link sweeps' neighbour offsets and reciprocal divisions, compiled for
the host and compared with the general index functions (site_offsets_check.cu)."""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_site_offsets_match_the_general_index_functions(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = tmp_path / "site_offsets_check"
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                           "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "paper_1305_3440_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "site_offsets_check.cu"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
