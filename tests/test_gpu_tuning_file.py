"""The autotuner's file (LGT_AUTOTUNE_CACHE): configurations that a format and gauge
have kernels for are taken from it, others are not."""
import os
import subprocess
import sys

import pytest

from test_gpu_fixed_links import lgt  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_HEAD = """
import sys
import numpy as np
sys.path.insert(0, {root!r}); sys.path.insert(0, {tests!r})
import oracle as O
from paper_1305_3440_gb300 import lgt, synth
from lattice_np import check_fp32_bound, fp32_half_sweep_bound
"""


def run_with(tmp_path, lines, code):
    import torch
    name = torch.cuda.get_device_name().replace(" ", "_")
    cache = tmp_path / "tuned"
    cache.write_text("".join(f"{f} {g} {a} {d[0]} {d[1]} {d[2]} {d[3]} {name} {c}\n" for f, g, a, d, c in lines))
    code = _HEAD.format(root=ROOT, tests=os.path.join(ROOT, "tests")) + code
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, LGT_AUTOTUNE_CACHE=str(cache)),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr


def test_lines_without_a_kernel_are_passed_over(lgt, tmp_path):
    """Lines naming a configuration that the format or gauge has no kernel for (as
    another build's file, or an edited one, may): contexts of all these kinds are
    tuned afresh, sweep and end in a documented configuration."""
    d = (4, 4, 6, 8)
    lines = [(5, 0, 0, d, 0), (6, 0, 0, d, 13), (6, 1, 0, d, 15), (4, 0, 0, d, 9), (4, 1, 0, d, 15), (7, 0, 1, d, 16),
             (0, 0, 0, d, 4), (0, 2, 0, d, 16), (2, 2, 0, d, 11), (1, 0, 1, d, 14), (6, 0, 0, d, 99), (6, 0, 0, d, -1)]
    run_with(tmp_path, lines, f"""
dims = {d}
U = synth.field(dims, 0.3, 97)
for gauge, algo, bulk, want, polish in ((0, 0, 1, "fix", "or"), (0, 0, 2, "fix", "or"), (1, 0, 2, "fix", "or"),
                                        (0, 1, 1, None, "sr"), (0, 0, 0, "f64", "f64"), (2, 0, 0, "mag", "mag"),
                                        (2, 0, 2, "mag12", "mag")):
    kinds = {{"fix": (3, 4, 8, 9, 16), "or": (0, 1, 2, 3, 4, 11, 16), "sr": (0, 1, 2, 3, 11), "f64": (0, 1, 2, 3, 16),
             "mag": (0, 1, 2, 3), "mag12": (0, 1, 2, 3, 13, 14), None: (0, 1, 2, 3, 4, 5, 6, 8, 9, 11)}}
    ctx = lgt.lgt_create(lgt.lgt_params_default(dims=dims, gauge=gauge, algo=algo, bulk=bulk, p=0.8, seed=3), U)
    lgt.lgt_sweep(ctx, 2)
    if bulk:
        lgt.lgt_promote(ctx)
        lgt.lgt_sweep(ctx, 2)
    assert np.isfinite(lgt.lgt_get_links(ctx, dims)).all()
    st = lgt.lgt_get_stats(ctx)
    lgt.lgt_destroy(ctx)
    if bulk:
        assert st.launch_config[0] in kinds[want], (gauge, algo, bulk, list(st.launch_config))
    assert st.launch_config[1] in kinds[polish], (gauge, algo, bulk, list(st.launch_config))
print("ok")
""")


@pytest.mark.parametrize("bulk,cfg", [("FP64", c) for c in (0, 1, 2, 3)] + [("FP32_12", c) for c in (0, 1, 2, 3, 13, 14)])
def test_maximally_abelian_configurations_from_the_file(lgt, tmp_path, bulk, cfg):
    """Each configuration that the tuner may pick in the maximally Abelian gauge, forced
    through the file: the stats report it and half-sweeps match the oracle (bounds of
    test_mag_half_sweep_matches_oracle)."""
    d = (4, 6, 10, 14)
    run_with(tmp_path, [(0 if bulk == "FP64" else 2, 2, 0, d, cfg)], f"""
dims = {d}
U = synth.field(dims, 0.5, 98)
for parity in (0, 1):
    ref = U.copy()
    O.half_sweep(ref, parity, gauge=O.MAG, omega=1.7)
    bound = fp32_half_sweep_bound(O.site_conditioning(U, parity, gauge=O.MAG, omega=1.7), parity, 32.0)
    ctx = lgt.lgt_create(lgt.lgt_params_default(dims=dims, gauge=lgt.LGT_MAG, bulk=lgt.LGT_{bulk}, omega=1.7), U)
    lgt.lgt_half_sweep(ctx, parity)
    out = lgt.lgt_get_working_links(ctx, dims)
    cfgs = list(lgt.lgt_get_stats(ctx).launch_config)
    lgt.lgt_destroy(ctx)
    assert cfgs[{1 if bulk == "FP64" else 0}] == {cfg}, cfgs
    err = np.abs(out - ref)
    if {bulk == "FP64"}:
        assert err.max() < 1e-12, err.max()
    else:
        ratio = check_fp32_bound(err, bound)[0]
        assert ratio <= 1.0, ratio
print("ok")
""")
