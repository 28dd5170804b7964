"""The four-threads-per-site sweeps read a site's G (or D) in all four lanes of a
quad and write it from three of them, and the lanes past a slice's last site hold
the indices of another warp's site: a run must not depend on the order in which
lanes and warps come by."""
import os
import subprocess
import sys

import pytest

from test_gpu_fixed_links import lgt  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

# slices of 66, 132 and 20 sites of a parity: the last block holds 2, 4 and 20 of 32
DIMS = [(2, 2, 2, 33 * 2), (4, 2, 6, 22), (2, 2, 2, 10)]

_RUN = """
import sys
import numpy as np
sys.path.insert(0, {root!r})
from paper_1305_3440_gb300 import lgt, synth
for dims in {dims}:
    for gauge in (0, 1):
        U = synth.field(dims, 0.5, 95)
        kw = dict(dims=dims, gauge=gauge, bulk=lgt.LGT_FP32_12, omega=1.7)
        first = None
        for again in range(3):
            ctx = lgt.lgt_create(lgt.lgt_params_default(**kw), U)
            lgt.lgt_sweep(ctx, 150)
            bulk = lgt.lgt_get_working_links(ctx, dims)
            F, th, _, _ = lgt.lgt_estimate(ctx, dims[0])
            lgt.lgt_promote(ctx)
            lgt.lgt_sweep(ctx, 150)
            full = lgt.lgt_get_links(ctx, dims)
            st = lgt.lgt_get_stats(ctx)
            lgt.lgt_destroy(ctx)
            assert list(st.launch_config) == [4, 4], list(st.launch_config)
            assert np.isfinite(bulk).all() and np.isfinite(full).all() and np.isfinite([F, th]).all()
            if first is None:
                first = bulk, full, F, th
            assert all(np.array_equal(a, b) for a, b in zip(first, (bulk, full, F, th))), (dims, gauge, again)
print("ok")
"""


def test_runs_are_reproducible_at_ragged_slices(lgt, tmp_path):
    """150 bulk and 150 polish sweeps in the four-thread configuration, three times
    over: the same links, F and theta bit for bit."""
    import torch
    name = torch.cuda.get_device_name().replace(" ", "_")
    cache = tmp_path / "tuned"
    cache.write_text("".join(f"{fmt} {gauge} 0 {d[0]} {d[1]} {d[2]} {d[3]} {name} 4\n"
                             for fmt in (4, 6) for gauge in (0, 1) for d in DIMS))
    code = _RUN.format(root=os.path.dirname(os.path.dirname(os.path.abspath(__file__))), dims=DIMS)
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, LGT_AUTOTUNE_CACHE=str(cache)),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
